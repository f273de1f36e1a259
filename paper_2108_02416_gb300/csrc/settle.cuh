// The exact lower median of single coordinates, for those that the tile kernel
// (sweep_impl.cuh) leaves open: equal values in many files (units that are off,
// gradients kept in 16 bits), a NaN, an overflowed counter.
//
// The rows' values of the open coordinates among 32 neighbours are read once,
// into shared memory, and a warp bisects the key range of one coordinate at a
// time; each step draws the range in to the keys that occur in it.  Equal values
// end at once, two values after one step, 455 continuous ones after about
// twelve, and 32 steps always suffice.  (Four radix passes over the rows in
// global memory took 6.9 ms for 1,048,576 coordinates of 455 equal values, this
// 0.7.)
#pragma once

#include "median_common.cuh"

namespace aspis {

// Words of shared memory for the keys of `most` coordinates.
__host__ __device__ constexpr int settle_words(int n, int most)
{
    return most * ((n + 31) / 32 * 32) + 32;
}

// The range of a coordinate's keys i0, i0 + step, ...; the values become keys
// (read again by the same lane alone).
__device__ __forceinline__ void key_range(uint32_t *keys, int i0, int step, int n, uint32_t &lo, uint32_t &hi)
{
    lo = 0xffffffffu;
    hi = 0u;
#pragma unroll 8
    for (int i = i0; i < n; i += step) {
        const uint32_t x = to_key(keys[i]);
        keys[i] = x;
        lo = min(lo, x);
        hi = max(hi, x);
    }
}

// How many of them are up to mid, the largest of those, and the next one above.
__device__ __forceinline__ void key_split(const uint32_t *keys, int i0, int step, int n, uint32_t mid, uint32_t &low,
                                          uint32_t &below, uint32_t &above)
{
    low = 0u;
    below = 0u;
    above = 0xffffffffu;
#pragma unroll 8
    for (int i = i0; i < n; i += step) {
        const uint32_t x = keys[i];
        if (x <= mid) {
            ++low;
            below = max(below, x);
        } else {
            above = min(above, x);
        }
    }
}

// Bit k of open: coordinate c0 + k is settled.  Called by a whole block of NT
// threads; row_of(i) is the i-th of the n aggregated rows, stage holds
// settle_words(n, number of bits) words.
template <int NT, class Row>
__device__ __forceinline__ void settle(const float *copies, int64_t ld, int n, Row row_of, int64_t c0, uint32_t open,
                                       uint32_t *stage, float *out)
{
    constexpr int kNW = NT / 32;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, many = __popc(open);
    const uint32_t krank = (uint32_t)((n - 1) / 2);
    // a warp copies one word of 2^sh coordinates from 32 / 2^sh rows, to 32 banks
    const int sh = 32 - __clz(many - 1), rows = 32 >> sh, pitch = (n + 31) / 32 * 32 + rows;
    const int mine = lane & ((1 << sh) - 1);
    if (mine < many) {
        const float *at = copies + c0 + __fns(open, 0, mine + 1);
        const uint32_t to = (uint32_t)__cvta_generic_to_shared(stage + mine * pitch);
#pragma unroll 4
        for (int i = w * rows + (lane >> sh); i < n; i += kNW * rows)
            cp_async4(to + i * 4u, at + (int64_t)row_of(i) * ld);
        cp_async_commit();
        cp_async_wait_all();
    }
    __syncthreads();
    uint32_t lo, hi, low, below, above;                         // the median lies in [lo, hi]
    if (many * 2 > kNW) {
        // a warp per coordinate
        for (int q = w; q < many; q += kNW) {
            uint32_t *keys = stage + q * pitch;
            key_range(keys, lane, 32, n, lo, hi);
            lo = __reduce_min_sync(full, lo);
            hi = __reduce_max_sync(full, hi);
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo) / 2u;
                key_split(keys, lane, 32, n, mid, low, below, above);
                if (krank < __reduce_add_sync(full, low)) hi = __reduce_max_sync(full, below);
                else lo = __reduce_min_sync(full, above);
            }
            if (lane == 0) out[c0 + __fns(open, 0, q + 1)] = __uint_as_float(from_key(lo));
        }
    } else {
        // few coordinates: the warps share them, 2 or more each
        __shared__ uint32_t part[kNW][3];
        const int share = kNW / many, q = w % many, s = w / many;
        uint32_t *keys = stage + q * pitch;
        auto combine = [&](uint32_t a, uint32_t b, uint32_t c) {
            a = __reduce_add_sync(full, a);
            b = __reduce_max_sync(full, b);
            c = __reduce_min_sync(full, c);
            if (lane == 0) {
                part[w][0] = a;
                part[w][1] = b;
                part[w][2] = c;
            }
            __syncthreads();
            const int from = (q + (lane < share ? lane : 0) * many);
            low = __reduce_add_sync(full, lane < share ? part[from][0] : 0u);
            below = __reduce_max_sync(full, part[from][1]);
            above = __reduce_min_sync(full, part[from][2]);
        };
        const int i0 = s < share ? s * 32 + lane : n;
        key_range(keys, i0, share * 32, n, lo, hi);
        combine(0u, hi, lo);
        lo = above;
        hi = below;
        while (__syncthreads_or(lo < hi)) {
            const uint32_t mid = lo + (hi - lo) / 2u;
            key_split(keys, i0, share * 32, n, mid, low, below, above);
            combine(low, below, above);
            if (lo < hi) {
                if (krank < low) hi = below;
                else lo = above;
            }
        }
        if (s == 0 && lane == 0) out[c0 + __fns(open, 0, q + 1)] = __uint_as_float(from_key(lo));
    }
    __syncthreads();
}

}  // namespace aspis
