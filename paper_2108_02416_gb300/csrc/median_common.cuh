// Pieces of the coordinate-wise aggregation: the totalOrder
// key map, the value-space bin map, tag matching, compensated sums and the
// search modes of the lower median.
#pragma once

#include <utility>

#include <stdint.h>

namespace aspis {

constexpr int kNB = 128;          // key-space histogram rows of the exact path
constexpr int kLogNB = 7;         // key bits resolved per key-space pass
constexpr int kVB = 256;          // value-space histogram rows
constexpr int kTopBin = 254;      // value-space bins are 0..kTopBin
constexpr uint32_t kPadTag = 0xFFu;   // tag byte of a missing row: no value-space bin

// IEEE totalOrder as unsigned order: flip all bits of negatives, the sign
// bit of non-negatives.  A bijection, so the median's bits come back exactly.
__device__ __forceinline__ uint32_t to_key(uint32_t u)
{
    return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}

__device__ __forceinline__ uint32_t from_key(uint32_t k)
{
    return k ^ ((uint32_t)((int32_t)~k >> 31) | 0x80000000u);
}

// Value-space bin of x, as the bits of 2^23 + bin: y = sat(x*s + c) in
// [0, 1] (fma with saturation: NaN gives +0), then 2^23 + rint(254*y), whose
// low byte is the bin 0..254.  Both steps are correctly rounded and
// non-decreasing, so the map is monotone in the IEEE totalOrder of every
// non-NaN x (+0 and -0 share a bin) and always lands in 0..254, whatever s
// and c are.  NaNs are detected separately.
__device__ __forceinline__ uint32_t vbin_bits(float x, float s, float c)
{
    float y;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(x), "f"(s), "f"(c));
    return __float_as_uint(fmaf(y, (float)kTopBin, 8388608.0f));
}

enum { M_DONE = 0, M_VH, M_VC, M_VM, M_KA, M_KH, M_KC };

// Four tag bytes against the target bytes of vbx: 0x80 in each byte whose tag
// equals its target, 0 elsewhere.  Exact for every byte value: the sum of a
// byte's low seven bits and 0x7F sets its top bit iff they are not all zero
// and cannot carry into the next byte.  (Targets of coordinates that search
// nothing are 0xFF, equal to the padding tag; callers skip such hits.)
__device__ __forceinline__ uint32_t tag_match(uint32_t w, uint32_t vbx)
{
    const uint32_t x = w ^ vbx;
    return ~(((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x) & 0x80808080u;
}

// Two-sum: s + e == a + b exactly (Knuth); no products, so nothing to fuse.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    const float bp = s - a;
    e = (a - (s - bp)) + (b - bp);
}

// Histogram increment.  No memory clobber: the counters are read only after a
// block barrier, so ordinary loads and stores may move across these.
template <uint32_t INC>
__device__ __forceinline__ void red_shared(uint32_t saddr)
{
    asm volatile("red.shared.add.u32 [%0], %1;\n" ::"r"(saddr), "n"(INC));
}

__device__ __forceinline__ void cp_async4(uint32_t saddr, const void *g)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(saddr), "l"(g) : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void *p)
{
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p));
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// ascending bitonic sorting network over N registers (N a power of two)
template <int N>
__device__ __forceinline__ void sort_net(uint32_t (&y)[N])
{
#pragma unroll
    for (int k = 2; k <= N; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int l = i ^ j;
                if (l > i) {
                    const uint32_t a = y[i], b = y[l];
                    const bool up = (i & k) == 0;
                    y[i] = up ? min(a, b) : max(a, b);
                    y[l] = up ? max(a, b) : min(a, b);
                }
            }
}

// the 32 values of a warp (one per lane) sorted ascending across the lanes
// (bitonic: lane i meets lane i ^ j; the lower lane of an ascending block
// keeps the minimum)
__device__ __forceinline__ uint32_t warp_sort32(uint32_t x, int lane)
{
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
            const bool up = (lane & k) == 0, lower = (lane & j) == 0;
            x = lower == up ? min(x, y) : max(x, y);
        }
    return x;
}

// flag |= 1 if any of a, b, c, e is NaN (one compare per pair)
__device__ __forceinline__ void nan_check(uint32_t &flag, float a, float b, float c, float e)
{
    asm("{\n .reg .pred p;\n setp.nan.f32 p, %1, %2;\n setp.nan.or.f32 p, %3, %4, p;\n"
        " @p mov.b32 %0, 1;\n}\n" : "+r"(flag) : "f"(a), "f"(b), "f"(c), "f"(e));
}

// the low bytes of four words, packed into one word
__device__ __forceinline__ uint32_t pack4(uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3)
{
    return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
}

// mean of the values x[s] of the slots s in m (fp32: x0 plus the
// mean of the deviations from it; 0 where a copy equals x0 bit for bit); s0 = the
// lowest slot of m, k = |m|; every index is a compile-time slot
template <int R>
__device__ __forceinline__ float mean_masked(const float (&x)[R], uint32_t m, int s0, int k)
{
    if (k == R) {                          // all copies: nothing to pick, a constant divisor
        const uint32_t b = __float_as_uint(x[0]);
        float sum = 0.f;
#pragma unroll
        for (int s = 1; s < R; ++s)
            sum = __fadd_rn(sum, __float_as_uint(x[s]) == b ? 0.f : __fsub_rn(x[s], x[0]));
        return sum == 0.f ? x[0] : __fadd_rn(x[0], __fdiv_rn(sum, (float)R));
    }
    float x0 = x[0];
#pragma unroll
    for (int s = 1; s < R; ++s)
        if (s == s0) x0 = x[s];
    const uint32_t b0 = __float_as_uint(x0);
    float acc = 0.f;
#pragma unroll
    for (int s = 0; s < R; ++s)
        if ((m >> s) & 1u) {
            const float e = __float_as_uint(x[s]) == b0 ? 0.f : __fsub_rn(x[s], x0);
            acc = __fadd_rn(acc, e);
        }
    return acc == 0.f ? x0 : __fadd_rn(x0, __fdiv_rn(acc, (float)k));
}

// Ascending odd-even merge sort of N <= 64 keys in registers (Batcher 1968):
// the comparators of the 32-key (64-key) network, those that touch a key beyond
// N dropped (they would meet the largest key).
struct Network {
    int n = 0;
    unsigned char a[544] = {}, b[544] = {};
};

template <int N>
__host__ __device__ constexpr Network merge_network()
{
    constexpr int kWide = N <= 32 ? 32 : 64;
    Network net{};
    for (int p = 1; p < kWide; p *= 2)
        for (int k = p; k >= 1; k /= 2)
            for (int j = k % p; j + k < kWide; j += 2 * k)
                for (int i = 0; i < k; ++i)
                    if (i + j + k < N && (i + j) / (2 * p) == (i + j + k) / (2 * p)) {
                        net.a[net.n] = (unsigned char)(i + j);
                        net.b[net.n] = (unsigned char)(i + j + k);
                        ++net.n;
                    }
    return net;
}

template <int A, int B, int N>
__device__ __forceinline__ void compare_exchange(uint32_t (&y)[N])
{
    const uint32_t a = y[A], b = y[B];
    y[A] = min(a, b);
    y[B] = max(a, b);
}

template <int N, int... I>
__device__ __forceinline__ void merge_sort(uint32_t (&y)[N], std::integer_sequence<int, I...>)
{
    constexpr Network net = merge_network<N>();
    (compare_exchange<net.a[I], net.b[I]>(y), ...);
}

template <int N>
__device__ __forceinline__ void merge_sort(uint32_t (&y)[N])
{
    merge_sort<N>(y, std::make_integer_sequence<int, merge_network<N>().n>{});
}

}  // namespace aspis
