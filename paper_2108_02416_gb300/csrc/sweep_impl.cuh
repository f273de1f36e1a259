// The kernel declared in sweep.cuh, instantiated per number of copies in
// sweep_r*.cu.
#pragma once

#include "settle.cuh"
#include "sweep.cuh"

namespace aspis {
namespace {

// Repairs: the kernel runs only where bit 1 of gate->success asks for it, and
// the last block to leave takes the request back (blocks are counted from bit
// 8 up; every block has read the request by then).  gate = NULL: always.
__device__ __forceinline__ bool gate_open(const aspis_detection *gate)
{
    return !gate || (*(volatile const int32_t *)&gate->success & 2);
}

__device__ __forceinline__ void gate_leave(aspis_detection *gate)
{
    if (!gate) return;
    const int32_t old = atomicAdd(&gate->success, 256);
    if ((old >> 8) == (int32_t)gridDim.x - 1) *(volatile int32_t *)&gate->success = old & 1;
}

constexpr int kNT = 384, kWarps = kNT / 32;
constexpr int TC = 128;                     // coordinates per tile, four per lane
// What the sweep computes: the median with tag bytes, the mean, or the median
// without tags, from a second pass over the chosen rows.
enum Mode { TAGGED = 0, MEAN = 1, TWO_PASS = 2 };
// List entries per coordinate (CAP; the two-pass median's bins are wider).  A
// bin has n / 120 members on average.  Two blocks share the SM up to 456 files
// with 32 entries and up to kPairFiles with 16, which are hardly ever exceeded
// there by continuous values (495 files, d = 1,048,576: 456 us, 723 with a block
// alone); values kept in 16 bits, whose grid is coarser than the bins, do exceed
// them (1,211 and 820).  A block alone takes 64 where they fit (kLongFiles): of
// such values at 816 files it leaves 881 coordinates of 524,288 open, not 56,173
// (672 us, not 1,136).
template <int MODE, int CAP>
__host__ __device__ constexpr int list_cap() { return MODE == TWO_PASS ? 96 : CAP; }
constexpr int kHistWords = kVB * 32;        // four 8-bit counters per (bin, lane)
constexpr int kBPW = (kVB + kWarps - 1) / kWarps;
constexpr int kSample = 2 * kWarps;         // sampled values per coordinate
constexpr float kReach = 14.0f;             // farthest bin from the centre, in inner ranges of the sample
constexpr int kDropped = 15;                // slot of a file that is not aggregated
// per-coordinate state, arrays of TC words
//   S_VS, S_VC  scale and offset of the value bins
//   S_PEND      the pending tile's listed bin: count | rank in it << 8
//   S_BIN       target bin, kListed where its members are listed
//   S_PART      the bin search's partial sums (six arrays' room)
enum { S_VS, S_VC, S_LCNT, S_PEND, S_BIN, S_PART, kStateWords = S_PART + 6 };
static_assert(6 * TC * 4 >= kWarps * 32 * 8, "room for the partial sums");
constexpr uint32_t kListed = 0x100u, kLive = 0x200u;

struct SweepLayout {
    size_t tags, hist, list, state, meta, total;
};

template <int MODE, int CAP>
__host__ __device__ inline SweepLayout sweep_layout(int64_t f)
{
    SweepLayout L{};
    int64_t per_warp = (f + kWarps - 1) / kWarps;
    if (per_warp < 8) per_warp = 8;          // the sampled keys use a warp's first eight tag rows
    size_t o = 0;
    L.tags = o; o += MODE == TAGGED ? (size_t)per_warp * kWarps * 128 : 0;
    L.hist = o; o += MODE != MEAN ? (size_t)kHistWords * 4 : 0;
    L.list = o; o += (size_t)list_cap<MODE, CAP>() * TC * 4;      // (the mean: its partial sums)
    L.state = o; o += MODE != MEAN ? (size_t)kStateWords * TC * 4 : 0;
    L.meta = o; o += ((size_t)f * 4 + 15) / 16 * 16;
    L.total = o;
    return L;
}

// A row start is aligned to W floats (4, 2 or 1), the widest load it allows: a
// lane holds W neighbouring coordinates of each of the 4 / W parts of the
// tile's 128-float row segment.  off_of: element k of a lane, from its first;
// seg_at: coordinate c of a tile (lane c / 4, element c % 4), from the tile's.
template <int W>
__host__ __device__ constexpr int off_of(int k)
{
    return k % W + k / W * 32 * W;
}

template <int W>
__device__ __forceinline__ int seg_at(int c)
{
    return (c >> 2) * W + off_of<W>(c & 3);
}

// the first kl elements of a lane (a pair or four are loaded whole: what lies
// beyond d is padding of the same row)
template <int W, bool STREAM>
__device__ __forceinline__ void load_lane(uint4 &x, const char *p, int kl)
{
    if constexpr (W == 4) {
        const uint4 *e = reinterpret_cast<const uint4 *>(p);
        if (kl > 0) x = STREAM ? __ldcs(e) : __ldcg(e);
    } else if constexpr (W == 2) {
        const uint2 *e = reinterpret_cast<const uint2 *>(p);
        if (kl > 0) {
            const uint2 y = STREAM ? __ldcs(e) : __ldca(e);
            x.x = y.x;
            x.y = y.y;
        }
        if (kl > 2) {
            const uint2 y = STREAM ? __ldcs(e + 32) : __ldca(e + 32);
            x.z = y.x;
            x.w = y.y;
        }
    } else {
        // (the four 128-byte parts of an unaligned segment share lines: through L1)
        const unsigned int *e = reinterpret_cast<const unsigned int *>(p);
        if (kl > 0) x.x = STREAM ? __ldcs(e) : __ldca(e);
        if (kl > 1) x.y = STREAM ? __ldcs(e + 32) : __ldca(e + 32);
        if (kl > 2) x.z = STREAM ? __ldcs(e + 64) : __ldca(e + 64);
        if (kl > 3) x.w = STREAM ? __ldcs(e + 96) : __ldca(e + 96);
    }
}

__device__ __forceinline__ uint32_t el(const uint4 &x, int k)
{
    return k == 0 ? x.x : k == 1 ? x.y : k == 2 ? x.z : x.w;
}

__device__ __forceinline__ uint32_t vdiff(const uint4 &a, const uint4 &b)
{
    return (a.x ^ b.x) | (a.y ^ b.y) | (a.z ^ b.z) | (a.w ^ b.w);
}

// The file (a multiple of 8) that a tile's order starts from: its first kSample
// files are the sample, so as few of them as possible shall be marked (bit 31:
// their copies differ).  Neighbours in file order share workers, and with them
// distortions, so some window has few even where a quarter of all files is
// distorted.  (A sample spread over the file order is as good, but rows taken
// from all over the copies at a tile's start cost 7 to 10% of the pass at 61
// GB, read once or twice, prefetched or not.)  Called by the whole block; marked
// holds n words, in the list, which every layout makes long enough.
__device__ __forceinline__ int cleanest_start(const uint32_t *marked, int n, int *best)
{
    if (n < 2 * kSample) return 0;
    for (int i = threadIdx.x * 8; i < n; i += kNT * 8) {
        int cnt = 0;
        for (int q = 0; q < kSample; ++q) cnt += (int)(marked[i + q < n ? i + q : i + q - n] >> 31);
        atomicMin(best, (cnt << 16) | i);
    }
    __syncthreads();
    return *best & 0xFFFF;
}

// Files whose copies one thread holds in registers at a time (minb blocks
// share the SM's registers).  Measured on whole rounds: with two blocks, R = 3
// takes 3.52 ms per 2^22 coordinates of 455 files with 2 files in flight,
// 4.50 with 3 (the extra registers spill) and 4.79 with 1.
__host__ __device__ constexpr int batch_files(int R, int minb)
{
    return minb == 1 ? (R <= 2 ? 8 : 4) : R <= 2 ? 4 : 2;
}

// Whether one of the lane's keys (a: entry `lane`, b: entry `lane + 32`) is the
// element of rank rk among the warp's first cnt <= 64 entries: every lane
// counts the entries below and at its own, by independent shuffles.  Returns 1
// for a, 2 for b, 0 for neither.
__device__ __forceinline__ int warp_ranked(uint32_t a, uint32_t b, uint32_t cnt, uint32_t rk)
{
    const unsigned full = 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t lta = 0u, lea = 0u, ltb = 0u, leb = 0u;
#pragma unroll 4
    for (uint32_t e = 0; e < cnt; ++e) {
        const uint32_t y = __shfl_sync(full, e < 32u ? a : b, (int)(e & 31u));
        lta += y < a;
        lea += y <= a;
        ltb += y < b;
        leb += y <= b;
    }
    if (lane < cnt && lta <= rk && rk < lea) return 1;
    if (lane + 32u < cnt && ltb <= rk && rk < leb) return 2;
    return 0;
}

// The coordinates that a block left open (kOpen in its part of out), at the end
// of its sweep: for few tiles of few files (kSettleFiles), where fixup_kernel's
// launch costs more (the round of 84 files of three at d = 4,096: 28 us, 31 with
// fixup_kernel; equal at 220 files, but 36 and 36 at 455 and 55 and 51 at 1,140).
// In larger calls the mere presence of this call costs the sweep 5 to 9%.  stage:
// room for 32 coordinates' keys.
__device__ __noinline__ void settle_open(const SweepArgs &A, uint32_t *stage, const uint32_t *meta, int n,
                                         int64_t t0, int64_t tstep)
{
    __shared__ uint32_t open_s[TC / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t c0 = t0 * TC; c0 < A.d; c0 += tstep * TC) {
        if (w < TC / 32) {
            const int64_t c = c0 + w * 32 + lane;
            const uint32_t x = c < A.d ? __ldcg(reinterpret_cast<const unsigned int *>(A.out) + c) : 0u;
            const uint32_t m = __ballot_sync(0xffffffffu, x == kOpen);
            if (lane == 0) open_s[w] = m;
        }
        __syncthreads();
        for (int g = 0; g < TC / 32; ++g)
            if (open_s[g])
                settle<kNT>(A.copies, A.ld, n, [&](int i) { return meta[i]; }, c0 + g * 32, open_s[g], stage, A.out);
        __syncthreads();
    }
}

// AVG: a file's value is the average of its copies in slot_mask; the meta word
// holds the mask in place of slot and pair word.
template <int R, int W, int MODE, int MINB, bool AVG, int CAP, bool SETTLE>
__global__ void __launch_bounds__(kNT, MINB)
sweep_kernel(const SweepArgs A)
{
    chain();
    if (R == 1 && !gate_open(A.gate)) return;
    constexpr int kShort = MINB == 1 || (MODE == TWO_PASS && R == 1) ? 16 : 8;   // longest list one thread sorts
    constexpr int kF = R == 1 && W == 4 && MODE == MEAN ? 6 : batch_files(R, MINB);
    constexpr int kRows = kF * R;
    static_assert(kF >= 2, "the sample is the first two files of every warp");
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr uint32_t cap = (uint32_t)list_cap<MODE, CAP>();
    const SweepLayout L = sweep_layout<MODE, CAP>(A.f);
    uint32_t *tags = reinterpret_cast<uint32_t *>(smem + L.tags);     // [warp's file][kWarps][32]
    // the sampled keys: a warp's own first tag rows, which nothing else reads,
    // or (no tags) the list, empty at a tile's start
    uint32_t *keys = reinterpret_cast<uint32_t *>(smem + (MODE == TWO_PASS ? L.list : L.tags));
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem + L.hist);     // [kVB][32]
    uint32_t *list = reinterpret_cast<uint32_t *>(smem + L.list);     // [cap][TC]
    uint32_t *st = reinterpret_cast<uint32_t *>(smem + L.state);      // [kStateWords][TC]
    // by place in the tile's order: slot | pair word << 4 | file << 16, or
    // (R = 1) the kept row
    uint32_t *meta = reinterpret_cast<uint32_t *>(smem + L.meta);
    uint2 *part = reinterpret_cast<uint2 *>(st + S_PART * TC);        // [kWarps][32]
    __shared__ int n_s, start_s, warp_tot[kWarps];
    __shared__ int n_long[2];           // listed bins with more than kShort members, by tile parity
    __shared__ uint8_t long_c[TC];

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned full = 0xffffffffu;
    const int f = A.f;
    const int64_t d = A.d;
    const uint64_t ldb = (uint64_t)A.ld * 4u;
    const uint32_t hist_s = (uint32_t)__cvta_generic_to_shared(hist);
    const uint32_t list_s = (uint32_t)__cvta_generic_to_shared(list);
    auto S = [&](int k, int c) -> uint32_t & { return st[k * TC + c]; };

    if (tid == 0) {
        n_s = 0;
        start_s = 0x7fffffff;
        n_long[0] = n_long[1] = 0;
    }
    if constexpr (MODE != MEAN) {
        for (int i = tid; i < TC; i += kNT) {
            S(S_LCNT, i) = 0u;
            S(S_PEND, i) = 0u;
        }
        for (int i = tid * 4; i < kHistWords; i += kNT * 4)
            *reinterpret_cast<uint4 *>(hist + i) = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
    int n = 0, start = 0;
    if constexpr (R == 1) {
        // the kept rows in file order
        for (int b0 = 0; b0 < f; b0 += kNT) {
            const int i = b0 + tid, s = i < f ? (int)A.sel[i] : -1;
            const unsigned m = __ballot_sync(full, s >= 0);
            if (lane == 0) warp_tot[w] = __popc(m);
            __syncthreads();
            int off = n;
            for (int q = 0; q < kWarps; ++q) {
                off += q < w ? warp_tot[q] : 0;
                n += warp_tot[q];
            }
            // (a mean takes them in this order, a median from a chosen start)
            uint32_t *to = MODE != MEAN ? list : meta;
            if (s >= 0)
                to[off + __popc(m & ((1u << lane) - 1u))] = (uint32_t)(i * A.r + s) | (s > 0 ? 0x80000000u : 0u);
            __syncthreads();
        }
        if constexpr (MODE != MEAN) {
            start = cleanest_start(list, n, &start_s);
            for (int i = tid; i < n; i += kNT) meta[(i < start ? n : 0) + i - start] = list[i] & 0x7fffffffu;
            __syncthreads();
        } else {
            for (int i = tid; i < n; i += kNT) meta[i] &= 0x7fffffffu;
            __syncthreads();
        }
        if (n == 0) {
            if (tid == 0) {
                if (blockIdx.x == 0) A.det->status = ASPIS_E_EMPTY;
                gate_leave(A.gate);
            }
            return;
        }
    } else {
        if constexpr (MODE != MEAN) {
            for (int i = tid; i < f; i += kNT) {
                const bool marked = AVG ? A.slot_mask[i] != (1u << R) - 1u : A.sel[i] < 0 || A.sel[i] >= kUnclean;
                list[i] = marked ? 0x80000000u : 0u;
            }
            __syncthreads();
            start = cleanest_start(list, f, &start_s);
        }
        if constexpr (MODE == MEAN) {
            // the kept files first, in file order, and the others from the end: a
            // warp sums the same values in the same order as the separate mean
            for (int b0 = 0; b0 < f; b0 += kNT) {
                const int i = b0 + tid, s = i < f ? (int)A.sel[i] : -1;
                const unsigned m = __ballot_sync(full, s >= 0);
                if (lane == 0) warp_tot[w] = __popc(m);
                __syncthreads();
                int off = n + __popc(m & ((1u << lane) - 1u));
                for (int q = 0; q < kWarps; ++q) {
                    off += q < w ? warp_tot[q] : 0;
                    n += warp_tot[q];
                }
                if (i < f)
                    meta[s >= 0 ? off : f - 1 - (i - off)] =
                        (uint32_t)(s < 0 ? kDropped : s & (kUnclean - 1)) | ((uint32_t)i << 16);
                __syncthreads();
            }
        } else {
            int mine = 0;
            for (int i = tid; i < f; i += kNT) {
                const int s = A.sel[i];
                meta[(i < start ? f : 0) + i - start] =
                    (AVG ? (uint32_t)A.slot_mask[i] : (uint32_t)(s < 0 ? kDropped : s & (kUnclean - 1))) |
                    ((uint32_t)i << 16);
                mine += AVG ? A.slot_mask[i] != 0 : s >= 0;
            }
            mine = __reduce_add_sync(full, mine);
            if (lane == 0 && mine) atomicAdd(&n_s, mine);
            __syncthreads();
            n = n_s;
        }
    }
    const uint32_t krank = (uint32_t)((n - 1) / 2);
    // With more files the bins span more than the sample's range, so that the
    // 8-bit counters of the two outer bins (4% of the values on average, up to
    // four times that) hold; a wider span puts more members in a bin.
    const float widen = n <= 640 ? 0.0f : n <= 1024 ? 0.125f : n <= 2500 ? 0.25f : n <= 4096 ? 0.375f : 0.5f;
    const int64_t ntiles = (d + TC - 1) / TC;

    const int nf = R == 1 ? n : f;                                    // files of a tile
    const int nmine = nf > w ? (nf - w + kWarps - 1) / kWarps : 0;    // of this warp
    auto word_of = [&](int j) -> uint32_t { return meta[w + j * kWarps]; };
    // the slot of the chosen (AVG: of the first averaged) copy
    auto slot_of = [&](int j) -> int {
        if constexpr (AVG) return word_of(j) & 0xFFu ? __ffs((int)(word_of(j) & 0xFFu)) - 1 : kDropped;
        return R == 1 ? 0 : (int)(word_of(j) & 15u);
    };
    // a file's copies start here, from the lane's base in row 0
    auto file_at = [&](const char *base, int j) -> const char * {
        return base + (uint64_t)(R == 1 ? word_of(j) : (word_of(j) >> 16) * R) * ldb;
    };
    // the lane's part of tile t: address in row 0, and how many of its four
    // coordinates exist
    auto lane_base = [&](int64_t t) -> const char * {
        return reinterpret_cast<const char *>(A.copies + t * TC + lane * W);
    };
    auto live_of = [&](int64_t t) -> int {
        if (t >= ntiles) return 0;
        const int64_t left = d - t * TC;
        if (left >= TC) return 4;
        int kl = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) kl += lane * W + off_of<W>(k) < left;
        return kl;
    };
    auto load_file = [&](uint4 (&x)[R], const char *p, int kl, uint32_t mask) {
#pragma unroll
        for (int s = 0; s < R; ++s) {
            if (AVG && !((mask >> s) & 1u)) continue;
            const char *q = p + (uint64_t)s * ldb;
            // the copies of slot 0 are the usual choice: they stay in L2 for
            // the member lists, the others are first to go
            if (s == 0 || (W < 4 && MODE == MEAN)) load_lane<W, false>(x[s], q, kl);
            else load_lane<W, true>(x[s], q, kl);
        }
    };

    uint4 xa[kF][R];
    {
        const char *p = lane_base(blockIdx.x);
        const int kl = live_of(blockIdx.x);
#pragma unroll
        for (int u = 0; u < kF; ++u) {
#pragma unroll
            for (int s = 0; s < R; ++s) xa[u][s] = make_uint4(0u, 0u, 0u, 0u);
            if (u < nmine) load_file(xa[u], file_at(p, u), kl, word_of(u));
        }
    }

    uint32_t open_cnt = 0u;             // coordinates left to fixup_kernel (threads < TC)
    bool have_p = false;
    int64_t c0_p = 0;
    int par = 0;

    // Rank the pending tile's listed bins: lists of at most kShort keys one
    // thread per coordinate, longer ones (queued by the bin search) one warp
    // per coordinate.
    auto rank_pending = [&](int parity) {
        if (tid < TC) {
            const int c = tid;
            const uint32_t cnt = S(S_PEND, c) & 0xFFu, rk = S(S_PEND, c) >> 8;
            if (cnt != 0u && cnt <= (uint32_t)kShort) {
                uint32_t y[kShort];
#pragma unroll
                for (int e = 0; e < kShort; ++e) y[e] = (uint32_t)e < cnt ? to_key(list[e * TC + c]) : 0xffffffffu;
                sort_net<kShort>(y);
                uint32_t res = y[0];
#pragma unroll
                for (int e = 1; e < kShort; ++e) res = (uint32_t)e == rk ? y[e] : res;
                A.out[c0_p + seg_at<W>(c)] = __uint_as_float(from_key(res));
            }
        }
        const int nl = n_long[parity];
        for (int q = (w - TC / 32 + kWarps) % kWarps; q < nl; q += kWarps) {
            const int c = long_c[q];
            const uint32_t cnt = S(S_PEND, c) & 0xFFu, rk = S(S_PEND, c) >> 8;
            if (cap <= 32u || cnt <= 32u) {
                const uint32_t x = warp_sort32((uint32_t)lane < cnt ? to_key(list[lane * TC + c]) : 0xffffffffu, lane);
                const uint32_t res = __shfl_sync(full, x, (int)rk);
                if (lane == 0) A.out[c0_p + seg_at<W>(c)] = __uint_as_float(from_key(res));
                continue;
            }
            if (cap <= 64u || cnt <= 64u) {
                // (equal keys: several lanes write the same bits)
                const uint32_t a = list[lane * TC + c], b = (uint32_t)lane + 32u < cnt ? list[(lane + 32) * TC + c] : 0u;
                const int is = warp_ranked(to_key(a), to_key(b), cnt, rk);
                if (is) A.out[c0_p + seg_at<W>(c)] = __uint_as_float(is == 1 ? a : b);
                continue;
            }
            for (uint32_t e = (uint32_t)lane; e < cnt; e += 32u) {
                const uint32_t x = to_key(list[e * TC + c]);
                uint32_t lt = 0u, le = 0u;
                for (uint32_t i = 0; i < cnt; ++i) {
                    const uint32_t y = to_key(list[i * TC + c]);
                    lt += y < x;
                    le += y <= x;
                }
                if (lt <= rk && rk < le) A.out[c0_p + seg_at<W>(c)] = __uint_as_float(from_key(x));
            }
        }
    };

    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t c0 = t * TC, tn = t + gridDim.x;
        const int kl = live_of(t), kln = live_of(tn);
        const bool ragged = d - c0 < TC;
        const char *lb = lane_base(t), *lbn = lane_base(kln ? tn : t);

        // values beyond d do not count as differences
        auto mask_tail = [&](uint4 (&x)[R]) {
#pragma unroll
            for (int s = 0; s < R; ++s) {
                if (kl < 1) x[s].x = 0u;
                if (kl < 2) x[s].y = 0u;
                if (kl < 3) x[s].z = 0u;
                if (kl < 4) x[s].w = 0u;
            }
        };
        // files j.. of a batch into L2, one 128-byte line per lane.  An
        // unaligned segment lies in five lines; the fifth is left to the next
        // tile where it would take one more instruction per batch (which cost
        // 3 to 5% with two or four copies; without it three copies lost 14%).
        constexpr int kLines = W < 4 && MODE != MEAN && (kRows * 5 + 31) / 32 == (kRows * 4 + 31) / 32 ? 5 : 4;
        auto prefetch_batch = [&](int64_t cb, int j) {
#pragma unroll
            for (int q0 = 0; q0 < kRows * kLines; q0 += 32) {
                const int q = q0 + lane, row = q / kLines, col = q % kLines * 32, jp = j + row / R;
                if (q < kRows * kLines && jp < nmine && cb + col < d && (!AVG || (word_of(jp) >> (row % R)) & 1u))
                    prefetch_l2(file_at(reinterpret_cast<const char *>(A.copies + cb + col), jp) +
                                (uint64_t)(row % R) * ldb);
            }
        };
        // One pass over this warp's files, kF at a time; a file's registers
        // are refilled as soon as it is compared, the last ones with the next
        // tile's first files.  fn(v, j): the guessed copy of the warp's j-th
        // file; skip(j): a file without one.  (TWO_PASS: refilled with the
        // second pass's first rows instead.)
        auto chosen_at = [&](int j) -> const char * { return file_at(lb, j) + (uint64_t)slot_of(j) * ldb; };
        auto load_chosen = [&](uint4 &x, int j) {
            if (j < nmine && slot_of(j) != kDropped) load_lane<W, false>(x, chosen_at(j), kl);
        };
        auto sweep = [&](auto fn, auto skip) {
            auto file = [&](uint4 (&x)[R], int j) {
                if constexpr (R == 1) {
                    fn(x[0], j);
                    return;
                }
                if constexpr (AVG) {
                    const uint32_t m = word_of(j) & 0xFFu;
                    if (!m) {
                        skip(j);
                        return;
                    }
                    const int s0 = __ffs((int)m) - 1, many = __popc(m);
                    uint32_t v[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        float a[R];
#pragma unroll
                        for (int s = 0; s < R; ++s) a[s] = __uint_as_float(el(x[s], k));
                        v[k] = __float_as_uint(mean_masked<R>(a, m, s0, many));
                    }
                    float *to = A.means + (int64_t)(word_of(j) >> 16) * A.ldm + c0 + lane * 4;
                    if (kl == 4) {
                        __stcg(reinterpret_cast<uint4 *>(to), make_uint4(v[0], v[1], v[2], v[3]));
                    } else {
#pragma unroll
                        for (int k = 0; k < 3; ++k)
                            if (k < kl) to[k] = __uint_as_float(v[k]);
                    }
                    fn(make_uint4(v[0], v[1], v[2], v[3]), j);
                    return;
                }
                if (ragged) mask_tail(x);
                const int slot = slot_of(j);
                uint32_t df = 0u;
#pragma unroll
                for (int s = 1; s < R; ++s) df |= vdiff(x[0], x[s]);
                uint4 v = x[0];
                if (__any_sync(full, df != 0u)) {
                    uint32_t neq = 0u;
                    int p = 0;
#pragma unroll
                    for (int s = 0; s < R; ++s)
#pragma unroll
                        for (int q = s + 1; q < R; ++q, ++p) neq |= (vdiff(x[s], x[q]) != 0u ? 1u : 0u) << p;
                    neq = __reduce_or_sync(full, neq);
                    if (lane == 0) meta[w + j * kWarps] |= neq << 4;
#pragma unroll
                    for (int s = 1; s < R; ++s)
                        if (slot == s) v = x[s];
                }
                if (slot != kDropped) fn(v, j);
                else skip(j);
            };
            int j0 = 0;
            for (; j0 + kF < nmine; j0 += kF) {
                prefetch_batch(c0, j0 + 2 * kF);             // the batch after next
#pragma unroll
                for (int u = 0; u < kF; ++u) {
                    file(xa[u], j0 + u);
                    const int jn = j0 + kF + u;
                    if (jn < nmine) load_file(xa[u], file_at(lb, jn), kl, word_of(jn));
                }
            }
#pragma unroll
            for (int u = 0; u < kF; ++u) {
                if (j0 + u < nmine) file(xa[u], j0 + u);
                if constexpr (MODE == TWO_PASS) {
#pragma unroll
                    for (int s = 0; s < R; ++s) load_chosen(xa[u][s], u * R + s);
                } else {
                    if (u < nmine) load_file(xa[u], file_at(lbn, u), kln, word_of(u));
                }
            }
        };

        if constexpr (MODE == MEAN) {
            // ---- mean: compensated per-thread sums, combined in warp order
            float sm[4], se[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) sm[k] = se[k] = 0.f;
            sweep([&](const uint4 &v, int) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float ns, ne;
                    two_sum(sm[k], __uint_as_float(el(v, k)), ns, ne);
                    sm[k] = ns;
                    se[k] += ne;
                }
            }, [](int) {});
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                list[(2 * w) * TC + lane * 4 + k] = __float_as_uint(sm[k]);
                list[(2 * w + 1) * TC + lane * 4 + k] = __float_as_uint(se[k]);
            }
            __syncthreads();
            if (tid < TC && c0 + seg_at<W>(tid) < d && n > 0) {
                float a = 0.f, ae = 0.f;
                for (int u = 0; u < kWarps; ++u) {
                    float ns, ne;
                    two_sum(a, __uint_as_float(list[(2 * u) * TC + tid]), ns, ne);
                    a = ns;
                    ae += ne + __uint_as_float(list[(2 * u + 1) * TC + tid]);
                }
                A.out[c0 + seg_at<W>(tid)] = (float)(((double)a + (double)ae) / (double)n);
            }
            __syncthreads();
        } else {
            // ---- keys of a sample, the first two files of every warp, in
            // the warp's own tag rows; where a warp has fewer, the smallest
            // or the largest key (NaNs, which no range below keeps) in turn
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int slot = u < nmine ? slot_of(u) : kDropped;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    uint32_t q = el(xa[u][0], k);
#pragma unroll
                    for (int s = 1; s < R; ++s)
                        if (slot == s) q = el(xa[u][s], k);
                    keys[(w + (u * 4 + k) * kWarps) * 32 + lane] = slot == kDropped ? ((w ^ u) & 1 ? 0xffffffffu : 0u) : to_key(q);
                }
            }
            __syncthreads();                                        // (A)
            // ---- value bins: thread (k, lane) sorts its coordinate's sample.
            // Bins 1..253 span the sample's range, cut to kReach inner ranges
            // (the four middle values) to either side of its median; values
            // outside go to bins 0 and 254.  A distorted copy in the sample
            // would otherwise stretch the range and crowd every other value
            // into a few bins; the middle holds while at most 10 of the 24
            // lie on one side of the honest values.  The widest inner range
            // of four lanes counts, as one alone can be tiny by chance.
            if (tid < TC) {
                const int k = w, c = lane * 4 + k;
                uint32_t y[kSample];
#pragma unroll
                for (int q = 0; q < kSample; ++q)
                    y[q] = keys[(q % kWarps + (q / kWarps * 4 + k) * kWarps) * 32 + lane];
                merge_sort<kSample>(y);
                float xlo = __uint_as_float(from_key(y[0])), xhi = __uint_as_float(from_key(y[kSample - 1]));
                const float i0 = __uint_as_float(from_key(y[kSample / 2 - 2]));
                const float i1 = __uint_as_float(from_key(y[kSample / 2 + 1]));
                float reach = kReach * (i1 - i0);
                reach = fmaxf(reach, __shfl_xor_sync(full, reach, 1));
                reach = fmaxf(reach, __shfl_xor_sync(full, reach, 2));
                if (reach > 0.f && reach < 1e38f) {
                    const float mid = 0.5f * i0 + 0.5f * i1;
                    xlo = fmaxf(xlo, mid - reach);
                    xhi = fminf(xhi, mid + reach);
                }
                const float more = widen * (xhi - xlo);
                xlo -= more;
                xhi += more;
                const float sc = (252.0f / 254.0f) / (xhi - xlo);
                const float cc = fmaf(-xlo, sc, 1.0f / 254.0f);
                const bool ok = isfinite(xlo) && isfinite(xhi) && xhi > xlo && isfinite(sc) && sc > 0.f &&
                                isfinite(cc);
                S(S_VS, c) = __float_as_uint(ok ? sc : 0.f);
                S(S_VC, c) = __float_as_uint(ok ? cc : 0.f);
                S(S_BIN, c) = c0 + seg_at<W>(c) < d && n > 0 ? kLive | (ok ? 0u : 0xFFu) : 0u;
            }
            __syncthreads();                                        // (B)
            const float4 vs = *reinterpret_cast<const float4 *>(&S(S_VS, lane * 4));
            const float4 vc = *reinterpret_cast<const float4 *>(&S(S_VC, lane * 4));
            const uint32_t hb = hist_s + (uint32_t)lane * 4u - (0x4B000000u << 7);

            // ---- sweep: compare, histogram and tag words of the guessed copies
            uint32_t nanf = 0u;
            sweep([&](const uint4 &v, int j) {
                const uint32_t b0 = vbin_bits(__uint_as_float(v.x), vs.x, vc.x);
                const uint32_t b1 = vbin_bits(__uint_as_float(v.y), vs.y, vc.y);
                const uint32_t b2 = vbin_bits(__uint_as_float(v.z), vs.z, vc.z);
                const uint32_t b3 = vbin_bits(__uint_as_float(v.w), vs.w, vc.w);
                red_shared<1u>((b0 << 7) + hb);
                red_shared<0x100u>((b1 << 7) + hb);
                red_shared<0x10000u>((b2 << 7) + hb);
                red_shared<0x1000000u>((b3 << 7) + hb);
                nan_check(nanf, __uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z),
                          __uint_as_float(v.w));
                if constexpr (MODE == TAGGED) tags[(w + j * kWarps) * 32 + lane] = pack4(b0, b1, b2, b3);
            }, [&](int j) {
                if constexpr (MODE == TAGGED) tags[(w + j * kWarps) * 32 + lane] = kPadTag * 0x01010101u;
            });
            // a NaN adds one to the lane's lowest bins, so that their totals
            // are not n
            if (nanf) red_shared<0x01010101u>(hist_s + (uint32_t)lane * 4u);
            cp_async_wait_all();
            __syncthreads();                                        // (C)
            {
                // per-warp partial sums over bins [kBPW*w, kBPW*w + kBPW): the
                // 8-bit counters as two pairs of 16-bit fields
                uint32_t ps0 = 0u, ps1 = 0u;
#pragma unroll
                for (int b = 0; b < kBPW; ++b)
                    if (w * kBPW + b < kVB) {
                        const uint32_t x = hist[(w * kBPW + b) * 32 + lane];
                        ps0 += x & 0x00FF00FFu;
                        ps1 += (x >> 8) & 0x00FF00FFu;
                    }
                part[w * 32 + lane] = make_uint2(ps0, ps1);
            }
            if (MODE == TAGGED && have_p) rank_pending(par ^ 1);
            if (tid == 0) n_long[par] = 0;
            __syncthreads();                                        // (D)
            // ---- bin search, one thread per coordinate
            if (tid < TC) {
                const int c = tid, lc = c >> 2, k = c & 3;
                uint32_t pend = 0u, word = 0u;
                const uint32_t state = S(S_BIN, c);
                if (state == kLive) {
                    const uint16_t *p16 = reinterpret_cast<const uint16_t *>(part) + lc * 4 + (k & 1) * 2 + (k >> 1);
                    uint32_t pu[kWarps], tot = 0u, rem = krank;
#pragma unroll
                    for (int u = 0; u < kWarps; ++u) {
                        pu[u] = p16[u * 128];
                        tot += pu[u];
                    }
                    int owner = kWarps - 1;
                    bool fd = false;
#pragma unroll
                    for (int u = 0; u < kWarps; ++u) {
                        const bool hit = !fd && rem < pu[u];
                        if (hit) owner = u;
                        if (!fd && !hit) rem -= pu[u];
                        fd |= hit;
                    }
                    const uint32_t *h = hist + lc;
                    uint32_t bin = min(owner * kBPW + kBPW, kVB) - 1, cnt = 0u, cbs[kBPW];
                    bool f2 = false;
#pragma unroll
                    for (int i = 0; i < kBPW; ++i) {
                        const int b = owner * kBPW + i;
                        cbs[i] = b < kVB ? (h[b * 32] >> (8 * k)) & 0xFFu : 0u;
                    }
#pragma unroll
                    for (int i = 0; i < kBPW; ++i) {
                        const bool hit = !f2 && rem < cbs[i];
                        if (hit) {
                            bin = owner * kBPW + i;
                            cnt = cbs[i];
                        }
                        if (!f2 && !hit) rem -= cbs[i];
                        f2 |= hit;
                    }
                    // an overflowed counter or a NaN changes the coordinate's total
                    if (tot == (uint32_t)n && cnt <= cap) {
                        word = bin | kListed;
                        pend = cnt | (rem << 8);
                        if (cnt > (uint32_t)kShort) long_c[atomicAdd(&n_long[par], 1)] = (uint8_t)c;
                    }
                }
                if (state != 0u && word == 0u) {                    // left to fixup_kernel
                    A.out[c0 + seg_at<W>(c)] = __uint_as_float(kOpen);
                    ++open_cnt;
                }
                S(S_BIN, c) = word;
                S(S_PEND, c) = pend;
                S(S_LCNT, c) = 0u;
            }
            __syncthreads();                                        // (E)
            for (int i = tid * 4; i < kHistWords; i += kNT * 4)
                *reinterpret_cast<uint4 *>(hist + i) = make_uint4(0u, 0u, 0u, 0u);

            // ---- the listed bins' members into the coordinates' lists: the
            // tag words (eight at a time) against the target bins, each
            // member's value by a 4-byte cp.async while it is still in L2;
            // the copies land during the next sweep
            if constexpr (MODE == TWO_PASS) {
                // ---- second pass over the chosen rows (the registers hold
                // the first kRows of them): the values in their coordinate's
                // target bin go straight into its list
                const uint4 tg = *reinterpret_cast<const uint4 *>(&S(S_BIN, lane * 4));
                const uint32_t t0 = (tg.x & kListed) ? 0x4B000000u | (tg.x & 0xFFu) : 0xFFFFFFFFu;
                const uint32_t t1 = (tg.y & kListed) ? 0x4B000000u | (tg.y & 0xFFu) : 0xFFFFFFFFu;
                const uint32_t t2 = (tg.z & kListed) ? 0x4B000000u | (tg.z & 0xFFu) : 0xFFFFFFFFu;
                const uint32_t t3 = (tg.w & kListed) ? 0x4B000000u | (tg.w & 0xFFu) : 0xFFFFFFFFu;
                auto take = [&](const uint4 &v, int j) {
                    if (j >= nmine || slot_of(j) == kDropped) return;
                    const bool m0 = vbin_bits(__uint_as_float(v.x), vs.x, vc.x) == t0;
                    const bool m1 = vbin_bits(__uint_as_float(v.y), vs.y, vc.y) == t1;
                    const bool m2 = vbin_bits(__uint_as_float(v.z), vs.z, vc.z) == t2;
                    const bool m3 = vbin_bits(__uint_as_float(v.w), vs.w, vc.w) == t3;
                    if (m0 | m1 | m2 | m3) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (!(k == 0 ? m0 : k == 1 ? m1 : k == 2 ? m2 : m3)) continue;
                            const int c = lane * 4 + k;
                            const uint32_t at = atomicAdd(&S(S_LCNT, c), 1u);
                            if (at < cap) list[at * TC + c] = el(v, k);
                        }
                    }
                };
                int j0 = 0;
                for (; j0 + kRows < nmine; j0 += kRows) {
                    // the batch after next into L2
#pragma unroll
                    for (int q0 = 0; q0 < kRows * 4; q0 += 32) {
                        const int q = q0 + lane, jp = j0 + 2 * kRows + q / 4;
                        if (q < kRows * 4 && jp < nmine && c0 + (q & 3) * 32 < d && slot_of(jp) != kDropped)
                            prefetch_l2(file_at(reinterpret_cast<const char *>(A.copies + c0 + (q & 3) * 32), jp) +
                                        (uint64_t)slot_of(jp) * ldb);
                    }
#pragma unroll
                    for (int i = 0; i < kRows; ++i) {
                        take(xa[i / R][i % R], j0 + i);
                        load_chosen(xa[i / R][i % R], j0 + kRows + i);
                    }
                }
#pragma unroll
                for (int u = 0; u < kF; ++u) {
#pragma unroll
                    for (int s = 0; s < R; ++s) take(xa[u][s], j0 + u * R + s);
                    if (u < nmine) load_file(xa[u], file_at(lbn, u), kln, word_of(u));
                }
                if (tn < ntiles) prefetch_batch(tn * TC, kF);
                __syncthreads();
                c0_p = c0;
                rank_pending(par);
                __syncthreads();
                continue;
            }
            const uint4 tg = *reinterpret_cast<const uint4 *>(&S(S_BIN, lane * 4));
            const uint32_t vbx = pack4(tg.x, tg.y, tg.z, tg.w);
            const uint32_t vmask = ((tg.x >> 8) & 1u) * 0xFFu | ((tg.y >> 8) & 1u) * 0xFF00u |
                                   ((tg.z >> 8) & 1u) * 0xFF0000u | ((tg.w >> 8) & 1u) * 0xFF000000u;
            if (vmask) {
                for (int g = 0; g < nmine; g += 8) {
                    uint32_t m = 0u;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (g + i < nmine) m |= tag_match(tags[(w + (g + i) * kWarps) * 32 + lane], vbx) >> (7 - i);
                    for (m &= vmask; m; m &= m - 1u) {
                        const int b = __ffs(m) - 1;
                        const int k = b >> 3, j = g + (b & 7), c = lane * 4 + k;
                        const uint32_t at = atomicAdd(&S(S_LCNT, c), 1u);
                        if (at < cap)
                            cp_async4(list_s + (at * TC + c) * 4u,
                                      AVG ? reinterpret_cast<const char *>(A.means + (int64_t)(word_of(j) >> 16) * A.ldm +
                                                                           c0 + c)
                                          : file_at(lb, j) + (uint64_t)slot_of(j) * ldb + off_of<W>(k) * 4);
                    }
                }
                cp_async_commit();
            }
            if (tn < ntiles) prefetch_batch(tn * TC, kF);   // the next tile's second batch
            have_p = true;
            c0_p = c0;
            par ^= 1;
        }
    }
    __syncthreads();
    if constexpr (MODE != MEAN) {
        // the last tile's listed members are ranked once their copies land
        if (MODE == TAGGED && have_p) {
            cp_async_wait_all();
            __syncthreads();
            rank_pending(par ^ 1);
        }
        if (tid < TC) {
            open_cnt = __reduce_add_sync(full, open_cnt);
            if (lane == 0 && open_cnt) atomicAdd(&A.det->median_exact, open_cnt);
        }
        if constexpr (SETTLE) {
            // (the tags and the counters after them are done with)
            static_assert(kHistWords >= 32 * 32, "the tags' f rows of 32 words are up to 32 rows short of the keys");
            if (__syncthreads_or(open_cnt != 0u)) settle_open(A, tags, meta, n, blockIdx.x, gridDim.x);
        }
    }
    if constexpr (R == 1) {
        if (tid == 0) gate_leave(A.gate);
    } else if constexpr (!AVG) {
        for (int i = tid; i < f; i += kNT) {
            const uint32_t neq = (meta[i] >> 4) & 0xFFFu;
            if (neq) atomicOr(&A.file_neq[meta[i] >> 16], neq);
        }
    }
}

template <int R, int W, int MODE, int MINB, bool AVG = false, int CAP = 32, bool SETTLE = false>
cudaError_t try_sweep(bool &ok, const SweepArgs &A, bool chained, cudaStream_t stream)
{
    ok = false;
    const SweepLayout L = sweep_layout<MODE, CAP>(A.f);
    if (L.total > smem_cap()) return cudaSuccess;
    auto kern = sweep_kernel<R, W, MODE, MINB, AVG, CAP, SETTLE>;
    static Residency resident;
    const int per_sm = resident.blocks(kern, kNT, L.total);
    if (per_sm < MINB) return cudaSuccess;                // the next configuration is tried
    const int64_t ntiles = (A.d + TC - 1) / TC;
    int64_t grid = (int64_t)sm_count() * per_sm;
    if (grid > ntiles) grid = ntiles;
    ok = true;
    if (chained) return launch_chained(kern, grid, kNT, L.total, stream, A);
    kern<<<(unsigned)grid, kNT, L.total, stream>>>(A);
    return cudaGetLastError();
}

template <int R, int W>
cudaError_t sweep_for(bool &ok, bool &open, const SweepArgs &A, int mode, bool chained, cudaStream_t stream)
{
    open = mode == 0;
    ok = false;
    if (mode == 1) return try_sweep<R, W, MEAN, 2>(ok, A, chained, stream);
    // One block alone on its SM has more rows in flight: taken where the tags
    // leave no room for a second one, and where there are no more tiles than
    // SMs anyway.
    const bool alone = (A.d + TC - 1) / TC <= sm_count();
    cudaError_t e = cudaSuccess;
    if constexpr (R == 1) {
        if (alone && A.f <= kSettleFiles) {
            e = try_sweep<R, W, TAGGED, 1, false, 32, true>(ok, A, chained, stream);
            if (ok) open = false;
            return e;
        }
    }
    if ((!alone || R == 2) && A.f <= kPairFiles) {
        e = try_sweep<R, W, TAGGED, 2>(ok, A, chained, stream);
        if (e == cudaSuccess && !ok) e = try_sweep<R, W, TAGGED, 2, false, 16>(ok, A, chained, stream);
    }
    if constexpr (R == 2) {
        return e;                     // two copies: at most 465 files
    } else {
        if (e != cudaSuccess || ok) return e;
        if (A.f <= kTagFiles) {
            e = A.f <= kLongFiles ? try_sweep<R, W, TAGGED, 1, false, 64>(ok, A, chained, stream)
                                  : try_sweep<R, W, TAGGED, 1>(ok, A, chained, stream);
            if (e != cudaSuccess || ok) return e;
        }
        return try_sweep<R, W, TWO_PASS, 2>(ok, A, chained, stream);
    }
}

}  // namespace

template <int R>
cudaError_t launch_sweep(bool &ok, bool &open, const SweepArgs &A, int mode, bool chained, cudaStream_t stream)
{
    switch (load_width(A.copies, A.ld)) {
    case 4: return sweep_for<R, 4>(ok, open, A, mode, chained, stream);
    case 2: return sweep_for<R, 2>(ok, open, A, mode, chained, stream);
    default: return sweep_for<R, 1>(ok, open, A, mode, chained, stream);
    }
}

template <int R>
cudaError_t launch_sweep_averages(bool &ok, const SweepArgs &A, cudaStream_t stream)
{
    ok = false;
    const bool chained = false;
    cudaError_t e = cudaSuccess;
    if ((A.d + TC - 1) / TC > sm_count()) e = try_sweep<R, 4, TAGGED, 2, true>(ok, A, chained, stream);
    if (e != cudaSuccess || ok) return e;
    if (R == 2 || A.f <= kLongFiles) return try_sweep<R, 4, TAGGED, 1, true, 64>(ok, A, chained, stream);
    if constexpr (R > 2) e = try_sweep<R, 4, TAGGED, 1, true>(ok, A, chained, stream);
    return e;
}

}  // namespace aspis
