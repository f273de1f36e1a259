// The round in one pass over the copies (steps 1-5).
//
// Run one after the other, the compare reads all f*r rows and the aggregation
// reads the f chosen rows again.  The aggregation needs the selection only to
// know which copy of a file to take, and that can be guessed: an adversary
// that distorts a copy distorts it nearly everywhere, so a few coordinates of
// every row already show which copies differ.
//   sample   pair words of every file from up to 128 coordinates;
//   decide   graph, maximum cliques and selection from those words: a guess;
//   sweep    one pass over all copies: every pair compared in full, and the
//            guessed copies' values, while they are in registers, aggregated
//            (lower median or mean);
//   decide   graph, cliques and selection again, from the full words.  Where
//            the selection equals the guess, the aggregate is the round's;
//   repair   otherwise (distortions outside the sample) the separate
//            aggregation runs over the chosen rows.  It is always launched
//            and returns at once when the guess held.
//   fixup    the few coordinates whose median the sweep left open.
// The outputs are those of the separate steps.  All state between the kernels
// is in the caller's buffers: the guess in sel, the request for a repair in
// det->success (bit 1), taken back by the repair's last block, open
// coordinates as a bit pattern in out.
//
// The sweep is bound by HBM (61.0 GB in 9.5 ms = 6.4 TB/s at 455 files of
// three copies and 11.2M coordinates; the separate passes took 8.7 + 4.9 ms).
// With one copy per file (R = 1) it is the separate aggregation: 0.43 ms at
// 455 files and 2^20 coordinates.
#include <utility>

#include "aspis_internal.cuh"
#include "detect_common.cuh"
#include "median_common.cuh"

namespace aspis {
namespace {

// ------------------------------------------------------------------ sample

constexpr int kSampleThreads = 128;
constexpr int kSegments = 4;                 // of 32 coordinates, spread over the row

// one warp per file: its pair word over the sampled coordinates
template <int R>
__global__ void __launch_bounds__(kSampleThreads)
sample_kernel(const uint32_t *__restrict__ copies, int64_t f, int64_t d, int64_t ld,
              uint32_t *__restrict__ file_neq)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * (kSampleThreads / 32) + (threadIdx.x >> 5);
    if (i >= f) return;
    const uint32_t *row = copies + i * R * ld;
    uint32_t x[kSegments][R];
#pragma unroll
    for (int g = 0; g < kSegments; ++g) {
        const int64_t c = ((d * (2 * g + 1) / (2 * kSegments)) & ~(int64_t)31) + lane;
#pragma unroll
        for (int s = 0; s < R; ++s) x[g][s] = c < d ? __ldg(row + s * ld + c) : 0u;
    }
    uint32_t neq = 0u;
#pragma unroll
    for (int g = 0; g < kSegments; ++g) {
        int p = 0;
#pragma unroll
        for (int s = 0; s < R; ++s)
#pragma unroll
            for (int t = s + 1; t < R; ++t, ++p) neq |= (x[g][s] != x[g][t] ? 1u : 0u) << p;
    }
    neq = __reduce_or_sync(0xffffffffu, neq);
    if (lane == 0) file_neq[i] = neq;
}

// ------------------------------------------------------------------ decide

constexpr int kDecideThreads = 1024;

// Steps 2-4 in one block (f <= ASPIS_MAX_AGG_FILES): three launches less than
// the separate kernels, which take 3 + 4..18 + 3 us one after the other.
//   GUESS    sel and det from the sampled words; file_neq is cleared for the
//            sweep, and kUnclean set in sel where copies of the file differ
//   VERIFY   the round's adj, det and sel; bit 1 of det->success is set where
//            sel held another guess
//   PLAIN    adj, det and sel
enum Decide { GUESS, VERIFY, PLAIN };
constexpr int kUnclean = 16;

template <int R, Decide WHAT>
__global__ void __launch_bounds__(kDecideThreads)
decide_kernel(uint32_t *__restrict__ file_neq, const uint8_t *__restrict__ fw, int f, int K,
              uint32_t *__restrict__ adj_out, aspis_detection *det, int8_t *__restrict__ sel)
{
    __shared__ uint32_t dis[32], adj[32];
    __shared__ Frame stack[32][32];
    __shared__ int best, kept, success_s;
    __shared__ uint32_t clique_s;
    const int tid = threadIdx.x;
    if (tid < 32) dis[tid] = 0u;
    if (tid == 0) {
        best = 0;
        kept = 0;
    }
    __syncthreads();
    for (int i = tid; i < f; i += kDecideThreads) {
        const uint32_t w = file_neq[i];
        if (w) add_disagreements(w, fw + i * R, R, dis);
    }
    __syncthreads();
    if (tid < 32) {
        const uint32_t all = (1u << K) - 1u;                 // K <= 31
        const uint32_t row = tid < K ? ~dis[tid] & all & ~(1u << tid) : 0u;
        adj[tid] = row;
        if (WHAT != GUESS && tid < K) adj_out[tid] = row;
        const uint32_t budget = det->node_budget ? det->node_budget : kDefaultNodeBudget;
        __syncwarp();
        const CliqueResult c = max_cliques_warp<true>(adj, K, budget, stack, &best);
        if (tid == 0) {
            clique_s = c.first;
            success_s = (c.n_max == 1u && !c.over) ? 1 : 0;
            det->clique_mask = c.first;
            det->omega = c.omega;
            det->n_max_cliques = c.n_max;
            det->status = c.over ? ASPIS_E_LIMIT : ASPIS_OK;
            det->search_nodes = c.nodes;
            if (WHAT != VERIFY) det->median_exact = 0u;
        }
    }
    __syncthreads();
    const bool success = success_s != 0;
    int mine = 0, differs = 0;
    for (int i = tid; i < f; i += kDecideThreads) {
        const uint32_t w = success && WHAT != GUESS ? 0u : file_neq[i];
        const int pick = chosen_slot<R>(success, clique_s, fw + i * R, w);
        if (WHAT == VERIFY) {
            const int was = sel[i];
            if ((was < 0 ? was : was & (kUnclean - 1)) != pick) differs = 1;
        }
        sel[i] = (int8_t)(WHAT == GUESS && w && pick >= 0 ? pick | kUnclean : pick);
        if (WHAT == GUESS) file_neq[i] = 0u;
        mine += pick >= 0;
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if ((tid & 31) == 0 && mine) atomicAdd(&kept, mine);
    differs = __syncthreads_or(differs);     // (always 0 but for VERIFY)
    if (tid == 0) {
        det->n_sel = kept;
        det->success = success_s | (differs ? 2 : 0);
        if (differs) det->median_exact = 0u;
    }
}

// ------------------------------------------------------------------- sweep

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
constexpr int kCap = 32;                    // list entries per coordinate
constexpr int kHistWords = kVB * 32;        // four 8-bit counters per (bin, lane)
constexpr int kBPW = (kVB + kWarps - 1) / kWarps;
constexpr int kShort = 8;                   // longest list one thread sorts
constexpr int kSample = 2 * kWarps;         // sampled values per coordinate
constexpr float kReach = 14.0f;             // farthest bin from the centre, in inner ranges of the sample
constexpr int kDropped = 15;                // slot of a file that is not aggregated
// Bits of a coordinate that the sweep leaves to fixup_kernel.  They may also
// be a median's own bits (a NaN payload): computing that one again gives it.
constexpr uint32_t kOpen = 0x7FA5C3E1u;

// per-coordinate state, arrays of TC words
//   S_VS, S_VC  scale and offset of the value bins
//   S_PEND      the pending tile's listed bin: count | rank in it << 8
//   S_BIN       target bin, kListed where its members are listed
//   S_PART      the bin search's partial sums (six arrays' room)
enum { S_VS, S_VC, S_LCNT, S_PEND, S_BIN, S_PART, kStateWords = S_PART + 6 };
static_assert(6 * TC * 4 >= kWarps * 32 * 8, "room for the partial sums");
constexpr uint32_t kListed = 0x100u, kLive = 0x200u;

// Tag bytes bound the files of a median tile: two blocks share an SM up to
// about 460 files, one block has it up to kTileFiles, where the 8-bit counters
// of bins over the sample's range still hold.
constexpr int64_t kTileFiles = 640;
static_assert(kTileFiles <= kCap * TC, "the kept rows fit the list while they are put in order");
constexpr int64_t kMinValues = 100'000'000;  // fp32 values of the smallest round taken in one pass

struct SweepArgs {
    const float *copies;
    int64_t d, ld;
    int f;
    const int8_t *sel;
    aspis_detection *det;
    float *out;
    uint32_t *file_neq;              // R > 1: pair words, ORed
    int r;                           // R = 1: row i * r + sel[i] is file i's
    aspis_detection *gate;           // R = 1: run only where a repair was asked for, or NULL
};

struct SweepLayout {
    size_t tags, hist, list, state, meta, total;
};

template <int MODE>
__host__ __device__ inline SweepLayout sweep_layout(int64_t f)
{
    SweepLayout L{};
    int64_t per_warp = (f + kWarps - 1) / kWarps;
    if (per_warp < 8) per_warp = 8;          // the sampled keys use a warp's first eight tag rows
    size_t o = 0;
    L.tags = o; o += MODE == 0 ? (size_t)per_warp * kWarps * 128 : 0;
    L.hist = o; o += MODE == 0 ? (size_t)kHistWords * 4 : 0;
    L.list = o; o += (size_t)kCap * TC * 4;
    L.state = o; o += MODE == 0 ? (size_t)kStateWords * TC * 4 : 0;
    L.meta = o; o += ((size_t)f * 4 + 15) / 16 * 16;
    L.total = o;
    return L;
}

// coordinate c of a tile (lane c / 4, element c % 4) in the tile's row segment
template <bool VEC>
__device__ __forceinline__ int seg_at(int c)
{
    return VEC ? c : (c >> 2) + 32 * (c & 3);
}

__device__ __forceinline__ uint32_t el(const uint4 &x, int k)
{
    return k == 0 ? x.x : k == 1 ? x.y : k == 2 ? x.z : x.w;
}

__device__ __forceinline__ uint32_t vdiff(const uint4 &a, const uint4 &b)
{
    return (a.x ^ b.x) | (a.y ^ b.y) | (a.z ^ b.z) | (a.w ^ b.w);
}

// Ascending odd-even merge sort of N <= 32 keys in registers (Batcher 1968):
// the comparators of the 32-key network, those that touch a key beyond N
// dropped (they would meet the largest key).
struct Network {
    int n = 0;
    unsigned char a[192] = {}, b[192] = {};
};

template <int N>
__host__ __device__ constexpr Network merge_network()
{
    Network net{};
    for (int p = 1; p < 32; p *= 2)
        for (int k = p; k >= 1; k /= 2)
            for (int j = k % p; j + k < 32; j += 2 * k)
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

// The file (a multiple of 8) that a tile's order starts from: its first kSample
// files are the sample, so as few of them as possible shall be marked (bit 31:
// their copies differ).  Neighbours in file order share workers, and with them
// distortions, so some window has few even where a quarter of all files is
// distorted.  (A sample spread over the file order is as good, but rows taken
// from all over the copies at a tile's start cost 7 to 10% of the pass at 61
// GB, read once or twice, prefetched or not.)  Called by the whole block; n <=
// kTileFiles.
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

template <int R, bool VEC, int MODE, int MINB>
__global__ void __launch_bounds__(kNT, MINB)
sweep_kernel(const SweepArgs A)
{
    if (R == 1 && !gate_open(A.gate)) return;
    constexpr int kF = batch_files(R, MINB);
    constexpr int kRows = kF * R;
    static_assert(kF >= 2, "the sample is the first two files of every warp");
    extern __shared__ __align__(16) unsigned char smem[];
    const SweepLayout L = sweep_layout<MODE>(A.f);
    uint32_t *tags = reinterpret_cast<uint32_t *>(smem + L.tags);     // [warp's file][kWarps][32]
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem + L.hist);     // [kVB][32]
    uint32_t *list = reinterpret_cast<uint32_t *>(smem + L.list);     // [kCap][TC]
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
    if constexpr (MODE == 0) {
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
            uint32_t *to = MODE == 0 ? list : meta;
            if (s >= 0)
                to[off + __popc(m & ((1u << lane) - 1u))] = (uint32_t)(i * A.r + s) | (s > 0 ? 0x80000000u : 0u);
            __syncthreads();
        }
        if constexpr (MODE == 0) {
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
        if constexpr (MODE == 0) {
            for (int i = tid; i < f; i += kNT) list[i] = A.sel[i] < 0 || A.sel[i] >= kUnclean ? 0x80000000u : 0u;
            __syncthreads();
            start = cleanest_start(list, f, &start_s);
        }
        int mine = 0;
        for (int i = tid; i < f; i += kNT) {
            const int s = A.sel[i];
            meta[(i < start ? f : 0) + i - start] =
                (uint32_t)(s < 0 ? kDropped : s & (kUnclean - 1)) | ((uint32_t)i << 16);
            mine += s >= 0;
        }
        mine = __reduce_add_sync(full, mine);
        if (lane == 0 && mine) atomicAdd(&n_s, mine);
        __syncthreads();
        n = n_s;
    }
    const uint32_t krank = (uint32_t)((n - 1) / 2);
    const int64_t ntiles = (d + TC - 1) / TC;

    const int nf = R == 1 ? n : f;                                    // files of a tile
    const int nmine = nf > w ? (nf - w + kWarps - 1) / kWarps : 0;    // of this warp
    auto word_of = [&](int j) -> uint32_t { return meta[w + j * kWarps]; };
    auto slot_of = [&](int j) -> int { return R == 1 ? 0 : (int)(word_of(j) & 15u); };
    // a file's copies start here, from the lane's base in row 0
    auto file_at = [&](const char *base, int j) -> const char * {
        return base + (uint64_t)(R == 1 ? word_of(j) : (word_of(j) >> 16) * R) * ldb;
    };
    // the lane's part of tile t: address in row 0, and how many of its four
    // coordinates exist
    auto lane_base = [&](int64_t t) -> const char * {
        return reinterpret_cast<const char *>(A.copies + t * TC + (VEC ? lane * 4 : lane));
    };
    auto live_of = [&](int64_t t) -> int {
        if (t >= ntiles) return 0;
        const int64_t left = d - t * TC;
        if (left >= TC) return 4;
        const int64_t q = VEC ? left - lane * 4 : (left - lane + 31) / 32;
        return q < 0 ? 0 : q > 4 ? 4 : (int)q;
    };
    auto load_file = [&](uint4 (&x)[R], const char *p, int kl) {
#pragma unroll
        for (int s = 0; s < R; ++s) {
            const char *q = p + (uint64_t)s * ldb;
            if constexpr (VEC) {
                // the copies of slot 0 are the usual choice: they stay in L2
                // for the member lists, the others are first to go
                const uint4 *e = reinterpret_cast<const uint4 *>(q);
                if (kl > 0) x[s] = s == 0 ? __ldcg(e) : __ldcs(e);
            } else {
                const unsigned int *e = reinterpret_cast<const unsigned int *>(q);
                if (kl > 0) x[s].x = __ldcg(e);
                if (kl > 1) x[s].y = __ldcg(e + 32);
                if (kl > 2) x[s].z = __ldcg(e + 64);
                if (kl > 3) x[s].w = __ldcg(e + 96);
            }
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
            if (u < nmine) load_file(xa[u], file_at(p, u), kl);
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
                A.out[c0_p + seg_at<VEC>(c)] = __uint_as_float(from_key(res));
            }
        }
        const int nl = n_long[parity];
        for (int q = (w - TC / 32 + kWarps) % kWarps; q < nl; q += kWarps) {
            const int c = long_c[q];
            const uint32_t cnt = S(S_PEND, c) & 0xFFu, rk = S(S_PEND, c) >> 8;
            const uint32_t x = warp_sort32((uint32_t)lane < cnt ? to_key(list[lane * TC + c]) : 0xffffffffu, lane);
            const uint32_t res = __shfl_sync(full, x, (int)rk);
            if (lane == 0) A.out[c0_p + seg_at<VEC>(c)] = __uint_as_float(from_key(res));
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
        // files j.. of a batch into L2, one 128-byte line per lane
        auto prefetch_batch = [&](int64_t cb, int j) {
#pragma unroll
            for (int q0 = 0; q0 < kRows * 4; q0 += 32) {
                const int q = q0 + lane, row = q / 4, jp = j + row / R;
                if (q < kRows * 4 && jp < nmine && cb + (q & 3) * 32 < d)
                    prefetch_l2(file_at(reinterpret_cast<const char *>(A.copies + cb + (q & 3) * 32), jp) +
                                (uint64_t)(row % R) * ldb);
            }
        };
        // One pass over this warp's files, kF at a time; a file's registers
        // are refilled as soon as it is compared, the last ones with the next
        // tile's first files.  fn(v, j): the guessed copy of the warp's j-th
        // file; skip(j): a file without one.
        auto sweep = [&](auto fn, auto skip) {
            auto file = [&](uint4 (&x)[R], int j) {
                if constexpr (R == 1) {
                    fn(x[0], j);
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
                    if (jn < nmine) load_file(xa[u], file_at(lb, jn), kl);
                }
            }
#pragma unroll
            for (int u = 0; u < kF; ++u) {
                if (j0 + u < nmine) file(xa[u], j0 + u);
                if (u < nmine) load_file(xa[u], file_at(lbn, u), kln);
            }
        };

        if constexpr (MODE == 1) {
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
            if (tid < TC && c0 + seg_at<VEC>(tid) < d && n > 0) {
                float a = 0.f, ae = 0.f;
                for (int u = 0; u < kWarps; ++u) {
                    float ns, ne;
                    two_sum(a, __uint_as_float(list[(2 * u) * TC + tid]), ns, ne);
                    a = ns;
                    ae += ne + __uint_as_float(list[(2 * u + 1) * TC + tid]);
                }
                A.out[c0 + seg_at<VEC>(tid)] = (float)(((double)a + (double)ae) / (double)n);
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
                    tags[(w + (u * 4 + k) * kWarps) * 32 + lane] = slot == kDropped ? ((w ^ u) & 1 ? 0xffffffffu : 0u) : to_key(q);
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
                    y[q] = tags[(q % kWarps + (q / kWarps * 4 + k) * kWarps) * 32 + lane];
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
                const float sc = (252.0f / 254.0f) / (xhi - xlo);
                const float cc = fmaf(-xlo, sc, 1.0f / 254.0f);
                const bool ok = isfinite(xlo) && isfinite(xhi) && xhi > xlo && isfinite(sc) && sc > 0.f &&
                                isfinite(cc);
                S(S_VS, c) = __float_as_uint(ok ? sc : 0.f);
                S(S_VC, c) = __float_as_uint(ok ? cc : 0.f);
                S(S_BIN, c) = c0 + seg_at<VEC>(c) < d && n > 0 ? kLive | (ok ? 0u : 0xFFu) : 0u;
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
                tags[(w + j * kWarps) * 32 + lane] = pack4(b0, b1, b2, b3);
            }, [&](int j) { tags[(w + j * kWarps) * 32 + lane] = kPadTag * 0x01010101u; });
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
            if (have_p) rank_pending(par ^ 1);
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
                    if (tot == (uint32_t)n && cnt <= (uint32_t)kCap) {
                        word = bin | kListed;
                        pend = cnt | (rem << 8);
                        if (cnt > (uint32_t)kShort) long_c[atomicAdd(&n_long[par], 1)] = (uint8_t)c;
                    }
                }
                if (state != 0u && word == 0u) {                    // left to fixup_kernel
                    A.out[c0 + seg_at<VEC>(c)] = __uint_as_float(kOpen);
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
                        if (at < (uint32_t)kCap)
                            cp_async4(list_s + (at * TC + c) * 4u,
                                      file_at(lb, j) + (uint64_t)slot_of(j) * ldb + (VEC ? k : 32 * k) * 4);
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
    if constexpr (MODE == 0) {
        // the last tile's listed members are ranked once their copies land
        if (have_p) {
            cp_async_wait_all();
            __syncthreads();
            rank_pending(par ^ 1);
        }
        if (tid < TC) {
            open_cnt = __reduce_add_sync(full, open_cnt);
            if (lane == 0 && open_cnt) atomicAdd(&A.det->median_exact, open_cnt);
        }
    }
    if constexpr (R == 1) {
        if (tid == 0) gate_leave(A.gate);
    } else {
        for (int i = tid; i < f; i += kNT) {
            const uint32_t neq = (meta[i] >> 4) & 0xFFFu;
            if (neq) atomicOr(&A.file_neq[meta[i] >> 16], neq);
        }
    }
}

// ------------------------------------------------------------------- fixup

// The coordinates that the sweep left open (kOpen in out): a NaN among the
// values, a value bin with more members than a list holds, an overflowed
// counter, no spread in the sample.  Returns at once when det says that there
// are none.  A block takes 32 coordinates at a time.
//   Few of them open: one after the other, the values spread over the block's
//   threads and their keys selected bit by bit (a load latency and 32 counting
//   barriers).
//   Else an 8-bit radix select of all 32 at once: four passes over the rows'
//   128-byte segments, which stay in L2.
constexpr int kFixThreads = 512, kFixWarps = kFixThreads / 32;
constexpr int kFixPer = ASPIS_MAX_AGG_FILES / kFixThreads;
constexpr int kFixFew = 6;
static_assert(kFixPer * kFixThreads == ASPIS_MAX_AGG_FILES, "every kept value has a thread");

__global__ void __launch_bounds__(kFixThreads)
fixup_kernel(const SweepArgs A)
{
    if (*(volatile const uint32_t *)&A.det->median_exact == 0u) return;
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem);              // [256][32]
    uint16_t *rows = reinterpret_cast<uint16_t *>(hist + 256 * 32);   // kept rows
    __shared__ int warp_tot[kFixWarps];
    __shared__ uint32_t pre[32], rnk[32], open_s;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, f = A.f;
    const unsigned full = 0xffffffffu;
    const uint32_t *copies = reinterpret_cast<const uint32_t *>(A.copies);
    const int64_t ntiles = (A.d + 31) / 32;
    int n = -1;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t c0 = t * 32;
        if (w == 0) {
            const uint32_t x = c0 + lane < A.d ? __float_as_uint(A.out[c0 + lane]) : 0u;
            const uint32_t m = __ballot_sync(full, x == kOpen);
            if (lane == 0) open_s = m;
        }
        __syncthreads();
        uint32_t open = open_s;
        __syncthreads();
        if (!open) continue;
        if (n < 0) {                       // the kept rows, once a block has work
            n = 0;
            for (int b0 = 0; b0 < f; b0 += kFixThreads) {
                const int i = b0 + tid, s = i < f ? (int)A.sel[i] : -1;
                const unsigned m = __ballot_sync(full, s >= 0);
                if (lane == 0) warp_tot[w] = __popc(m);
                __syncthreads();
                int off = n;
                for (int q = 0; q < kFixWarps; ++q) {
                    off += q < w ? warp_tot[q] : 0;
                    n += warp_tot[q];
                }
                if (s >= 0) rows[off + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(i * A.r + s);
                __syncthreads();
            }
        }
        const uint32_t krank = (uint32_t)((n - 1) / 2);
        if (__popc(open) <= kFixFew) {
            for (; open; open &= open - 1u) {
                const int64_t c = c0 + __ffs(open) - 1;
                uint32_t key[kFixPer];
#pragma unroll
                for (int u = 0; u < kFixPer; ++u) {
                    const int i = tid + u * kFixThreads;
                    key[u] = i < n ? to_key(__ldcg(copies + (int64_t)rows[i] * A.ld + c)) : 0u;
                }
                uint32_t prefix = 0u, rk = krank;
                for (int b = 31; b >= 0; --b) {
                    // keys that match the prefix above bit b and have bit b clear
                    uint32_t below = 0u;
#pragma unroll
                    for (int u = 0; u < kFixPer; ++u)
                        if (u * kFixThreads < n)
                            below += (uint32_t)__syncthreads_count(tid + u * kFixThreads < n &&
                                                                   (key[u] >> b) == (prefix >> b));
                    if (rk >= below) {
                        rk -= below;
                        prefix |= 1u << b;
                    }
                }
                if (tid == 0) A.out[c] = __uint_as_float(from_key(prefix));
            }
            __syncthreads();
            continue;
        }
        const bool live = c0 + lane < A.d;
        if (tid < 32) {
            pre[tid] = 0u;
            rnk[tid] = krank;
        }
        for (int p = 0; p < 4; ++p) {
            const int sh = 24 - 8 * p;
            const uint32_t pmask = p == 0 ? 0u : 0xFFFFFFFFu << (32 - 8 * p);
            for (int i = tid; i < 256 * 32; i += kFixThreads) hist[i] = 0u;
            __syncthreads();
            const uint32_t want = pre[lane];
            for (int j0 = w; j0 < n; j0 += kFixWarps * 8) {
                uint32_t v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int j = j0 + u * kFixWarps;
                    v[u] = live && j < n ? __ldcg(copies + (int64_t)rows[j] * A.ld + c0 + lane) : 0u;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int j = j0 + u * kFixWarps;
                    const uint32_t key = to_key(v[u]);
                    if (live && j < n && (key & pmask) == want) atomicAdd(&hist[((key >> sh) & 0xFFu) * 32 + lane], 1u);
                }
            }
            __syncthreads();
            // a warp settles two coordinates: a warp scan over the 256 digits
            for (int cc = w; cc < 32; cc += kFixWarps) {
                uint32_t cb[8], sum = 0u;
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                    cb[b] = hist[(lane * 8 + b) * 32 + cc];
                    sum += cb[b];
                }
                uint32_t inc = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(full, inc, o);
                    if (lane >= o) inc += y;
                }
                const uint32_t rk = rnk[cc], exc = inc - sum;
                const bool mine = exc <= rk && rk < inc;
                uint32_t dig = 0u, r2 = rk - exc;
                if (mine) {
                    bool hit = false;
#pragma unroll
                    for (int b = 0; b < 8; ++b) {
                        if (!hit && r2 < cb[b]) {
                            dig = (uint32_t)(lane * 8 + b);
                            hit = true;
                        }
                        if (!hit) r2 -= cb[b];
                    }
                }
                const unsigned bal = __ballot_sync(full, mine);
                const int src = bal ? __ffs(bal) - 1 : 0;
                dig = __shfl_sync(full, dig, src);
                r2 = __shfl_sync(full, r2, src);
                if (lane == 0 && bal) {
                    pre[cc] |= dig << sh;
                    rnk[cc] = r2;
                }
            }
            __syncthreads();
        }
        if (w == 0 && ((open >> lane) & 1u)) A.out[c0 + lane] = __uint_as_float(from_key(pre[lane]));
        __syncthreads();
    }
}

cudaError_t launch_fixup(const SweepArgs &A, cudaStream_t stream)
{
    const size_t smem = 256 * 32 * 4 + ((size_t)A.f * 2 + 15) / 16 * 16;
    const int64_t ntiles = (A.d + 31) / 32;
    int64_t grid = (int64_t)sm_count() * 4;
    if (grid > ntiles) grid = ntiles;
    fixup_kernel<<<(unsigned)grid, kFixThreads, smem, stream>>>(A);
    return cudaGetLastError();
}

template <int R, bool VEC, int MODE, int MINB>
cudaError_t try_sweep(bool &launched, const SweepArgs &A, cudaStream_t stream)
{
    launched = false;
    const SweepLayout L = sweep_layout<MODE>(A.f);
    auto kern = sweep_kernel<R, VEC, MODE, MINB>;
    if (L.total > smem_cap()) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.total);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kNT, L.total);
    if (e != cudaSuccess) return e;
    if (per_sm < MINB) return cudaSuccess;
    const int64_t ntiles = (A.d + TC - 1) / TC;
    int64_t grid = (int64_t)sm_count() * per_sm;
    if (grid > ntiles) grid = ntiles;
    kern<<<(unsigned)grid, kNT, L.total, stream>>>(A);
    launched = true;
    return cudaGetLastError();
}

template <int R>
cudaError_t fused(bool &done, const SweepArgs &A, const uint8_t *fw, int K, uint32_t *adj, int8_t *sel,
                  int mode, bool vec, cudaStream_t stream)
{
    sample_kernel<R><<<(unsigned)((A.f + 3) / 4), kSampleThreads, 0, stream>>>(
        reinterpret_cast<const uint32_t *>(A.copies), A.f, A.d, A.ld, A.file_neq);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    decide_kernel<R, GUESS><<<1, kDecideThreads, 0, stream>>>(A.file_neq, fw, A.f, K, adj, A.det, sel);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    bool ok = false;
    if (mode == 1) {
        e = vec ? try_sweep<R, true, 1, 2>(ok, A, stream) : try_sweep<R, false, 1, 2>(ok, A, stream);
    } else {
        e = vec ? try_sweep<R, true, 0, 2>(ok, A, stream) : try_sweep<R, false, 0, 2>(ok, A, stream);
        if (e == cudaSuccess && !ok)
            e = vec ? try_sweep<R, true, 0, 1>(ok, A, stream) : try_sweep<R, false, 0, 1>(ok, A, stream);
    }
    if (e != cudaSuccess) return e;
    if (!ok) return cudaErrorInvalidValue;
    decide_kernel<R, VERIFY><<<1, kDecideThreads, 0, stream>>>(A.file_neq, fw, A.f, K, adj, A.det, sel);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return launch_aggregate_tiles(done, A.copies, A.f, R, A.d, A.ld, sel, A.det, mode, A.out, stream, A.det);
}

template <int R>
cudaError_t decide(uint32_t *file_neq, const uint8_t *fw, int f, int K, uint32_t *adj, aspis_detection *det,
                   int8_t *sel, cudaStream_t stream)
{
    decide_kernel<R, PLAIN><<<1, kDecideThreads, 0, stream>>>(file_neq, fw, f, K, adj, det, sel);
    return cudaGetLastError();
}

// the separate aggregation of the chosen rows
template <bool VEC>
cudaError_t aggregate_rows(bool &ok, const SweepArgs &A, int mode, cudaStream_t stream)
{
    if (mode == 1) return try_sweep<1, VEC, 1, 2>(ok, A, stream);
    cudaError_t e = try_sweep<1, VEC, 0, 2>(ok, A, stream);
    if (e == cudaSuccess && !ok) e = try_sweep<1, VEC, 0, 1>(ok, A, stream);
    return e == cudaSuccess && ok ? launch_fixup(A, stream) : e;
}

}  // namespace

cudaError_t launch_aggregate_tiles(bool &done, const float *copies, int64_t f, int r, int64_t d, int64_t ld,
                                   const int8_t *sel, aspis_detection *det, int mode, float *out,
                                   cudaStream_t stream, aspis_detection *gate)
{
    done = false;
    if (mode == 0 && f > kTileFiles) return cudaSuccess;
    const bool vec = (uintptr_t)copies % 16 == 0 && ld % 4 == 0;
    const SweepArgs A{copies, d, ld, (int)f, sel, det, out, nullptr, r, gate};
    return vec ? aggregate_rows<true>(done, A, mode, stream) : aggregate_rows<false>(done, A, mode, stream);
}

cudaError_t launch_decide(uint32_t *file_neq, const uint8_t *fw, int64_t f, int r, int K, uint32_t *adj,
                          aspis_detection *det, int8_t *sel, cudaStream_t stream)
{
    switch (r) {
    case 2: return decide<2>(file_neq, fw, (int)f, K, adj, det, sel, stream);
    case 3: return decide<3>(file_neq, fw, (int)f, K, adj, det, sel, stream);
    case 4: return decide<4>(file_neq, fw, (int)f, K, adj, det, sel, stream);
    case 5: return decide<5>(file_neq, fw, (int)f, K, adj, det, sel, stream);
    case 6: return decide<6>(file_neq, fw, (int)f, K, adj, det, sel, stream);
    case 7: return decide<7>(file_neq, fw, (int)f, K, adj, det, sel, stream);
    case 8: return decide<8>(file_neq, fw, (int)f, K, adj, det, sel, stream);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_round_fused(bool &done, const float *copies, int64_t f, int r, int K, int64_t d, int64_t ld,
                               const uint8_t *fw, uint32_t *file_neq, uint32_t *adj, aspis_detection *det,
                               int8_t *sel, int mode, float *out, cudaStream_t stream)
{
    done = false;
    const bool vec = (uintptr_t)copies % 16 == 0 && ld % 4 == 0;
    // The guess, its check and the empty repair cost about 20 us; the bytes
    // not read again are worth that from about 350 MB of copies on (455 files
    // of three: 102 us against 99 for the separate steps at 358 MB, 137
    // against 142 at 537 MB).
    if (r > 5 || f * r * d < kMinValues) return cudaSuccess;
    if (mode == 0 && f > kTileFiles) return cudaSuccess;
    const SweepArgs A{copies, d, ld, (int)f, sel, det, out, file_neq, r, nullptr};
    switch (r) {
    case 2: return fused<2>(done, A, fw, K, adj, sel, mode, vec, stream);
    case 3: return fused<3>(done, A, fw, K, adj, sel, mode, vec, stream);
    case 4: return fused<4>(done, A, fw, K, adj, sel, mode, vec, stream);
    default: return fused<5>(done, A, fw, K, adj, sel, mode, vec, stream);
    }
}

}  // namespace aspis
