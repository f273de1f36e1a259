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
//            and returns at once when the guess held.  (A round whose guess
//            is wrong takes 3 to 7% longer than taken apart, one whose guess
//            holds about 30% less: 1,332, 925 and 1,284 us at 455 files of
//            three and d = 1,048,576, 10.2, 6.9 and 9.9 ms at 8,388,608.)
//   fixup    the few coordinates whose median the sweep left open.
// The outputs are those of the separate steps.  All state between the kernels
// is in the caller's buffers: the guess in sel, the request for a repair in
// det->success (bit 1), taken back by the repair's last block, open
// coordinates as a bit pattern in out.
//
// The sweep is bound by HBM (61.0 GB in 9.8 ms = 6.2 TB/s at 455 files of
// three copies and 11.2M coordinates; the separate passes take 8.7 + 4.4 ms).
// With one copy per file (R = 1) it is the separate aggregation: 0.43 ms at
// 455 files and 2^20 coordinates.
#include "aspis_internal.cuh"
#include "detect_common.cuh"
#include "median_common.cuh"
#include "settle.cuh"
#include "sweep.cuh"

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
    chain();
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
constexpr int64_t kMinValues = 100'000'000;  // fp32 values of the smallest round taken in one pass
constexpr int64_t kMinAverages = 20'000'000; // and of the smallest averages that feed the median directly

// Steps 2-4 in one block (f <= ASPIS_MAX_AGG_FILES): three launches less than
// the separate kernels, which take 3 + 4..18 + 3 us one after the other.
//   GUESS    sel and det from the sampled words; file_neq is cleared for the
//            sweep, and kUnclean set in sel where copies of the file differ
//   VERIFY   the round's adj, det and sel; bit 1 of det->success is set where
//            sel held another guess
//   PLAIN    adj, det and sel
enum Decide { GUESS, VERIFY, PLAIN };

template <int R, Decide WHAT>
__global__ void __launch_bounds__(kDecideThreads)
decide_kernel(uint32_t *__restrict__ file_neq, const uint8_t *__restrict__ fw, int f, int K,
              uint32_t *__restrict__ adj_out, aspis_detection *det, int8_t *__restrict__ sel)
{
    __shared__ uint32_t dis[32], adj[32];
    __shared__ Frame stack[32][32];
    __shared__ int best, kept, success_s;
    __shared__ uint32_t clique_s;
    chain();
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

// ------------------------------------------------------------------- fixup

// The coordinates that the sweep left open (kOpen in out): a NaN among the
// values, a value bin with more members than a list holds, an overflowed
// counter, no spread in the sample.  Returns at once when det says that there
// are none.  A block looks through 32 * masks coordinates at a time (32 at a time
// took 50 us for a few open ones among 1,048,576) and settles what it finds, up
// to `most` of 32 neighbours together.
constexpr int kFixThreads = 256, kFixWarps = kFixThreads / 32, kFixMasks = 32;

__host__ __device__ constexpr size_t fixup_rows(int f)
{
    return ((size_t)f * 2 + 15) / 16 * 16;
}

__global__ void __launch_bounds__(kFixThreads)
fixup_kernel(const SweepArgs A, int masks, int most)
{
    chain();
    if (*(volatile const uint32_t *)&A.det->median_exact == 0u) return;
    extern __shared__ __align__(16) unsigned char smem[];
    uint16_t *rows = reinterpret_cast<uint16_t *>(smem);              // kept rows
    uint32_t *stage = reinterpret_cast<uint32_t *>(smem + fixup_rows(A.f));
    __shared__ int warp_tot[kFixWarps];
    __shared__ uint32_t open_s[kFixMasks];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, f = A.f;
    const unsigned full = 0xffffffffu;
    const int64_t step = (int64_t)gridDim.x * 32;
    int n = -1;
    for (int64_t c0 = (int64_t)blockIdx.x * 32; c0 < A.d; c0 += masks * step) {
        uint32_t any = 0u;
        for (int g = w; g < masks; g += kFixWarps) {
            const int64_t c = c0 + g * step + lane;
            const uint32_t x = c < A.d ? __float_as_uint(A.out[c]) : 0u;
            const uint32_t m = __ballot_sync(full, x == kOpen);
            if (lane == 0) open_s[g] = m;
            any |= m;
        }
        if (!__syncthreads_or(any != 0u)) continue;
        if (n < 0) {                       // the kept rows, once a block has work: a part of the files per warp
            const int per = (f + kFixThreads - 1) / kFixThreads * 32, i0 = w * per, i1 = min(f, i0 + per);
            int mine = 0;
#pragma unroll 4
            for (int i = i0 + lane; i < i0 + per; i += 32) mine += i < i1 && A.sel[i] >= 0;
            mine = __reduce_add_sync(full, mine);
            if (lane == 0) warp_tot[w] = mine;
            __syncthreads();
            int off = 0;
            n = 0;
            for (int q = 0; q < kFixWarps; ++q) {
                off += q < w ? warp_tot[q] : 0;
                n += warp_tot[q];
            }
            for (int i = i0 + lane; i < i0 + per; i += 32) {
                const int s = i < i1 ? (int)A.sel[i] : -1;
                const unsigned m = __ballot_sync(full, s >= 0);
                if (s >= 0) rows[off + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(i * A.r + s);
                off += __popc(m);
            }
            __syncthreads();
            if (n == 0) return;            // (these were the caller's own bits)
        }
        for (int g = 0; g < masks; ++g)
            for (uint32_t left = open_s[g], open; left; left &= ~open) {
                open = __popc(left) <= most ? left : left & ((2u << __fns(left, 0, most)) - 1u);
                settle<kFixThreads>(A.copies, A.ld, n, [&](int i) { return rows[i]; }, c0 + g * step, open, stage,
                                    A.out);
            }
        __syncthreads();
    }
}

// Keys of 32 neighbours where three blocks share an SM, of 16 where two do,
// else of 8 (a sector of every row).
cudaError_t launch_fixup(const SweepArgs &A, cudaStream_t stream)
{
    const int most = A.f <= 544 ? 32 : A.f <= 1632 ? 16 : 8;
    const size_t smem = fixup_rows(A.f) + (size_t)settle_words(A.f, most) * 4;
    static Residency resident;
    const int per_sm = resident.blocks(fixup_kernel, kFixThreads, smem);
    if (per_sm < 1) return cudaErrorInvalidValue;
    const int64_t masks = (A.d + 31) / 32;
    int64_t grid = (int64_t)sm_count() * per_sm;
    if (grid > masks) grid = masks;
    const int64_t at_once = (masks + grid - 1) / grid < kFixMasks ? (masks + grid - 1) / grid : kFixMasks;
    return launch_chained(fixup_kernel, grid, kFixThreads, smem, stream, A, (int)at_once, most);
}

template <int R>
cudaError_t fused(bool &done, const SweepArgs &A, const uint8_t *fw, int K, uint32_t *adj, int8_t *sel,
                  int mode, cudaStream_t stream)
{
    sample_kernel<R><<<(unsigned)((A.f + 3) / 4), kSampleThreads, 0, stream>>>(
        reinterpret_cast<const uint32_t *>(A.copies), A.f, A.d, A.ld, A.file_neq);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_chained(decide_kernel<R, GUESS>, 1, kDecideThreads, 0, stream, A.file_neq, fw, A.f, K, adj, A.det, sel);
    if (e != cudaSuccess) return e;
    bool ok = false, open = false;
    if ((e = launch_sweep<R>(ok, open, A, mode, true, stream)) != cudaSuccess) return e;
    if (!ok) return cudaErrorInvalidValue;
    e = launch_chained(decide_kernel<R, VERIFY>, 1, kDecideThreads, 0, stream, A.file_neq, fw, A.f, K, adj, A.det, sel);
    if (e != cudaSuccess) return e;
    done = true;
    return launch_aggregate(A.copies, A.f, R, A.d, A.ld, sel, A.det, mode, A.out, stream, A.det, true);
}

template <int R>
cudaError_t decide(uint32_t *file_neq, const uint8_t *fw, int f, int K, uint32_t *adj, aspis_detection *det,
                   int8_t *sel, cudaStream_t stream)
{
    return launch_chained(decide_kernel<R, PLAIN>, 1, kDecideThreads, 0, stream, file_neq, fw, f, K, adj, det, sel);
}

}  // namespace

cudaError_t launch_aggregate(const float *copies, int64_t f, int r, int64_t d, int64_t ld, const int8_t *sel,
                             aspis_detection *det, int mode, float *out, cudaStream_t stream,
                             aspis_detection *gate, bool chained)
{
    if (f > ASPIS_MAX_AGG_FILES || f * r > 65535) return cudaErrorInvalidValue;
    const SweepArgs A{copies, d, ld, (int)f, sel, det, out, nullptr, r, gate, nullptr, nullptr, 0};
    // Few files: whole values sorted in registers (89 us for the round against 52 at
    // 35 files of three, d = 400,000; 24 against 23 at 4,096).
    if (mode == 0 && f <= kFewFiles && !gate) return launch_aggregate_few(copies, f, r, d, ld, sel, det, out, chained, stream);
    // Many files: one pass over narrow tiles (2,024 files, d = 9,000: 28 us, 92 for
    // two passes over wide ones) or two passes with more rows in flight (3,003
    // files: 126 us against 165).
    if (mode == 0 && f > kTagFiles && !gate) return launch_aggregate_many(copies, f, r, d, ld, sel, det, out, stream);
    // 517 to 1,330 files: a block of 128-coordinate tiles has an SM to itself.  Up to
    // about 950 files two of 64-coordinate ones share it (us, wide and narrow, 816
    // files: 35 and 26 at d = 4,096, 54 and 51 at 36,928, 273 and 243 at 262,144, 988
    // and 946 at 1,048,576).  Where rows are not 16-byte aligned, narrower tiles are
    // also better while the wide ones make up to three waves (1,287 files, 4-byte
    // rows: 60 and 50 at 16,317, 88 and 69 at 24,865, 117 and 108 at 48,173, but 1,560
    // and 2,640 at 1,048,577).
    if (mode == 0 && f > kPairFiles && !gate) {
        bool done = false;
        const bool few = (d + 127) / 128 <= 3 * (int64_t)sm_count();
        const cudaError_t e = launch_aggregate_narrow(done, copies, f, r, d, ld, sel, det, out, few, stream);
        if (e != cudaSuccess) return e;
        if (done) return launch_fixup(A, stream);
    }
    // The mean by itself: tiles of 32 loads per row (of 512, 256 or 128 bytes) where
    // the 128-coordinate tiles are few, and for 8-byte rows of few files (us, wide
    // and narrow): 455 files, d = 3,661, 23.0 and 17.5; 3,276, 10,172, 62.9 and
    // 48.0; 1,330, 25,060, 43.9 and 39.3, 250,624, 228 and 224; 4-byte rows of 1,330,
    // 25,061, 47.2 and 50.0; 8-byte rows of 84, 3,968,254, 410 and 296, of 3,276,
    // 101,750, 237 and 251.  Within a round the wide tiles start early, which is worth
    // 3 us (3,003 files of five, d = 6,662: 148 and 126).
    if (mode == 1 && !gate && (!chained || f > kTagFiles)) {
        const int width = load_width(copies, ld);
        if ((d + 127) / 128 <= (width == 1 ? 1 : 4) * (int64_t)sm_count() || (width == 2 && f <= kPairFiles))
            return launch_aggregate_mean(copies, f, r, d, ld, sel, det, out, stream);
    }
    bool ok = false, open = false;
    const cudaError_t e = launch_sweep<1>(ok, open, A, mode, chained, stream);
    if (e != cudaSuccess) return e;
    if (!ok) return cudaErrorInvalidValue;
    // (a repair that does not run has settled nothing of the one-pass sweep)
    return open || (gate && mode == 0) ? launch_fixup(A, stream) : cudaSuccess;
}

cudaError_t launch_average_median(bool &done, const float *copies, int64_t f, int r, int64_t d, int64_t ld,
                                  const uint8_t *slot_mask, const int8_t *sel, float *means, int64_t ldm,
                                  aspis_detection *det, float *out, cudaStream_t stream)
{
    done = false;
    // (62 against 54 us at 455 files of three and d = 4,096, 73 against 75 at
    // 16,384, 176 against 199 at 65,536; with few files the tiles' fixed work costs
    // more than reading the averages again: 1,079 against 786 us at 35 and 4,000,000)
    if (r > 5 || f <= kFewFiles || f > kTagFiles || f * r * d < kMinAverages) return cudaSuccess;
    const SweepArgs A{copies, d, ld, (int)f, sel, det, out, nullptr, r, nullptr, slot_mask, means, ldm};
    cudaError_t e;
    switch (r) {
    case 2: e = launch_sweep_averages<2>(done, A, stream); break;
    case 3: e = launch_sweep_averages<3>(done, A, stream); break;
    case 4: e = launch_sweep_averages<4>(done, A, stream); break;
    default: e = launch_sweep_averages<5>(done, A, stream); break;
    }
    if (e != cudaSuccess || !done) return e;
    // open coordinates: from the averages, one row per file
    const SweepArgs F{means, d, ldm, (int)f, sel, det, out, nullptr, 1, nullptr, nullptr, nullptr, 0};
    return launch_fixup(F, stream);
}

// Whether the one-pass round beats the separate compare and aggregation, from
// the bytes that each moves, the rates measured for them (TB/s on GB300) and the
// launches (the guess, its check and the empty repair: 30 us against 10).  Tiles
// of 128 coordinates run one per resident block at a time, and a last wave that
// is nearly empty costs about 0.4 of a full one (its blocks have the bandwidth
// for themselves): the one-pass mean of 3,003 files of five copies takes 550 us
// against 482 with 316 tiles on 304 blocks, 1,309 against 1,355 with 1,024.
// width: floats that a row start is aligned to (4, 2 or 1).
bool one_pass_pays(int64_t f, int r, int64_t d, int mode, int width)
{
    // few files (35 of three, d = 11,173,962): 1,223 us apart, 1,332 with the copies
    // compared and sorted in registers in one pass, 1,736 with the tile kernel
    if (mode == 0 && f <= kFewFiles) return false;
    const bool many = mode == 0 && f > kTagFiles;                       // two passes over the chosen rows
    const int64_t tiles = (d + 127) / 128;
    const int64_t blocks = (int64_t)sm_count() * (mode == 1 || many || f <= kPairFiles ? 2 : 1);
    const double full = (double)((tiles + blocks - 1) / blocks * blocks) / (double)tiles;
    const double all = (double)f * r * (double)d * 4e-6, chosen = all / r;      // MB: us at 1 TB/s
    if (many) {
        // The separate median has tags and one pass in 64-coordinate (rows of 4-byte
        // alignment: 32-coordinate) tiles up to kNarrowFiles files; beyond them two
        // passes over 16-byte rows, one in 32-coordinate tiles over others.  Many
        // rows far apart cost both ways page walks.  Fitted to 15 clusters of 1,540
        // to 5,985 files, 2 x 10^7 to 6 x 10^9 values and the three alignments; the
        // better way or one within 5% of it is taken, some of it (one pass and apart
        // in us):
        //   16 bytes  1,540 of three   d = 151,512    751 and   817   670,992  2,914 and 3,474
        //             2,002 of five        104,892  1,007 and   921   309,688  2,586 and 2,677
        //             2,600 of three       134,612  1,168 and 1,114   397,432  3,021 and 3,165
        //             3,003 of five         46,620    896 and   880    69,928  1,029 and 1,116
        //             4,368 of five         32,048    792 and   979    73,260  1,638 and 1,785
        //    8 bytes  2,002 of five        159,842  1,788 and 1,590   309,690  3,089 and 3,512
        //             3,276 of three        40,702    716 and   562   162,802  2,009 and 2,231
        //             4,368 of five         18,314    659 and   486   274,726  6,720 and 6,940
        //    4 bytes  2,024 of three        32,937    314 and   313   172,925  1,270 and 1,582
        //             4,845 of four        159,957  4,202 and 3,752   309,597  7,201 and 7,855
        const double once = (all + chosen) * (1.0 + 0.6 * (full - 1.0));
        if (f > kNarrowFiles && width < 4)
            return once / (6.23 - 0.377e-3 * (double)f) + 180.0 < all / 5.7 + chosen / 1.9 + 10.0;
        if (width == 4)
            return once / 6.3 + 180.0 <
                   all / 7.1 + (f <= kNarrowFiles ? chosen / 2.7 + 10.0 : chosen / 2.6 + 0.1 * (double)f - 90.0);
        return width == 2 ? once / 5.5 + 180.0 < all / 5.8 + chosen / 2.7 + 10.0
                          : once / 5.4 + 180.0 < all / 5.9 + chosen / 1.75 + 10.0;
    }
    if (f * r * d < kMinValues) return false;
    // 517 to 1,330 files in 4-byte loads (1,287 of five, d = 48,173: 356 and 330 us;
    // 1,330 of three, 40,101: 249 and 230, 77,693: 309 and 411)
    if (mode == 0 && width == 1 && f > kPairFiles)
        return all / 4.7 * full + 30.0 < all / 5.6 + chosen / 2.3 + 10.0;
    const double wave = 1.0 + 0.4 * (full - 1.0);
    return all / 6.3 * wave + 30.0 < all / 7.1 + chosen / (mode == 1 ? 5.6 : 4.4) * wave + 10.0;
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
    if (r > 5 || !one_pass_pays(f, r, d, mode, load_width(copies, ld))) return cudaSuccess;
    const SweepArgs A{copies, d, ld, (int)f, sel, det, out, file_neq, r, nullptr, nullptr, nullptr, 0};
    switch (r) {
    case 2: return fused<2>(done, A, fw, K, adj, sel, mode, stream);
    case 3: return fused<3>(done, A, fw, K, adj, sel, mode, stream);
    case 4: return fused<4>(done, A, fw, K, adj, sel, mode, stream);
    default: return fused<5>(done, A, fw, K, adj, sel, mode, stream);
    }
}

}  // namespace aspis
