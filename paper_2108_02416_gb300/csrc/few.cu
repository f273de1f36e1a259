// Lower median of at most kFewFiles files: a thread holds one value of every
// file and sorts them.  The tile kernel (sweep.cuh) spends the same 3 to 4 us on
// a tile's bins, search and lists however few files there are; this one has no
// barrier per tile and needs no alignment.  Small lengths are bound by latency,
// large ones by the sort's minima and maxima.  The whole round of 35 files of
// three copies, before and after: 43 and 27 us at d = 100,000, 89 and 52 at
// 400,000, 342 and 228 at 2,000,000, 1,736 and 1,223 at 11,173,962.
#include "sweep.cuh"

namespace aspis {
namespace {

constexpr int kFewThreads = 64;
constexpr int kFewBatch = 9;                // rows in flight per thread beyond those being placed
constexpr int kMid = (kFewFiles - 1) / 2;   // the sorted place of the lower median
static_assert(kFewFiles % (2 * kFewBatch) == 0, "batches in pairs");

// One coordinate per thread, any alignment.  Files that are not aggregated, and
// those beyond f, hold the smallest or the largest key, as many of each as put
// the median at kMid; of the sort only the comparators that reach kMid remain.
__global__ void __launch_bounds__(kFewThreads)
few_kernel(const float *copies, int f, int r, int64_t d, int64_t ld, const int8_t *sel, aspis_detection *det,
           float *out)
{
    chain();
    __shared__ int row_s[kFewFiles];        // the chosen row, or -1: low, -2: high
    __shared__ int n_s;
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31;
    constexpr int kG = (kFewFiles + 31) / 32;
    if (tid < 32) {
        int n = 0, absent = 0, row[kG], place[kG];
#pragma unroll
        for (int g = 0; g < kG; ++g) {
            const int i = g * 32 + lane;
            const int s = i < f ? (int)sel[i] : -1;
            const unsigned in = __ballot_sync(full, s >= 0), no = __ballot_sync(full, s < 0 && i < kFewFiles);
            row[g] = s >= 0 ? i * r + s : -1;
            place[g] = absent + __popc(no & ((1u << lane) - 1u));
            n += __popc(in);
            absent += __popc(no);
        }
        const int low = kMid - (n - 1) / 2;
#pragma unroll
        for (int g = 0; g < kG; ++g)
            if (g * 32 + lane < kFewFiles) row_s[g * 32 + lane] = row[g] >= 0 ? row[g] : place[g] < low ? -1 : -2;
        if (lane == 0) n_s = n;
    }
    __syncthreads();
    if (n_s == 0) {
        if (tid == 0 && blockIdx.x == 0) det->status = ASPIS_E_EMPTY;
        return;
    }
    for (int64_t c = (int64_t)blockIdx.x * kFewThreads + tid; c < d; c += (int64_t)gridDim.x * kFewThreads) {
        const uint32_t *at = reinterpret_cast<const uint32_t *>(copies) + c;
        uint32_t xa[kFewBatch], xb[kFewBatch], y[kFewFiles];
        auto load = [&](uint32_t (&x)[kFewBatch], int i0) {
#pragma unroll
            for (int u = 0; u < kFewBatch; ++u) {
                const int row = row_s[i0 + u];
                x[u] = row >= 0 ? __ldg(at + (int64_t)row * ld) : 0u;
            }
        };
        auto place = [&](const uint32_t (&x)[kFewBatch], int i0) {
#pragma unroll
            for (int u = 0; u < kFewBatch; ++u) {
                const int row = row_s[i0 + u];
                y[i0 + u] = row >= 0 ? to_key(x[u]) : row == -1 ? 0u : 0xffffffffu;
            }
        };
        load(xa, 0);
#pragma unroll
        for (int i0 = 0; i0 < kFewFiles; i0 += 2 * kFewBatch) {
            load(xb, i0 + kFewBatch);
            place(xa, i0);
            if (i0 + 2 * kFewBatch < kFewFiles) load(xa, i0 + 2 * kFewBatch);
            place(xb, i0 + kFewBatch);
        }
        merge_sort<kFewFiles>(y);
        out[c] = __uint_as_float(from_key(y[kMid]));
    }
}

}  // namespace

cudaError_t launch_aggregate_few(const float *copies, int64_t f, int r, int64_t d, int64_t ld, const int8_t *sel,
                                 aspis_detection *det, float *out, bool chained, cudaStream_t stream)
{
    static Residency resident;
    const int per_sm = resident.blocks(few_kernel, kFewThreads, 0);
    int64_t grid = (int64_t)sm_count() * (per_sm > 0 ? per_sm : 1);
    const int64_t tiles = (d + kFewThreads - 1) / kFewThreads;
    if (grid > tiles) grid = tiles;
    if (chained) return launch_chained(few_kernel, grid, kFewThreads, 0, stream, copies, (int)f, r, d, ld, sel, det, out);
    few_kernel<<<(unsigned)grid, kFewThreads, 0, stream>>>(copies, (int)f, r, d, ld, sel, det, out);
    return cudaGetLastError();
}

}  // namespace aspis
