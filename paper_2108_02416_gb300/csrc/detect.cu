// Steps 3-4 of the PS round.
//
// detect: all maximum cliques of G (Algorithm 3), one warp (max_cliques_warp).
// Each lane has a node budget; running out sets ASPIS_E_LIMIT and
// success = 0, so a pathological graph ends the search instead of stalling
// the stream.
//
// select: one copy per file (Algorithm 1): Case 1 honest copy / Case 2
// majority class of bitwise-equal copies, read from the mismatch word.
#include "aspis_internal.cuh"
#include "detect_common.cuh"

namespace aspis {
namespace {

__global__ void __launch_bounds__(32)
detect_kernel(const uint32_t *__restrict__ adj_g, int K, aspis_detection *det)
{
    __shared__ uint32_t adj[32];
    __shared__ Frame stack[32][32];          // [depth][lane]
    __shared__ int shared_best;
    const int v = threadIdx.x;
    const unsigned full = 0xffffffffu;
    const uint32_t row = v < K ? adj_g[v] : 0u;
    adj[v] = row;
    if (v == 0) shared_best = 0;
    const uint32_t budget = det->node_budget ? det->node_budget : kDefaultNodeBudget;
    // the closure step needs a symmetric graph without self loops, as
    // aspis_check writes it: column u (a ballot) must equal row u
    uint32_t col = 0u;
#pragma unroll
    for (int u = 0; u < 32; ++u) {
        const uint32_t m = __ballot_sync(full, (row >> u) & 1u);
        if (v == u) col = m;
    }
    const bool plain = __all_sync(full, col == row && !((row >> v) & 1u));
    __syncwarp();
    const CliqueResult c = plain ? max_cliques_warp<true>(adj, K, budget, stack, &shared_best)
                                 : max_cliques_warp<false>(adj, K, budget, stack, &shared_best);
    if (v == 0) {
        det->clique_mask = c.first;
        det->omega = c.omega;
        det->n_max_cliques = c.n_max;
        det->success = (c.n_max == 1u && !c.over) ? 1 : 0;
        det->n_sel = 0;
        det->median_exact = 0u;
        det->status = c.over ? ASPIS_E_LIMIT : ASPIS_OK;
        det->search_nodes = c.nodes;
    }
}

template <int R>
__global__ void __launch_bounds__(256)
select_kernel(const uint32_t *__restrict__ file_neq, aspis_detection *det,
              const uint8_t *__restrict__ fw, int64_t f, int8_t *__restrict__ sel)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int success = det->success;
    const uint32_t clique = det->clique_mask;
    int pick = -1;
    if (i < f) {
        pick = chosen_slot<R>(success != 0, clique, fw + i * R, success ? 0u : file_neq[i]);
        sel[i] = (int8_t)pick;
    }
    const int kept = __syncthreads_count(pick >= 0);
    if (threadIdx.x == 0 && kept) atomicAdd(&det->n_sel, kept);
}

}  // namespace

cudaError_t launch_detect(const uint32_t *adj, int K, aspis_detection *det, cudaStream_t stream)
{
    detect_kernel<<<1, 32, 0, stream>>>(adj, K, det);
    return cudaGetLastError();
}

cudaError_t launch_select(const uint32_t *file_neq, aspis_detection *det,
                          const uint8_t *dev_file_workers, int64_t f, int r, int8_t *sel,
                          cudaStream_t stream)
{
    const unsigned grid = (unsigned)((f + 255) / 256);
    switch (r) {
    case 2: select_kernel<2><<<grid, 256, 0, stream>>>(file_neq, det, dev_file_workers, f, sel); break;
    case 3: select_kernel<3><<<grid, 256, 0, stream>>>(file_neq, det, dev_file_workers, f, sel); break;
    case 4: select_kernel<4><<<grid, 256, 0, stream>>>(file_neq, det, dev_file_workers, f, sel); break;
    case 5: select_kernel<5><<<grid, 256, 0, stream>>>(file_neq, det, dev_file_workers, f, sel); break;
    case 6: select_kernel<6><<<grid, 256, 0, stream>>>(file_neq, det, dev_file_workers, f, sel); break;
    case 7: select_kernel<7><<<grid, 256, 0, stream>>>(file_neq, det, dev_file_workers, f, sel); break;
    case 8: select_kernel<8><<<grid, 256, 0, stream>>>(file_neq, det, dev_file_workers, f, sel); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace aspis
