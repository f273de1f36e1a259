// sweep_kernel for one row per file (the separate aggregation).
#include "sweep_impl.cuh"

namespace aspis {
template cudaError_t launch_sweep<1>(bool &, bool &, const SweepArgs &, int, bool, cudaStream_t);
}  // namespace aspis
