// sweep_kernel for 2 copies per file.
#include "sweep_impl.cuh"

namespace aspis {
template cudaError_t launch_sweep<2>(bool &, bool &, const SweepArgs &, int, bool, cudaStream_t);
template cudaError_t launch_sweep_averages<2>(bool &, const SweepArgs &, cudaStream_t);
}  // namespace aspis
