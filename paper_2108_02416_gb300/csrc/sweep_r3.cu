// sweep_kernel for 3 copies per file.
#include "sweep_impl.cuh"

namespace aspis {
template cudaError_t launch_sweep<3>(bool &, bool &, const SweepArgs &, int, bool, cudaStream_t);
template cudaError_t launch_sweep_averages<3>(bool &, const SweepArgs &, cudaStream_t);
}  // namespace aspis
