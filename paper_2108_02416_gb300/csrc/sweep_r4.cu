// sweep_kernel for 4 copies per file.
#include "sweep_impl.cuh"

namespace aspis {
template cudaError_t launch_sweep<4>(bool &, bool &, const SweepArgs &, int, bool, cudaStream_t);
template cudaError_t launch_sweep_averages<4>(bool &, const SweepArgs &, cudaStream_t);
}  // namespace aspis
