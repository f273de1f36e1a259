// sweep_kernel for 5 copies per file.
#include "sweep_impl.cuh"

namespace aspis {
template cudaError_t launch_sweep<5>(bool &, bool &, const SweepArgs &, int, bool, cudaStream_t);
template cudaError_t launch_sweep_averages<5>(bool &, const SweepArgs &, cudaStream_t);
}  // namespace aspis
