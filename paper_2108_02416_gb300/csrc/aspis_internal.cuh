// Internal declarations shared by the libaspis translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "aspis.h"

namespace aspis {

// Launch helpers: enqueue on `stream`, return cudaGetLastError().
// launch_compare overwrites file_neq entirely.
cudaError_t launch_compare(const float *copies, int64_t f, int r, int64_t d,
                           int64_t ld, uint32_t *file_neq, cudaStream_t stream);
cudaError_t launch_graph(const uint32_t *file_neq, const uint8_t *dev_file_workers,
                         int64_t f, int r, int K, uint32_t *adj, cudaStream_t stream);
cudaError_t launch_detect(const uint32_t *adj, int K, aspis_detection *det,
                          cudaStream_t stream);
cudaError_t launch_select(const uint32_t *file_neq, aspis_detection *det,
                          const uint8_t *dev_file_workers, int64_t f, int r,
                          int8_t *sel, cudaStream_t stream);
// gate: a repair of the one-pass round (round.cu), or NULL.  chained: the
// kernel before it on the stream is one of the same call that calls chain().
cudaError_t launch_aggregate(const float *copies, int64_t f, int r, int64_t d,
                             int64_t ld, const int8_t *sel, aspis_detection *det,
                             int mode, float *out, cudaStream_t stream,
                             aspis_detection *gate = nullptr, bool chained = false);
// Averages of the copies in slot_mask into means (16-byte aligned rows) and
// their lower median in one pass; done = false (and nothing enqueued) where the
// separate passes are better or the only ones.
cudaError_t launch_average_median(bool &done, const float *copies, int64_t f, int r, int64_t d, int64_t ld,
                                  const uint8_t *slot_mask, const int8_t *sel, float *means, int64_t ldm,
                                  aspis_detection *det, float *out, cudaStream_t stream);
// The lower median for f > kTagFiles (aggregate.cu).
cudaError_t launch_aggregate_many(const float *copies, int64_t f, int r, int64_t d, int64_t ld,
                                  const int8_t *sel, aspis_detection *det, float *out, cudaStream_t stream);
// The lower median in 64-coordinate tiles, two blocks per SM where the files'
// tag bytes allow it; few: else also one block, or (rows of 4-byte alignment)
// 32-coordinate tiles.  fixup_kernel has to follow.  done = false (and nothing
// enqueued) where the 128-coordinate tiles of sweep_kernel are better.
cudaError_t launch_aggregate_narrow(bool &done, const float *copies, int64_t f, int r, int64_t d, int64_t ld,
                                    const int8_t *sel, aspis_detection *det, float *out, bool few,
                                    cudaStream_t stream);
// The mean in tiles of 32 loads of the widest kind that the rows allow.
cudaError_t launch_aggregate_mean(const float *copies, int64_t f, int r, int64_t d, int64_t ld, const int8_t *sel,
                                  aspis_detection *det, float *out, cudaStream_t stream);
// At most kFewFiles files (sweep.cuh), median.
cudaError_t launch_aggregate_few(const float *copies, int64_t f, int r, int64_t d, int64_t ld, const int8_t *sel,
                                 aspis_detection *det, float *out, bool chained, cudaStream_t stream);
// Steps 2-4 (graph, maximum cliques, selection) in one launch, for f <=
// ASPIS_MAX_AGG_FILES.
cudaError_t launch_decide(uint32_t *file_neq, const uint8_t *dev_file_workers, int64_t f, int r, int K,
                          uint32_t *adj, aspis_detection *det, int8_t *sel, cudaStream_t stream);
// The whole round in one pass over the copies; done = false (and nothing
// enqueued) where the separate steps have to run.
cudaError_t launch_round_fused(bool &done, const float *copies, int64_t f, int r, int K, int64_t d,
                               int64_t ld, const uint8_t *dev_file_workers, uint32_t *file_neq,
                               uint32_t *adj, aspis_detection *det, int8_t *sel, int mode,
                               float *out, cudaStream_t stream);

// Number of SMs of the current device (cached per device).
int sm_count();

// Dynamic shared memory a block may ask for on the current device (cached).
size_t smem_cap();

// Kernels of one call that follow one another are launched as programmatic
// dependents: the next one's blocks are scheduled while this one still runs and
// wait in chain() for its end and its writes, which hides the 2 to 3 us between
// dependent kernels.  Every kernel of a chain calls chain() before it touches
// global memory; the first one is launched plainly, and so waits for all earlier
// work on the stream.  Measured: the separate kernels of a round over 455 files
// of three and d = 36,932 65 us against 72, over 35 files and d = 4,096 21.3 against
// 23.3, the six of the one-pass round at d = 1,048,576 1,222 against 1,225.
__device__ __forceinline__ void chain()
{
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), int64_t grid, int threads, size_t smem, cudaStream_t stream,
                           A... args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Blocks of one kernel that an SM holds, asked of the runtime once per device
// and amount of dynamic shared memory (the last amount is kept, in one word, so
// that threads cannot see half of another's answer).
class Residency {
public:
    template <class K>
    int blocks(K kernel, int threads, size_t smem)
    {
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 0 || dev >= 64) dev = 0;
        const uint64_t known = last_[dev].load(std::memory_order_relaxed);
        if ((known >> 8) == smem + 1) return (int)(known & 0xFFu);
        // (always the same limit: another thread's call may need more than this one)
        if (smem > 0 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_cap()) !=
                            cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        last_[dev].store(((uint64_t)(smem + 1) << 8) | (uint64_t)(n < 255 ? n : 255), std::memory_order_relaxed);
        return n;
    }

private:
    std::atomic<uint64_t> last_[64] = {};
};

__host__ __device__ inline int pair_count(int r) { return r * (r - 1) / 2; }

}  // namespace aspis
