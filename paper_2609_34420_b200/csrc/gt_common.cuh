// Shared host/device helpers of the CUDA library (status word, argument checks, launch checks).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>

#include <atomic>
#include <utility>

#include "../../include/gt_attn.h"

namespace gt {

// Workspace header: the first 256 bytes of every workspace.
//   word 0 : device status (gt_status), written by kernels, read+cleared by gt_check
//   word 1 : debug detail of the first failing wait (site id)
//   word 2 : work counter of persistent kernels (reset by each call)
//   word 3 : number of work items (written by set-up kernels)
constexpr size_t kHeaderBytes = 256;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline bool misaligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; }

inline gt_status validate_batch(const gt_batch* b)
{
    if (b == nullptr) return GT_ERR_INVALID_ARG;
    if (b->n_total < 1 || b->n_graphs < 1 || b->max_seqlen < 1 || b->max_seqlen > b->n_total) return GT_ERR_INVALID_ARG;
    if (b->n_graphs > 1 && b->cu_seqlens == nullptr) return GT_ERR_INVALID_ARG;
    if (b->n_graphs == 1 && b->max_seqlen != b->n_total) return GT_ERR_INVALID_ARG;
    return GT_OK;
}

#define GT_CUDA_TRY(expr)                                                              \
    do {                                                                               \
        cudaError_t e__ = (expr);                                                      \
        if (e__ != cudaSuccess) {                                                      \
            if (getenv("GT_DEBUG"))                                                    \
                fprintf(stderr, "[gt_attn] %s failed: %s (%s:%d)\n", #expr,           \
                        cudaGetErrorString(e__), __FILE__, __LINE__);                  \
            return GT_ERR_CUDA;                                                        \
        }                                                                              \
    } while (0)

// Kernels of this library are launched so that a kernel may start while the one before it in the stream is still running
// (programmatic dependent launch): its set-up -- barriers, tensor memory, tables in registers -- and the launch itself then
// overlap with the other's end.  Every such kernel calls grid_wait() before its first access to global memory, which returns
// when everything before it in the stream is complete and visible, and grid_release() as soon as the next kernel may start
// its own set-up.  (A kernel that is not of this library releases at its end; one that does not wait starts when all is done.)
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Params, typename... Args>
inline gt_status launch_overlapped_cluster(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem_bytes, int cluster, cudaStream_t stream,
                                           Args&&... args)
{
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    GT_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...));
    return GT_OK;
}
template <typename... Params, typename... Args>
inline gt_status launch_overlapped(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem_bytes, cudaStream_t stream, Args&&... args)
{
    return launch_overlapped_cluster(kernel, grid, threads, smem_bytes, 1, stream, std::forward<Args>(args)...);
}

// Lets a kernel use up to `bytes` of dynamic shared memory, once per device: `granted` is that kernel's own (a bit per device),
// `bytes` always the same, so it does not matter how many threads ask at once.
template <class Kernel>
inline gt_status grant_smem(Kernel kernel, std::atomic<uint64_t>& granted, size_t bytes)
{
    int dev = 0;
    GT_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 64 && ((granted.load(std::memory_order_relaxed) >> dev) & 1u)) return GT_OK;
    GT_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    if (dev < 64) granted.fetch_or(1ull << dev, std::memory_order_relaxed);
    return GT_OK;
}

// Number of SMs of the current device (cached per device).
int sm_count();

__device__ __forceinline__ void report_timeout(uint32_t* status, uint32_t site)
{
    if (atomicCAS(status, 0u, (uint32_t)GT_ERR_DEVICE_TIMEOUT) == 0u) status[1] = site;
}

}  // namespace gt
