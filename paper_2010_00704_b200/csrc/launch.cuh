// Host side of a launch.  A call on a small layer is a few microseconds of GPU work, so what the host does per launch
// counts: device properties and kernel attributes are looked up once per process (and device), not once per call.
#pragma once
#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>
#include "bcnn.h"

namespace bcnn {

// Multiprocessors of the current device (148 where the query fails).
int sm_count();
// Resident blocks of `kernel` per multiprocessor (at least 1).
int blocks_per_sm(const void *kernel, int threads, size_t smem);
// Clusters of `cluster` blocks of `kernel` that the device holds at a time; 0 where the query fails.  Fewer than its multiprocessors give in sum:
// a cluster lies within one processing cluster (at one block a multiprocessor fifteen of eight, 33 of four, 74 of two on 148).
int max_clusters(const void *kernel, int cluster, int threads, size_t smem);
// Raises the kernel's dynamic shared-memory limit to `bytes` on the current device; the driver is asked on the first
// call only.  The limit is a property of the kernel, not of a launch: callers always pass the same `bytes` for a kernel,
// so a captured launch stays valid whatever later calls with other shapes ask for.
bool allow_smem(const void *kernel, int bytes);

template <typename T> struct Same { using type = T; };

// Every kernel is launched as a programmatic dependent of what the stream runs before it: its blocks may start while that
// kernel is still finishing, and wait (pdl_wait) before they touch global memory.  Measured on B200: kernels launched one
// by one on a stream otherwise start on a 2.048 us grid (a kernel of 3.3 us repeats every 6.1 us, as a programmatic
// dependent every 3.6 us), and consecutive kernels of a CUDA graph are 0.7 us apart, as dependents 0.2 us.
//   * pdl_wait: by every thread that reads or writes global memory, before the first access, in EVERY kernel - a kernel
//     that does not wait would let the one after it overtake the one before it;
//   * pdl_trigger: the next kernel's blocks may be scheduled.  A kernel that allocates tensor memory calls it behind the
//     allocation only: a waiting block of the next kernel must not take the columns this grid still needs.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// kernel<<<grid, threads, smem, stream>>>(args...), the arguments converted to the kernel's parameter types; in clusters of CLUSTER blocks.
template <int CLUSTER = 1, typename... P>
int launch(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, typename Same<P>::type... args)
{
    void *argv[] = {const_cast<void *>(static_cast<const void *>(&args))...};
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = CLUSTER;
    attrs[1].val.clusterDim.y = attrs[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attrs;
    cfg.numAttrs = CLUSTER > 1 ? 2 : 1;
    if (cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(kernel), argv) == cudaSuccess) return BCNN_OK;
    (void)cudaGetLastError();                 // a refused launch leaves no error behind for the caller's next check
    return BCNN_ERR_CUDA;
}

}  // namespace bcnn
