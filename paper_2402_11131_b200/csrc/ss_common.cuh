// Internal helpers shared by the CUDA translation units of libss_msa.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "ss_msa.h"

namespace ss {

// Workspace header: word 0 = device status, the rest of the first 256 bytes is reserved.
constexpr size_t kWsHeaderBytes = 256;

__device__ __forceinline__ void set_status(void* workspace, int32_t code) {
    atomicCAS(reinterpret_cast<int*>(workspace), 0, code);   // keep the first error
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline int sm_count() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
        cached[dev] = n;
    }
    return cached[dev];
}

// Programmatic dependent launch.  A kernel launched with launch_after_previous may be scheduled while the
// previous kernel of the stream drains; it must call wait_for_previous_kernel() before it touches global
// memory, which restores plain stream order for everything after the call.
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The other half: lets the next kernel of the stream be scheduled from here on.  Called after the wait only, so at most
// two kernels of a stream are ever on the GPU: what ran before the previous kernel is complete.  A kernel that writes tree
// descriptors calls it only once they are in memory, or not at all: an attention call behind it may promise that they are
// stable and reads them before its wait.
__device__ __forceinline__ void release_next_kernel() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// `cluster` CTAs along x form a cluster; early: may be scheduled while the previous kernel of the stream drains
template <typename... KArgs, typename... Args>
inline cudaError_t launch_rows(void (*kernel)(KArgs...), dim3 grid, dim3 block, int cluster, bool early, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (early) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = static_cast<unsigned>(cluster);
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = static_cast<unsigned>(n);
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_after_previous(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t stream, Args... args) {
    return launch_rows(kernel, grid, block, 1, true, stream, args...);
}

}  // namespace ss
