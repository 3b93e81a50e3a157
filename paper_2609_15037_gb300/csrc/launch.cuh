// Kernel launches that may begin before the kernel in front of them has ended
// (programmatic dependent launch).  The refresh is a chain of several hundred
// short kernels, a small model's step one of three: a launch's own latency and
// the next kernel's setup run beside the end of the kernel in front.
//
// A kernel launched this way calls pdl_begin() before it touches memory that
// earlier kernels write: it lets the kernel behind it be launched once all its
// CTAs have begun, and waits until the kernel in front has ended and its writes
// are visible (which that kernel in turn did).  Behind anything but such a
// kernel the launch is an ordinary one.
#pragma once

#include <cuda_runtime.h>
#include <type_traits>

namespace moara {

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}
#endif

// cluster: CTAs per cluster along x (1: none); overlap: whether the kernel may
// begin early (off where events of another stream stand between the two)
template <class... P, class... A>
cudaError_t launch_if(bool overlap, void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster,
                      const A&... args) {
    static_assert((std::is_same<typename std::remove_cv<P>::type, A>::value && ...), "exact argument types");
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    void* ptrs[] = {const_cast<void*>(static_cast<const void*>(&args))...};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, reinterpret_cast<const void*>(fn), ptrs);
    // reported here: a later call that asks for the runtime's last error must not meet it again
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

template <class... P, class... A>
cudaError_t launch(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster, const A&... args) {
    return launch_if(true, fn, grid, block, smem, s, cluster, args...);
}

}  // namespace moara
