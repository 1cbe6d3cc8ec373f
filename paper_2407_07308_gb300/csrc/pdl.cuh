// pdl.cuh -- programmatic dependent launch for the hot kernels.
//
// A kernel launched with the attribute may have its CTAs made resident while
// the previous kernel on its stream is still finishing (that kernel lets its
// dependents launch once all of its CTAs have started, pdl_trigger); it finds
// its unit and fetches tables that no kernel writes (twiddles, level
// constants, key words) and then waits until all prerequisite grids have
// completed and their memory operations are visible (pdl_wait) -- before it
// reads or writes anything another kernel touches.  Every kernel of this kind
// waits in every CTA, so completion carries over from launch to launch.  In a
// captured graph the launches become programmatic edges.  A kernel launched
// without the attribute passes both at once.
//
// Where it is used: always on a context's own stream, where every launch
// follows the one before (launch and prologue are then hidden: one less-than
// on the small ring 668 -> 508 us, one LT + EQ at N = 2^14 2249 -> 2116 us,
// tournament of 8 ciphertexts 171.8 -> 164.3 ms); under the dependency
// scheduler, whose streams run side by side, only for launches of at most
// FHE_PDL_THREADS threads per SM, since waiting CTAs hold slots that another
// stream's kernels would use (16 pairs as a graph: 9.62 ms without, 9.63 at
// 256, 9.69 at 512, 9.84 with all; 32 uneven requests 46.8, 46.5, 46.5, 46.3).
#pragma once
#include <cuda_runtime.h>

#include <utility>

#ifndef FHE_PDL_THREADS
#define FHE_PDL_THREADS 256
#endif

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void pdl_begin()
{
    pdl_trigger();
    pdl_wait();
}

template <class... KArgs, class... Args>
inline void launch_attrs(void (*kernel)(KArgs...), bool overlap, int cluster, int grid, int block, size_t smem,
                         cudaStream_t s, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (overlap) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)n;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);  // errors surface in cudaGetLastError
}

template <class... KArgs, class... Args>
inline void launch_pdl_smem(void (*kernel)(KArgs...), bool overlap, int grid, int block, size_t smem, cudaStream_t s,
                            Args &&...args)
{
    if (!overlap)
        kernel<<<grid, block, smem, s>>>(std::forward<Args>(args)...);
    else
        launch_attrs(kernel, true, 1, grid, block, smem, s, std::forward<Args>(args)...);
}

// grid a multiple of cluster (above 8, the portable size, the kernel opts in)
template <class... KArgs, class... Args>
inline void launch_pdl_cluster(void (*kernel)(KArgs...), bool overlap, int grid, int block, int cluster, cudaStream_t s,
                               Args &&...args)
{
    if (cluster > 8) cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    launch_attrs(kernel, overlap, cluster, grid, block, 0, s, std::forward<Args>(args)...);
}

template <class... KArgs, class... Args>
inline void launch_pdl(void (*kernel)(KArgs...), bool overlap, int grid, int block, cudaStream_t s, Args &&...args)
{
    launch_pdl_smem(kernel, overlap, grid, block, 0, s, std::forward<Args>(args)...);
}
