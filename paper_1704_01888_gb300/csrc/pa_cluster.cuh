// pa_cluster.cuh -- helpers of kernels whose blocks work as a thread-block
// cluster: reductions through distributed shared memory, and their launch.
#pragma once
#include <cooperative_groups.h>

#include <climits>

#include "pa_internal.cuh"

namespace pa {

namespace cg = cooperative_groups;

namespace dev {

// Smallest and largest of lo and hi over the cluster; every thread receives
// both.  sc: 64 ints, mine: 2 ints read by the other blocks.
__device__ __forceinline__ void cluster_extremes(cg::cluster_group &cl, int &lo, int &hi, int *sc, int *mine)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    lo = __reduce_min_sync(0xFFFFFFFFu, lo);
    hi = __reduce_max_sync(0xFFFFFFFFu, hi);
    if (lane == 0) {
        sc[warp] = lo;
        sc[32 + warp] = hi;
    }
    __syncthreads();
    if (warp == 0) {
        const int l = __reduce_min_sync(0xFFFFFFFFu, lane < nw ? sc[lane] : INT_MAX);
        const int h = __reduce_max_sync(0xFFFFFFFFu, lane < nw ? sc[32 + lane] : INT_MIN);
        if (lane == 0) {
            mine[0] = l;
            mine[1] = h;
        }
    }
    cl.sync();
    if (warp == 0) {
        const int C = (int)cl.num_blocks();
        const int *theirs = cl.map_shared_rank(mine, lane < C ? lane : 0);
        const int l = __reduce_min_sync(0xFFFFFFFFu, theirs[0]);
        const int h = __reduce_max_sync(0xFFFFFFFFu, theirs[1]);
        if (lane == 0) {
            sc[0] = l;
            sc[1] = h;
        }
    }
    __syncthreads();
    lo = sc[0];
    hi = sc[1];
}

}  // namespace dev

// Launches `blocks` blocks in clusters of C.
template <typename... P, typename... A>
cudaError_t launch_clusters(void (*kernel)(P...), int C, int blocks, int threads, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return launch_result(cudaLaunchKernelEx(&cfg, kernel, (P)args...));
}

}  // namespace pa
