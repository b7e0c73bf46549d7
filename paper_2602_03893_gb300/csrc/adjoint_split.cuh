// adjoint_split.cuh -- the sensors of an adjoint's tile divided over the CTAs of a thread-block cluster
// (gridDim.y of them, one cluster per tile).
#pragma once
#include <cooperative_groups.h>

#include "gpair_internal.cuh"

namespace gp {

// Each thread's N sums over the cluster's CTAs, in the order of the ranks, by the first CTA's threads
// (true there, false in the others).  at: which of the tile's sums they are -- every CTA has a thread
// for each, not always the same one.  part: N floats of shared memory per thread.
template <int N>
__device__ __forceinline__ bool split_sum(float (&sum)[N], float* part, int at) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
#pragma unroll
    for (int u = 0; u < N; ++u) part[u * blockDim.x + at] = sum[u];
    cl.sync();
    if (blockIdx.y == 0)
        for (unsigned c = 1; c < gridDim.y; ++c) {
            const float* other = cl.map_shared_rank(part, c);
#pragma unroll
            for (int u = 0; u < N; ++u) sum[u] += other[u * blockDim.x + at];
        }
    cl.sync();                       // the others' shared memory stays until it has been read
    return blockIdx.y == 0;
}

// CTAs that share a tile's sensors: a power of two up to 8, doubled while the grid stays within one wave
// of `ctas` per SM and each CTA keeps at least 4 sensors.  16 bricks and 128 sensors: 74 us for the 16
// CTAs, 40 us for 8 times as many (20 steps of a 16^3 reconstruction 2476 -> 1778 us).  More than a wave
// is not split: CTAs that walk the sensors in the same order share their rows in L1, and 4096 bricks split
// eightfold for an even last wave took the mid workload's two discretised adjoints from 1.4 to 2.1 ms.
inline int adj_split(int64_t ntiles, int Nd, int ctas) {
    int split = 1;
    while (split < 8 && ntiles * split * 2 <= (int64_t)device_sms() * ctas && Nd >= 8 * split) split *= 2;
    return split;
}

template <typename... Args>
inline cudaError_t launch_split(void (*kern)(Args...), unsigned tiles, int split, int threads, size_t smem,
                                cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles, split);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = split;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = split > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}


}  // namespace gp
