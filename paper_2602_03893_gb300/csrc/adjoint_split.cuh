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

// CTAs that share a tile's sensors, a power of two up to 8: doubled while the CTAs stay within a wave of `ctas` per SM and
// keep `least` sensors each (idle SMs), and while they stay within some waves and keep 64.
// rows: the tiles gather the sensors' rows of a table through L1, and CTAs that walk the sensors in the same order share
// them there.  Such grids are split only where unsplit they are less than a wave, up to four waves.  The amplitude
// adjoint with 1, 2, 4 and 8 CTAs a tile: 16 bricks, 128 sensors: 74 us with 1, 17 us with 8; 675 bricks, 952
// sensors: 609, 600, 441, 370 us; 1024 bricks, 512 sensors: 337, 316, 305, 279 us; but 3900 bricks, 47 sensors: 76 us
// with 1, 154 with 4, 241 with 8.  Without such rows up to 16 waves, for the last wave's sake: the gradient step
// of 1024 tiles of free centres and 512 sensors 3498, 3435, 3424, 3413 us.
inline int adj_split(int64_t ntiles, int Nd, int ctas, int least, bool rows) {
    const int64_t wave = (int64_t)device_sms() * ctas;
    const int64_t most = rows ? (ntiles < wave ? 4 * wave : 0) : 16 * wave;
    int split = 1;
    while (split < 8 && ((ntiles * split * 2 <= wave && Nd >= 2 * least * split) ||
                         (ntiles * split * 2 <= most && Nd >= 128 * split)))
        split *= 2;
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
