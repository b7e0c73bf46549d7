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
// keep `least` sensors each (idle SMs), and while they stay within 16 waves and keep 64, for the last wave's sake: the
// gradient step of 1024 tiles of free centres and 512 sensors 3498, 3435, 3424, 3413 us.
inline int adj_split(int64_t ntiles, int Nd, int ctas, int least) {
    const int64_t wave = (int64_t)device_sms() * ctas;
    int split = 1;
    while (split < 8 && ((ntiles * split * 2 <= wave && Nd >= 2 * least * split) ||
                         (ntiles * split * 2 <= 16 * wave && Nd >= 128 * split)))
        split *= 2;
    return split;
}

// The same for the amplitude adjoints of lattices, whose tiles gather the sensors' rows of a table through L1: CTAs that
// walk the sensors in the same order share them there, so that a split costs more than its barrier, and grids that
// fill half of the chip's warps already lose by it.  Microseconds with 1, 2, 4 and 8 CTAs a tile, exact adjoint (the
// discretised one is alike), at the lines of the rule (152 SMs):
//    54 tiles,  128 sensors:   70   43   29   21        768 tiles,  128 sensors:   72   79   70   87
//   150         128            70   41   27   33        768         300           160  172  140  155 (84 100 83 96)
//   288         128            70   43   31   46        768         512           266  290  231  226
//   512         128            69   45   51   62       1024         300           169  176  180  194
//   512        1024           496  295  310  308       1352         512           305  428  365  360
//  1024          33            28   33   45   70       2048        1024           761 1089  965  984
inline int adj_split_rows(int64_t ntiles, int Nd) {
    const int64_t sms = device_sms();
    if (ntiles * 8 <= 4 * sms && Nd >= 64) return 8;
    if (ntiles * 4 <= 8 * sms && Nd >= 32) return 4;
    if (ntiles * 2 <= 8 * sms) return Nd >= 16 ? 2 : 1;
    if (ntiles <= 6 * sms) return Nd >= 512 ? 8 : Nd >= 300 ? 4 : 1;
    return 1;
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
