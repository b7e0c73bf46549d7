// voxelize.cu -- Eq. (2) (the Gaussian source field p0) sampled at voxel centres, each
// Gaussian truncated to the box |r_a - c_a| <= k sigma on every axis.
//
// Lattice case (Gaussians on the output lattice, shared sigma): the field is A convolved with
// the 1-D taps exp(-(m h)^2 / 2 sigma^2), |m h| <= k sigma, along x, y and z in turn -- one kernel for up
// to six taps a side, three separable gather passes for more (HBM-bound).
// Any other Gaussian set: small boxes of factors are scattered with atomics; larger ones, where they cover the volume
// several times, are gathered by tiles of the volume.  Very large sets, and calls under stream capture, scatter all.
#include <algorithm>

#include "gpair_internal.cuh"

namespace gp {

constexpr int VOX_MAXTAP = 64;

struct Taps {
    int mm;                      // taps m = -mm..mm
    float t[2 * VOX_MAXTAP + 1];
};

// out = in convolved with taps along one axis.  Threads run along x, blocks over (y, z) rows,
// so no voxel index is divided and every tap's loads are coalesced across the warp.
constexpr int VOX_THREADS = 256;
template <int AXIS>
__global__ void __launch_bounds__(VOX_THREADS)
vox_pass_kernel(const float* __restrict__ in, float* __restrict__ out, int nx, int ny, int nz, Taps taps) {
    const int ix = blockIdx.x * VOX_THREADS + threadIdx.x;
    if (ix >= nx) return;
    const int64_t stride = AXIS == 0 ? 1 : (AXIS == 1 ? (int64_t)nx : (int64_t)nx * ny);
    for (int iz = blockIdx.z; iz < nz; iz += gridDim.z)
        for (int iy = blockIdx.y; iy < ny; iy += gridDim.y) {
            const int64_t v = ((int64_t)iz * ny + iy) * nx + ix;
            const int c = AXIS == 0 ? ix : (AXIS == 1 ? iy : iz), n = AXIS == 0 ? nx : (AXIS == 1 ? ny : nz);
            const int lo = max(-taps.mm, -c), hi = min(taps.mm, n - 1 - c);
            float acc = 0.f;
            for (int m = lo; m <= hi; ++m) acc = fmaf(taps.t[m + taps.mm], __ldg(in + v + m * stride), acc);
            out[v] = acc;
        }
}

// The same pass with the tap count fixed at compile time: the 2 MM + 1 loads of a voxel issue
// together (out-of-volume taps load nothing and add fmaf(t, 0, acc) = acc, so the sum is the
// one above, term for term).
template <int AXIS, int MM>
__global__ void __launch_bounds__(VOX_THREADS)
vox_pass_fixed_kernel(const float* __restrict__ in, float* __restrict__ out, int nx, int ny, int nz, Taps taps) {
    const int ix = blockIdx.x * VOX_THREADS + threadIdx.x;
    if (ix >= nx) return;
    const int64_t stride = AXIS == 0 ? 1 : (AXIS == 1 ? (int64_t)nx : (int64_t)nx * ny);
    for (int iz = blockIdx.z; iz < nz; iz += gridDim.z)
        for (int iy = blockIdx.y; iy < ny; iy += gridDim.y) {
            const int64_t v = ((int64_t)iz * ny + iy) * nx + ix;
            const int c = AXIS == 0 ? ix : (AXIS == 1 ? iy : iz), n = AXIS == 0 ? nx : (AXIS == 1 ? ny : nz);
            float val[2 * MM + 1];
#pragma unroll
            for (int m = -MM; m <= MM; ++m)
                val[m + MM] = (unsigned)(c + m) < (unsigned)n ? __ldg(in + v + m * stride) : 0.f;
            float acc = 0.f;
#pragma unroll
            for (int m = 0; m <= 2 * MM; ++m) acc = fmaf(taps.t[m], val[m], acc);
            out[v] = acc;
        }
}

// The y or z pass with VOX_RUN consecutive outputs per thread along the pass axis: they share
// their taps' inputs, so a thread loads VOX_RUN + 2 MM values instead of VOX_RUN (2 MM + 1).
// Each output's sum is the one above, term for term.
constexpr int VOX_RUN = 4;
template <int AXIS, int MM>
__global__ void __launch_bounds__(VOX_THREADS)
vox_pass_run_kernel(const float* __restrict__ in, float* __restrict__ out, int nx, int ny, int nz, Taps taps) {
    static_assert(AXIS == 1 || AXIS == 2, "runs along y or z");
    const int ix = blockIdx.x * VOX_THREADS + threadIdx.x;
    if (ix >= nx) return;
    const int n = AXIS == 1 ? ny : nz;
    const int nruns = (n + VOX_RUN - 1) / VOX_RUN;
    const int64_t stride = AXIS == 1 ? (int64_t)nx : (int64_t)nx * ny;
    // blockIdx.y runs over (run, other axis) pairs, blockIdx.z over the rest when they exceed 65535
    for (int64_t u = blockIdx.y + (int64_t)blockIdx.z * gridDim.y; u < (int64_t)nruns * (AXIS == 1 ? nz : ny);
         u += (int64_t)gridDim.y * gridDim.z) {
        const int run = (int)(u % nruns), other = (int)(u / nruns);
        const int c0 = run * VOX_RUN;
        const int iy = AXIS == 1 ? c0 : other, iz = AXIS == 1 ? other : c0;
        const int64_t v0 = ((int64_t)iz * ny + iy) * nx + ix;
        float val[VOX_RUN + 2 * MM];
#pragma unroll
        for (int k = 0; k < VOX_RUN + 2 * MM; ++k) {
            const int c = c0 - MM + k;
            val[k] = (unsigned)c < (unsigned)n ? __ldg(in + v0 + (int64_t)(k - MM) * stride) : 0.f;
        }
#pragma unroll
        for (int r = 0; r < VOX_RUN; ++r) {
            if (c0 + r >= n) break;
            float acc = 0.f;
#pragma unroll
            for (int m = 0; m <= 2 * MM; ++m) acc = fmaf(taps.t[m], val[r + m], acc);
            out[v0 + (int64_t)r * stride] = acc;
        }
    }
}

// All three passes in one kernel, for taps fixed at compile time.  A CTA owns VF_TX x VF_TY outputs of tz
// planes, four outputs along x to a thread, and marches z through the tz + 2 MM input planes it needs.
// A thread convolves up to two runs of four inputs of the next plane along x (16-byte loads where rows are
// whole vectors) into one of two shared buffers, while it convolves its own outputs of the current
// plane along y from the other; the last 2 MM + 1 such values stay in registers for the sum along z.
// One barrier a plane.  The volume is read once from DRAM and written once (the halos come from L2).
// Each output is the same three sums as the separate passes', in the same order, so the result is the
// same.
//
// Bound by memory.  With one output to a thread, 32 x 8 columns and three barriers a plane it took 50 us
// for 256 x 256 x 128 voxels, 32 us now.
constexpr int VF_TX = 64, VF_TY = 16, VF_THREADS = VF_TX / 4 * VF_TY;

constexpr int vf_ctas(int mm) { return mm <= 3 ? 3 : 2; }       // resident per SM (registers)

// VEC: nx a multiple of 4 and both volumes 16-byte aligned.
template <int MM, bool VEC>
__global__ void __launch_bounds__(VF_THREADS, vf_ctas(MM))
vox_fused_kernel(const float* __restrict__ in, float* __restrict__ out, int nx, int ny, int nz, int tz, Taps taps) {
    constexpr int ROWS = VF_TY + 2 * MM, GX = VF_TX / 4, ITEMS = ROWS * GX;
    constexpr int NI = (ITEMS + VF_THREADS - 1) / VF_THREADS;               // runs of four a thread convolves along x
    constexpr int HV = (MM + 3) / 4, NL = 4 + 8 * HV;                       // vectors of halo a side, values loaded
    constexpr int NR = 2 * MM + 1;
    __shared__ __align__(16) float Sx[2][ROWS][VF_TX];
    const int t = threadIdx.x, gx = t % GX, ty = t / GX;
    const int x0 = blockIdx.x * VF_TX, y0 = blockIdx.y * VF_TY, z0 = blockIdx.z * tz;
    const int64_t plane = (int64_t)nx * ny;
    const int zn = min(tz, nz - z0);
    float pre[NI][NL];
    auto load = [&](int zi) {
#pragma unroll
        for (int u = 0; u < NI; ++u) {
            const int q = t + u * VF_THREADS, y = y0 - MM + q / GX, x = x0 + (q % GX) * 4 - 4 * HV;
            const bool row = q < ITEMS && (unsigned)y < (unsigned)ny && (unsigned)zi < (unsigned)nz;
            const float* src = in + (int64_t)zi * plane + (int64_t)y * nx;
            if (VEC) {
#pragma unroll
                for (int v = 0; v < NL / 4; ++v) {
                    const bool ok = row && (unsigned)(x + 4 * v) < (unsigned)nx;
                    const float4 f = ok ? __ldg(reinterpret_cast<const float4*>(src + x + 4 * v)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    pre[u][4 * v] = f.x; pre[u][4 * v + 1] = f.y; pre[u][4 * v + 2] = f.z; pre[u][4 * v + 3] = f.w;
                }
            } else {
#pragma unroll
                for (int v = 4 * HV - MM; v < 4 * HV + 4 + MM; ++v)
                    pre[u][v] = row && (unsigned)(x + v) < (unsigned)nx ? __ldg(src + x + v) : 0.f;
            }
        }
    };
    auto along_x = [&](int buf) {
#pragma unroll
        for (int u = 0; u < NI; ++u) {
            const int q = t + u * VF_THREADS;
            if (q >= ITEMS) break;
            float o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float acc = 0.f;
#pragma unroll
                for (int m = 0; m < NR; ++m) acc = fmaf(taps.t[m], pre[u][4 * HV - MM + k + m], acc);
                o[k] = acc;
            }
            *reinterpret_cast<float4*>(&Sx[buf][q / GX][(q % GX) * 4]) = make_float4(o[0], o[1], o[2], o[3]);
        }
    };
    float ring[NR][4];                       // ring[NR - 1] is the newest plane's
#pragma unroll
    for (int m = 0; m < NR; ++m)
#pragma unroll
        for (int k = 0; k < 4; ++k) ring[m][k] = 0.f;
    const int xo = x0 + gx * 4, yo = y0 + ty;
    load(z0 - MM);
    along_x(0);
    __syncthreads();
    const int planes = zn + 2 * MM;
#pragma unroll 1
    for (int i = 0; i < planes; ++i) {
        const bool more = i + 1 < planes;
        if (more) load(z0 - MM + i + 1);     // in flight during this plane's sums
#pragma unroll
        for (int m = 0; m < NR - 1; ++m)
#pragma unroll
            for (int k = 0; k < 4; ++k) ring[m][k] = ring[m + 1][k];
#pragma unroll
        for (int k = 0; k < 4; ++k) ring[NR - 1][k] = 0.f;
#pragma unroll
        for (int m = 0; m < NR; ++m) {       // the (x, y)-convolved values of plane z0 - MM + i
            const float4 v = *reinterpret_cast<const float4*>(&Sx[i & 1][ty + m][gx * 4]);
            ring[NR - 1][0] = fmaf(taps.t[m], v.x, ring[NR - 1][0]);
            ring[NR - 1][1] = fmaf(taps.t[m], v.y, ring[NR - 1][1]);
            ring[NR - 1][2] = fmaf(taps.t[m], v.z, ring[NR - 1][2]);
            ring[NR - 1][3] = fmaf(taps.t[m], v.w, ring[NR - 1][3]);
        }
        if (i >= 2 * MM && yo < ny) {        // plane z0 + i - 2 MM has all its z neighbours
            float o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                o[k] = 0.f;
#pragma unroll
                for (int m = 0; m < NR; ++m) o[k] = fmaf(taps.t[m], ring[m][k], o[k]);
            }
            float* dst = out + (int64_t)(z0 + i - 2 * MM) * plane + (int64_t)yo * nx + xo;
            if (VEC) {
                if (xo < nx) *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (xo + k < nx) dst[k] = o[k];
            }
        }
        if (more) along_x((i + 1) & 1);
        __syncthreads();
    }
}

template <int MM>
static void vox_passes_fixed(const float* A, float* vol, float* tmp, const gpair_grid& og, const Taps& taps,
                             dim3 grid, cudaStream_t st) {
    // planes a CTA: as few (but 4) as one wave of CTAs covers the volume with; 32 where the columns alone are more
    // (each CTA reads the 2 MM planes of overlap again)
    const int64_t cols = (int64_t)((og.nx + VF_TX - 1) / VF_TX) * ((og.ny + VF_TY - 1) / VF_TY);
    const int64_t chunks = (int64_t)device_sms() * vf_ctas(MM) / cols;
    const int tz = chunks < 1 ? 32 : (int)std::max<int64_t>(4, (og.nz + chunks - 1) / chunks);
    const dim3 fgrid((og.nx + VF_TX - 1) / VF_TX, (og.ny + VF_TY - 1) / VF_TY, (og.nz + tz - 1) / tz);
    if (fgrid.y <= 65535 && fgrid.z <= 65535) {
        const bool vec = og.nx % 4 == 0 && (((uintptr_t)A | (uintptr_t)vol) & 15) == 0;
        if (vec) vox_fused_kernel<MM, true><<<fgrid, VF_THREADS, 0, st>>>(A, vol, og.nx, og.ny, og.nz, tz, taps);
        else vox_fused_kernel<MM, false><<<fgrid, VF_THREADS, 0, st>>>(A, vol, og.nx, og.ny, og.nz, tz, taps);
        return;
    }
    vox_pass_fixed_kernel<0, MM><<<grid, VOX_THREADS, 0, st>>>(A, vol, og.nx, og.ny, og.nz, taps);
    const int64_t gy = (int64_t)((og.ny + VOX_RUN - 1) / VOX_RUN) * og.nz;
    const int64_t gz = (int64_t)((og.nz + VOX_RUN - 1) / VOX_RUN) * og.ny;
    auto rgrid = [&](int64_t units) {
        const unsigned y = (unsigned)(units < 65535 ? units : 65535);
        const int64_t z = (units + y - 1) / y;
        return dim3(grid.x, y, (unsigned)(z < 65535 ? z : 65535));
    };
    vox_pass_run_kernel<1, MM><<<rgrid(gy), VOX_THREADS, 0, st>>>(vol, tmp, og.nx, og.ny, og.nz, taps);
    vox_pass_run_kernel<2, MM><<<rgrid(gz), VOX_THREADS, 0, st>>>(tmp, vol, og.nx, og.ny, og.nz, taps);
}

// Gaussian i of the set: centre, width and amplitude.
struct VoxG { float A, cx, cy, cz, s; };
__device__ __forceinline__ VoxG vox_gaussian(const GaussDev& g, int64_t i) {
    VoxG q;
    q.A = g.A[i];
    if (g.grid) {
        const int ix = (int)(i % g.nx), iy = (int)((i / g.nx) % g.ny), iz = (int)(i / ((int64_t)g.nx * g.ny));
        q.cx = (float)(g.ox + (ix + 0.5) * (double)g.h);
        q.cy = (float)(g.oy + (iy + 0.5) * (double)g.h);
        q.cz = (float)(g.oz + (iz + 0.5) * (double)g.h);
        q.s = g.sigma;
    } else {
        q.cx = g.cx[i]; q.cy = g.cy[i]; q.cz = g.cz[i]; q.s = g.sg[i];
    }
    return q;
}
__device__ __forceinline__ float vox_half(float k, float s) { return k * s * (1.f + 1e-6f); }
__device__ __forceinline__ float vox_c2(float s) { return -0.72134752044448170368f / (s * s); }

// The voxels [lo, hi] of an axis that the box of a centre c may hold; the ends' own test is exact.
__device__ __forceinline__ int2 vox_range(float c, float half, float o, float inv, int n) {
    return make_int2(max(0, (int)floorf((c - half - o) * inv - 0.5f)), min(n - 1, (int)ceilf((c + half - o) * inv - 0.5f)));
}

// Add A prod_a f_a to the box of voxels within k sigma per axis, voxel by voxel.
__device__ __forceinline__ void vox_scatter_one(const VoxG& q, const gpair_grid& og, float k, float* __restrict__ vol) {
    const float cx = q.cx, cy = q.cy, cz = q.cz;
    const float half = vox_half(k, q.s), c2 = vox_c2(q.s);
    const float inv = 1.f / og.dx;
    const int2 X = vox_range(cx, half, og.ox, inv, og.nx), Y = vox_range(cy, half, og.oy, inv, og.ny),
               Z = vox_range(cz, half, og.oz, inv, og.nz);
    for (int iz = Z.x; iz <= Z.y; ++iz) {
        const float rz = og.oz + (iz + 0.5f) * og.dx - cz;
        if (fabsf(rz) > half) continue;
        const float fz = q.A * ex2_approx(rz * rz * c2);
        for (int iy = Y.x; iy <= Y.y; ++iy) {
            const float ry = og.oy + (iy + 0.5f) * og.dx - cy;
            if (fabsf(ry) > half) continue;
            const float fyz = fz * ex2_approx(ry * ry * c2);
            for (int ix = X.x; ix <= X.y; ++ix) {
                const float rx = og.ox + (ix + 0.5f) * og.dx - cx;
                if (fabsf(rx) > half) continue;
                atomicAdd(&vol[((int64_t)iz * og.ny + iy) * og.nx + ix], fyz * ex2_approx(rx * rx * c2));
            }
        }
    }
}

// One thread per Gaussian: scatter its box into the volume.
__global__ void vox_scatter_kernel(GaussDev g, gpair_grid og, float k, float* __restrict__ vol) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= g.M) return;
    const VoxG q = vox_gaussian(g, i);
    if (q.A == 0.f) return;
    vox_scatter_one(q, og, k, vol);
}

// ------------------------------------------------------------------------------------------
// The same sum, the large boxes by gathering.  The scatter costs an exponential and an L2 atomic per voxel of a box
// (about 230 G atomics/s), a thread a box; a tile of 8^3 voxels costs a Gaussian that reaches it 24 exponentials and 512
// FMAs, and every tile costs microseconds of finding them.  So boxes of up to VOX_SMALL voxels are scattered by a thread
// each, and the others are taken by tiles or scattered by a warp each, whichever vox_tile_us says is faster.  Only the
// device knows the widths, so every launch after the first two looks at the counts and leaves when it has nothing to do:
//   vox_clear_kernel   the volume and the counts are zero
//   vox_split_kernel   a thread to a Gaussian: small boxes scattered, the others listed and counted by cells (32 an axis)
//   vox_place_kernel   the listed ones in the cells' Morton order, for compact groups
//   vox_boxes_kernel   a bounding box for every 32 and every 1024 of them
//   vox_tile_kernel    the tiles, or a warp to each listed box
// Small sets in small volumes (VOX_DIRECT_*) take one launch: the tiles, with the set itself for the prepared entries.
// A Gaussian with a value that is not finite is scattered, whatever its box: the outer product of a tile would carry it
// to voxels outside.
//
// A tile is a CTA's, whose warps keep the whole of it in registers (16 voxels a lane: x = lane % 8, two rows of y, eight
// planes of z) and share the Gaussians that reach it; the warps' tiles are added in shared memory and every voxel is
// written once.  Finding them: the warps share the test of the boxes of 1024, then each goes down through the ones that
// meet the tile, testing 32 boxes at a time, one to a lane; the entries found wait in the warp's queue until 32 are
// there, one to a lane for the factors.
//
// Bound by FMA issue and shared-memory reads, no longer by the L2's atomics: 262,144 Gaussians of 6 to 24 voxels a side
// into 128^3 took 3992 us as a scatter (857 M atomics) and take 305.  Microseconds with a thread's scatter for every box,
// with tiles for every box of sorted sets, and now (side of the volume, Gaussians, mean side of their boxes):
//   128  262144  8   643  195  169        256    1000  6    57   231   26        512  100000  2     95   1924   101
//   128  262144 18  7300  456  453        256  100000  2    21   325   27        512  100000  6    532   2063   478
//    64    4096 12   267   29   21        256  100000  8   296   385  195        512  100000 30  53157   3047  3222
//   128  100000  2    16  100   21        256 1000000  2    51  1057   59        512 4000000  2    579  23025   585
//   128 1000000  6  1022  438  349        256 1000000 12  8025  1616 1229        512 4000000  8  29146  24401 27670
// The sets of two-voxel boxes pay for the three launches that leave, 6 to 9 us.
//
// In thin sets of many (VOX_THIN: under 64 Gaussians a tile) in volumes of over VOX_THIN_TILES tiles, boxes of up to
// VOX_SMALL_THIN voxels are scattered: 100,000 Gaussians of 6 voxels a side into 256^3 take 141 us, listed 395.
//
// The scatter takes all of sets whose prepared entries would need more than about 0.8 GB (VOX_TILE_MAX) and where
// Gaussians crowd the voxels (more than VOX_TILE_PER_VOXEL each): there are too few tiles then to fill the chip, and
// boxes are a few voxels; and of lattices whose one width makes it the faster way.
constexpr int64_t VOX_TILE_MAX = (int64_t)1 << 24;
constexpr int64_t VOX_TILE_PER_VOXEL = 8;
constexpr int VOX_SMALL = 64, VOX_SMALL_THIN = 343, VOX_THIN = 64;
constexpr int64_t VOX_THIN_M = 32768, VOX_THIN_TILES = 8192;
constexpr int64_t VOX_DIRECT_M = 4096, VOX_DIRECT_TILES = 4096, VOX_DIRECT_TESTS = (int64_t)1 << 21;
constexpr int VT = 8;                         // tile side, voxels
constexpr int VT_N = VT * VT * VT;
constexpr int VT_WARPS = 8, VT_CTAS = 4;      // warps of a CTA, CTAs per SM
constexpr int VT_ROW = 28;                    // factor row of one Gaussian: x 0-7, y 8-15 as (y, y + 4) pairs,
                                              // z 16-23, 4 words of padding (conflict-free 16-byte stores)
constexpr int VT_GROUP = 32, VT_SUPER = 1024;
constexpr float VT_MARGIN = 0.25f;            // voxels by which the boxes exceed the exact test of a factor
constexpr int VC_BITS = 5, VC_SIDE = 1 << VC_BITS;        // cells of the volume, an axis
constexpr int VC_CELLS = VC_SIDE * VC_SIDE * VC_SIDE, VC_BLOCKS = VC_CELLS / 8;      // and blocks of eight of them
constexpr int VC_THREADS = 256, VC_PLACE = 1024;

// Programmatic launches: the two kernels after the split start before the one ahead of them ends and wait here for its
// results, so that they cost no launch gap where they find nothing to do.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

struct VoxCounts {
    unsigned long long voxels;                // of the listed boxes
    unsigned count;                           // listed Gaussians
    alignas(16) int cell[VC_CELLS];           // listed per cell, in Morton order
    int taken[VC_CELLS];                      // and placed so far
};
struct VoxBox { float lo[3], hi[3], pad[2]; };          // 32 bytes, two 16-byte loads
// Microseconds that the tiles take for c boxes of v voxels, and the rates that they are weighed against: fits to 240 sets
// of 1 to 4,000,000 boxes of 5 to 30 voxels a side in 32^3 to 512^3 voxels, each with both, that choose the faster one
// or one within a third of it but for boxes crowded in a part of the volume (2.6 times).
__host__ __device__ __forceinline__ float vox_tile_us(float nt, float c, float v) {
    const float r = (cbrtf(v / c) + VT - 1) / VT;       // tiles that a box reaches, along an axis
    return nt * 2.8e-3f + c * 1.2e-4f + c * r * r * r * 5.9e-5f + nt * c * 1.5e-8f;
}
constexpr float VOX_US_L2 = 2.3e-6f, VOX_US_DRAM = 5.3e-6f;      // a voxel of a warp's scatter, volumes in L2 and beyond
constexpr float VOX_US_LATTICE = 1.25e-6f;                      // of a lattice's, whose threads' atomics coincide

struct VoxSet {                               // scratch
    VoxCounts* n;
    int* list;                                // the listed Gaussians, in no particular order
    float4* u;                                // in place: centre and half width in voxel units (half width < 0: none)
    float4* c;                                // centre, k sigma
    float2* w;                                // amplitude, -1 / (2 sigma^2 ln 2)
    VoxBox *gbox, *sbox;                      // per 32 and per 1024 entries
    float nt, per_voxel;                      // tiles of the volume, microseconds a voxel of a warp's scatter
    // Whether the tiles take the listed boxes.
    __device__ __forceinline__ bool tiles() const {
        const float c = (float)n->count, v = (float)n->voxels;
        return vox_tile_us(nt, c, v) < v * per_voxel + c * 7e-4f + v / c * 3e-3f;
    }
};

__global__ void vox_clear_kernel(float* __restrict__ vol, int64_t n, int* __restrict__ counts, int nc) {
    const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = first; i < n; i += step) vol[i] = 0.f;
    for (int64_t i = first; i < nc; i += step) counts[i] = 0;
}

// Finite in voxel units too, in which the tiles look for it.
__device__ __forceinline__ bool vox_finite(const VoxG& q, const gpair_grid& og, float half, float c2) {
    const float inv = 1.f / og.dx;
    return isfinite(q.A) && isfinite(half * inv) && isfinite(c2) && isfinite((q.cx - og.ox) * inv) &&
           isfinite((q.cy - og.oy) * inv) && isfinite((q.cz - og.oz) * inv);
}

__device__ __forceinline__ int vox_cell(const VoxG& q, const gpair_grid& og) {
    const float inv = 1.f / og.dx;
    const float u[3] = {(q.cx - og.ox) * inv, (q.cy - og.oy) * inv, (q.cz - og.oz) * inv};
    const int n[3] = {og.nx, og.ny, og.nz};
    int r = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float side = (float)max(VT / 2, (n[a] + VC_SIDE - 1) / VC_SIDE);
        const int c = (int)fminf(fmaxf(u[a] / side, 0.f), (float)(VC_SIDE - 1));
#pragma unroll
        for (int b = 0; b < VC_BITS; ++b) r |= (c >> b & 1) << (3 * b + a);
    }
    return r;
}

__global__ void __launch_bounds__(VC_THREADS)
vox_split_kernel(GaussDev g, gpair_grid og, float k, float small, float* __restrict__ vol, VoxSet V) {
    __shared__ unsigned wn[VC_THREADS / 32], wv[VC_THREADS / 32], base;
    const int64_t i = blockIdx.x * (int64_t)VC_THREADS + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    VoxG q = {};
    if (i < g.M) q = vox_gaussian(g, i);
    unsigned voxels = 0;                      // of a box to be listed
    if (q.A != 0.f) {
        const float half = vox_half(k, q.s), inv = 1.f / og.dx, side = 2.f * half * inv;
        // a large box that the volume cuts is listed too: a thread would walk its face alone
        if (side * side * side > small && vox_finite(q, og, half, vox_c2(q.s))) {
            const int2 X = vox_range(q.cx, half, og.ox, inv, og.nx), Y = vox_range(q.cy, half, og.oy, inv, og.ny),
                       Z = vox_range(q.cz, half, og.oz, inv, og.nz);
            const float w = min((float)(X.y - X.x + 1), side), h = min((float)(Y.y - Y.x + 1), side),
                        d = min((float)(Z.y - Z.x + 1), side);
            if (w > 0.f && h > 0.f && d > 0.f) voxels = (unsigned)fminf(fmaxf(w * h * d, 1.f), 16777216.f);
            q.A = 0.f;                        // not for the scatter
        }
    }
    const unsigned listed = __ballot_sync(0xffffffffu, voxels > 0);
    const unsigned sum = __reduce_add_sync(0xffffffffu, voxels);
    if (lane == 0) { wn[warp] = __popc(listed); wv[warp] = sum; }
    if (__syncthreads_or(listed != 0)) {
        if (threadIdx.x == 0) {               // one place for the block, the warps' parts of it after another
            unsigned n = 0;
            unsigned long long v = 0;
            for (int w = 0; w < VC_THREADS / 32; ++w) {
                const unsigned m = wn[w];
                wn[w] = n;
                n += m;
                v += wv[w];
            }
            base = atomicAdd(&V.n->count, n);
            atomicAdd(&V.n->voxels, v);
        }
        __syncthreads();
        if (voxels) {
            V.list[base + wn[warp] + __popc(listed & ((1u << lane) - 1u))] = (int)i;
            atomicAdd(&V.n->cell[vox_cell(q, og)], 1);
        }
    }
    // last: with anything after it, the warps' lanes would wait for one another at the ends of the loops (4,000,000 boxes of
    // two voxels a side: 187 us, 150 like this)
    if (q.A != 0.f) vox_scatter_one(q, og, k, vol);
}

__global__ void __launch_bounds__(VC_PLACE)
vox_place_kernel(GaussDev g, gpair_grid og, float k, VoxSet V) {
    grid_launch_next();
    grid_wait();
    const unsigned count = V.n->count;
    if (count == 0 || !V.tiles()) return;
    // where each block of cells begins: every CTA sums the counts for itself
    __shared__ int first[VC_BLOCKS];
    __shared__ int wsum[VC_PLACE / 32];
    constexpr int PER = VC_BLOCKS / VC_PLACE;
    const int t = threadIdx.x, lane = t & 31;
    int c[PER], mine = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int4* p = reinterpret_cast<const int4*>(V.n->cell + (t * PER + q) * 8);
        const int4 a = p[0], b = p[1];
        c[q] = a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
        mine += c[q];
    }
    int x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += u;
    }
    if (lane == 31) wsum[t >> 5] = x;
    __syncthreads();
    int start = x - mine;
    for (int w = 0; w < t >> 5; ++w) start += wsum[w];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        first[t * PER + q] = start;
        start += c[q];
    }
    __syncthreads();
    const unsigned whole = (count + VT_SUPER - 1) / VT_SUPER * VT_SUPER;
    for (unsigned e = blockIdx.x * VC_PLACE + t; e < whole; e += gridDim.x * VC_PLACE) {
        if (e >= count) {                     // the last super's rest
            V.u[e] = make_float4(0.f, 0.f, 0.f, -INFINITY);
            continue;
        }
        const VoxG q = vox_gaussian(g, V.list[e]);
        const float half = vox_half(k, q.s), inv = 1.f / og.dx;
        const int cell = vox_cell(q, og);
        int at = first[cell >> 3] + atomicAdd(&V.n->taken[cell], 1);
        for (int b = cell & ~7; b < cell; ++b) at += V.n->cell[b];
        V.u[at] = make_float4((q.cx - og.ox) * inv - 0.5f, (q.cy - og.oy) * inv - 0.5f, (q.cz - og.oz) * inv - 0.5f,
                              half * inv + VT_MARGIN);
        V.c[at] = make_float4(q.cx, q.cy, q.cz, half);
        V.w[at] = make_float2(q.A, vox_c2(q.s));
    }
}

__global__ void __launch_bounds__(VT_SUPER)
vox_boxes_kernel(VoxSet V) {
    grid_wait();
    const unsigned count = V.n->count;
    if (count == 0 || !V.tiles()) return;
    __shared__ float sb[6][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (unsigned s = blockIdx.x; s < (count + VT_SUPER - 1) / VT_SUPER; s += gridDim.x) {
        const unsigned e = s * VT_SUPER + threadIdx.x;
        const float4 u = V.u[e];
        float b[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
        if (u.w >= 0.f) {
            b[0] = u.x - u.w; b[1] = u.y - u.w; b[2] = u.z - u.w;
            b[3] = u.x + u.w; b[4] = u.y + u.w; b[5] = u.z + u.w;
        }
        auto join = [&] {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    const float v = __shfl_xor_sync(0xffffffffu, b[q], o);
                    b[q] = q < 3 ? fminf(b[q], v) : fmaxf(b[q], v);
                }
        };
        auto store = [&](VoxBox* p) {
            reinterpret_cast<float4*>(p)[0] = make_float4(b[0], b[1], b[2], b[3]);
            reinterpret_cast<float2*>(p)[2] = make_float2(b[4], b[5]);
        };
        join();
        if (lane == 0) {
            store(V.gbox + e / VT_GROUP);
#pragma unroll
            for (int q = 0; q < 6; ++q) sb[q][warp] = b[q];
        }
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int q = 0; q < 6; ++q) b[q] = sb[q][lane];
            join();
            if (lane == 0) store(V.sbox + s);
        }
        __syncthreads();
    }
}

// A warp to a box: the lanes along x, rows and planes in turn; the factors and their products as vox_scatter_one's.
__device__ __forceinline__ void vox_scatter_warp(const VoxG& q, const gpair_grid& og, float k, int lane, float* __restrict__ vol) {
    const float half = vox_half(k, q.s), c2 = vox_c2(q.s), inv = 1.f / og.dx;
    const int2 X = vox_range(q.cx, half, og.ox, inv, og.nx), Y = vox_range(q.cy, half, og.oy, inv, og.ny),
               Z = vox_range(q.cz, half, og.oz, inv, og.nz);
    const int64_t wx = X.y - X.x + 1, wy = Y.y - Y.x + 1;
    for (int64_t p = lane; p < wx * wy; p += 32) {        // this lane's columns of the box
        const int iy = Y.x + (int)(p / wx), ix = X.x + (int)(p % wx);
        const float ry = og.oy + (iy + 0.5f) * og.dx - q.cy, rx = og.ox + (ix + 0.5f) * og.dx - q.cx;
        if (fabsf(ry) > half || fabsf(rx) > half) continue;
        const float fy = ex2_approx(ry * ry * c2), fx = ex2_approx(rx * rx * c2);
        for (int iz = Z.x; iz <= Z.y; ++iz) {
            const float rz = og.oz + (iz + 0.5f) * og.dx - q.cz;
            if (fabsf(rz) > half) continue;
            atomicAdd(&vol[((int64_t)iz * og.ny + iy) * og.nx + ix], q.A * ex2_approx(rz * rz * c2) * fy * fx);
        }
    }
}

// DIRECT: the set itself in place of the prepared entries (V unused), every voxel of the volume is written: one launch.
template <bool DIRECT>
__global__ void __launch_bounds__(VT_WARPS * 32, VT_CTAS)
vox_tile_kernel(GaussDev g, gpair_grid og, float k, VoxSet V, int ntx, int nty, int ntiles, float* __restrict__ vol) {
    __shared__ __align__(16) float F[VT_WARPS][VT_GROUP * VT_ROW];
    __shared__ int queue[VT_WARPS][2 * VT_GROUP];
    __shared__ uint32_t sups[DIRECT ? 1 : VOX_TILE_MAX / VT_SUPER / 32];
    static_assert(VT_GROUP * VT_ROW >= VT_N, "the warps' tiles take the factors' place at the end");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned count = 0;
    if constexpr (!DIRECT) {
        count = V.n->count;
        if (count == 0) return;
        if (!V.tiles()) {
            for (unsigned e = blockIdx.x * VT_WARPS + warp; e < count; e += gridDim.x * VT_WARPS)
                vox_scatter_warp(vox_gaussian(g, V.list[e]), og, k, lane, vol);
            return;
        }
    }
    float* Fw = F[warp];
    int* qw = queue[warp];
    const uint32_t lt = (1u << lane) - 1u;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
        const int x0 = tx * VT, y0 = ty * VT, z0 = tz * VT;
        const float tlo[3] = {(float)x0, (float)y0, (float)z0};
        const float thi[3] = {(float)(x0 + VT - 1), (float)(y0 + VT - 1), (float)(z0 + VT - 1)};
        auto meets = [&](const VoxBox* p) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(p));
            const float2 h = __ldg(reinterpret_cast<const float2*>(p) + 2);
            return a.x <= thi[0] && a.y <= thi[1] && a.z <= thi[2] && a.w >= tlo[0] && h.x >= tlo[1] && h.y >= tlo[2];
        };
        auto reaches = [&](float4 u) {        // centre and half width in voxel units
            return u.x - u.w <= thi[0] && u.y - u.w <= thi[1] && u.z - u.w <= thi[2] && u.x + u.w >= tlo[0] &&
                   u.y + u.w >= tlo[1] && u.z + u.w >= tlo[2];
        };
        // acc[p][r]: planes 2p and 2p + 1 of row y = lane / 8 + 4 r
        float2 acc[VT / 2][2];
#pragma unroll
        for (int p = 0; p < VT / 2; ++p) acc[p][0] = acc[p][1] = make_float2(0.f, 0.f);

        // the first n (<= 32) entries of the queue: factors by the lanes, then their outer products
        auto batch = [&](int n) {
            if (lane < n) {
                const int e = qw[lane];
                float4 c;
                float2 w;
                if constexpr (DIRECT) {
                    const VoxG q = vox_gaussian(g, e);
                    c = make_float4(q.cx, q.cy, q.cz, vox_half(k, q.s));
                    w = make_float2(q.A, vox_c2(q.s));
                } else {
                    c = __ldg(V.c + e);
                    w = __ldg(V.w + e);
                }
                float f[3 * VT];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const float o = q == 0 ? og.ox : (q == 1 ? og.oy : og.oz), cc = q == 0 ? c.x : (q == 1 ? c.y : c.z);
                    const int i0 = q == 0 ? x0 : (q == 1 ? y0 : z0);
#pragma unroll
                    for (int m = 0; m < VT; ++m) {
                        const float r = o + ((float)(i0 + m) + 0.5f) * og.dx - cc;
                        const float v = fabsf(r) <= c.w ? ex2_approx(r * r * w.y) : 0.f;
                        f[q * VT + (q == 1 ? (m & 3) * 2 + (m >> 2) : m)] = q == 2 ? w.x * v : v;
                    }
                }
                float4* row = reinterpret_cast<float4*>(Fw + lane * VT_ROW);
#pragma unroll
                for (int m = 0; m < 3 * VT / 4; ++m) row[m] = make_float4(f[4 * m], f[4 * m + 1], f[4 * m + 2], f[4 * m + 3]);
            }
            __syncwarp();
#pragma unroll 4
            for (int j = 0; j < n; ++j) {
                const float* row = Fw + j * VT_ROW;
                const float fx = row[lane & 7];
                const float2 fy = *reinterpret_cast<const float2*>(row + VT + 2 * (lane >> 3));
                const float4 za = *reinterpret_cast<const float4*>(row + 2 * VT), zb = *reinterpret_cast<const float4*>(row + 2 * VT + 4);
                const float w0 = fx * fy.x, w1 = fx * fy.y;
                const float2 W0 = make_float2(w0, w0), W1 = make_float2(w1, w1);
                const float2 z[4] = {make_float2(za.x, za.y), make_float2(za.z, za.w), make_float2(zb.x, zb.y), make_float2(zb.z, zb.w)};
#pragma unroll
                for (int p = 0; p < VT / 2; ++p) {
                    acc[p][0] = __ffma2_rn(z[p], W0, acc[p][0]);
                    acc[p][1] = __ffma2_rn(z[p], W1, acc[p][1]);
                }
            }
            __syncwarp();
        };
        int qn = 0;
        bool found = false;
        auto take = [&](int e, bool hit) {    // entry e of this lane into the queue
            const uint32_t hm = __ballot_sync(0xffffffffu, hit);
            if (hit) qw[qn + __popc(hm & lt)] = e;
            qn += __popc(hm);
            __syncwarp();
            if (qn >= VT_GROUP) {
                found = true;
                batch(VT_GROUP);
                qn -= VT_GROUP;
                const int rest = lane < qn ? qw[VT_GROUP + lane] : 0;
                __syncwarp();
                if (lane < qn) qw[lane] = rest;
                __syncwarp();
            }
        };
        if constexpr (DIRECT) {
            const float inv = 1.f / og.dx;
            for (int e0 = warp * 32; e0 < g.M; e0 += VT_WARPS * 32) {
                const int e = e0 + lane;
                VoxG q = {};
                if (e < g.M) q = vox_gaussian(g, e);
                const float half = vox_half(k, q.s);
                const bool odd = q.A != 0.f && !vox_finite(q, og, half, vox_c2(q.s));
                const float4 u = make_float4((q.cx - og.ox) * inv - 0.5f, (q.cy - og.oy) * inv - 0.5f,
                                             (q.cz - og.oz) * inv - 0.5f, half * inv + VT_MARGIN);
                take(e, q.A != 0.f && !odd && half >= 0.f && reaches(u));
                // values that are not finite, voxel by voxel as the scatter has them
                for (uint32_t om = __ballot_sync(0xffffffffu, odd); om; om &= om - 1) {
                    const VoxG o = vox_gaussian(g, e0 + __ffs(om) - 1);
                    const float oh = vox_half(k, o.s), c2 = vox_c2(o.s);
                    const int2 X = vox_range(o.cx, oh, og.ox, inv, og.nx), Y = vox_range(o.cy, oh, og.oy, inv, og.ny),
                               Z = vox_range(o.cz, oh, og.oz, inv, og.nz);
                    const int ix = x0 + (lane & 7);
                    const float rx = og.ox + (ix + 0.5f) * og.dx - o.cx;
                    if (ix < X.x || ix > X.y || fabsf(rx) > oh) continue;
#pragma unroll
                    for (int v = 0; v < 16; ++v) {
                        const int iy = y0 + (lane >> 3) + 4 * (v & 1), iz = z0 + (v >> 1);
                        const float ry = og.oy + (iy + 0.5f) * og.dx - o.cy, rz = og.oz + (iz + 0.5f) * og.dx - o.cz;
                        if (iy < Y.x || iy > Y.y || iz < Z.x || iz > Z.y || fabsf(ry) > oh || fabsf(rz) > oh) continue;
                        const float t = o.A * ex2_approx(rz * rz * c2) * ex2_approx(ry * ry * c2) * ex2_approx(rx * rx * c2);
                        float2& to = acc[v >> 2][v & 1];
                        if (v >> 1 & 1) to.y += t; else to.x += t;
                    }
                }
                __syncwarp();
            }
        } else {
            // the supers that reach the tile, a bit each, 32 to a warp's test
            const int ns = (int)((count + VT_SUPER - 1) / VT_SUPER), nw = (ns + 31) / 32;
            for (int w = warp; w < nw; w += VT_WARPS) {
                const int sl = 32 * w + lane;
                const uint32_t m = __ballot_sync(0xffffffffu, sl < ns && meets(V.sbox + min(sl, ns - 1)));
                if (lane == 0) sups[w] = m;
            }
            __syncthreads();
            int turn = 0;
            for (int w = 0; w < nw; ++w) {
                uint32_t sm = sups[w];
                while (sm) {
                    const int sup = 32 * w + __ffs(sm) - 1;
                    sm &= sm - 1;
                    uint32_t gm = __ballot_sync(0xffffffffu, meets(V.gbox + (int64_t)sup * (VT_SUPER / VT_GROUP) + lane));
                    while (gm) {                   // the groups in turn to the warps
                        const int grp = __ffs(gm) - 1;
                        gm &= gm - 1;
                        if ((turn++ & (VT_WARPS - 1)) != warp) continue;
                        const int e = sup * VT_SUPER + grp * VT_GROUP + lane;
                        take(e, reaches(__ldg(V.u + e)));
                    }
                }
            }
        }
        if (qn) batch(qn);
        // no Gaussian reaches the tile: its voxels have what the scatter left them
        if (!DIRECT && !__syncthreads_or(found || qn)) continue;

        // this warp's tile in place of its factors: voxel (z, y, x) at z * 64 + y * 8 + x
#pragma unroll
        for (int p = 0; p < VT / 2; ++p)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                Fw[(2 * p) * 64 + r * 32 + lane] = acc[p][r].x;
                Fw[(2 * p + 1) * 64 + r * 32 + lane] = acc[p][r].y;
            }
        __syncthreads();
#pragma unroll
        for (int v = threadIdx.x; v < VT_N; v += VT_WARPS * 32) {
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < VT_WARPS; ++q) s += F[q][v];
            const int x = x0 + (v & 7), y = y0 + ((v >> 3) & 7), z = z0 + (v >> 6);
            if (x < og.nx && y < og.ny && z < og.nz) {
                float* to = vol + ((int64_t)z * og.ny + y) * og.nx + x;
                if (DIRECT) *to = s;
                else atomicAdd(to, s);            // one writer; an add that nothing waits for
            }
        }
        __syncthreads();                     // the tile has been read
    }
}

static int vox_blocks(int64_t n) {
    int64_t b = (n + 255) / 256;
    if (b > (int64_t)device_sms() * 32) b = (int64_t)device_sms() * 32;
    return (int)(b < 1 ? 1 : b);
}

bool vox_is_lattice(const GaussDev& g, const gpair_grid& og) {
    return g.grid && og.nx == g.nx && og.ny == g.ny && og.nz == g.nz && og.dx == g.h &&
           (double)og.ox == g.ox && (double)og.oy == g.oy && (double)og.oz == g.oz;
}

// Entries that the tile path has room for, in whole supers.
static int64_t vox_entries(const GaussDev& g) { return (g.M + VT_SUPER - 1) / VT_SUPER * VT_SUPER; }

static int64_t vox_tiles(const gpair_grid& og) {
    return (int64_t)((og.nx + VT - 1) / VT) * ((og.ny + VT - 1) / VT) * ((og.nz + VT - 1) / VT);
}

constexpr int64_t VOX_L2 = 100 << 20;       // bytes of a volume that L2 holds
constexpr size_t VOX_COUNTS = (sizeof(VoxCounts) + 255) & ~(size_t)255;

// Small sets in small volumes go to the tiles as they are.
static bool vox_direct(const GaussDev& g, const gpair_grid& og) {
    const int64_t nt = vox_tiles(og);
    return g.M <= VOX_DIRECT_M && nt <= VOX_DIRECT_TILES && g.M * nt <= VOX_DIRECT_TESTS;
}

// Scratch of the tile path, 0: the scatter takes the call, or the tiles without any.
size_t vox_tile_bytes(const GaussDev& g, const gpair_grid& og, float k) {
    const int64_t n = vox_entries(g), nt = vox_tiles(og);
    if (vox_direct(g, og) || n > VOX_TILE_MAX || nt > INT32_MAX / 2 || n > VOX_TILE_PER_VOXEL * (nt * VT_N)) return 0;
    if (g.grid) {                             // one width: the host knows
        const double side = 2.0 * (double)k * g.sigma / og.dx, v = side * side * side;
        if (v <= VOX_SMALL || v * g.M * VOX_US_LATTICE < vox_tile_us((float)nt, (float)g.M, (float)(v * g.M))) return 0;
    }
    return VOX_COUNTS + (size_t)n * 44 + (size_t)(n / VT_GROUP + n / VT_SUPER) * sizeof(VoxBox);
}

static cudaError_t launch_vox_tiles(const GaussDev& g, const gpair_grid& og, float k, float* vol, void* prep,
                                    cudaStream_t st) {
    const int64_t n = vox_entries(g), ng = n / VT_GROUP, ns = n / VT_SUPER, nv = (int64_t)og.nx * og.ny * og.nz;
    VoxSet V;
    V.n = static_cast<VoxCounts*>(prep);
    V.u = reinterpret_cast<float4*>(static_cast<char*>(prep) + VOX_COUNTS);
    V.c = V.u + n;
    V.gbox = reinterpret_cast<VoxBox*>(V.c + n);
    V.sbox = V.gbox + ng;
    V.w = reinterpret_cast<float2*>(V.sbox + ns);
    V.list = reinterpret_cast<int*>(V.w + n);
    V.nt = (float)vox_tiles(og);
    V.per_voxel = nv * 4 > VOX_L2 ? VOX_US_DRAM : VOX_US_L2;
    vox_clear_kernel<<<vox_blocks(nv), 256, 0, st>>>(vol, nv, reinterpret_cast<int*>(prep), (int)(sizeof(VoxCounts) / 4));
    const int ntx = (og.nx + VT - 1) / VT, nty = (og.ny + VT - 1) / VT, nt = (int)vox_tiles(og);
    const float small = g.M >= VOX_THIN_M && nt > VOX_THIN_TILES && g.M < (int64_t)VOX_THIN * nt ? VOX_SMALL_THIN : VOX_SMALL;
    vox_split_kernel<<<(unsigned)((g.M + VC_THREADS - 1) / VC_THREADS), VC_THREADS, 0, st>>>(g, og, k, small, vol, V);
    cudaError_t e = cudaGetLastError();
    const int64_t sms = device_sms();
    auto launch = [&](auto kern, int64_t ctas, int threads, auto... args) {
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3(threads);
        cfg.stream = st;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, kern, args...);
    };
    launch(vox_place_kernel, std::min<int64_t>((n + VC_PLACE - 1) / VC_PLACE, sms), VC_PLACE, g, og, k, V);
    launch(vox_boxes_kernel, std::min<int64_t>(ns, 2 * sms), VT_SUPER, V);
    // a few CTAs to every place for one, each with tiles a grid apart: they end together and an empty grid is soon gone
    const int64_t ctas = std::min<int64_t>(std::max<int64_t>(nt, (g.M + VT_WARPS - 1) / VT_WARPS), 4 * VT_CTAS * sms);
    // launched in turn: CTAs that start while others still hold some SMs crowd the rest
    if (e == cudaSuccess) vox_tile_kernel<false><<<(unsigned)ctas, VT_WARPS * 32, 0, st>>>(g, og, k, V, ntx, nty, nt, vol);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// tmp: scratch volume of the same size (lattice case); prep: vox_tile_bytes() of scratch (others;
// null: the scatter).
cudaError_t launch_voxelize(const GaussDev& g, const gpair_grid& og, float k, float* vol, float* tmp, void* prep,
                            cudaStream_t st) {
    const int64_t nv = (int64_t)og.nx * og.ny * og.nz;
    if (vox_is_lattice(g, og)) {
        Taps taps;
        const double half = (double)k * g.sigma;
        int mm = (int)floor(half / g.h * (1.0 + 1e-9));
        if (mm > VOX_MAXTAP) return cudaErrorInvalidValue;
        taps.mm = mm;
        for (int m = -mm; m <= mm; ++m) {
            double r = m * (double)g.h;
            taps.t[m + mm] = (float)exp(-r * r / (2.0 * (double)g.sigma * g.sigma));
        }
        const dim3 grid((og.nx + VOX_THREADS - 1) / VOX_THREADS, og.ny < 65535 ? og.ny : 65535,
                        og.nz < 65535 ? og.nz : 65535);
        switch (mm) {
            case 1: vox_passes_fixed<1>(g.A, vol, tmp, og, taps, grid, st); break;
            case 2: vox_passes_fixed<2>(g.A, vol, tmp, og, taps, grid, st); break;
            case 3: vox_passes_fixed<3>(g.A, vol, tmp, og, taps, grid, st); break;
            case 4: vox_passes_fixed<4>(g.A, vol, tmp, og, taps, grid, st); break;
            case 5: vox_passes_fixed<5>(g.A, vol, tmp, og, taps, grid, st); break;
            case 6: vox_passes_fixed<6>(g.A, vol, tmp, og, taps, grid, st); break;
            default:
                vox_pass_kernel<0><<<grid, VOX_THREADS, 0, st>>>(g.A, vol, og.nx, og.ny, og.nz, taps);
                vox_pass_kernel<1><<<grid, VOX_THREADS, 0, st>>>(vol, tmp, og.nx, og.ny, og.nz, taps);
                vox_pass_kernel<2><<<grid, VOX_THREADS, 0, st>>>(tmp, vol, og.nx, og.ny, og.nz, taps);
        }
        return cudaGetLastError();
    }
    if (vox_direct(g, og)) {
        const int ntx = (og.nx + VT - 1) / VT, nty = (og.ny + VT - 1) / VT, nt = (int)vox_tiles(og);
        vox_tile_kernel<true><<<nt, VT_WARPS * 32, 0, st>>>(g, og, k, VoxSet{}, ntx, nty, nt, vol);
        return cudaGetLastError();
    }
    if (prep) return launch_vox_tiles(g, og, k, vol, prep, st);
    vox_clear_kernel<<<vox_blocks(nv), 256, 0, st>>>(vol, nv, nullptr, 0);
    vox_scatter_kernel<<<(unsigned)((g.M + 255) / 256), 256, 0, st>>>(g, og, k, vol);
    return cudaGetLastError();
}

}  // namespace gp
