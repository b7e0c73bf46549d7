// voxelize.cu -- Eq. (2) (the Gaussian source field p0) sampled at voxel centres, each
// Gaussian truncated to the box |r_a - c_a| <= k sigma on every axis.
//
// Lattice case (Gaussians on the output lattice, shared sigma): the field is A convolved with
// the 1-D taps exp(-(m h)^2 / 2 sigma^2), |m h| <= k sigma, along x, y and z in turn -- three
// separable gather passes, each one coalesced read and write of the volume (HBM-bound).
// Any other Gaussian set: tiles of the volume gather the separable boxes of factors of the Gaussians that
// reach them; very large sets, and calls under stream capture, scatter them instead.
#include <algorithm>

#include "gpair_internal.cuh"

namespace gp {

size_t spatial_order_bytes(int64_t M);
cudaError_t launch_spatial_perm(const GaussDev& g, void* scratch, const int** perm, cudaStream_t st);

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

__global__ void zero_kernel(float* p, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = 0.f;
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

// Add A prod_a f_a to the box of voxels within k sigma per axis, voxel by voxel.
__device__ __forceinline__ void vox_scatter_one(const VoxG& q, const gpair_grid& og, float k, float* __restrict__ vol) {
    const float cx = q.cx, cy = q.cy, cz = q.cz;
    const float half = vox_half(k, q.s), c2 = vox_c2(q.s);
    const float inv = 1.f / og.dx;
    const int xa = max(0, (int)floorf((cx - half - og.ox) * inv - 0.5f)), xb = min(og.nx - 1, (int)ceilf((cx + half - og.ox) * inv - 0.5f));
    const int ya = max(0, (int)floorf((cy - half - og.oy) * inv - 0.5f)), yb = min(og.ny - 1, (int)ceilf((cy + half - og.oy) * inv - 0.5f));
    const int za = max(0, (int)floorf((cz - half - og.oz) * inv - 0.5f)), zb = min(og.nz - 1, (int)ceilf((cz + half - og.oz) * inv - 0.5f));
    for (int iz = za; iz <= zb; ++iz) {
        const float rz = og.oz + (iz + 0.5f) * og.dx - cz;
        if (fabsf(rz) > half) continue;
        const float fz = q.A * ex2_approx(rz * rz * c2);
        for (int iy = ya; iy <= yb; ++iy) {
            const float ry = og.oy + (iy + 0.5f) * og.dx - cy;
            if (fabsf(ry) > half) continue;
            const float fyz = fz * ex2_approx(ry * ry * c2);
            for (int ix = xa; ix <= xb; ++ix) {
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
// The same sum by gathering.  The volume is cut into tiles of 8^3 voxels, one CTA each, whose warps
// keep the whole tile in registers (16 voxels a lane: x = lane % 8, two rows of y, eight planes of z)
// and share the Gaussians that reach it; the warps' tiles are added in shared memory and every voxel
// is written once.  A Gaussian costs a tile 24 exponentials (8 per axis, zero outside its box)
// and 512 FMAs of their outer product, against one exponential and one L2 atomic per voxel of its box.
//
// Finding them: the entries come in a spatially compact order (free centres: the Morton order; a
// lattice: its 8 x 8 x 4 bricks), every 32 of them under one bounding box and every 1024 under another,
// in voxel units.  A warp tests 32 boxes at a time, one to a lane, and goes down through the ones
// that meet the tile; the entries found wait in the warp's queue until 32 are there, one to
// a lane for the factors.
//
// Bound by FMA issue and shared-memory reads, no longer by the L2's atomics: 262,144 Gaussians of 3 to
// 24 voxels a side into 128^3 took 3955 us as a scatter (857 M atomics) and take 354 us, 46 of them
// the order.
//
// The scatter stays for sets whose prepared entries would need more than about a gigabyte
// (VOX_TILE_MAX) and where Gaussians crowd the voxels (more than VOX_TILE_PER_VOXEL each): there are
// too few tiles then to fill the chip, and boxes are a few voxels.
constexpr int64_t VOX_TILE_MAX = (int64_t)1 << 24;
constexpr int64_t VOX_TILE_PER_VOXEL = 8;
constexpr int VT = 8;                         // tile side, voxels
constexpr int VT_N = VT * VT * VT;
constexpr int VT_WARPS = 8;
constexpr int VT_ROW = 28;                    // factor row of one Gaussian: x 0-7, y 8-15 as (y, y + 4) pairs,
                                              // z 16-23, 4 words of padding (conflict-free 16-byte stores)
constexpr int VT_GROUP = 32, VT_SUPER = 1024;
constexpr float VT_MARGIN = 0.25f;            // voxels by which the boxes exceed the exact test of a factor

struct VoxBox { float lo[3], hi[3], pad[2]; };          // 32 bytes, two 16-byte loads
struct VoxSet {                               // the prepared entries (scratch)
    float4* u;                                // centre and half width in voxel units (half width < 0: skipped)
    float4* c;                                // centre, k sigma
    float2* w;                                // amplitude, -1 / (2 sigma^2 ln 2)
    VoxBox *gbox, *sbox;                      // per 32 and per 1024 entries
    int* odd;                                 // per 1024 entries: 1 when one of them is not finite
    int64_t n;                                // entries, a multiple of VT_SUPER
};

// Entry e -> Gaussian, -1: none.
__device__ __forceinline__ int64_t vox_entry(const GaussDev& g, const int* perm, int64_t e) {
    if (!g.grid) return e < g.M ? (perm ? perm[e] : e) : -1;
    const int64_t t = e / TILE;
    if (t >= g.ntiles) return -1;
    const int l = (int)(e % TILE);
    const int ix = (int)(t % g.ntx) * BX + (l & (BX - 1)), iy = (int)((t / g.ntx) % g.nty) * BY + ((l / BX) & (BY - 1)),
              iz = (int)(t / ((int64_t)g.ntx * g.nty)) * BZ + l / (BX * BY);
    return ix < g.nx && iy < g.ny && iz < g.nz ? ((int64_t)iz * g.ny + iy) * g.nx + ix : -1;
}

// A Gaussian with a value that is not finite reaches voxels outside its box through the zeros of the
// outer product; these few go voxel by voxel afterwards (vox_odd_kernel).
// So do those whose place in voxel units is not.
__device__ __forceinline__ bool vox_finite(const VoxG& q, const gpair_grid& og, float half, float c2) {
    const float inv = 1.f / og.dx;
    return isfinite(q.A) && isfinite(half * inv) && isfinite(c2) && isfinite((q.cx - og.ox) * inv) &&
           isfinite((q.cy - og.oy) * inv) && isfinite((q.cz - og.oz) * inv);
}

__global__ void __launch_bounds__(VT_SUPER)
vox_prepare_kernel(GaussDev g, gpair_grid og, float k, const int* __restrict__ perm, VoxSet V) {
    __shared__ float sb[6][32];
    const int64_t e = blockIdx.x * (int64_t)VT_SUPER + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = vox_entry(g, perm, e);
    float4 u = make_float4(0.f, 0.f, 0.f, -INFINITY), c = make_float4(0.f, 0.f, 0.f, -1.f);
    float2 w = make_float2(0.f, 0.f);
    float b[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    bool odd = false;
    if (i >= 0) {
        const VoxG q = vox_gaussian(g, i);
        const float half = vox_half(k, q.s), c2 = vox_c2(q.s);
        odd = q.A != 0.f && !vox_finite(q, og, half, c2);
        if (q.A != 0.f && !odd && half >= 0.f) {
            const float inv = 1.f / og.dx;
            u = make_float4((q.cx - og.ox) * inv - 0.5f, (q.cy - og.oy) * inv - 0.5f, (q.cz - og.oz) * inv - 0.5f,
                            half * inv + VT_MARGIN);
            c = make_float4(q.cx, q.cy, q.cz, half);
            w = make_float2(q.A, c2);
            b[0] = u.x - u.w; b[1] = u.y - u.w; b[2] = u.z - u.w;
            b[3] = u.x + u.w; b[4] = u.y + u.w; b[5] = u.z + u.w;
        }
    }
    V.u[e] = u;
    V.c[e] = c;
    V.w[e] = w;
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
    const int any_odd = __syncthreads_or(odd);
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < 6; ++q) b[q] = sb[q][lane];
        join();
        if (lane == 0) {
            store(V.sbox + blockIdx.x);
            V.odd[blockIdx.x] = any_odd;
        }
    }
}

__global__ void __launch_bounds__(VT_WARPS * 32, 4)
vox_tile_kernel(gpair_grid og, VoxSet V, int ntx, int nty, float* __restrict__ vol) {
    __shared__ __align__(16) float F[VT_WARPS][VT_GROUP * VT_ROW];
    __shared__ int queue[VT_WARPS][2 * VT_GROUP];
    static_assert(VT_GROUP * VT_ROW >= VT_N, "the warps' tiles take the factors' place at the end");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tx = blockIdx.x % ntx, ty = (blockIdx.x / ntx) % nty, tz = blockIdx.x / (ntx * nty);
    const int x0 = tx * VT, y0 = ty * VT, z0 = tz * VT;
    const float tlo[3] = {(float)x0, (float)y0, (float)z0};
    const float thi[3] = {(float)(x0 + VT - 1), (float)(y0 + VT - 1), (float)(z0 + VT - 1)};
    auto meets = [&](const VoxBox* p) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(p));
        const float2 h = __ldg(reinterpret_cast<const float2*>(p) + 2);
        return a.x <= thi[0] && a.y <= thi[1] && a.z <= thi[2] && a.w >= tlo[0] && h.x >= tlo[1] && h.y >= tlo[2];
    };
    float* Fw = F[warp];
    int* qw = queue[warp];
    const uint32_t lt = (1u << lane) - 1u;
    // acc[p][r]: planes 2p and 2p + 1 of row y = lane / 8 + 4 r
    float2 acc[VT / 2][2];
#pragma unroll
    for (int p = 0; p < VT / 2; ++p) acc[p][0] = acc[p][1] = make_float2(0.f, 0.f);

    // the first n (<= 32) entries of the queue: factors by the lanes, then their outer products
    auto batch = [&](int n) {
        if (lane < n) {
            const int e = qw[lane];
            const float4 c = __ldg(V.c + e);
            const float2 w = __ldg(V.w + e);
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

    const int ns = (int)(V.n / VT_SUPER);
    int qn = 0, turn = 0;
    for (int s0 = 0; s0 < ns; s0 += 32) {
        uint32_t sm = __ballot_sync(0xffffffffu, s0 + lane < ns && meets(V.sbox + min(s0 + lane, ns - 1)));
        while (sm) {
            const int sup = s0 + __ffs(sm) - 1;
            sm &= sm - 1;
            uint32_t gm = __ballot_sync(0xffffffffu, meets(V.gbox + (int64_t)sup * (VT_SUPER / VT_GROUP) + lane));
            while (gm) {                       // the groups in turn to the warps
                const int grp = __ffs(gm) - 1;
                gm &= gm - 1;
                if ((turn++ & (VT_WARPS - 1)) != warp) continue;
                const int e = sup * VT_SUPER + grp * VT_GROUP + lane;
                const float4 u = __ldg(V.u + e);
                const bool hit = u.x - u.w <= thi[0] && u.y - u.w <= thi[1] && u.z - u.w <= thi[2] &&
                                 u.x + u.w >= tlo[0] && u.y + u.w >= tlo[1] && u.z + u.w >= tlo[2];
                const uint32_t hm = __ballot_sync(0xffffffffu, hit);
                if (hit) qw[qn + __popc(hm & lt)] = e;
                qn += __popc(hm);
                __syncwarp();
                if (qn >= VT_GROUP) {
                    batch(VT_GROUP);
                    qn -= VT_GROUP;
                    const int rest = lane < qn ? qw[VT_GROUP + lane] : 0;
                    __syncwarp();
                    if (lane < qn) qw[lane] = rest;
                    __syncwarp();
                }
            }
        }
    }
    if (qn) batch(qn);

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
        if (x < og.nx && y < og.ny && z < og.nz) vol[((int64_t)z * og.ny + y) * og.nx + x] = s;
    }
}

// The Gaussians that the tiles left out for a value that is not finite.
__global__ void __launch_bounds__(VT_SUPER)
vox_odd_kernel(GaussDev g, gpair_grid og, float k, const int* __restrict__ perm, const int* __restrict__ odd,
               float* __restrict__ vol) {
    if (!odd[blockIdx.x]) return;
    const int64_t i = vox_entry(g, perm, blockIdx.x * (int64_t)VT_SUPER + threadIdx.x);
    if (i < 0) return;
    const VoxG q = vox_gaussian(g, i);
    if (q.A != 0.f && !vox_finite(q, og, vox_half(k, q.s), vox_c2(q.s))) vox_scatter_one(q, og, k, vol);
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

// Entries of the tile path: the Gaussians (a lattice's in whole bricks), in whole supers.
static int64_t vox_entries(const GaussDev& g) {
    const int64_t n = g.grid ? g.ntiles * TILE : g.M;
    return (n + VT_SUPER - 1) / VT_SUPER * VT_SUPER;
}

// Free sets of up to this many Gaussians are not sorted: a tile's 256 threads test every one of them.
constexpr int64_t VOX_SORT_MIN = 4096;

static size_t vox_set_bytes(int64_t n) { return (size_t)n * 40 + (size_t)(n / VT_GROUP + n / VT_SUPER) * sizeof(VoxBox) + (size_t)(n / VT_SUPER) * 4; }

// Scratch of the tile path, 0: the scatter takes the call.
size_t vox_tile_bytes(const GaussDev& g, const gpair_grid& og) {
    const int64_t n = vox_entries(g);
    const int64_t nt = (int64_t)((og.nx + VT - 1) / VT) * ((og.ny + VT - 1) / VT) * ((og.nz + VT - 1) / VT);
    if (n > VOX_TILE_MAX || nt > INT32_MAX || n > VOX_TILE_PER_VOXEL * (nt * VT_N)) return 0;
    return vox_set_bytes(n) + 256 + (!g.grid && g.M > VOX_SORT_MIN ? spatial_order_bytes(g.M) : 0);
}

static cudaError_t launch_vox_tiles(const GaussDev& g, const gpair_grid& og, float k, float* vol, void* prep,
                                    cudaStream_t st) {
    VoxSet V;
    V.n = vox_entries(g);
    const int64_t ng = V.n / VT_GROUP, ns = V.n / VT_SUPER;
    V.u = static_cast<float4*>(prep);
    V.c = V.u + V.n;
    V.gbox = reinterpret_cast<VoxBox*>(V.c + V.n);
    V.sbox = V.gbox + ng;
    V.w = reinterpret_cast<float2*>(V.sbox + ns);
    V.odd = reinterpret_cast<int*>(V.w + V.n);
    const int* perm = nullptr;
    if (!g.grid && g.M > VOX_SORT_MIN) {
        char* so = static_cast<char*>(prep) + ((vox_set_bytes(V.n) + 255) & ~(size_t)255);
        const cudaError_t e = launch_spatial_perm(g, so, &perm, st);
        if (e != cudaSuccess) return e;
    }
    vox_prepare_kernel<<<(unsigned)ns, VT_SUPER, 0, st>>>(g, og, k, perm, V);
    const int ntx = (og.nx + VT - 1) / VT, nty = (og.ny + VT - 1) / VT, ntz = (og.nz + VT - 1) / VT;
    vox_tile_kernel<<<(unsigned)((int64_t)ntx * nty * ntz), VT_WARPS * 32, 0, st>>>(og, V, ntx, nty, vol);
    vox_odd_kernel<<<(unsigned)ns, VT_SUPER, 0, st>>>(g, og, k, perm, V.odd, vol);
    return cudaGetLastError();
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
    if (prep) return launch_vox_tiles(g, og, k, vol, prep, st);
    zero_kernel<<<vox_blocks(nv), 256, 0, st>>>(vol, nv);
    vox_scatter_kernel<<<(unsigned)((g.M + 255) / 256), 256, 0, st>>>(g, og, k, vol);
    return cudaGetLastError();
}

}  // namespace gp
