// metrics.cu -- the image metrics the paper tabulates for reconstructions (Results, Table 1): the
// maximum amplitude projection along z, and MSE / PSNR / SSIM of an image against a reference.
// The paper gives no formulas; the common definitions are used: SSIM (Wang et al., 2004) with a
// uniform window of `win` samples per axis, sample (N / (N - 1)) variances and covariance,
// C1 = (0.01 R)^2, C2 = (0.03 R)^2 for the data range R, averaged over the positions whose window
// lies inside the image.  The local sums are separable box filters (x, then y, then z) of five
// fields (x, y, x^2, y^2, x y): fused for windows up to 9 (ssim_zfirst_kernel) and up to 15
// (ssim_march_kernel), which also sum the squared differences, else one coalesced pass per axis through device memory.
#include "gpair_internal.cuh"

namespace gp {

constexpr int MET_THREADS = 256;
// CTAs of the persistent passes: 4 per SM of the current device.
#define MET_BLOCKS (4 * device_sms())

// A block takes 64 columns, four threads to a column with every fourth plane each, eight planes' loads in
// flight: HBM-bound.  256 x 256 x 128: 8.1 us; 11.5 with one thread to a column, which left half the chip idle.
constexpr int ZM_X = 64, ZM_Z = MET_THREADS / ZM_X;
__global__ void __launch_bounds__(MET_THREADS)
zmap_kernel(const float* __restrict__ vol, int nx, int ny, int nz, float* __restrict__ out) {
    __shared__ float part[ZM_Z][ZM_X];
    const int64_t nxy = (int64_t)nx * ny;
    const int tx = threadIdx.x % ZM_X, tz = threadIdx.x / ZM_X;
    for (int64_t i0 = (int64_t)blockIdx.x * ZM_X; i0 < nxy; i0 += (int64_t)gridDim.x * ZM_X) {
        const int64_t i = i0 + tx;
        float m = __int_as_float(0x7FFFFFFF);      // fmaxf passes a NaN by
        if (i < nxy)
#pragma unroll 8
            for (int z = tz; z < nz; z += ZM_Z) m = fmaxf(m, vol[(int64_t)z * nxy + i]);
        part[tz][tx] = m;
        __syncthreads();
        if (tz == 0 && i < nxy) {
            for (int q = 1; q < ZM_Z; ++q) m = fmaxf(m, part[q][tx]);
            out[i] = m;
        }
        __syncthreads();
    }
}

// Box sums along x of the five fields of (x, y), valid where p <= ix < nx - p.
__global__ void box_x_kernel(const float* __restrict__ a, const float* __restrict__ b, int nx, int ny, int nz, int p,
                             float* __restrict__ S) {
    const int64_t M = (int64_t)nx * ny * nz;
    for (int row = blockIdx.x; row < ny * nz; row += gridDim.x)
        for (int ix = p + threadIdx.x; ix < nx - p; ix += blockDim.x) {
            const int64_t i = (int64_t)row * nx + ix;
            float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, s4 = 0.f;
            for (int d = -p; d <= p; ++d) {
                const float u = a[i + d], v = b[i + d];
                s0 += u; s1 += v; s2 = fmaf(u, u, s2); s3 = fmaf(v, v, s3); s4 = fmaf(u, v, s4);
            }
            S[i] = s0; S[M + i] = s1; S[2 * M + i] = s2; S[3 * M + i] = s3; S[4 * M + i] = s4;
        }
}

// Box sums of the five fields along y (axis 1) or z (axis 2), valid where the window fits on that
// axis (and on the axes summed before).
__global__ void box_yz_kernel(const float* __restrict__ S, int nx, int ny, int nz, int p, int axis,
                              float* __restrict__ T) {
    const int64_t M = (int64_t)nx * ny * nz;
    const int64_t stride = axis == 1 ? nx : (int64_t)nx * ny;
    for (int row = blockIdx.x; row < ny * nz; row += gridDim.x) {
        const int iy = row % ny, iz = row / ny;
        const int c = axis == 1 ? iy : iz, n = axis == 1 ? ny : nz;
        if (c < p || c >= n - p) continue;
        if (axis == 2 && (iy < p || iy >= ny - p)) continue;
        for (int ix = p + threadIdx.x; ix < nx - p; ix += blockDim.x) {
            const int64_t i = (int64_t)row * nx + ix;
            for (int f = 0; f < 5; ++f) {
                float s = 0.f;
                for (int d = -p; d <= p; ++d) s += S[f * M + i + d * stride];
                T[f * M + i] = s;
            }
        }
    }
}

// SSIM at every interior position from the five box sums; FP64 block partials of the sum.
__global__ void __launch_bounds__(MET_THREADS)
ssim_kernel(const float* __restrict__ S, int nx, int ny, int nz, int p, int pz, float invN, float cov, float C1,
            float C2, double* __restrict__ partial) {
    __shared__ double red[MET_THREADS / 32];
    const int64_t M = (int64_t)nx * ny * nz;
    double acc = 0.0;
    for (int row = blockIdx.x; row < ny * nz; row += gridDim.x) {
        const int iy = row % ny, iz = row / ny;
        if (iy < p || iy >= ny - p || iz < pz || iz >= nz - pz) continue;
        for (int ix = p + threadIdx.x; ix < nx - p; ix += blockDim.x) {
            const int64_t i = (int64_t)row * nx + ix;
            const float mx = S[i] * invN, my = S[M + i] * invN;
            const float sxx = cov * (S[2 * M + i] * invN - mx * mx);
            const float syy = cov * (S[3 * M + i] * invN - my * my);
            const float sxy = cov * (S[4 * M + i] * invN - mx * my);
            acc += (double)(((2.f * mx * my + C1) * (2.f * sxy + C2)) / ((mx * mx + my * my + C1) * (sxx + syy + C2)));
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) red[w] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < MET_THREADS / 32; ++k) s += red[k];
        partial[blockIdx.x] = s;
    }
}

__global__ void sum_partials_kernel(const double* __restrict__ partial, int n, double* __restrict__ out) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < n; ++k) s += partial[k];    // fixed order
        *out = s;
    }
}

// Fused MSE + SSIM, marching along z.  A CTA owns a column of SS_TX x SS_TY output positions and
// a chunk of SS_ZC planes.  Per input plane it stages x and y with a p-voxel halo in x and y,
// box-sums the five fields along x (shared memory), then along y for its own positions, and keeps
// the last 2 pz + 1 such planes in a per-thread ring; an output plane's z box sum adds the ring
// in plane order.  The summation order per position is that of the separable passes above (x, y,
// then z), so every position's SSIM is the same FP32 value; only x and y cross HBM.  Per-thread
// sums of (x - y)^2 over the CTA's own voxels and of SSIM over its interior positions are
// compensated FP32, then FP64 per CTA: partial[2 b] and partial[2 b + 1].
constexpr int SS_TX = 32, SS_TY = 8, SS_ZC = 16, SS_PMAX = 7;
// staged entries per thread: (SS_TY + 2 p)(SS_TX + 2 p) <= 22 * 46 = 1012 <= 4 * 256
constexpr int SS_STAGE = ((SS_TY + 2 * SS_PMAX) * (SS_TX + 2 * SS_PMAX) + 255) / 256;
static_assert(SS_TX * SS_TY == MET_THREADS, "one thread per output column position");

__host__ __device__ __forceinline__ size_t ssim_march_floats(int p, int pz) {
    return (size_t)2 * (SS_TY + 2 * p) * (SS_TX + 2 * p) + (size_t)5 * (SS_TY + 2 * p) * SS_TX +
           (size_t)(2 * pz + 1) * 5 * SS_TY * SS_TX;
}

__global__ void __launch_bounds__(MET_THREADS)
ssim_march_kernel(const float* __restrict__ x, const float* __restrict__ y, int nx, int ny, int nz, int p, int pz,
                  float invN, float cov, float C1, float C2, double* __restrict__ partial) {
    extern __shared__ float ssm[];
    __shared__ double red[2][MET_THREADS / 32];
    const int SW = SS_TX + 2 * p, SH = SS_TY + 2 * p, R = 2 * pz + 1;
    float* sa = ssm;                              // [SH][SW]
    float* sb = sa + SH * SW;                     // [SH][SW]
    float* xb = sb + SH * SW;                     // [5][SH][SS_TX]
    float* ring = xb + 5 * SH * SS_TX;            // [R][5][SS_TY][SS_TX]
    const int tx = threadIdx.x % SS_TX, ty = threadIdx.x / SS_TX;
    const int ncx = (nx + SS_TX - 1) / SS_TX, ncy = (ny + SS_TY - 1) / SS_TY, ncz = (nz + SS_ZC - 1) / SS_ZC;
    const int nitems = ncx * ncy * ncz;
    KahanF ksq, kss;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
        const int cx = item % ncx, cy = (item / ncx) % ncy, cz = item / (ncx * ncy);
        const int X0 = cx * SS_TX, Y0 = cy * SS_TY, Z0 = cz * SS_ZC, Z1 = min(Z0 + SS_ZC, nz);
        const int gx = X0 + tx, gy = Y0 + ty;
        const bool own_xy = gx < nx && gy < ny;
        const bool in_xy = gx >= p && gx < nx - p && gy >= p && gy < ny - p;
        const int zlo = max(Z0 - pz, 0), zhi = min(Z1 - 1 + pz, nz - 1);
        // this thread's staging entries q = threadIdx.x + k MET_THREADS (k < SS_STAGE), loaded one
        // plane ahead into registers so that the loads overlap the previous plane's sums
        float pa[SS_STAGE], pb[SS_STAGE];
        auto load_plane = [&](int zi) {
            const float* xp = x + (int64_t)zi * ny * nx;
            const float* yp = y + (int64_t)zi * ny * nx;
#pragma unroll
            for (int k = 0; k < SS_STAGE; ++k) {
                const int q = threadIdx.x + k * MET_THREADS;
                const int r = q / SW, c = q - r * SW;
                const int ix = X0 - p + c, iy = Y0 - p + r;
                const bool ok = q < SH * SW && ix >= 0 && ix < nx && iy >= 0 && iy < ny;
                const int64_t o = (int64_t)iy * nx + ix;
                pa[k] = ok ? __ldg(xp + o) : 0.f;
                pb[k] = ok ? __ldg(yp + o) : 0.f;
            }
        };
        load_plane(zlo);
        for (int zi = zlo; zi <= zhi; ++zi) {
            __syncthreads();   // the previous plane's readers of sa, sb and xb are done
#pragma unroll
            for (int k = 0; k < SS_STAGE; ++k) {
                const int q = threadIdx.x + k * MET_THREADS;
                if (q < SH * SW) {
                    sa[q] = pa[k];
                    sb[q] = pb[k];
                }
            }
            if (zi < zhi) load_plane(zi + 1);
            __syncthreads();
            if (own_xy && zi >= Z0 && zi < Z1) {
                const float d = sa[(ty + p) * SW + tx + p] - sb[(ty + p) * SW + tx + p];
                ksq.add(d * d);
            }
            for (int q = threadIdx.x; q < SH * SS_TX; q += MET_THREADS) {   // box along x
                const int r = q / SS_TX, c = q - r * SS_TX;
                const float* ra = sa + r * SW + c;
                const float* rb = sb + r * SW + c;
                float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, s4 = 0.f;
                for (int d = 0; d <= 2 * p; ++d) {
                    const float u = ra[d], v = rb[d];
                    s0 += u; s1 += v; s2 = fmaf(u, u, s2); s3 = fmaf(v, v, s3); s4 = fmaf(u, v, s4);
                }
                xb[q] = s0; xb[SH * SS_TX + q] = s1; xb[2 * SH * SS_TX + q] = s2; xb[3 * SH * SS_TX + q] = s3;
                xb[4 * SH * SS_TX + q] = s4;
            }
            __syncthreads();
            float* rslot = ring + (size_t)(zi % R) * 5 * SS_TY * SS_TX + ty * SS_TX + tx;
            for (int f = 0; f < 5; ++f) {                                      // box along y (own position)
                const float* col = xb + (size_t)f * SH * SS_TX + ty * SS_TX + tx;
                float s = 0.f;
                for (int d = 0; d <= 2 * p; ++d) s += col[d * SS_TX];
                rslot[f * SS_TY * SS_TX] = s;
            }
            // output plane zi - pz, once its 2 pz + 1 planes are in the ring (this thread's own entries)
            const int zo = zi - pz;
            if (in_xy && zo >= Z0 && zo < Z1 && zo >= pz && zo < nz - pz) {
                float S[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
                for (int zz = zo - pz; zz <= zo + pz; ++zz) {
                    const float* slot = ring + (size_t)(zz % R) * 5 * SS_TY * SS_TX + ty * SS_TX + tx;
#pragma unroll
                    for (int f = 0; f < 5; ++f) S[f] += slot[f * SS_TY * SS_TX];
                }
                const float mx = S[0] * invN, my = S[1] * invN;
                const float sxx = cov * (S[2] * invN - mx * mx);
                const float syy = cov * (S[3] * invN - my * my);
                const float sxy = cov * (S[4] * invN - mx * my);
                kss.add(((2.f * mx * my + C1) * (2.f * sxy + C2)) / ((mx * mx + my * my + C1) * (sxx + syy + C2)));
            }
        }
    }
    double a = (double)ksq.s - (double)ksq.c, b = (double)kss.s - (double)kss.c;
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        red[0][w] = a;
        red[1][w] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sa2 = 0.0, sb2 = 0.0;
        for (int k = 0; k < MET_THREADS / 32; ++k) {
            sa2 += red[0][k];
            sb2 += red[1][k];
        }
        partial[2 * blockIdx.x] = sa2;
        partial[2 * blockIdx.x + 1] = sb2;
    }
}

// The same for the windows up to 9, z first.  A CTA covers SZ_PX x SZ_PY positions, of which the inner
// (SZ_PX - 2 P) x (SZ_PY - 2 P) are the voxels it owns, and marches z through a chunk of planes.  Each
// thread keeps the last 2 PZ + 1 values of x and y of its four positions in registers and forms their
// five sums along z there (no shared memory); the plane of sums goes to shared memory once, is
// box-summed along x (a thread takes 4 neighbouring outputs from 4 + 2 P inputs, 16 bytes at a time) and
// along y (4 outputs from 4 + 2 P rows).  Two barriers per plane.
// What bounds it: shared-memory bandwidth, about 50 words per output position (the kernel above, which
// sums one output at a time along x, y and z in shared memory, moves about 110), and FP32 issue.
// 256 x 256 x 128 voxels, window 7: 125 us, the kernel above 270; one 256 x 256 image 5.8 us, above 17.
// One CTA per SM 162 us, three (64 registers, spills) 284, the z loop unrolled by the ring's length 144.
constexpr int SZ_PX = 64, SZ_PY = 20, SZ_NP = 4, SZ_THREADS = SZ_PX * SZ_PY / SZ_NP;
constexpr int SZ_PITCH = SZ_PX + 4, SZ_PMAX = 4;
constexpr int SZ_CTAS = 2;

template <int P, bool VOL>
__global__ void __launch_bounds__(SZ_THREADS, SZ_CTAS)
ssim_zfirst_kernel(const float* __restrict__ x, const float* __restrict__ y, int nx, int ny, int nz, int zc,
                   unsigned nitems, float invN, float cov, float C1, float C2, double* __restrict__ partial) {
    constexpr int PZ = VOL ? P : 0, R = 2 * PZ + 1, OX = SZ_PX - 2 * P, OY = SZ_PY - 2 * P;
    constexpr int XS = (OX + 3) / 4, YS = (OY + 3) / 4;      // strips of four outputs
    static_assert(XS * SZ_PY <= SZ_THREADS && YS * OX <= SZ_THREADS, "one strip per thread");
    static_assert(4 * (XS - 1) + 4 + 2 * P <= SZ_PITCH, "a strip's inputs stay in the padded row");
    extern __shared__ __align__(16) float szm[];
    float (*zs)[SZ_PY][SZ_PITCH] = reinterpret_cast<float (*)[SZ_PY][SZ_PITCH]>(szm);                    // [5]
    float (*xb)[SZ_PY][SZ_PX] = reinterpret_cast<float (*)[SZ_PY][SZ_PX]>(szm + 5 * SZ_PY * SZ_PITCH);   // [5]
    __shared__ double red[2][SZ_THREADS / 32];
    const int t = threadIdx.x;
    const unsigned ncx = (nx + OX - 1) / OX, ncy = (ny + OY - 1) / OY;
    const int64_t plane = (int64_t)nx * ny;
    KahanF ksq, kss;
    for (int q = t; q < 5 * SZ_PY * (SZ_PITCH - SZ_PX); q += SZ_THREADS)      // the pad feeds unused outputs only
        zs[q / (SZ_PY * 4)][(q / 4) % SZ_PY][SZ_PX + q % 4] = 0.f;
    for (unsigned it = blockIdx.x; it < nitems; it += gridDim.x) {
        const unsigned cx = it % ncx, rest = it / ncx;
        const int X0 = (int)cx * OX, Y0 = (int)(rest % ncy) * OY, Z0 = (int)(rest / ncy) * zc, Z1 = min(Z0 + zc, nz);
        // this thread's positions: offsets in a plane (-1: outside the volume), and whether the CTA owns them
        int off[SZ_NP];
        unsigned own = 0;
#pragma unroll
        for (int i = 0; i < SZ_NP; ++i) {
            const int q = t + i * SZ_THREADS, col = q % SZ_PX, row = q / SZ_PX;
            const int gx = X0 - P + col, gy = Y0 - P + row;
            const bool ok = gx >= 0 && gx < nx && gy >= 0 && gy < ny;
            off[i] = ok ? gy * nx + gx : -1;
            own |= (unsigned)(ok && col >= P && col < SZ_PX - P && row >= P && row < SZ_PY - P) << i;
        }
        float rx[SZ_NP][R], ry[SZ_NP][R], px[SZ_NP], py[SZ_NP];
#pragma unroll
        for (int i = 0; i < SZ_NP; ++i)
#pragma unroll
            for (int k = 0; k < R; ++k) rx[i][k] = ry[i][k] = 0.f;
        const int zlo = max(Z0 - PZ, 0), zhi = min(Z1 - 1 + PZ, nz - 1);
        auto load = [&](int zi) {
            const float* xp = x + zi * plane;
            const float* yp = y + zi * plane;
#pragma unroll
            for (int i = 0; i < SZ_NP; ++i) {
                px[i] = off[i] >= 0 ? __ldg(xp + off[i]) : 0.f;
                py[i] = off[i] >= 0 ? __ldg(yp + off[i]) : 0.f;
            }
        };
        load(zlo);
#pragma unroll 1
        for (int zi = zlo; zi <= zhi; ++zi) {
            const bool mine = zi >= Z0 && zi < Z1;
#pragma unroll
            for (int i = 0; i < SZ_NP; ++i) {
#pragma unroll
                for (int k = 0; k < R - 1; ++k) { rx[i][k] = rx[i][k + 1]; ry[i][k] = ry[i][k + 1]; }
                rx[i][R - 1] = px[i];
                ry[i][R - 1] = py[i];
                if (mine && (own >> i & 1)) {
                    const float d = px[i] - py[i];
                    ksq.add(d * d);
                }
            }
            if (zi < zhi) load(zi + 1);
            const int zo = zi - PZ;                        // the plane whose z window is complete
            if (zo < max(Z0, PZ) || zo >= min(Z1, nz - PZ)) continue;
#pragma unroll
            for (int i = 0; i < SZ_NP; ++i) {
                float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, s4 = 0.f;
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const float u = rx[i][k], v = ry[i][k];
                    s0 += u; s1 += v; s2 = fmaf(u, u, s2); s3 = fmaf(v, v, s3); s4 = fmaf(u, v, s4);
                }
                const int q = t + i * SZ_THREADS, col = q % SZ_PX, row = q / SZ_PX;
                zs[0][row][col] = s0; zs[1][row][col] = s1; zs[2][row][col] = s2; zs[3][row][col] = s3; zs[4][row][col] = s4;
            }
            __syncthreads();
            if (t < XS * SZ_PY) {
                const int row = t / XS, c = 4 * (t - row * XS);
#pragma unroll
                for (int f = 0; f < 5; ++f) {
                    constexpr int NV = (2 * P + 4 + 3) / 4;
                    float v[4 * NV];
#pragma unroll
                    for (int k = 0; k < NV; ++k) {
                        const float4 q = *reinterpret_cast<const float4*>(&zs[f][row][c + 4 * k]);
                        v[4 * k] = q.x; v[4 * k + 1] = q.y; v[4 * k + 2] = q.z; v[4 * k + 3] = q.w;
                    }
                    // outputs o = 0 .. 3 sum v[o .. o + 2 P]; v[3 .. 2 P] is common to the four (P >= 2)
                    float o0, o1, o2, o3;
                    if constexpr (P >= 2) {
                        float m = v[3];
#pragma unroll
                        for (int k = 4; k <= 2 * P; ++k) m += v[k];
                        const float l = v[1] + v[2], h = v[2 * P + 1] + v[2 * P + 2];
                        o0 = (v[0] + l) + m;
                        o1 = (l + m) + v[2 * P + 1];
                        o2 = (v[2] + m) + h;
                        o3 = (m + h) + v[2 * P + 3];
                    } else {
                        o0 = v[0] + v[1] + v[2]; o1 = v[1] + v[2] + v[3]; o2 = v[2] + v[3] + v[4]; o3 = v[3] + v[4] + v[5];
                    }
                    *reinterpret_cast<float4*>(&xb[f][row][c]) = make_float4(o0, o1, o2, o3);
                }
            }
            __syncthreads();
            if (t < YS * OX) {
                const int c = t % OX, r0 = 4 * (t / OX);
                const int gx = X0 + c;
                float S[5][4];
#pragma unroll
                for (int f = 0; f < 5; ++f) {
                    float v[2 * P + 4];
#pragma unroll
                    for (int k = 0; k < 2 * P + 4; ++k) v[k] = r0 + k < SZ_PY ? xb[f][r0 + k][c] : 0.f;
                    if constexpr (P >= 2) {
                        float m = v[3];
#pragma unroll
                        for (int k = 4; k <= 2 * P; ++k) m += v[k];
                        const float l = v[1] + v[2], h = v[2 * P + 1] + v[2 * P + 2];
                        S[f][0] = (v[0] + l) + m;
                        S[f][1] = (l + m) + v[2 * P + 1];
                        S[f][2] = (v[2] + m) + h;
                        S[f][3] = (m + h) + v[2 * P + 3];
                    } else {
                        S[f][0] = v[0] + v[1] + v[2]; S[f][1] = v[1] + v[2] + v[3]; S[f][2] = v[2] + v[3] + v[4]; S[f][3] = v[3] + v[4] + v[5];
                    }
                }
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    const int gy = Y0 + r0 + o;
                    if (r0 + o < OY && gx >= P && gx < nx - P && gy >= P && gy < ny - P) {
                        const float mx = S[0][o] * invN, my = S[1][o] * invN;
                        const float sxx = cov * (S[2][o] * invN - mx * mx);
                        const float syy = cov * (S[3][o] * invN - my * my);
                        const float sxy = cov * (S[4][o] * invN - mx * my);
                        kss.add(((2.f * mx * my + C1) * (2.f * sxy + C2)) / ((mx * mx + my * my + C1) * (sxx + syy + C2)));
                    }
                }
            }
        }
        __syncthreads();       // the last plane's readers are done before the next item's sums
    }
    double a = (double)ksq.s - (double)ksq.c, b = (double)kss.s - (double)kss.c;
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((t & 31) == 0) {
        red[0][t >> 5] = a;
        red[1][t >> 5] = b;
    }
    __syncthreads();
    if (t == 0) {
        double sa2 = 0.0, sb2 = 0.0;
        for (int k = 0; k < SZ_THREADS / 32; ++k) {
            sa2 += red[0][k];
            sb2 += red[1][k];
        }
        partial[2 * blockIdx.x] = sa2;
        partial[2 * blockIdx.x + 1] = sb2;
    }
}

// Launches the kernel above; returns the CTAs (partials) it used, 0 where its 32-bit indices do not reach.
template <int P, bool VOL>
static int launch_zfirst(const float* x, const float* y, int nx, int ny, int nz, float invN, float cov, float C1, float C2,
                         double* partial, cudaStream_t st) {
    constexpr int OX = SZ_PX - 2 * P, OY = SZ_PY - 2 * P, PZ = VOL ? P : 0;
    const int64_t cols = (int64_t)((nx + OX - 1) / OX) * ((ny + OY - 1) / OY), slots = (int64_t)SZ_CTAS * device_sms();
    // the chunk length whose waves of CTAs take the fewest planes (a chunk of zc reads zc + 2 PZ)
    int zc = nz;
    int64_t cost = INT64_MAX;
    for (int n = 1; n <= 64 && n <= nz; ++n) {
        const int c = (nz + n - 1) / n;
        const int64_t w = (cols * ((nz + c - 1) / c) + slots - 1) / slots * (c + 2 * PZ);
        if (w < cost) { cost = w; zc = c; }
    }
    const int64_t items = cols * ((nz + zc - 1) / zc);
    if (items >= ((int64_t)1 << 31) || (int64_t)nx * ny >= ((int64_t)1 << 31)) return 0;
    const int nb = (int)(items < slots ? items : slots);
    constexpr int sm = 5 * SZ_PY * (SZ_PITCH + SZ_PX) * (int)sizeof(float);
    if (cudaFuncSetAttribute(ssim_zfirst_kernel<P, VOL>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm) != cudaSuccess) return 0;
    ssim_zfirst_kernel<P, VOL><<<nb, SZ_THREADS, sm, st>>>(x, y, nx, ny, nz, zc, (unsigned)items, invN, cov, C1, C2, partial);
    return nb;
}

// res[0] = sum (x - ref)^2 over all voxels, res[2] = sum of SSIM over the interior positions: each
// thread sums a fixed stride of the CTA partials, then a fixed tree (deterministic).
__global__ void __launch_bounds__(MET_THREADS)
ssim_march_finish_kernel(const double* __restrict__ partial, int n, double* __restrict__ res) {
    __shared__ double sa[MET_THREADS], sb[MET_THREADS];
    double a = 0.0, b = 0.0;
    for (int k = threadIdx.x; k < n; k += MET_THREADS) {
        a += partial[2 * k];
        b += partial[2 * k + 1];
    }
    sa[threadIdx.x] = a;
    sb[threadIdx.x] = b;
    __syncthreads();
    for (int w = MET_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            sa[threadIdx.x] += sa[threadIdx.x + w];
            sb[threadIdx.x] += sb[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        res[0] = sa[0];
        res[2] = sb[0];
    }
}

size_t ssim_march_partial_doubles() { return 2 * (size_t)MET_BLOCKS; }
int metrics_march_pmax() { return SS_PMAX; }

// cudaErrorNotSupported when the window is wider than the fused kernel handles (caller falls back).
cudaError_t launch_metrics_march(const float* x, const float* y, int nx, int ny, int nz, int win, float range,
                                 double* partial, double* res, cudaStream_t st) {
    const int p = (win - 1) / 2, pz = nz > 1 ? p : 0;
    if (p > SS_PMAX) return cudaErrorNotSupported;
    const double N = nz > 1 ? (double)win * win * win : (double)win * win;
    cudaError_t e;
    const float C1 = (0.01f * range) * (0.01f * range), C2 = (0.03f * range) * (0.03f * range);
    const float invN = (float)(1.0 / N), cov = (float)(N / (N - 1.0));
    int nb = 0;
    switch (p <= SZ_PMAX ? 2 * p + (nz > 1) : 0) {
#define GP_ZF(P) case 2 * P: nb = launch_zfirst<P, false>(x, y, nx, ny, nz, invN, cov, C1, C2, partial, st); break; \
                 case 2 * P + 1: nb = launch_zfirst<P, true>(x, y, nx, ny, nz, invN, cov, C1, C2, partial, st); break;
        GP_ZF(1) GP_ZF(2) GP_ZF(3) GP_ZF(4)
#undef GP_ZF
    }
    if (nb == 0) {
        const size_t sm = ssim_march_floats(p, pz) * sizeof(float);
        e = cudaFuncSetAttribute(ssim_march_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        nb = MET_BLOCKS;
        ssim_march_kernel<<<nb, MET_THREADS, sm, st>>>(x, y, nx, ny, nz, p, pz, invN, cov, C1, C2, partial);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ssim_march_finish_kernel<<<1, MET_THREADS, 0, st>>>(partial, nb, res);
    return cudaGetLastError();
}

cudaError_t launch_zmap(const float* vol, int nx, int ny, int nz, float* out, cudaStream_t st) {
    const int64_t nb = ((int64_t)nx * ny + ZM_X - 1) / ZM_X, most = (int64_t)16 * device_sms();
    zmap_kernel<<<(unsigned)(nb < most ? nb : most), MET_THREADS, 0, st>>>(vol, nx, ny, nz, out);
    return cudaGetLastError();
}

size_t ssim_scratch_bytes(int64_t M) { return (size_t)M * 10 * sizeof(float) + sizeof(double) * (MET_BLOCKS + 1); }

// out (device): the sum of SSIM over the interior positions.
cudaError_t launch_ssim_sum(const float* x, const float* y, int nx, int ny, int nz, int win, float range, void* scratch,
                            double* out, cudaStream_t st) {
    const int64_t M = (int64_t)nx * ny * nz;
    float* A = static_cast<float*>(scratch);
    float* B = A + 5 * M;
    double* partial = reinterpret_cast<double*>(B + 5 * M);
    const int p = (win - 1) / 2, pz = nz > 1 ? p : 0;
    const int dimsN = nz > 1 ? 3 : 2;
    const double N = dimsN == 3 ? (double)win * win * win : (double)win * win;
    box_x_kernel<<<MET_BLOCKS, MET_THREADS, 0, st>>>(x, y, nx, ny, nz, p, A);
    box_yz_kernel<<<MET_BLOCKS, MET_THREADS, 0, st>>>(A, nx, ny, nz, p, 1, B);
    const float* S = B;
    if (nz > 1) {
        box_yz_kernel<<<MET_BLOCKS, MET_THREADS, 0, st>>>(B, nx, ny, nz, p, 2, A);
        S = A;
    }
    const float C1 = (0.01f * range) * (0.01f * range), C2 = (0.03f * range) * (0.03f * range);
    ssim_kernel<<<MET_BLOCKS, MET_THREADS, 0, st>>>(S, nx, ny, nz, p, pz, (float)(1.0 / N), (float)(N / (N - 1.0)), C1,
                                                    C2, partial);
    sum_partials_kernel<<<1, 32, 0, st>>>(partial, MET_BLOCKS, out);
    return cudaGetLastError();
}

}  // namespace gp
