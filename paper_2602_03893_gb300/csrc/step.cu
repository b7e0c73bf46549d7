// step.cu -- elementwise and reduction kernels of one reconstruction iteration (Algorithm 2):
// the nonnegative parameterisation x = (z + eps)^2 and its chain rule (Methods, NPC), the data
// loss |y - b|^2 / N and residual norm reduced in FP64, the Adam update, and the exact line
// search step of the steepest-descent variant.  All HBM-bound; FP64 is used only inside the
// reductions.
#include "gpair_internal.cuh"
#include "step_sched.cuh"

#include <atomic>
#include <cmath>

namespace gp {

constexpr int RED_THREADS = 256;
// Block partials of the FP64 reductions: 4 per SM of the current device; a second pass sums them in
// order.
int red_blocks();
#define RED_BLOCKS red_blocks()

__global__ void npc_kernel(const float* __restrict__ z, float* __restrict__ x, int64_t M, int npc, float eps) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        float zi = z[i];
        x[i] = npc ? (zi + eps) * (zi + eps) : zi;
    }
}

__device__ __forceinline__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k];
    return s;
}

// r = y - b; delta = scale * r (may alias nothing); partial[blk][0] = sum r^2 (FP64).
__global__ void __launch_bounds__(RED_THREADS)
resid_kernel(const float* __restrict__ y, const float* __restrict__ b, float* __restrict__ delta, float scale,
             int64_t n, double* __restrict__ partial) {
    __shared__ double red[RED_THREADS / 32];
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float r = y[i] - b[i];
        acc += (double)r * (double)r;
        delta[i] = scale * r;
    }
    double s = block_sum(acc, red);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// Generic FP64 reductions: partial[blk] = (sum (a - b)^2, sum a * c).  b, c may be NULL.
__global__ void __launch_bounds__(RED_THREADS)
reduce2_kernel(const float* __restrict__ a, const float* __restrict__ b, const float* __restrict__ c, int64_t n,
               double* __restrict__ partial) {
    __shared__ double red[RED_THREADS / 32];
    double s0 = 0.0, s1 = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double ai = a[i];
        double d = b ? ai - (double)b[i] : ai;
        s0 += d * d;
        if (c) s1 += ai * (double)c[i];
    }
    double t0 = block_sum(s0, red);
    double t1 = block_sum(s1, red);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = t0;
        partial[2 * blockIdx.x + 1] = t1;
    }
}

// out[q] = sum_blk partial[blk * stride + q] for q < nq, in block order (deterministic).
__device__ __forceinline__ void finish_sums(const double* __restrict__ partial, int nblk, int stride, int nq,
                                            double* __restrict__ out) {
    __shared__ double red[RED_THREADS / 32];
    for (int q = 0; q < nq; ++q) {
        double acc = 0.0;
        for (int k = threadIdx.x; k < nblk; k += blockDim.x) acc += partial[(size_t)k * stride + q];
        double s = block_sum(acc, red);
        if (threadIdx.x == 0) out[q] = s;
        __syncthreads();
    }
}
__global__ void finish_kernel(const double* __restrict__ partial, int nblk, int stride, int nq,
                              double* __restrict__ out) {
    finish_sums(partial, nblk, stride, nq, out);
}

// Adam on z with gradient g_x (and the NPC chain rule g_z = g_x * 2 (z + eps)).
// Per-step scalars of Algorithm 2 on the device, so that a step's launches do not change from one
// step to the next (and can be replayed as a CUDA graph): the CAWR step size of step t and Adam's
// bias corrections 1 / (1 - b1^(t+1)), 1 / sqrt(1 - b2^(t+1)), the powers kept as running
// products.  One thread; FP64 only for the products (GB300's FP64 pipe is slow, and a chain of
// FP64 pow / cos / divide took ~11 us).  Advances t.
__device__ __forceinline__ void schedule_step(const SchedParams& p, StepSched* __restrict__ sd) {
    const int t = sd->t;
    // SGDR: periods T0, T0 T_mult, ...; T_cur counts iterations since the last restart
    const int T0 = p.T0 > 0 ? p.T0 : 1;
    float phase;                                   // T_cur / T_i
    if (p.T_mult <= 1.0) {
        phase = (float)(t % T0) / (float)T0;
    } else {
        double Tcur = t, Ti = T0;
        for (int guard = 0; Tcur >= Ti && guard < 4096; ++guard) {   // O(log t) periods
            Tcur -= Ti;
            Ti *= p.T_mult;
        }
        phase = (float)(Tcur / Ti);
    }
    sd->eta = (float)p.eta_min + 0.5f * (float)(p.eta_max - p.eta_min) * (1.f + cospif(phase));
    const double b1t = sd->b1t * p.beta1, b2t = sd->b2t * p.beta2;   // beta^(t+1)
    sd->b1t = b1t;
    sd->b2t = b2t;
    sd->inv_c1 = 1.f / (float)(1.0 - b1t);
    sd->inv_sqrt_c2 = rsqrtf((float)(1.0 - b2t));
    sd->t = t + 1;
}

// Block 0: out[0] = the sum of the residual's partials; block 1: the step's scalars, a launch less.
__global__ void finish_schedule_kernel(const double* __restrict__ partial, int nblk, double* __restrict__ out,
                                       SchedParams p, StepSched* __restrict__ sd) {
    if (blockIdx.x == 0) finish_sums(partial, nblk, 1, 1, out);
    else if (threadIdx.x == 0) schedule_step(p, sd);
}

__global__ void set_step_kernel(StepSched* __restrict__ sd, int t, double b1t, double b2t) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        sd->t = t;
        sd->b1t = b1t;
        sd->b2t = b2t;
    }
}

// x: the amplitudes of the new iterate, as npc_kernel gives them.
__global__ void adam_kernel(float* __restrict__ z, float* __restrict__ m, float* __restrict__ v, float* __restrict__ x,
                            const float* __restrict__ gx, int64_t M, int npc, float eps, float b1, float b2,
                            float adam_eps, const StepSched* __restrict__ sd) {
    const float eta = sd->eta, inv_c1 = sd->inv_c1, inv_sqrt_c2 = sd->inv_sqrt_c2;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        float zi = z[i];
        float g = gx[i];
        if (npc) g *= 2.f * (zi + eps);
        float mi = b1 * m[i] + (1.f - b1) * g;
        float vi = b2 * v[i] + (1.f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        zi = zi - eta * (mi * inv_c1) / (sqrtf(vi) * inv_sqrt_c2 + adam_eps);
        z[i] = zi;
        x[i] = npc ? (zi + eps) * (zi + eps) : zi;
    }
}

// x <- x - alpha g with alpha = num / den read from device memory (exact line search).
__global__ void ls_update_kernel(float* __restrict__ x, const float* __restrict__ g, int64_t M,
                                 const double* __restrict__ nd) {
    const double den = nd[1];
    const float alpha = den > 0.0 ? (float)(nd[0] / den) : 0.f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x)
        x[i] -= alpha * g[i];
}

// dot(r, Fg) and |Fg|^2 into partials (for the line search).
__global__ void __launch_bounds__(RED_THREADS)
ls_dots_kernel(const float* __restrict__ r, const float* __restrict__ Fg, int64_t n, double* __restrict__ partial) {
    __shared__ double red[RED_THREADS / 32];
    double s0 = 0.0, s1 = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double f = Fg[i];
        s0 += (double)r[i] * f;
        s1 += f * f;
    }
    double t0 = block_sum(s0, red);
    double t1 = block_sum(s1, red);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = t0;
        partial[2 * blockIdx.x + 1] = t1;
    }
}

static int ew_blocks(int64_t n) {
    int64_t b = (n + 255) / 256;
    if (b > (int64_t)device_sms() * 32) b = (int64_t)device_sms() * 32;
    return (int)(b < 1 ? 1 : b);
}

cudaError_t launch_npc(const float* z, float* x, int64_t M, int npc, float eps, cudaStream_t st) {
    npc_kernel<<<ew_blocks(M), 256, 0, st>>>(z, x, M, npc, eps);
    return cudaGetLastError();
}

// partial must hold RED_BLOCKS doubles; out[0] = sum r^2.  sd (optional): the schedule advances too.
cudaError_t launch_resid(const float* y, const float* b, float* delta, float scale, int64_t n, double* partial,
                         double* out, const SchedParams& p, StepSched* sd, cudaStream_t st) {
    resid_kernel<<<RED_BLOCKS, RED_THREADS, 0, st>>>(y, b, delta, scale, n, partial);
    if (sd) finish_schedule_kernel<<<2, RED_THREADS, 0, st>>>(partial, RED_BLOCKS, out, p, sd);
    else finish_kernel<<<1, RED_THREADS, 0, st>>>(partial, RED_BLOCKS, 1, 1, out);
    return cudaGetLastError();
}

// partial must hold 2 * RED_BLOCKS doubles; out[0..1].
cudaError_t launch_reduce2(const float* a, const float* b, const float* c, int64_t n, double* partial, double* out,
                           cudaStream_t st) {
    reduce2_kernel<<<RED_BLOCKS, RED_THREADS, 0, st>>>(a, b, c, n, partial);
    finish_kernel<<<1, RED_THREADS, 0, st>>>(partial, RED_BLOCKS, 2, 2, out);
    return cudaGetLastError();
}

cudaError_t launch_ls(const float* r, const float* Fg, int64_t n, float* x, const float* g, int64_t M,
                      double* partial, double* nd, cudaStream_t st) {
    ls_dots_kernel<<<RED_BLOCKS, RED_THREADS, 0, st>>>(r, Fg, n, partial);
    finish_kernel<<<1, RED_THREADS, 0, st>>>(partial, RED_BLOCKS, 2, 2, nd);
    ls_update_kernel<<<ew_blocks(M), 256, 0, st>>>(x, g, M, nd);
    return cudaGetLastError();
}

// t steps taken: the running products are beta^t.
cudaError_t launch_set_step(StepSched* sd, int t, const SchedParams& p, cudaStream_t st) {
    set_step_kernel<<<1, 32, 0, st>>>(sd, t, std::pow(p.beta1, (double)t), std::pow(p.beta2, (double)t));
    return cudaGetLastError();
}

cudaError_t launch_adam(float* z, float* m, float* v, float* x, const float* gx, int64_t M, int npc, float eps, float b1,
                        float b2, float adam_eps, const StepSched* sd, cudaStream_t st) {
    adam_kernel<<<ew_blocks(M), 256, 0, st>>>(z, m, v, x, gx, M, npc, eps, b1, b2, adam_eps, sd);
    return cudaGetLastError();
}

int red_blocks() { return 4 * device_sms(); }

int device_sms() {
    constexpr int MAXDEV = 64;
    static std::atomic<int> cache[MAXDEV];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 1; }
    if (dev < 0 || dev >= MAXDEV) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
            cudaGetLastError();
            return 1;
        }
        return n;
    }
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
        cudaGetLastError();
        return 1;
    }
    cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

// ---- vessel continuity regulariser (Methods: R_VCR = R_H + beta R_TV) on a lattice image --------
// Readings of the unspecified parts: central first differences (x[i+1] - x[i-1]) / 2; second
// differences x[i+1] - 2 x[i] + x[i-1] and the four-point mixed stencil / 4 (counted twice in the
// Frobenius sum, D_pq = D_qp); Neumann boundaries (neighbour indices clamped per axis); unit voxel
// spacing; eps inside each square root.  Image x fastest.

// One fused pass marching along z.  A CTA covers 32 x VM_PY field positions, one thread each (a warp is
// a row), of which the inner 30 x (VM_PY - 2) are the voxels it owns, and a chunk of planes.  Per step it
// has one plane of x in shared memory (with one more voxel of halo, neighbour indices clamped per
// axis: the Neumann reading); each thread reads its eight neighbours there once and keeps what the
// stencils need of them for three planes in registers.  From planes z - 1, z, z + 1 it forms its
// weighted fields at plane z,
//   F_k = m_k (D_k x) / sqrt(sH + eps)  (k = xx, yy, zz, xy, xz, yz; m = 1, 1, 1, 2, 2, 2),
//   F_{6+d} = beta (D_d x) / sqrt(sT + eps),
// sH = sum_{p,q} (D_pq x)^2, sT = sum_d (D_d x)^2, zero outside the volume, and hands the ones that
// neighbours along y need on through shared memory, along x through warp shuffles.
// The gradient sum_k D_k^T F_k is separable per axis: with S_o the clamped shift, (S_o^T F)[j] =
// F[j - o], plus F[j] itself where j + o leaves the volume.  So along an axis, with lo / hi telling
// whether j is its first / last node,
//   (S_+ - S_-)^T F      = F[j-1] - F[j+1] + (hi - lo) F[j],
//   (S_+ - 2 + S_-)^T F  = F[j-1] + F[j+1] + (hi + lo - 2) F[j],
// exact on faces, edges and corners alike; the mixed fields take the first form along both axes.  The
// z part of plane z goes to planes z - 1, z and z + 1: each thread carries the sums of two pending
// planes.  Only x and g cross HBM.  Two sets of buffers: one barrier per plane.
// What bounds it: shared-memory and shuffle issue, 25 accesses per position and plane, and the plane's
// chain of loads, square roots and one barrier.  256 x 256 x 128: 109 us, where the form with nine field
// planes in shared memory (72 accesses per voxel, two barriers a plane) took 214.  Rows per CTA x CTAs per
// SM: 16 x 2 109 us, 16 x 3 (40 registers, spills) 125, 32 x 1 110, 8 x 4 118.
// The value sum sqrt(sH + eps) + beta sqrt(sT + eps) over the CTA's own voxels is compensated FP32 per
// thread and FP64 per CTA (partial[blockIdx.x]).
constexpr int VM_PY = 16, VM_CTAS = 2;                 // field rows of a CTA, CTAs per SM
constexpr int VM_THREADS = 32 * VM_PY;
constexpr int VM_OX = 30, VM_OY = VM_PY - 2;           // voxels owned
constexpr int VM_XW = 34, VM_XH = VM_PY + 2, VM_XN = VM_XW * VM_XH;   // staged x plane
constexpr int VM_STAGE = (VM_XN + VM_THREADS - 1) / VM_THREADS;

__device__ __forceinline__ double block_sum_n(double v, double* red, int warps) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < warps; ++k) s += red[k];
    return s;
}

template <bool GRAD>
__global__ void __launch_bounds__(VM_THREADS, VM_CTAS)
vcr_march_kernel(const float* __restrict__ x, int nx, int ny, int nz, float beta, float eps, float lam,
                 float* __restrict__ g, double* __restrict__ partial, int zc, unsigned nitems) {
    __shared__ float xs[2][VM_XN];
    __shared__ float fs[GRAD ? 2 : 1][GRAD ? 4 : 1][GRAD ? VM_THREADS : 1];   // A, B, yz, xy rows (see below)
    __shared__ double red[VM_PY];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const unsigned ncx = (nx + VM_OX - 1) / VM_OX, ncy = (ny + VM_OY - 1) / VM_OY;
    const int64_t plane = (int64_t)nx * ny;
    KahanF acc;    // this thread's own voxels; FP64 from the CTA sum on
    for (unsigned it = blockIdx.x; it < nitems; it += gridDim.x) {
        const unsigned cx = it % ncx, rest = it / ncx;
        const int X0 = (int)cx * VM_OX, Y0 = (int)(rest % ncy) * VM_OY, Z0 = (int)(rest / ncy) * zc;
        const int Z1 = min(Z0 + zc, nz);
        const int px = X0 - 1 + lane, py = Y0 - 1 + row;               // this thread's field position
        const bool inside = px >= 0 && px < nx && py >= 0 && py < ny;
        const bool own = inside && lane >= 1 && lane <= VM_OX && row >= 1 && row <= VM_OY;
        const float hix = px == nx - 1 ? 1.f : 0.f, lox = px == 0 ? 1.f : 0.f;
        const float hiy = py == ny - 1 ? 1.f : 0.f, loy = py == 0 ? 1.f : 0.f;
        const float ex = hix - lox, ax = hix + lox - 2.f, ey = hiy - loy, ay = hiy + loy - 2.f;
        // this thread's staging entries: offsets in a plane, the same for every plane of the item
        int64_t off[VM_STAGE];
#pragma unroll
        for (int u = 0; u < VM_STAGE; ++u) {
            const int q = threadIdx.x + u * VM_THREADS, a = q % VM_XW, b = q / VM_XW;
            const int ix = min(max(X0 - 2 + a, 0), nx - 1), iy = min(max(Y0 - 2 + b, 0), ny - 1);
            off[u] = q < VM_XN ? (int64_t)iy * nx + ix : -1;
        }
        float pre[VM_STAGE];
        auto load_plane = [&](int zi) {
            const float* xp = x + (int64_t)min(max(zi, 0), nz - 1) * plane;
#pragma unroll
            for (int u = 0; u < VM_STAGE; ++u) pre[u] = off[u] >= 0 ? __ldg(xp + off[u]) : 0.f;
        };
        auto store_plane = [&](int s) {
#pragma unroll
            for (int u = 0; u < VM_STAGE; ++u)
                if (off[u] >= 0) xs[s & 1][threadIdx.x + u * VM_THREADS] = pre[u];
        };
        // Step s reads x plane Z0 - 2 + s, forms the fields of plane zf = Z0 - 3 + s (s >= 2) and finishes
        // the gradient of plane zf - 1 (s >= 4); x plane s + 1 is stored and plane s + 2 loaded meanwhile.
        load_plane(Z0 - 2);
        __syncthreads();                 // the previous item's readers are done
        store_plane(0);
        load_plane(Z0 - 1);
        __syncthreads();
        // of x: the centre and the x and y differences of the last three planes, and the in-plane second
        // differences of the last two
        float c0 = 0.f, cm = 0.f, dx0 = 0.f, dxm = 0.f, dy0 = 0.f, dym = 0.f, hxx0 = 0.f, hyy0 = 0.f, hxy0 = 0.f;
        float hold = 0.f, zplus = 0.f;   // gradient of plane zf - 1 without its part from zf; part of zf - 1 for zf
        for (int s = 0; Z0 - 4 + s < Z1; ++s) {
            const float* xp = &xs[s & 1][(row + 1) * VM_XW + lane + 1];
            const float cp = xp[0];
            const float xr = xp[1], xl = xp[-1], yr = xp[VM_XW], yl = xp[-VM_XW];
            const float dxp = xr - xl, dyp = yr - yl;
            const float hxxp = (xr - cp) + (xl - cp), hyyp = (yr - cp) + (yl - cp);
            const float hxyp = 0.25f * ((xp[VM_XW + 1] - xp[1 - VM_XW]) - (xp[VM_XW - 1] - xp[-VM_XW - 1]));
            if (s + 1 < Z1 - Z0 + 4) store_plane(s + 1);
            if (s + 2 < Z1 - Z0 + 4) load_plane(Z0 + s);
            const int zf = Z0 - 3 + s;
            float fzz = 0.f, fz = 0.f, fxz = 0.f, fyz = 0.f, fxy = 0.f, fxx = 0.f, fx = 0.f, fyy = 0.f, fy = 0.f;
            if (s >= 2 && inside && zf >= 0 && zf < nz) {
                const float hzz = (cp - c0) + (cm - c0), d1z = 0.5f * (cp - cm);
                const float hxz = 0.25f * (dxp - dxm), hyz = 0.25f * (dyp - dym);
                const float d1x = 0.5f * dx0, d1y = 0.5f * dy0;
                const float sH = hxx0 * hxx0 + hyy0 * hyy0 + hzz * hzz + 2.f * (hxy0 * hxy0 + hxz * hxz + hyz * hyz) + eps;
                const float sT = d1x * d1x + d1y * d1y + d1z * d1z + eps;
                if (GRAD) {
                    const float wH = rsqrtf(sH), wT = 0.5f * beta * rsqrtf(sT);
                    fxx = wH * hxx0; fyy = wH * hyy0; fzz = wH * hzz;
                    const float wM = 0.5f * wH;              // the factor 2 of the mixed fields and the 1/4 of their stencil
                    fxy = wM * hxy0; fxz = wM * hxz; fyz = wM * hyz;
                    fx = wT * d1x; fy = wT * d1y; fz = wT * d1z;     // with the 1/2 of their stencil
                }
                if (own && zf >= Z0 && zf < Z1) acc.add(sqrtf(sH) + beta * sqrtf(sT));
            }
            if constexpr (GRAD) {
                float (*F)[VM_THREADS] = fs[s & 1];
                F[0][threadIdx.x] = fyy + fy;                // A: what the row above adds
                F[1][threadIdx.x] = fyy - fy;                // B: what the row below adds
                F[2][threadIdx.x] = fyz;
                F[3][threadIdx.x] = fxy;
            }
            __syncthreads();
            if constexpr (GRAD) if (s >= 2) {
                float (*F)[VM_THREADS] = fs[s & 1];
                const int up = max((int)threadIdx.x - 32, 0), dn = min((int)threadIdx.x + 32, VM_THREADS - 1);  // rows 0 and VM_PY - 1 own nothing
                // along y, then x, the mixed xy field; the terms that take j itself only on the faces
                float q = F[3][up] - F[3][dn];
                float in = F[0][up] + F[1][dn] + ay * fyy;
                float by = F[2][up] - F[2][dn];
                if (ey != 0.f) {
                    q += ey * fxy;
                    in += ey * fy;
                    by += ey * fyz;
                }
                in += __shfl_up_sync(0xffffffffu, fxx + fx, 1) + __shfl_down_sync(0xffffffffu, fxx - fx, 1) + ax * fxx;
                in += __shfl_up_sync(0xffffffffu, q, 1) - __shfl_down_sync(0xffffffffu, q, 1);
                float b = __shfl_up_sync(0xffffffffu, fxz, 1) - __shfl_down_sync(0xffffffffu, fxz, 1);
                if (ex != 0.f) {
                    in += ex * (fx + q);
                    b += ex * fxz;
                }
                b += by + fz;                        // what plane zf gives its neighbours along z
                const float hiz = zf == nz - 1 ? 1.f : 0.f, loz = zf == 0 ? 1.f : 0.f;
                in += (hiz + loz - 2.f) * fzz;
                if (hiz != loz) in += (hiz - loz) * b;
                const int jz = zf - 1;
                if (own && jz >= Z0 && jz < Z1) {
                    const int64_t j = (int64_t)jz * plane + (int64_t)py * nx + px;
                    g[j] = fmaf(lam, hold + (fzz - b), g[j]);
                }
                hold = zplus + in;
                zplus = fzz + b;
            }
            cm = c0; c0 = cp;
            dxm = dx0; dx0 = dxp;
            dym = dy0; dy0 = dyp;
            hxx0 = hxxp; hyy0 = hyyp; hxy0 = hxyp;
        }
    }
    const double tot = block_sum_n((double)acc.s - (double)acc.c, red, VM_PY);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

// Planes per item and the item count: the chunk length whose waves of CTAs take the fewest plane
// steps (a chunk of zc planes takes zc + 4).
static int vcr_chunk(int nx, int ny, int nz, int slots, int64_t& items) {
    const int64_t cols = (int64_t)((nx + VM_OX - 1) / VM_OX) * ((ny + VM_OY - 1) / VM_OY);
    int best = nz;
    int64_t cost = INT64_MAX;
    for (int n = 1; n <= 64 && n <= nz; ++n) {
        const int zc = (nz + n - 1) / n;
        const int64_t its = cols * ((nz + zc - 1) / zc), c = (its + slots - 1) / slots * (zc + 4);
        if (c < cost) { cost = c; best = zc; }
    }
    items = cols * ((nz + best - 1) / best);
    return best;
}

// value_out (device, may be NULL): R_VCR(x) in FP64.  g (may be NULL): g += lam grad R_VCR(x).
// partial: RED_BLOCKS doubles.
cudaError_t launch_vcr(const float* x, int nx, int ny, int nz, float beta, float eps, float lam, double* partial,
                       double* value_out, float* g, cudaStream_t st) {
    const int slots = VM_CTAS * device_sms();
    int64_t items = 0;
    const int zc = vcr_chunk(nx, ny, nz, slots, items);
    if (items >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
    const int nb = (int)(items < slots ? items : slots);
    if (g) vcr_march_kernel<true><<<nb, VM_THREADS, 0, st>>>(x, nx, ny, nz, beta, eps, lam, g, partial, zc, (unsigned)items);
    else vcr_march_kernel<false><<<nb, VM_THREADS, 0, st>>>(x, nx, ny, nz, beta, eps, lam, nullptr, partial, zc, (unsigned)items);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (value_out) {
        finish_kernel<<<1, RED_THREADS, 0, st>>>(partial, nb, 1, 1, value_out);
        e = cudaGetLastError();
    }
    return e;
}

// Failure-detection self-test: one warp waits on a shared-memory barrier that nothing completes,
// with a bound of `polls` polls; the wait gives up, the timeout goes into the status word and the
// kernel returns normally (no trap, nothing in flight).
__global__ void wait_selftest_kernel(uint32_t polls, int* status) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncwarp();
    const bool ok = mbar_wait_n(&bar, 0u, polls);
    __syncwarp();
    if (threadIdx.x == 0) {
        if (!ok) set_status(status, DEV_TIMEOUT);
        mbar_inval(&bar);
    }
}

cudaError_t launch_wait_selftest(uint32_t polls, int* status, cudaStream_t st) {
    wait_selftest_kernel<<<1, 32, 0, st>>>(polls, status);
    return cudaGetLastError();
}

}  // namespace gp
