// assa.cu -- the paper's discretised operator (Methods, adaptive supersampling alignment;
// Algorithm 1) for grid Gaussians sharing one width.  Each pair's time of flight is snapped to
// the nearest sample of a grid alpha times finer than fs, the pair's mass A / r accumulates at
// that sample, the impulse lines are convolved with the sampled pulse h and decimated back to
// fs.  The adjoint transposes each stage: zero filling, correlation with h, back-projection.
//
// Forward decomposition: as the exact forward (forward.cu), CTA = (slab of bricks, 8 sensors),
// one warp per sensor, bricks streamed through a ring of TMA-filled shared buffers.  Each warp
// keeps its sensor's impulse line over the slab's band on the fine grid in shared memory and
// adds every pair's mass there with a shared-memory atomic; after the slab it convolves and
// decimates the band into the slab's partial row (summed over slabs by slab_reduce_kernel).
// The adds are 32-bit integer adds of the mass in fixed point, which the shared-memory units
// execute at about twice the rate of float adds.  A warp scales its masses by
// q = ASSA_QMAX d_min / max|A|, d_min the sensor's distance to the slab's box, so that each
// scaled mass is below ASSA_QMAX = 2^19 in magnitude, and every ASSA_FLUSH bricks (at most
// 2^12 pairs) it converts the integer band into a float band and clears it: no band value can
// leave the int32 range, and each mass is rounded to 2^-19 of the largest.  A warp whose sensor
// touches the slab's box, or a non-finite max|A|, keeps float adds.
// Adjoint: the correlated residual dconv_j[k] = sum_n h[alpha n - k] delta_j[n] is formed once
// per sensor (assa_dconv_kernel); then one thread per Gaussian gathers dconv at its snapped
// samples over all sensors, Kahan-compensated, and writes its gradient once.
#include <cuda.h>

#include <cmath>
#include <cstring>
#include <type_traits>

#include "adjoint_split.cuh"
#include "gpair_internal.cuh"

namespace gp {

constexpr int ASSA_SPC = 8;
constexpr int ASSA_THREADS = 32 * ASSA_SPC;
constexpr int ASSA_RING = 4;
constexpr float ASSA_QMAX = 0.99f * 524288.f;      // 0.99 * 2^19: bound of a scaled mass
constexpr int ASSA_FLUSH = 16;                     // bricks per integer band (16 * 256 = 2^12 pairs)

struct AssaSmem {
    float tileA[ASSA_RING][TILE];
    uint64_t full[ASSA_RING];
    int released[ASSA_RING];
    int issued[ASSA_RING];
    int abort;
};
constexpr size_t ASSA_HDR = (sizeof(AssaSmem) + 127) & ~(size_t)127;

// Impulse band of one (slab, sensor) on the fine grid: samples alpha w - K .. alpha (w + LB - 1) + K.
__host__ __device__ __forceinline__ int assa_zb(int LB, int alpha, int K) { return (alpha * LB + 2 * K + 3) & ~3; }

// Snapping by the float representation: for |x| < 2^22, x + 1.5 * 2^23 rounds to the nearest
// integer in the float's mantissa, so its bits minus SNAP_BITS are that integer: round(x), which is
// floor(x + 1/2) except at exact ties (rounded to even there; the oracle bounds tie decisions).
constexpr float SNAP_MAGIC = 12582912.f;           // 1.5 * 2^23
constexpr unsigned SNAP_BITS = 0x4B400000u;         // its bits

// Snapped fine sample of a pair, alpha n0 + round(phi alpha / Delta): base = alpha n0 - SNAP_BITS
// (wrapping).
__device__ __forceinline__ int assa_snap(float phi, float aInvD, unsigned base) {
    return (int)((unsigned)__float_as_int(fmaf(phi, aInvD, SNAP_MAGIC)) + base);
}

// alpha n0, clamped far outside any record (the snapped sample then fails the range tests).
__device__ __forceinline__ int assa_an0(int alpha, int n0) {
    const long long an = (long long)alpha * n0;
    return (int)max(min(an, (long long)(1 << 30)), -(long long)(1 << 30));
}

// max |A| over the amplitudes, as the bits of a non-negative float (ordered like the floats;
// a NaN amplitude gives a NaN).  *out must be zero before the launch.
__global__ void assa_amax_kernel(const float* __restrict__ A, int64_t M, unsigned* __restrict__ out) {
    unsigned m = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, (unsigned)__float_as_int(fabsf(A[i])));
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

__global__ void __launch_bounds__(ASSA_THREADS)
assa_fwd_kernel(GaussDev g, ArrDev a, const SlabInfo* __restrict__ slabs, float* __restrict__ partial,
                int2* __restrict__ rows, int LB, int* status, int use_tma, const __grid_constant__ CUtensorMap tmap,
                const __grid_constant__ AssaTable T, const unsigned* __restrict__ amax_bits) {
    static_assert(BX == 8 && BY == 8 && BZ == 4 && TILE == 256,
                  "lane offsets below assume lane + 32 q -> (lane & 7, (lane >> 3) + 4 (q & 1), q >> 1)");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    AssaSmem& S = *reinterpret_cast<AssaSmem*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int alpha = T.alpha, K = T.K;
    const int ZB = assa_zb(LB, alpha, K);
    float* zb = reinterpret_cast<float*>(smem_raw + ASSA_HDR) + (size_t)warp * 2 * ZB;   // float band
    int* zi = reinterpret_cast<int*>(zb + ZB);                                          // fixed-point band

    const int slab = blockIdx.y;
    const int j = blockIdx.x * ASSA_SPC + warp;
    const bool has_sensor = j < a.Nd;
    const SlabInfo sl = slabs[slab];
    const int nTiles = sl.t_end - sl.t_begin;
    const size_t row = (size_t)slab * a.Nd + (has_sensor ? j : 0);
    float* prow = partial + row * LB;
    const int Nup = alpha * a.Nt;

    // the slab's sample band for this sensor; a.k * sigma covers the pulse half-width plus half
    // a fine step of snapping
    float sx = 0.f, sy = 0.f, sz = 0.f;
    int n_lo = 0, n_hi = -1;
    float qscale = 0.f;                    // 0: float adds
    if (has_sensor) {
        sx = a.xyz[3 * j]; sy = a.xyz[3 * j + 1]; sz = a.xyz[3 * j + 2];
        if (nTiles > 0) {
            double dmin, dmax;
            box_distance(sl, sx, sy, sz, dmin, dmax);
            const float amax = __int_as_float((int)*amax_bits);
            if (amax > 0.f && amax <= 3.0e38f && dmin > 0.0) qscale = (float)((double)ASSA_QMAX * dmin / (double)amax);
            double ks = (double)a.k * sl.smax;
            double lo = floor(((dmin - ks) / a.v - a.t0) * a.fs) - 2.0;
            double hi = ceil(((dmax + ks) / a.v - a.t0) * a.fs) + 2.0;
            if (lo < 0) lo = 0;
            if (hi > a.Nt - 1) hi = a.Nt - 1;
            if (lo <= hi) { n_lo = (int)lo; n_hi = (int)hi; }
        }
    }
    const int w = n_lo & ~3;
    bool active = has_sensor && n_lo <= n_hi;
    if (active && n_hi + 1 - w > LB) {     // cannot happen with the host's band bound
        set_status(status, DEV_CAPACITY);
        n_hi = w + LB - 1;
    }
    if (lane == 0 && has_sensor) rows[row] = make_int2(w, active ? min(LB, a.Nt - w) : 0);
    if (threadIdx.x == 0) {
        S.abort = 0;
        for (int b = 0; b < ASSA_RING; ++b) {
            S.released[b] = 0;
            S.issued[b] = -1;
            mbar_init(&S.full[b], 1);
        }
        fence_mbar_init();
    }
    for (int q = lane; q < ZB; q += 32) {
        zb[q] = 0.f;
        zi[q] = 0;
    }
    const bool fixedp = qscale > 0.f;     // warp-uniform
    const float inv_q = fixedp ? 1.f / qscale : 0.f;
    // integer band -> float band, cleared for the next bricks
    auto flush = [&]() {
        __syncwarp();
        for (int q = lane; q < ZB; q += 32) {
            const int v = zi[q];
            if (v != 0) {
                zb[q] = fmaf((float)v, inv_q, zb[q]);
                zi[q] = 0;
            }
        }
        __syncwarp();
    };
    __syncthreads();

    const bool tma = use_tma != 0;
    auto fill = [&](int TT) {
        const int b = TT % ASSA_RING;
        int tx, ty, tz;
        slab_brick(sl, TT, tx, ty, tz);
        if (tma) {
            if (lane == 0) {
                S.issued[b] = TT;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive_expect_tx(&S.full[b], TILE * sizeof(float));
                tma_load_3d(&S.tileA[b][0], &tmap, tx * BX, ty * BY, tz * BZ, &S.full[b]);
            }
        } else {
            for (int q = lane; q < TILE; q += 32) {
                const int gx = tx * BX + (q & (BX - 1)), gy = ty * BY + ((q / BX) & (BY - 1)), gz = tz * BZ + q / (BX * BY);
                const bool ok = gx < g.nx && gy < g.ny && gz < g.nz;
                S.tileA[b][q] = ok ? g.A[((int64_t)gz * g.ny + gy) * g.nx + gx] : 0.f;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.full[b]);
        }
    };
    if (warp == 0)
        for (int TT = 0; TT < ASSA_RING && TT < nTiles; ++TT) fill(TT);

    const float aInvD = (float)alpha * a.invDelta;     // fine samples per metre
    const int kb0 = alpha * w - K;                     // fine sample at zb[0]
    const float h = g.h;
    const float ox = ((float)(lane & 7) - 0.5f * (BX - 1)) * h;
    const float oy0 = ((float)(lane >> 3) - 0.5f * (BY - 1)) * h;
    const float oy1 = ((float)((lane >> 3) + 4) - 0.5f * (BY - 1)) * h;

    PairRef refs;
    int t = 0;
    bool ok = true;
    for (; t < nTiles; ++t) {
        const int b = t % ASSA_RING;
        if (!mbar_wait(&S.full[b], (uint32_t)((t / ASSA_RING) & 1))) {
            ok = false;
            break;
        }
        if (active) {
            if ((t & 31) == 0 && t + lane < nTiles) {
                int tx, ty, tz;
                slab_brick(sl, t + lane, tx, ty, tz);
                refs = make_ref(g.ox + (tx * BX + BX / 2) * (double)g.h, g.oy + (ty * BY + BY / 2) * (double)g.h,
                                g.oz + (tz * BZ + BZ / 2) * (double)g.h, sx, sy, sz, a);
            }
            const int src = t & 31;
            PairRef r;
            r.v0x = __shfl_sync(0xffffffffu, refs.v0x, src);
            r.v0y = __shfl_sync(0xffffffffu, refs.v0y, src);
            r.v0z = __shfl_sync(0xffffffffu, refs.v0z, src);
            r.R0 = __shfl_sync(0xffffffffu, refs.R0, src);
            r.phi0 = __shfl_sync(0xffffffffu, refs.phi0, src);
            r.n0 = __shfl_sync(0xffffffffu, refs.n0, src);
            const unsigned base = (unsigned)assa_an0(alpha, r.n0) - SNAP_BITS;
            const float ax = ox * (2.f * r.v0x + ox);
            const float ay0 = oy0 * (2.f * r.v0y + oy0), ay1 = oy1 * (2.f * r.v0y + oy1);
#pragma unroll
            for (int q = 0; q < TILE / 32; ++q) {
                const float Ai = S.tileA[b][lane + 32 * q];
                const float oz = ((float)(q >> 1) - 0.5f * (BZ - 1)) * h;
                const float num = (ax + ((q & 1) ? ay1 : ay0)) + oz * (2.f * r.v0z + oz);
                float invR, phi;
                pair_phase_num(r, num, invR, phi);
                // snapped fine sample: floor((R / v - t0) alpha fs + 1/2) = alpha n0 + floor(phi alpha / Delta + 1/2)
                const int k = assa_snap(phi, aInvD, base);
                const int kb = k - kb0;
                if (Ai != 0.f && k >= 0 && k < Nup && kb >= 0 && kb < ZB) {
                    if (fixedp)   // round(A / r q): |.| < 2^19, so the float representation gives it
                        atomicAdd(&zi[kb], __float_as_int(fmaf(Ai * invR, qscale, SNAP_MAGIC)) - (int)SNAP_BITS);
                    else
                        atomicAdd(&zb[kb], Ai * invR);
                }
            }
            if (fixedp && (t + 1) % ASSA_FLUSH == 0) flush();
        }
        // release the slot; the warp that releases it last refills it with tile t + ASSA_RING
        __syncwarp();
        int last = 0;
        if (lane == 0) {
            __threadfence_block();
            last = (atomicAdd(&S.released[b], 1) + 1) % ASSA_SPC == 0;
            if (last) __threadfence_block();
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last && t + ASSA_RING < nTiles) fill(t + ASSA_RING);
    }
    if (!ok && lane == 0) {
        set_status(status, DEV_TIMEOUT);
        S.abort = 1;
    }
    __syncthreads();
    if (S.abort) {
        if (tma && threadIdx.x == 0)
            for (int b = 0; b < ASSA_RING; ++b)
                if (S.issued[b] >= 0) mbar_wait(&S.full[b], (uint32_t)((S.issued[b] / ASSA_RING) & 1));
        return;
    }
    if (active) {
        if (fixedp) flush();
        // y[n] = sum_m z[m] h[alpha n - m]; sample n = w + q needs zb[alpha q .. alpha q + 2K]
        const int wend = min(a.Nt, w + LB);
        for (int q = lane; q < wend - w; q += 32) {
            const float* zq = zb + (size_t)alpha * q;
            float y = 0.f;
            for (int tt = 0; tt <= 2 * K; ++tt) y = fmaf(zq[tt], T.hr[tt], y);   // h[alpha n - m] = h[K - tt]
            prow[q] = y;
        }
    }
}

// The forward with the lanes of a warp owning 32 sensors, for slabs of at most ASSA_FLUSH bricks.  All lanes
// take the same Gaussian; a lane adds its pair's mass, in fixed point as above, to an integer band of its
// own, [sample][lane] in shared memory: 32 different banks whatever samples the lanes address, and a
// shared-memory add that nothing waits for.  The band holds the fine samples between the
// sensor's nearest and farthest distance to the slab, not the pulse's margins; an impulse outside the
// record goes to the entry after the last.  After the slab a lane scales its band to floats and
// convolves it, eight outputs at a time over a window of registers.  A lane whose masses have no bound
// (sensor in the slab's box, amplitudes not finite) adds floats.
//
// Bound by the MUFU pipe (two operations a pair) and instruction issue; with a warp to a sensor the
// lanes' samples met in the same banks and every pair had its own range tests (48 instructions a
// pair).  1.07e9 pairs: 1.71 ms, 0.89 ms now.
constexpr int ASSA_LANES_MAXW = 4, ASSA_LANES_Q = 8;

struct AssaLanesHdr {
    float tileA[ASSA_RING][TILE];
    uint64_t full[ASSA_RING];
    int released[ASSA_RING];
    int issued[ASSA_RING];
    int abort;
};
constexpr size_t ASSA_LANES_HDR = (sizeof(AssaLanesHdr) + 127) & ~(size_t)127;

// Entries of a lane's band for a slab whose centres span `diag` metres.  The band starts up to two samples before
// the nearest distance to the slab's box, which lies up to `widened` metres before the nearest centre
// (brick_block): the six entries more than the span cover the first and a sample of the second.
int assa_lanes_nz(double diag, double widened, double invDelta, int alpha) {
    const double fine = invDelta * alpha, extra = fmax(0.0, ceil(widened * fine) - 1.0);
    return (int)fmin(ceil(diag * 1.00001 * fine) + 6.0 + extra, (double)(1 << 24));
}
size_t assa_lanes_smem(int NW, int NZ) { return ASSA_LANES_HDR + (size_t)NW * (NZ + 1) * 32 * sizeof(int); }

// Slabs of sb bricks that divide the blocks of qb bricks in which the kernel above walks the lattice: a slab's masses
// take its block's scale, so that both kernels round each mass alike.  kx x ky slabs across.
struct AssaSlabs {
    int sb[3], qb[3], kx, ky;
};

__global__ void __launch_bounds__(ASSA_LANES_MAXW * 32, 2)
assa_fwd_lanes_kernel(GaussDev g, ArrDev a, const AssaSlabs slabs, float* __restrict__ partial,
                      int2* __restrict__ rows, int LB, int NZ, int* status, int use_tma,
                      const __grid_constant__ CUtensorMap tmap, const __grid_constant__ AssaTable T,
                      const unsigned* __restrict__ amax_bits) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    AssaLanesHdr& S = *reinterpret_cast<AssaLanesHdr*>(smem_raw);
    const int NW = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int* Z = reinterpret_cast<int*>(smem_raw + ASSA_LANES_HDR) + (size_t)warp * (NZ + 1) * 32 + lane;    // [entry * 32]
    const int alpha = T.alpha, K = T.K;
    const int j = (blockIdx.x * NW + warp) * 32 + lane;
    const bool has_sensor = j < a.Nd;
    const size_t row = (size_t)blockIdx.y * a.Nd + (has_sensor ? j : 0);
    const int Nup = alpha * a.Nt;
    // this CTA's slab and its block
    const int si[3] = {(int)(blockIdx.y % slabs.kx), (int)(blockIdx.y / slabs.kx % slabs.ky), (int)(blockIdx.y / (slabs.kx * slabs.ky))};
    const int nt[3] = {g.ntx, g.nty, g.ntz};
    int b0[3], bd[3], q0[3], qd[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int per = (slabs.qb[q] + slabs.sb[q] - 1) / slabs.sb[q], sub = si[q] % per * slabs.sb[q];
        q0[q] = si[q] / per * slabs.qb[q];
        qd[q] = min(slabs.qb[q], nt[q] - q0[q]);
        b0[q] = q0[q] + sub;
        bd[q] = min(slabs.sb[q], qd[q] - sub);
    }
    if (bd[0] <= 0 || bd[1] <= 0 || bd[2] <= 0) {          // past the block's end at a ragged face
        if (has_sensor) rows[row] = make_int2(0, 0);
        return;
    }
    const SlabInfo sl = brick_block(g, b0[0], b0[1], b0[2], bd[0], bd[1], bd[2]);
    const int nTiles = sl.t_end;

    // the lane's samples of the slab, [w, w + LBe), and its impulses' fine samples, [lo, lo + cnt)
    float sx = 0.f, sy = 0.f, sz = 0.f, qscale = 0.f;
    int n_lo = 0, n_hi = -1, lo = 0, cnt = 0;
    if (has_sensor) {
        sx = a.xyz[3 * j]; sy = a.xyz[3 * j + 1]; sz = a.xyz[3 * j + 2];
        double dmin, dmax;
        box_distance(sl, sx, sy, sz, dmin, dmax);
        const float amax = __int_as_float((int)*amax_bits);
        double qmin, qmax;
        box_distance(brick_block(g, q0[0], q0[1], q0[2], qd[0], qd[1], qd[2]), sx, sy, sz, qmin, qmax);
        if (amax > 0.f && amax <= 3.0e38f && qmin > 0.0) qscale = (float)((double)ASSA_QMAX * qmin / (double)amax);
        const double ks = (double)a.k * sl.smax;
        double l = floor(((dmin - ks) / a.v - a.t0) * a.fs) - 2.0;
        double u = ceil(((dmax + ks) / a.v - a.t0) * a.fs) + 2.0;
        if (l < 0) l = 0;
        if (u > a.Nt - 1) u = a.Nt - 1;
        if (l <= u) { n_lo = (int)l; n_hi = (int)u; }
        const double k0 = fmin(fmax(floor((dmin / a.v - a.t0) * a.fs * alpha) - 1.0, -1073741824.0), 1073741824.0);
        lo = max((int)k0, 0);
        cnt = max(0, min((int)k0 + NZ, Nup) - lo);
    }
    const int w = n_lo & ~3;
    bool active = has_sensor && n_lo <= n_hi;
    if (active && n_hi + 1 - w > LB) {     // cannot happen with the host's band bound
        set_status(status, DEV_CAPACITY);
        n_hi = w + LB - 1;
    }
    const int LBe = active ? min(min(LB, a.Nt - w), n_hi + 1 - w) : 0;
    if (has_sensor) rows[row] = make_int2(w, LBe);
    if (threadIdx.x == 0) {
        S.abort = 0;
        for (int b = 0; b < ASSA_RING; ++b) {
            S.released[b] = 0;
            S.issued[b] = -1;
            mbar_init(&S.full[b], 1);
        }
        fence_mbar_init();
    }
    for (int q = 0; q <= NZ; ++q) Z[q * 32] = 0;       // 0 and 0.f
    const bool fixedp = qscale > 0.f;
    const bool all_fixed = __all_sync(0xffffffffu, fixedp || !active);
    const float inv_q = fixedp ? 1.f / qscale : 0.f;
    __syncthreads();

    const bool tma = use_tma != 0;
    auto fill = [&](int TT) {
        const int b = TT % ASSA_RING;
        int tx, ty, tz;
        slab_brick(sl, TT, tx, ty, tz);
        if (tma) {
            if (lane == 0) {
                S.issued[b] = TT;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive_expect_tx(&S.full[b], TILE * sizeof(float));
                tma_load_3d(&S.tileA[b][0], &tmap, tx * BX, ty * BY, tz * BZ, &S.full[b]);
            }
        } else {
            for (int q = lane; q < TILE; q += 32) {
                const int gx = tx * BX + (q & (BX - 1)), gy = ty * BY + ((q / BX) & (BY - 1)), gz = tz * BZ + q / (BX * BY);
                const bool ok = gx < g.nx && gy < g.ny && gz < g.nz;
                S.tileA[b][q] = ok ? g.A[((int64_t)gz * g.ny + gy) * g.nx + gx] : 0.f;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.full[b]);
        }
    };
    if (warp == 0)
        for (int TT = 0; TT < ASSA_RING && TT < nTiles; ++TT) fill(TT);

    auto both = [](float v) { return make_float2(v, v); };
    const float h = g.h;
    const float2 aD = both((float)alpha * a.invDelta), magic = both(SNAP_MAGIC), qs = both(qscale);
    bool ok = true, touched = false;
    for (int t = 0; t < nTiles; ++t) {
        const int b = t % ASSA_RING;
        if (!mbar_wait(&S.full[b], (uint32_t)((t / ASSA_RING) & 1))) {
            ok = false;
            break;
        }
        const float* tile = S.tileA[b];
        bool any = false;                  // a brick without amplitudes adds nothing
#pragma unroll
        for (int q = 0; q < TILE / 32 / 4; ++q) {
            const float4 v = reinterpret_cast<const float4*>(tile)[lane * (TILE / 32 / 4) + q];
            any |= (v.x != 0.f) | (v.y != 0.f) | (v.z != 0.f) | (v.w != 0.f);
        }
        if (__any_sync(0xffffffffu, any) && active) {
            touched = true;
            int tx, ty, tz;
            slab_brick(sl, t, tx, ty, tz);
            const PairRef r = make_ref(g.ox + (tx * BX + BX / 2) * (double)h, g.oy + (ty * BY + BY / 2) * (double)h,
                                       g.oz + (tz * BZ + BZ / 2) * (double)h, sx, sy, sz, a);
            const unsigned base = (unsigned)assa_an0(alpha, r.n0) - SNAP_BITS - (unsigned)lo;
            const float2 R0 = both(r.R0), phi0 = both(r.phi0);
            float2 ax[BX / 2];
#pragma unroll
            for (int l = 0; l < BX; ++l) {
                const float o = ((float)l - 0.5f * (BX - 1)) * h, v = o * fmaf(2.f, r.v0x, o);
                if (l & 1) ax[l >> 1].y = v; else ax[l >> 1].x = v;
            }
            auto brick = [&](auto fx) {
#pragma unroll 1
                for (int ly = 0; ly < BY; ++ly) {
                    const float oy = ((float)ly - 0.5f * (BY - 1)) * h;
                    const float2 oy2 = both(oy), Yc = both(fmaf(2.f, r.v0y, oy));
                    float2 axy[BX / 2];
#pragma unroll
                    for (int u = 0; u < BX / 2; ++u) axy[u] = __ffma2_rn(oy2, Yc, ax[u]);
#pragma unroll
                    for (int lz = 0; lz < BZ; ++lz) {
                        const float oz = ((float)lz - 0.5f * (BZ - 1)) * h;
                        const float2 az = both(__fmul_rn(oz, fmaf(2.f, r.v0z, oz)));
                        const float4 a0 = *reinterpret_cast<const float4*>(tile + (lz * BY + ly) * BX);
                        const float4 a1 = *reinterpret_cast<const float4*>(tile + (lz * BY + ly) * BX + 4);
                        const float2 A[BX / 2] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), make_float2(a1.x, a1.y),
                                                  make_float2(a1.z, a1.w)};
#pragma unroll
                        for (int u = 0; u < BX / 2; ++u) {
                            const float2 num = __fadd2_rn(axy[u], az);
                            const float2 R2 = __ffma2_rn(R0, R0, num);
                            const float2 invR = make_float2(rsqrtf(R2.x), rsqrtf(R2.y));
                            const float2 den = __ffma2_rn(R2, invR, R0);
                            float2 rc;
                            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc.x) : "f"(den.x));
                            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc.y) : "f"(den.y));
                            const float2 k = __ffma2_rn(__ffma2_rn(num, rc, phi0), aD, magic);
                            int* z0 = Z + min((unsigned)__float_as_int(k.x) + base, (unsigned)cnt) * 32u;
                            int* z1 = Z + min((unsigned)__float_as_int(k.y) + base, (unsigned)cnt) * 32u;
                            const float2 mass = __fmul2_rn(A[u], invR);
                            if (fx) {
                                const float2 q = __ffma2_rn(mass, qs, magic);
                                atomicAdd(z0, __float_as_int(q.x) - (int)SNAP_BITS);
                                atomicAdd(z1, __float_as_int(q.y) - (int)SNAP_BITS);
                            } else if (fixedp) {
                                const float2 q = __ffma2_rn(mass, qs, magic);
                                *z0 += __float_as_int(q.x) - (int)SNAP_BITS;
                                *z1 += __float_as_int(q.y) - (int)SNAP_BITS;
                            } else {
                                if (A[u].x != 0.f) *z0 = __float_as_int(__int_as_float(*z0) + mass.x);
                                if (A[u].y != 0.f) *z1 = __float_as_int(__int_as_float(*z1) + mass.y);
                            }
                        }
                    }
                }
            };
            if (all_fixed) brick(std::true_type{}); else brick(std::false_type{});
        }
        // release the slot; the warp that releases it last refills it with tile t + ASSA_RING
        __syncwarp();
        int last = 0;
        if (lane == 0) {
            __threadfence_block();
            last = (atomicAdd(&S.released[b], 1) + 1) % NW == 0;
            if (last) __threadfence_block();
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last && t + ASSA_RING < nTiles) fill(t + ASSA_RING);
    }
    if (!ok && lane == 0) {
        set_status(status, DEV_TIMEOUT);
        S.abort = 1;
    }
    __syncthreads();
    if (S.abort) {
        if (tma && threadIdx.x == 0)
            for (int b = 0; b < ASSA_RING; ++b)
                if (S.issued[b] >= 0) mbar_wait(&S.full[b], (uint32_t)((S.issued[b] / ASSA_RING) & 1));
        return;
    }
    if (!active) return;
    if (!touched) {            // a slab without amplitudes: an empty row
        rows[row] = make_int2(w, 0);
        return;
    }
    float* F = reinterpret_cast<float*>(Z);
    for (int q = 0; q <= NZ; ++q) F[q * 32] = q < cnt ? (fixedp ? (float)Z[q * 32] * inv_q : F[q * 32]) : 0.f;
    // y[n] = sum_m z[m] h[alpha n - m]: output w + q sums entries alpha (w + q) - K - lo + tt, tt = 0 .. 2K, the
    // taps tt = c, c + alpha, ... of one residue c at a time, so that the next tap's entries are this tap's
    // shifted by one output
    float4* prow = reinterpret_cast<float4*>(partial + row * LB);
    for (int q0 = 0; q0 < LBe; q0 += ASSA_LANES_Q) {
        float acc[ASSA_LANES_Q];
#pragma unroll
        for (int u = 0; u < ASSA_LANES_Q; ++u) acc[u] = 0.f;
        for (int c = 0; c < alpha; ++c) {
            int at = alpha * (w + q0) - K - lo + c;
            auto entry = [&] {
                const float v = F[min((unsigned)at, (unsigned)NZ) * 32u];        // entry NZ is zero
                at += alpha;
                return v;
            };
            float V[ASSA_LANES_Q];
#pragma unroll
            for (int u = 0; u < ASSA_LANES_Q - 1; ++u) V[u] = entry();
            for (int tt = c; tt <= 2 * K;) {
#pragma unroll
                for (int i = 0; i < ASSA_LANES_Q; ++i, tt += alpha) {
                    if (tt > 2 * K) break;
                    V[(i + ASSA_LANES_Q - 1) % ASSA_LANES_Q] = entry();
                    const float hv = T.hr[tt];                                 // h[alpha n - m] = h[K - tt]
#pragma unroll
                    for (int u = 0; u < ASSA_LANES_Q; ++u) acc[u] = fmaf(V[(i + u) % ASSA_LANES_Q], hv, acc[u]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < ASSA_LANES_Q; u += 4)          // LB is a multiple of 4; outputs past LBe are not read
            if (q0 + u < LBe) prow[(q0 + u) >> 2] = make_float4(acc[u], acc[u + 1], acc[u + 2], acc[u + 3]);
    }
}

// A sensor's row of dconv: its alpha N_t fine samples and a zero.
__host__ __device__ __forceinline__ int assa_dconv_row(int alpha, int Nt) { return alpha * Nt + 1; }

// dconv_j[k] = sum_n h[alpha n - k] delta_j[n], k = 0 .. alpha Nt - 1 (zero filling and the
// correlation with the flipped pulse in one pass).  The outputs of one residue, k = alpha q + r, are a filter of delta
// with taps of their own: a block takes DC_PER samples q from each of its threads, residue by residue, so that
// the taps are uniform and serve DC_PER outputs each.  4.2e6 samples, alpha = 2: 87 us with a thread to an
// output, 28 us.
constexpr int DC_THREADS = 256, DC_PER = 4;
__device__ __forceinline__ int floor_div(int a, int b) { return (a >= 0) ? a / b : -((-a + b - 1) / b); }

__global__ void __launch_bounds__(DC_THREADS)
assa_dconv_kernel(const float* __restrict__ delta, int Nt, const __grid_constant__ AssaTable T,
                  float* __restrict__ dconv) {
    extern __shared__ float sd[];                  // samples q0 - M .. q0 + DC_THREADS DC_PER + M
    const int j = blockIdx.y, t = threadIdx.x;
    const int alpha = T.alpha, K = T.K, M = K / alpha + 1;
    const int q0 = blockIdx.x * DC_THREADS * DC_PER;
    const float* dj = delta + (size_t)j * Nt;
    for (int c = t; c < DC_THREADS * DC_PER + 2 * M + 1; c += DC_THREADS) {
        const int n = q0 - M + c;
        sd[c] = (n >= 0 && n < Nt) ? dj[n] : 0.f;
    }
    __syncthreads();
    float* row = dconv + (size_t)j * assa_dconv_row(alpha, Nt);
    for (int r = 0; r < alpha; ++r) {
        const int i1 = -floor_div(-(r - K), alpha), i2 = (r + K) / alpha;      // n - q with |alpha n - k| <= K
        float acc[DC_PER];
#pragma unroll
        for (int u = 0; u < DC_PER; ++u) acc[u] = 0.f;
        for (int i = i1; i <= i2; ++i) {
            const float h = T.hr[K - alpha * i + r];
#pragma unroll
            for (int u = 0; u < DC_PER; ++u) acc[u] = fmaf(h, sd[t + u * DC_THREADS + M + i], acc[u]);
        }
#pragma unroll
        for (int u = 0; u < DC_PER; ++u) {
            const int q = q0 + t + u * DC_THREADS;
            if (q < Nt) row[(size_t)alpha * q + r] = acc[u];
        }
    }
    if (blockIdx.x == 0 && t == 0) row[(size_t)alpha * Nt] = 0.f;      // the entry of every sample outside the record
}

size_t assa_dconv_smem(const AssaTable& T) { return (size_t)(DC_THREADS * DC_PER + 2 * (T.K / T.alpha + 1) + 1) * sizeof(float); }

// g_i = sum_j dconv_j[k_ij] / r_ij.  One CTA of 64 threads per brick, four Gaussians to a thread (x and
// x + 4, two planes each; the planes through packed FP32 arithmetic, which rounds each half as the scalar
// operation does).  The FP64 references of a chunk of 64 sensors, one to a thread, are
// double-buffered.  A snapped sample outside the record reads the sensor's zero entry, one past its end.
// A brick's sensors may be divided over the CTAs of a cluster.
//
// A node on which a sensor lies has no time of flight and adds nothing.  It reads the zero entry, but 0 / 0 is not
// a number: a CTA that finds such a sum gathers again, dropping 1 / R at the zero entry (CHECK).
//
// Bound by instruction issue.  With a Gaussian to a thread 25 instructions a pair; 1.07e9 pairs: 955 us, 771 us now.
constexpr int ASSA_ADJ_THREADS = 64, ASSA_ADJ_PER = TILE / ASSA_ADJ_THREADS, ASSA_ADJ_CTAS = 14;
constexpr int ASSA_ADJ_SC = 64;
struct __align__(16) AssaRef {
    float v2x, v2y, v2z, R0;     // 2 (c0 - s), |c0 - s|
    float phi0;
    unsigned base;               // alpha n0 - SNAP_BITS (wrapping)
    const float* row;            // the sensor's row of dconv
};
static_assert(sizeof(AssaRef) == 32, "two 16-byte loads");

template <bool SPLIT>
__global__ void __launch_bounds__(ASSA_ADJ_THREADS, ASSA_ADJ_CTAS)
assa_adj_kernel(GaussDev g, ArrDev a, const float* __restrict__ dconv, const __grid_constant__ AssaTable T,
                float* __restrict__ gA, int per) {
    __shared__ AssaRef refs2[2][ASSA_ADJ_SC];
    __shared__ float part[SPLIT ? TILE : 1];
    const int64_t t = blockIdx.x;
    const int l = threadIdx.x;
    const int tx = (int)(t % g.ntx), ty = (int)((t / g.ntx) % g.nty), tz = (int)(t / ((int64_t)g.ntx * g.nty));
    // a warp takes a 4 x 4 x 2 block of nodes per gather (planes 0 and 2, or 1 and 3), so that the snapped
    // positions of its 32 Gaussians for one sensor -- the residual entries it gathers -- stay close together
    static_assert(BX == 8 && BY == 8 && BZ == 4 && ASSA_ADJ_THREADS == 64, "brick of 8 x 8 x 4, 2 warps");
    const int lx = l & 3, ly = ((l >> 2) & 3) | (((l >> 5) & 1) << 2), lz = ((l >> 4) & 1) << 1;
    const int alpha = T.alpha, Nt = a.Nt;
    const float aInvD = (float)alpha * a.invDelta;
    const float dx0 = ((float)lx - 0.5f * (BX - 1)) * g.h, dx1 = ((float)(lx + 4) - 0.5f * (BX - 1)) * g.h;
    const float dy = ((float)ly - 0.5f * (BY - 1)) * g.h;
    const float2 dz = make_float2(((float)lz - 0.5f * (BZ - 1)) * g.h, ((float)(lz + 1) - 0.5f * (BZ - 1)) * g.h);
    const float2 dx[2] = {make_float2(dx0, dx0), make_float2(dx1, dx1)}, dy2 = make_float2(dy, dy);
    float2 d2[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) d2[u] = __ffma2_rn(dx[u], dx[u], __ffma2_rn(dy2, dy2, __fmul2_rn(dz, dz)));
    const double c0x = g.ox + (tx * BX + BX / 2) * (double)g.h;
    const double c0y = g.oy + (ty * BY + BY / 2) * (double)g.h;
    const double c0z = g.oz + (tz * BZ + BZ / 2) * (double)g.h;
    const unsigned zero_entry = (unsigned)(alpha * Nt);
    auto ref = [&](int j) {
        const PairRef p = ref_doubled(make_ref(c0x, c0y, c0z, a.xyz[3 * j], a.xyz[3 * j + 1], a.xyz[3 * j + 2], a));
        AssaRef r;
        r.v2x = p.v0x; r.v2y = p.v0y; r.v2z = p.v0z;
        r.R0 = p.R0;
        r.phi0 = p.phi0;
        r.base = (unsigned)assa_an0(alpha, p.n0) - SNAP_BITS;         // see assa_snap
        r.row = dconv + (size_t)j * assa_dconv_row(alpha, Nt);
        return r;
    };
    auto both = [](float v) { return make_float2(v, v); };
    const float2 magic = both(SNAP_MAGIC), aD = both(aInvD);
    KahanF kA[ASSA_ADJ_PER];         // FP32 over 32 sensors, compensated from there on
    const int jb = SPLIT ? blockIdx.y * per : 0, je = SPLIT ? min(a.Nd, jb + per) : a.Nd;
    auto gather = [&](auto CHECK) {
#pragma unroll
        for (int u = 0; u < ASSA_ADJ_PER; ++u) kA[u] = KahanF();
        if (jb + l < je) refs2[0][l] = ref(jb + l);
        int cur = 0;
        for (int j0 = jb; j0 < je; j0 += ASSA_ADJ_SC, cur ^= 1) {
            const int nsc = min(ASSA_ADJ_SC, je - j0);
            __syncthreads();
            if (j0 + ASSA_ADJ_SC + l < je) refs2[cur ^ 1][l] = ref(j0 + ASSA_ADJ_SC + l);
            for (int q0 = 0; q0 < nsc; q0 += 32) {
                float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                const AssaRef* rp = refs2[cur] + q0;
                const int nq = min(32, nsc - q0);
#pragma unroll 4
                for (int q = 0; q < nq; ++q) {
                    const AssaRef r = rp[q];
                    const float2 R0 = both(r.R0);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const float2 num = __ffma2_rn(dx[u], both(r.v2x), __ffma2_rn(dy2, both(r.v2y), __ffma2_rn(dz, both(r.v2z), d2[u])));
                        const float2 R2 = __ffma2_rn(R0, R0, num);
                        float2 iR = make_float2(rsqrtf(R2.x), rsqrtf(R2.y));
                        const float2 den = __ffma2_rn(R2, iR, R0);
                        float2 rc;
                        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc.x) : "f"(den.x));
                        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc.y) : "f"(den.y));
                        const float2 s = __ffma2_rn(__ffma2_rn(num, rc, both(r.phi0)), aD, magic);
                        const unsigned ka = min((unsigned)__float_as_int(s.x) + r.base, zero_entry);
                        const unsigned kb = min((unsigned)__float_as_int(s.y) + r.base, zero_entry);
                        if (CHECK) {
                            if (ka == zero_entry) iR.x = 0.f;
                            if (kb == zero_entry) iR.y = 0.f;
                        }
                        acc[u] = __ffma2_rn(make_float2(__ldg(r.row + ka), __ldg(r.row + kb)), iR, acc[u]);
                    }
                }
                kA[0].add(acc[0].x); kA[1].add(acc[0].y);
                kA[2].add(acc[1].x); kA[3].add(acc[1].y);
            }
        }
    };
    gather(std::false_type{});
    bool nan = false;
#pragma unroll
    for (int u = 0; u < ASSA_ADJ_PER; ++u) nan |= kA[u].s != kA[u].s;
    if (__syncthreads_or(nan)) gather(std::true_type{});
    float sum[ASSA_ADJ_PER];
#pragma unroll
    for (int u = 0; u < ASSA_ADJ_PER; ++u) sum[u] = kA[u].s;
    if constexpr (SPLIT)
        if (!split_sum<ASSA_ADJ_PER>(sum, part, l)) return;
#pragma unroll
    for (int u = 0; u < ASSA_ADJ_PER; ++u) {
        const int gx = tx * BX + lx + (u >> 1) * 4, gy = ty * BY + ly, gz = tz * BZ + lz + (u & 1);
        if (gx < g.nx && gy < g.ny && gz < g.nz) gA[((int64_t)gz * g.ny + gy) * g.nx + gx] = sum[u];
    }
}

// ---- host side -----------------------------------------------------------------------------

size_t assa_fwd_smem(int LB, const AssaTable& T) {
    return ASSA_HDR + (size_t)ASSA_SPC * 2 * assa_zb(LB, T.alpha, T.K) * sizeof(float);
}

// ev (optional): two events recorded immediately before and after the main kernel.  amax: 4 bytes
// of device scratch for max |A|.
cudaError_t launch_assa_forward(const GaussDev& g, const ArrDev& a, const SlabInfo* si, int S, float* partial,
                                int2* rows, int LB, int* status, const CUtensorMap* tmap, const AssaTable& T,
                                unsigned* amax, const cudaEvent_t* ev, cudaStream_t st) {
    static const CUtensorMap zero_map = [] { CUtensorMap z; memset(&z, 0, sizeof(z)); return z; }();
    const size_t smem = assa_fwd_smem(LB, T);
    cudaError_t e = cudaFuncSetAttribute(assa_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(amax, 0, sizeof(unsigned), st)) != cudaSuccess) return e;
    assa_amax_kernel<<<4 * device_sms(), 256, 0, st>>>(g.A, g.M, amax);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    dim3 grid((a.Nd + ASSA_SPC - 1) / ASSA_SPC, S);
    if (ev && (e = cudaEventRecord(ev[0], st)) != cudaSuccess) return e;
    assa_fwd_kernel<<<grid, ASSA_THREADS, smem, st>>>(g, a, si, partial, rows, LB, status, tmap != nullptr,
                                                      tmap ? *tmap : zero_map, T, amax);
    e = cudaGetLastError();
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[1], st);
    return e;
}

// The same by the lanes kernel: S rows a sensor, slabs of sb bricks in blocks of qb, NW warps and NZ entries a lane.
cudaError_t launch_assa_forward_lanes(const GaussDev& g, const ArrDev& a, const int sb[3], const int qb[3], int S,
                                      float* partial, int2* rows, int LB, int NW, int NZ, int* status,
                                      const CUtensorMap* tmap, const AssaTable& T, unsigned* amax, const cudaEvent_t* ev,
                                      cudaStream_t st) {
    static const CUtensorMap zero_map = [] { CUtensorMap z; memset(&z, 0, sizeof(z)); return z; }();
    const size_t smem = assa_lanes_smem(NW, NZ);
    cudaError_t e = cudaFuncSetAttribute(assa_fwd_lanes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(amax, 0, sizeof(unsigned), st)) != cudaSuccess) return e;
    assa_amax_kernel<<<4 * device_sms(), 256, 0, st>>>(g.A, g.M, amax);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    AssaSlabs s;
    const int nt[3] = {g.ntx, g.nty, g.ntz};
    int k[3];
    for (int q = 0; q < 3; ++q) {
        s.sb[q] = sb[q];
        s.qb[q] = qb[q];
        k[q] = (nt[q] + qb[q] - 1) / qb[q] * ((qb[q] + sb[q] - 1) / sb[q]);
    }
    s.kx = k[0]; s.ky = k[1];
    if (ev && (e = cudaEventRecord(ev[0], st)) != cudaSuccess) return e;
    assa_fwd_lanes_kernel<<<dim3((a.Nd + 32 * NW - 1) / (32 * NW), S), 32 * NW, smem, st>>>(
        g, a, s, partial, rows, LB, NZ, status, tmap != nullptr, tmap ? *tmap : zero_map, T, amax);
    e = cudaGetLastError();
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[1], st);
    return e;
}

size_t assa_dconv_bytes(const ArrDev& a, const AssaTable& T) { return (size_t)a.Nd * assa_dconv_row(T.alpha, a.Nt) * sizeof(float); }

cudaError_t launch_assa_adjoint(const GaussDev& g, const ArrDev& a, const float* delta, float* gA, const AssaTable& T,
                                float* dconv, const cudaEvent_t* ev, cudaStream_t st) {
    dim3 dgrid((a.Nt + DC_THREADS * DC_PER - 1) / (DC_THREADS * DC_PER), a.Nd);
    assa_dconv_kernel<<<dgrid, DC_THREADS, assa_dconv_smem(T), st>>>(delta, a.Nt, T, dconv);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (ev && (e = cudaEventRecord(ev[0], st)) != cudaSuccess) return e;
    const int split = adj_split_rows(g.ntiles, a.Nd);
    e = launch_split(split > 1 ? assa_adj_kernel<true> : assa_adj_kernel<false>, (unsigned)g.ntiles, split, ASSA_ADJ_THREADS, 0, st, g, a, (const float*)dconv, T,
                     gA, (a.Nd + split - 1) / split);
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[1], st);
    return e;
}

}  // namespace gp
