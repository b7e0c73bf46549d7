// spatial_order.cu -- a spatially compact order of free-centre Gaussians for the forward: the
// Morton order of their centres in the set's bounding box, so that the 256 consecutive Gaussians
// of a tile lie close together and the sensor-lane kernel's sample bands stay short.  The
// forward is a sum over Gaussians, so the order changes its result only by FP32 summation order.
//
// The order is a stable sort of 18-bit Morton keys (64 cells per axis, finer than a tile of 256
// Gaussians needs): equal keys keep their index order, so the result is deterministic.
// Up to SO_ONE_MAX Gaussians one CTA does all of it, a bitonic sort of (key, index) words in shared
// memory: seven launches less.  Larger sets go through an LSD radix sort in two passes of 9 bits:
// per-block digit counts, a scan of each digit's counts over the blocks, and a scatter whose
// ranks inside a block follow the index order through warp-level match masks.  Then one gather
// writes the permuted centres, widths and amplitudes.
//
// Latency and launches bound it at every size in use.  262,144 Gaussians: 131 us with blocks of 4096
// keys (64 CTAs) and one CTA scanning all counts, 46 us now; 1500: 57 us, 20 us now.
#include <cfloat>

#include "gpair_internal.cuh"

namespace gp {

constexpr int SO_THREADS = 256, SO_WARPS = SO_THREADS / 32;
constexpr int SO_BB_BLOCKS = 256;           // blocks of the bounding-box reduction
constexpr int SO_AXIS_BITS = 6;             // Morton key: 6 bits per axis
constexpr int SO_DIGIT = 9, SO_RADIX = 1 << SO_DIGIT, SO_PASSES = 3 * SO_AXIS_BITS / SO_DIGIT;
constexpr int SO_ONE_THREADS = 1024, SO_ONE_BITS = 13, SO_ONE_MAX = 1 << SO_ONE_BITS;
static_assert(SO_ONE_BITS + 3 * SO_AXIS_BITS < 32, "key and index in one word, the last word free");
static_assert(SO_BB_BLOCKS == SO_THREADS, "a block joins the boxes, one to a thread");

// Keys per block of a radix pass: 1024, more where that would be over 1024 blocks.
inline int64_t so_chunk(int64_t M) {
    int64_t c = 1024;
    while ((M + c - 1) / c > 1024) c *= 2;
    return c;
}
inline int so_blocks(int64_t M) { return (int)((M + so_chunk(M) - 1) / so_chunk(M)); }
inline size_t align256_sz(size_t x) { return (x + 255) & ~(size_t)255; }

// scratch: keys[2][M], vals[2][M], counts [radix][blocks] and [radix] totals, box partials, permuted arrays [5][M]
size_t spatial_order_bytes(int64_t M) {
    const size_t a = align256_sz((size_t)M * 4);
    return 4 * a + align256_sz((size_t)SO_RADIX * (so_blocks(M) + 1) * 4) + align256_sz((size_t)SO_BB_BLOCKS * 6 * 4) +
           5 * a;
}

struct SoBox { float mn[3], mx[3]; };

__device__ __forceinline__ void so_join(SoBox& b, const SoBox& o) {
#pragma unroll
    for (int q = 0; q < 3; ++q) { b.mn[q] = fminf(b.mn[q], o.mn[q]); b.mx[q] = fmaxf(b.mx[q], o.mx[q]); }
}

// Join over the block (every thread gets it); sh: one box per warp.
__device__ __forceinline__ SoBox so_block_join(SoBox b, SoBox* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        SoBox v;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            v.mn[q] = __shfl_xor_sync(0xffffffffu, b.mn[q], o);
            v.mx[q] = __shfl_xor_sync(0xffffffffu, b.mx[q], o);
        }
        so_join(b, v);
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = b;
    __syncthreads();
    b = sh[0];
    for (int w = 1; w < (int)blockDim.x / 32; ++w) so_join(b, sh[w]);
    return b;
}

__device__ __forceinline__ SoBox so_empty() {
    return {{FLT_MAX, FLT_MAX, FLT_MAX}, {-FLT_MAX, -FLT_MAX, -FLT_MAX}};
}

__device__ __forceinline__ SoBox so_range_box(const GaussDev& g, int64_t first, int64_t stride) {
    SoBox b = so_empty();
    for (int64_t i = first; i < g.M; i += stride) {
        const float c[3] = {g.cx[i], g.cy[i], g.cz[i]};
#pragma unroll
        for (int q = 0; q < 3; ++q) { b.mn[q] = fminf(b.mn[q], c[q]); b.mx[q] = fmaxf(b.mx[q], c[q]); }
    }
    return b;
}

__global__ void __launch_bounds__(SO_THREADS) so_box_kernel(GaussDev g, SoBox* __restrict__ part) {
    __shared__ SoBox sh[SO_WARPS];
    const SoBox b = so_block_join(so_range_box(g, blockIdx.x * (int64_t)SO_THREADS + threadIdx.x,
                                               (int64_t)gridDim.x * SO_THREADS), sh);
    if (threadIdx.x == 0) part[blockIdx.x] = b;
}

// the axis bits spread three apart (bit b to bit 3b), for interleaving x, y, z from the lowest bit
__device__ __forceinline__ uint32_t spread_bits(uint32_t v) {
    uint32_t r = 0;
#pragma unroll
    for (int b = 0; b < SO_AXIS_BITS; ++b) r |= ((v >> b) & 1u) << (3 * b);
    return r;
}

__device__ __forceinline__ uint32_t so_key(const GaussDev& g, const SoBox& box, int64_t i) {
    const float c[3] = {g.cx[i], g.cy[i], g.cz[i]};
    uint32_t k = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float lo = box.mn[q], ext = box.mx[q] - lo;
        const float t = ext > 0.f ? (c[q] - lo) / ext : 0.f;
        const float top = (float)((1 << SO_AXIS_BITS) - 1);
        const uint32_t u = (uint32_t)fminf(fmaxf(t * top, 0.f), top);
        k |= spread_bits(u) << q;
    }
    return k;
}

__device__ __forceinline__ void so_gather_one(const GaussDev& g, int64_t i, int64_t j, float* __restrict__ out) {
    const int64_t M = g.M;
    out[i] = g.cx[j];
    out[M + i] = g.cy[j];
    out[2 * M + i] = g.cz[j];
    out[3 * M + i] = g.sg[j];
    out[4 * M + i] = g.A[j];
}

// The whole order of up to SO_ONE_MAX Gaussians: Mp words (a power of two of at least 64) of dynamic
// shared memory.  out: the permuted arrays.
__global__ void __launch_bounds__(SO_ONE_THREADS)
so_one_kernel(GaussDev g, int Mp, float* __restrict__ out) {
    extern __shared__ uint32_t so_word[];
    __shared__ SoBox sh[SO_ONE_THREADS / 32];
    const int M = (int)g.M, t = threadIdx.x;
    const SoBox box = so_block_join(so_range_box(g, t, SO_ONE_THREADS), sh);
    for (int i = t; i < Mp; i += SO_ONE_THREADS)
        so_word[i] = i < M ? so_key(g, box, i) << SO_ONE_BITS | (uint32_t)i : 0xffffffffu;
    __syncthreads();
    for (int k = 2; k <= Mp; k <<= 1)
        for (int h = k >> 1; h > 0; h >>= 1) {
            for (int u = t; u < Mp / 2; u += SO_ONE_THREADS) {
                const int i = ((u & ~(h - 1)) << 1) | (u & (h - 1));
                const uint32_t a = so_word[i], b = so_word[i + h];
                if ((a > b) == ((i & k) == 0)) { so_word[i] = b; so_word[i + h] = a; }
            }
            // pairs of up to 32 words apart stay inside a warp's 64 words
            if (h > 32 || h == 1) __syncthreads(); else __syncwarp();
        }
    for (int i = t; i < M; i += SO_ONE_THREADS) {
        so_gather_one(g, i, (int)(so_word[i] & (SO_ONE_MAX - 1)), out);
    }
}

// Radix pass, step 1: the block's digit counts, stored digit-major: hist[d * nblocks + block].  The
// first pass (g.M > 0 keys to form) joins the boxes and writes the keys and indices too.
template <bool FIRST>
__global__ void __launch_bounds__(SO_THREADS)
so_hist_kernel(GaussDev g, const SoBox* __restrict__ part, uint32_t* __restrict__ keys, int* __restrict__ vals,
               int64_t chunk, int shift, int* __restrict__ hist) {
    __shared__ int h[SO_RADIX];
    __shared__ SoBox sh[SO_WARPS];
    for (int d = threadIdx.x; d < SO_RADIX; d += SO_THREADS) h[d] = 0;
    SoBox box;
    if (FIRST) box = so_block_join(part[threadIdx.x], sh);
    __syncthreads();
    const int64_t b0 = blockIdx.x * chunk;
    for (int64_t q = threadIdx.x; q < chunk; q += SO_THREADS) {
        const int64_t i = b0 + q;
        if (i >= g.M) break;
        uint32_t k;
        if (FIRST) {
            k = so_key(g, box, i);
            keys[i] = k;
            vals[i] = (int)i;
        } else {
            k = keys[i];
        }
        atomicAdd(&h[(k >> shift) & (SO_RADIX - 1)], 1);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < SO_RADIX; d += SO_THREADS) hist[(int64_t)d * gridDim.x + blockIdx.x] = h[d];
}

// Step 2: one warp per digit: the exclusive scan of its counts over the blocks, and its total.
__global__ void __launch_bounds__(SO_THREADS) so_scan_kernel(int* __restrict__ hist, int nb, int* __restrict__ total) {
    const int d = blockIdx.x * SO_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    int* row = hist + (int64_t)d * nb;
    int carry = 0;
    for (int b0 = 0; b0 < nb; b0 += 32) {
        const int v = b0 + lane < nb ? row[b0 + lane] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        if (b0 + lane < nb) row[b0 + lane] = carry + x - v;
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) total[d] = carry;
}

// Step 3: stable scatter.  Each warp owns a contiguous eighth of the block's keys: it counts its
// digits, the warps' counts give each its start per digit, and it then takes its keys 32 at a time
// in index order, the lanes of equal digit ranked by a match mask.
__global__ void __launch_bounds__(SO_THREADS)
so_scatter_kernel(const uint32_t* __restrict__ kin, const int* __restrict__ vin, int64_t n, int64_t chunk, int shift,
                  const int* __restrict__ hist, const int* __restrict__ total, uint32_t* __restrict__ kout,
                  int* __restrict__ vout) {
    __shared__ int cnt[SO_WARPS][SO_RADIX];
    __shared__ int wsum[SO_WARPS];
    static_assert(SO_RADIX == 2 * SO_THREADS, "two digits a thread");
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    for (int q = t; q < SO_WARPS * SO_RADIX; q += SO_THREADS) (&cnt[0][0])[q] = 0;
    // where each digit begins: thread t scans the totals of digits 2t and 2t + 1
    const int t0 = total[2 * t], t1 = total[2 * t + 1];
    int x = t0 + t1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += u;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    const int64_t seg = chunk / SO_WARPS, s0 = blockIdx.x * chunk + warp * seg;
    const int64_t s1 = s0 + seg < n ? s0 + seg : n;
    for (int64_t i = s0 + lane; i < s1; i += 32) atomicAdd(&cnt[warp][(kin[i] >> shift) & (SO_RADIX - 1)], 1);
    int start = x - t0 - t1;
    for (int w = 0; w < warp; ++w) start += wsum[w];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int d = 2 * t + k;
        int acc = start + (k ? t0 : 0) + hist[(int64_t)d * gridDim.x + blockIdx.x];
#pragma unroll
        for (int w = 0; w < SO_WARPS; ++w) {
            const int c = cnt[w][d];
            cnt[w][d] = acc;
            acc += c;
        }
    }
    __syncthreads();
    uint32_t lt;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
    for (int64_t i0 = s0; i0 < s1; i0 += 32) {
        const int64_t i = i0 + lane;
        const bool ok = i < s1;
        const uint32_t key = ok ? kin[i] : 0u;
        const int val = ok ? vin[i] : 0;
        const int d = ok ? (int)((key >> shift) & (SO_RADIX - 1)) : SO_RADIX;     // SO_RADIX: no key
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(peers & lt);
        const int at = ok ? cnt[warp][d] : 0;
        __syncwarp();
        if (ok && rank == 0) cnt[warp][d] = at + __popc(peers);
        if (ok) {
            kout[at + rank] = key;
            vout[at + rank] = val;
        }
        __syncwarp();
    }
}

__global__ void so_gather_kernel(GaussDev g, const int* __restrict__ perm, float* __restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < g.M) so_gather_one(g, i, perm[i], out);
}

// gp: g with its arrays replaced by the permuted copies in scratch (spatial_order_bytes(g.M)).
cudaError_t launch_spatial_order(const GaussDev& g, void* scratch, GaussDev& gp, cudaStream_t st) {
    const int64_t M = g.M;
    if (M > 0x7FFFFFFF) return cudaErrorNotSupported;
    const size_t a = align256_sz((size_t)M * 4);
    char* p = static_cast<char*>(scratch);
    float* out = reinterpret_cast<float*>(p + spatial_order_bytes(M) - 5 * a);
    gp = g;
    gp.cx = out;
    gp.cy = out + M;
    gp.cz = out + 2 * M;
    gp.sg = out + 3 * M;
    gp.A = out + 4 * M;
    if (M <= SO_ONE_MAX) {
        int Mp = 64;
        while (Mp < M) Mp <<= 1;
        so_one_kernel<<<1, SO_ONE_THREADS, (size_t)Mp * 4, st>>>(g, Mp, out);
        return cudaGetLastError();
    }
    uint32_t* keys[2] = {reinterpret_cast<uint32_t*>(p), reinterpret_cast<uint32_t*>(p + a)};
    int* vals[2] = {reinterpret_cast<int*>(p + 2 * a), reinterpret_cast<int*>(p + 3 * a)};
    const int nb = so_blocks(M);
    const int64_t chunk = so_chunk(M);
    int* hist = reinterpret_cast<int*>(p + 4 * a);
    int* total = hist + (size_t)SO_RADIX * nb;
    SoBox* part = reinterpret_cast<SoBox*>(p + 4 * a + align256_sz((size_t)SO_RADIX * (nb + 1) * 4));
    so_box_kernel<<<SO_BB_BLOCKS, SO_THREADS, 0, st>>>(g, part);
    for (int pass = 0; pass < SO_PASSES; ++pass) {
        const int in = pass & 1, shift = SO_DIGIT * pass;
        if (pass == 0) so_hist_kernel<true><<<nb, SO_THREADS, 0, st>>>(g, part, keys[in], vals[in], chunk, shift, hist);
        else so_hist_kernel<false><<<nb, SO_THREADS, 0, st>>>(g, part, keys[in], vals[in], chunk, shift, hist);
        so_scan_kernel<<<SO_RADIX / SO_WARPS, SO_THREADS, 0, st>>>(hist, nb, total);
        so_scatter_kernel<<<nb, SO_THREADS, 0, st>>>(keys[in], vals[in], M, chunk, shift, hist, total, keys[in ^ 1],
                                                     vals[in ^ 1]);
    }
    static_assert(SO_PASSES % 2 == 0, "the order ends in buffer 0");
    so_gather_kernel<<<(unsigned)((M + 255) / 256), 256, 0, st>>>(g, vals[0], out);
    return cudaGetLastError();
}

}  // namespace gp
