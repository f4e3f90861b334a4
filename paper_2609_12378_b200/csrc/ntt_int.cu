// The N = 2^16 transform on the integer pipe (context option CKKS_OPT_NTT_FP_SHARE below 8: of every eight limbs, those from
// the share on take this path; the FP64 kernels of ntt.cu skip them).
//
// Lazy arithmetic.  Residues travel as 64-bit words that are only congruent to the value: with 50-bit primes there are 14
// spare bits.  The twiddle product uses an under-estimate of floor(x w'/2^64) built from three 32x32 products (the low x low
// product is dropped, the cross products keep their high halves), at most 3 below the exact quotient, so the product lands
// in [0, 5q) for ANY 64-bit x.  Forward (Cooley-Tukey): X' = X + T, Y' = X - T + 5q; magnitudes grow by at most 5q per
// stage, 81q < 2^57 after 16 stages, one exact reduction at the end.  Inverse (Gentleman-Sande): X' = U + V doubles the
// bound per stage, Y' = (U - V + bound q) w' is back in [0, 5q); 8 stages keep everything below 1280 q < 2^61, so one lazy
// reduction between the passes suffices.
#include "common.cuh"

namespace {

constexpr uint32_t THREADS = 256;

__device__ __forceinline__ u64 mulhi_under(u64 x, u64 a) {
    const uint32_t x0 = (uint32_t)x, x1 = (uint32_t)(x >> 32), a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32);
    return (u64)x1 * a1 + __umulhi(x1, a0) + __umulhi(x0, a1);
}
// x * w mod q up to a multiple of q, in [0, 5q), for any 64-bit x
__device__ __forceinline__ u64 mul_tw(u64 x, ulonglong2 w, u64 q) { return x * w.x - mulhi_under(x, w.y) * q; }

// 4 Cooley-Tukey stages on 16 registers; stage twiddles tw[ml*base + i], ml = 1,2,4,8
__device__ __forceinline__ void fwd16(u64 (&x)[16], const ulonglong2 *__restrict__ tw, uint32_t base, u64 q, u64 q5) {
#pragma unroll
    for (uint32_t ml = 1; ml < 16; ml <<= 1) {
        const uint32_t tl = 8 / ml;
#pragma unroll
        for (uint32_t i = 0; i < ml; i++) {
            const ulonglong2 w = __ldg(&tw[ml * base + i]);
#pragma unroll
            for (uint32_t j = 0; j < tl; j++) {
                const uint32_t k1 = 2 * i * tl + j, k2 = k1 + tl;
                const u64 t = mul_tw(x[k2], w, q);
                x[k2] = x[k1] + q5 - t;
                x[k1] = x[k1] + t;
            }
        }
    }
}

// 4 Gentleman-Sande stages (ml = 8,4,2,1); `bound` = multiple of q bounding the inputs on entry
template <uint32_t BOUND>
__device__ __forceinline__ void inv16(u64 (&x)[16], const ulonglong2 *__restrict__ tw, uint32_t base, u64 q) {
    uint32_t b = BOUND;
#pragma unroll
    for (uint32_t ml = 8; ml >= 1; ml >>= 1) {
        const uint32_t tl = 8 / ml;
        const u64 off = (u64)b * q;
#pragma unroll
        for (uint32_t i = 0; i < ml; i++) {
            const ulonglong2 w = __ldg(&tw[ml * base + i]);
#pragma unroll
            for (uint32_t j = 0; j < tl; j++) {
                const uint32_t k1 = 2 * i * tl + j, k2 = k1 + tl;
                const u64 u = x[k1], v = x[k2];
                x[k1] = u + v;
                x[k2] = mul_tw(u + off - v, w, q);
            }
        }
        b = 2 * b > 5 ? 2 * b : 5;
    }
}
// bound after the 4 stages of inv16<b>: b -> max(2b, 5) four times, i.e. 1 -> 40, 5 -> 80, 40 -> 640, 80 -> 1280

// exact reduction of a lazy word (< 2^64) to [0, q): qinv64 = floor(2^64 / q)
__device__ __forceinline__ u64 reduce_exact(u64 x, u64 q, u64 qinv64) {
    u64 r = x - __umul64hi(x, qinv64) * q;     // in [0, 2q)
    return r >= q ? r - q : r;
}

__global__ void __launch_bounds__(THREADS) int_fwd_cols(DevTables c, u64 *base, LimbMap map, uint32_t fp_share) {
    grid_dep_sync();
    __shared__ u64 sm[256 * 16];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) < fp_share) return;
    const u64 q = c.mod[prime], q5 = 5 * q;
    const ulonglong2 *tw = c.tw_fwd + ((size_t)prime << 16);
    const uint32_t cc = threadIdx.x & 15, r = threadIdx.x >> 4;
    u64 *g = base + (limb_index(map, blockIdx.y) << 16) + blockIdx.x * 16 + cc;
    u64 x[16];
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = g[(size_t)(r + 16 * k) * 256];
    fwd16(x, tw, 1, q, q5);
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) sm[(r + 16 * k) * 16 + cc] = x[k];
    __syncthreads();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = sm[(16 * r + k) * 16 + cc];
    fwd16(x, tw, 16 + r, q, q5);
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) g[(size_t)(16 * r + k) * 256] = x[k];
}

constexpr uint32_t ROW_PAD = 256 + 16;
__device__ __forceinline__ uint32_t padded(uint32_t i) { return i + (i >> 4); }

__global__ void __launch_bounds__(THREADS) int_fwd_rows(DevTables c, u64 *base, LimbMap map, uint32_t fp_share) {
    grid_dep_sync();
    __shared__ u64 sm[16 * ROW_PAD];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) < fp_share) return;
    const u64 q = c.mod[prime], q5 = 5 * q;
    const ulonglong2 *tw = c.tw_fwd + ((size_t)prime << 16);
    const uint32_t t = threadIdx.x & 15, rl = threadIdx.x >> 4, row = blockIdx.x * 16 + rl;
    u64 *g = base + (limb_index(map, blockIdx.y) << 16) + (size_t)row * 256;
    u64 *s = sm + rl * ROW_PAD;
    u64 x[16];
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = g[t + 16 * k];
    fwd16(x, tw, 256 + row, q, q5);
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) s[padded(t + 16 * k)] = x[k];
    __syncwarp();   // a row lives in one half warp
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = s[padded(16 * t + k)];
    fwd16(x, tw, 16 * (256 + row) + t, q, q5);
    const u64 qinv64 = c.mu64[prime];
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) s[padded(16 * t + k)] = reduce_exact(x[k], q, qinv64);
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) g[t + 16 * k] = s[padded(t + 16 * k)];
}

// src (if any): limb x of entry y / period lies at src + entry * src_stride words + x * src_lpitch limbs
__global__ void __launch_bounds__(THREADS) int_inv_rows(DevTables c, u64 *base, LimbMap map, uint32_t fp_share, const u64 *src, size_t src_stride, uint32_t src_lpitch) {
    grid_dep_sync();
    __shared__ u64 sm[16 * ROW_PAD];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) < fp_share) return;
    const u64 q = c.mod[prime];
    const ulonglong2 *tw = c.tw_inv + ((size_t)prime << 16);
    const uint32_t t = threadIdx.x & 15, rl = threadIdx.x >> 4, row = blockIdx.x * 16 + rl;
    u64 *g = base + (limb_index(map, blockIdx.y) << 16) + (size_t)row * 256;
    const u64 *gs = src ? src + (blockIdx.y / map.period) * src_stride + (((size_t)(blockIdx.y % map.period) * src_lpitch) << 16) + (size_t)row * 256 : g;
    u64 *s = sm + rl * ROW_PAD;
    u64 x[16];
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) s[padded(t + 16 * k)] = gs[t + 16 * k];
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = s[padded(16 * t + k)];
    inv16<1>(x, tw, 16 * (256 + row) + t, q);
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) s[padded(16 * t + k)] = x[k];
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = s[padded(t + 16 * k)];
    inv16<40>(x, tw, 256 + row, q);
    const ulonglong2 one = make_ulonglong2(1, c.mu64[prime]);
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) g[t + 16 * k] = mul_tw(x[k], one, q);   // lazy reduction to [0, 5q)
}

__global__ void __launch_bounds__(THREADS) int_inv_cols(DevTables c, u64 *base, LimbMap map, uint32_t fp_share) {
    grid_dep_sync();
    __shared__ u64 sm[256 * 16];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) < fp_share) return;
    const u64 q = c.mod[prime];
    const ulonglong2 *tw = c.tw_inv + ((size_t)prime << 16);
    const uint32_t cc = threadIdx.x & 15, r = threadIdx.x >> 4;
    u64 *g = base + (limb_index(map, blockIdx.y) << 16) + blockIdx.x * 16 + cc;
    u64 x[16];
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = g[(size_t)(16 * r + k) * 256];
    inv16<5>(x, tw, 16 + r, q);
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) sm[(16 * r + k) * 16 + cc] = x[k];
    __syncthreads();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = sm[(r + 16 * k) * 16 + cc];
    inv16<80>(x, tw, 1, q);
    const ulonglong2 ni = c.n_inv[prime];
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) g[(size_t)(r + 16 * k) * 256] = mul_shoup(x[k], ni.x, ni.y, q);
}

}  // namespace

// the limbs of a grid of ny limbs that the FP64 kernels leave out (whole periods of the map per call)
// src: as launch_ntt's, in the unscattered form
void launch_ntt_int(const ckks_ctx *c, u64 *b, uint32_t ny, const LimbMap &map, bool inverse, const NttSource &src, cudaStream_t s) {
    const dim3 grid(16, ny);
    const uint32_t share = c->ntt_fp_share;
    if (!inverse) {
        launch(int_fwd_cols, grid, THREADS, 0, s, c->dev, b, map, share);
        launch(int_fwd_rows, grid, THREADS, 0, s, c->dev, b, map, share);
    } else {
        launch(int_inv_rows, grid, THREADS, 0, s, c->dev, b, map, share, src.lpitch ? src.ptr.base : nullptr, src.ptr.stride, src.lpitch);
        launch(int_inv_cols, grid, THREADS, 0, s, c->dev, b, map, share);
    }
}
