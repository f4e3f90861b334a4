// Batched negacyclic NTT / inverse NTT, N = 2^10 .. 2^16.
//
// Forward: merged Cooley-Tukey, natural-order input, bit-reversed output, stages m = 1, 2, .., N/2 with butterfly distance
// t = N/(2m) and twiddle psi^bitrev(m+i) for block i.  Inverse: Gentleman-Sande, the same stages backwards, then N^-1.
//
// A limb is viewed as R rows of 256 coefficients (R = N/256 = 2^LOGR).  The stages with distance >= 256 couple rows only
// ("column pass": a CTA owns all R rows of a strip of columns), the stages with distance < 256 stay inside a row ("row
// pass": 16 threads per row).  Every pass holds its coefficients in registers and does its stages in one or two groups of up
// to four, with one exchange through shared memory between the groups; a limb makes two trips through memory per transform.
// The results of the column pass (forward) or row pass (inverse) stay signed doubles until the other pass has read them.
//
// Arithmetic: 50-bit residues as signed integers in doubles, exact while below 2^53.  The FP64 pipe multiplies two of them
// exactly in two instructions where the integer pipe needs several 32x32 products:
//   p = y w (rounded), e = fma(y, w, -p) (exact low part), k = round(p * (1/q)) by adding and subtracting 1.5 * 2^52 (or
//   1.5 * 2^53), r = fma(-k, q, p) + e = y w - k q exactly.
// The kernels are bound by FP64 issue (eight instructions per butterfly), so what is kept small is everything around the
// butterflies: range reductions, conversions, and load/store instructions.
#include "common.cuh"

namespace {

// ML consecutive twiddles w (ML = 1, 2, 4, 8; the index is a multiple of ML) with the widest loads that fit.
// SH: from a copy in shared memory.
template <uint32_t ML, bool SH = false>
__device__ __forceinline__ void load_tw(const double *p, double (&v)[ML]) {
    if (SH) {
        if (ML == 1) v[0] = *p;
#pragma unroll
        for (uint32_t i = 0; i + 1 < ML; i += 2) {
            const double2 w = *reinterpret_cast<const double2 *>(p + i);
            v[i] = w.x; v[(i + 1) % ML] = w.y;
        }
        return;
    }
    if (ML == 1) v[0] = __ldg(p);
    if (ML == 2) asm volatile("ld.global.nc.v2.f64 {%0,%1}, [%2];" : "=d"(v[0]), "=d"(v[ML > 1 ? 1 : 0]) : "l"(p));
    if (ML >= 4) {
#pragma unroll
        for (uint32_t i = 0; i < ML; i += 4)
            asm volatile("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(v[i]), "=d"(v[(i + 1) % ML]), "=d"(v[(i + 2) % ML]), "=d"(v[(i + 3) % ML]) : "l"(p + i));
    }
}

// ---- range bookkeeping ---------------------------------------------------------------------------------------------
// B = bound in units of q (q > 2^49, everything below 8 q <= 2^53 is exact).  The twiddle tables hold centred
// representatives, |w| <= q/2, and the quotient estimate is within 2^-52 relative, so for |y| <= B q the product y w - k q
// comes out below
//   T(B) = (1/2 + B/8) q   when k is rounded to the nearest integer (needs B < 4:  |y w/q| < 2^51), and below
//   Tc(B) = (1 + B/8) q    when k is rounded to the nearest even integer ("coarse", needs B < 8).
// A Cooley-Tukey stage (u, v) -> (u + v w, u - v w) takes B to B + T(B), or to 1/2 + T(B) if u is reduced first (three
// instructions for half of the values; the product needs no reduced v).  From a canonical input the stages reach
//   1.63 2.33 3.12 4.01 | 5.51c 7.20c | u reduced: 2.40c 3.20,
// the row pass goes on with 4.10 5.61c 7.31c | u reduced: 2.42c | 3.22 4.12 5.64c 7.35c and one exact reduction at the end:
// two half reductions on the way for sixteen stages.  Smaller rings reduce u in their last column stage instead, which
// keeps the row pass's input at or below 3.20 for every N.

// Stage s (1 .. LOGR) of the forward column pass.
__host__ __device__ constexpr bool col_coarse(uint32_t s) { return s >= 5 && s <= 7; }
__host__ __device__ constexpr bool col_reduce(uint32_t logr, uint32_t s) { return logr >= 4 && s == (logr < 7 ? logr : 7); }

// one Cooley-Tukey stage on 2 ML tl registers starting at x: blocks of 2 tl, twiddles tw[ML * base + i]
template <uint32_t ML, uint32_t RADIX, bool COARSE, bool REDUCE_U, bool SH = false, uint32_t E>
__device__ __forceinline__ void fwd_stage(double (&x)[E], uint32_t x0, const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    constexpr uint32_t tl = RADIX / 2 / ML;
    double w[ML];
    load_tw<ML, SH>(tw + ML * base, w);
#pragma unroll
    for (uint32_t i = 0; i < ML; i++)
#pragma unroll
        for (uint32_t j = 0; j < tl; j++) {
            const uint32_t k1 = x0 + 2 * i * tl + j, k2 = k1 + tl;
            const double t = mulmod_pq<COARSE ? 1 : 0>(x[k2], w[i], q, qinv);
            const double u = REDUCE_U ? reduce_d(x[k1], q, qinv) : x[k1];
            x[k2] = __dsub_rn(u, t);
            x[k1] = __dadd_rn(u, t);
        }
}
// stages S0 + 1 .. S0 + G of the column pass on one sub-transform of 2^G registers
template <uint32_t LOGR, uint32_t S0, uint32_t G, bool SH = false, uint32_t E>
__device__ __forceinline__ void fwd_col_group(double (&x)[E], uint32_t x0, const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    constexpr uint32_t RX = 1u << G;
    fwd_stage<1, RX, col_coarse(S0 + 1), col_reduce(LOGR, S0 + 1), SH>(x, x0, tw, base, q, qinv);
    if constexpr (G >= 2) fwd_stage<2, RX, col_coarse(S0 + 2), col_reduce(LOGR, S0 + 2), SH>(x, x0, tw, base, q, qinv);
    if constexpr (G >= 3) fwd_stage<4, RX, col_coarse(S0 + 3), col_reduce(LOGR, S0 + 3), SH>(x, x0, tw, base, q, qinv);
    if constexpr (G >= 4) fwd_stage<8, RX, col_coarse(S0 + 4), col_reduce(LOGR, S0 + 4), SH>(x, x0, tw, base, q, qinv);
}
// row pass, first four stages: 3.20 q in, 4.10 5.61c 7.31c | u reduced 2.42c out
__device__ __forceinline__ void fwd_row_open(double (&x)[16], const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    fwd_stage<1, 16, false, false>(x, 0, tw, base, q, qinv);
    fwd_stage<2, 16, true, false>(x, 0, tw, base, q, qinv);
    fwd_stage<4, 16, true, false>(x, 0, tw, base, q, qinv);
    fwd_stage<8, 16, true, true>(x, 0, tw, base, q, qinv);
}
// row pass, last four stages: 2.42 q in, 3.22 4.12 5.64c 7.35c out
__device__ __forceinline__ void fwd_row_close(double (&x)[16], const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    fwd_stage<1, 16, false, false>(x, 0, tw, base, q, qinv);
    fwd_stage<2, 16, false, false>(x, 0, tw, base, q, qinv);
    fwd_stage<4, 16, true, false>(x, 0, tw, base, q, qinv);
    fwd_stage<8, 16, true, false>(x, 0, tw, base, q, qinv);
}

// Gentleman-Sande: (u, v) -> (u + v, (u - v) w).  Sums double the bound and products fall back to T(Bu + Bv), so after a
// group of stages only the few registers that were sums several times over are large, and the registers' positions are
// known at compile time: gs_plan walks the bounds and marks which registers to reduce before a stage (where a pair would
// reach 8 q, or 4 q in the last stage, whose products must round to nearest), which pairs need the coarse product, and
// which to reduce after the group because they exceed `thr` (the next group starts from the largest of what is left).  33
// reductions per sixteen registers and transform at N = 2^16, where reducing all of them once per group took 80.
struct GsPlan {
    uint32_t pre[4], coarse[4], post;
    double out;
};
__host__ __device__ constexpr GsPlan gs_plan(uint32_t stages, double in, double thr, bool last) {
    GsPlan p{};
    double b[16] = {};
    const uint32_t n = 1u << stages;
    for (uint32_t k = 0; k < n; k++) b[k] = in;
    for (uint32_t s = 0; s < stages; s++) {
        const uint32_t tl = 1u << s;
        const double lim = last && s + 1 == stages ? 4.0 : 7.99;
        for (uint32_t k = 0; k < n; k++) {
            if (k & tl) continue;
            for (uint32_t r = 0; r < 2 && b[k] + b[k + tl] >= lim; r++) {
                const uint32_t big = b[k] >= b[k + tl] ? k : k + tl;
                b[big] = 0.5;
                p.pre[s] |= 1u << big;
            }
            const double sum = b[k] + b[k + tl];
            if (sum >= 4.0) p.coarse[s] |= 1u << k;
            b[k] = sum;
            b[k + tl] = (sum >= 4.0 ? 1.0 : 0.5) + sum / 8.0;
        }
    }
    for (uint32_t k = 0; k < n; k++) {
        if (!last && b[k] > thr) { b[k] = 0.5; p.post |= 1u << k; }
        if (b[k] > p.out) p.out = b[k];
    }
    return p;
}
__host__ __device__ constexpr uint32_t gs_pre(uint32_t st, double in, double thr, bool last, uint32_t s) { return gs_plan(st, in, thr, last).pre[s]; }
__host__ __device__ constexpr uint32_t gs_coarse(uint32_t st, double in, double thr, bool last, uint32_t s) { return gs_plan(st, in, thr, last).coarse[s]; }
__host__ __device__ constexpr uint32_t gs_post(uint32_t st, double in, double thr, bool last) { return gs_plan(st, in, thr, last).post; }
__host__ __device__ constexpr double gs_out(uint32_t st, double in, double thr) { return gs_plan(st, in, thr, false).out; }

// The groups of the inverse: row pass 1 and 2 (four stages each), column pass first and last.  Bounds on entry:
__host__ __device__ constexpr double inv_in(int group) {
    return group == 1 ? 1.0 : group == 2 ? gs_out(4, 1.0, 1.75) : gs_out(4, gs_out(4, 1.0, 1.75), 2.01);
}

template <uint32_t MASK, uint32_t N_, uint32_t E>
__device__ __forceinline__ void reduce_masked(double (&x)[E], uint32_t x0, double q, double qinv) {
#pragma unroll
    for (uint32_t k = 0; k < N_; k++)
        if (MASK >> k & 1) x[x0 + k] = reduce_d(x[x0 + k], q, qinv);
}
// stage s (distance 2^s) of a group of G stages
template <uint32_t S, uint32_t G, uint32_t PRE, uint32_t COARSE, bool SH, uint32_t E>
__device__ __forceinline__ void inv_stage(double (&x)[E], uint32_t x0, const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    constexpr uint32_t tl = 1u << S, ML = (1u << G) / 2 / tl;
    double w[ML];
    load_tw<ML, SH>(tw + ML * base, w);
    reduce_masked<PRE, (1u << G)>(x, x0, q, qinv);
#pragma unroll
    for (uint32_t i = 0; i < ML; i++)
#pragma unroll
        for (uint32_t j = 0; j < tl; j++) {
            const uint32_t k = 2 * i * tl + j, k1 = x0 + k, k2 = k1 + tl;
            const double u = x[k1], v = x[k2], d = __dsub_rn(u, v);
            x[k1] = __dadd_rn(u, v);
            x[k2] = (COARSE >> k & 1) ? mulmod_pq<1>(d, w[i], q, qinv) : mulmod_pq<0>(d, w[i], q, qinv);
        }
}
// the first NST of a group of G stages, entry bound IN(group) of the plan (G, in, thr, LAST)
#define INV_STAGE(S, G, IN, THR, LAST) inv_stage<S, G, gs_pre(G, IN, THR, LAST, S), gs_coarse(G, IN, THR, LAST, S), SH>(x, x0, tw, base, q, qinv)
template <int GROUP>        // 1, 2: the row pass
__device__ __forceinline__ void inv_row_group(double (&x)[16], const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    constexpr uint32_t x0 = 0;
    constexpr bool SH = false;
    constexpr double in = inv_in(GROUP), thr = GROUP == 1 ? 1.75 : 2.01;
    INV_STAGE(0, 4, in, thr, false);
    INV_STAGE(1, 4, in, thr, false);
    INV_STAGE(2, 4, in, thr, false);
    INV_STAGE(3, 4, in, thr, false);
    reduce_masked<gs_post(4, in, thr, false), 16>(x, 0, q, qinv);
}
template <uint32_t G, bool SH = false, uint32_t E>       // the column pass's first group (of two)
__device__ __forceinline__ void inv_col_open(double (&x)[E], uint32_t x0, const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    constexpr double in = inv_in(3), thr = 1.01;
    INV_STAGE(0, G, in, thr, false);
    if constexpr (G >= 2) INV_STAGE(1, G, in, thr, false);
    if constexpr (G >= 3) INV_STAGE(2, G, in, thr, false);
    if constexpr (G >= 4) INV_STAGE(3, G, in, thr, false);
    reduce_masked<gs_post(G, in, thr, false), (1u << G)>(x, x0, q, qinv);
}
// The last group (twiddle base 1); the last stage has N^-1 (or the caller's constant) folded in: x1 = (u + v) c0,
// x2 = (u - v) c1, both products of values below 4 q rounded to nearest, so the results are below q and one conditional
// addition makes them canonical.  c0 = {N^-1, N^-1/q}, c1 = {w_1 N^-1, that / q}, centred.
template <uint32_t G, uint32_t B, bool SH = false, uint32_t E>     // B: stages of the open group before it (0: none)
__device__ __forceinline__ void inv_col_last(double (&x)[E], const double *__restrict__ tw, double q, double qinv, double2 c0, double2 c1) {
    constexpr uint32_t x0 = 0, base = 1;
    constexpr double in = B ? gs_out(B, inv_in(3), 1.01) : inv_in(3);
    if constexpr (G >= 2) INV_STAGE(0, G, in, 9.0, true);
    if constexpr (G >= 3) INV_STAGE(1, G, in, 9.0, true);
    if constexpr (G >= 4) INV_STAGE(2, G, in, 9.0, true);
    reduce_masked<gs_pre(G, in, 9.0, true, G - 1), (1u << G)>(x, 0, q, qinv);
    constexpr uint32_t tl = (1u << G) / 2;
#pragma unroll
    for (uint32_t j = 0; j < tl; j++) {
        const double u = x[j], v = x[j + tl];
        x[j] = mulmod_d<0>(__dadd_rn(u, v), c0, q);
        x[j + tl] = mulmod_d<0>(__dsub_rn(u, v), c1, q);
    }
}
#undef INV_STAGE

// ---- measurement aid: the forward butterflies on registers only ------------------
// Every thread runs `iters` radix-16 groups (4 stages, 32 butterflies, with the transform's range reductions and twiddle
// fetches, the latter from a 17 KiB window that stays in L1) on 16 registers; nothing else touches memory.  Three CTAs of 256
// threads per SM: 24 warps, the inverse transform's occupancy (the forward passes run at 32).
constexpr uint32_t F_THREADS = 256;
__global__ void __launch_bounds__(F_THREADS, 3) butterfly_probe_kernel(DevTables c, uint32_t iters, u64 *sink) {
    grid_dep_sync();
    const double q = c.modd[0].x, qinv = c.modd[0].y;
    const double *tw = c.twd_fwd;
    double x[16];
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = (double)(threadIdx.x * 16 + k + 1);
    uint32_t base = 16 + (threadIdx.x & 255);
    for (uint32_t it = 0; it < iters; it++) {
        fwd_row_open(x, tw, base, q, qinv);
        base = 16 + ((base * 5 + 1) & 255);
    }
    double acc = 0.0;
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) acc = __dadd_rn(acc, x[k]);
    if (acc == 0.5) sink[blockIdx.x * F_THREADS + threadIdx.x] = 1;      // never true for integer-valued sums
}

// The column pass of a limb uses entries 1 .. R - 1 of its twiddle table (2 KiB at N = 2^16).  At that size a CTA fetches them
// once into shared memory: stage by stage from global memory they cost every stage a trip to L2, because the streamed data
// leaves them nothing of L1 (768 limbs: forward 150 -> 141 us, inverse 161 -> 156).  Smaller rings' few CTAs are bound by latency
// and keep the direct loads (the barrier costs them 0.2 us), and so do the row passes, where a CTA's entries are its own
// (forward 155 -> 157, inverse 147 -> 171 us with its first-group entries in shared memory).
template <uint32_t LOGR> constexpr bool TW_SHARED = LOGR == 8;
template <uint32_t R>
__device__ __forceinline__ void stage_tw(double *dst, const double *tw) {
    for (uint32_t e = threadIdx.x; e < R; e += blockDim.x) dst[e] = tw[e];
}

// The end of a CTA whose limb is left out.  With limbs on the integer path that may be every CTA of a grid (a digit's own limb and
// seven integer ones), and a grid that has not waited for the one before it lets the one after it pass that too.
__device__ __forceinline__ void leave_out(uint32_t fp_share) {
    if (fp_share < 8) grid_dep_sync();
}

// ---- column passes -------------------------------------------------------------------------------------------------
// Shape per LOGR: the R-point column transform is split into a first group of A stages (registers R/2^A rows apart) and a
// second of B stages (2^B consecutive rows; a thread holds 2^(A-B) of these), E = 2^A registers per thread, COLS columns per
// CTA.  N = 2^16: radix 16 x 16, strips of 16 columns (128-byte row pieces), 256 threads.  Smaller rings take fewer
// registers per thread so that the few limbs of a small ciphertext still spread over the GPU, and wider strips.
template <uint32_t LOGR>
struct ColShape {
    static constexpr uint32_t A = LOGR == 8 ? 4 : LOGR == 7 ? 4 : LOGR == 6 ? 3 : LOGR == 5 ? 3 : LOGR;
    static constexpr uint32_t B = LOGR - A, E = 1u << A, R = 1u << LOGR;
    static constexpr uint32_t COLS = LOGR >= 6 ? 16 : LOGR == 5 ? 32 : 128;
    static constexpr uint32_t THREADS = R * COLS / E;
};

enum { SRC_LIMBS = 0, SRC_COEFS = 1, SRC_LIFT = 2, SRC_DOUBLES = 3 };

// forward: SRC_LIMBS in place; SRC_COEFS: signed 64-bit coefficients [batch][N], reduced modulo the limb's prime on load;
// SRC_LIFT: one residue limb per period modulo prime src_prime, lifted to its centred representative (rescale);
// SRC_DOUBLES in place, signed doubles of at most q / 2 instead of residues (the conversions)
template <uint32_t LOGR, int SRC>
__global__ void __launch_bounds__(ColShape<LOGR>::THREADS, 1024 / ColShape<LOGR>::THREADS) ntt_fwd_cols(DevTables c, u64 *base, LimbMap map, uint32_t fp_share,
                                                                                                    const u64 *src, uint32_t src_prime) {
    using S = ColShape<LOGR>;
    __shared__ double sm[S::B ? S::R * S::COLS : 1];
    constexpr bool SH = TW_SHARED<LOGR>;
    __shared__ __align__(16) double stw[SH ? S::R : 2];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) >= fp_share) return leave_out(fp_share);
    const double q = c.modd[prime].x, qinv = c.modd[prime].y;
    const double *tw = c.twd_fwd + ((size_t)prime << c.log_n);
    const uint32_t cc = threadIdx.x % S::COLS, r = threadIdx.x / S::COLS;
    u64 *g = base + (limb_index(map, blockIdx.y) << c.log_n) + blockIdx.x * S::COLS + cc;
    const u64 *gs = SRC == SRC_LIMBS || SRC == SRC_DOUBLES ? g : src + ((size_t)(blockIdx.y / map.period) << c.log_n) + blockIdx.x * S::COLS + cc;
    constexpr uint32_t RS = S::R / S::E;          // rows between a thread's registers in the first group
    double x[S::E];
    if (SH) stage_tw<S::R>(stw, tw);
    const double *tws = SH ? stw : tw;
    grid_dep_sync();
    if (SRC == SRC_COEFS) {
        // coefficients below 2^49 (every weight of ordinary size at the scale of a prime) are residues as they are, signed;
        // anything larger in a warp takes the integer reduction
        long long v[S::E];
        uint32_t big = 0;
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) {
            v[k] = (long long)gs[(size_t)(r + RS * k) * 256];
            const uint32_t hi = (uint32_t)(v[k] >> 32);
            big |= hi ^ (uint32_t)((int)hi >> 31);
        }
        if (__any_sync(0xffffffffu, big >= (1u << 17))) {
            const u64 qi = c.mod[prime], mu = c.mu[prime];
#pragma unroll
            for (uint32_t k = 0; k < S::E; k++) {
                const u64 m = barrett112(0, v[k] < 0 ? (u64)(-v[k]) : (u64)v[k], qi, mu);
                x[k] = u64_to_d((v[k] < 0 && m) ? qi - m : m);
            }
        } else {
#pragma unroll
            for (uint32_t k = 0; k < S::E; k++) x[k] = __dsub_rn(__longlong_as_double(v[k] + 0x4338000000000000ll), MAGIC0);
        }
    } else if (SRC == SRC_DOUBLES) {
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) x[k] = reinterpret_cast<const double *>(gs)[(size_t)(r + RS * k) * 256];
    } else if (SRC == SRC_LIFT) {
        const u64 ql = c.mod[src_prime];
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) x[k] = centre_d(gs[(size_t)(r + RS * k) * 256], ql);
    } else {
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) x[k] = u64_to_d(gs[(size_t)(r + RS * k) * 256]);
    }
    if (SH) __syncthreads();
    else __syncwarp();  // keeps all loads in front of the butterflies: interleaved with them they were 10 % slower
    fwd_col_group<LOGR, 0, S::A, SH>(x, 0, tws, 1, q, qinv);
    if constexpr (S::B > 0) {
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) sm[(r + RS * k) * S::COLS + cc] = x[k];
        __syncthreads();
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) x[k] = sm[(S::E * r + k) * S::COLS + cc];
#pragma unroll
        for (uint32_t j = 0; j < (S::E >> S::B); j++)
            fwd_col_group<LOGR, S::A, S::B, SH>(x, j << S::B, tws, (1u << S::A) + r * (S::E >> S::B) + j, q, qinv);
    }
    constexpr uint32_t OS = S::B ? 1 : RS;        // without a second group the registers are still RS rows apart
#pragma unroll
    for (uint32_t k = 0; k < S::E; k++) reinterpret_cast<double *>(g)[(size_t)((S::B ? S::E : 1) * r + OS * k) * 256] = x[k];
}

// inverse (the last pass): the first group on 2^B consecutive rows, the last on rows 2^B apart, then the folded scaling
template <uint32_t LOGR>
__global__ void __launch_bounds__(ColShape<LOGR>::THREADS, 768 / ColShape<LOGR>::THREADS) ntt_inv_cols(DevTables c, u64 *base, LimbMap map, uint32_t fp_share,
                                                                                                   const double2 *scale) {
    using S = ColShape<LOGR>;
    __shared__ double sm[S::B ? S::R * S::COLS : 1];
    constexpr bool SH = TW_SHARED<LOGR>;
    __shared__ __align__(16) double stw[SH ? S::R : 2];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) >= fp_share) return leave_out(fp_share);
    const double q = c.modd[prime].x, qinv = c.modd[prime].y;
    const double *tw = c.twd_inv + ((size_t)prime << c.log_n);
    const uint32_t cc = threadIdx.x % S::COLS, r = threadIdx.x / S::COLS;
    u64 *g = base + (limb_index(map, blockIdx.y) << c.log_n) + blockIdx.x * S::COLS + cc;
    const double2 *sc = scale ? scale + 2 * (blockIdx.y % map.period) : c.n_inv_d + 2 * prime;
    const double2 c0 = sc[0], c1 = sc[1];
    constexpr uint32_t RS = S::R / S::E;
    double x[S::E];
    if (SH) stage_tw<S::R>(stw, tw);
    const double *tws = SH ? stw : tw;
    grid_dep_sync();
    if constexpr (S::B > 0) {
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) x[k] = reinterpret_cast<const double *>(g)[(size_t)(S::E * r + k) * 256];
        if (SH) __syncthreads();
#pragma unroll
        for (uint32_t j = 0; j < (S::E >> S::B); j++) inv_col_open<S::B, SH>(x, j << S::B, tws, (1u << S::A) + r * (S::E >> S::B) + j, q, qinv);
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) sm[(S::E * r + k) * S::COLS + cc] = x[k];
        __syncthreads();
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) x[k] = sm[(r + RS * k) * S::COLS + cc];
    } else {
#pragma unroll
        for (uint32_t k = 0; k < S::E; k++) x[k] = reinterpret_cast<const double *>(g)[(size_t)(r + RS * k) * 256];
        if (SH) __syncthreads();
    }
    inv_col_last<S::A, S::B, SH>(x, tws, q, qinv, c0, c1);
#pragma unroll
    for (uint32_t k = 0; k < S::E; k++) g[(size_t)(r + RS * k) * 256] = canonical_d(x[k], q);
}

// ---- row passes ----------------------------------------------------------------------------------------------------
// 16 threads per row, a row in one half warp, so warps need no barrier between them; 4 rows per CTA (16 were
// 2 % slower: finer CTAs keep the phases of an SM's warps apart).  In the exchange row two spare words
// follow every 16, so that a thread's own 16 consecutive coefficients are a 16-byte aligned block at a pitch of 144 bytes:
// 8-byte accesses of consecutive lanes and 16-byte accesses to the own block are both conflict free.  Words enter and leave
// through the row too, as pairs: lane t of a half warp moves words 2 t + 32 k and 2 t + 32 k + 1, so that every global access
// is 16 bytes per lane and 256 consecutive bytes per half warp (32 bytes per lane cost the load/store pipe one pass per lane,
// and 128-byte bulk copies per thread keep issuing while they are waited for: forward 162 -> 155, inverse 159 -> 146 us at 768 limbs).
__device__ __forceinline__ uint32_t padded(uint32_t i) { return i + 2 * (i >> 4); }
constexpr uint32_t ROW_PAD = 256 + 32, ROW_CTA = 4;

// forward, EP 0: in place; 1: the tail of a ModDown or rescale, (u - NTT(conv)) c + sigma_g(add), written to its final
// place; 2: into a tiled buffer; 3: as 1 with u formed here from BETA digits and the key.  EP 3 is bound by HBM (the key words and the
// results); one pair of words per step at 64 registers: two pairs at 96 registers and 20 warps per SM took 1750 us for 64
// rotations, four pairs at 128 registers 1910, against 1550.
template <int EP, bool WIDE, uint32_t BETA = 1, bool ADDP = false>
__global__ void __launch_bounds__(16 * ROW_CTA, 64 / ROW_CTA) ntt_fwd_rows(DevTables c, u64 *base, LimbMap map, uint32_t fp_share, const __grid_constant__ NttEpilogue ep) {
    __shared__ __align__(16) double sm[ROW_CTA * ROW_PAD];
    // EP 3: the entries and components of a limb next to each other, for the sake of its digits and key words in L2
    const uint32_t yl = EP == 3 ? ((blockIdx.y >> 1) % ep.nb * 2 + (blockIdx.y & 1)) * ep.level + (blockIdx.y >> 1) / ep.nb : blockIdx.y;
    const int prime = limb_prime(map, yl);
    if (prime < 0 || (yl & 7) >= fp_share) return leave_out(fp_share);
    const double q = c.modd[prime].x, qinv = c.modd[prime].y;
    const double *tw = c.twd_fwd + ((size_t)prime << c.log_n);
    const uint32_t t = threadIdx.x & 15, rl = threadIdx.x >> 4, row = blockIdx.x * ROW_CTA + rl, R = c.N >> 8;
    u64 *g = base + (limb_index(map, yl) << c.log_n) + (size_t)row * 256;
    double *s = sm + rl * ROW_PAD;
    double x[16];
    grid_dep_sync();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = reinterpret_cast<const double *>(g)[t + 16 * k];
    __syncwarp();
    fwd_row_open(x, tw, R + row, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) s[padded(t + 16 * k)] = x[k];
    __syncwarp();
    double *blk = s + 18 * t;                 // this thread's 16 consecutive coefficients
#pragma unroll
    for (uint32_t k = 0; k < 16; k += 2) {
        const double2 v = *reinterpret_cast<const double2 *>(blk + k);
        x[k] = v.x; x[k + 1] = v.y;
    }
    fwd_row_close(x, tw, 16 * (R + row) + t, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 16; k += 2) *reinterpret_cast<double2 *>(blk + k) = make_double2(x[k], x[k + 1]);
    __syncwarp();
    const double *sp = s + 2 * t + 2 * (t >> 3);          // padded(2 t); word 2 t + 32 k is 36 k further
    if (EP == 1 || EP == 3) {
        const uint32_t y = yl + ep.y0, i = y % ep.level, comp = (y / ep.level) % ep.ncomp, bz = y / (ep.ncomp * ep.level);
        const double2 pinv = ep.pinv[i];
        const uint32_t p0 = row * 256 + 2 * t;
        // grouped: entry bz is key bz / group applied to member bz % group (own: to the entry itself)
        const uint32_t rot = ep.group ? bz / ep.group : bz, mem = ep.group ? bz % ep.group : bz;
        const uint32_t gal = (uint32_t)(ep.multi ? ep.mgalois[rot] : ep.galois);
        const u64 *add = (ep.add_comps >> comp & 1) ? ep.add.at(ep.own ? bz : mem) + (((size_t)comp * (EP == 3 ? ep.add_level : ep.level) + i) << c.log_n) : nullptr;
        const u64 *acc = ep.accumulate ? ep.acc.at(bz) + (((size_t)comp * ep.level + i) << c.log_n) + p0 : nullptr;
        const uint32_t bstep = ep.tl.R ? ep.tl.R * 64 : 64;    // words from one 64-word block of the destination to the next
        u64 *dst = ep.tl.R ? const_cast<u64 *>(ep.out.base) + tiled_index(ep.tl.R, c.N, ep.tl.row0 + rot * ep.rot_rows + (ep.group ? mem : bz) * ep.tl.row_stride + comp, i, row * 256) + 2 * t
                           : const_cast<u64 *>(ep.group ? ep.out.base + rot * ep.rot_stride + mem * ep.out.stride : ep.out.at(bz)) +
                                 (((size_t)comp * ep.level + i) << c.log_n) + p0;
        if (EP == 3) {
            // u = sum_j digit_j key_j; add joins it times P (rescale: the result is scaled by (P q_l)^-1) or the result as it is
            const size_t ks = (size_t)2 * c.T << c.log_n;
            const uint32_t de = ep.shared ? 0 : ep.group && !ep.own ? mem : bz, own = i / c.alpha;
            const u64 *kp = (ep.multi ? ep.mevk[rot] : ep.evk) + (((size_t)comp * c.T + i) << c.log_n) + p0;
            const u64 *eb = ep.ext + (((size_t)de * BETA * ep.nt + i) << c.log_n), *od = ep.d.at(de) + ((size_t)i << c.log_n);
            const double pq = ADDP ? c.dn_p_mod_d[i] : 0.0;
#pragma unroll
            for (uint32_t k = 0; k < 8; k++) {
                const uint32_t sr = galois_src(p0 + 32 * k, gal, c.log_n), so = sr & ~1u;
                const bool odd = sr & 1;
                ulonglong2 kv[BETA], ev[BETA], z;
#pragma unroll
                for (uint32_t j = 0; j < BETA; j++) {
                    kv[j] = ld_pair<true>(kp + j * ks + 32 * k);
                    ev[j] = ld_pair<true>((j == own ? od : eb + (((size_t)j * ep.nt) << c.log_n)) + so);
                }
                if (add) z = ld_pair<true>(add + so);
                __syncwarp();
                // the permutation maps the pair onto a pair, possibly swapped: summed in the digits' order, crossed with the key's
                double s0 = 0.0, s1 = 0.0;
                if (ADDP && add) { s0 = mulmod_dd(u64_to_d(z.x), pq, q, qinv); s1 = mulmod_dd(u64_to_d(z.y), pq, q, qinv); }
#pragma unroll
                for (uint32_t j = 0; j < BETA; j++) {
                    s0 = __dadd_rn(s0, mulmod_dd(u64_to_d(ev[j].x), u64_to_d(odd ? kv[j].y : kv[j].x), q, qinv));
                    s1 = __dadd_rn(s1, mulmod_dd(u64_to_d(ev[j].y), u64_to_d(odd ? kv[j].x : kv[j].y), q, qinv));
                }
                // |u - v| < (0.75 (BETA + 1) + 0.5) q <= 3.5 q, below 2^52: the product may round its quotient to even
                if (BETA > 3) { s0 = reduce_d(s0, q, qinv); s1 = reduce_d(s1, q, qinv); }
                const double2 v = *reinterpret_cast<const double2 *>(sp + 36 * k);
                double r0 = mulmod_d<1>(__dsub_rn(odd ? s1 : s0, reduce_d(v.x, q, qinv)), pinv, q);
                double r1 = mulmod_d<1>(__dsub_rn(odd ? s0 : s1, reduce_d(v.y, q, qinv)), pinv, q);
                if (!ADDP && add) {
                    r0 = __dadd_rn(r0, u64_to_d(odd ? z.y : z.x));
                    r1 = __dadd_rn(r1, u64_to_d(odd ? z.x : z.y));
                }
                if (ep.accumulate) {
                    const ulonglong2 o = ld_pair<true>(acc + 32 * k);
                    r0 = __dadd_rn(r0, u64_to_d(o.x));
                    r1 = __dadd_rn(r1, u64_to_d(o.y));
                }
                st_pair<true>(dst + (k >> 1) * bstep + (k & 1) * 32, make_ulonglong2(canonical_d(reduce_d(r0, q, qinv), q), canonical_d(reduce_d(r1, q, qinv), q)));
            }
            return;
        }
        const u64 *up = ep.u.at(bz) + (((size_t)comp * ep.nt + i) << c.log_n) + p0;
        // the other operands are fetched four pairs at a time, all in flight together (one pair per step, behind the step's
        // arithmetic, was latency bound: 332 us against 243 for 16 key switches at level 24)
        ulonglong2 ua[4], aa[4];
        uint32_t sr[4];
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) {
            if ((k & 3) == 0) {
#pragma unroll
                for (uint32_t h = 0; h < 4; h++) {
                    ua[h] = ld_pair<WIDE>(up + 32 * (k + h));
                    if (add) {      // the permutation maps the pair onto a pair, possibly swapped
                        sr[h] = galois_src(p0 + 32 * (k + h), gal, c.log_n);
                        aa[h] = ld_pair<WIDE>(add + (sr[h] & ~1u));
                    }
                }
                __syncwarp();
            }
            u64 *d = dst + (k >> 1) * bstep + (k & 1) * 32;
            const double2 v = *reinterpret_cast<const double2 *>(sp + 36 * k);
            const ulonglong2 uu = ua[k & 3], a = aa[k & 3];
            // |u - v| < 1.5 q, times P^-1 -> |.| < 0.9 q, plus up to two residues, reduced once
            double r0 = mulmod_d<0>(__dsub_rn(u64_to_d(uu.x), reduce_d(v.x, q, qinv)), pinv, q);
            double r1 = mulmod_d<0>(__dsub_rn(u64_to_d(uu.y), reduce_d(v.y, q, qinv)), pinv, q);
            if (add) {
                const bool odd = sr[k & 3] & 1;
                r0 = __dadd_rn(r0, u64_to_d(odd ? a.y : a.x));
                r1 = __dadd_rn(r1, u64_to_d(odd ? a.x : a.y));
            }
            if (ep.accumulate) {
                const ulonglong2 o = ld_pair<WIDE>(acc + 32 * k);
                r0 = __dadd_rn(r0, u64_to_d(o.x));
                r1 = __dadd_rn(r1, u64_to_d(o.y));
            }
            st_pair<WIDE>(d, make_ulonglong2(canonical_d(reduce_d(r0, q, qinv), q), canonical_d(reduce_d(r1, q, qinv), q)));
        }
        return;
    }
    u64 *dst = g + 2 * t;
    uint32_t bstep = 64;
    if (EP == 2) {
        const uint32_t y = blockIdx.y + ep.y0, i = y % ep.level, b = y / ep.level;
        dst = const_cast<u64 *>(ep.out.base) + tiled_index(ep.tl.R, c.N, ep.tl.row0 + b * ep.tl.row_stride, i, row * 256) + 2 * t;
        bstep = ep.tl.R * 64;
    }
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) {
        const double2 v = *reinterpret_cast<const double2 *>(sp + 36 * k);
        st_pair<WIDE>(dst + (k >> 1) * bstep + (k & 1) * 32, make_ulonglong2(canonical_d(reduce_d(v.x, q, qinv), q), canonical_d(reduce_d(v.y, q, qinv), q)));
    }
}

// inverse (the first pass); src (if any): the input limbs lie elsewhere, entry y / period at src.ptr.at(), limbs src.lpitch apart.
// BETA: the input is the inner product of BETA digits with a key, formed here (a launch and the sum's trip through memory
// less: 64 hoisted rotations at N = 2^16, level 24, 4110 -> 4005 us)
template <bool WIDE, uint32_t BETA = 0, class Src = NttSource>
__global__ void __launch_bounds__(16 * ROW_CTA, 48 / ROW_CTA) ntt_inv_rows(DevTables c, u64 *base, LimbMap map, uint32_t fp_share, const __grid_constant__ Src src) {
    __shared__ __align__(16) double sm[ROW_CTA * ROW_PAD];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) >= fp_share) return leave_out(fp_share);
    const double q = c.modd[prime].x, qinv = c.modd[prime].y;
    const double *tw = c.twd_inv + ((size_t)prime << c.log_n);
    const uint32_t t = threadIdx.x & 15, rl = threadIdx.x >> 4, row = blockIdx.x * ROW_CTA + rl, R = c.N >> 8;
    u64 *g = base + (limb_index(map, blockIdx.y) << c.log_n) + (size_t)row * 256;
    const u64 *gs = g;
    if constexpr (BETA == 0)
        if (src.lpitch) gs = src.ptr.at(blockIdx.y / map.period) + (((size_t)(blockIdx.y % map.period) * src.lpitch) << c.log_n) + (size_t)row * 256;
    double *s = sm + rl * ROW_PAD, *blk = s + 18 * t;
    double *sp = s + 2 * t + 2 * (t >> 3);
    double x[16];
    grid_dep_sync();
    if constexpr (BETA > 0) {
        const uint32_t e = blockIdx.y / map.period, comp = e & 1, bz = e >> 1, xl = src.x0 + blockIdx.y % map.period, p0 = row * 256 + 2 * t;
        const uint32_t rot = src.group ? bz / src.group : bz, mem = src.group ? bz % src.group : bz;
        const uint32_t gal = (uint32_t)(src.multi ? src.mgalois[rot] : src.galois), de = src.shared ? 0 : src.group && !src.own ? mem : bz;
        const bool main = xl < src.add_level;               // a q-limb: some digit has it among its own, P add counts
        const uint32_t own = main ? xl / c.alpha : BETA;
        const size_t ks = (size_t)2 * c.T << c.log_n;
        const u64 *kp = (src.multi ? src.mevk[rot] : src.evk) + (((size_t)comp * c.T + prime) << c.log_n) + p0;
        const u64 *eb = src.ext + (((size_t)de * BETA * src.nt + xl) << c.log_n), *od = src.d.at(de) + ((size_t)xl << c.log_n);
        const u64 *add = src.add_p && main ? src.add.at(bz) + (((size_t)comp * src.add_level + xl) << c.log_n) + p0 : nullptr;
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) {
            const uint32_t sr = galois_src(p0 + 32 * k, gal, c.log_n), so = sr & ~1u;
            const bool odd = sr & 1;
            ulonglong2 kv[BETA], ev[BETA];
#pragma unroll
            for (uint32_t j = 0; j < BETA; j++) {
                kv[j] = ld_pair<true>(kp + j * ks + 32 * k);
                ev[j] = ld_pair<true>((j == own ? od : eb + (((size_t)j * src.nt) << c.log_n)) + so);
            }
            __syncwarp();
            double s0 = 0.0, s1 = 0.0;
            if (add) {
                const ulonglong2 z = ld_pair<true>(add + 32 * k);
                const double pq = c.dn_p_mod_d[xl];
                s0 = mulmod_dd(u64_to_d(z.x), pq, q, qinv); s1 = mulmod_dd(u64_to_d(z.y), pq, q, qinv);
            }
#pragma unroll
            for (uint32_t j = 0; j < BETA; j++) {
                s0 = __dadd_rn(s0, mulmod_dd(u64_to_d(odd ? ev[j].y : ev[j].x), u64_to_d(kv[j].x), q, qinv));
                s1 = __dadd_rn(s1, mulmod_dd(u64_to_d(odd ? ev[j].x : ev[j].y), u64_to_d(kv[j].y), q, qinv));
            }
            *reinterpret_cast<double2 *>(sp + 36 * k) = make_double2(reduce_d(s0, q, qinv), reduce_d(s1, q, qinv));
        }
    } else {
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) {
            const ulonglong2 v = ld_pair<WIDE>(gs + 2 * t + 32 * k);
            x[2 * k] = u64_to_d(v.x); x[2 * k + 1] = u64_to_d(v.y);
        }
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) *reinterpret_cast<double2 *>(sp + 36 * k) = make_double2(x[2 * k], x[2 * k + 1]);
    }
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 16; k += 2) {
        const double2 v = *reinterpret_cast<const double2 *>(blk + k);
        x[k] = v.x; x[k + 1] = v.y;
    }
    inv_row_group<1>(x, tw, 16 * (R + row) + t, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 16; k += 2) *reinterpret_cast<double2 *>(blk + k) = make_double2(x[k], x[k + 1]);
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = s[padded(t + 16 * k)];
    inv_row_group<2>(x, tw, R + row, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) reinterpret_cast<double *>(g)[t + 16 * k] = x[k];
}

// ---- both passes in one kernel: a cluster of CTAs per limb --------------------------------------------------------------
// CL CTAs hold a limb in shared memory: CTA c does the column stages of 256 / CL columns, the values cross to the CTAs that
// own their rows through distributed shared memory, and CTA d does the row stages of R / CL rows (inverse: the other way
// round).  Two cluster barriers: one, split around the second group's arithmetic, keeps values from landing in an exchange buffer
// that is still being read; the other follows the crossing.
template <uint32_t LOGR>
struct ClShape {
    static constexpr uint32_t LOG = LOGR, R = 1u << LOGR, CL = LOGR == 6 ? 8 : 4;
    static constexpr uint32_t A = 4, B = LOGR - 4;                             // column stages: 4, then 0 .. 2
    static constexpr uint32_t COLS = 256 / CL, ROWS = R / CL, THREADS = ROWS * 16;
    static constexpr uint32_t SMEM = (ROWS * ROW_PAD > R * COLS ? ROWS * ROW_PAD : R * COLS) * 8;
};
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_addr(const double *p, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_store(uint32_t a, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(a), "d"(v) : "memory"); }

template <uint32_t LOGR>
__global__ void __launch_bounds__(ClShape<LOGR>::THREADS, 1024 / ClShape<LOGR>::THREADS) ntt_fwd_cluster(DevTables c, u64 *base, LimbMap map, bool doubles) {
    using S = ClShape<LOGR>;
    extern __shared__ __align__(16) double dsm[];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0) return;                  // the whole cluster
    const double q = c.modd[prime].x, qinv = c.modd[prime].y;
    const double *tw = c.twd_fwd + ((size_t)prime << c.log_n);
    const uint32_t rank = blockIdx.x;
    u64 *limb = base + (limb_index(map, blockIdx.y) << c.log_n);
    double x[16];
    {
        const uint32_t cc = threadIdx.x % S::COLS, r = threadIdx.x / S::COLS;
        constexpr uint32_t RS = S::R / 16;
        const u64 *gs = limb + rank * S::COLS + cc;
        grid_dep_sync();
#pragma unroll
        for (uint32_t k = 0; k < 16; k++) {
            const u64 v = gs[(size_t)(r + RS * k) * 256];
            x[k] = doubles ? __longlong_as_double((long long)v) : u64_to_d(v);
        }
        __syncwarp();
        fwd_col_group<LOGR, 0, 4>(x, 0, tw, 1, q, qinv);
        if constexpr (S::B > 0) {
#pragma unroll
            for (uint32_t k = 0; k < 16; k++) dsm[(r + RS * k) * S::COLS + cc] = x[k];
            __syncthreads();
#pragma unroll
            for (uint32_t k = 0; k < 16; k++) x[k] = dsm[(16 * r + k) * S::COLS + cc];
            cluster_arrive();
#pragma unroll
            for (uint32_t j = 0; j < (16u >> S::B); j++) fwd_col_group<LOGR, 4, S::B>(x, j << S::B, tw, 16 + r * (16 >> S::B) + j, q, qinv);
        } else {
            cluster_arrive();
        }
        cluster_wait();                     // (without a second group: the peers have started)
        // 16 consecutive rows (S::B = 0: all of them) of one column to the CTAs that own them
        const uint32_t col = padded(rank * S::COLS + cc);
#pragma unroll
        for (uint32_t k0 = 0; k0 < 16; k0 += S::ROWS) {
            const uint32_t row = (S::B ? 16 * r : 0) + k0;
            const uint32_t a = cluster_addr(dsm + col, row / S::ROWS);
#pragma unroll
            for (uint32_t k = 0; k < S::ROWS; k++) cluster_store(a + k * ROW_PAD * 8, x[k0 + k]);
        }
        cluster_arrive();
        cluster_wait();
    }
    const uint32_t t = threadIdx.x & 15, rl = threadIdx.x >> 4, row = rank * S::ROWS + rl;
    double *s = dsm + rl * ROW_PAD, *blk = s + 18 * t;
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = s[padded(t + 16 * k)];
    fwd_row_open(x, tw, S::R + row, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) s[padded(t + 16 * k)] = x[k];
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 16; k += 2) {
        const double2 v = *reinterpret_cast<const double2 *>(blk + k);
        x[k] = v.x; x[k + 1] = v.y;
    }
    fwd_row_close(x, tw, 16 * (S::R + row) + t, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 16; k += 2) *reinterpret_cast<double2 *>(blk + k) = make_double2(x[k], x[k + 1]);
    __syncwarp();
    const double *sp = s + 2 * t + 2 * (t >> 3);
    u64 *dst = limb + (size_t)row * 256 + 2 * t;
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) {
        const double2 v = *reinterpret_cast<const double2 *>(sp + 36 * k);
        st_pair<true>(dst + 32 * k, make_ulonglong2(canonical_d(reduce_d(v.x, q, qinv), q), canonical_d(reduce_d(v.y, q, qinv), q)));
    }
}

template <uint32_t LOGR>
__global__ void __launch_bounds__(ClShape<LOGR>::THREADS, 1024 / ClShape<LOGR>::THREADS) ntt_inv_cluster(DevTables c, u64 *base, LimbMap map, const __grid_constant__ NttSource src,
                                                                                                           const double2 *scale) {
    using S = ClShape<LOGR>;
    extern __shared__ __align__(16) double dsm[];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0) return;
    const double q = c.modd[prime].x, qinv = c.modd[prime].y;
    const double *tw = c.twd_inv + ((size_t)prime << c.log_n);
    const uint32_t rank = blockIdx.x;
    u64 *limb = base + (limb_index(map, blockIdx.y) << c.log_n);
    double x[16];
    {
        const uint32_t t = threadIdx.x & 15, rl = threadIdx.x >> 4, row = rank * S::ROWS + rl;
        const u64 *gs = (src.lpitch ? src.ptr.at(blockIdx.y / map.period) + (((size_t)(blockIdx.y % map.period) * src.lpitch) << c.log_n) : limb) + (size_t)row * 256;
        double *s = dsm + rl * ROW_PAD, *blk = s + 18 * t, *sp = s + 2 * t + 2 * (t >> 3);
        grid_dep_sync();
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) {
            const ulonglong2 v = ld_pair<true>(gs + 2 * t + 32 * k);
            x[2 * k] = u64_to_d(v.x); x[2 * k + 1] = u64_to_d(v.y);
        }
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) *reinterpret_cast<double2 *>(sp + 36 * k) = make_double2(x[2 * k], x[2 * k + 1]);
        __syncwarp();
#pragma unroll
        for (uint32_t k = 0; k < 16; k += 2) {
            const double2 v = *reinterpret_cast<const double2 *>(blk + k);
            x[k] = v.x; x[k + 1] = v.y;
        }
        inv_row_group<1>(x, tw, 16 * (S::R + row) + t, q, qinv);
#pragma unroll
        for (uint32_t k = 0; k < 16; k += 2) *reinterpret_cast<double2 *>(blk + k) = make_double2(x[k], x[k + 1]);
        __syncwarp();
#pragma unroll
        for (uint32_t k = 0; k < 16; k++) x[k] = s[padded(t + 16 * k)];
        cluster_arrive();
        inv_row_group<2>(x, tw, S::R + row, q, qinv);
        cluster_wait();
        // columns t + 16 k of this row to the CTAs that own them
        constexpr uint32_t KC = S::COLS / 16;
#pragma unroll
        for (uint32_t k0 = 0; k0 < 16; k0 += KC) {
            const uint32_t a = cluster_addr(dsm + row * S::COLS + t, k0 / KC);
#pragma unroll
            for (uint32_t k = 0; k < KC; k++) cluster_store(a + k * 128, x[k0 + k]);
        }
        cluster_arrive();
        cluster_wait();
    }
    const uint32_t cc = threadIdx.x % S::COLS, r = threadIdx.x / S::COLS;
    constexpr uint32_t RS = S::R / 16;
    const double2 *sc = scale ? scale + 2 * (blockIdx.y % map.period) : c.n_inv_d + 2 * prime;
    const double2 c0 = sc[0], c1 = sc[1];
    if constexpr (S::B > 0) {
#pragma unroll
        for (uint32_t k = 0; k < 16; k++) x[k] = dsm[(16 * r + k) * S::COLS + cc];
#pragma unroll
        for (uint32_t j = 0; j < (16u >> S::B); j++) inv_col_open<S::B>(x, j << S::B, tw, 16 + r * (16 >> S::B) + j, q, qinv);
#pragma unroll
        for (uint32_t k = 0; k < 16; k++) dsm[(16 * r + k) * S::COLS + cc] = x[k];
        __syncthreads();
    }
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) x[k] = dsm[(r + RS * k) * S::COLS + cc];
    inv_col_last<4, S::B>(x, tw, q, qinv, c0, c1);
    u64 *g = limb + rank * S::COLS + cc;
#pragma unroll
    for (uint32_t k = 0; k < 16; k++) g[(size_t)(r + RS * k) * 256] = canonical_d(x[k], q);
}

template <uint32_t LOGR>
void launch_cols(const ckks_ctx *c, u64 *b, uint32_t ny, const LimbMap &map, bool inverse, uint32_t share, const NttPrologue *pro, const double2 *scale, cudaStream_t s) {
    const dim3 grid(256 / ColShape<LOGR>::COLS, ny);
    const uint32_t th = ColShape<LOGR>::THREADS;
    if (inverse) launch(ntt_inv_cols<LOGR>, grid, th, 0, s, c->dev, b, map, share, scale);
    else if (!pro) launch(ntt_fwd_cols<LOGR, SRC_LIMBS>, grid, th, 0, s, c->dev, b, map, share, (const u64 *)nullptr, 0u);
    else if (pro->doubles) launch(ntt_fwd_cols<LOGR, SRC_DOUBLES>, grid, th, 0, s, c->dev, b, map, share, (const u64 *)nullptr, 0u);
    else if (pro->lift) launch(ntt_fwd_cols<LOGR, SRC_LIFT>, grid, th, 0, s, c->dev, b, map, share, pro->src, pro->src_prime);
    else launch(ntt_fwd_cols<LOGR, SRC_COEFS>, grid, th, 0, s, c->dev, b, map, share, pro->src, 0u);
}

}  // namespace

// Transforms of a few limbs of a small ring without a fused prologue or epilogue, both passes in one launch.  Returns false outside
// its range, N = 2^12 .. 2^14 and at most two CTAs per SM.  For short calls: these are bound by the host, whom a launch costs
// 2 us (N = 2^14: product and rescale 53 -> 47 us; N = 2^13: rotation 33.5 -> 29.5 us), while on the device this kernel's 5.8 to
// 7.8 us lose to the two passes' 2.3 to 3.7 us each, so that longer calls keep those (a 64 x 64 projection at N = 2^13: 177 against
// 188 us).  At N = 2^16 the same form with 8 and 16 CTAs per cluster took 431 and 417 us against 305 for 768 limbs.
static bool launch_ntt_small(const ckks_ctx *c, u64 *base, uint32_t nlimbs, const LimbMap &map, bool inverse, cudaStream_t s, const NttSource *src, const double2 *inv_scale, bool doubles) {
    if (c->log_n < 12 || c->log_n > 14 || !aligned16(base) || (src && !aligned16(src->ptr))) return false;
    auto run = [&](auto shape) {
        using S = decltype(shape);
        if (nlimbs * S::CL > 2 * (uint32_t)c->sms) return false;
        const dim3 grid(S::CL, nlimbs);
        if (inverse) launch_clusters(ntt_inv_cluster<S::LOG>, S::CL, grid, S::THREADS, S::SMEM, s, c->dev, base, map, src ? *src : NttSource{}, inv_scale);
        else launch_clusters(ntt_fwd_cluster<S::LOG>, S::CL, grid, S::THREADS, S::SMEM, s, c->dev, base, map, doubles);
        return true;
    };
    return c->log_n == 14 ? run(ClShape<6>()) : c->log_n == 13 ? run(ClShape<5>()) : run(ClShape<4>());
}

void launch_ntt(const ckks_ctx *c, u64 *base, uint32_t nlimbs_total, const LimbMap &map, bool inverse, cudaStream_t s, const NttEpilogue *ep,
                const NttPrologue *pro, const NttSource *src, const double2 *inv_scale, bool alone) {
    if (alone && !ep && (!pro || pro->doubles) && launch_ntt_small(c, base, nlimbs_total, map, inverse, s, src, inv_scale, pro != nullptr)) return;
    const uint32_t R = c->N >> 8;
    // the integer path (an option, N = 2^16) has no fused forms: those take all limbs on the FP64 pipe
    const uint32_t share = (ep || pro || inv_scale || (src && src->ptr.n) || c->log_n != 16) ? 8 : c->ntt_fp_share;
    // grid.y is limited to 65535: go in chunks that are whole repeats of the limb map, a period of every digit where they differ (a
    // multiple of 8 limbs apart only matters to the integer share, which is a choice of limbs and not part of the result)
    const uint32_t repeat = map.period * map.nbeta, chunk = std::max(1u, 32768 / repeat) * repeat;
    for (uint32_t y0 = 0; y0 < nlimbs_total; y0 += chunk) {
        const uint32_t ny = nlimbs_total - y0 < chunk ? nlimbs_total - y0 : chunk;
        u64 *b = base + (limb_index(map, y0) << c->log_n);
        NttPrologue pr;
        if (pro) pr = *pro;
        if (pr.src) { pr.src += (size_t)(y0 / map.period) << c->log_n; }
        NttSource sr;
        if (src) { sr = *src; if (!sr.ptr.n) sr.ptr.base += (size_t)(y0 / map.period) * sr.ptr.stride; }
        auto cols = [&]() {
            switch (c->log_n) {
                case 16: return launch_cols<8>(c, b, ny, map, inverse, share, pro ? &pr : nullptr, inv_scale, s);
                case 15: return launch_cols<7>(c, b, ny, map, inverse, share, pro ? &pr : nullptr, inv_scale, s);
                case 14: return launch_cols<6>(c, b, ny, map, inverse, share, pro ? &pr : nullptr, inv_scale, s);
                case 13: return launch_cols<5>(c, b, ny, map, inverse, share, pro ? &pr : nullptr, inv_scale, s);
                case 12: return launch_cols<4>(c, b, ny, map, inverse, share, pro ? &pr : nullptr, inv_scale, s);
                case 11: return launch_cols<3>(c, b, ny, map, inverse, share, pro ? &pr : nullptr, inv_scale, s);
                default: return launch_cols<2>(c, b, ny, map, inverse, share, pro ? &pr : nullptr, inv_scale, s);
            }
        };
        const dim3 grid(R / ROW_CTA, ny);
        if (share > 0 && !inverse) {
            cols();
            bool wide = aligned16(ep ? (const void *)nullptr : (const void *)b);
            if (ep) wide = aligned16(ep->u) && aligned16(ep->add) && aligned16(ep->acc) && aligned16(ep->out) && (ep->rot_stride & 1) == 0;
            NttEpilogue e = ep ? *ep : NttEpilogue{};
            e.y0 = y0;
            const int mode = ep ? ep->mode : 0;
            static constexpr decltype(&ntt_fwd_rows<0, true>) inner[2][IP_FUSED_BETA] = {
                {ntt_fwd_rows<3, true, 1>, ntt_fwd_rows<3, true, 2>, ntt_fwd_rows<3, true, 3>, ntt_fwd_rows<3, true, 4>},
                {ntt_fwd_rows<3, true, 1, true>, ntt_fwd_rows<3, true, 2, true>, ntt_fwd_rows<3, true, 3, true>, ntt_fwd_rows<3, true, 4, true>}};
            auto *k = mode == 3 ? inner[e.add_p][e.beta - 1]
                    : mode == 1 ? (wide ? ntt_fwd_rows<1, true> : ntt_fwd_rows<1, false>)
                    : mode == 2 ? (wide ? ntt_fwd_rows<2, true> : ntt_fwd_rows<2, false>)
                                : (wide ? ntt_fwd_rows<0, true> : ntt_fwd_rows<0, false>);
            launch(k, grid, 16 * ROW_CTA, 0, s, c->dev, b, map, share, e);
        } else if (share > 0) {
            const NttSource none{};
            const bool wide = src ? aligned16(src->ptr) : aligned16(b);
            static constexpr decltype(&ntt_inv_rows<true, 1, NttEpilogue>) inner[IP_FUSED_BETA] = {
                ntt_inv_rows<true, 1, NttEpilogue>, ntt_inv_rows<true, 2, NttEpilogue>, ntt_inv_rows<true, 3, NttEpilogue>, ntt_inv_rows<true, 4, NttEpilogue>};
            if (ep) launch(inner[ep->beta - 1], grid, 16 * ROW_CTA, 0, s, c->dev, b, map, share, *ep);
            else launch(wide ? ntt_inv_rows<true> : ntt_inv_rows<false>, grid, 16 * ROW_CTA, 0, s, c->dev, b, map, share, src ? sr : none);
            cols();
        }
        if (share < 8) launch_ntt_int(c, b, ny, map, inverse, sr, s);
    }
}

// grid: three CTAs per SM, all resident at once.  Returns the butterflies one launch performs.
uint64_t launch_butterfly_probe(const ckks_ctx *c, uint32_t iters, u64 *sink, cudaStream_t s) {
    const uint32_t ctas = (uint32_t)c->sms * 3;
    launch(butterfly_probe_kernel, ctas, F_THREADS, 0, s, c->dev, iters, sink);
    return (uint64_t)ctas * F_THREADS * iters * 32;
}
