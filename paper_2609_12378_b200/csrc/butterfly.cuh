// Butterflies of the negacyclic transform on registers, shared by the transform kernels (ntt.cu) and by the kernel that runs an
// inverse column pass, a basis conversion and a forward column pass in one (conv_ntt.cu).
#pragma once
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
// keeps the row pass's input at or below 3.20 for every N.  From 1.25 q, which the conversions of conv_ntt.cu hand over, it is
//   1.91 2.64 3.48 4.41 | 5.96c 7.71c | 2.46c 3.27 and 4.18 5.70c 7.42c | 2.43c | 3.23 4.13 5.65c 7.36c.

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

// Row passes.
// 16 threads per row, a row in one half warp, so warps need no barrier between them; 4 rows per CTA (16 were
// 2 % slower: finer CTAs keep the phases of an SM's warps apart).  In the exchange row two spare words
// follow every 16, so that a thread's own 16 consecutive coefficients are a 16-byte aligned block at a pitch of 144 bytes:
// 8-byte accesses of consecutive lanes and 16-byte accesses to the own block are both conflict free.  Words enter and leave
// through the row too, as pairs: lane t of a half warp moves words 2 t + 32 k and 2 t + 32 k + 1, so that every global access
// is 16 bytes per lane and 256 consecutive bytes per half warp (32 bytes per lane cost the load/store pipe one pass per lane,
// and 128-byte bulk copies per thread keep issuing while they are waited for: forward 162 -> 155, inverse 159 -> 146 us at 768 limbs).
__device__ __forceinline__ uint32_t padded(uint32_t i) { return i + 2 * (i >> 4); }
constexpr uint32_t ROW_PAD = 256 + 32, ROW_CTA = 4;


// ---- a row by a warp: eight coefficients per lane, stages in groups of 3, 3 and 2 -----------------------------------------------
// Half the chain of dependent operations and twice the warps of sixteen lanes per row, for more exchanges: where a launch is bound by
// latency (mid_rows.cu, the row passes of few limbs).  The exchange row has four spare words behind every 32.
constexpr uint32_t WROW_PAD = 256 + 32;
__device__ __forceinline__ uint32_t wrow_at(uint32_t i) { return i + 4 * (i >> 5); }
// words t + 32 k of the row in v (3.27 q) -> the row's results at s, in order, at most half a prime; base: R + row
__device__ __forceinline__ void wrow_forward(double (&v)[8], double *s, uint32_t t, const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    const uint32_t b32 = wrow_at(t / 4 * 32) + t % 4;              // word 32 b + s, the lane's place in the middle group
    fwd_stage<1, 8, false, false>(v, 0, tw, base, q, qinv);
    fwd_stage<2, 8, true, false>(v, 0, tw, base, q, qinv);
    fwd_stage<4, 8, true, false>(v, 0, tw, base, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) s[t + 36 * k] = v[k];
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) v[k] = s[b32 + 4 * k];
    fwd_stage<1, 8, true, true>(v, 0, tw, 8 * base + t / 4, q, qinv);
    fwd_stage<2, 8, false, false>(v, 0, tw, 8 * base + t / 4, q, qinv);
    fwd_stage<4, 8, false, false>(v, 0, tw, 8 * base + t / 4, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) s[b32 + 4 * k] = v[k];
    __syncwarp();
    // words 4 t .. and 128 + 4 t ..
#pragma unroll
    for (uint32_t h = 0; h < 2; h++) {
        double *blk = s + wrow_at(4 * t) + 144 * h;
#pragma unroll
        for (uint32_t k = 0; k < 4; k += 2) {
            const double2 w = *reinterpret_cast<const double2 *>(blk + k);
            v[4 * h + k] = w.x; v[4 * h + k + 1] = w.y;
        }
        fwd_stage<1, 4, true, false>(v, 4 * h, tw, 64 * base + 32 * h + t, q, qinv);
        fwd_stage<2, 4, true, false>(v, 4 * h, tw, 64 * base + 32 * h + t, q, qinv);
#pragma unroll
        for (uint32_t k = 0; k < 4; k += 2)
            *reinterpret_cast<double2 *>(blk + k) = make_double2(reduce_d(v[4 * h + k], q, qinv), reduce_d(v[4 * h + k + 1], q, qinv));
    }
}
// Bounds of the inverse row pass in groups of 2, 3 and 3 stages from canonical residues; it ends below inv_in(3) (see gs_plan)
constexpr double WROW_IN0 = 1.0, WROW_T0 = 1.5, WROW_IN1 = gs_out(2, WROW_IN0, WROW_T0), WROW_T1 = 1.44, WROW_IN2 = gs_out(3, WROW_IN1, WROW_T1), WROW_T2 = 1.8;
static_assert(gs_out(3, WROW_IN2, WROW_T2) <= inv_in(3), "the column pass takes these values");
#define WROW_INV(S, G, IN, THR, X0, BASE) inv_stage<S, G, gs_pre(G, IN, THR, false, S), gs_coarse(G, IN, THR, false, S), false>(v, X0, tw, BASE, q, qinv)
// the row at s, in order -> words t + 32 k in v
__device__ __forceinline__ void wrow_inverse(double (&v)[8], double *s, uint32_t t, const double *__restrict__ tw, uint32_t base, double q, double qinv) {
    const uint32_t b32 = wrow_at(t / 4 * 32) + t % 4;
#pragma unroll
    for (uint32_t h = 0; h < 2; h++) {
        double *blk = s + wrow_at(4 * t) + 144 * h;
#pragma unroll
        for (uint32_t k = 0; k < 4; k += 2) {
            const double2 w = *reinterpret_cast<const double2 *>(blk + k);
            v[4 * h + k] = w.x; v[4 * h + k + 1] = w.y;
        }
        WROW_INV(0, 2, WROW_IN0, WROW_T0, 4 * h, 64 * base + 32 * h + t);
        WROW_INV(1, 2, WROW_IN0, WROW_T0, 4 * h, 64 * base + 32 * h + t);
        reduce_masked<gs_post(2, WROW_IN0, WROW_T0, false), 4>(v, 4 * h, q, qinv);
#pragma unroll
        for (uint32_t k = 0; k < 4; k += 2) *reinterpret_cast<double2 *>(blk + k) = make_double2(v[4 * h + k], v[4 * h + k + 1]);
    }
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) v[k] = s[b32 + 4 * k];
    WROW_INV(0, 3, WROW_IN1, WROW_T1, 0, 8 * base + t / 4);
    WROW_INV(1, 3, WROW_IN1, WROW_T1, 0, 8 * base + t / 4);
    WROW_INV(2, 3, WROW_IN1, WROW_T1, 0, 8 * base + t / 4);
    reduce_masked<gs_post(3, WROW_IN1, WROW_T1, false), 8>(v, 0, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) s[b32 + 4 * k] = v[k];
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) v[k] = s[t + 36 * k];
    WROW_INV(0, 3, WROW_IN2, WROW_T2, 0, base);
    WROW_INV(1, 3, WROW_IN2, WROW_T2, 0, base);
    WROW_INV(2, 3, WROW_IN2, WROW_T2, 0, base);
    reduce_masked<gs_post(3, WROW_IN2, WROW_T2, false), 8>(v, 0, q, qinv);
}
#undef WROW_INV

}  // namespace
