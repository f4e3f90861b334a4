// Inverse column pass, basis conversion and forward column pass in one kernel.
//
// Between the row passes of a key switch's transforms everything stays inside a column: the inverse transform of a conversion's
// source limbs ends with their column pass, the conversion takes each coefficient by itself, and the forward transform of its
// targets starts with their column pass.  A CTA takes a strip of columns of all sources of one conversion, keeps their
// coefficients in shared memory and walks a chunk of the targets, so that neither the sources' coefficients nor the converted
// limbs make a trip through memory between these steps, and three launches are one.
#include <type_traits>

#include "butterfly.cuh"

namespace {

// Shape for R = 2^LOGR rows: strips of 2048 words (eight columns at N = 2^16), one CTA of 16 warps per SM, four groups of TG = 128
// threads.  A transform of a limb's strip is a group's, sixteen coefficients per thread, as in the column passes of ntt.cu: radix 16,
// an exchange, the other stages.  For the targets the groups have different roles, so that every scheduler always has warps of both
// kinds and none waits for the other's loads: two convert, CPT = 8 coefficients per thread with all their sources in registers, and
// pass one target after the other through BUFFERS buffers to the two that transform them.  (All groups doing both in turn, with the
// sources in shared memory: 395 us for the ModDowns of sixteen hoisted rotations at N = 2^16, level 24; with the sources in registers
// and a barrier of the CTA per batch of targets: 416; in this form 354, the FP64 pipe busy 71 % of its cycles.  The three kernels this
// replaces take 344 one by one, but move another 64 MiB per rotation, which under the power limit costs more than they save.)
template <uint32_t LOGR>
struct StripShape {
    static constexpr uint32_t R = 1u << LOGR, A = 4, B = LOGR - A, E = 16, RS = R / E;
    static constexpr uint32_t LIMB = 2048, COLS = LIMB / R, TG = LIMB / E, GROUPS = 4, THREADS = TG * GROUPS, CONV = 2 * TG, CPT = LIMB / CONV;
    static constexpr uint32_t BUFFERS = 4;
    // exchange index: with eight columns a half warp reads two rows sixteen apart, which this puts into different banks
    static __device__ __forceinline__ uint32_t at(uint32_t row, uint32_t cc) { return (COLS == 8 ? row ^ (row >> 4 & 1) : row) * COLS + cc; }
};
constexpr uint32_t STRIP_CHUNK = 32, STRIP_NS = 8;         // targets and sources of a CTA at most
// Registers per thread of the two roles.  256 (176 + 80) = 512 x 128, which is what the CTA is launched with (every instance is compiled
// to 128): more in sum would wait for registers that nobody gives back.  Eight sources spill: 36 to 96 bytes per thread stored, 64 to 144
// read, more of them the larger the ring.
constexpr uint32_t CONV_REGS = 176, NTT_REGS = 80;
static_assert(CONV_REGS + NTT_REGS == 256, "the two halves of the CTA share the registers of its launch");

__device__ __forceinline__ void group_sync(uint32_t id, uint32_t threads) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void group_arrive(uint32_t id, uint32_t threads) { asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); }

// out[p] (+)= sum_a y[p][a] w[a] mod t (see CONV_SIGMA; out enters below t).  The quotient of the whole sum is formed in two roundings,
// k = round(lo / t + round(hi / t)), hi / t below 2^51 and the low parts with out below 2^53: |out| <= (1/2 + 1/4 + 1/2) t = 1.25 t.
// FULL: ns = NS, without a branch per source, so that the constants' fetches run ahead of the products.
template <bool FIRST, bool FULL, uint32_t NS, uint32_t CPT>
__device__ __forceinline__ void strip_dot(const double (&y)[CPT][NS], const double *w, uint32_t ns, double t, double tinv, double (&out)[CPT]) {
    double H[CPT];
#pragma unroll
    for (uint32_t a = 0; a < NS; a++) {
        if (!FULL && a >= ns) break;
        const double wa = w[a];
#pragma unroll
        for (uint32_t p = 0; p < CPT; p++) {
            const double h = a ? H[p] : CONV_SIGMA;
            H[p] = __fma_rn(y[p][a], wa, h);
            const double l = __fma_rn(y[p][a], wa, -__dsub_rn(H[p], h));
            out[p] = FIRST && a == 0 ? l : __dadd_rn(out[p], l);
        }
    }
#pragma unroll
    for (uint32_t p = 0; p < CPT; p++) {
        const double hs = __dsub_rn(H[p], CONV_SIGMA);
        const double k = __dsub_rn(__fma_rn(out[p], tinv, __fma_rn(hs, tinv, MAGIC0)), MAGIC0);
        out[p] = __dadd_rn(out[p], __fma_rn(-k, t, hs));
    }
}

// The CTAs of a launch: strips by chunks of targets (x, y), or, with `whole`, in one row: the first `whole` take a strip with all its
// targets, the others one of the `split` remaining ones with `chunk` targets.  (The short launches are of the first kind, which has no
// arithmetic in the way of their start: a rotation at N = 2^15, level 4 30.4 us, with one row for both and two divisions 31.0.)
struct StripGrid { uint32_t whole, split, chunk; };

// src: limbs after the inverse row pass (signed doubles); dst: limbs for the forward row pass.  NS: sources at most
template <uint32_t LOGR, int MODE, uint32_t NS>
__global__ void __launch_bounds__(StripShape<LOGR>::THREADS, 1) conv_cols(DevTables c, const double *src, double *dst, uint32_t level, uint32_t targets, StripGrid grid) {
    using S = StripShape<LOGR>;
    constexpr uint32_t E = S::E, R = S::R, RS = S::RS, LIMB = S::LIMB, COLS = S::COLS, TG = S::TG, GROUPS = S::GROUPS, CPT = S::CPT;
    constexpr bool RESC = MODE == CONV_DOWN_RS;
    extern __shared__ __align__(16) double ssm[];
    const uint32_t grp = threadIdx.x / TG, tid = threadIdx.x % TG, cc = tid % COLS, r = tid / COLS;
    constexpr uint32_t STRIPS = 256 / COLS;                   // of an item
    uint32_t strip = blockIdx.x, x0 = blockIdx.y * grid.chunk, take = grid.chunk;
    if (grid.whole) {
        if (strip < grid.whole) take = targets;
        else
#pragma unroll 1
            for (; strip >= grid.whole + grid.split; strip -= grid.split) x0 += grid.chunk;
    }
    const uint32_t col = strip % STRIPS * COLS + cc;
    double *bufs = ssm;                                       // [sources][LIMB] (the dropped limb last); the first BUFFERS pass targets later
    double *stw = bufs + (NS > S::BUFFERS ? NS : S::BUFFERS) * LIMB + (RESC ? LIMB : 0);       // [GROUPS][R] twiddles
    double2 *s_m = reinterpret_cast<double2 *>(stw + GROUPS * R);       // the targets' primes and inverses
    double *s_w = reinterpret_cast<double *>(s_m + STRIP_CHUNK);        // [targets of the chunk (+ the dropped limb)][NS] constants
    double *dropped = bufs + (NS > S::BUFFERS ? NS : S::BUFFERS) * LIMB;
    // the conversion's sources and targets
    const uint32_t item = strip / STRIPS;
    const uint32_t beta = MODE == CONV_UP ? (level + c.alpha - 1) / c.alpha : 1, j = MODE == CONV_UP ? item % beta : 0, bz = item / beta;
    const uint32_t lo = j * c.alpha, nd = MODE == CONV_UP ? min(c.alpha, level - lo) : c.K;
    const uint32_t nt = level + c.K;
    const uint32_t x1 = min(x0 + take, MODE == CONV_UP ? nt - nd : targets);      // ModUp: counted without the digit's own limbs
    if (x0 >= x1) return;
    auto target_limb = [&](uint32_t xt) { return MODE == CONV_UP && xt >= lo ? xt + nd : xt; };
    auto target_prime = [&](uint32_t xt) { const uint32_t x = target_limb(xt); return MODE == CONV_UP && x >= level ? c.L + (x - level) : x; };
    if (threadIdx.x < x1 - x0) s_m[threadIdx.x] = c.modd[target_prime(x0 + threadIdx.x)];
    for (uint32_t e = threadIdx.x; e < (x1 - x0 + RESC) * NS; e += S::THREADS) {
        const uint32_t xi = e / NS, a = e % NS;
        if (a >= nd) continue;
        if (MODE == CONV_UP) s_w[e] = c.up_hat_mod_d[(((size_t)level * c.dnum + j) * c.T + target_prime(x0 + xi)) * c.alpha + a];
        else s_w[e] = c.dn_hat_mod_d[(size_t)(RESC && xi == x1 - x0 ? targets : x0 + xi) * c.K + a];
    }
    src += MODE == CONV_UP ? ((size_t)bz * level + lo) << c.log_n : ((size_t)item * nt + level) << c.log_n;
    dst += (size_t)(item * (MODE == CONV_UP ? nt : targets)) << c.log_n;
    double x[E];
    grid_dep_sync();
    // ---- sources (the dropped limb last): inverse column pass (see ntt_inv_cols), each in a buffer of its own
    for (uint32_t a = grp; a < nd + RESC; a += GROUPS) {
        const bool drop = RESC && a == nd;
        const uint32_t prime = MODE == CONV_UP ? lo + a : drop ? level - 1 : c.L + a;
        const double q = c.modd[prime].x, qinv = c.modd[prime].y;
        const double *tw = c.twd_inv + ((size_t)prime << c.log_n);
        const double2 *sc = MODE == CONV_UP ? c.inv_scale_up + 2 * ((size_t)level * c.L + lo + a)
                            : RESC          ? c.inv_scale_rs + 2 * ((size_t)(level - 1) * (c.K + 1) + (drop ? 0 : 1 + a))
                                            : c.inv_scale_dn + 2 * a;
        const double2 c0 = sc[0], c1 = sc[1];
        const double *g = src + (drop ? -((ptrdiff_t)1 << c.log_n) : (ptrdiff_t)a << c.log_n) + col;
        double *ex = drop ? dropped : bufs + a * LIMB, *tws = stw + grp * R;
#pragma unroll
        for (uint32_t k = 0; k < E; k++) x[k] = g[(size_t)(E * r + k) * 256];
        for (uint32_t e = tid; e < R; e += TG) tws[e] = tw[e];
        group_sync(1 + grp, TG);
        if constexpr (S::B > 0) {
#pragma unroll
            for (uint32_t i = 0; i < (E >> S::B); i++) inv_col_open<S::B, true>(x, i << S::B, tws, (1u << S::A) + r * (E >> S::B) + i, q, qinv);
#pragma unroll
            for (uint32_t k = 0; k < E; k++) ex[S::at(E * r + k, cc)] = x[k];
            group_sync(1 + grp, TG);
#pragma unroll
            for (uint32_t k = 0; k < E; k++) x[k] = ex[S::at(r + RS * k, cc)];
        }
        inv_col_last<S::A, S::B, true>(x, tws, q, qinv, c0, c1);
        group_sync(1 + grp, TG);                              // the exchange and the twiddles have been read
#pragma unroll
        for (uint32_t k = 0; k < E; k++) ex[(r + RS * k) * COLS + cc] = reduce_d(x[k], q, qinv);
    }
    __syncthreads();
    constexpr uint32_t FULL = 1 + GROUPS, EMPTY = FULL + S::BUFFERS, PASS = S::CONV + TG;        // barriers of a buffer and who takes part
    if (threadIdx.x < S::CONV) {
        // ---- conversions
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(CONV_REGS));
        double y[CPT][NS];
#pragma unroll
        for (uint32_t p = 0; p < CPT; p++)
#pragma unroll
            for (uint32_t a = 0; a < NS; a++) y[p][a] = a < nd ? bufs[a * LIMB + threadIdx.x + p * S::CONV] : 0.0;
        if (RESC) {
            // the dropped limb's share of the ModDown is finished here, r = centre((u_l - conv_l) P^-1 mod q_l); every target's
            // conversion gets P r on top, so that (u_i - NTT(conv_i + P r)) (P q_l)^-1 is the rescaled ModDown: one transform of
            // each remaining limb, where ModDown and rescale after each other take two
            const double2 md = c.modd[targets], pinv = c.dn_p_inv_d[targets];
            double v[CPT];
            strip_dot<true, false, NS, CPT>(y, s_w + (x1 - x0) * NS, nd, md.x, md.y, v);
#pragma unroll
            for (uint32_t p = 0; p < CPT; p++) {
                double *d = dropped + threadIdx.x + p * S::CONV;
                *d = reduce_d(mulmod_d<0>(__dsub_rn(*d, v[p]), pinv, md.x), md.x, md.y);
            }
        }
        group_sync(1, S::CONV);                               // the sources have been read
        auto convert = [&](auto full) {
#pragma unroll 1
            for (uint32_t xt = x0; xt < x1; xt++) {
                const uint32_t b = (xt - x0) % S::BUFFERS;
                const double2 md = s_m[xt - x0];
                double v[CPT];
                if (RESC) {
                    const double pq = c.dn_p_mod_d[xt];
#pragma unroll
                    for (uint32_t p = 0; p < CPT; p++) v[p] = mulmod_dd(dropped[threadIdx.x + p * S::CONV], pq, md.x, md.y);
                }
                strip_dot<!RESC, decltype(full)::value, NS, CPT>(y, s_w + (xt - x0) * NS, nd, md.x, md.y, v);
                if (xt - x0 >= S::BUFFERS) group_sync(EMPTY + b, PASS);
#pragma unroll
                for (uint32_t p = 0; p < CPT; p++) bufs[b * LIMB + threadIdx.x + p * S::CONV] = v[p];
                group_arrive(FULL + b, PASS);
            }
        };
        if (nd == NS) convert(std::true_type());
        else convert(std::false_type());
    } else {
        // ---- forward column passes (see ntt_fwd_cols), every other target
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(NTT_REGS));
        const uint32_t first = x0 + grp - S::CONV / TG;
        auto fetch = [&](uint32_t xt, double *to) {
            const double *tw = c.twd_fwd + ((size_t)target_prime(xt) << c.log_n);
            const uint32_t sa = (uint32_t)__cvta_generic_to_shared(to);
            for (uint32_t e = tid; e < R; e += TG) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa + 8 * e), "l"(tw + e) : "memory");
        };
        double *tws = stw + 2 * (grp - S::CONV / TG) * R;     // two buffers of this group
        if (first < x1) fetch(first, tws);
        uint32_t turn = 0;
#pragma unroll 1
        for (uint32_t xt = first; xt < x1; xt += GROUPS - S::CONV / TG, turn ^= 1) {
            const uint32_t b = (xt - x0) % S::BUFFERS;
            const double q = s_m[xt - x0].x, qinv = s_m[xt - x0].y;
            const double *twp = tws + turn * R;
            double *ex = bufs + b * LIMB;
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            group_sync(FULL + b, PASS);                       // (also: the group's twiddles have arrived, the last ones have been read)
            if (xt + GROUPS - S::CONV / TG < x1) fetch(xt + GROUPS - S::CONV / TG, tws + (turn ^ 1) * R);
#pragma unroll
            for (uint32_t k = 0; k < E; k++) x[k] = ex[(r + RS * k) * COLS + cc];
            fwd_col_group<LOGR, 0, S::A, true>(x, 0, twp, 1, q, qinv);
            if constexpr (S::B > 0) {
                group_sync(1 + grp, TG);
#pragma unroll
                for (uint32_t k = 0; k < E; k++) ex[S::at(r + RS * k, cc)] = x[k];
                group_sync(1 + grp, TG);
#pragma unroll
                for (uint32_t k = 0; k < E; k++) x[k] = ex[S::at(E * r + k, cc)];
            }
            if (xt + S::BUFFERS < x1) group_arrive(EMPTY + b, PASS);
            if constexpr (S::B > 0)
#pragma unroll
                for (uint32_t i = 0; i < (E >> S::B); i++)
                    fwd_col_group<LOGR, S::A, S::B, true>(x, i << S::B, twp, (1u << S::A) + r * (E >> S::B) + i, q, qinv);
            double *g = dst + ((size_t)target_limb(xt) << c.log_n) + col;
#pragma unroll
            for (uint32_t k = 0; k < E; k++) g[(size_t)(E * r + k) * 256] = x[k];
        }
    }
}

template <uint32_t LOGR>
constexpr size_t strip_smem(int mode, uint32_t ns) {
    using S = StripShape<LOGR>;
    return ((size_t)((ns > S::BUFFERS ? ns : S::BUFFERS) + (mode == CONV_DOWN_RS)) * S::LIMB + S::GROUPS * S::R + (STRIP_CHUNK + 1) * ns + 2 * STRIP_CHUNK) * sizeof(double);
}
using StripKernel = decltype(&conv_cols<8, 0, 1>);
// by mode and log2 of the sources' register arrays
template <uint32_t LOGR>
constexpr StripKernel strip_kernels[3][4] = {
    {conv_cols<LOGR, CONV_UP, 1>, conv_cols<LOGR, CONV_UP, 2>, conv_cols<LOGR, CONV_UP, 4>, conv_cols<LOGR, CONV_UP, 8>},
    {conv_cols<LOGR, CONV_DOWN, 1>, conv_cols<LOGR, CONV_DOWN, 2>, conv_cols<LOGR, CONV_DOWN, 4>, conv_cols<LOGR, CONV_DOWN, 8>},
    {conv_cols<LOGR, CONV_DOWN_RS, 1>, conv_cols<LOGR, CONV_DOWN_RS, 2>, conv_cols<LOGR, CONV_DOWN_RS, 4>, conv_cols<LOGR, CONV_DOWN_RS, 8>}};

// f(std::integral_constant<uint32_t, log2 of the rows>)
template <class F>
auto for_ring(const ckks_ctx *c, F f) {
    switch (c->log_n) {
        case 16: return f(std::integral_constant<uint32_t, 8>());
        case 15: return f(std::integral_constant<uint32_t, 7>());
        case 14: return f(std::integral_constant<uint32_t, 6>());
        case 13: return f(std::integral_constant<uint32_t, 5>());
        default: return f(std::integral_constant<uint32_t, 4>());
    }
}
uint32_t strip_sources(const ckks_ctx *c, int mode, uint32_t level) { return mode == CONV_UP ? std::min(c->alpha, level) : c->K; }
// (of a ModUp the most that a digit has: the last one's)
uint32_t strip_targets(const ckks_ctx *c, int mode, uint32_t level) {
    return mode == CONV_UP ? (level + c->alpha - 1) / c->alpha * c->alpha - c->alpha + c->K : mode == CONV_DOWN ? level : level - 1;
}

// The cheapest grid for `strips` strips, one CTA per SM at a time.  A CTA's time is its targets in groups of four and half as much per
// round of sources, which every chunk of the same strip repeats.  As many strips as fill whole waves can go by one CTA each; cut into
// chunks, the others share out the last wave.  (N = 2^16, level 24, in a burst and back to back under the power limit: eight hoisted
// rotations, 512 strips, 3.46 waves, by the separate kernels 576 and 566 us, by a CTA per strip 588 and 559, so 575 and 545; fourteen, 6.05
// waves, 910 and 924, 931 and 918, 911 and 878.)
struct StripPlan { StripGrid grid; dim3 ctas; uint32_t cost, full; };        // full: the cost if all SMs were busy throughout, times their number
StripPlan strip_plan(const ckks_ctx *c, int mode, uint32_t level, uint32_t strips) {
    const uint32_t targets = strip_targets(c, mode, level), sms = (uint32_t)c->sms, rounds = (strip_sources(c, mode, level) + (mode == CONV_DOWN_RS) + 3) / 4;
    auto cta = [&](uint32_t n) { return (std::min(n, targets) + 3) / 4 * 2 + rounds; };
    StripPlan p{};
    p.full = strips * cta(targets);
    p.cost = ~0u;
    const uint32_t waves = targets <= STRIP_CHUNK ? strips / sms : 0;
    for (uint32_t w = 0;; w = waves) {
        const uint32_t whole = w * sms, split = strips - whole;
        for (uint32_t ch = 4; ch <= STRIP_CHUNK && ch < targets + 4; ch += 4) {
            const uint32_t n = (targets + ch - 1) / ch, cost = w * cta(targets) + (split * n + sms - 1) / sms * cta(ch);
            if (cost <= p.cost) p = {{whole, split, ch}, whole ? dim3(whole + split * n) : dim3(split, n), cost, p.full};
        }
        if (w == waves) break;
    }
    return p;
}

}  // namespace

bool conv_strip_prepare(const ckks_ctx *c) {
    if (c->log_n < 12) return false;
    return for_ring(c, [](auto logr) {
        bool ok = true;
        for (int mode = 0; mode < 3; mode++)
            for (uint32_t i = 0; i < 4 && ok; i++) {
                StripKernel k = strip_kernels<decltype(logr)::value>[mode][i];
                cudaFuncAttributes fa;
                ok = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)strip_smem<decltype(logr)::value>(mode, 1u << i)) == cudaSuccess &&
                     cudaFuncGetAttributes(&fa, k) == cudaSuccess && (fa.numRegs + 7) / 8 * 8 * 2 == (int)(CONV_REGS + NTT_REGS);
            }
        if (!ok) cudaGetLastError();
        return ok;
    });
}

// Whether a conversion of `items` items runs here.  It can from N = 2^12 on with at most eight sources, whose coefficients fit the
// registers.  At N = 2^16 a strip takes an SM as long as the separate kernels do, and what it saves is traffic: batches of four strips
// per SM and more, and of three with eight targets and more where the last wave is nearly full, take the same time in a burst (0.98 to
// 1.02 of it) and under the power limit 0.91 to 1.01 of it, most of them 0.96 and less (64 hoisted rotations at level 24 3952 -> 3750 us,
// sixteen products 2056 -> 1950).  Seven hoisted rotations at level 5, 3.03 waves, would go from 205 to 216 us and from 152 to 164, eight
// from 171 to 175.  The few strips of one ciphertext (96 for ModUp, 64 for ModDown) leave a third of the GPU idle or repeat their sources'
// transforms (a rotation 149 -> 156).
// The separate kernels of smaller rings are bound by latency, and fewer launches win from the first ciphertext on (N = 2^15: rotation
// 49.5 -> 43.9, product and rescale 71.7 -> 66.3; N = 2^14: ModUp 29.3 -> 28.4), but for ModDowns of a few strips (29.3 -> 30.7) and, at
// N = 2^13, for ModUps inside longer calls (a 64 x 64 projection 172.4 -> 175.3; a rotation of its own 30.7 -> 29.2).
bool conv_strip(const ckks_ctx *c, int mode, uint32_t level, uint32_t items, bool alone) {
    if (!c->strips || c->conv_kernel == CKKS_CONV_TENSOR || items > 65535 || strip_sources(c, mode, level) > STRIP_NS) return false;
    const uint32_t strips = (c->N >> 11) * items, sms = (uint32_t)c->sms;
    if (strips >= 4 * sms || (c->log_n < 16 && (mode == CONV_UP ? alone || c->log_n > 13 : strips >= 32))) return true;
    if (strips < 3 * sms || strip_targets(c, mode, level) < 8) return false;
    const StripPlan p = strip_plan(c, mode, level, strips);
    return 10 * p.full >= 9 * sms * p.cost;
}

void launch_conv_strip(const ckks_ctx *c, int mode, const u64 *src, u64 *dst, uint32_t level, uint32_t items, cudaStream_t s) {
    const uint32_t ns = strip_sources(c, mode, level), i = ns <= 1 ? 0 : ns <= 2 ? 1 : ns <= 4 ? 2 : 3;
    for_ring(c, [&](auto logr) {
        constexpr uint32_t LOGR = decltype(logr)::value;
        using S = StripShape<LOGR>;
        const StripPlan p = strip_plan(c, mode, level, 256 / S::COLS * items);
        launch(strip_kernels<LOGR>[mode][i], p.ctas, S::THREADS, strip_smem<LOGR>(mode, 1u << i), s, c->dev, reinterpret_cast<const double *>(src), reinterpret_cast<double *>(dst),
               level, strip_targets(c, mode, level), p.grid);
    });
}
