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
#include "butterfly.cuh"

namespace {

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

// The end of a CTA whose limb is left out.  With limbs on the integer path that may be every CTA of a grid (a digit's own limb and
// seven integer ones), and a grid that has not waited for the one before it lets the one after it pass that too.
__device__ __forceinline__ void leave_out(uint32_t fp_share) {
    if (fp_share < 8) grid_dep_sync();
}

// ---- column passes -------------------------------------------------------------------------------------------------
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

// ---- row passes (see ROW_PAD) --------------------------------------------------------------------------------------------
// forward, EP 0: in place; 1: the tail of a ModDown or rescale, (u - NTT(conv)) c + sigma_g(add), written to its final
// place; 2: into a tiled buffer; 3: as 1 with u formed here from BETA digits and the key.  EP 3 is bound by HBM (the key words and the
// results); one pair of words per step at 64 registers: two pairs at 96 registers and 20 warps per SM took 1750 us for 64
// rotations, four pairs at 128 registers 1910, against 1550.
template <int EP, bool WIDE, uint32_t BETA = 1>
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
        const u64 *add = (ep.add_comps >> comp & 1) ? ep.add.at(ep.own ? bz : mem) + (((size_t)comp * ep.level + i) << c.log_n) : nullptr;
        const u64 *acc = ep.accumulate ? ep.acc.at(bz) + (((size_t)comp * ep.level + i) << c.log_n) + p0 : nullptr;
        const uint32_t bstep = ep.tl.R ? ep.tl.R * 64 : 64;    // words from one 64-word block of the destination to the next
        u64 *dst = ep.tl.R ? const_cast<u64 *>(ep.out.base) + tiled_index(ep.tl.R, c.N, ep.tl.row0 + rot * ep.rot_rows + (ep.group ? mem : bz) * ep.tl.row_stride + comp, i, row * 256) + 2 * t
                           : const_cast<u64 *>(ep.group ? ep.out.base + rot * ep.rot_stride + mem * ep.out.stride : ep.out.at(bz)) +
                                 (((size_t)comp * ep.level + i) << c.log_n) + p0;
        if (EP == 3) {
            // u = sum_j digit_j key_j
            const size_t ks = (size_t)2 * c.T << c.log_n;
            const uint32_t de = ep.group ? mem : 0, own = i / c.alpha;
            const u64 *kp = ep.mevk[rot] + (((size_t)comp * c.T + i) << c.log_n) + p0;
            const u64 *eb = ep.ext + (((size_t)de * BETA * ep.nt + i) << c.log_n), *od = ep.d.at(de) + ((size_t)i << c.log_n);
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
#pragma unroll
                for (uint32_t j = 0; j < BETA; j++) {
                    s0 = __dadd_rn(s0, mulmod_dd(u64_to_d(ev[j].x), u64_to_d(odd ? kv[j].y : kv[j].x), q, qinv));
                    s1 = __dadd_rn(s1, mulmod_dd(u64_to_d(ev[j].y), u64_to_d(odd ? kv[j].x : kv[j].y), q, qinv));
                }
                // |u - v| < (0.75 BETA + 0.5) q <= 2.75 q, below 2^52: the product may round its quotient to even
                if (BETA > 3) { s0 = reduce_d(s0, q, qinv); s1 = reduce_d(s1, q, qinv); }
                const double2 v = *reinterpret_cast<const double2 *>(sp + 36 * k);
                double r0 = mulmod_d<1>(__dsub_rn(odd ? s1 : s0, reduce_d(v.x, q, qinv)), pinv, q);
                double r1 = mulmod_d<1>(__dsub_rn(odd ? s0 : s1, reduce_d(v.y, q, qinv)), pinv, q);
                if (add) {
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
        const uint32_t e = blockIdx.y / map.period, comp = e & 1, bz = e >> 1, xl = src.nt - map.period + blockIdx.y % map.period, p0 = row * 256 + 2 * t;
        const uint32_t rot = src.group ? bz / src.group : bz, mem = src.group ? bz % src.group : bz;
        const uint32_t gal = (uint32_t)src.mgalois[rot], de = src.group ? mem : 0;
        const size_t ks = (size_t)2 * c.T << c.log_n;
        const u64 *kp = src.mevk[rot] + (((size_t)comp * c.T + prime) << c.log_n) + p0;
        const u64 *eb = src.ext + (((size_t)de * BETA * src.nt + xl) << c.log_n);
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) {
            const uint32_t sr = galois_src(p0 + 32 * k, gal, c.log_n), so = sr & ~1u;
            const bool odd = sr & 1;
            ulonglong2 kv[BETA], ev[BETA];
#pragma unroll
            for (uint32_t j = 0; j < BETA; j++) {
                kv[j] = ld_pair<true>(kp + j * ks + 32 * k);
                ev[j] = ld_pair<true>(eb + (((size_t)j * src.nt) << c.log_n) + so);
            }
            __syncwarp();
            double s0 = 0.0, s1 = 0.0;
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

// ---- row passes of few limbs: a row by a warp -----------------------------------------------------------------------------
// forward, EP 0 and 1 as in ntt_fwd_rows; the other operands are on their way while the row is transformed
template <int EP, bool WIDE>
__global__ void __launch_bounds__(32 * ROW_CTA, 6) ntt_fwd_wrows(DevTables c, u64 *base, LimbMap map, uint32_t fp_share, const __grid_constant__ NttEpilogue ep) {
    __shared__ __align__(16) double sm[ROW_CTA][WROW_PAD];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) >= fp_share) return leave_out(fp_share);
    const double q = c.modd[prime].x, qinv = c.modd[prime].y;
    const double *tw = c.twd_fwd + ((size_t)prime << c.log_n);
    const uint32_t t = threadIdx.x & 31, rl = threadIdx.x >> 5, row = blockIdx.x * ROW_CTA + rl, R = c.N >> 8;
    u64 *g = base + (limb_index(map, blockIdx.y) << c.log_n) + (size_t)row * 256;
    double *s = sm[rl], v[8];
    grid_dep_sync();
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) v[k] = reinterpret_cast<const double *>(g)[t + 32 * k];
    const double *sp = s + wrow_at(2 * t);                // word 2 t + 64 k is 72 k further
    if (EP == 0) {
        __syncwarp();
        wrow_forward(v, s, t, tw, R + row, q, qinv);
        __syncwarp();
#pragma unroll
        for (uint32_t k = 0; k < 4; k++) {
            const double2 w = *reinterpret_cast<const double2 *>(sp + 72 * k);
            st_pair<WIDE>(g + 2 * t + 64 * k, make_ulonglong2(canonical_d(w.x, q), canonical_d(w.y, q)));
        }
        return;
    }
    const uint32_t y = blockIdx.y + ep.y0, i = y % ep.level, comp = (y / ep.level) % ep.ncomp, bz = y / (ep.ncomp * ep.level);
    const double2 pinv = ep.pinv[i];
    const uint32_t p0 = row * 256 + 2 * t;
    // grouped: entry bz is key bz / group applied to member bz % group (own: to the entry itself)
    const uint32_t rot = ep.group ? bz / ep.group : bz, mem = ep.group ? bz % ep.group : bz;
    const uint32_t gal = (uint32_t)(ep.multi ? ep.mgalois[rot] : ep.galois);
    const u64 *add = (ep.add_comps >> comp & 1) ? ep.add.at(ep.own ? bz : mem) + (((size_t)comp * ep.level + i) << c.log_n) : nullptr;
    const u64 *acc = ep.accumulate ? ep.acc.at(bz) + (((size_t)comp * ep.level + i) << c.log_n) + p0 : nullptr;
    const uint32_t bstep = ep.tl.R ? ep.tl.R * 64 : 64;        // words from one 64-word block of the destination to the next
    u64 *dst = ep.tl.R ? const_cast<u64 *>(ep.out.base) + tiled_index(ep.tl.R, c.N, ep.tl.row0 + rot * ep.rot_rows + (ep.group ? mem : bz) * ep.tl.row_stride + comp, i, row * 256) + 2 * t
                       : const_cast<u64 *>(ep.group ? ep.out.base + rot * ep.rot_stride + mem * ep.out.stride : ep.out.at(bz)) + (((size_t)comp * ep.level + i) << c.log_n) + p0;
    const u64 *up = ep.u.at(bz) + (((size_t)comp * ep.nt + i) << c.log_n) + p0;
    ulonglong2 ua[4], aa[4];
    uint32_t sr[4];
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) {
        ua[k] = ld_pair<WIDE>(up + 64 * k);
        if (add) {      // the permutation maps the pair onto a pair, possibly swapped
            sr[k] = galois_src(p0 + 64 * k, gal, c.log_n);
            aa[k] = ld_pair<WIDE>(add + (sr[k] & ~1u));
        }
    }
    __syncwarp();
    wrow_forward(v, s, t, tw, R + row, q, qinv);
    __syncwarp();
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) {
        const double2 w = *reinterpret_cast<const double2 *>(sp + 72 * k);
        // |u - v| < 1.5 q, times P^-1 -> |.| < 0.9 q, plus up to two residues, reduced once
        double r0 = mulmod_d<0>(__dsub_rn(u64_to_d(ua[k].x), w.x), pinv, q);
        double r1 = mulmod_d<0>(__dsub_rn(u64_to_d(ua[k].y), w.y), pinv, q);
        if (add) {
            const bool odd = sr[k] & 1;
            r0 = __dadd_rn(r0, u64_to_d(odd ? aa[k].y : aa[k].x));
            r1 = __dadd_rn(r1, u64_to_d(odd ? aa[k].x : aa[k].y));
        }
        if (ep.accumulate) {
            const ulonglong2 o = ld_pair<WIDE>(acc + 64 * k);
            r0 = __dadd_rn(r0, u64_to_d(o.x));
            r1 = __dadd_rn(r1, u64_to_d(o.y));
        }
        st_pair<WIDE>(dst + k * bstep, make_ulonglong2(canonical_d(reduce_d(r0, q, qinv), q), canonical_d(reduce_d(r1, q, qinv), q)));
    }
}

// inverse; src as in ntt_inv_rows
template <bool WIDE>
__global__ void __launch_bounds__(32 * ROW_CTA, 8) ntt_inv_wrows(DevTables c, u64 *base, LimbMap map, uint32_t fp_share, const __grid_constant__ NttSource src) {
    __shared__ __align__(16) double sm[ROW_CTA][WROW_PAD];
    const int prime = limb_prime(map, blockIdx.y);
    if (prime < 0 || (blockIdx.y & 7) >= fp_share) return leave_out(fp_share);
    const double q = c.modd[prime].x, qinv = c.modd[prime].y;
    const double *tw = c.twd_inv + ((size_t)prime << c.log_n);
    const uint32_t t = threadIdx.x & 31, rl = threadIdx.x >> 5, row = blockIdx.x * ROW_CTA + rl, R = c.N >> 8;
    u64 *g = base + (limb_index(map, blockIdx.y) << c.log_n) + (size_t)row * 256;
    const u64 *gs = src.lpitch ? src.ptr.at(blockIdx.y / map.period) + (((size_t)(blockIdx.y % map.period) * src.lpitch) << c.log_n) + (size_t)row * 256 : g;
    double *s = sm[rl], v[8];
    grid_dep_sync();
    ulonglong2 w[4];
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) w[k] = ld_pair<WIDE>(gs + 2 * t + 64 * k);
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) *reinterpret_cast<double2 *>(s + wrow_at(2 * t) + 72 * k) = make_double2(u64_to_d(w[k].x), u64_to_d(w[k].y));
    __syncwarp();
    wrow_inverse(v, s, t, tw, R + row, q, qinv);
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) reinterpret_cast<double *>(g)[t + 32 * k] = v[k];
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

static void run_ntt(const ckks_ctx *c, u64 *base, uint32_t nlimbs_total, const LimbMap &map, bool inverse, cudaStream_t s, const NttEpilogue *ep,
                    const NttPrologue *pro, const NttSource *src, const double2 *inv_scale, NttPart part) {
    const uint32_t R = c->N >> 8;
    // the integer path (an option, N = 2^16) has no fused forms: those take all limbs on the FP64 pipe
    const uint32_t share = (ep || pro || inv_scale || part != NTT_BOTH || (src && src->ptr.n) || c->log_n != 16) ? 8 : c->ntt_fp_share;
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
        // A row by a warp where the launch is bound by latency: up to six CTAs of four rows per SM.  (Rotation at N = 2^14, 192 CTAs,
        // 28.8 -> 27.3 us; at N = 2^15, 768 CTAs, 44.1 -> 43.4; the 64 x 64 projection at N = 2^13 175.4 -> 168.7; from there on the
        // additional exchanges cost more: rotation at N = 2^16, level 9, 1152 CTAs, 72.0 -> 74.0.)
        const bool few = (uint64_t)grid.x * ny <= 6 * (uint64_t)c->sms;
        if (share > 0 && !inverse) {
            if (part & NTT_COLS) cols();
            if (!(part & NTT_ROWS)) continue;
            bool wide = aligned16(ep ? (const void *)nullptr : (const void *)b);
            if (ep) wide = aligned16(ep->u) && aligned16(ep->add) && aligned16(ep->acc) && aligned16(ep->out) && (ep->rot_stride & 1) == 0;
            NttEpilogue e = ep ? *ep : NttEpilogue{};
            e.y0 = y0;
            const int mode = ep ? ep->mode : 0;
            static constexpr decltype(&ntt_fwd_rows<0, true>) inner[IP_FUSED_BETA] = {ntt_fwd_rows<3, true, 1>, ntt_fwd_rows<3, true, 2>, ntt_fwd_rows<3, true, 3>,
                                                                                      ntt_fwd_rows<3, true, 4>};
            auto *k = mode == 3 ? inner[e.beta - 1]
                    : mode == 1 ? (wide ? ntt_fwd_rows<1, true> : ntt_fwd_rows<1, false>)
                    : mode == 2 ? (wide ? ntt_fwd_rows<2, true> : ntt_fwd_rows<2, false>)
                                : (wide ? ntt_fwd_rows<0, true> : ntt_fwd_rows<0, false>);
            if (mode < 2 && few)
                launch(mode ? (wide ? ntt_fwd_wrows<1, true> : ntt_fwd_wrows<1, false>) : (wide ? ntt_fwd_wrows<0, true> : ntt_fwd_wrows<0, false>), grid, 32 * ROW_CTA, 0, s, c->dev, b, map,
                       share, e);
            else launch(k, grid, 16 * ROW_CTA, 0, s, c->dev, b, map, share, e);
        } else if (share > 0) {
            const NttSource none{};
            const bool wide = src ? aligned16(src->ptr) : aligned16(b);
            static constexpr decltype(&ntt_inv_rows<true, 1, NttEpilogue>) inner[IP_FUSED_BETA] = {
                ntt_inv_rows<true, 1, NttEpilogue>, ntt_inv_rows<true, 2, NttEpilogue>, ntt_inv_rows<true, 3, NttEpilogue>, ntt_inv_rows<true, 4, NttEpilogue>};
            if (!(part & NTT_ROWS)) {
            } else if (ep) {
                launch(inner[ep->beta - 1], grid, 16 * ROW_CTA, 0, s, c->dev, b, map, share, *ep);
            } else if (few) {
                launch(wide ? ntt_inv_wrows<true> : ntt_inv_wrows<false>, grid, 32 * ROW_CTA, 0, s, c->dev, b, map, share, src ? sr : none);
            } else {
                launch(wide ? ntt_inv_rows<true> : ntt_inv_rows<false>, grid, 16 * ROW_CTA, 0, s, c->dev, b, map, share, src ? sr : none);
            }
            if (part & NTT_COLS) cols();
        }
        if (share < 8) launch_ntt_int(c, b, ny, map, inverse, sr, s);
    }
}

void launch_ntt(const ckks_ctx *c, u64 *base, uint32_t nlimbs_total, const LimbMap &map, bool inverse, cudaStream_t s, const NttEpilogue *ep,
                const NttPrologue *pro, const NttSource *src, const double2 *inv_scale, bool alone) {
    if (alone && !ep && (!pro || pro->doubles) && launch_ntt_small(c, base, nlimbs_total, map, inverse, s, src, inv_scale, pro != nullptr)) return;
    run_ntt(c, base, nlimbs_total, map, inverse, s, ep, pro, src, inv_scale, NTT_BOTH);
}
void launch_ntt_part(const ckks_ctx *c, NttPart part, u64 *base, uint32_t nlimbs_total, const LimbMap &map, bool inverse, cudaStream_t s, const NttEpilogue *ep,
                     const NttPrologue *pro, const NttSource *src, const double2 *inv_scale) {
    run_ntt(c, base, nlimbs_total, map, inverse, s, ep, pro, src, inv_scale, part);
}

// grid: three CTAs per SM, all resident at once.  Returns the butterflies one launch performs.
uint64_t launch_butterfly_probe(const ckks_ctx *c, uint32_t iters, u64 *sink, cudaStream_t s) {
    const uint32_t ctas = (uint32_t)c->sms * 3;
    launch(butterfly_probe_kernel, ctas, F_THREADS, 0, s, c->dev, iters, sink);
    return (uint64_t)ctas * F_THREADS * iters * 32;
}
