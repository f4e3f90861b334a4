// Hybrid key switching (dnum digits, K special primes) and rescale.
//
// KeySwitch(d, evk):  d (evaluation domain, `level` limbs)
//   1. to the coefficient domain (inverse NTT)
//   2. ModUp: every active digit j is extended from its own limbs to all active
//      q-limbs and all special limbs by a centred fast basis conversion
//         y_a = centre([d_a * qhat_a^-1]_{q_a}),  ext_j[t] = sum_a y_a (qhat_a mod t)  mod t
//   3. NTT of the converted limbs (own limbs keep their evaluation values)
//   4. inner product with the key: u_c[t] = sum_j ext_j[t] * evk_{j,c}[t]
//   5. ModDown: inverse NTT of the special limbs, centred conversion P -> q_i,
//      NTT, out_i = (u_i - conv_i) * P^-1 mod q_i.
// Rescale drops the last limb the same way with a single source limb.
#include "common.cuh"

namespace {

constexpr uint32_t THREADS = 256, IP_THREADS = 128;
// of the conversions: 128 threads even out what an SM gets (ModDown of products 184 -> 172 us in the degree-63 polynomial, the
// hoisted rotations' 615 -> 601; 64 threads fetch their constants too often, 618)
constexpr uint32_t CONV_THREADS = 128;

// ---- basis conversions (see CONV_SIGMA), any number of sources, reduced once per eight: the quotient of the high part, rounded to nearest,
// leaves |r| <= 1.1 t, and with the low parts and a reduced carry of the previous eight sources the sum stays below 2^53.
// A thread takes CPT adjacent coefficients, so that a pair of constants from shared memory serves 2 CPT pairs.
// out enters holding a further summand below t (FIRST: nothing)
template <bool FIRST, uint32_t NS, uint32_t CPT>
__device__ __forceinline__ void conv_dot(const double (&y)[CPT][NS], const double *w, double t, double tinv, double (&out)[CPT]) {
    double H[CPT], lo[CPT];
#pragma unroll
    for (uint32_t p = 0; p < CPT; p++) { H[p] = CONV_SIGMA; lo[p] = FIRST ? 0.0 : out[p]; }
#pragma unroll
    for (uint32_t a = 0; a < NS; a++) {
        const double wa = w[a];
#pragma unroll
        for (uint32_t p = 0; p < CPT; p++) {
            const double Hn = __fma_rn(y[p][a], wa, H[p]);
            const double l = __fma_rn(y[p][a], wa, -__dsub_rn(Hn, H[p]));
            lo[p] = FIRST && a == 0 ? l : __dadd_rn(lo[p], l);
            H[p] = Hn;
            if ((a & 7) == 7 || a + 1 == NS) {
                const double hs = __dsub_rn(H[p], CONV_SIGMA);
                const double k = __dsub_rn(__fma_rn(hs, tinv, MAGIC0), MAGIC0);
                lo[p] = reduce_d(__dadd_rn(lo[p], __fma_rn(-k, t, hs)), t, tinv);
                H[p] = CONV_SIGMA;
            }
        }
    }
#pragma unroll
    for (uint32_t p = 0; p < CPT; p++) out[p] = lo[p];
}

// centred source residues of CPT adjacent coefficients
template <uint32_t CPT>
__device__ __forceinline__ void conv_load(const u64 *p, u64 (&v)[CPT]) {
    if (CPT == 2) {
        const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(p);
        v[0] = w.x; v[CPT - 1] = w.y;
    } else {
        v[0] = *p;
    }
}
// The results stay signed doubles, at most t / 2, for the transform that follows: three instructions less here and one there
// (64 hoisted rotations: conversion 648 -> 602 us; one rotation 155.6 -> 153.1).
template <uint32_t CPT>
__device__ __forceinline__ void conv_store(u64 *p, const double (&v)[CPT]) {
    if (CPT == 2) *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[CPT - 1]);
    else *reinterpret_cast<double *>(p) = v[0];
}

// coefficients per thread: two while their sources fit the registers and the buffers take 16-byte accesses
inline uint32_t conv_cpt(uint32_t ns, const void *a, const void *b) { return ns <= 8 && (((uintptr_t)a | (uintptr_t)b) & 15) == 0 ? 2 : 1; }

// targets per CTA (grid y) for `items` conversions of `targets` targets over gx CTAs: all of them, unless that leaves fewer than
// 512 threads (four CTAs) per SM.  Every chunk loads and centres its sources again, which costs more than a machine that is
// only partly filled (one ciphertext at N = 2^16, level 24: ModUp with 24, 8, 5 targets per CTA 21.7, 22.7, 26.0 us, taken with
// CTAs of 256 threads, two per SM).
constexpr uint32_t CONV_CHUNK_MAX = 32;
inline uint32_t conv_chunk(const ckks_ctx *c, uint32_t gx, uint32_t items, uint32_t targets) {
    const uint32_t want = (uint32_t)c->sms * (512 / CONV_THREADS);
    uint32_t chunks = (want + gx * items - 1) / (gx * items);
    chunks = std::max(1u, std::min(chunks, (targets + 1) / 2));
    return std::min(CONV_CHUNK_MAX, (targets + chunks - 1) / chunks);
}

// ext[j][x][k] for the limbs x of q_0..q_{level-1}, p_0..p_{K-1} outside digit j, from dcoef (coefficient domain).  A thread
// owns CPT coefficients of one digit: it forms the centred y_a of the digit's limbs once and walks a chunk of CHUNK target
// limbs (blockIdx.y), so the source limbs are read once per chunk.
// dcoef already holds [d_a qhat_a^-1] (the inverse transform multiplied it in), so only the centring is left.
template <uint32_t ALPHA, uint32_t CPT>
__global__ void __launch_bounds__(CONV_THREADS) modup_kernel(DevTables c, const u64 *dcoef, u64 *ext, uint32_t level, uint32_t CHUNK) {
    // the CTA's conversion constants (qhat_a mod t; t and 1/t), fetched once
    __shared__ __align__(16) double s_w[CONV_CHUNK_MAX][ALPHA];
    __shared__ double2 s_m[CONV_CHUNK_MAX];
    const uint32_t k = (blockIdx.x * CONV_THREADS + threadIdx.x) * CPT;
    const uint32_t beta = (level + c.alpha - 1) / c.alpha, j = blockIdx.z % beta, bz = blockIdx.z / beta;
    const uint32_t nt = level + c.K, lo = j * c.alpha, hi = min(lo + c.alpha, level), nd = hi - lo;
    const uint32_t x0 = blockIdx.y * CHUNK, x1 = min(x0 + CHUNK, nt - nd);       // targets, counted without the digit's own limbs
    if (x0 >= x1) return;
    const size_t cb = (size_t)level * c.dnum + j;
    for (uint32_t e = threadIdx.x; e < (x1 - x0) * ALPHA; e += CONV_THREADS) {
        const uint32_t xi = e / ALPHA, a = e % ALPHA, xt = x0 + xi, x = xt < lo ? xt : xt + nd, t = x < level ? x : c.L + (x - level);
        s_w[xi][a] = a < nd ? c.up_hat_mod_d[(cb * c.T + t) * c.alpha + a] : 0.0;
        if (a == 0) s_m[xi] = c.modd[t];
    }
    dcoef += ((size_t)bz * level + lo) * c.N + k;
    ext += ((size_t)bz * beta + j) * nt * c.N + k;
    double y[CPT][ALPHA];
    grid_dep_sync();
#pragma unroll
    for (uint32_t a = 0; a < ALPHA; a++) {
        u64 v[CPT];
        if (a < nd) conv_load<CPT>(dcoef + (size_t)a * c.N, v);
#pragma unroll
        for (uint32_t p = 0; p < CPT; p++) {
            y[p][a] = 0.0;
            if (a < nd) {
                const u64 qa = c.mod[lo + a];
                y[p][a] = centre_d(v[p], qa);
            }
        }
    }
    __syncthreads();
    for (uint32_t xt = x0; xt < x1; xt++) {
        const double2 md = s_m[xt - x0];
        double r[CPT];
        conv_dot<true>(y, s_w[xt - x0], md.x, md.y, r);
        conv_store<CPT>(ext + (size_t)(xt < lo ? xt : xt + nd) * c.N, r);
    }
}

template <uint32_t ALPHA>
void launch_modup(const ckks_ctx *c, const u64 *dcoef, u64 *ext, uint32_t level, uint32_t nb, cudaStream_t s) {
    const uint32_t nt = level + c->K, beta = (level + c->alpha - 1) / c->alpha;
    const uint32_t cpt = conv_cpt(ALPHA, dcoef, ext), gx = c->N / (CONV_THREADS * cpt), targets = nt - (level - (beta - 1) * c->alpha);   // the last digit has the most targets
    const uint32_t CHUNK = conv_chunk(c, gx, beta * nb, targets);
    const dim3 grid(gx, (targets + CHUNK - 1) / CHUNK, beta * nb);
    constexpr uint32_t WIDE = ALPHA <= 8 ? 2 : 1;
    launch(cpt == WIDE ? modup_kernel<ALPHA, WIDE> : modup_kernel<ALPHA, 1>, grid, CONV_THREADS, 0, s, c->dev, dcoef, ext, level, CHUNK);
}

// u[comp][x][p] = sum_j ext[j][x][pi_g(p)] * evk[j][comp][kt(x)][p]          (any number of digits)
__global__ void __launch_bounds__(THREADS) inner_product_generic_kernel(DevTables c, const u64 *ext, const __grid_constant__ Ptrs dp, uint32_t d0, const u64 *evk, u64 g,
                                                                        u64 *u, uint32_t level, int has_multi, const __grid_constant__ KsMulti multi, int acc_u, int has_add,
                                                                        const __grid_constant__ Ptrs add) {
    const uint32_t p = blockIdx.x * THREADS + threadIdx.x;
    const uint32_t x = blockIdx.z, bz = blockIdx.y;     // batch varies faster than the limb: a key limb is reused from L2
    const uint32_t nt = level + c.K, beta = (level + c.alpha - 1) / c.alpha;
    const uint32_t kt = x < level ? x : c.L + (x - level);
    if (has_multi) { evk = multi.evk[bz]; g = multi.galois[bz]; }     // shared digits, per-entry key and permutation
    else ext += (size_t)bz * beta * nt * c.N;
    const u64 *d = dp.at(d0 + (has_multi ? 0 : bz));
    grid_dep_sync();
    const uint32_t own = x < level ? x / c.alpha : beta;        // the digit that has x among its own limbs
    const uint32_t src = galois_src(p, (uint32_t)g, c.log_n);
    u += (size_t)bz * 2 * nt * c.N;
    // products on the FP64 pipe: each is reduced to |r| <= 0.75 m as it is formed, the few digits are summed exactly
    const double2 md = c.modd[kt];
    double a0 = 0.0, a1 = 0.0;
    if (has_add && x < level) {
        const u64 *z = add.at(bz) + (size_t)x * c.N + p;
        a0 = mulmod_dd(u64_to_d(z[0]), c.dn_p_mod_d[x], md.x, md.y);
        a1 = mulmod_dd(u64_to_d(z[(size_t)level * c.N]), c.dn_p_mod_d[x], md.x, md.y);
    }
    for (uint32_t j = 0; j < beta; j++) {
        const double e = u64_to_d((j == own ? d + (size_t)x * c.N : ext + ((size_t)j * nt + x) * c.N)[src]);
        a0 = __dadd_rn(a0, mulmod_dd(e, u64_to_d(evk[(((size_t)j * 2 + 0) * c.T + kt) * c.N + p]), md.x, md.y));
        a1 = __dadd_rn(a1, mulmod_dd(e, u64_to_d(evk[(((size_t)j * 2 + 1) * c.T + kt) * c.N + p]), md.x, md.y));
        if ((j & 7) == 7) { a0 = reduce_d(a0, md.x, md.y); a1 = reduce_d(a1, md.x, md.y); }
    }
    u64 r0 = canonical_d(reduce_d(a0, md.x, md.y), md.x), r1 = canonical_d(reduce_d(a1, md.x, md.y), md.x);
    if (acc_u) {        // a sum of key-switched terms kept in the extended basis
        const u64 m = c.mod[kt];
        r0 = add_mod(r0, u[((size_t)0 * nt + x) * c.N + p], m);
        r1 = add_mod(r1, u[((size_t)1 * nt + x) * c.N + p], m);
    }
    u[((size_t)0 * nt + x) * c.N + p] = r0;
    u[((size_t)1 * nt + x) * c.N + p] = r1;
}

// The same for BETA <= 8 digits, two adjacent coefficients per thread.  pi_g maps the pair (p, p + 1), p even, onto a
// pair (s, s ^ 1), so digits and key words both move as 16-byte loads.  Without `multi` a thread walks `bch` batch
// entries (blockIdx.y picks the chunk) with the key words of its pair held in registers; with it, an entry is one
// of up to KS_MULTI keys applied to the same digits.
constexpr uint32_t IP_MAX_BETA = 8, IP_TERMS_MAX_BETA = 4;
template <uint32_t BETA, bool ADD>
__global__ void __launch_bounds__(IP_THREADS) inner_product_kernel(DevTables c, const u64 *ext, const __grid_constant__ Ptrs d, const u64 *evk, u64 g, u64 *u,
                                                                uint32_t level, uint32_t nb, uint32_t bch, int has_multi, const __grid_constant__ KsMulti multi,
                                                                int acc_u, const __grid_constant__ Ptrs add) {
    const uint32_t p = (blockIdx.x * IP_THREADS + threadIdx.x) * 2;
    const uint32_t x = blockIdx.z;     // chunks of a limb run together: its key words (and shared digits) come from L2
    uint32_t b0 = blockIdx.y * bch, b1 = min(b0 + bch, nb), e0 = has_multi ? 0 : b0;      // entries; first digits entry
    const uint32_t nt = level + c.K;
    const uint32_t kt = x < level ? x : c.L + (x - level);
    const double2 md = c.modd[kt];
    const size_t js = (size_t)nt * c.N, ks = (size_t)c.T * c.N;
    if (has_multi && multi.group) {     // key r on a chunk of the group's members
        const uint32_t cpr = (multi.group + bch - 1) / bch, r = blockIdx.y / cpr, ch = blockIdx.y % cpr;
        e0 = ch * bch;
        b0 = r * multi.group + e0;
        if (multi.own) e0 = b0;
        b1 = min(b0 + bch, (r + 1) * multi.group);
        evk = multi.evk[r]; g = multi.galois[r];
    } else if (has_multi) { evk = multi.evk[b0]; g = multi.galois[b0]; }
    const uint32_t src = galois_src(p, (uint32_t)g, c.log_n);
    const bool odd = src & 1;
    grid_dep_sync();
    // all loads of a step are issued before the first product (the barrier keeps the compiler from spreading them out): the
    // kernel is bound by how many of its scattered 16-byte reads are in flight
    ulonglong2 kv[BETA][2], ev[BETA];             // [digit][component]
#pragma unroll
    for (uint32_t j = 0; j < BETA; j++)
#pragma unroll
        for (uint32_t cm = 0; cm < 2; cm++) kv[j][cm] = *reinterpret_cast<const ulonglong2 *>(evk + ((size_t)j * 2 + cm) * ks + (size_t)kt * c.N + p);
    const uint32_t own = x < level ? x / c.alpha : BETA;       // the digit that has x among its own limbs: it lies in d
    const size_t off = (size_t)x * c.N + (src & ~1u);
    u64 *o = u + b0 * 2 * js + (size_t)x * c.N + p;
    const double pq = ADD && x < level ? c.dn_p_mod_d[x] : 0.0;
    double k[BETA][2][2];                         // [digit][component][coefficient of the pair]
    for (uint32_t b = b0; b < b1; b++, o += 2 * js) {
        const uint32_t be = b - b0 + e0;
#pragma unroll
        for (uint32_t j = 0; j < BETA; j++)
            ev[j] = *reinterpret_cast<const ulonglong2 *>((j == own ? d.at(be) : ext + ((size_t)be * BETA + j) * js) + off);
        ulonglong2 z[2];
        if (ADD && x < level)
#pragma unroll
            for (uint32_t cm = 0; cm < 2; cm++) z[cm] = *reinterpret_cast<const ulonglong2 *>(add.at(b) + ((size_t)cm * level + x) * c.N + p);
        __syncwarp();
        if (b == b0) {
#pragma unroll
            for (uint32_t j = 0; j < BETA; j++)
#pragma unroll
                for (uint32_t cm = 0; cm < 2; cm++) {
                    k[j][cm][0] = u64_to_d(kv[j][cm].x);
                    k[j][cm][1] = u64_to_d(kv[j][cm].y);
                }
        }
        double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
        if (ADD && x < level)
#pragma unroll
            for (uint32_t cm = 0; cm < 2; cm++) {
                acc[cm][0] = mulmod_dd(u64_to_d(z[cm].x), pq, md.x, md.y);
                acc[cm][1] = mulmod_dd(u64_to_d(z[cm].y), pq, md.x, md.y);
            }
#pragma unroll
        for (uint32_t j = 0; j < BETA; j++) {
            const double d0 = u64_to_d(odd ? ev[j].y : ev[j].x), d1 = u64_to_d(odd ? ev[j].x : ev[j].y);
#pragma unroll
            for (uint32_t cm = 0; cm < 2; cm++) {
                acc[cm][0] = __dadd_rn(acc[cm][0], mulmod_dd(d0, k[j][cm][0], md.x, md.y));
                acc[cm][1] = __dadd_rn(acc[cm][1], mulmod_dd(d1, k[j][cm][1], md.x, md.y));
            }
        }
#pragma unroll
        for (uint32_t cm = 0; cm < 2; cm++) {
            ulonglong2 r;
            r.x = canonical_d(reduce_d(acc[cm][0], md.x, md.y), md.x);
            r.y = canonical_d(reduce_d(acc[cm][1], md.x, md.y), md.x);
            if (acc_u) {
                const ulonglong2 old = *reinterpret_cast<const ulonglong2 *>(o + cm * js);
                const u64 m = c.mod[kt];
                r.x = add_mod(r.x, old.x, m);
                r.y = add_mod(r.y, old.y, m);
            }
            *reinterpret_cast<ulonglong2 *>(o + cm * js) = r;
        }
    }
}

// The inner product of several terms at once (see ks_inner_terms): like inner_product_kernel, but every term has its
// own digits, key, permutation and first component, and the running sums of a chunk of IP_BCH batch entries stay in
// registers over the terms.
// Two entries per thread at 64 registers and 32 warps per SM: four entries at 85 registers kept too few loads in flight (the
// 4096 x 4096 projection's share: 20.2 -> 17.4 ms; one entry 19.9, two at 48 registers 21.3).
constexpr uint32_t IP_BCH = 2;
template <uint32_t BETA>
__global__ void __launch_bounds__(IP_THREADS, 8) inner_product_terms_kernel(DevTables c, const u64 *ext, size_t term_stride, const u64 *d, size_t d_stride,
                                                                         const __grid_constant__ IpTerms tm, uint32_t nterm, size_t c0_stride,
                                                                         u64 *u, uint32_t level, uint32_t nb, int acc_u) {
    const uint32_t p = (blockIdx.x * IP_THREADS + threadIdx.x) * 2;
    const uint32_t x = blockIdx.z, b0 = blockIdx.y * IP_BCH;
    const uint32_t nt = level + c.K;
    const uint32_t kt = x < level ? x : c.L + (x - level);
    const double2 md = c.modd[kt];
    const size_t js = (size_t)nt * c.N, ks = (size_t)c.T * c.N;
    const double pq = x < level ? c.dn_p_mod_d[x] : 0.0;
    const uint32_t own = x < level ? x / c.alpha : BETA;       // the digit that has x among its own limbs: it lies in d
    double acc[IP_BCH][2][2];
#pragma unroll
    for (uint32_t bi = 0; bi < IP_BCH; bi++) acc[bi][0][0] = acc[bi][0][1] = acc[bi][1][0] = acc[bi][1][1] = 0.0;
    grid_dep_sync();
    for (uint32_t t = 0; t < nterm; t++) {
        const uint32_t src = galois_src(p, (uint32_t)tm.galois[t], c.log_n);
        const bool odd = src & 1;
        const u64 *evk = tm.evk[t];
        double k[BETA][2][2];
#pragma unroll
        for (uint32_t j = 0; j < BETA; j++)
#pragma unroll
            for (uint32_t cm = 0; cm < 2; cm++) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(evk + ((size_t)j * 2 + cm) * ks + (size_t)kt * c.N + p);
                k[j][cm][0] = u64_to_d(v.x);
                k[j][cm][1] = u64_to_d(v.y);
            }
        const uint32_t so = src & ~1u;
        const u64 *z = (x < level && tm.c0[t]) ? tm.c0[t] + b0 * c0_stride + (size_t)x * c.N : nullptr;
        // no branch in here, so that the loads of all entries of the chunk are in flight together: an entry past the end
        // of the batch repeats the last one and is not stored
#pragma unroll
        for (uint32_t bi = 0; bi < IP_BCH; bi++) {
            const uint32_t bc = min(bi, nb - 1 - b0);
            double sum[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
            for (uint32_t j = 0; j < BETA; j++) {
                const u64 *ej = (j == own ? d + (size_t)(t * nb + b0 + bc) * d_stride
                                          : ext + t * term_stride + ((size_t)(b0 + bc) * BETA + j) * js) + (size_t)x * c.N;
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(ej + so);
                const double d0 = u64_to_d(odd ? v.y : v.x), d1 = u64_to_d(odd ? v.x : v.y);
#pragma unroll
                for (uint32_t cm = 0; cm < 2; cm++) {
                    sum[cm][0] = __dadd_rn(sum[cm][0], mulmod_dd(d0, k[j][cm][0], md.x, md.y));
                    sum[cm][1] = __dadd_rn(sum[cm][1], mulmod_dd(d1, k[j][cm][1], md.x, md.y));
                }
            }
            if (z) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(z + bc * c0_stride + so);
                sum[0][0] = __dadd_rn(sum[0][0], mulmod_dd(u64_to_d(odd ? v.y : v.x), pq, md.x, md.y));
                sum[0][1] = __dadd_rn(sum[0][1], mulmod_dd(u64_to_d(odd ? v.x : v.y), pq, md.x, md.y));
            }
            // at most BETA + 1 products of size 0.75 m on top of a reduced sum: far below 2^53
#pragma unroll
            for (uint32_t cm = 0; cm < 2; cm++) {
                acc[bi][cm][0] = reduce_d(__dadd_rn(acc[bi][cm][0], sum[cm][0]), md.x, md.y);
                acc[bi][cm][1] = reduce_d(__dadd_rn(acc[bi][cm][1], sum[cm][1]), md.x, md.y);
            }
        }
    }
    const u64 m = c.mod[kt];
#pragma unroll
    for (uint32_t bi = 0; bi < IP_BCH; bi++) {
        if (b0 + bi >= nb) break;
        u64 *o = u + (size_t)(b0 + bi) * 2 * js + (size_t)x * c.N + p;
#pragma unroll
        for (uint32_t cm = 0; cm < 2; cm++) {
            ulonglong2 r;
            r.x = canonical_d(acc[bi][cm][0], md.x);
            r.y = canonical_d(acc[bi][cm][1], md.x);
            if (acc_u) {
                const ulonglong2 old = *reinterpret_cast<const ulonglong2 *>(o + cm * js);
                r.x = add_mod(r.x, old.x, m);
                r.y = add_mod(r.y, old.y, m);
            }
            *reinterpret_cast<ulonglong2 *>(o + cm * js) = r;
        }
    }
}

// conv[comp][i][k] = sum_a centre([u_{p_a} Phat_a^-1]) (Phat_a mod q_i)  mod q_i   (coefficient domain)
// Same shape as ModUp: the K centred special residues are formed once per thread, then a chunk of targets is walked.
// RS, the conversion of a ModDown that a rescale follows: u's limb `targets` (the one to drop, q_l) lies in the coefficient
// domain too.  Its share of the ModDown is finished here, r = centre((u_l - conv_l) P^-1 mod q_l), and every target's conv
// gets P r on top, so that (u_i - NTT(conv_i + P r)) (P q_l)^-1 is the rescaled ModDown: one transform of each remaining
// limb, where ModDown and rescale after each other take two (and four more launches).
template <uint32_t KK, uint32_t CPT, bool RS>
__global__ void __launch_bounds__(CONV_THREADS) moddown_conv_kernel(DevTables c, const u64 *u, u64 *conv, uint32_t level, uint32_t targets, uint32_t CHUNK) {
    __shared__ __align__(16) double s_w[CONV_CHUNK_MAX + RS][KK];     // Phat_a mod q_i (the last row: of the dropped limb)
    __shared__ double2 s_m[CONV_CHUNK_MAX];                           // q_i, 1 / q_i
    __shared__ double s_p[RS ? CONV_CHUNK_MAX : 1];                   // P mod q_i
    const uint32_t k = (blockIdx.x * CONV_THREADS + threadIdx.x) * CPT;
    const uint32_t comp = blockIdx.z & 1, bz = blockIdx.z >> 1;
    const uint32_t nt = level + c.K;
    const uint32_t i0 = blockIdx.y * CHUNK, i1 = min(i0 + CHUNK, targets);
    for (uint32_t e = threadIdx.x; e < (i1 - i0) * KK; e += CONV_THREADS) {
        const uint32_t ii = e / KK, a = e % KK;
        s_w[ii][a] = a < c.K ? c.dn_hat_mod_d[(size_t)(i0 + ii) * c.K + a] : 0.0;
        if (a == 0) s_m[ii] = c.modd[i0 + ii];
        if (RS && a == 0) s_p[ii] = c.dn_p_mod_d[i0 + ii];
    }
    if (RS && threadIdx.x < KK) s_w[CONV_CHUNK_MAX + RS - 1][threadIdx.x] = threadIdx.x < c.K ? c.dn_hat_mod_d[(size_t)targets * c.K + threadIdx.x] : 0.0;
    u += (((size_t)bz * 2 + comp) * nt + level) * c.N + k;
    conv += ((size_t)bz * 2 + comp) * targets * c.N + k;
    double y[CPT][KK], r[CPT];
    grid_dep_sync();
#pragma unroll
    for (uint32_t a = 0; a < KK; a++) {
        u64 v[CPT];
        if (a < c.K) conv_load<CPT>(u + (size_t)a * c.N, v);
#pragma unroll
        for (uint32_t p = 0; p < CPT; p++) {
            y[p][a] = 0.0;
            if (a < c.K) {
                const u64 pa = c.mod[c.L + a];
                y[p][a] = centre_d(v[p], pa);
            }
        }
    }
    __syncthreads();
    if (RS) {
        const double2 md = c.modd[targets], pinv = c.dn_p_inv_d[targets];
        u64 v[CPT];
        conv_load<CPT>(u - c.N, v);
        conv_dot<true>(y, s_w[CONV_CHUNK_MAX + RS - 1], md.x, md.y, r);
#pragma unroll
        for (uint32_t p = 0; p < CPT; p++)
            r[p] = centre_d(canonical_d(reduce_d(mulmod_d<0>(__dsub_rn(u64_to_d(v[p]), r[p]), pinv, md.x), md.x, md.y), md.x), c.mod[targets]);
    }
    for (uint32_t i = i0; i < i1; i++) {
        const double2 md = s_m[i - i0];
        double x[CPT];
        if (RS)
#pragma unroll
            for (uint32_t p = 0; p < CPT; p++) x[p] = mulmod_dd(r[p], s_p[i - i0], md.x, md.y);
        conv_dot<!RS>(y, s_w[i - i0], md.x, md.y, x);
        conv_store<CPT>(conv + (size_t)i * c.N, x);
    }
}

template <uint32_t KK, bool RS>
void launch_moddown_conv(const ckks_ctx *c, const u64 *u, u64 *conv, uint32_t level, uint32_t nb, cudaStream_t s) {
    const uint32_t targets = level - RS, cpt = conv_cpt(KK, u, conv), gx = c->N / (CONV_THREADS * cpt), CHUNK = conv_chunk(c, gx, 2 * nb, targets);
    const dim3 grid(gx, (targets + CHUNK - 1) / CHUNK, 2 * nb);
    constexpr uint32_t WIDE = KK <= 8 ? 2 : 1;
    launch(cpt == WIDE ? moddown_conv_kernel<KK, WIDE, RS> : moddown_conv_kernel<KK, 1, RS>, grid, CONV_THREADS, 0, s, c->dev, u, conv, level, targets, CHUNK);
}

// register-array size for a digit / special-prime count: next of 1, 2, 4, 8, 16, 32, 64
#define DISPATCH_POW2(n, CALL)                      \
    do {                                            \
        if ((n) <= 1) { CALL(1); }                  \
        else if ((n) <= 2) { CALL(2); }             \
        else if ((n) <= 4) { CALL(4); }             \
        else if ((n) <= 8) { CALL(8); }             \
        else if ((n) <= 16) { CALL(16); }           \
        else if ((n) <= 32) { CALL(32); }           \
        else { CALL(64); }                          \
    } while (0)

// dst row (row0 + i * row_step + comp) of a tiled buffer <- component comp of ciphertext i, blockIdx.z = 2 i + comp
__global__ void __launch_bounds__(THREADS) to_tiled_kernel(DevTables c, const u64 *src, size_t src_stride, u64 *dst, uint32_t R,
                                                           uint32_t row0, uint32_t row_step) {
    grid_dep_sync();
    const uint32_t p = (blockIdx.x * THREADS + threadIdx.x) * 2, i = blockIdx.y, r = blockIdx.z >> 1, comp = blockIdx.z & 1;
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(src + r * src_stride + ((size_t)comp * gridDim.y + i) * c.N + p);
    *reinterpret_cast<ulonglong2 *>(dst + tiled_index(R, c.N, row0 + r * row_step + comp, i, p)) = v;
}

// dst[x] = first[x] + sum_r terms[r][x] over [nct][2][level][N] words (grid y: limbs of all ciphertexts)
__global__ void __launch_bounds__(THREADS) sum_kernel(DevTables c, u64 *dst, const u64 *first, const u64 *terms, uint32_t n, size_t stride, uint32_t level) {
    const size_t off = (size_t)blockIdx.y * c.N + (blockIdx.x * THREADS + threadIdx.x) * 2;
    const u64 q = c.mod[blockIdx.y % level];
    grid_dep_sync();
    ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(first + off);
    for (uint32_t r = 0; r < n; r++) {
        const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(terms + r * stride + off);
        a.x = add_mod(a.x, b.x, q);
        a.y = add_mod(a.y, b.y, q);
    }
    *reinterpret_cast<ulonglong2 *>(dst + off) = a;
}

// u[b][0][i][p] += P sigma_g(c0[b][i])[p]   (first component's q-limbs of the extended-basis sum)
__global__ void __launch_bounds__(THREADS) p_c0_acc_kernel(DevTables c, const u64 *c0, size_t c0_stride, u64 g, u64 *u, size_t u_stride) {
    grid_dep_sync();
    const uint32_t p = blockIdx.x * THREADS + threadIdx.x, i = blockIdx.y, b = blockIdx.z;
    const double2 md = c.modd[i];
    u64 *d = u + b * u_stride + (size_t)i * c.N + p;
    const double v = mulmod_dd(u64_to_d(c0[b * c0_stride + (size_t)i * c.N + galois_src(p, (uint32_t)g, c.log_n)]), c.dn_p_mod_d[i], md.x, md.y);
    *d = add_mod(*d, canonical_d(reduce_d(v, md.x, md.y), md.x), c.mod[i]);
}

}  // namespace

size_t ks_workspace_limbs(const ckks_ctx *c, uint32_t level) {
    const size_t beta = (level + c->alpha - 1) / c->alpha, nt = level + c->K;
    return level + beta * nt + 2 * nt + 2 * (size_t)level;
}

// Workspace for nb key switches running side by side: dcoef [nb][level], ext [nb][beta][level+K],
// u [nb][2][level+K], conv [nb][2][level].
KsWorkspace ks_carve(const ckks_ctx *c, uint32_t level, void *ws, uint32_t nb) {
    const size_t beta = (level + c->alpha - 1) / c->alpha, nt = level + c->K, N = c->N;
    KsWorkspace w;
    w.dcoef = (u64 *)ws;
    w.ext = w.dcoef + (size_t)nb * level * N;
    w.u = w.ext + (size_t)nb * beta * nt * N;
    w.conv = w.u + (size_t)nb * 2 * nt * N;
    return w;
}

// whether the conversions run on the tensor cores (context option CKKS_CONV_TENSOR: bit-identical, slower on B200); they take
// the inverse transform's plain output, the FP64 kernels one with qhat^-1 (Phat^-1) multiplied in
static bool conv_tensor(const ckks_ctx *c) { return c->conv_kernel == CKKS_CONV_TENSOR && c->dev.conv_groups; }

static const NttPrologue CONV_OUT{nullptr, false, 0, true};     // what the FP64 conversions leave

void ks_modup(const ckks_ctx *c, const Ptrs &d, uint32_t level, KsWorkspace &w, cudaStream_t s, uint32_t nb) {
    const uint32_t beta = (level + c->alpha - 1) / c->alpha, nt = level + c->K;
    w.d = d;
    NttSource src;
    src.ptr = d; src.lpitch = 1;
    if (conv_strip(c, CONV_UP, level, nb * beta, w.alone)) {
        launch_ntt_part(c, NTT_ROWS, w.dcoef, nb * level, plain_map(0, level), true, s, nullptr, nullptr, &src);
        launch_conv_strip(c, CONV_UP, w.dcoef, w.ext, level, nb * beta, s);
        if (!w.mid) launch_ntt_part(c, NTT_ROWS, w.ext, nb * beta * nt, ext_map(level, c->K, c->L, c->alpha, beta), false, s);
        return;
    }
    launch_ntt(c, w.dcoef, nb * level, plain_map(0, level), true, s, nullptr, nullptr, &src,
               conv_tensor(c) ? nullptr : c->dev.inv_scale_up + (size_t)level * c->L * 2, w.alone);
    if (conv_tensor(c)) {
        launch_modup_mma(c, w.dcoef, w.ext, level, nb, s);
    } else {
#define CALL_UP(A) launch_modup<A>(c, w.dcoef, w.ext, level, nb, s)
        DISPATCH_POW2(c->alpha, CALL_UP);
#undef CALL_UP
    }
    if (w.mid) launch_ntt_part(c, NTT_COLS, w.ext, nb * beta * nt, ext_map(level, c->K, c->L, c->alpha, beta), false, s, nullptr, conv_tensor(c) ? nullptr : &CONV_OUT);
    else launch_ntt(c, w.ext, nb * beta * nt, ext_map(level, c->K, c->L, c->alpha, beta), false, s, nullptr, conv_tensor(c) ? nullptr : &CONV_OUT, nullptr, nullptr, w.alone);
}

void ks_inner(const ckks_ctx *c, const u64 *evk, uint32_t level, u64 ext_galois, const KsWorkspace &w, cudaStream_t s, uint32_t nb,
              bool acc_u, const KsMulti *multi, const Ptrs *add) {
    const uint32_t N = c->N, nt = level + c->K;
    const uint32_t beta = (level + c->alpha - 1) / c->alpha;
    const int au = acc_u ? 1 : 0;
    bool aligned = aligned16(w.ext) && aligned16(w.u) && aligned16(w.d) && (multi || aligned16(evk));
    const uint32_t nkeys = multi ? (multi->group ? nb / multi->group : nb) : 0;
    for (uint32_t b = 0; b < nkeys; b++) aligned = aligned && aligned16(multi->evk[b]);
    if (add) aligned = aligned && aligned16(*add);
    const bool fast = beta <= IP_MAX_BETA && aligned && (!add || beta > IP_FUSED_BETA);       // (mid_rows adds to fewer digits' products)
    const Ptrs pa = add ? *add : Ptrs();
    if (multi && multi->group && !fast) {       // grouped entries without the fast kernel: one key at a time
        for (uint32_t r = 0; r < nkeys; r++) {
            KsWorkspace wr = w;
            wr.u = w.u + (size_t)r * multi->group * 2 * nt * N;
            if (multi->own) {
                wr.ext = w.ext + (size_t)r * multi->group * beta * nt * N;
                wr.d.base += r * multi->group * w.d.stride;
            }
            ks_inner(c, multi->evk[r], level, multi->galois[r], wr, s, multi->group, acc_u, nullptr);
        }
        return;
    }
    const KsMulti m = multi ? *multi : KsMulti{};
    if (fast) {
        // batch entries per thread: enough chunks left to fill the machine, key words reused across a chunk (sixteen entries, 4 ->
        // 8 per thread: 13.9 -> 12.7 ms of the 4096 x 4096 projection; half of these shares: 15.9 ms)
        const uint32_t grp = multi ? multi->group : 0, per = grp ? grp : nb;
        const uint32_t bch = (multi && !grp) ? 1 : (per >= 16 ? 8 : per >= 8 ? 4 : per >= 4 ? 2 : 1);
        const dim3 grid(N / (2 * IP_THREADS), grp ? (nb / grp) * ((grp + bch - 1) / bch) : (nb + bch - 1) / bch, nt);
        using K = decltype(&inner_product_kernel<1, false>);
        static constexpr K plain[IP_MAX_BETA] = {inner_product_kernel<1, false>, inner_product_kernel<2, false>, inner_product_kernel<3, false>, inner_product_kernel<4, false>,
                                                 inner_product_kernel<5, false>, inner_product_kernel<6, false>, inner_product_kernel<7, false>, inner_product_kernel<8, false>};
        static constexpr K adding[IP_MAX_BETA - IP_FUSED_BETA] = {inner_product_kernel<5, true>, inner_product_kernel<6, true>, inner_product_kernel<7, true>, inner_product_kernel<8, true>};
        launch(add ? adding[beta - 1 - IP_FUSED_BETA] : plain[beta - 1], grid, IP_THREADS, 0, s, c->dev, w.ext, w.d, evk, ext_galois, w.u, level, nb, bch, multi ? 1 : 0, m, au, pa);
    } else {
        launch(inner_product_generic_kernel, dim3(N / THREADS, nb, nt), THREADS, 0, s, c->dev, w.ext, w.d, 0u, evk, ext_galois, w.u, level, multi ? 1 : 0, m, au,
               add ? 1 : 0, pa);
    }
}

// mid_rows takes up to IP_FUSED_BETA digits and 16-byte accesses (one rotation at N = 2^16, level 24: 153 -> 149.4 us, at N = 2^14 32.8 ->
// 29.4; the degree-63 polynomial 2139 -> 2091; projections of 24 tokens, which sum their giant steps, 32.1 -> 31.7 ms)
bool ks_mid(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, const Ptrs &d, const u64 *const *evk, uint32_t nkeys) {
    // plain transforms around the tensor cores' conversions: a share of their limbs may be on the integer pipe, which runs whole transforms
    if (conv_tensor(c) && c->ntt_fp_share < 8 && c->log_n == 16) return false;
    bool ok = (level + c->alpha - 1) / c->alpha <= IP_FUSED_BETA && aligned16(w.ext) && aligned16(w.u) && aligned16(d);
    for (uint32_t k = 0; k < nkeys; k++) ok = ok && aligned16(evk[k]);
    return ok;
}
// Sums of terms: a row's terms follow one another in its CTA, so that few CTAs make a long chain, where separate launches transform all
// terms' digits side by side.  mid_rows takes them from three CTAs per SM on (sums of sixteen terms: N = 2^15, level 12, 512 CTAs, 459 ->
// 432 us; level 10, 448 CTAs, 401 -> 386; but level 8, 384 CTAs, 273 -> 282; N = 2^14, level 6, 128 CTAs, 191 -> 252; N = 2^13, level 4, 40
// CTAs, 149 -> 223; lazy projections of one to three shards there 1.07 to 1.22 times as long), and short chains of two terms
// everywhere (N = 2^13, level 4, 40.3 -> 39.6 us; of four 48.5 -> 60.4).
bool ks_mid_sum(const ckks_ctx *c, uint32_t level, uint32_t nterm, uint32_t nb) {
    return nterm <= 2 || (uint64_t)(c->N >> 10) * nb * (level + c->K) >= 3 * (uint64_t)c->sms;
}
static void mid_inner(const ckks_ctx *c, const u64 *evk, uint32_t level, u64 galois, const KsWorkspace &w, uint32_t inv_from, cudaStream_t s, uint32_t nb, const KsMulti *multi,
                      const Ptrs *add) {
    MidArgs a{};
    a.ext = w.ext; a.d = w.d; a.u = w.u;
    a.nterm = 1; a.nb = nb; a.level = level; a.inv_from = inv_from;
    a.evk[0] = evk; a.galois[0] = galois;
    if (multi) {
        a.group = multi->group;
        for (uint32_t r = 0; r < nb / multi->group; r++) { a.evk[r] = multi->evk[r]; a.galois[r] = multi->galois[r]; }
    }
    if (add) { a.has_add = 1; a.add = *add; }
    launch_mid_rows(c, a, (level + c->alpha - 1) / c->alpha, s);
}

// Whether the row pass that ends a ModDown forms the inner product's q-limbs itself (mode 3 of the epilogue), so that the sum u
// is written and read back for the special limbs only.  It does where keys share digits (digits of one key go through mid_rows), a key
// word serves fewer than four entries (four or more share it from registers in inner_product_kernel, where this form would read it from
// L2 for each) and the pass fills the GPU once: below that its eight steps of dependent reads cost more than the traffic (64 hoisted
// rotations at N = 2^16, level 24: 4550 -> 4110 us; the key/value projections of 24 tokens 35.9 -> 34.3 ms).  Operands have to take
// 16-byte accesses.
static bool inner_fused(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, uint32_t nb, const KsMulti *multi) {
    if (!multi || multi->own) return false;
    const uint32_t beta = (level + c->alpha - 1) / c->alpha, nkeys = multi->group ? nb / multi->group : nb;
    bool ok = multi->group < 4 && beta <= IP_FUSED_BETA && nb * 2 * level <= 32768 && (uint64_t)nb * 2 * level * (c->N >> 10) >= 16 * (uint64_t)c->sms &&
              aligned16(w.ext) && aligned16(w.d);
    for (uint32_t b = 0; b < nkeys; b++) ok = ok && aligned16(multi->evk[b]);
    return ok;
}
// the part of the epilogue that describes the inner product
static void fuse_inner(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, uint32_t nb, const KsMulti &multi, NttEpilogue &ep) {
    ep.mode = 3;
    ep.ext = w.ext; ep.d = w.d; ep.nb = nb;
    ep.beta = (level + c->alpha - 1) / c->alpha;
    for (uint32_t b = 0; b < KS_MULTI; b++) ep.mevk[b] = multi.evk[b];
}
static bool out_aligned(const NttEpilogue &ep) { return aligned16(ep.add) && aligned16(ep.acc) && aligned16(ep.out) && (ep.rot_stride & 1) == 0; }

// the ModDown of w.u; fused: of a w.u whose special limbs alone exist
static NttEpilogue moddown_epilogue(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, const KsOut &o, uint32_t nb, const KsMulti *multi) {
    NttEpilogue ep{};      // the last NTT pass finishes the ModDown itself
    ep.mode = 1;
    ep.u = Ptrs(w.u, (size_t)2 * (level + c->K) * c->N);
    ep.add = o.add; ep.out = o.out; ep.add_comps = o.add_comps;
    ep.pinv = c->dev.dn_p_inv_d;
    ep.ncomp = 2; ep.level = level; ep.nt = level + c->K;
    ep.galois = o.galois; ep.acc = o.acc; ep.accumulate = o.acc.n || o.acc.base ? 1 : 0; ep.tl = o.tiled;
    if (multi) {
        ep.multi = 1; ep.group = multi->group; ep.own = multi->own; ep.rot_rows = multi->rot_rows; ep.rot_stride = multi->rot_stride;
        for (uint32_t b = 0; b < KS_MULTI; b++) { ep.mgalois[b] = multi->galois[b]; ep.out.p[b] = multi->out[b]; }
        if (!multi->group) ep.out.n = nb;
    }
    return ep;
}
static void moddown(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, NttEpilogue ep, cudaStream_t s, uint32_t nb) {
    const uint32_t N = c->N, nt = level + c->K, K = c->K;
    // the K special limbs of every (batch, component): groups of K limbs, nt limbs apart
    const bool strip = conv_strip(c, CONV_DOWN, level, 2 * nb);
    const NttPart first = NttPart((w.mid ? 0 : NTT_ROWS) | (strip ? 0 : NTT_COLS));
    const double2 *scale = conv_tensor(c) ? nullptr : c->dev.inv_scale_dn;
    if (first == NTT_BOTH)
        launch_ntt(c, w.u + (size_t)level * N, nb * 2 * K, pitched_map(c->L, K, nt), true, s, ep.mode == 3 ? &ep : nullptr, nullptr, nullptr, scale, w.alone);
    else if (first)
        launch_ntt_part(c, first, w.u + (size_t)level * N, nb * 2 * K, pitched_map(c->L, K, nt), true, s, ep.mode == 3 ? &ep : nullptr, nullptr, nullptr, scale);
    if (strip) {
        launch_conv_strip(c, CONV_DOWN, w.u, w.conv, level, 2 * nb, s);
        launch_ntt_part(c, NTT_ROWS, w.conv, nb * 2 * level, plain_map(0, level), false, s, &ep);
        return;
    }
    if (conv_tensor(c)) {
        launch_moddown_conv_mma(c, w.u, w.conv, level, nb, s);
    } else {
#define CALL_DN(A) launch_moddown_conv<A, false>(c, w.u, w.conv, level, nb, s)
        DISPATCH_POW2(K, CALL_DN);
#undef CALL_DN
    }
    launch_ntt(c, w.conv, nb * 2 * level, plain_map(0, level), false, s, &ep, conv_tensor(c) ? nullptr : &CONV_OUT);
}
void ks_moddown(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, const KsOut &o, cudaStream_t s, uint32_t nb, const KsMulti *multi) {
    KsWorkspace wd = w;
    wd.mid = false;         // all of u is in the evaluation domain
    moddown(c, level, wd, moddown_epilogue(c, level, wd, o, nb, multi), s, nb);
}
void ks_apply(const ckks_ctx *c, const u64 *evk, uint32_t level, const KsWorkspace &w, const KsOut &o, cudaStream_t s, uint32_t nb, const KsMulti *multi) {
    NttEpilogue ep = moddown_epilogue(c, level, w, o, nb, multi);
    if (w.mid) {
        mid_inner(c, evk, level, o.galois, w, level, s, nb, multi, nullptr);
        moddown(c, level, w, ep, s, nb);
        return;
    }
    if (inner_fused(c, level, w, nb, multi) && out_aligned(ep)) fuse_inner(c, level, w, nb, *multi, ep);
    else ks_inner(c, evk, level, o.galois, w, s, nb, false, multi);
    moddown(c, level, w, ep, s, nb);
}

// The tensor-core conversions have no form that carries the dropped limb along
bool ks_fused_rescale(const ckks_ctx *c) { return !conv_tensor(c); }

// ModDown and rescale at once, bit for bit what they give one after the other (see moddown_conv_kernel); the polynomial of
// degree 63 at N = 2^16, level 24, whose products all end this way: 2615 -> 2295 us.
void ks_apply_rescale(const ckks_ctx *c, const u64 *evk, uint32_t level, const KsWorkspace &w, const Ptrs &add, const Ptrs &out, cudaStream_t s, uint32_t nb) {
    const uint32_t N = c->N, K = c->K, nt = level + K, m = level - 1;
    NttEpilogue ep{};
    ep.mode = 1;
    ep.u = Ptrs(w.u, (size_t)2 * nt * N);
    ep.out = out;
    ep.pinv = c->dev.rs_p_inv_d + (size_t)m * c->L;
    ep.ncomp = 2; ep.level = m; ep.nt = nt; ep.galois = 1;
    const bool strip = conv_strip(c, CONV_DOWN_RS, level, 2 * nb);
    if (w.mid) mid_inner(c, evk, level, 1, w, m, s, nb, nullptr, &add);
    else ks_inner(c, evk, level, 1, w, s, nb, false, nullptr, &add);
    // the dropped limb and the K special limbs of every (batch, component), nt limbs apart
    const NttPart first = NttPart((w.mid ? 0 : NTT_ROWS) | (strip ? 0 : NTT_COLS));
    if (first)
        launch_ntt_part(c, first, w.u + (size_t)m * N, nb * 2 * (K + 1), tail_map(m, level, K, c->L), true, s, nullptr, nullptr, nullptr,
                        c->dev.inv_scale_rs + (size_t)m * (K + 1) * 2);
    if (strip) {
        launch_conv_strip(c, CONV_DOWN_RS, w.u, w.conv, level, 2 * nb, s);
        launch_ntt_part(c, NTT_ROWS, w.conv, nb * 2 * m, plain_map(0, m), false, s, &ep);
        return;
    }
#define CALL_DN(A) launch_moddown_conv<A, true>(c, w.u, w.conv, level, nb, s)
    DISPATCH_POW2(K, CALL_DN);
#undef CALL_DN
    launch_ntt(c, w.conv, nb * 2 * m, plain_map(0, m), false, s, &ep, &CONV_OUT);
}

void ks_inner_terms(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, size_t term_stride, const IpTerms &terms, uint32_t nterm,
                    size_t c0_stride, cudaStream_t s, uint32_t nb, bool acc_u) {
    const uint32_t N = c->N, nt = level + c->K, beta = (level + c->alpha - 1) / c->alpha;
    if (w.mid) {
        MidArgs a{};
        a.ext = w.ext; a.d = w.d; a.u = w.u;
        a.nterm = nterm; a.nb = nb; a.level = level; a.inv_from = nt;
        a.term_stride = term_stride; a.c0_stride = c0_stride; a.acc_u = acc_u ? 1 : 0;
        for (uint32_t t = 0; t < nterm; t++) { a.evk[t] = terms.evk[t]; a.galois[t] = terms.galois[t]; a.c0[t] = terms.c0[t]; }
        launch_mid_rows(c, a, beta, s);
        return;
    }
    bool aligned = aligned16(w.ext) && aligned16(w.u) && (term_stride & 1) == 0 && (c0_stride & 1) == 0 && aligned16(w.d);
    for (uint32_t t = 0; t < nterm; t++) aligned = aligned && aligned16(terms.evk[t]) && aligned16(terms.c0[t]);
    if (beta <= IP_TERMS_MAX_BETA && aligned) {
        const dim3 grid(N / (2 * IP_THREADS), (nb + IP_BCH - 1) / IP_BCH, nt);
        auto *k = beta == 1 ? inner_product_terms_kernel<1> : beta == 2 ? inner_product_terms_kernel<2> : beta == 3 ? inner_product_terms_kernel<3> : inner_product_terms_kernel<4>;
        launch(k, grid, IP_THREADS, 0, s, c->dev, w.ext, term_stride, w.d.base, w.d.stride, terms, nterm, c0_stride, w.u, level, nb, acc_u ? 1 : 0);
        return;
    }
    // any number of digits, any alignment: one term at a time through the generic kernel, then its P c0
    for (uint32_t t = 0; t < nterm; t++) {
        launch(inner_product_generic_kernel, dim3(N / THREADS, nb, nt), THREADS, 0, s, c->dev, w.ext + t * term_stride, w.d, t * nb, terms.evk[t], terms.galois[t],
               w.u, level, 0, KsMulti{}, (acc_u || t > 0) ? 1 : 0, 0, Ptrs());
        if (terms.c0[t])
            launch(p_c0_acc_kernel, dim3(N / THREADS, level, nb), THREADS, 0, s, c->dev, terms.c0[t], c0_stride, terms.galois[t], w.u, (size_t)2 * nt * N);
    }
}

void launch_to_tiled(const ckks_ctx *c, const u64 *src, size_t src_stride, uint32_t n, u64 *dst, uint32_t R, uint32_t row0,
                     uint32_t row_step, uint32_t level, cudaStream_t s) {
    for (uint32_t r0 = 0; r0 < n; r0 += 16384) {
        const uint32_t nr = std::min(16384u, n - r0);
        launch(to_tiled_kernel, dim3(c->N / (2 * THREADS), level, 2 * nr), THREADS, 0, s, c->dev, src + r0 * src_stride, src_stride, dst, R,
               row0 + r0 * row_step, row_step);
    }
}

void launch_sum(const ckks_ctx *c, u64 *dst, const u64 *first, const u64 *terms, uint32_t n, uint32_t nct, uint32_t level, cudaStream_t s) {
    const size_t ct = (size_t)2 * level * c->N;
    for (uint32_t i0 = 0; i0 < nct; i0 += 256) {        // grid y holds 2 level (at most 128) limbs per ciphertext
        const uint32_t m = std::min(256u, nct - i0);
        launch(sum_kernel, dim3(c->N / (2 * THREADS), m * 2 * level), THREADS, 0, s, c->dev, dst + i0 * ct, first + i0 * ct, terms + i0 * ct, n, nct * ct, level);
    }
}

// Drops the last limb of every component: its inverse transform (out of place), then the forward transform whose first pass
// lifts it to its centred representative modulo every remaining prime and whose last pass finishes (in - NTT(lift)) q_last^-1.
// Four launches for the whole batch; copies of the last limbs, the lift and the final step were kernels of their own before
// (10 operations, 63 -> 36 us for one ciphertext at N = 2^16, level 17).
// ws: [nb][ncomp][N] last limbs + [nb][ncomp][level-1][N]
void launch_rescale(const ckks_ctx *c, const Ptrs &in, const Ptrs &out, uint32_t ncomp, uint32_t level, u64 *ws, cudaStream_t s, uint32_t nb, bool alone) {
    const size_t N = c->N;
    u64 *last = ws, *tmp = ws + (size_t)nb * ncomp * N;
    NttSource src;
    src.ptr = in; src.lpitch = level;
    if (in.n) for (uint32_t b = 0; b < in.n; b++) src.ptr.p[b] += (size_t)(level - 1) * N;
    else src.ptr.base += (size_t)(level - 1) * N;
    launch_ntt(c, last, nb * ncomp, same_map(level - 1, ncomp), true, s, nullptr, nullptr, &src, nullptr, alone);
    NttPrologue pro{last, true, level - 1};
    NttEpilogue ep{};
    ep.mode = 1;
    ep.u = in; ep.out = out;
    ep.pinv = c->dev.rs_inv_d + (size_t)(level - 1) * c->L;
    ep.ncomp = ncomp; ep.level = level - 1; ep.nt = level; ep.galois = 1;
    launch_ntt(c, tmp, nb * ncomp * (level - 1), plain_map(0, level - 1), false, s, &ep, &pro);
}
