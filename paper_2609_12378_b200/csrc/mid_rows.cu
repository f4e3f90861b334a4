// What lies between the two column-wise kernels of a key switch whose digits serve one key: the forward row pass of the extended
// digits, their inner product with the key, and the inverse row pass of the limbs that ModDown converts.
//
// sigma_g maps rows of 256 words onto rows (a word's row is the low part of its bit-reversed index, and the low part of g (2 b + 1)
// follows from the low part of b), so that a row of the result needs one row of each digit: nothing but the sums leaves the SM,
// where the digits' evaluation form made a trip through memory (36 MiB out and 96 MiB in per ciphertext at N = 2^16, level 24) and
// two launches were one more.  Digits that many keys share (hoisted rotations, baby steps) keep that form: it is computed once.
#include "butterfly.cuh"

namespace {

// A warp per row, eight coefficients per lane (stages in groups of 3, 3 and 2), so that the sums of both components fit 64 registers:
// the kernel waits for its key words and digits, and 32 warps per SM wait for more of them at a time (16 lanes per row with
// sixteen coefficients and 128 registers: 54 us for one ciphertext at N = 2^16, level 24).  Sums over terms hold theirs throughout, and at
// five CTAs per SM those of three and four digits spill (144 and 220 bytes per thread stored).
constexpr uint32_t MID_ROWS = 4;

template <uint32_t BETA, bool TERMS>
__global__ void __launch_bounds__(32 * MID_ROWS, TERMS ? 5 : 8) mid_rows(DevTables c, const __grid_constant__ MidArgs a) {
    __shared__ __align__(16) double sm[BETA][MID_ROWS][WROW_PAD];
    const uint32_t t = threadIdx.x & 31, rl = threadIdx.x >> 5, row = blockIdx.x * MID_ROWS + rl, R = c.N >> 8;
    // special limbs, which have the most to do, first: they would stretch the last wave (rotation at N = 2^15 42.6 -> 40.8 us, at
    // N = 2^16 150.9 -> 149.7)
    const uint32_t bz = blockIdx.y, nt = a.level + c.K, x = TERMS ? blockIdx.z : nt - 1 - blockIdx.z, kt = x < a.level ? x : c.L + (x - a.level);
    const double q = c.modd[kt].x, qinv = c.modd[kt].y;
    const uint32_t p0 = row * 256 + 2 * t, own = x < a.level ? x / c.alpha : BETA;       // own: the digit that has x among its own limbs
    const size_t limb = (size_t)1 << c.log_n;
    double s0[8], s1[8];               // sums of words p0 + 64 k, p0 + 64 k + 1 of both components
    if (TERMS)
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) s0[k] = s1[k] = 0.0;
    grid_dep_sync();
    const uint32_t nterm = TERMS ? a.nterm : 1;
#pragma unroll 1
    for (uint32_t term = 0; term < nterm; term++) {
        const uint32_t key = a.group ? bz / a.group : term;
        const uint32_t gal = (uint32_t)a.galois[key], srow = galois_src(row << 8, gal, c.log_n) >> 8;
#pragma unroll 1
        for (uint32_t j = 0; j < BETA; j++) {
            double *s = sm[j][rl];
            if (j == own) {
                const u64 *d = a.d.at(term * a.nb + bz) + x * limb + srow * 256 + 2 * t;
                ulonglong2 w[4];
#pragma unroll
                for (uint32_t k = 0; k < 4; k++) w[k] = ld_pair<true>(d + 64 * k);
#pragma unroll
                for (uint32_t k = 0; k < 4; k++) *reinterpret_cast<double2 *>(s + wrow_at(2 * t) + 72 * k) = make_double2(u64_to_d(w[k].x), u64_to_d(w[k].y));
                continue;
            }
            const double *tw = c.twd_fwd + ((size_t)kt << c.log_n);
            const double *g = reinterpret_cast<const double *>(a.ext + term * a.term_stride) + (((size_t)bz * BETA + j) * nt + x) * limb + srow * 256 + t;
            double v[8];
#pragma unroll
            for (uint32_t k = 0; k < 8; k++) v[k] = g[32 * k];
            wrow_forward(v, s, t, tw, R + srow, q, qinv);
        }
        __syncwarp();
        const u64 *c0 = TERMS && x < a.level && a.c0[term] ? a.c0[term] + bz * a.c0_stride + x * limb + srow * 256 : nullptr;
        const u64 *kp = a.evk[key] + kt * limb + p0;
        const size_t kc = c.T * limb;          // from a key's component to the next, digit by digit
#pragma unroll
        for (uint32_t k = 0; k < 4; k++) {
            const uint32_t sr = galois_src(p0 + 64 * k, gal, c.log_n) & 255, so = sr & ~1u;
            const bool odd = sr & 1;             // the permutation maps the pair onto a pair, possibly swapped
            ulonglong2 kv[BETA][2];
#pragma unroll
            for (uint32_t j = 0; j < BETA; j++) {
                kv[j][0] = ld_pair<true>(kp + 2 * j * kc + 64 * k);
                kv[j][1] = ld_pair<true>(kp + (2 * j + 1) * kc + 64 * k);
            }
            if (!TERMS) s0[2 * k] = s0[2 * k + 1] = s1[2 * k] = s1[2 * k + 1] = 0.0;
            if (TERMS && c0) {
                const ulonglong2 z = ld_pair<true>(c0 + so);
                const double pq = c.dn_p_mod_d[x];
                s0[2 * k] = __dadd_rn(s0[2 * k], mulmod_dd(u64_to_d(odd ? z.y : z.x), pq, q, qinv));
                s0[2 * k + 1] = __dadd_rn(s0[2 * k + 1], mulmod_dd(u64_to_d(odd ? z.x : z.y), pq, q, qinv));
            }
#pragma unroll
            for (uint32_t j = 0; j < BETA; j++) {
                const double2 e = *reinterpret_cast<const double2 *>(sm[j][rl] + wrow_at(so));
                const double e0 = odd ? e.y : e.x, e1 = odd ? e.x : e.y;
                s0[2 * k] = __dadd_rn(s0[2 * k], mulmod_dd(e0, u64_to_d(kv[j][0].x), q, qinv));
                s0[2 * k + 1] = __dadd_rn(s0[2 * k + 1], mulmod_dd(e1, u64_to_d(kv[j][0].y), q, qinv));
                s1[2 * k] = __dadd_rn(s1[2 * k], mulmod_dd(e0, u64_to_d(kv[j][1].x), q, qinv));
                s1[2 * k + 1] = __dadd_rn(s1[2 * k + 1], mulmod_dd(e1, u64_to_d(kv[j][1].y), q, qinv));
            }
            // at most BETA + 1 products of 0.75 q on top of half a prime
            s0[2 * k] = reduce_d(s0[2 * k], q, qinv); s0[2 * k + 1] = reduce_d(s0[2 * k + 1], q, qinv);
            s1[2 * k] = reduce_d(s1[2 * k], q, qinv); s1[2 * k + 1] = reduce_d(s1[2 * k + 1], q, qinv);
            asm volatile("" ::: "memory");       // one step's words at a time: the registers hold no more
        }
        __syncwarp();
    }
    // what is added in place: P times a ciphertext (q-limbs), or the sum that u holds
    const u64 *add = a.has_add && x < a.level ? a.add.at(bz) + x * limb + p0 : nullptr;
    u64 *u = a.u + ((size_t)bz * 2 * nt + x) * limb + p0;
    const double *twi = c.twd_inv + ((size_t)kt << c.log_n);
#pragma unroll
    for (uint32_t cm = 0; cm < 2; cm++, u += nt * limb) {
        double (&v)[8] = cm ? s1 : s0;
        if (add || a.acc_u) {
            const u64 *o = add ? add + cm * a.level * limb : u;
            const double pq = add ? c.dn_p_mod_d[x] : 1.0;
#pragma unroll
            for (uint32_t k = 0; k < 4; k++) {
                const ulonglong2 z = ld_pair<true>(o + 64 * k);
                v[2 * k] = reduce_d(__dadd_rn(v[2 * k], mulmod_dd(u64_to_d(z.x), pq, q, qinv)), q, qinv);
                v[2 * k + 1] = reduce_d(__dadd_rn(v[2 * k + 1], mulmod_dd(u64_to_d(z.y), pq, q, qinv)), q, qinv);
            }
        }
        if (x < a.inv_from) {
#pragma unroll
            for (uint32_t k = 0; k < 4; k++) st_pair<true>(u + 64 * k, make_ulonglong2(canonical_d(v[2 * k], q), canonical_d(v[2 * k + 1], q)));
            continue;
        }
        double *s = sm[0][rl];
#pragma unroll
        for (uint32_t k = 0; k < 4; k++) *reinterpret_cast<double2 *>(s + wrow_at(2 * t) + 72 * k) = make_double2(v[2 * k], v[2 * k + 1]);
        __syncwarp();
        wrow_inverse(v, s, t, twi, R + row, q, qinv);
        double *g = reinterpret_cast<double *>(u) - t;
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) g[32 * k] = v[k];
        __syncwarp();
    }
}

}  // namespace

void launch_mid_rows(const ckks_ctx *c, const MidArgs &a, uint32_t beta, cudaStream_t s) {
    using K = decltype(&mid_rows<1, false>);
    static constexpr K one[IP_FUSED_BETA] = {mid_rows<1, false>, mid_rows<2, false>, mid_rows<3, false>, mid_rows<4, false>};
    static constexpr K terms[IP_FUSED_BETA] = {mid_rows<1, true>, mid_rows<2, true>, mid_rows<3, true>, mid_rows<4, true>};
    launch((a.nterm > 1 || a.c0[0] ? terms : one)[beta - 1], dim3((c->N >> 8) / MID_ROWS, a.nb, a.level + c->K), 32 * MID_ROWS, 0, s, c->dev, a);
}
