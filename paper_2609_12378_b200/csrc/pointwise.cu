// Pointwise (coefficient-wise) kernels on evaluation-domain limbs: ciphertext x
// plaintext multiply-accumulate, addition, tensor product.
// All are streaming kernels bound by HBM bandwidth: 128-bit loads and stores,
// one pass over each operand.
#include "common.cuh"

namespace {

constexpr uint32_t THREADS = 256;
constexpr uint32_t MAC_MAX = 32;   // ciphertexts per launch

struct MacArgs {
    const u64 *ct[MAC_MAX];
    u64 *acc[MAC_MAX];
};

// acc[s][c][i][k] (+)= ct[s][c][i][k] * pt[i][k]; one thread owns two adjacent coefficients of one (c, i).
template <bool INIT>
__global__ void __launch_bounds__(THREADS) mac_kernel(DevTables c, MacArgs a, uint32_t ncts, const u64 *pt, uint32_t level) {
    grid_dep_sync();
    const uint32_t half = c.N / 2;
    const uint32_t x = blockIdx.x * THREADS + threadIdx.x;   // pair index inside the limb
    const uint32_t limb = blockIdx.y, comp = blockIdx.z;
    if (x >= half) return;
    const u64 q = c.mod[limb], mu = c.mu[limb];
    const ulonglong2 p = reinterpret_cast<const ulonglong2 *>(pt + (size_t)limb * c.N)[x];
    const size_t off = ((size_t)comp * level + limb) * half + x;
    for (uint32_t s = 0; s < ncts; s++) {
        ulonglong2 v = reinterpret_cast<const ulonglong2 *>(a.ct[s])[off];
        ulonglong2 r;
        r.x = mul_mod(v.x, p.x, q, mu);
        r.y = mul_mod(v.y, p.y, q, mu);
        ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(a.acc[s]) + off;
        if (!INIT) {
            ulonglong2 o = *dst;
            r.x = add_mod(r.x, o.x, q);
            r.y = add_mod(r.y, o.y, q);
        }
        *dst = r;
    }
}

__global__ void __launch_bounds__(THREADS) add_kernel(DevTables c, const u64 *a, const u64 *b, u64 *out, uint32_t level) {
    grid_dep_sync();
    const uint32_t half = c.N / 2;
    const uint32_t x = blockIdx.x * THREADS + threadIdx.x;
    if (x >= half) return;
    const u64 q = c.mod[blockIdx.y % level];
    const size_t off = (size_t)blockIdx.y * half + x;
    ulonglong2 u = reinterpret_cast<const ulonglong2 *>(a)[off], v = reinterpret_cast<const ulonglong2 *>(b)[off];
    reinterpret_cast<ulonglong2 *>(out)[off] = make_ulonglong2(add_mod(u.x, v.x, q), add_mod(u.y, v.y, q));
}

// Operands enter the product kernels as 50-bit residues in doubles: a product is six FP64 instructions (mulmod_dd, |r| <= 0.75 q),
// where the integer pipe's 128-bit product and Barrett step cost about four times as much issue time.
template <bool WIDE>
__device__ __forceinline__ void pair_d(const u64 *p, double (&v)[2]) {
    const ulonglong2 w = ld_pair<WIDE>(p);
    v[0] = u64_to_d(w.x); v[1] = u64_to_d(w.y);
}
template <bool WIDE>
__device__ __forceinline__ void store_pair(u64 *p, const double (&v)[2], double q, double qinv) {
    st_pair<WIDE>(p, make_ulonglong2(canonical_d(reduce_d(v[0], q, qinv), q), canonical_d(reduce_d(v[1], q, qinv), q)));
}

// (a0 b0, a0 b1 + a1 b0) -> e01 [2][level][N];  a1 b1 -> e2 [level][N], for the products blockIdx.z; two coefficients per thread
template <bool WIDE>
__global__ void __launch_bounds__(THREADS) tensor_kernel(DevTables c, const __grid_constant__ TensorArgs t, uint32_t level) {
    const uint32_t k = (blockIdx.x * THREADS + threadIdx.x) * 2, limb = blockIdx.y, z = blockIdx.z;
    const double q = c.modd[limb].x, qinv = c.modd[limb].y;
    const size_t o = (size_t)limb * c.N + k;
    const CtView va = t.a[z], vb = t.b[z];
    grid_dep_sync();
    double a0[2], a1[2], b0[2], b1[2], r0[2], r1[2], r2[2];
    pair_d<WIDE>(va.p + o, a0); pair_d<WIDE>(va.p + va.comp + o, a1);
    pair_d<WIDE>(vb.p + o, b0); pair_d<WIDE>(vb.p + vb.comp + o, b1);
#pragma unroll
    for (uint32_t i = 0; i < 2; i++) {
        r0[i] = mulmod_dd(a0[i], b0[i], q, qinv);
        r1[i] = __dadd_rn(mulmod_dd(a0[i], b1[i], q, qinv), mulmod_dd(a1[i], b0[i], q, qinv));
        r2[i] = mulmod_dd(a1[i], b1[i], q, qinv);
    }
    store_pair<WIDE>(t.e01[z] + o, r0, q, qinv);
    store_pair<WIDE>(t.e01[z] + (size_t)level * c.N + o, r1, q, qinv);
    store_pair<WIDE>(t.e2[z] + o, r2, q, qinv);
}

// out = in * v (MUL) or in + v on component 0 (the constant polynomial v, a signed integer, has the value v mod q in
// every position of the evaluation domain); blockIdx.y = component * level + limb
template <bool MUL>
__global__ void __launch_bounds__(THREADS) const_kernel(DevTables c, const __grid_constant__ Ptrs inp, long long v, const __grid_constant__ Ptrs outp, uint32_t level) {
    grid_dep_sync();
    const uint32_t half = c.N / 2;
    const uint32_t x = blockIdx.x * THREADS + threadIdx.x;
    if (x >= half) return;
    const uint32_t limb = blockIdx.y % level;
    const u64 q = c.mod[limb], mu = c.mu[limb];
    const u64 m = (u64)(v < 0 ? -v : v) % q;
    u64 r = (v < 0 && m) ? q - m : m;
    if (!MUL && blockIdx.y >= level) r = 0;
    const size_t off = (size_t)blockIdx.y * half + x;
    const ulonglong2 u = reinterpret_cast<const ulonglong2 *>(inp.at(blockIdx.z))[off];
    reinterpret_cast<ulonglong2 *>(const_cast<u64 *>(outp.at(blockIdx.z)))[off] =
        MUL ? make_ulonglong2(mul_mod(u.x, r, q, mu), mul_mod(u.y, r, q, mu)) : make_ulonglong2(add_mod(u.x, r, q), add_mod(u.y, r, q));
}

// e[o] (+)= sum_{i < n} tensor(a_i, b[o]_i), n <= TS_MAX terms per launch, NO outputs that share the first operands.  Sums of
// products of size 0.75 q (1.5 q for the middle component) are reduced every four terms; one canonical step per component at the
// end, with the previous partial sum added unless INIT.  Bound by the operands' HBM traffic, which four outputs at a time cut to
// 5/8 of one at a time (the attention products: one query set against several key sets, the probabilities against every value
// channel).
template <bool INIT, bool WIDE, uint32_t NO>
__global__ void __launch_bounds__(THREADS) tensor_sum_kernel(DevTables c, const __grid_constant__ TensorSumArgs t, uint32_t n, uint32_t level) {
    const uint32_t k = (blockIdx.x * THREADS + threadIdx.x) * 2, limb = blockIdx.y;
    const double q = c.modd[limb].x, qinv = c.modd[limb].y;
    const size_t o0 = (size_t)limb * c.N + k, o1 = o0 + (size_t)level * c.N;
    grid_dep_sync();
    double s[NO][3][2];
#pragma unroll
    for (uint32_t o = 0; o < NO; o++)
        if (INIT) s[o][0][0] = s[o][0][1] = s[o][1][0] = s[o][1][1] = s[o][2][0] = s[o][2][1] = 0.0;
        else { pair_d<WIDE>(t.e01[o] + o0, s[o][0]); pair_d<WIDE>(t.e01[o] + o1, s[o][1]); pair_d<WIDE>(t.e2[o] + o0, s[o][2]); }
    for (uint32_t i = 0; i < n; i++) {
        double a0[2], a1[2], b0[NO][2], b1[NO][2];
        pair_d<WIDE>(t.a[i].p + o0, a0); pair_d<WIDE>(t.a[i].p + t.a[i].comp + o0, a1);
#pragma unroll
        for (uint32_t o = 0; o < NO; o++) { pair_d<WIDE>(t.b[o][i].p + o0, b0[o]); pair_d<WIDE>(t.b[o][i].p + t.b[o][i].comp + o0, b1[o]); }
#pragma unroll
        for (uint32_t o = 0; o < NO; o++)
#pragma unroll
            for (uint32_t j = 0; j < 2; j++) {
                s[o][0][j] = __dadd_rn(s[o][0][j], mulmod_dd(a0[j], b0[o][j], q, qinv));
                s[o][1][j] = __dadd_rn(s[o][1][j], __dadd_rn(mulmod_dd(a0[j], b1[o][j], q, qinv), mulmod_dd(a1[j], b0[o][j], q, qinv)));
                s[o][2][j] = __dadd_rn(s[o][2][j], mulmod_dd(a1[j], b1[o][j], q, qinv));
                if ((i & 3) == 3)
#pragma unroll
                    for (uint32_t m = 0; m < 3; m++) s[o][m][j] = reduce_d(s[o][m][j], q, qinv);
            }
    }
#pragma unroll
    for (uint32_t o = 0; o < NO; o++) {
        store_pair<WIDE>(t.e01[o] + o0, s[o][0], q, qinv);
        store_pair<WIDE>(t.e01[o] + o1, s[o][1], q, qinv);
        store_pair<WIDE>(t.e2[o] + o0, s[o][2], q, qinv);
    }
}

// out[o] (+)= sum_j v[o][j] x[j] for up to LIN_MAX inputs and outputs of the ciphertexts blockIdx.z / 2 (component blockIdx.z & 1),
// constants as signed integers; cst[o] q_{level-1} is added to the first component (so that a rescale turns it into the
// constant cst[o]).  The inputs are read once for all outputs; the constants' residues modulo this limb's prime are formed
// once per CTA.
template <bool WIDE>
__global__ void __launch_bounds__(THREADS) lincomb_kernel(DevTables c, const __grid_constant__ LinArgs t, uint32_t level) {
    __shared__ double s_v[LIN_MAX][LIN_MAX + 1];
    const uint32_t k = (blockIdx.x * THREADS + threadIdx.x) * 2, limb = blockIdx.y, comp = blockIdx.z & 1, z = blockIdx.z >> 1;
    const double q = c.modd[limb].x, qinv = c.modd[limb].y;
    for (uint32_t e = threadIdx.x; e < t.no * (LIN_MAX + 1); e += THREADS) {
        const uint32_t o = e / (LIN_MAX + 1), j = e % (LIN_MAX + 1);
        const long long v = j < LIN_MAX ? t.v[o][j] : t.cst[o];
        const u64 m = c.mod[limb], r = (u64)(v < 0 ? -v : v) % m;
        double d = v < 0 ? -(double)r : (double)r;
        if (j == LIN_MAX) d = comp || limb + 1 == level ? 0.0 : mulmod_dd(d, (double)(c.mod[level - 1] % m), q, qinv);
        s_v[o][j] = d;
    }
    grid_dep_sync();
    const size_t off = (size_t)limb * c.N + k, oo = (size_t)comp * level * c.N + off;
    ulonglong2 x[LIN_MAX];
#pragma unroll
    for (uint32_t j = 0; j < LIN_MAX; j++)
        if (j < t.nx) x[j] = ld_pair<WIDE>(t.x[j].at(z) + comp * t.xc[j] + off);
    __syncthreads();
    for (uint32_t o = 0; o < t.no; o++) {
        u64 *dst = const_cast<u64 *>(t.out[o].at(z)) + oo;
        double r[2] = {s_v[o][LIN_MAX], s_v[o][LIN_MAX]};
        if (t.accumulate) {
            double old[2];
            pair_d<WIDE>(dst, old);
            r[0] = __dadd_rn(r[0], old[0]); r[1] = __dadd_rn(r[1], old[1]);
        }
        // |sum| <= (0.75 + 1) q + LIN_MAX / 2 * 0.75 q, twice with a reduction between: below 8 q
#pragma unroll
        for (uint32_t j = 0; j < LIN_MAX; j++) {
            if (j < t.nx) {
                r[0] = __dadd_rn(r[0], mulmod_dd(u64_to_d(x[j].x), s_v[o][j], q, qinv));
                r[1] = __dadd_rn(r[1], mulmod_dd(u64_to_d(x[j].y), s_v[o][j], q, qinv));
            }
            if (j == LIN_MAX / 2 - 1) { r[0] = reduce_d(r[0], q, qinv); r[1] = reduce_d(r[1], q, qinv); }
        }
        store_pair<WIDE>(dst, r, q, qinv);
    }
}

}  // namespace

// out[x] = 1.0 where lo <= x / B < hi and t0 <= x % Ti < t1, else 0.0 (slot masks of the attention layout's conversions)
__global__ void __launch_bounds__(THREADS) slot_mask_kernel(double *out, uint32_t n, uint32_t B, uint32_t lo, uint32_t hi, uint32_t Ti, uint32_t t0,
                                                            uint32_t t1) {
    grid_dep_sync();
    const uint32_t x = blockIdx.x * THREADS + threadIdx.x;
    if (x >= n) return;
    const uint32_t blk = x / B, t = x % Ti;
    out[x] = (blk >= lo && blk < hi && t >= t0 && t < t1) ? 1.0 : 0.0;
}

void launch_slot_mask(const ckks_ctx *c, double *out, uint32_t B, uint32_t lo, uint32_t hi, uint32_t Ti, uint32_t t0, uint32_t t1, cudaStream_t s) {
    launch(slot_mask_kernel, (c->n + THREADS - 1) / THREADS, THREADS, 0, s, out, c->n, B, lo, hi, Ti, t0, t1);
}

void launch_const(const ckks_ctx *c, const Ptrs &in, long long v, bool mul, const Ptrs &out, uint32_t ncomp, uint32_t level, cudaStream_t s, uint32_t n) {
    dim3 grid((c->N / 2 + THREADS - 1) / THREADS, ncomp * level, n);
    if (mul) launch(const_kernel<true>, grid, THREADS, 0, s, c->dev, in, v, out, level);
    else launch(const_kernel<false>, grid, THREADS, 0, s, c->dev, in, v, out, level);
}

template <uint32_t NO>
static void tensor_sum(const ckks_ctx *c, const CtView *a, const CtView *const *b, uint32_t n, u64 *const *e01, u64 *const *e2, uint32_t level, cudaStream_t s) {
    const dim3 grid(c->N / (2 * THREADS), level);
    for (uint32_t i0 = 0; i0 < n; i0 += TS_MAX) {
        TensorSumArgs args;
        const uint32_t m = std::min(TS_MAX, n - i0);
        bool wide = true;
        for (uint32_t i = 0; i < m; i++) { args.a[i] = a[i0 + i]; wide = wide && aligned16(args.a[i]); }
        for (uint32_t o = 0; o < NO; o++) {
            args.e01[o] = e01[o]; args.e2[o] = e2[o];
            wide = wide && aligned16(e01[o]) && aligned16(e2[o]);
            for (uint32_t i = 0; i < m; i++) { args.b[o][i] = b[o][i0 + i]; wide = wide && aligned16(args.b[o][i]); }
        }
        auto *k = i0 == 0 ? (wide ? tensor_sum_kernel<true, true, NO> : tensor_sum_kernel<true, false, NO>)
                          : (wide ? tensor_sum_kernel<false, true, NO> : tensor_sum_kernel<false, false, NO>);
        launch(k, grid, THREADS, 0, s, c->dev, args, m, level);
    }
}

void launch_tensor_sum(const ckks_ctx *c, const CtView *a, const CtView *const *b, uint32_t n, u64 *const *e01, u64 *const *e2, uint32_t no, uint32_t level,
                       cudaStream_t s) {
    for (; no >= 4; no -= 4, b += 4, e01 += 4, e2 += 4) tensor_sum<4>(c, a, b, n, e01, e2, level, s);
    if (no >= 2) { tensor_sum<2>(c, a, b, n, e01, e2, level, s); no -= 2; b += 2; e01 += 2; e2 += 2; }
    if (no) tensor_sum<1>(c, a, b, n, e01, e2, level, s);
}

void launch_lincomb(const ckks_ctx *c, const LinArgs &args, uint32_t n, uint32_t level, cudaStream_t s) {
    bool wide = true;
    for (uint32_t j = 0; j < args.nx; j++) wide = wide && aligned16(args.x[j]) && (args.xc[j] & 1) == 0;
    for (uint32_t o = 0; o < args.no; o++) wide = wide && aligned16(args.out[o]);
    launch(wide ? lincomb_kernel<true> : lincomb_kernel<false>, dim3(c->N / (2 * THREADS), level, 2 * n), THREADS, 0, s, c->dev, args, level);
}

void launch_mul_plain_acc(const ckks_ctx *c, const u64 *const *cts, u64 *const *accs, uint32_t ncts, const u64 *pt,
                          uint32_t level, bool init, cudaStream_t s) {
    dim3 grid((c->N / 2 + THREADS - 1) / THREADS, level, 2);
    for (uint32_t s0 = 0; s0 < ncts; s0 += MAC_MAX) {
        MacArgs a;
        uint32_t n = ncts - s0 < MAC_MAX ? ncts - s0 : MAC_MAX;
        for (uint32_t i = 0; i < n; i++) { a.ct[i] = cts[s0 + i]; a.acc[i] = accs[s0 + i]; }
        launch(init ? mac_kernel<true> : mac_kernel<false>, grid, THREADS, 0, s, c->dev, a, n, pt, level);
    }
}

void launch_add(const ckks_ctx *c, const u64 *a, const u64 *b, u64 *out, uint32_t ncomp, uint32_t level, cudaStream_t s) {
    dim3 grid((c->N / 2 + THREADS - 1) / THREADS, ncomp * level);
    launch(add_kernel, grid, THREADS, 0, s, c->dev, a, b, out, level);
}

void launch_tensor(const ckks_ctx *c, const TensorArgs &args, uint32_t n, uint32_t level, cudaStream_t s) {
    bool wide = true;
    for (uint32_t i = 0; i < n; i++) wide = wide && aligned16(args.a[i]) && aligned16(args.b[i]) && aligned16(args.e01[i]) && aligned16(args.e2[i]);
    launch(wide ? tensor_kernel<true> : tensor_kernel<false>, dim3(c->N / (2 * THREADS), level, n), THREADS, 0, s, c->dev, args, level);
}
