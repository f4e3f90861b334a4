// Shared declarations of the ckks_b200 library: context, device tables,
// modular arithmetic for 50-bit primes, kernel launch entry points.
#pragma once
#include <algorithm>

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/ckks_b200.h"

typedef unsigned long long u64;
typedef unsigned __int128 u128;

// ---------------------------------------------------------------------------
// Device-side view of the context tables (plain pointers, passed by value).
// Prime index space t: 0..L-1 = q_i, L..L+K-1 = p_k.
// ---------------------------------------------------------------------------
struct DevTables {
    uint32_t log_n, N, L, K, alpha, T, dnum;
    const u64 *mod;          // [T]
    const u64 *mu;           // [T] floor(2^112 / prime)
    const u64 *mu64;         // [T] floor(2^64 / prime)
    const double2 *modd;     // [T] {prime, 1/prime} as doubles
    const ulonglong2 *tw_fwd;  // [T][N] {psi^bitrev(i), Shoup companion}, index m+i (integer transform: N = 2^16 only)
    const ulonglong2 *tw_inv;  // [T][N] inverses of the same
    const ulonglong2 *n_inv;   // [T] {N^-1, Shoup}
    // fp64 tables of the transform: the centred representative of w as a double, same
    // indexing (the transform estimates a product's quotient from the rounded product and 1/q, so the table holds w alone)
    const double *twd_fwd, *twd_inv;    // [T][N]
    const double2 *n_inv_d;             // [T][2] {N^-1, N^-1/q}, {w N^-1, that/q} for the inverse's last twiddle w, all centred
    // inverse-transform scalings that deliver the basis conversions' first factor y = [d qhat^-1], pairs
    // {N^-1 qhat^-1, last inverse twiddle times that}, each {v, v / prime} centred
    const double2 *inv_scale_up;   // [(L+1)][L][2]   ModUp: level, limb
    const double2 *inv_scale_dn;   // [K][2]          ModDown: special limb
    const double2 *inv_scale_rs;   // [L][1 + K][2]   ModDown with rescale: dropped limb (N^-1 alone), then the special limbs
    // ModUp, per level l (1..L), digit j, source a < alpha:
    const ulonglong2 *up_hat_inv;  // [(L+1)][dnum][alpha]        {qhat^-1 mod q_src, Shoup}
    const double *up_hat_mod_d;    // [(L+1)][dnum][T][alpha]     centred qhat mod target
    // ModDown:
    const ulonglong2 *dn_hat_inv;  // [K]      {Phat_k^-1 mod p_k, Shoup}
    const double *dn_hat_mod_d;    // [L][K]   centred Phat_k mod q_i
    const double2 *dn_p_inv_d;     // [L]      {P^-1 mod q_i, that / q_i} as doubles
    const double *dn_p_mod_d;      // [L]      P mod q_i as a double
    // Tensor-core basis conversion (conv_mma.cu; conv_groups = 0 when alpha or K exceeds 8 sources): byte matrices of
    // the conversion constants in the B-fragment order of mma.m16n8k32, [group of 8 targets][13 diagonals][2 k-steps]
    // [lane][2] words; targets are the non-own limbs of the digit in ascending order (ModUp) or q_0.. (ModDown)
    const uint32_t *up_bmat;       // [(L+1)][dnum][conv_groups][13][2][64]
    const uint32_t *dn_bmat;       // [conv_groups][13][2][64]
    const double2 *two52_d;        // [T] {2^52 mod prime, that / prime}
    uint32_t conv_groups;
    // Rescale:
    const double2 *rs_inv_d;       // [L(last)][L(i)] {q_last^-1 mod q_i, that / q_i} as doubles
    const double2 *rs_p_inv_d;     // [L(last)][L(i)] {(q_last P)^-1 mod q_i, that / q_i}
    // Encode:
    const uint32_t *enc_src;       // [n] slot index feeding FFT input position pos (bit-reversed e_j)
    const double2 *enc_omega;      // [n] exp(2 pi i t / n)
    const double2 *enc_omega_st;   // [min(n, 1024)] the same values stage by stage: entry half + j = omega^(j n / (2 half)), half = 1, 2, .. (entry 0 unused)
    const double2 *enc_omega_st2;  // [n] second-pass twiddles by stage and row: entry (hr + jr) * ch + col = omega^((jr ch + col) n / (2 hr ch)), ch = min(n, 1024)
    const double2 *enc_zeta;       // [n] exp(2 pi i k / 2N)
    int *range_flag;               // [0] sticky encode overflow flag, [1] sticky device-side wait timeout flag
};

struct ckks_ctx {
    uint32_t log_n, N, n, L, K, dnum, alpha, T;
    int device, sms;
    std::vector<u64> mod;        // host copy of the primes
    std::vector<u64> pow5;       // 5^j mod 2N, j < n (host)
    DevTables dev;               // pointers into `allocs`
    std::vector<void *> allocs;  // device allocations owned by the context
    std::string cuda_error;
    // options (ckks_context_set_option); host-side state read when a call is made
    uint32_t ntt_fp_share = 8;               // of every 8 limbs, how many take the double-precision NTT path
    int ntt_bulk_store = 1;                  // kept for get and set; selects nothing
    int conv_kernel = 0;                     // basis conversions: 0 = FP64 pipe, 1 = tensor cores (conv_mma.cu)
    int mac_kernel = 82;                     // projection multiply-accumulate kernel (see launch_mac_mma)
    bool strips = false;                     // conversions may run in strips (conv_strip_prepare)
    long long wait_cycles = 2000000000ll;    // clock bound of every device-side wait (about a second)
    // Streams of the context.  ckks_attention_pack, whose work is many independent single-ciphertext chains, spreads them over
    // `lanes` streams, lane 0 being the caller's: a single ciphertext's kernels fill the GPU for at most one wave, so
    // independent chains overlap.  Forked from and joined to the caller's stream by events.
    int lanes = 4;
    cudaStream_t lane_stream[3] = {nullptr, nullptr, nullptr};
    cudaEvent_t lane_event[4] = {nullptr, nullptr, nullptr, nullptr};
};

// The context's streams as lanes for independent chains: lane 0 is the caller's stream.  fork() makes the other lanes wait
// for what the caller's stream has been given so far, join() makes the caller's stream wait for all of them.
struct Lanes {
    ckks_ctx *c;
    cudaStream_t caller;
    uint32_t n;
    Lanes(ckks_ctx *ctx, void *stream) : c(ctx), caller((cudaStream_t)stream), n((uint32_t)std::max(1, std::min(ctx->lanes, 4))) {}
    void *at(uint32_t i) const { return i % n == 0 ? (void *)caller : (void *)c->lane_stream[i % n - 1]; }
    void fork() const {
        if (n == 1) return;
        int prev = 0;
        cudaGetDevice(&prev);
        cudaSetDevice(c->device);
        cudaEventRecord(c->lane_event[0], caller);
        for (uint32_t i = 1; i < n; i++) cudaStreamWaitEvent(c->lane_stream[i - 1], c->lane_event[0], 0);
        cudaSetDevice(prev);
    }
    void join() const {
        if (n == 1) return;
        int prev = 0;
        cudaGetDevice(&prev);
        cudaSetDevice(c->device);
        for (uint32_t i = 1; i < n; i++) {
            cudaEventRecord(c->lane_event[i], c->lane_stream[i - 1]);
            cudaStreamWaitEvent(caller, c->lane_event[i], 0);
        }
        cudaSetDevice(prev);
    }
};
inline uint32_t lane_count(const ckks_ctx *c) { return (uint32_t)std::max(1, std::min(c->lanes, 4)); }

// ---------------------------------------------------------------------------
// "Tiled" operand layout of the projection's multiply-accumulate.  R rows (one row = one plaintext, or one
// component of one ciphertext) of [level][N] words are stored so that, for a limb i and a block of 64
// coefficients, all R rows are adjacent:   index(r, i, p) = (((i * N/64) + p/64) * R + r) * 64 + p % 64.
// The multiply-accumulate walks all rows of a few coefficients; in the plain [row][level][N] layout those
// words are 12-24 MiB apart (one TLB entry and one DRAM page per 64 bytes), here they are one 512-byte step apart.
// ---------------------------------------------------------------------------
__host__ __device__ inline size_t tiled_index(uint32_t R, uint32_t N, uint32_t r, uint32_t i, uint32_t p) {
    return ((((size_t)i * (N >> 6)) + (p >> 6)) * R + r) * 64 + (p & 63);
}
// where a key-switch result goes when it is written straight into a tiled buffer: component c of batch entry b
// becomes row row0 + b * row_stride + c of a buffer with R rows (R = 0: plain layout)
struct TiledOut { uint32_t R = 0, row0 = 0, row_stride = 0; };

// ---------------------------------------------------------------------------
// Limb addressing for batched limb-wise kernels (NTT): limb y of a buffer
// [..][period][N] -> prime index, or -1 to skip the limb.
//   kind 0: prime = first + y % period
//   kind 1: "extended" layout [batch][digit][level + K]: x = y % period is q_x for
//           x < level, else p_{x-level}; with skip_own the digit's own limbs
//           (which never leave the evaluation domain) are skipped.
// ---------------------------------------------------------------------------
struct LimbMap {      // kind 2: prime = first for every limb
    uint32_t kind, first, period, pitch, level, L, alpha, nbeta, skip_own;
};
// limbs [..][period][N] contiguous, limb x of every period under prime first + x
inline LimbMap plain_map(uint32_t first, uint32_t period) { return LimbMap{0, first, period, period, 0, 0, 0, 1, 0}; }
// same, but consecutive periods start `pitch` limbs apart (a sub-range of limbs of a larger array)
inline LimbMap pitched_map(uint32_t first, uint32_t period, uint32_t pitch) { return LimbMap{0, first, period, pitch, 0, 0, 0, 1, 0}; }
// limbs [..][period][N], all under one prime
inline LimbMap same_map(uint32_t prime, uint32_t period) { return LimbMap{2, prime, period, period, 0, 0, 0, 1, 0}; }
// extended digits [batch][beta][level + K]
inline LimbMap ext_map(uint32_t level, uint32_t K, uint32_t L, uint32_t alpha, uint32_t beta) {
    return LimbMap{1, 0, level + K, level + K, level, L, alpha, beta, 1};
}
// limbs first .. level + K - 1 of every polynomial of the extended basis, polynomials level + K limbs apart
inline LimbMap tail_map(uint32_t first, uint32_t level, uint32_t K, uint32_t L) { return LimbMap{1, first, level + K - first, level + K, level, L, 0, 1, 0}; }

__host__ __device__ inline int limb_prime(const LimbMap &m, uint32_t y) {
    uint32_t x = y % m.period;
    if (m.kind == 0) return (int)(m.first + x);
    if (m.kind == 2) return (int)m.first;
    if (m.skip_own) {
        uint32_t j = (y / m.period) % m.nbeta, lo = j * m.alpha, hi = lo + m.alpha < m.level ? lo + m.alpha : m.level;
        if (x >= lo && x < hi) return -1;
    }
    x += m.first;
    return x < m.level ? (int)x : (int)(m.L + (x - m.level));
}
// index (in limbs) of limb y from the base pointer
__host__ __device__ inline size_t limb_index(const LimbMap &m, uint32_t y) { return (size_t)(y / m.period) * m.pitch + y % m.period; }

// ---------------------------------------------------------------------------
// Modular arithmetic, primes in (2^49, 2^50).
// ---------------------------------------------------------------------------

// x * w mod q for a constant w with companion wp = floor(w 2^64 / q); result in [0, 2q) for ANY 64-bit x.
__device__ __forceinline__ u64 mul_shoup_lazy(u64 x, u64 w, u64 wp, u64 q) {
    return x * w - __umul64hi(x, wp) * q;
}
__device__ __forceinline__ u64 mul_shoup(u64 x, u64 w, u64 wp, u64 q) {
    u64 r = mul_shoup_lazy(x, w, wp, q);
    return r >= q ? r - q : r;
}
__device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) { u64 s = a + b; return s >= q ? s - q : s; }
__device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

// (hi:lo) mod q for a value below 2^112; mu = floor(2^112 / q).
// qhat = floor((x >> 48) mu / 2^64) is in (x/q - 2, x/q], so one conditional subtraction finishes.
__device__ __forceinline__ u64 barrett112(u64 hi, u64 lo, u64 q, u64 mu) {
    u64 xh = (hi << 16) | (lo >> 48);
    u64 qhat = __umul64hi(xh, mu);
    u64 r = lo - qhat * q;
    return r >= q ? r - q : r;
}
__device__ __forceinline__ u64 mul_mod(u64 a, u64 b, u64 q, u64 mu) {
    return barrett112(__umul64hi(a, b), a * b, q, mu);
}
// 128-bit lazy accumulator: acc += a * b
__device__ __forceinline__ void mac128(u64 &hi, u64 &lo, u64 a, u64 b) {
    u64 pl = a * b, ph = __umul64hi(a, b);
    lo += pl;
    hi += ph + (lo < pl);
}
// Representative of the centred lift of y (mod src) taken modulo dst, for primes of equal bit length:
// y <= (src-1)/2 stays, else y - src + dst (positive because dst > src/2).
__device__ __forceinline__ u64 centred_to(u64 y, u64 src, u64 dst) {
    return y > (src >> 1) ? y + dst - src : y;
}

// ---------------------------------------------------------------------------
// Double-precision modular arithmetic for 50-bit primes (FP64 pipe).  Values are
// signed integers held in doubles, exact while below 2^53 in magnitude.
//   mulmod_d: y * w - k q with k = round(y * (w/q)); exact; |result| <= (1/2 + |y| 2^-53) q
//             (COARSE: k rounded to even, valid for |y w / q| < 2^52, |result| <= (1 + ..) q).
// ---------------------------------------------------------------------------
constexpr double MAGIC0 = 6755399441055744.0;    // 1.5 * 2^52: rounds |v| < 2^51 to the nearest integer
constexpr double MAGIC1 = 13510798882111488.0;   // 1.5 * 2^53: rounds |v| < 2^52 to the nearest even integer
constexpr double TWO52 = 4503599627370496.0;
// Basis conversions: out[t] = sum_a y_a C[a][t] mod t with centred sources |y_a| <= q_a / 2 and centred constants |C| <= t / 2 (a dense
// contraction, bound by the FP64 pipe).  The exact 100-bit products of up to eight sources are summed as they are:
//   H' = fma(y, C, H) starting from H = 1.5 * 2^102 rounds the running sum to multiples of 2^50 (|sum| <= 8 * 2^98 =
//   2^101 keeps H inside [2^102, 2^103)); h = H' - H is exact, l = fma(y, C, -h) is the exact rest, |l| <= 2^49,
// so the sum is (H - 1.5 * 2^102) + sum l, four instructions per (source, target) pair where a reduction of every product took seven.
// The high part is below 2 q t, its quotient by t below 2^51; the low parts are at most 8 * 2^49.
constexpr double CONV_SIGMA = 0x1.8p+102;

template <int COARSE>
__device__ __forceinline__ double mulmod_d(double y, double2 w, double q) {
    const double p = __dmul_rn(y, w.x);
    const double e = __fma_rn(y, w.x, -p);
    const double M = COARSE ? MAGIC1 : MAGIC0;
    const double k = __dsub_rn(__fma_rn(y, w.y, M), M);
    return __dadd_rn(__fma_rn(-k, q, p), e);
}
// The same with the quotient estimated from the rounded product, k = round(p * (1/q)): p and 1/q are each within 2^-53
// relative, so the estimate is as close as with a precomputed w * (1/q), and no per-twiddle multiply is needed.
template <int COARSE>
__device__ __forceinline__ double mulmod_pq(double y, double w, double q, double qinv) {
    const double p = __dmul_rn(y, w);
    const double e = __fma_rn(y, w, -p);
    const double M = COARSE ? MAGIC1 : MAGIC0;
    const double k = __dsub_rn(__fma_rn(p, qinv, M), M);
    return __dadd_rn(__fma_rn(-k, q, p), e);
}
// x * y - k q for two variable residues 0 <= x, y < q (as doubles): exact, |result| <= 0.75 q
__device__ __forceinline__ double mulmod_dd(double x, double y, double q, double qinv) {
    const double p = __dmul_rn(x, y);
    const double e = __fma_rn(x, y, -p);
    const double k = __dsub_rn(__fma_rn(p, qinv, MAGIC0), MAGIC0);
    return __dadd_rn(__fma_rn(-k, q, p), e);
}
__device__ __forceinline__ double reduce_d(double v, double q, double qinv) {   // to |v| <= q/2
    const double k = __dsub_rn(__fma_rn(v, qinv, MAGIC0), MAGIC0);
    return __fma_rn(-k, q, v);
}
__device__ __forceinline__ double u64_to_d(u64 x) { return __dsub_rn(__longlong_as_double((long long)(x | 0x4330000000000000ull)), TWO52); }
__device__ __forceinline__ u64 d_to_u64(double v) { return (u64)__double_as_longlong(__dadd_rn(v, TWO52)) & 0x000FFFFFFFFFFFFFull; }
__device__ __forceinline__ u64 canonical_d(double v, double q) { return d_to_u64(v < 0.0 ? __dadd_rn(v, q) : v); }

__device__ __forceinline__ uint32_t bitrev_n(uint32_t x, uint32_t bits) { return __brev(x) >> (32 - bits); }
// index p' with stored[p] of sigma_g(a) = stored[p'] of a (evaluation domain, bit-reversed); g = 1: identity.  The exponents
// live modulo 2N <= 2^17, so 32-bit products do.
__device__ __forceinline__ uint32_t galois_src(uint32_t p, uint32_t g, uint32_t log_n) {
    if (g == 1) return p;
    const uint32_t e = g * (2 * bitrev_n(p, log_n) + 1);
    return bitrev_n((e >> 1) & ((1u << log_n) - 1), log_n);
}
// centred representative of a canonical residue
__device__ __forceinline__ double centre_d(u64 v, u64 q) { return v > (q >> 1) ? __dsub_rn(u64_to_d(v), (double)q) : u64_to_d(v); }

// Kernel launches issued by this library since it was loaded (all contexts, all streams).
extern unsigned long long g_kernel_launches;
inline void count_launches(unsigned n = 1) { g_kernel_launches += n; }

// Launches are programmatic dependent launches: a kernel's CTAs may become resident as soon as every CTA of the kernel before
// it on the stream has exited, and grid_dep_sync waits until that kernel's writes are visible.  Until then a kernel may only
// read the context's tables.  Between dependent kernels of a few microseconds this hides the launch latency and the table
// fetches (a rotation of one ciphertext, 11 launches at the time, nine now: 208 -> 186 us).  No kernel triggers its dependents earlier: CTAs that
// wait for the last wave of a large launch take the slots and the issue cycles it needs (64 hoisted rotations 1 % slower,
// the 4096 x 4096 projection 3 %; for grids of at most one wave alone, one rotation 156 -> 160 us).
__device__ __forceinline__ void grid_dep_sync() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
template <class... P, class... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    count_launches();
}

// the same for a kernel of clusters of `cl` CTAs along x
template <class... P, class... A>
inline void launch_clusters(void (*kernel)(P...), uint32_t cl, dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cl; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    count_launches();
}

// ---------------------------------------------------------------------------
// Internal launchers (each validates nothing; the C ABI layer does).
// ---------------------------------------------------------------------------
// Up to KS_MULTI key switches that share one set of extended digits but differ in key, Galois element and output
// buffer (hoisted rotations): batch entry b uses evk[b], galois[b], out[b].
constexpr uint32_t KS_MULTI = 16;
struct KsMulti {
    const u64 *evk[KS_MULTI];
    u64 galois[KS_MULTI];
    u64 *out[KS_MULTI];
    // group > 0: `group` ciphertexts with their own digits take every one of the keys; batch entry b = r * group + m is key r
    // applied to member m's digits, added to member m's addend, and written to the tiled row
    // row0 + r * rot_rows + m * row_stride + component, or (plain layout) to out + r * rot_stride + m * out_stride words
    // (out[] is not used); own != 0: entry b has digits and an addend of its own instead of member m's
    uint32_t group, own, rot_rows;
    size_t rot_stride;
};

// Batch entries of a buffer: entry b at base + b * stride words, or (n > 0) at p[b]
struct Ptrs {
    const u64 *base = nullptr;
    size_t stride = 0;
    uint32_t n = 0;
    const u64 *p[KS_MULTI] = {};
    Ptrs() = default;
    __host__ __device__ Ptrs(const u64 *b, size_t s) : base(b), stride(s) {}
    __host__ __device__ const u64 *at(uint32_t b) const { return n ? p[b] : base + b * stride; }
};

// Two adjacent words with one 16-byte access (WIDE) or two 8-byte ones: kernels come in both forms, chosen by aligned16 on the
// host, because callers' buffers need only be 8-byte aligned.
template <bool WIDE>
__device__ __forceinline__ ulonglong2 ld_pair(const u64 *p) {
    return WIDE ? *reinterpret_cast<const ulonglong2 *>(p) : make_ulonglong2(p[0], p[1]);
}
template <bool WIDE>
__device__ __forceinline__ void st_pair(u64 *p, ulonglong2 v) {
    if (WIDE) *reinterpret_cast<ulonglong2 *>(p) = v;
    else { p[0] = v.x; p[1] = v.y; }
}
inline bool aligned16(const void *p) { return ((uintptr_t)p & 15) == 0; }
inline bool aligned16(const Ptrs &p) {
    if (!p.n) return aligned16(p.base) && (p.stride & 1) == 0;
    for (uint32_t i = 0; i < p.n; i++)
        if (!aligned16(p.p[i])) return false;
    return true;
}

// Epilogue of the forward transform, for a buffer of limbs laid out [b][ncomp][level].
//   mode 1: instead of storing NTT(conv) the last pass finishes a ModDown or a rescale:
//           out[b][comp][i][p] = (u[b][comp][i][p] - NTT(conv)[p]) pinv[i] + sigma_g(add[b][comp][i])[p] + acc[b][comp][i][p]
//           u: [ncomp][nt][N] words per entry; add: [..][level][N] words, taken for the components in the mask add_comps;
//           acc (if given): [ncomp][level][N] words per entry;
//           out: plain ([ncomp][level][N] per entry) or tiled (tl.R != 0, component comp of entry b in row
//           tl.row0 + b * tl.row_stride + comp)
//   mode 3: as mode 1, but the sum u is not read: it is formed here, u = <digits, key>.  Digits are read through sigma_galois
//           as well; beta <= IP_FUSED_BETA of them (inverse: the input is not read but formed as u, for the special limbs; the
//           map's periods are the entries' components)
//   mode 2: the transform's own result is stored, but into a tiled buffer (out.base): limb y = b * level + i becomes row
//           tl.row0 + b * tl.row_stride, limb i
constexpr uint32_t IP_FUSED_BETA = 4;
struct NttEpilogue {
    int mode;
    Ptrs u, add, out, acc;
    const double2 *pinv;   // [level] {constant, constant / q_i}
    uint32_t add_comps, ncomp, level, nt;
    u64 galois;
    int accumulate;        // acc is given
    TiledOut tl;
    int multi;             // batch entry b adds through mgalois[b]
    u64 mgalois[KS_MULTI];
    // KsMulti's grouped form: entry b = r * group + m takes mgalois[r] and add.at(m) and goes to row
    // tl.row0 + r * rot_rows + m * tl.row_stride + comp, or to out.base + r * rot_stride + m * out.stride
    uint32_t group, own, rot_rows;
    size_t rot_stride;
    // mode 3: extended digits [member][beta][nt][N] and the digits' own limbs (not grouped: one member's), a key per rotation, the batch
    const u64 *ext, *mevk[KS_MULTI];
    Ptrs d;
    uint32_t beta, nb;
    uint32_t y0;           // (filled in) first limb of the launch
};
// Prologue of the forward transform: the first pass reads one buffer [batch][N] (batch = limb index / map.period) instead of
// `base`: signed 64-bit coefficients, or (lift) residues modulo prime src_prime whose centred representatives are meant.
// doubles: the buffer itself, which holds signed doubles of at most half a prime (the conversions' output).
struct NttPrologue {
    const u64 *src = nullptr;
    bool lift = false;
    uint32_t src_prime = 0;
    bool doubles = false;
};
// Source of the inverse transform: the first pass reads limb x of entry b at ptr.at(b) + x * lpitch limbs, so the transform
// runs out of place and the input stays as it is (b = limb index / map.period, x = limb index % map.period).
struct NttSource {
    Ptrs ptr;
    uint32_t lpitch = 0;
};
// alone: the chain of launches belongs to a short call of its own, which for a small ring the host bounds: fewest launches.
// inv_scale (inverse): pairs [map.period][2] that replace {N^-1, last twiddle N^-1} for limb x of every period (device
// pointer), so that the output is scaled by a per-limb constant.
void launch_ntt(const ckks_ctx *c, u64 *base, uint32_t nlimbs_total, const LimbMap &map, bool inverse, cudaStream_t s,
                const NttEpilogue *ep = nullptr, const NttPrologue *pro = nullptr, const NttSource *src = nullptr, const double2 *inv_scale = nullptr, bool alone = false);
// One of the two passes alone, or both; limbs are signed doubles between the passes
enum NttPart { NTT_ROWS = 1, NTT_COLS = 2, NTT_BOTH = 3 };
void launch_ntt_part(const ckks_ctx *c, NttPart part, u64 *base, uint32_t nlimbs_total, const LimbMap &map, bool inverse, cudaStream_t s, const NttEpilogue *ep = nullptr,
                     const NttPrologue *pro = nullptr, const NttSource *src = nullptr, const double2 *inv_scale = nullptr);
// What lies between an inverse and a forward row pass (conv_ntt.cu): the sources' inverse column pass, a basis conversion, the targets'
// forward column pass.  CONV_UP: ModUp of one digit (an item: entry * digits + digit; src [entry][level], dst [item][level + K]);
// CONV_DOWN: ModDown of one component (item: entry * 2 + component; src [item][level + K], dst [item][targets]);
// CONV_DOWN_RS: that of a ModDown which a rescale follows.
enum { CONV_UP = 0, CONV_DOWN = 1, CONV_DOWN_RS = 2 };
// Once per context: whether it can run, i.e. the ring has an instance, and the compiler gave the kernels the registers that their roles
// share out (with fewer they would wait for ones that nobody gives back).  Without it the conversions take their separate kernels.
bool conv_strip_prepare(const ckks_ctx *c);
bool conv_strip(const ckks_ctx *c, int mode, uint32_t level, uint32_t items, bool alone = false);     // alone: see launch_ntt
void launch_conv_strip(const ckks_ctx *c, int mode, const u64 *src, u64 *dst, uint32_t level, uint32_t items, cudaStream_t s);
void launch_ntt_int(const ckks_ctx *c, u64 *b, uint32_t ny, const LimbMap &map, bool inverse, const NttSource &src, cudaStream_t s);

void launch_mul_plain_acc(const ckks_ctx *c, const u64 *const *cts, u64 *const *accs, uint32_t ncts, const u64 *pt,
                          uint32_t level, bool init, cudaStream_t s);
void launch_add(const ckks_ctx *c, const u64 *a, const u64 *b, u64 *out, uint32_t ncomp, uint32_t level, cudaStream_t s);
// A two-component ciphertext at some level inside a buffer of a higher one: component 1 lies comp words behind component 0
struct CtView { const u64 *p; size_t comp; };
inline bool aligned16(const CtView &v) { return aligned16(v.p) && (v.comp & 1) == 0; }
// e01[z], e2[z] = tensor(a[z], b[z]) for z < n
struct TensorArgs { CtView a[KS_MULTI], b[KS_MULTI]; u64 *e01[KS_MULTI], *e2[KS_MULTI]; };
void launch_tensor(const ckks_ctx *c, const TensorArgs &args, uint32_t n, uint32_t level, cudaStream_t s);
// slot values 1.0 on the slots x with lo <= x / B < hi and t0 <= x % Ti < t1, else 0.0 (n doubles on the device)
void launch_slot_mask(const ckks_ctx *c, double *out, uint32_t B, uint32_t lo, uint32_t hi, uint32_t Ti, uint32_t t0, uint32_t t1, cudaStream_t s);
// out = in * v or in + v (component 0 only) for the constant polynomial v
void launch_const(const ckks_ctx *c, const Ptrs &in, long long v, bool mul, const Ptrs &out, uint32_t ncomp, uint32_t level, cudaStream_t s, uint32_t n = 1);
// e01[o], e2[o] = sum_i tensor(a_i, b[o]_i) for `no` outputs that share the first operands (host arrays of n views each)
constexpr uint32_t TS_MAX = 16, TS_OUT = 4;
struct TensorSumArgs { CtView a[TS_MAX], b[TS_OUT][TS_MAX]; u64 *e01[TS_OUT], *e2[TS_OUT]; };
void launch_tensor_sum(const ckks_ctx *c, const CtView *a, const CtView *const *b, uint32_t n, u64 *const *e01, u64 *const *e2, uint32_t no, uint32_t level,
                       cudaStream_t s);
// out[o] (+)= sum_{j < nx} v[o][j] x[j] + cst[o] q_{level-1} (first component), o < no, for n ciphertexts each (see lincomb_kernel)
constexpr uint32_t LIN_MAX = 8;
struct LinArgs {
    Ptrs x[LIN_MAX], out[LIN_MAX];        // inputs: component 1 lies xc words behind component 0; outputs: [2][level][N]
    size_t xc[LIN_MAX];
    long long v[LIN_MAX][LIN_MAX], cst[LIN_MAX];
    uint32_t nx, no;
    int accumulate;
};
void launch_lincomb(const ckks_ctx *c, const LinArgs &args, uint32_t n, uint32_t level, cudaStream_t s);

// Key switch pieces.  Sizes in limbs: d [level], ext [beta][level+K], u [2][level+K], conv [2][level].
// d: the evaluation-domain input of the last ks_modup.  A digit's own limbs are not copied into ext; the inner product reads
// them from d, which has to stay as it is until then.
struct KsWorkspace {
    u64 *dcoef, *ext, *u, *conv;
    Ptrs d;
    bool alone = false;     // the key switch is an entry point's only one: see launch_ntt
    bool mid = false;       // ext is left after the column pass, for launch_mid_rows (set before ks_modup, see ks_mid)
};
size_t ks_workspace_limbs(const ckks_ctx *c, uint32_t level);
KsWorkspace ks_carve(const ckks_ctx *c, uint32_t level, void *ws, uint32_t nb = 1);
// nb key switches side by side: d (evaluation domain, [level][N] per entry) -> ext (evaluation domain, all digits without
// their own limbs).  A rotation applies its sigma_g to the extended digits when the inner product reads them (ext_galois
// below): the centred conversion commutes with the permutation and the sign flips of sigma_g, so this equals extending
// sigma_g(d), and d is never copied.
void ks_modup(const ckks_ctx *c, const Ptrs &d, uint32_t level, KsWorkspace &w, cudaStream_t s, uint32_t nb = 1);
// inner product with evk (digits read through sigma_{ext_galois}; 1 = identity): leaves u = <digits, evk> in the extended basis
// (w.u, nb entries); with acc_u it adds to what w.u holds, so that a sum of key-switched terms can share one ks_moddown; with
// `add` ([2][level][N] words per entry, no multi) it adds P add to both components.
void ks_inner(const ckks_ctx *c, const u64 *evk, uint32_t level, u64 ext_galois, const KsWorkspace &w, cudaStream_t s, uint32_t nb = 1,
              bool acc_u = false, const KsMulti *multi = nullptr, const Ptrs *add = nullptr);
// ModDown and the final combination out_c = sigma_galois(add_c) + k_c + acc_c (add taken for the components in add_comps, acc if
// given: [2][level][N] words per entry, possibly out itself)
struct KsOut {
    Ptrs add, out, acc;
    uint32_t add_comps = 0;
    u64 galois = 1;
    TiledOut tiled;
};
void ks_moddown(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, const KsOut &o, cudaStream_t s, uint32_t nb = 1, const KsMulti *multi = nullptr);
// Whether launch_mid_rows takes the digits d of key switches, which serve one key each (nkeys keys in all)
bool ks_mid(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, const Ptrs &d, const u64 *const *evk, uint32_t nkeys);
// and whether it is to take a sum of nterm terms of nb entries each
bool ks_mid_sum(const ckks_ctx *c, uint32_t level, uint32_t nterm, uint32_t nb);
// Both together: out = ModDown(<digits, key>) and the final combination, digits read through the permutation of o.galois
void ks_apply(const ckks_ctx *c, const u64 *evk, uint32_t level, const KsWorkspace &w, const KsOut &o, cudaStream_t s, uint32_t nb = 1, const KsMulti *multi = nullptr);
// out = rescale(ModDown(<digits, key>) + add), level - 1 limbs per component, without the tensor-core conversions (see ks_fused_rescale)
void ks_apply_rescale(const ckks_ctx *c, const u64 *evk, uint32_t level, const KsWorkspace &w, const Ptrs &add, const Ptrs &out, cudaStream_t s, uint32_t nb);
bool ks_fused_rescale(const ckks_ctx *c);
// A sum of up to IP_TERMS key-switched terms in one pass over the extended basis:
//   u[b] (+)= sum_t ( <ext[t][b] read through sigma_{g_t}, evk_t>  +  P sigma_{g_t}(c0_t[b]) on component 0's q-limbs )
// ext holds term t's digits of batch entry b at ext + t * term_stride + b * beta * (level + K) * N words, the own limbs of the
// digits lie at w.d.at(t * nb + b); c0[t]
// (may be null) points at term t's first-component limbs, entries c0_stride words apart.  Adding P c0 before the
// ModDown equals adding c0 after it, exactly.
constexpr uint32_t IP_TERMS = 4;
struct IpTerms {
    const u64 *evk[IP_TERMS];
    u64 galois[IP_TERMS];
    const u64 *c0[IP_TERMS];
};
void ks_inner_terms(const ckks_ctx *c, uint32_t level, const KsWorkspace &w, size_t term_stride, const IpTerms &terms, uint32_t nterm,
                    size_t c0_stride, cudaStream_t s, uint32_t nb, bool acc_u);
// The middle of a key switch whose digits serve one key each (mid_rows.cu): forward row pass of the extended digits (ext, after the
// column pass), inner product, inverse row pass of the limbs from inv_from on.
//   u[b] (+)= sum_t ( <ext[t][b] read through sigma_{g_t}, evk_t>  +  P sigma_{g_t}(c0_t[b]) )  +  P add[b]
// terms as in ks_inner_terms; with one term, entry b may have key b / group instead (group > 0)
struct MidArgs {
    const u64 *ext;
    Ptrs d, add;
    u64 *u;
    const u64 *evk[KS_MULTI], *c0[IP_TERMS];
    u64 galois[KS_MULTI];
    size_t term_stride, c0_stride;
    uint32_t nterm, nb, level, group, inv_from;
    int has_add, acc_u;
};
void launch_mid_rows(const ckks_ctx *c, const MidArgs &a, uint32_t beta, cudaStream_t s);
// The basis conversions on the tensor cores (contexts with byte matrices: at most 8 sources)
void launch_modup_mma(const ckks_ctx *c, const u64 *dcoef, u64 *ext, uint32_t level, uint32_t nb, cudaStream_t s);
void launch_moddown_conv_mma(const ckks_ctx *c, const u64 *u, u64 *conv, uint32_t level, uint32_t nb, cudaStream_t s);
// both components of n ciphertexts, src_stride words apart, into rows row0 + i * row_step + component of a tiled buffer with R rows
void launch_to_tiled(const ckks_ctx *c, const u64 *src, size_t src_stride, uint32_t n, u64 *dst, uint32_t R, uint32_t row0,
                     uint32_t row_step, uint32_t level, cudaStream_t s);
// dst = first + sum_{r < n} terms[r] for nct ciphertexts side by side (terms n * nct of them); first may be dst
void launch_sum(const ckks_ctx *c, u64 *dst, const u64 *first, const u64 *terms, uint32_t n, uint32_t nct, uint32_t level, cudaStream_t s);

// Tensor-core multiply-accumulate of a giant-step group (mac_mma.cu)
bool mac_mma_supported(const ckks_ctx *c, uint32_t J);
// baby, pts: tiled buffers with 2 * S * J rows ((shard * J + j) * 2 + component) and G * J rows (g * J + j)
// the baby buffer may hold Jx >= J rows per shard and component, of which rows j0 .. j0 + J - 1 are used (Jx = 0: J);
// accumulate: add to acc instead of overwriting it
bool launch_mac_mma(const ckks_ctx *c, const u64 *baby, const u64 *pts, u64 *acc, uint32_t J, uint32_t S, uint32_t G, uint32_t level,
                    cudaStream_t s, uint32_t Jx = 0, uint32_t j0 = 0, bool accumulate = false);

// the same contraction on the integer pipe, any J (mac_tile.cu): baby rows (s J + j) 2 + c, pts rows g J + j, both tiled
void launch_mac_tile(const ckks_ctx *c, const u64 *baby, const u64 *pts, u64 *acc, uint32_t J, uint32_t S, uint32_t G, uint32_t level,
                     cudaStream_t s);

// register-resident forward butterflies (measurement aid, ntt.cu); sink: device scratch of SMs * 4 * 256 words
uint64_t launch_butterfly_probe(const ckks_ctx *c, uint32_t iters, u64 *sink, cudaStream_t s);

// the same on tcgen05 / TMEM (mac_umma.cu); J <= 64
bool mac_umma_supported(const ckks_ctx *c, uint32_t J);
bool launch_mac_umma(const ckks_ctx *c, const u64 *baby, const u64 *pts, u64 *acc, uint32_t J, uint32_t S, uint32_t G, uint32_t level,
                     cudaStream_t s, uint32_t Jx = 0, uint32_t j0 = 0, bool accumulate = false);

// nb ciphertexts (at most KS_MULTI when the pointers are scattered) of ncomp components; ws: nb * ncomp * level limbs
void launch_rescale(const ckks_ctx *c, const Ptrs &in, const Ptrs &out, uint32_t ncomp, uint32_t level, u64 *ws, cudaStream_t s, uint32_t nb = 1,
                    bool alone = false);

size_t encode_workspace_bytes(const ckks_ctx *c, uint32_t batch);
// tiled.R != 0: plaintext b is written as row tiled.row0 + b * tiled.row_stride of the tiled buffer
// `tiled_out`; `out` is then only the scratch between the two NTT passes.
void launch_encode(const ckks_ctx *c, const double *re, const double *im, uint32_t batch, double scale, uint32_t level,
                   u64 *out, void *ws, cudaStream_t s, TiledOut tiled = TiledOut(), u64 *tiled_out = nullptr);
// Slot vectors of generalised diagonals, [count][n] fp64, for k = k0 .. k0+count-1 of one block pair, diagonal k pre-rotated by its
// giant step's share k - k % B.
void launch_extract_diagonals(const ckks_ctx *c, const double *W, uint32_t d_out_total, uint32_t in0, uint32_t m_in,
                              uint32_t out0, uint32_t m_out, uint32_t F, uint32_t T, uint32_t k0, uint32_t count,
                              uint32_t B, double *slots, cudaStream_t s);

// ---- sequences shared by the entry points (api.cu, poly.cu, attention.cu) -------------------------------------------
void relinearise(const ckks_ctx *c, const u64 *rlk, const Ptrs &e2, const Ptrs &o, uint32_t level, KsWorkspace &w, cudaStream_t s, uint32_t nb = 1);
void relin_rescale(const ckks_ctx *c, const u64 *rlk, const Ptrs &e2, const Ptrs &e01, const Ptrs &out, uint32_t level, u64 *ksw, cudaStream_t s,
                   uint32_t nb = 1);
void rotate_ks(const ckks_ctx *c, const ckks_evk *key, const Ptrs &in, const Ptrs &out, uint32_t level, KsWorkspace &w, cudaStream_t s, uint32_t nb = 1,
               const Ptrs *acc = nullptr);
size_t product_bytes(const ckks_ctx *c, uint32_t level);
void mul_rescale(const ckks_ctx *c, const CtView *a, const CtView *b, u64 *const *out, uint32_t n, const u64 *rlk, uint32_t level, void *ws, uint32_t chunk,
                 cudaStream_t s);
void sum_rescale(const ckks_ctx *c, const std::vector<std::vector<CtView>> &a, const std::vector<std::vector<CtView>> &b, u64 *const *out, uint32_t n,
                 const u64 *rlk, uint32_t level, void *ws, cudaStream_t s, size_t ws_bytes = SIZE_MAX);
size_t rotate_grid_bytes(const ckks_ctx *c, uint32_t level, uint32_t n, uint32_t nrot);
void rotate_grid(const ckks_ctx *c, const CtView *in, uint32_t n, const ckks_evk *keys, uint32_t nrot, u64 *out, size_t rot_stride, size_t ct_stride,
                 uint32_t level, void *ws, cudaStream_t s, size_t ws_bytes = SIZE_MAX);
// The polynomial of ckks_poly_eval_tree for n ciphertexts side by side (at most KS_MULTI; all at one level and scale).  plan
// first: it fixes levels, scales and constants and reports their errors before anything is launched.
struct TreePlan {
    uint32_t degree, level, Lt;
    double out_scale;
    std::vector<uint32_t> lvl;          // of x^k
    std::vector<long long> v;           // constants of x^k, v[0] for the constant term
};
int poly_tree_plan(const ckks_ctx *c, uint32_t level, double scale, const double *coeffs, uint32_t degree, TreePlan &p);
size_t poly_tree_bytes(const ckks_ctx *c, uint32_t level, uint32_t degree, uint32_t n);
void poly_tree_run(const ckks_ctx *c, const TreePlan &p, const Ptrs &x, const Ptrs &out, uint32_t n, const u64 *rlk, void *ws, cudaStream_t s);
bool const_value(double c, double scale, long long *v);
inline bool poly_bsgs_shape_ok(uint32_t degree, uint32_t m) { return m >= 2 && !(m & (m - 1)) && m <= degree; }
struct DeviceGuard {
    int prev = 0;
    explicit DeviceGuard(int dev) { cudaGetDevice(&prev); if (prev != dev) cudaSetDevice(dev); else prev = -1; }
    ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};
inline int finish(ckks_ctx *c) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { c->cuda_error = cudaGetErrorString(e); return CKKS_ERR_CUDA; }
    return CKKS_OK;
}
inline bool scales_agree(double a, double b) { return fabs(a - b) <= ldexp(fmax(fabs(a), fabs(b)), -30); }
inline bool ct_ok(const ckks_ct *ct) { return ct && ct->data; }
inline bool level_ok(const ckks_ctx *c, uint32_t level) { return level >= 1 && level <= c->L; }
inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
