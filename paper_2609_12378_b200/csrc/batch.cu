// Sequences of launches that several entry points share, all over many ciphertexts side by side: one ciphertext's launches
// are one or two waves of CTAs each, sixteen ciphertexts' fill the GPU, and a switching key is read once for all of them.
#include "common.cuh"

// o[i] (2 x level limbs) += key switch of e2[i], nb side by side
void relinearise(const ckks_ctx *c, const u64 *rlk, const Ptrs &e2, const Ptrs &o, uint32_t level, KsWorkspace &w, cudaStream_t s, uint32_t nb) {
    w.mid = ks_mid(c, level, w, e2, &rlk, 1);
    ks_modup(c, e2, level, w, s, nb);
    KsOut ko;
    ko.add = ko.out = o;
    ko.add_comps = 3;
    ks_apply(c, rlk, level, w, ko, s, nb);
}
// out[i] = rescale(e01[i] + key switch of e2[i]); ksw: the workspace of nb key switches
void relin_rescale(const ckks_ctx *c, const u64 *rlk, const Ptrs &e2, const Ptrs &e01, const Ptrs &out, uint32_t level, u64 *ksw, cudaStream_t s, uint32_t nb) {
    KsWorkspace w = ks_carve(c, level, ksw, nb);
    if (!ks_fused_rescale(c)) {
        relinearise(c, rlk, e2, e01, level, w, s, nb);
        launch_rescale(c, e01, out, 2, level, ksw, s, nb);
        return;
    }
    w.mid = ks_mid(c, level, w, e2, &rlk, 1) && aligned16(e01);
    ks_modup(c, e2, level, w, s, nb);
    ks_apply_rescale(c, rlk, level, w, e01, out, s, nb);
}
// One product's share of a batch: the tensor product's two parts and a key-switch workspace (whose bytes the rescale reuses)
size_t product_bytes(const ckks_ctx *c, uint32_t level) { return ((size_t)3 * level + ks_workspace_limbs(c, level)) * c->N * sizeof(u64); }

// out[i] = rescale(relin(a[i] b[i])), up to `chunk` products side by side; ws: min(n, chunk) * product_bytes
void mul_rescale(const ckks_ctx *c, const CtView *a, const CtView *b, u64 *const *out, uint32_t n, const u64 *rlk, uint32_t level, void *ws, uint32_t chunk,
                 cudaStream_t s) {
    const size_t N = c->N, ctl = (size_t)2 * level * N, ptl = (size_t)level * N;
    for (uint32_t i0 = 0; i0 < n; i0 += chunk) {
        const uint32_t m = std::min(chunk, n - i0);
        u64 *e01 = (u64 *)ws, *e2 = e01 + m * ctl, *ksw = e2 + m * ptl;
        TensorArgs ta;
        Ptrs po;
        po.n = m;
        for (uint32_t i = 0; i < m; i++) {
            ta.a[i] = a[i0 + i]; ta.b[i] = b[i0 + i];
            ta.e01[i] = e01 + i * ctl; ta.e2[i] = e2 + i * ptl;
            po.p[i] = out[i0 + i];
        }
        launch_tensor(c, ta, m, level, s);
        relin_rescale(c, rlk, Ptrs(e2, ptl), Ptrs(e01, ctl), po, level, ksw, s, m);
    }
}

// out = rotation of nb ciphertexts by one key (+ acc, both components, where acc is given; acc may be out, out must not be in)
void rotate_ks(const ckks_ctx *c, const ckks_evk *key, const Ptrs &in, const Ptrs &out, uint32_t level, KsWorkspace &w, cudaStream_t s, uint32_t nb,
               const Ptrs *acc) {
    Ptrs c1 = in;
    const size_t ptl = (size_t)level * c->N;
    if (in.n) for (uint32_t b = 0; b < in.n; b++) c1.p[b] += ptl;
    else c1.base += ptl;
    const u64 *evk = (const u64 *)key->data;
    w.mid = ks_mid(c, level, w, c1, &evk, 1);
    ks_modup(c, c1, level, w, s, nb);
    KsOut ko;
    ko.add = in; ko.out = out;
    ko.add_comps = 1; ko.galois = key->galois;
    if (acc) ko.acc = *acc;
    ks_apply(c, evk, level, w, ko, s, nb);
}

static bool same_views(const std::vector<CtView> &x, const std::vector<CtView> &y) {
    return x.size() == y.size() && std::equal(x.begin(), x.end(), y.begin(), [](const CtView &u, const CtView &v) { return u.p == v.p && u.comp == v.comp; });
}

// out[i] = rescale(relin(sum_t a[i][t] b[i][t])) for n sums of nterm products; ws: min(n, KS_MULTI) * product_bytes, or a ws_bytes
// of at least one product_bytes, which takes as many sums side by side as it holds
void sum_rescale(const ckks_ctx *c, const std::vector<std::vector<CtView>> &a, const std::vector<std::vector<CtView>> &b, u64 *const *out, uint32_t n,
                 const u64 *rlk, uint32_t level, void *ws, cudaStream_t s, size_t ws_bytes) {
    const size_t N = c->N, ctl = (size_t)2 * level * N, ptl = (size_t)level * N;
    const uint32_t side = (uint32_t)std::min<size_t>(KS_MULTI, ws_bytes / product_bytes(c, level));
    for (uint32_t i0 = 0; i0 < n; i0 += side) {
        const uint32_t m = std::min(side, n - i0);
        u64 *e01 = (u64 *)ws, *e2 = e01 + m * ctl, *ksw = e2 + m * ptl;
        Ptrs po;
        po.n = m;
        for (uint32_t i = 0; i < m;) {
            // neighbours with the same first operands share a pass over them
            const CtView *pb[KS_MULTI];
            u64 *p01[KS_MULTI], *p2[KS_MULTI];
            uint32_t r = 0;
            for (; i + r < m && (r == 0 || same_views(a[i0 + i], a[i0 + i + r])); r++) {
                pb[r] = b[i0 + i + r].data();
                p01[r] = e01 + (i + r) * ctl; p2[r] = e2 + (i + r) * ptl;
                po.p[i + r] = out[i0 + i + r];
            }
            launch_tensor_sum(c, a[i0 + i].data(), pb, (uint32_t)a[i0 + i].size(), p01, p2, r, level, s);
            i += r;
        }
        relin_rescale(c, rlk, Ptrs(e2, ptl), Ptrs(e01, ctl), po, level, ksw, s, m);
    }
}

// ---- many ciphertexts times many rotations -------------------------------------------------------------------------
// Up to GRID_CTS ciphertexts share a pass: each is extended once, every key is applied to all of them (and read once for
// them), GRID_ENTRIES key switches side by side.
constexpr uint32_t GRID_CTS = 8, GRID_ENTRIES = 32;
static uint32_t grid_keys(uint32_t members, uint32_t nrot) { return std::min(nrot, std::min(KS_MULTI, std::max(1u, GRID_ENTRIES / members))); }
static size_t grid_bytes(const ckks_ctx *c, uint32_t level, uint32_t members, uint32_t keys) {
    const size_t beta = (level + c->alpha - 1) / c->alpha, nt = level + c->K;
    return (members * (level + beta * nt) + (size_t)members * keys * (2 * nt + 2 * level)) * c->N * sizeof(u64);
}
size_t rotate_grid_bytes(const ckks_ctx *c, uint32_t level, uint32_t n, uint32_t nrot) {
    const uint32_t m = std::min(n, GRID_CTS);
    return grid_bytes(c, level, m, grid_keys(m, nrot));
}
// rotation r of ciphertext i (components comp words apart, taken at `level`) -> out + r * rot_stride + i * ct_stride
// ws: rotate_grid_bytes, or a ws_bytes of at least what one ciphertext and one key take, which lets as many share a pass as fit
void rotate_grid(const ckks_ctx *c, const CtView *in, uint32_t n, const ckks_evk *keys, uint32_t nrot, u64 *out, size_t rot_stride, size_t ct_stride,
                 uint32_t level, void *ws, cudaStream_t s, size_t ws_bytes) {
    if (!n || !nrot) return;
    const size_t beta = (level + c->alpha - 1) / c->alpha, nt = level + c->K, N = c->N;
    uint32_t mmax = std::min(n, GRID_CTS), kmax = grid_keys(mmax, nrot);
    for (; mmax > 1 && grid_bytes(c, level, mmax, kmax) > ws_bytes; kmax = grid_keys(mmax, nrot)) mmax--;
    while (kmax > 1 && grid_bytes(c, level, mmax, kmax) > ws_bytes) kmax--;
    KsWorkspace w;
    w.dcoef = (u64 *)ws;
    w.ext = w.dcoef + (size_t)mmax * level * N;
    w.u = w.ext + mmax * beta * nt * N;
    w.conv = w.u + (size_t)mmax * kmax * 2 * nt * N;
    for (uint32_t i0 = 0; i0 < n; i0 += mmax) {
        const uint32_t m = std::min(mmax, n - i0);
        KsOut ko;
        ko.add.n = m; ko.add_comps = 1;
        ko.out = Ptrs(out + i0 * ct_stride, ct_stride);
        Ptrs c1;
        c1.n = m;
        for (uint32_t i = 0; i < m; i++) { ko.add.p[i] = in[i0 + i].p; c1.p[i] = in[i0 + i].p + in[i0 + i].comp; }
        ks_modup(c, c1, level, w, s, m);
        for (uint32_t r0 = 0; r0 < nrot; r0 += kmax) {
            const uint32_t nr = std::min(kmax, nrot - r0);
            KsMulti k{};
            k.group = m; k.rot_stride = rot_stride;
            for (uint32_t r = 0; r < nr; r++) { k.galois[r] = keys[r0 + r].galois; k.evk[r] = (const u64 *)keys[r0 + r].data; }
            ko.out.base = out + r0 * rot_stride + i0 * ct_stride;
            ks_apply(c, nullptr, level, w, ko, s, nr * m, &k);
        }
    }
}
