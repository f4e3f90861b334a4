// Polynomials of a ciphertext: power tree and baby-step / giant-step evaluation.
//
// A product with relinearisation and rescale of one ciphertext is a chain of launches of at most one or two waves, so the
// time goes with the number of chains one after the other.  The powers x^k with 2^(d-1) < k <= 2^d only need powers up to
// 2^(d-1) and all have operands at one level: they are formed side by side (mul_rescale), log2 steps instead of k - 1 (the
// giant powers likewise).  Truncated operands are read in place (CtView), the linear combinations of all blocks run as one
// launch that reads every power once, and their rescales as one batch.  Degree 63 in blocks of 8 at N = 2^16, level 24:
// 549 -> 118 operations, 6.4 -> 2.6 ms (2.2 with ModDown and rescale in one step).
#include "common.cuh"

namespace {

// powers 2..top of a sequence whose power 1 is given: at(i, k) = view of power k of ciphertext i, dst(i, k) = its buffer
template <class At, class Dst>
void powers(const ckks_ctx *c, uint32_t top, const std::vector<uint32_t> &lvl, uint32_t n, At at, Dst dst, const u64 *rlk, void *ws, uint32_t chunk, cudaStream_t s) {
    std::vector<CtView> a, b;
    std::vector<u64 *> out;
    for (uint32_t lo = 2; lo <= top;) {
        const uint32_t lv = std::min(lvl[lo / 2], lvl[lo - lo / 2]);
        uint32_t hi = lo;       // the run of powers whose operands are there and meet at the same level
        while (hi <= top && hi - hi / 2 < lo && std::min(lvl[hi / 2], lvl[hi - hi / 2]) == lv) hi++;
        a.clear(); b.clear(); out.clear();
        for (uint32_t i = 0; i < n; i++)
            for (uint32_t k = lo; k < hi; k++) { a.push_back(at(i, k / 2)); b.push_back(at(i, k - k / 2)); out.push_back(dst(i, k)); }
        mul_rescale(c, a.data(), b.data(), out.data(), (uint32_t)out.size(), rlk, lv, ws, chunk, s);
        lo = hi;
    }
}
// the longest run that powers() forms at once
uint32_t widest(uint32_t top) {
    uint32_t w = 1, d = 1;
    for (; 2 * d < top; d *= 2) w = d;
    return std::max(w, top > d ? top - d : 0u);
}

// out[o] (+)= sum_j v[o][j] x[j] + cst[o], any number of inputs and outputs, n ciphertexts each
struct Lin {
    std::vector<Ptrs> x, out;
    std::vector<size_t> xc;
    std::vector<std::vector<long long>> v;      // [output][input]
    std::vector<long long> cst;
};
void lincomb(const ckks_ctx *c, const Lin &l, uint32_t n, uint32_t level, bool accumulate, cudaStream_t s) {
    for (size_t o0 = 0; o0 < l.out.size(); o0 += LIN_MAX)
        for (size_t j0 = 0; j0 == 0 || j0 < l.x.size(); j0 += LIN_MAX) {
            LinArgs g{};
            g.nx = (uint32_t)std::min<size_t>(LIN_MAX, l.x.size() - j0);
            g.no = (uint32_t)std::min<size_t>(LIN_MAX, l.out.size() - o0);
            for (uint32_t j = 0; j < g.nx; j++) { g.x[j] = l.x[j0 + j]; g.xc[j] = l.xc[j0 + j]; }
            for (uint32_t o = 0; o < g.no; o++) {
                g.out[o] = l.out[o0 + o];
                for (uint32_t j = 0; j < g.nx; j++) g.v[o][j] = l.v[o0 + o][j0 + j];
                g.cst[o] = j0 ? 0 : l.cst[o0 + o];
            }
            g.accumulate = accumulate || j0 > 0;
            launch_lincomb(c, g, n, level, s);
        }
}

bool rlk_ok(const ckks_evk *rlk) { return rlk && rlk->data && rlk->galois == 0; }
size_t ct_words(const ckks_ctx *c, uint32_t level) { return (size_t)2 * level * c->N; }

}  // namespace

// ---- power tree ----------------------------------------------------------------------------------------------------
int poly_tree_plan(const ckks_ctx *c, uint32_t level, double scale, const double *coeffs, uint32_t degree, TreePlan &p) {
    std::vector<double> sc(degree + 1);
    p.degree = degree; p.level = level;
    p.lvl.assign(degree + 1, 0);
    p.v.assign(degree + 1, 0);
    p.lvl[1] = level; sc[1] = scale;
    for (uint32_t k = 2; k <= degree; k++) {
        const uint32_t a = k / 2, b = k - a, lv = std::min(p.lvl[a], p.lvl[b]);
        sc[k] = sc[a] * sc[b] / (double)c->mod[lv - 1];
        p.lvl[k] = lv - 1;
    }
    p.Lt = p.lvl[degree];
    const double T = scale * (double)c->mod[p.Lt - 1];
    p.out_scale = T / (double)c->mod[p.Lt - 1];
    bool any = false;
    for (uint32_t k = 1; k <= degree; k++) {
        if (coeffs[k] == 0.0) continue;
        any = true;
        if (!const_value(coeffs[k], T / sc[k], &p.v[k])) return CKKS_ERR_RANGE;
    }
    if (!any) return CKKS_ERR_ARG;
    return const_value(coeffs[0], p.out_scale, &p.v[0]) ? CKKS_OK : CKKS_ERR_RANGE;
}

static uint32_t tree_chunk(uint32_t degree, uint32_t n) { return std::min<uint32_t>(KS_MULTI, n * widest(degree)); }

// the powers x^2.. and the sum of every ciphertext, then the products side by side (their bytes serve the last rescale too)
size_t poly_tree_bytes(const ckks_ctx *c, uint32_t level, uint32_t degree, uint32_t n) {
    const uint32_t d = std::max<uint32_t>(degree, 2);
    return (size_t)n * d * ct_words(c, level) * sizeof(u64) +
           std::max((size_t)tree_chunk(d, n) * product_bytes(c, level), (size_t)n * ct_words(c, level) * sizeof(u64));
}

void poly_tree_run(const ckks_ctx *c, const TreePlan &p, const Ptrs &x, const Ptrs &out, uint32_t n, const u64 *rlk, void *ws, cudaStream_t s) {
    const size_t N = c->N, ctw = ct_words(c, p.level);
    u64 *pw = (u64 *)ws, *acc = pw + (size_t)n * (p.degree - 1) * ctw;      // x^k of ciphertext i at pw + ((k - 2) n + i) ctw
    void *rest = acc + n * ctw;
    auto dst = [&](uint32_t i, uint32_t k) { return pw + ((size_t)(k - 2) * n + i) * ctw; };
    auto at = [&](uint32_t i, uint32_t k) { return CtView{k == 1 ? x.at(i) : dst(i, k), (size_t)p.lvl[k] * N}; };
    powers(c, p.degree, p.lvl, n, at, dst, rlk, rest, tree_chunk(p.degree, n), s);
    Lin l;
    l.out = {Ptrs(acc, ctw)};
    l.cst = {p.v[0]};
    l.v.resize(1);
    for (uint32_t k = 1; k <= p.degree; k++) {
        if (!p.v[k]) continue;
        l.x.push_back(k == 1 ? x : Ptrs(dst(0, k), ctw));
        l.xc.push_back((size_t)p.lvl[k] * N);
        l.v[0].push_back(p.v[k]);
    }
    lincomb(c, l, n, p.Lt, false, s);
    launch_rescale(c, Ptrs(acc, ctw), out, 2, p.Lt, (u64 *)rest, s, n);
}

extern "C" int32_t ckks_poly_eval_tree(ckks_ctx *c, const ckks_ct *x, const double *coeffs, uint32_t degree, const ckks_evk *rlk,
                                       ckks_ct *out, void *ws, size_t ws_bytes, void *stream) {
    if (!c || !ct_ok(x) || !ct_ok(out) || x->ncomp != 2 || !coeffs || degree < 2) return CKKS_ERR_ARG;
    const uint32_t level = x->level;
    uint32_t depth = 0;
    while ((1u << depth) < degree) depth++;
    if (!level_ok(c, level) || level < depth + 2) return CKKS_ERR_LEVEL;
    if (!rlk_ok(rlk)) return CKKS_ERR_NO_KEY;
    if (!ws || ws_bytes < ckks_workspace_bytes(c, CKKS_OP_POLY_EVAL_TREE, level, degree)) return CKKS_ERR_WORKSPACE;
    TreePlan p;
    int rc = poly_tree_plan(c, level, x->scale, coeffs, degree, p);
    if (rc) return rc;
    DeviceGuard g(c->device);
    poly_tree_run(c, p, Ptrs((const u64 *)x->data, 0), Ptrs((const u64 *)out->data, 0), 1, (const u64 *)rlk->data, ws, (cudaStream_t)stream);
    rc = finish(c);
    if (rc == CKKS_OK) { out->level = p.Lt - 1; out->ncomp = 2; out->scale = p.out_scale; }
    return rc;
}

// ---- baby steps and giant steps ------------------------------------------------------------------------------------
namespace {

struct BsgsPlan {
    uint32_t degree, m, G, level, Lb, Lc;
    std::vector<uint32_t> lb, lg;                 // levels of x^k, y^i
    std::vector<uint32_t> blocks, const_only;     // giant indices with a block polynomial / with a constant alone
    std::vector<std::vector<long long>> bv;       // per block: constants of x^1 .. x^(m-1)
    std::vector<long long> bc, av, cv;            // block constants; block 0's constants of x^1 ..; those of the lone giants
    long long c0;
    double out_scale;
};

// levels, scales and constants in the order the definition fixes them (a product's scale divided by the dropped prime)
int bsgs_plan(const ckks_ctx *c, uint32_t level, double scale, const double *coeffs, uint32_t degree, uint32_t m, BsgsPlan &p) {
    const uint32_t G = degree / m + 1;
    p.degree = degree; p.m = m; p.G = G; p.level = level;
    auto q = [&](uint32_t l) { return (double)c->mod[l - 1]; };
    auto levels = [&](std::vector<uint32_t> &l, std::vector<double> &s, uint32_t top) {
        for (uint32_t k = 2; k <= top; k++) {
            const uint32_t lv = std::min(l[k / 2], l[k - k / 2]);
            if (lv < 2) return false;
            l[k] = lv - 1;
            s[k] = s[k / 2] * s[k - k / 2] / q(lv);
        }
        return true;
    };
    std::vector<double> sb(m + 1), sg(std::max<uint32_t>(G, 2));
    p.lb.assign(m + 1, 0); p.lg.assign(std::max<uint32_t>(G, 2), 0);
    p.lb[1] = level; sb[1] = scale;
    if (!levels(p.lb, sb, m)) return CKKS_ERR_LEVEL;
    p.lg[1] = p.lb[m]; sg[1] = sb[m];
    if (!levels(p.lg, sg, G - 1)) return CKKS_ERR_LEVEL;
    p.Lb = p.lb[m - 1];
    p.Lc = std::min(p.lg[G - 1], p.Lb - 1);
    if (p.Lb < 2 || p.Lc < 2) return CKKS_ERR_LEVEL;
    auto coef = [&](uint32_t k) { return k <= degree ? coeffs[k] : 0.0; };
    const double Tp = scale * q(p.Lc);
    for (uint32_t i = 1; i < G; i++) {
        const double Ti = (Tp / sg[i]) * q(p.Lb);
        std::vector<long long> v(m - 1, 0);
        bool any = false;
        for (uint32_t j = 1; j < m; j++) {
            if (coef(i * m + j) == 0.0) continue;
            any = true;
            if (!const_value(coef(i * m + j), Ti / sb[j], &v[j - 1])) return CKKS_ERR_RANGE;
        }
        long long k = 0;
        if (any) {
            if (!const_value(coef(i * m), Ti / q(p.Lb), &k)) return CKKS_ERR_RANGE;
            p.blocks.push_back(i); p.bv.push_back(v); p.bc.push_back(k);
        } else if (coef(i * m) != 0.0) {
            if (!const_value(coef(i * m), Tp / sg[i], &k)) return CKKS_ERR_RANGE;
            p.const_only.push_back(i); p.cv.push_back(k);
        }
    }
    p.av.assign(m - 1, 0);
    bool have = !p.blocks.empty() || !p.const_only.empty();
    for (uint32_t j = 1; j < m; j++) {
        if (coef(j) == 0.0) continue;
        have = true;
        if (!const_value(coef(j), Tp / sb[j], &p.av[j - 1])) return CKKS_ERR_RANGE;
    }
    if (!have) return CKKS_ERR_ARG;
    p.out_scale = Tp / q(p.Lc);
    return const_value(coef(0), p.out_scale, &p.c0) ? CKKS_OK : CKKS_ERR_RANGE;
}

// buffers per ciphertext: baby powers 2..m, giant powers 2..G-1, the blocks before and after their rescale
uint32_t bsgs_buffers(uint32_t degree, uint32_t m) {
    const uint32_t G = degree / m + 1;
    return (m - 1) + (G > 2 ? G - 2 : 0) + 2 * (G - 1);
}
uint32_t bsgs_chunk(uint32_t degree, uint32_t m, uint32_t n) {
    return std::min<uint32_t>(KS_MULTI, n * std::max(widest(m), widest(degree / m)));
}
size_t bsgs_bytes(const ckks_ctx *c, uint32_t level, uint32_t degree, uint32_t m, uint32_t n) {
    const size_t ctb = ct_words(c, level) * sizeof(u64);
    // the products' bytes also hold the rescales of all blocks and the giant-step sums with their key switch
    return (size_t)n * bsgs_buffers(degree, m) * ctb +
           std::max((size_t)std::max(bsgs_chunk(degree, m, n), n) * product_bytes(c, level), (size_t)n * (degree / m) * ctb);
}

void bsgs_run(const ckks_ctx *c, const BsgsPlan &p, const Ptrs &x, const Ptrs &out, uint32_t n, const u64 *rlk, void *ws, cudaStream_t s) {
    const size_t N = c->N, ctw = ct_words(c, p.level);
    const uint32_t m = p.m, G = p.G;
    u64 *next = (u64 *)ws;
    auto buffers = [&](uint32_t count) { u64 *b = next; next += (size_t)count * n * ctw; return b; };       // [count][n]
    u64 *bp = buffers(m - 1), *gp = buffers(G > 2 ? G - 2 : 0), *acc = buffers(G - 1), *blk = buffers(G - 1);
    void *rest = next;
    const uint32_t chunk = bsgs_chunk(p.degree, m, n);
    auto bdst = [&](uint32_t i, uint32_t k) { return bp + ((size_t)(k - 2) * n + i) * ctw; };
    auto bat = [&](uint32_t i, uint32_t k) { return CtView{k == 1 ? x.at(i) : bdst(i, k), (size_t)p.lb[k] * N}; };
    auto gdst = [&](uint32_t i, uint32_t k) { return gp + ((size_t)(k - 2) * n + i) * ctw; };
    auto gat = [&](uint32_t i, uint32_t k) { return k == 1 ? bat(i, m) : CtView{gdst(i, k), (size_t)p.lg[k] * N}; };
    powers(c, m, p.lb, n, bat, bdst, rlk, rest, chunk, s);
    powers(c, G - 1, p.lg, n, gat, gdst, rlk, rest, chunk, s);
    auto bptrs = [&](uint32_t k) { return k == 1 ? x : Ptrs(bdst(0, k), ctw); };
    // blocks B_i, i >= 1: one linear combination of the baby powers each, rescaled together
    const uint32_t nblk = (uint32_t)p.blocks.size();
    const size_t accw = (size_t)2 * p.Lb * N, blkw = (size_t)2 * (p.Lb - 1) * N;
    if (nblk) {
        Lin l;
        for (uint32_t j = 1; j < m; j++) { l.x.push_back(bptrs(j)); l.xc.push_back((size_t)p.lb[j] * N); }
        for (uint32_t b = 0; b < nblk; b++) l.out.push_back(Ptrs(acc + (size_t)b * n * accw, accw));
        l.v = p.bv; l.cst = p.bc;
        lincomb(c, l, n, p.Lb, false, s);
        launch_rescale(c, Ptrs(acc, accw), Ptrs(blk, blkw), 2, p.Lb, (u64 *)rest, s, nblk * n);
    }
    // S = sum_i B_i y^i, relinearised once; block 0 and the lone giants join it before the key switch, the constant term as
    // well (times the prime that the rescale divides by)
    const size_t sw = (size_t)2 * p.Lc * N, ew = (size_t)p.Lc * N;
    u64 *S = (u64 *)rest, *e2 = S + n * sw, *ksw = e2 + n * ew;
    for (uint32_t i = 0; i < n && nblk; i++) {
        std::vector<CtView> A, B;
        for (uint32_t b = 0; b < nblk; b++) {
            A.push_back(CtView{blk + ((size_t)b * n + i) * blkw, (size_t)(p.Lb - 1) * N});
            B.push_back(gat(i, p.blocks[b]));
        }
        const CtView *pb = B.data();
        u64 *p01 = S + i * sw, *p2 = e2 + i * ew;
        launch_tensor_sum(c, A.data(), &pb, nblk, &p01, &p2, 1, p.Lc, s);
    }
    Lin l;
    l.out = {Ptrs(S, sw)};
    l.cst = {p.c0};
    l.v.resize(1);
    for (uint32_t j = 1; j < m; j++)
        if (p.av[j - 1]) { l.x.push_back(bptrs(j)); l.xc.push_back((size_t)p.lb[j] * N); l.v[0].push_back(p.av[j - 1]); }
    for (size_t k = 0; k < p.const_only.size(); k++) {
        const uint32_t i = p.const_only[k];
        l.x.push_back(i == 1 ? bptrs(m) : Ptrs(gdst(0, i), ctw));
        l.xc.push_back(gat(0, i).comp);
        l.v[0].push_back(p.cv[k]);
    }
    lincomb(c, l, n, p.Lc, nblk > 0, s);
    if (nblk) relin_rescale(c, rlk, Ptrs(e2, ew), Ptrs(S, sw), out, p.Lc, ksw, s, n);
    else launch_rescale(c, Ptrs(S, sw), out, 2, p.Lc, ksw, s, n);
}

constexpr uint32_t POLY_BATCH = 4;      // ciphertexts evaluated side by side by the batch entry point

}  // namespace

extern "C" size_t ckks_poly_eval_bsgs_workspace_bytes(const ckks_ctx *c, uint32_t level, uint32_t degree, uint32_t m) {
    if (!c || !level_ok(c, level) || !poly_bsgs_shape_ok(degree, m)) return 0;
    return bsgs_bytes(c, level, degree, m, 1);
}

extern "C" size_t ckks_poly_eval_bsgs_batch_workspace_bytes(const ckks_ctx *c, uint32_t level, uint32_t degree, uint32_t m, uint32_t n) {
    if (!c || !level_ok(c, level) || !poly_bsgs_shape_ok(degree, m)) return 0;
    return bsgs_bytes(c, level, degree, m, std::min(std::max<uint32_t>(n, 1), POLY_BATCH));
}

static int32_t bsgs_entry(ckks_ctx *c, const ckks_ct *x, uint32_t n, const double *coeffs, uint32_t degree, uint32_t m, const ckks_evk *rlk, ckks_ct *out,
                          void *ws, size_t ws_bytes, size_t need, void *stream) {
    if (!level_ok(c, x[0].level)) return CKKS_ERR_LEVEL;
    if (!rlk_ok(rlk)) return CKKS_ERR_NO_KEY;
    std::vector<BsgsPlan> plans(n);
    std::vector<double> scale(n);           // x and out may be one array: its scales change on the way
    for (uint32_t i = 0; i < n; i++) scale[i] = x[i].scale;
    for (uint32_t i = 0; i < n; i++)
        if (i == 0 || scale[i] != scale[0]) {
            const int rc = bsgs_plan(c, x[i].level, scale[i], coeffs, degree, m, plans[i]);
            if (rc) return rc;
        }
    if (!ws || ws_bytes < need) return CKKS_ERR_WORKSPACE;
    DeviceGuard guard(c->device);
    for (uint32_t i = 0; i < n;) {
        // a run of ciphertexts of one scale: the constants depend on it
        const bool own = i == 0 || scale[i] != scale[0];
        const BsgsPlan &p = own ? plans[i] : plans[0];
        uint32_t k = 1;
        while (k < POLY_BATCH && i + k < n && scale[i + k] == scale[i]) k++;
        Ptrs px, po;
        px.n = po.n = k;
        for (uint32_t j = 0; j < k; j++) { px.p[j] = (const u64 *)x[i + j].data; po.p[j] = (const u64 *)out[i + j].data; }
        bsgs_run(c, p, px, po, k, (const u64 *)rlk->data, ws, (cudaStream_t)stream);
        for (uint32_t j = 0; j < k; j++) { out[i + j].level = p.Lc - 1; out[i + j].ncomp = 2; out[i + j].scale = p.out_scale; }
        i += k;
    }
    return finish(c);
}

extern "C" int32_t ckks_poly_eval_bsgs(ckks_ctx *c, const ckks_ct *x, const double *coeffs, uint32_t degree, uint32_t m, const ckks_evk *rlk,
                                       ckks_ct *out, void *ws, size_t ws_bytes, void *stream) {
    if (!c || !ct_ok(x) || !ct_ok(out) || x->ncomp != 2 || !coeffs || !poly_bsgs_shape_ok(degree, m)) return CKKS_ERR_ARG;
    return bsgs_entry(c, x, 1, coeffs, degree, m, rlk, out, ws, ws_bytes, ckks_poly_eval_bsgs_workspace_bytes(c, x->level, degree, m), stream);
}

extern "C" int32_t ckks_poly_eval_bsgs_batch(ckks_ctx *c, const ckks_ct *x, uint32_t n, const double *coeffs, uint32_t degree, uint32_t m,
                                             const ckks_evk *rlk, ckks_ct *out, void *ws, size_t ws_bytes, void *stream) {
    if (!c || !x || !out || !n || !coeffs || !poly_bsgs_shape_ok(degree, m)) return CKKS_ERR_ARG;
    for (uint32_t i = 0; i < n; i++)
        if (!ct_ok(&x[i]) || !ct_ok(&out[i]) || x[i].ncomp != 2) return CKKS_ERR_ARG;
    for (uint32_t i = 0; i < n; i++)
        if (x[i].level != x[0].level) return CKKS_ERR_LEVEL;
    return bsgs_entry(c, x, n, coeffs, degree, m, rlk, out, ws, ws_bytes, ckks_poly_eval_bsgs_batch_workspace_bytes(c, x[0].level, degree, m, n), stream);
}
