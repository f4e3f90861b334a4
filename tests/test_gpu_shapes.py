"""GPU parity at the sizes where a kernel's split of the work can go wrong (tile edges, remainders, the ends of a range),
against the CPU oracle, bit for bit."""
import numpy as np
import pytest

from paper_2609_12378_b200 import inputs
from tests.harness import params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,K,dnum,level", [(3, 1, 3, 3), (7, 4, 3, 5), (8, 8, 1, 8), (9, 9, 1, 9), (17, 17, 1, 17), (17, 17, 1, 8)])
def test_basis_conversion_at_the_ends_of_the_residues(L, K, dnum, level):
    """One to seventeen sources (one, two and three groups of eight, full and partial digits), every first factor
    [d qhat^-1] drawn from 0, 1, q - 1 and the two residues next to q / 2, where the unreduced sums are largest."""
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(10, L, K, dnum), context(10, L, K, dnum)
    o, g = P.oracle, inputs.rng(700, level + 100 * L)
    alpha = -(-L // dnum)
    d = np.empty((1, level, P.N), dtype=np.uint64)
    for i in range(level):
        q, lo = int(P.q[i]), i // alpha * alpha
        hat = 1
        for b in range(lo, min(lo + alpha, level)):
            hat = hat * (int(P.q[b]) if b != i else 1) % q
        ends = np.array([y * hat % q for y in (0, 1, q - 1, q // 2, q // 2 + 1)], dtype=np.uint64)
        d[0, i] = ends[g.integers(0, 5, P.N)]
        d[0, i, :64] = ends[3 + np.arange(64) % 2]          # all sources at q / 2 together
    ct = np.concatenate([inputs.uniform_residues(g, P.q[:level], P.N, 1), o.ntt(d)])
    key = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, dnum * 2).reshape(dnum, 2, L + K, P.N)
    gal = o.galois_element(3)
    out = ctx.rotate(ct_dev(ct, 1.0), key_dev(key, gal))
    assert np.array_equal(host(out.data), o.rotate(ct, key, gal))


@pytest.mark.parametrize("log_n", range(10, 17))
@pytest.mark.parametrize("batch,limbs", [(1, 1), (5, 3)])
def test_transforms_of_every_ring_at_extreme_residues(log_n, batch, limbs):
    """Both directions on constant, alternating and random limbs (the lazy ranges of the butterflies peak where every input
    is 0 or q - 1), in a 16-byte aligned buffer and in one that is only 8-byte aligned."""
    import torch
    from tests.gpu_util import context, host
    P, ctx = params(log_n, 3, 1, 3), context(log_n, 3, 1, 3)
    o, g = P.oracle, inputs.rng(710, log_n)
    x = inputs.uniform_residues(g, P.q[:limbs], P.N, batch)
    for i in range(limbs):
        q = int(P.q[i])
        x[0, i] = q - 1
        if batch > 1:
            x[1, i] = np.where(np.arange(P.N) & 1, q - 1, 0)
            x[2, i] = np.where(g.integers(0, 2, P.N), q - 1, 0)
            x[3, i] = np.where(g.integers(0, 2, P.N), q // 2, q // 2 + 1)
    fwd, inv = o.ntt(x), o.intt(x)
    for offset in (0, 1):
        buf = torch.zeros(x.size + 1, dtype=torch.int64, device="cuda").view(torch.uint64)
        y = buf[offset:offset + x.size].view(batch, limbs, P.N)
        y.copy_(torch.from_numpy(x))
        assert np.array_equal(host(ctx.ntt(y)), fwd)
        y.copy_(torch.from_numpy(x))
        assert np.array_equal(host(ctx.intt(y)), inv)
        assert int(buf[x.size if offset == 0 else 0]) == 0


@pytest.mark.parametrize("log_n,level", [(10, 2), (13, 3), (15, 3), (16, 2)])
@pytest.mark.parametrize("ncomp", [1, 2])
def test_rescale_components_and_alignment(log_n, level, ncomp):
    """One and two components; dropped residues at the ends of their centred range; one component in place; buffers that are
    only 8-byte aligned."""
    import torch
    from tests.gpu_util import context, ct_dev, host
    from paper_2609_12378_b200 import binding
    P, ctx = params(log_n, 3, 1, 3), context(log_n, 3, 1, 3)
    g = inputs.rng(720, log_n)
    x = inputs.uniform_residues(g, P.q[:level], P.N, ncomp)
    q = int(P.q[level - 1])
    d = np.array([0, 1, q - 1, q // 2, q // 2 + 1], dtype=np.uint64)[g.integers(0, 5, P.N)]
    full = np.zeros((1, 3, P.N), dtype=np.uint64)
    full[0, level - 1] = d
    x[0, level - 1] = P.oracle.ntt(full)[0, level - 1]
    want = P.oracle.rescale(x)
    out = ctx.rescale(ct_dev(x, 1.0))
    assert np.array_equal(host(out.data), want)
    buf = torch.zeros(x.size + 1, dtype=torch.int64, device="cuda").view(torch.uint64)
    y = buf[1:].view(ncomp, level, P.N)
    y.copy_(torch.from_numpy(x))
    assert np.array_equal(host(ctx.rescale(binding.Ciphertext(y, 1.0)).data), want)
    if ncomp == 1:
        ct = ct_dev(x, 1.0)
        short = binding.Ciphertext(ct.data.view(-1)[:(level - 1) * P.N].view(1, level - 1, P.N), 0.0)
        ctx.rescale(ct, out=short)
        assert np.array_equal(host(short.data), want)


@pytest.mark.parametrize("log_n", [11, 14, 16])
def test_encode_coefficients_of_every_size(log_n):
    """Coefficients below 2^49 are taken as residues as they are, larger ones (here up to 2^61) are reduced; a batch mixes
    both, and one plaintext has a single large coefficient's worth of slots."""
    from tests.gpu_util import context, dev, host
    P, ctx = params(log_n, 3, 1, 3), context(log_n, 3, 1, 3)
    g = inputs.rng(730, log_n)
    z = g.uniform(-1, 1, (4, P.n))
    z[1] *= 2.0 ** 20
    z[2] = 2.0 ** 9          # one coefficient of 2^59, the others zero
    z[3, 1:] = 0.0
    for scale in (2.0 ** 30, 2.0 ** 50):
        zz = z if scale < 2.0 ** 40 else z * np.array([[1.0], [2.0 ** -10], [1.0], [1.0]])
        got = host(ctx.encode(dev(zz), None, scale, 3))
        for b in range(4):
            assert np.array_equal(got[b], P.oracle.encode(zz[b], scale, 3)), (scale, b)


@pytest.mark.parametrize("degree,m,count", [(40, 16, 5), (23, 2, 1), (16, 16, 2)])
def test_polynomial_batches_and_combinations(degree, m, count):
    """More inputs (15) and more blocks (11) than one combination launch takes, a block that is only a constant, zero
    coefficients, ciphertexts of two scales in one batch, and the power tree of the same degree."""
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(10, 10, 4, 3), context(10, 10, 4, 3)
    o, g = P.oracle, inputs.rng(740, degree)
    rlk = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, 6).reshape(3, 2, 14, P.N)
    coeffs = g.uniform(-1, 1, degree + 1)
    coeffs[m + 1:2 * m] = 0.0
    coeffs[3] = 0.0
    cts = [inputs.uniform_residues(g, P.q[:9], P.N, 2) for _ in range(count)]
    scales = [2.0 ** 50 * (1.0 if i != 2 else 1.0 - 2.0 ** -6) for i in range(count)]
    got = ctx.poly_eval_bsgs_batch([ct_dev(c, s) for c, s in zip(cts, scales)], coeffs, m, key_dev(rlk, 0))
    for x, c, s in zip(got, cts, scales):
        want, so = o.poly_eval_bsgs(c, s, coeffs, rlk, m)
        assert x.level == want.shape[1] and x.scale == so and np.array_equal(host(x.data), want)
    want, so = o.poly_eval_tree(cts[0], scales[0], coeffs, rlk)
    x = ctx.poly_eval_tree(ct_dev(cts[0], scales[0]), coeffs, key_dev(rlk, 0))
    assert x.level == want.shape[1] and x.scale == so and np.array_equal(host(x.data), want)


def test_polynomial_batch_in_place():
    """Five ciphertexts (a run of four and one) in one array of descriptors for input and output, at a scale that multiplying and
    dividing by the dropped prime does not give back."""
    import ctypes as C
    import torch
    from paper_2609_12378_b200 import binding
    from oracle.ckks_oracle import Oracle
    from tests.gpu_util import GuardedContext, dev, host, key_dev
    N, r, primes = 1024, 1 + int(1.37 * 2.0 ** 49) // 2048 * 2048, []
    while len(primes) < 14:         # in the middle of the range: just below 2^50 every scale comes back
        if inputs.is_prime(r):
            primes.append(r)
        r += 2048
    qs, ps = (np.array(x, dtype=np.uint64) for x in (primes[:10], primes[10:]))
    o, ctx, g = Oracle(10, qs, ps, 3), GuardedContext(10, qs, ps, 3), inputs.rng(745, 0)
    rlk = inputs.uniform_residues(g, primes, N, 6).reshape(3, 2, 14, N)
    coeffs, m, level = g.uniform(-1, 1, 16), 4, 9
    cts = [inputs.uniform_residues(g, qs[:level], N, 2) for _ in range(5)]
    lc = o.poly_eval_bsgs(cts[0], 2.0 ** 50, coeffs, rlk, m)[0].shape[1]
    q = float(qs[lc])
    scale = next(s for s in 2.0 ** 50 * g.uniform(0.9, 1.1, 1000) if s * q / q != s)
    data, key = [dev(c) for c in cts], key_dev(rlk, 0)
    arr = (binding.CCt * 5)(*[binding.CCt(d.data_ptr(), level, 2, scale) for d in data])
    lib = binding.load()
    ws = torch.empty(lib.ckks_poly_eval_bsgs_batch_workspace_bytes(ctx._h, level, 15, m, 5), dtype=torch.uint8, device="cuda")
    ck = binding.CEvk(key.data.data_ptr(), 0)
    assert lib.ckks_poly_eval_bsgs_batch(ctx._h, arr, 5, (C.c_double * 16)(*coeffs), 15, m, C.byref(ck), arr, ws.data_ptr(), ws.numel(), None) == binding.OK
    for d, x, c in zip(data, arr, cts):
        want, so = o.poly_eval_bsgs(c, scale, coeffs, rlk, m)
        assert x.level == want.shape[1] and x.scale == so and so != scale
        assert np.array_equal(host(d).reshape(-1)[:want.size].reshape(want.shape), want)


@pytest.mark.parametrize("level", [1, 4, 6])
def test_products_and_rotations_in_place_and_unaligned(level):
    """Batches of 17 (a full chunk and one) whose results lie on their own operands or on another product's, rotations onto
    their own and each other's inputs, and operands that are only 8-byte aligned."""
    import torch
    from paper_2609_12378_b200 import binding
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(10, 6, 2, 3), context(10, 6, 2, 3)
    o, g = P.oracle, inputs.rng(750, level)
    allp = list(P.q) + list(P.p)
    key = inputs.uniform_residues(g, allp, P.N, 6).reshape(3, 2, 8, P.N)
    gal = o.galois_element(5)
    x = [inputs.uniform_residues(g, P.q[:level], P.N, 2) for _ in range(17)]
    y = [inputs.uniform_residues(g, P.q[:level], P.N, 2) for _ in range(17)]
    prod, rot = [o.mul_relin(a, b, key) for a, b in zip(x, y)], [o.rotate(a, key, gal) for a in x]

    def unaligned(a):
        buf = torch.zeros(a.size + 1, dtype=torch.int64, device="cuda").view(torch.uint64)
        t = buf[1:].view(*a.shape)
        t.copy_(torch.from_numpy(a))
        return binding.Ciphertext(t, 1.0)

    for put in (lambda a: ct_dev(a, 1.0), unaligned):
        for shift in (0, 1):        # results onto the same product's operand, or onto the next one's
            dx, dy = [put(a) for a in x], [put(b) for b in y]
            outs = dx[shift:] + dx[:shift]
            if shift == 0:
                ctx.mul_relin_batch(dx, dy, key_dev(key, 0), outs=outs)
            else:                   # the last result goes to an operand of the chunk before it, already used
                ctx.mul_relin_batch(dx[:16], dy[:16], key_dev(key, 0), outs=dx[1:16] + dx[:1])
                outs, want = dx[1:16] + dx[:1], prod[:16]
            for i, w in enumerate(prod if shift == 0 else want):
                assert np.array_equal(host(outs[i].data), w), (shift, i)
            dx = [put(a) for a in x[:16]]
            outs = dx[shift:] + dx[:shift]
            ctx.rotate_batch(dx, key_dev(key, gal), outs=outs)
            for i in range(16):
                assert np.array_equal(host(outs[i].data), rot[i]), (shift, i)
        assert np.array_equal(host(ctx.mul_relin(put(x[0]), put(y[0]), key_dev(key, 0)).data), prod[0])
        assert np.array_equal(host(ctx.rotate(put(x[0]), key_dev(key, gal)).data), rot[0])
        s = ctx.mul_relin_sum([put(a) for a in x], [put(b) for b in y], key_dev(key, 0))
        assert np.array_equal(host(s.data), o.mul_relin_sum(np.stack(x), np.stack(y), key))


@pytest.mark.parametrize("shift", [0, 1, 5])
def test_batches_whose_results_share_words(shift):
    """Sixteen products and rotations in one buffer whose results start `shift` limbs behind another product's operand (the last
    one's for the first result), and two results in one place: as if every operand had been read first and the results then
    written in order."""
    from paper_2609_12378_b200 import binding
    from tests.gpu_util import context, ct_dev, dev, host, key_dev
    P, ctx = params(13, 6, 1, 6), context(13, 6, 1, 6)
    o, g = P.oracle, inputs.rng(755, shift)
    n, level, N = 16, 6, P.N
    words = 2 * level * N
    key = inputs.uniform_residues(g, list(P.q) + list(P.p), N, 12).reshape(6, 2, 7, N)
    gal = o.galois_element(5)
    x = [inputs.uniform_residues(g, P.q, N, 2) for _ in range(n)]
    y = inputs.uniform_residues(g, P.q, N, 2)
    for place in ([n - 1] + list(range(n - 1)), [0, 1] + [3] * 2 + list(range(4, n))):
        for products in (True, False):
            flat = np.concatenate([a.reshape(-1) for a in x] + [np.zeros(words, dtype=np.uint64)])
            want = flat.copy()
            for a, p in zip(x, place):
                r = o.mul_relin(a, y, key) if products else o.rotate(a, key, gal)
                want[p * words + shift * N:(p + 1) * words + shift * N] = r.reshape(-1)
            buf = dev(flat)
            def cts(starts):
                return [binding.Ciphertext(buf[s:s + words].view(2, level, N), 1.0) for s in starts]
            ins, outs = cts(i * words for i in range(n)), cts(p * words + shift * N for p in place)
            if products:
                ctx.mul_relin_batch(ins, [ct_dev(y, 1.0)] * n, key_dev(key, 0), outs=outs)
            else:
                ctx.rotate_batch(ins, key_dev(key, gal), outs=outs)
            assert np.array_equal(host(buf), want), (place[0], products)


@pytest.mark.parametrize("log_n,batch,limbs", [(12, 1, 3), (12, 24, 3), (12, 25, 3), (13, 24, 3), (13, 25, 3), (14, 12, 3), (14, 13, 3)])
def test_transforms_at_the_cluster_limit(log_n, batch, limbs):
    """The last batch that one cluster per limb transforms and the first that goes in two passes: both directions."""
    from tests.gpu_util import context, dev, host
    P, ctx = params(log_n, 3, 1, 3), context(log_n, 3, 1, 3)
    x = inputs.uniform_residues(inputs.rng(770, log_n), P.q[:limbs], P.N, batch)
    assert np.array_equal(host(ctx.ntt(dev(x))), P.oracle.ntt(x))
    assert np.array_equal(host(ctx.intt(dev(x))), P.oracle.intt(x))


@pytest.mark.parametrize("d,S", [(64, 4), (64, 5), (64, 9), (64, 12), (64, 17)])
def test_multiply_accumulate_tile_widths(d, S):
    """Shard counts at which the multiply-accumulate changes between 8- and 16-column tiles, with partly filled tiles."""
    from tests.test_gpu_linear import _run
    _run(10, 3, 1, 3, 2, d, d, 8, S, 32, seed=780 + S, check_slots=False)


@pytest.mark.parametrize("lazy", [False, True])
@pytest.mark.parametrize("dnum,d_in,d_out,S,B", [
    (6, 128, 128, 1, 8),      # sixteen eager giants (fifteen rotations) in one pass, seven baby rotations in one
    (6, 64, 32, 3, 4),        # five giants per pass: a partial last pass; folded
    (3, 128, 128, 5, 4),      # lazy: two passes of the sum over four giants each
    (6, 64, 64, 17, 8),       # one giant per pass
    (8, 24, 16, 2, 4),        # eight digits; two input blocks
    (9, 16, 16, 2, 4),        # nine digits: one key at a time
])
def test_projection_passes_by_shard_count(dnum, d_in, d_out, S, B, lazy):
    """How many rotations share a pass depends on the number of shards and digits."""
    from tests.test_gpu_linear import _run
    _run(10, 9, -(-9 // dnum), dnum, 9, d_in, d_out, 4 if d_in > 24 else 32, S, B, seed=760 + S, check_slots=False, lazy=lazy)


@pytest.mark.parametrize("L,K,dnum,level", [(3, 1, 3, 3), (9, 9, 1, 9), (17, 17, 1, 16), (7, 4, 3, 5), (8, 1, 8, 8)])
def test_products_that_drop_a_limb(L, K, dnum, level):
    """ModDown and rescale in one step: one, two and three groups of eight special primes, full and partial digits, more digits
    than the unrolled inner products take, the lowest level; inputs at the ends of the residues."""
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(10, L, K, dnum), context(10, L, K, dnum)
    o, g = P.oracle, inputs.rng(770, level + 100 * L)
    x = inputs.uniform_residues(g, P.q[:level], P.N, 2)
    for i in range(level):
        x[:, i, ::7] = int(P.q[i]) - 1
    rlk = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, dnum * 2).reshape(dnum, 2, L + K, P.N)
    coeffs = [0.25, -0.5, 0.75]
    want, so = o.poly_eval(x, 2.0 ** 50, coeffs, rlk)
    got = ctx.poly_eval(ct_dev(x, 2.0 ** 50), coeffs, key_dev(rlk, 0))
    assert got.scale == so and np.array_equal(host(got.data), want)


@pytest.mark.parametrize("dnum", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("level", [9, 10])
def test_hoisted_rotations_with_and_without_a_stored_inner_product(dnum, level):
    """Sixteen rotations at N = 2^13: at ten limbs and up to four digits they form the inner product in the last row pass, at nine
    limbs or with five digits in a launch of its own."""
    from tests.gpu_util import context, ct_dev, host, key_dev
    K = -(-10 // dnum)
    P, ctx = params(13, 10, K, dnum), context(13, 10, K, dnum)
    o, g = P.oracle, inputs.rng(780, level + 100 * dnum)
    ct = inputs.uniform_residues(g, P.q[:level], P.N, 2)
    keys = [inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, dnum * 2).reshape(dnum, 2, 10 + K, P.N) for _ in range(16)]
    gs = [o.galois_element(r) for r in range(1, 17)]
    got = ctx.rotate_hoisted(ct_dev(ct, 1.0), [key_dev(k, e) for k, e in zip(keys, gs)])
    for x, want in zip(got, o.rotate_hoisted(ct, keys, gs)):
        assert np.array_equal(host(x.data), want)


@pytest.mark.parametrize("dnum,level", [(1, 21), (3, 22), (4, 22), (3, 19), (5, 22), (5, 19)])
def test_large_product_with_and_without_a_stored_inner_product(dnum, level):
    """x^2 at N = 2^16 with one to four digits, whose inner product is formed between the row passes and never stored for the limbs that
    ModDown converts, and with five, whose sum is."""
    from tests.gpu_util import context, ct_dev, host, key_dev
    K = -(-22 // dnum)
    P, ctx = params(16, 22, K, dnum), context(16, 22, K, dnum)
    o, g = P.oracle, inputs.rng(790, level + 100 * dnum)
    x = inputs.uniform_residues(g, P.q[:level], P.N, 2)
    rlk = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, dnum * 2).reshape(dnum, 2, 22 + K, P.N)
    want, so = o.poly_eval(x, 2.0 ** 50, [0.0, 0.5, 1.0], rlk)
    got = ctx.poly_eval(ct_dev(x, 2.0 ** 50), [0.0, 0.5, 1.0], key_dev(rlk, 0))
    assert got.scale == so and np.array_equal(host(got.data), want)


@pytest.mark.parametrize("share", [0, 1, 4, 7])
def test_integer_transforms_give_the_same_limbs(share):
    """N = 2^16 with some or all limbs on the integer transform: nine limbs both ways, rescales of one to three components (their
    dropped limbs lie a whole component apart) with a workspace and without, of four ciphertexts at once behind a projection,
    and a rotation whose ModUp takes the transform's plain output."""
    from paper_2609_12378_b200 import binding
    from tests.gpu_util import context, ct_dev, dev, host, key_dev
    from tests.test_gpu_linear import _run
    from tests.test_zz_no_alloc import _call_static
    P, ctx = params(16, 9, 3, 3), context(16, 9, 3, 3)
    o, g = P.oracle, inputs.rng(800, share)
    x = inputs.uniform_residues(g, P.q[:9], P.N, 3)
    key = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, 6).reshape(3, 2, 12, P.N)
    gal = o.galois_element(5)
    ctx.set_option(binding.OPT_NTT_FP_SHARE, share)
    try:
        assert np.array_equal(host(ctx.ntt(dev(x))), o.ntt(x))
        assert np.array_equal(host(ctx.intt(dev(x))), o.intt(x))
        for ncomp in (1, 2):
            assert np.array_equal(host(ctx.rescale(ct_dev(x[:ncomp], 1.0)).data), o.rescale(x[:ncomp])), ncomp
        short = np.ascontiguousarray(x[:, :2])
        out = dev(np.zeros((3, 1, P.N), dtype=np.uint64))
        assert _call_static(ctx, dev(short), 2, 3, 1.0, out)[0] == binding.OK
        assert np.array_equal(host(out), o.rescale(short))
        _run(16, 9, 3, 3, 2, 4, 4, 8192, 4, 2, seed=801, check_slots=False)
        ctx.set_option(binding.OPT_CONV_KERNEL, binding.CONV_TENSOR)
        assert np.array_equal(host(ctx.rotate(ct_dev(x[:2], 1.0), key_dev(key, gal)).data), o.rotate(x[:2], key, gal))
    finally:
        ctx.set_option(binding.OPT_CONV_KERNEL, binding.CONV_FP64)
        ctx.set_option(binding.OPT_NTT_FP_SHARE, 8)


@pytest.mark.parametrize("share", [1, 7])
def test_transforms_that_leave_out_every_limb_of_one_path(share):
    """One limb and one special prime with the tensor-core ModUp: at share 1 the FP64 transform of the extended digits has the
    digit's own limb alone, which it skips, and the integer one all the rest; eight rotations in a row without a pause."""
    from paper_2609_12378_b200 import binding
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(16, 3, 1, 3), context(16, 3, 1, 3)
    o, g = P.oracle, inputs.rng(810, share)
    x = inputs.uniform_residues(g, P.q[:1], P.N, 2)
    key = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, 6).reshape(3, 2, 4, P.N)
    gal = o.galois_element(5)
    ctx.set_option(binding.OPT_NTT_FP_SHARE, share)
    ctx.set_option(binding.OPT_CONV_KERNEL, binding.CONV_TENSOR)
    try:
        ct, k = ct_dev(x, 1.0), key_dev(key, gal)
        for _ in range(8):
            ct = ctx.rotate(ct, k)
        want = x
        for _ in range(8):
            want = o.rotate(want, key, gal)
        assert np.array_equal(host(ct.data), want)
    finally:
        ctx.set_option(binding.OPT_CONV_KERNEL, binding.CONV_FP64)
        ctx.set_option(binding.OPT_NTT_FP_SHARE, 8)


def test_key_switches_of_one_key_take_the_integer_share():
    """With the tensor-core conversions a rotation's transforms are plain ones, so that the share of limbs on the integer transform applies
    to them as it does in a hoisted rotation: the same number of launches."""
    from paper_2609_12378_b200 import binding
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(16, 3, 1, 3), context(16, 3, 1, 3)
    o, g = P.oracle, inputs.rng(815, 0)
    x = inputs.uniform_residues(g, P.q[:2], P.N, 2)
    key = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, 6).reshape(3, 2, 4, P.N)
    gal = o.galois_element(5)
    want, count = o.rotate(x, key, gal), []
    ctx.set_option(binding.OPT_CONV_KERNEL, binding.CONV_TENSOR)
    ctx.set_option(binding.OPT_NTT_FP_SHARE, 4)
    try:
        for call in (lambda: ctx.rotate_hoisted(ct_dev(x, 1.0), [key_dev(key, gal)])[0], lambda: ctx.rotate(ct_dev(x, 1.0), key_dev(key, gal))):
            before = binding.kernel_launches()
            got = call()
            count.append(binding.kernel_launches() - before)
            assert np.array_equal(host(got.data), want)
    finally:
        ctx.set_option(binding.OPT_CONV_KERNEL, binding.CONV_FP64)
        ctx.set_option(binding.OPT_NTT_FP_SHARE, 8)
    assert count[0] == count[1]


@pytest.mark.parametrize("log_n,L,K,dnum,level", [
    (12, 3, 1, 3, 3), (12, 8, 8, 1, 8), (12, 9, 9, 1, 9), (12, 7, 4, 3, 5), (12, 12, 3, 4, 12), (12, 10, 2, 5, 10), (12, 16, 8, 2, 11),
    (13, 12, 6, 2, 12), (14, 6, 2, 3, 5), (14, 16, 8, 2, 16), (15, 12, 4, 3, 9), (15, 8, 8, 1, 8), (16, 3, 3, 1, 3), (16, 10, 5, 2, 6)])
def test_key_switches_of_every_ring_and_digit_size(log_n, L, K, dnum, level):
    """One to nine sources per conversion, full and partial digits, one to five digits (four are the most whose row pass forms the inner
    product): a rotation whose sources lie at the ends of the residues, a sum of rotations over two groups of terms, a product that drops a
    limb and a rescale, all of it on one ciphertext and on several.  At N = 2^14 and 2^15 the ModUps run in strips, at 2^15 the ModDowns
    too; test_gpu_strips.py has the batches that do so on the other rings."""
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(log_n, L, K, dnum), context(log_n, L, K, dnum)
    o, g = P.oracle, inputs.rng(800, level + 100 * L + 10000 * log_n)
    alpha = -(-L // dnum)
    d = np.empty((1, level, P.N), dtype=np.uint64)
    for i in range(level):
        q, lo = int(P.q[i]), i // alpha * alpha
        hat = 1
        for b in range(lo, min(lo + alpha, level)):
            hat = hat * (int(P.q[b]) if b != i else 1) % q
        ends = np.array([y * hat % q for y in (0, 1, q - 1, q // 2, q // 2 + 1)], dtype=np.uint64)
        d[0, i] = ends[g.integers(0, 5, P.N)]
        d[0, i, :64] = ends[3 + np.arange(64) % 2]          # all sources at q / 2 together
    ct = np.concatenate([inputs.uniform_residues(g, P.q[:level], P.N, 1), o.ntt(d)])
    more = [inputs.uniform_residues(g, P.q[:level], P.N, 2) for _ in range(4)]
    keys = [inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, dnum * 2).reshape(dnum, 2, L + K, P.N) for _ in range(3)]
    gals = [o.galois_element(r) for r in (3, 64, P.n - 1)]
    dk = [key_dev(k, e) for k, e in zip(keys, gals)]
    assert np.array_equal(host(ctx.rotate(ct_dev(ct, 1.0), dk[0]).data), o.rotate(ct, keys[0], gals[0]))
    batch = ctx.rotate_batch([ct_dev(x, 1.0) for x in [ct] + more], dk[1])
    for got, x in zip(batch, [ct] + more):
        assert np.array_equal(host(got.data), o.rotate(x, keys[1], gals[1]))
    pick = [0, 1, 2, 0, 1]
    got = ctx.rotate_sum([ct_dev(x, 1.0) for x in [ct] + more], [dk[j] for j in pick])
    assert np.array_equal(host(got.data), o.rotate_sum(np.stack([ct] + more), [keys[j] for j in pick], [gals[j] for j in pick]))
    if level < 3:
        return
    coeffs = [0.25, -0.5, 0.75]
    for xs in ([ct], [ct] + more[:2]):
        outs = [ctx.poly_eval(ct_dev(x, 2.0 ** 50), coeffs, key_dev(keys[0], 0)) for x in xs]
        for got, x in zip(outs, xs):
            assert np.array_equal(host(got.data), o.poly_eval(x, 2.0 ** 50, coeffs, keys[0])[0])
    prod = ctx.mul_relin(ct_dev(ct, 1.0), ct_dev(more[0], 1.0), key_dev(keys[2], 0))
    want = o.mul_relin(ct, more[0], keys[2])
    assert np.array_equal(host(prod.data), want)
    assert np.array_equal(host(ctx.rescale(prod).data), o.rescale(want))


@pytest.mark.parametrize("log_n,batch,limbs", [(10, 1, 1), (12, 74, 3), (12, 75, 3), (15, 9, 3), (15, 14, 2), (16, 13, 1), (16, 7, 2)])
def test_transforms_on_either_side_of_a_row_per_warp(log_n, batch, limbs):
    """Both directions with the most limbs whose rows are taken by a warp each (six CTAs of four rows per SM of 148) and the fewest
    that are taken by half a warp each, in a buffer that is 16-byte aligned and in one that is not."""
    import torch
    from tests.gpu_util import context, host
    P, ctx = params(log_n, 3, 1, 3), context(log_n, 3, 1, 3)
    o, g = P.oracle, inputs.rng(810, log_n + 100 * batch)
    x = inputs.uniform_residues(g, P.q[:limbs], P.N, batch)
    x[0] = np.array([int(q) - 1 for q in P.q[:limbs]], dtype=np.uint64)[:, None]
    fwd, inv = o.ntt(x), o.intt(x)
    for offset in (0, 1):
        buf = torch.zeros(x.size + 1, dtype=torch.int64, device="cuda").view(torch.uint64)
        y = buf[offset:offset + x.size].view(batch, limbs, P.N)
        y.copy_(torch.from_numpy(x))
        assert np.array_equal(host(ctx.ntt(y)), fwd)
        y.copy_(torch.from_numpy(x))
        assert np.array_equal(host(ctx.intt(y)), inv)


@pytest.mark.parametrize("log_n,L,K,dnum,level", [(12, 4, 4, 1, 4), (13, 6, 1, 6, 4), (14, 8, 2, 4, 8), (15, 16, 4, 4, 13), (15, 16, 4, 4, 12), (15, 12, 4, 3, 10), (15, 12, 4, 3, 9)])
def test_sums_of_rotations_whose_terms_share_a_row_or_not(log_n, L, K, dnum, level):
    """Two terms, which follow one another in the kernel between the column passes on every ring, and five, which do so from three CTAs per
    SM on and otherwise have their digits transformed by a launch before the inner product: one to four digits, a partial one among
    them, on either side of the line."""
    import torch
    from paper_2609_12378_b200 import binding
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(log_n, L, K, dnum), context(log_n, L, K, dnum)
    o, g = P.oracle, inputs.rng(820, level + 100 * L + 10000 * log_n)
    cts = [inputs.uniform_residues(g, P.q[:level], P.N, 2) for _ in range(5)]
    keys = [inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, dnum * 2).reshape(dnum, 2, L + K, P.N) for _ in range(5)]
    gals = [o.galois_element(r) for r in (1, 5, 64, 3, P.n - 1)]
    dcts, dkeys = [ct_dev(x, 1.0) for x in cts], [key_dev(k, e) for k, e in zip(keys, gals)]
    launches = []
    for n in (2, 5):
        before = binding.kernel_launches()
        got = ctx.rotate_sum(dcts[:n], dkeys[:n])
        launches.append(binding.kernel_launches() - before)
        assert np.array_equal(host(got.data), o.rotate_sum(np.stack(cts[:n]), keys[:n], gals[:n]))
    one_kernel = (P.N >> 10) * (level + K) >= 3 * torch.cuda.get_device_properties(0).multi_processor_count
    assert launches[1] - launches[0] == (1 if one_kernel else 2)      # five terms take two passes


@pytest.mark.parametrize("L,K,dnum,level,separate", [(3, 1, 3, 3, (7, 8, 9)), (10, 8, 2, 9, (7,)), (24, 8, 3, 24, ())])
def test_last_wave_of_the_strips(L, K, dnum, level, separate):
    """Hoisted rotations at N = 2^16 whose strips (64 per rotation, on 148 SMs) fill three waves and a bit to six waves and a bit: whole strips
    and strips cut into chunks in one grid.  Where most of the last wave would be idle the separate kernels run, two launches more."""
    import torch
    from paper_2609_12378_b200 import binding
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(16, L, K, dnum), context(16, L, K, dnum)
    o, g = P.oracle, inputs.rng(840, level)
    ct = inputs.uniform_residues(g, P.q[:level], P.N, 2)
    keys = [inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, dnum * 2).reshape(dnum, 2, L + K, P.N) for _ in range(3)] * 5
    gals = [o.galois_element(r) for r in range(1, 16)]
    want = o.rotate_hoisted(ct, keys[:14], gals[:14])
    data, count = [key_dev(k, 0).data for k in keys[:3]], {}
    dkeys = [binding.SwitchKey(data[i % 3], e) for i, e in enumerate(gals)]
    for n in (6, 7, 8, 9, 14):
        before = binding.kernel_launches()
        got = ctx.rotate_hoisted(ct_dev(ct, 1.0), dkeys[:n])
        count[n] = binding.kernel_launches() - before
        for x, w in zip(got, want):
            assert np.array_equal(host(x.data), w)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert [n for n in (7, 8, 9, 14) if count[n] == count[14] + 2] == list(separate), count


FEWER_REGISTERS = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <cuda_runtime_api.h>
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *f) {
    cudaError_t (*real)(struct cudaFuncAttributes *, const void *) = dlsym(dlopen("libcudart.so.12", RTLD_LAZY | RTLD_NOLOAD), "cudaFuncGetAttributes");
    cudaError_t e = real(a, f);
    a->numRegs -= 32;
    return e;
}
"""
ROTATE_ONCE = """
import numpy as np
from paper_2609_12378_b200 import binding, inputs
from tests.gpu_util import context, ct_dev, host, key_dev
from tests.harness import params
P, ctx = params(15, 4, 2, 2), context(15, 4, 2, 2)
g = inputs.rng(830, 0)
x = inputs.uniform_residues(g, P.q, P.N, 2)
key = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, 4).reshape(2, 2, 6, P.N)
before = binding.kernel_launches()
y = host(ctx.rotate(ct_dev(x, 1.0), key_dev(key, P.oracle.galois_element(3))).data)
assert np.array_equal(y, P.oracle.rotate(x, key, P.oracle.galois_element(3)))
print(binding.kernel_launches() - before)
"""


def test_context_without_the_registers_of_the_strip_kernel(tmp_path):
    """A library whose strip kernels were compiled to other registers than their roles share out (here: whose runtime says so) makes
    contexts all the same and takes the separate kernels: the same rotation in more launches."""
    import os
    import subprocess
    import sys
    src, lib, root = tmp_path / "regs.c", tmp_path / "regs.so", os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src.write_text(FEWER_REGISTERS)
    subprocess.run(["gcc", "-shared", "-fPIC", "-I/usr/local/cuda/include", str(src), "-o", str(lib), "-ldl"], check=True)
    count = [int(subprocess.run([sys.executable, "-c", ROTATE_ONCE], cwd=root, env={**os.environ, **env}, check=True, stdout=subprocess.PIPE, timeout=300).stdout)
             for env in ({}, {"LD_PRELOAD": " ".join([str(lib), os.environ.get("LD_PRELOAD", "")]).strip()})]
    assert count[0] == 5 and count[1] > 5
