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
