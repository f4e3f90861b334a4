"""Conversions in strips (an inverse column pass, a basis conversion and a forward column pass in one kernel) against the separate kernels and
the checker, in batches that are large enough for them: sixteen rotations, nine hoisted ones and a polynomial of four ciphertexts, whose products
drop a limb four, eight and sixteen at a time, with one to eight sources, full and partial digits, on every ring that has the kernel.  A child
process whose CUDA runtime reports other registers than the kernel needs computes the same without strips; a conversion in a strip is
two launches less (one or none less where hoisted rotations on a small ring have a transform in one launch otherwise)."""
import hashlib
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2609_12378_b200 import binding, inputs
from tests.harness import params

pytestmark = pytest.mark.gpu

# log_n, L, K, dnum, level; launches that the three calls save (on 148 SMs)
CASES = [((12, 6, 1, 6, 6), (2, 1, 4)), ((12, 6, 2, 3, 6), (2, 1, 4)), ((12, 6, 3, 2, 6), (2, 1, 4)),
         ((12, 8, 4, 2, 7), (2, 1, 4)), ((12, 8, 8, 1, 8), (2, 2, 4)), ((13, 6, 1, 6, 6), (2, 1, 6)),
         ((13, 7, 2, 4, 7), (2, 1, 6)), ((13, 8, 4, 2, 8), (2, 1, 6)), ((13, 7, 7, 1, 7), (2, 2, 6)),
         ((14, 6, 1, 6, 6), (4, 2, 12)), ((14, 7, 4, 2, 7), (4, 2, 12)), ((14, 16, 8, 2, 11), (4, 3, 12)),
         ((15, 8, 2, 4, 8), (4, 4, 12)), ((15, 12, 6, 2, 9), (4, 4, 12)), ((16, 6, 1, 6, 6), (4, 0, 8)),
         ((16, 7, 2, 4, 7), (4, 0, 8)), ((16, 6, 3, 2, 6), (4, 0, 4)), ((16, 9, 4, 3, 9), (4, 2, 6)),
         ((16, 10, 5, 2, 8), (4, 2, 6)), ((16, 12, 6, 2, 12), (4, 2, 8)), ((16, 9, 7, 2, 9), (4, 2, 6)),
         ((16, 16, 8, 2, 12), (4, 2, 8))]


def run(log_n, L, K, dnum, level):
    """[launches, digest of the results] of each call, and what they were given and gave."""
    from tests.gpu_util import context, ct_dev, host, key_dev
    P, ctx = params(log_n, L, K, dnum), context(log_n, L, K, dnum)
    g = inputs.rng(850, level + 100 * L + 10000 * log_n)
    cts = list(inputs.uniform_residues(g, P.q[:level], P.N, 32).reshape(16, 2, level, P.N))
    keys = inputs.uniform_residues(g, list(P.q) + list(P.p), P.N, 3 * dnum * 2).reshape(3, dnum, 2, L + K, P.N)
    gals = [P.oracle.galois_element(r) for r in range(1, 10)]
    coeffs = [0.5 / (k + 1) for k in range(9)]
    dcts, data = [ct_dev(x, 2.0 ** 50) for x in cts], [key_dev(k, 0).data for k in keys]
    calls = [lambda: ctx.rotate_batch(dcts, binding.SwitchKey(data[0], gals[4])),
             lambda: ctx.rotate_hoisted(dcts[0], [binding.SwitchKey(data[i % 3], e) for i, e in enumerate(gals)]),
             lambda: ctx.poly_eval_bsgs_batch(dcts[:4], coeffs, 8, binding.SwitchKey(data[1], 0))]
    seen, results = [], []
    for call in calls:
        before = binding.kernel_launches()
        out = call()
        launches = binding.kernel_launches() - before
        results.append([host(x.data) for x in out])
        seen.append([launches, hashlib.sha256(b"".join(x.tobytes() for x in results[-1])).hexdigest()])
    return seen, (P.oracle, cts, keys, gals, coeffs), results


@pytest.fixture(scope="module")
def without_strips(tmp_path_factory):
    from tests.test_gpu_shapes import FEWER_REGISTERS
    where, root = tmp_path_factory.mktemp("strips"), os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    (where / "regs.c").write_text(FEWER_REGISTERS)
    subprocess.run(["gcc", "-shared", "-fPIC", "-I/usr/local/cuda/include", str(where / "regs.c"), "-o", str(where / "regs.so"), "-ldl"], check=True)
    code = "import json\nfrom tests import test_gpu_strips as t\nprint(json.dumps([t.run(*c)[0] for c, _ in t.CASES]))"
    env = {**os.environ, "LD_PRELOAD": " ".join([str(where / "regs.so"), os.environ.get("LD_PRELOAD", "")]).strip()}
    out = subprocess.run([sys.executable, "-c", code], cwd=root, env=env, check=True, stdout=subprocess.PIPE, timeout=600).stdout
    return json.loads(out.splitlines()[-1])


@pytest.mark.parametrize("index", range(len(CASES)), ids=["-".join(map(str, c)) for c, _ in CASES])
def test_strips_and_separate_kernels_agree(index, without_strips):
    import torch
    case, saved = CASES[index]
    seen, (o, cts, keys, gals, coeffs), (batch, hoisted, poly) = run(*case)
    for (_, got), (_, want) in zip(seen, without_strips[index]):
        assert got == want
    for i in (0, 15):
        assert np.array_equal(batch[i], o.rotate(cts[i], keys[0], gals[4]))
    assert np.array_equal(hoisted[8], o.rotate(cts[0], keys[2], gals[8]))
    assert np.array_equal(poly[3], o.poly_eval_bsgs(cts[3], 2.0 ** 50, coeffs, keys[1], 8)[0])
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert [a - b for (b, _), (a, _) in zip(seen, without_strips[index])] == list(saved)
