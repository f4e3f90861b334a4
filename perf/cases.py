"""Performance cases of the CKKS layer: what a server-side program has the library do, through paper_2609_12378_b200.binding.

Every case is one call (or the two calls that always come together) of the public API on inputs that are already on the GPU.
Ciphertexts and switching keys are uniform residues, which is what real ones look like to the kernels; weights, slot values
and polynomial coefficients are doubles of the size real ones have.  Every result is a whole number and has to be the same
bit for bit.

Parameter sets (ring exponent: ciphertext primes, special primes, key-switch digits): 16 is the set of the benchmark and of
the Llama-3-8B shapes, 13 the toy projection's, 14 and 15 are the sizes between them at the same security margin.
"""
import functools
import math

import torch

from paper_2609_12378_b200 import binding, inputs

PARAMS = {13: (6, 1, 6), 14: (6, 2, 3), 15: (12, 4, 3), 16: (24, 8, 3)}
SCALE = 2.0 ** 40


# ---------------------------------------------------------------------------------------------------------------- cases
def listed():
    return [
        # the two components of one toy-ring ciphertext, one way and the other: the smallest transform call there is
        {"name": "ntt_ring13", "op": "ntt", "log_n": 13, "batch": 2, "limbs": 6},
        # the NTT micro-benchmark: 32 polynomials of 24 limbs, one buffer forward and one back
        {"name": "ntt_32x24", "op": "ntt", "log_n": 16, "batch": 32, "limbs": 24},
        # weight diagonals encoded for a ciphertext-plaintext product: one baby-step group of a projection
        {"name": "encode_64", "op": "encode", "log_n": 16, "batch": 64, "level": 24},
        # one rotation of one ciphertext, a complete key switch: the unit of every rotate-and-add ladder
        {"name": "rotate_one", "op": "rotate", "log_n": 16, "level": 24},
        # 64 rotations of one ciphertext off a shared ModUp: the baby steps of a matrix product
        {"name": "rotate_hoisted_64", "op": "hoisted", "log_n": 16, "level": 24, "rotations": 64},
        # ciphertext x ciphertext product with relinearisation and rescale in the middle of the modulus chain, where the last
        # key-switch digit is partial
        {"name": "mul_rescale_level17", "op": "mul", "log_n": 16, "level": 17},
        # the same on a small ring: launches and latency
        {"name": "mul_rescale_ring14", "op": "mul", "log_n": 14, "level": 6},
        # an activation polynomial of the degree the paper gives SiLU, on one ciphertext
        {"name": "poly_degree63", "op": "poly", "log_n": 16, "level": 24, "count": 1, "degree": 63, "block": 8},
        # the toy projection: one ciphertext of 32 tokens x 64 features times 64 x 64
        {"name": "projection_toy", "op": "projection", "log_n": 13, "level": 6, "d_in": 64, "d_out": 64, "tokens": 32, "shards": 1,
         "baby": 8, "lazy": False},
        # 128 tokens through a 4096 x 4096 projection (query, output), the headline workload
        {"name": "projection_4096", "op": "projection", "log_n": 16, "level": 24, "d_in": 4096, "d_out": 4096, "tokens": 8, "shards": 16,
         "baby": 64, "lazy": True},
        # a short prompt (24 tokens: 3 shards) through the narrower key/value projection, which folds its result, with the
        # library's default schedule
        {"name": "projection_kv_24tokens", "op": "projection", "log_n": 16, "level": 24, "d_in": 4096, "d_out": 1024, "tokens": 8, "shards": 3,
         "baby": 64, "lazy": False},
        # scores, Softmax and probability x value of 128 tokens and 32 heads, 64 channels
        {"name": "attention_128tokens", "op": "attention", "log_n": 16, "level": 24, "tokens": 128, "heads": 32, "diag_block": 8,
         "group_baby": 4, "dim": 64},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["ntt", "ntt", "encode", "rotate", "hoisted", "mul", "mul", "poly", "projection", "projection", "attention"])
    log_n = rng.choice([13, 14, 15, 16, 16, 16])
    L = PARAMS[log_n][0]
    if op == "ntt":
        limbs = rng.randint(1, L)
        return {"op": op, "log_n": log_n, "batch": _log_uniform(rng, 1, 32), "limbs": limbs}
    if op == "encode":
        return {"op": op, "log_n": log_n, "batch": _log_uniform(rng, 1, 96), "level": rng.randint(1, L)}
    if op == "rotate":
        return {"op": op, "log_n": log_n, "level": rng.randint(1, L)}
    if op == "hoisted":
        return {"op": op, "log_n": log_n, "level": rng.randint(2, L), "rotations": _log_uniform(rng, 2, 64)}
    if op == "mul":
        return {"op": op, "log_n": log_n, "level": rng.randint(2, L)}
    if op == "poly":
        log_n = rng.choice([15, 16])
        level = rng.randint(10, PARAMS[log_n][0])
        return {"op": op, "log_n": log_n, "level": level, "count": rng.randint(1, 4), "degree": rng.randint(8, 63), "block": rng.choice([4, 8])}
    if op == "projection":
        lazy = rng.random() < 0.5
        if rng.random() < 0.4:      # small rings and matrices
            log_n = rng.choice([13, 14, 15])
            width = rng.choice([64, 128, 256])
            slots = 1 << (log_n - 1)
            return {"op": op, "log_n": log_n, "level": rng.randint(2, PARAMS[log_n][0]), "d_in": width, "d_out": width // rng.choice([1, 1, 2]),
                    "tokens": rng.choice([t for t in (4, 8, 16, 32) if t * width <= slots]), "shards": rng.randint(1, 4),
                    "baby": rng.choice([8, 16, 32]), "lazy": lazy}
        d_in, d_out = rng.choice([(4096, 4096), (4096, 1024), (4096, 2048), (2048, 2048), (1024, 4096), (6144, 4096)])
        return {"op": op, "log_n": 16, "level": rng.randint(8, 24), "d_in": d_in, "d_out": d_out, "tokens": 8, "shards": rng.randint(1, 10),
                "baby": rng.choice([32, 64]), "lazy": lazy}
    tokens = rng.choice([32, 64, 128])
    return {"op": op, "log_n": 16, "level": rng.randint(17, 24), "tokens": tokens, "heads": 32, "diag_block": rng.choice([4, 8]),
            "group_baby": rng.choice([1, 2, 4]), "dim": _log_uniform(rng, 4, 48)}


# -------------------------------------------------------------------------------------------------------------- prepare
@functools.lru_cache(maxsize=None)
def _context(log_n):
    """The context of a parameter set: a program builds it once and keeps it."""
    num_q, num_p, dnum = PARAMS[log_n]
    q, p = inputs.prime_chain(log_n, num_q, num_p)
    return binding.Context(log_n, q, p, dnum)


class _Source:
    """Seeded residues, keys and doubles on the GPU."""

    def __init__(self, ctx, seed):
        self.ctx, self.primes = ctx, ctx.q + ctx.p
        self.gen = torch.Generator(device=ctx.device)
        self.gen.manual_seed(seed)

    def residues(self, primes, *lead):
        out = torch.empty((*lead, len(primes), self.ctx.N), dtype=torch.int64, device=self.ctx.device)
        for i, m in enumerate(primes):
            out[..., i, :] = torch.randint(0, m, (*lead, self.ctx.N), generator=self.gen, device=self.ctx.device, dtype=torch.int64)
        return out.view(torch.uint64)

    def ciphertexts(self, count, level, scale=SCALE):
        return [binding.Ciphertext(x, scale) for x in self.residues(self.primes[:level], count, 2)]

    def keys(self, galois):
        data = self.residues(self.primes, len(galois), self.ctx.dnum, 2)
        return [binding.SwitchKey(k, g) for k, g in zip(data, galois)]

    def rotation_keys(self, rotations):
        return self.keys([self.ctx.galois_element(r) for r in rotations])

    def normal(self, shape, std):
        return torch.randn(shape, generator=self.gen, device=self.ctx.device, dtype=torch.float64) * std


def prepare(case, seed):
    ctx = _context(case["log_n"])
    src = _Source(ctx, seed)
    op, s = case["op"], {"case": case, "ctx": ctx}
    level = case.get("level")
    if op == "ntt":
        s["forward"] = src.residues(ctx.q[:case["limbs"]], case["batch"])
        s["backward"] = src.residues(ctx.q[:case["limbs"]], case["batch"])
    elif op == "encode":
        s["values"] = src.normal((case["batch"], ctx.n), 0.02)
        s["scale"] = float(ctx.q[level - 1])
    elif op == "rotate":
        s["ct"] = src.ciphertexts(1, level)[0]
        s["key"] = src.rotation_keys([8])[0]
    elif op == "hoisted":
        s["ct"] = src.ciphertexts(1, level)[0]
        s["keys"] = src.rotation_keys([8 * b for b in range(1, case["rotations"] + 1)])
    elif op == "mul":
        s["a"], s["b"] = src.ciphertexts(2, level)
        s["rlk"] = src.keys([0])[0]
    elif op == "poly":
        s["cts"] = src.ciphertexts(case["count"], level, 2.0 ** 50)
        s["coeffs"] = [0.5 * math.cos(1.7 * k + 0.3) / (k + 1) for k in range(case["degree"] + 1)]
        s["rlk"] = src.keys([0])[0]
    elif op == "projection":
        d_in, d_out = case["d_in"], case["d_out"]
        blocks = -(-d_in // (ctx.n // case["tokens"]))
        s["cts"] = src.ciphertexts(case["shards"] * blocks, level)
        s["keys"] = src.rotation_keys(ctx.linear_proj_rotations(d_in, d_out, case["tokens"], case["shards"], case["baby"]))
        s["W"] = src.normal((d_in, d_out), 0.02)
    else:
        dim = case["dim"]
        cts = src.ciphertexts(3 * dim, level, 2.0 ** 50)
        s["q"], s["k"], s["v"] = cts[:dim], cts[dim:2 * dim], cts[2 * dim:]
        s["shape"] = (case["tokens"], case["heads"], case["diag_block"])
        s["group_baby"] = min(case["group_baby"], case["tokens"] // case["diag_block"])
        s["keys"] = src.rotation_keys(ctx.attention_rotations(*s["shape"], group_baby=s["group_baby"]))
        s["rlk"] = src.keys([0])[0]
        # one doubling round with degree-4 polynomials: exp on [-4, 0] / 2 and an inverse square root
        s["exp"] = [1.0, 0.5, 0.125, 0.0208, 0.0026]
        s["rsqrt"] = [[2.1, -1.9, 1.2, -0.4, 0.05]]
    return s


# ------------------------------------------------------------------------------------------------------------------ run
def _words(t):
    """A result as signed words (a view: few torch operators take unsigned ones)."""
    return t.view(torch.int64)


def run(s):
    case, ctx = s["case"], s["ctx"]
    op = case["op"]
    if op == "ntt":
        return [_words(ctx.ntt(s["forward"])), _words(ctx.intt(s["backward"]))]
    if op == "encode":
        return _words(ctx.encode(s["values"], None, s["scale"], case["level"]))
    if op == "rotate":
        return _words(ctx.rotate(s["ct"], s["key"]).data)
    if op == "hoisted":
        return [_words(o.data) for o in ctx.rotate_hoisted(s["ct"], s["keys"])]
    if op == "mul":
        return _words(ctx.rescale(ctx.mul_relin(s["a"], s["b"], s["rlk"])).data)
    if op == "poly":
        if len(s["cts"]) == 1:
            return _words(ctx.poly_eval_bsgs(s["cts"][0], s["coeffs"], case["block"], s["rlk"]).data)
        return [_words(o.data) for o in ctx.poly_eval_bsgs_batch(s["cts"], s["coeffs"], case["block"], s["rlk"])]
    if op == "projection":
        return [_words(o.data) for o in ctx.linear_proj(s["cts"], s["W"], s["keys"], case["d_in"], case["d_out"], case["tokens"], case["shards"],
                                                case["baby"], lazy_moddown=case["lazy"])]
    return [_words(o.data) for o in ctx.attention(s["q"], s["k"], s["v"], 0.0, 1, s["exp"], s["rsqrt"], s["rlk"], s["keys"], *s["shape"],
                                          group_baby=s["group_baby"])]


# ----------------------------------------------------------------------------------------------------------------- work
# Operations: a modular product of two words of 50 bits is six double-precision operations (product, its error, quotient and
# remainder), a butterfly two more, a product added to a sum one more.
class _Work:
    def __init__(self, log_n):
        self.N, (self.L, self.K, self.dnum) = 1 << log_n, PARAMS[log_n]
        self.alpha = -(-self.L // self.dnum)
        self.limb = 8 * self.N
        self.butterflies = 8 * (self.N // 2) * log_n          # operations of one limb's transform
        self.pair = 7 * self.N                                # operations of one product and sum per coefficient
        self.flops = 0.0
        self.bytes = 0.0

    def key(self, level):
        """Bytes of the limbs of one switching key that a level uses."""
        return -(-level // self.alpha) * 2 * (level + self.K) * self.limb

    def ct(self, level):
        return 2 * level * self.limb

    def ntts(self, limbs, count=1):
        self.flops += count * limbs * self.butterflies

    def modup(self, level, count=1):
        nt = level + self.K
        own = [min(self.alpha, level - lo) for lo in range(0, level, self.alpha)]
        self.ntts(level + sum(nt - d for d in own), count)
        self.flops += count * self.pair * sum(d * (nt - d) for d in own)

    def inner(self, level, count=1):
        self.flops += count * self.pair * -(-level // self.alpha) * 2 * (level + self.K)

    def moddown(self, level, count=1):
        self.ntts(2 * self.K + 2 * level, count)
        self.flops += count * self.pair * 2 * level * (self.K + 1)

    def switch(self, level, count=1):
        self.modup(level, count); self.inner(level, count); self.moddown(level, count)

    def rescale(self, level, count=1):
        self.ntts(2 * level, count)
        self.flops += count * self.pair * 2 * (level - 1)

    def product(self, level, count=1):
        self.flops += count * self.pair * 4 * level

    def mul_rescale(self, level, count=1):
        self.product(level, count); self.switch(level, count); self.rescale(level, count)


def work(case):
    w = _Work(case["log_n"])
    op, level = case["op"], case.get("level")
    if op == "ntt":
        limbs = 2 * case["batch"] * case["limbs"]
        w.ntts(limbs)
        w.bytes = 2 * limbs * w.limb
    elif op == "encode":
        n = w.N // 2
        w.ntts(level, case["batch"])
        w.flops += case["batch"] * 5 * n * (case["log_n"] - 1)
        w.bytes = case["batch"] * (8 * n + level * w.limb)
    elif op == "rotate":
        w.switch(level)
        w.bytes = 2 * w.ct(level) + w.key(level)
    elif op == "hoisted":
        r = case["rotations"]
        w.modup(level); w.inner(level, r); w.moddown(level, r)
        w.bytes = w.ct(level) + r * (w.key(level) + w.ct(level))
    elif op == "mul":
        w.mul_rescale(level)
        w.bytes = 2 * w.ct(level) + w.key(level) + w.ct(level - 1)
    elif op == "poly":
        d, m = case["degree"], case["block"]
        giants = d // m
        lb = level - (m - 1).bit_length()
        w.mul_rescale(level, m - 1)
        w.mul_rescale(lb, max(giants - 1, 0))
        w.product(lb, d + giants); w.switch(lb); w.rescale(lb, giants + 1)
        w.flops *= case["count"]
        w.bytes = case["count"] * (w.ct(level) + w.ct(max(lb - 4, 1))) + w.key(level)
    elif op == "projection":
        S, B, F = case["shards"], case["baby"], (w.N // 2) // case["tokens"]
        keys = set(range(1, B))
        blocks = lambda d: [min(F, d - x) for x in range(0, d, F)]  # noqa: E731
        for m in blocks(case["d_in"]):
            w.modup(level, S); w.inner(level, S * (B - 1)); w.moddown(level, S * (B - 1))
        for o in blocks(case["d_out"]):
            giants = 0
            for m in blocks(case["d_in"]):
                diagonals = min(m, o)
                giants = max(giants, diagonals // B)
                w.ntts(level, diagonals)
                w.flops += diagonals * S * w.pair * 2 * level
                folds = max(m // o, 1).bit_length() - 1
            keys |= {g * B for g in range(1, giants)} | {o << f for f in range(folds)}
            w.modup(level, S * (giants - 1)); w.inner(level, S * (giants - 1))
            w.moddown(level, S if case["lazy"] else S * (giants - 1))
            w.switch(level, S * folds)
            w.rescale(level, S)
        w.bytes = 8 * case["d_in"] * case["d_out"] + len(keys) * w.key(level)
        w.bytes += S * (len(blocks(case["d_in"])) * w.ct(level) + len(blocks(case["d_out"])) * w.ct(level - 1))
    else:
        dim, E, G = case["dim"], case["diag_block"], case["tokens"] // case["diag_block"]
        Gb = min(case["group_baby"], G)
        Gg, ladder = G // Gb, E.bit_length() - 1
        w.modup(level, dim * ((Gb > 1) + (Gg > 1))); w.inner(level, dim * (Gb + Gg - 2)); w.moddown(level, dim * (Gb + Gg - 2))
        w.product(level, G * dim); w.switch(level, G); w.rescale(level, G); w.switch(level - 1, G - Gb)
        lv = level - 1                                       # Softmax: the exponential, a round's row sum, its polynomial, two products
        w.mul_rescale(lv, 3 * G); w.rescale(lv - 2, G)
        lv -= 3
        w.product(lv, G); w.switch(lv); w.rescale(lv); w.switch(lv - 1, ladder)
        w.mul_rescale(lv - 1, 3); w.rescale(lv - 3)
        w.mul_rescale(lv - 4, G); w.mul_rescale(lv - 5, G)
        lp = lv - 6
        w.modup(lp, dim); w.inner(lp, dim * (G - 1)); w.moddown(lp, dim * (G - 1))
        w.product(lp, dim * G); w.switch(lp, dim); w.rescale(lp, dim); w.switch(lp - 1, dim * ladder)
        keys = (Gb - 1) + 2 * (Gg - 1) + (G - 1) + ladder + 1
        w.bytes = 2 * dim * w.ct(level) + dim * (w.ct(lp) + w.ct(lp - 1)) + keys * w.key(lp)
    return {"bytes": w.bytes, "flops": w.flops}


def tolerance(case):
    return "exact"
