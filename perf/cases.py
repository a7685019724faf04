"""Performance cases: the encrypted operations and circuits a worker or key
holder runs through the package's public entry points, from one ciphertext of
a small ring to the full gradient step.

A case names an operation (`op`), the scheme parameters (ring degree 2^log_n,
`limbs` primes of `bits` bits, `special` special primes of `sbits` bits,
scale 2^`lscale`), the level the operands sit at and how many ciphertexts one
pass takes.  Ciphertexts are uniform residues, which is what an RLWE
ciphertext's words are; only the decryption case encrypts real data, because
there the values matter.  Contexts (primes, keys, tables) are kept between
preparations with the same parameters, as a program keeps them.
"""
from __future__ import annotations

import math
from collections import OrderedDict

import numpy as np
import torch

import paper_2006_10091_gb300 as he

# Parameter sets of the repository's workloads: (limbs, bits, special, sbits, lscale)
SMALL = dict(limbs=3, bits=40, special=1, sbits=60, lscale=30)    # small multiplication configuration, N = 2^12
STEP = dict(limbs=8, bits=40, special=2, sbits=59, lscale=40)     # gradient step, N = 2^14
SERVE = dict(limbs=20, bits=50, special=4, sbits=60, lscale=50)   # serving mix, N = 2^13 .. 2^16
LARGE = dict(limbs=24, bits=50, special=4, sbits=60, lscale=50)   # large configuration, N = 2^16
# gradient of the binomial loss as the paper's cubic
POLY = (0.5, -0.0843, 0.0, 0.0002)


def listed():
    return [
        # a key holder encrypting one short feature vector: host values in, one ciphertext out
        dict(name="encrypt_n12", op="encrypt", log_n=12, **SMALL, level=3, count=1),
        # the key holder reading a gradient step's result: one decryption and decoding to host slots
        dict(name="decrypt_n14", op="decrypt", log_n=14, **STEP, level=3, count=1),
        # one multiplication of the small configuration: launches and latency
        dict(name="mul_n12", op="mul", log_n=12, **SMALL, level=3, count=1),
        # the small configuration's sixteen pairs in one call
        dict(name="mul_n12_b16", op="mul", log_n=12, **SMALL, level=3, count=16),
        # one rotation at a serving ring size, an odd level and a last digit that is not full
        dict(name="rotate_n13", op="rotate", log_n=13, **SERVE, level=19, count=1, step=5),
        # a plaintext-weighted, shifted and rescaled ciphertext: the scoring of one request's packed features
        dict(name="affine_n15", op="affine", log_n=15, **SERVE, level=11, count=1),
        # one hoisted stage of the step's feature sum over part of a shard (an odd count)
        dict(name="rotsum_n14_b63", op="rotsum", log_n=14, **STEP, level=7, count=63, step=8, nrot=7),
        # multiplications at the large configuration
        dict(name="mul_n16_b8", op="mul", log_n=16, **LARGE, level=24, count=8),
        # the first stage of the large configuration's rotate-and-sum: unit steps, fifteen rotations
        dict(name="rotsum_n16_b4", op="rotsum", log_n=16, **LARGE, level=24, count=4, step=1, nrot=15),
        # encrypted inference of three requests of different sizes at serving parameters
        dict(name="infer_n13", op="infer", log_n=13, **SERVE, level=9, w_level=9, count=21, shards=3, g=16, lmask=34),
        # one mini-batch's gradient step on a small shard
        dict(name="step_n13_b5", op="step", log_n=13, **STEP, level=7, w_level=7, count=5, shards=1, g=8, lmask=27),
        # the full gradient step: 4096 samples x 784 features, eight samples per ciphertext
        dict(name="step_n14_b512", op="step", log_n=14, **STEP, level=8, w_level=8, count=512, shards=1, g=8, lmask=27),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["encrypt", "decrypt", "mul", "mul", "rotate", "affine", "rotsum", "rotsum", "infer", "step"])
    log_n = rng.randint(12, 16)
    if op in ("infer", "step"):  # circuits: five or more levels, an own key per rotation
        log_n = rng.randint(12, 14)
        bits = rng.choice([40, 50])
        case = dict(op=op, log_n=log_n, limbs=rng.randint(7, 10), bits=bits, special=rng.choice([1, 2, 4]),
                    sbits=rng.choice([59, 60]), lscale=bits)
        case["level"] = rng.randint(6, case["limbs"])
        case["w_level"] = rng.randint(6, case["level"])
        top = {12: 512, 13: 256, 14: 96}[log_n]
        case["count"] = _log_int(rng, 1, top)
        case["shards"] = rng.randint(1, min(4, case["count"]))
        case["g"] = 1 << rng.randint(2, 6)
        case["lmask"] = 27 if bits == 40 else 34
        return case
    case = dict(op=op, log_n=log_n, limbs=rng.randint(3, 24), bits=rng.choice([40, 45, 50, 55]),
                special=rng.choice([1, 2, 3, 4]), sbits=rng.choice([59, 60]), lscale=40)
    case["level"] = rng.randint(2, case["limbs"])
    # a one-prime digit size with many limbs makes as many digits: keys and work stay in the range of the listed cases
    if case["special"] == 1:
        case["limbs"] = min(case["limbs"], 8)
        case["level"] = min(case["level"], 8)
    words = (1 << log_n) * (case["level"] + case["special"])
    if op in ("encrypt", "decrypt", "affine"):
        case["count"] = 1
    elif op == "rotsum":
        case["count"] = _log_int(rng, 1, max(1, min(200, int(2.0e7 / words))))
        case["nrot"] = rng.choice([1, 3, 7, 15])
        case["step"] = 1 << rng.randint(0, 6)
    else:
        case["count"] = _log_int(rng, 1, max(1, min(600, int(4.0e7 / words))))
        if op == "rotate":
            case["step"] = rng.choice([1, 5, 8, 64, -1])
    return case


def _rot_steps(case):
    if case["op"] == "rotate":
        return (case["step"],)
    if case["op"] == "rotsum":
        return tuple(case["step"] * m for m in range(1, case["nrot"] + 1))
    if case["op"] in ("infer", "step"):
        return tuple(he.lr_rot_steps(1 << (case["log_n"] - 1), case["g"]))
    return ()


_contexts = OrderedDict()


def _context(case):
    key = (case["log_n"], case["limbs"], case["bits"], case["special"], case["sbits"], case["lscale"],
           _rot_steps(case))
    if key not in _contexts:
        while len(_contexts) >= 2:  # keys and scratch of unused parameter sets are given back
            _contexts.popitem(last=False)
        _contexts[key] = he.Context(case["log_n"], case["limbs"], case["bits"], case["special"], case["sbits"],
                                    2.0 ** case["lscale"], seed=1, rot_steps=_rot_steps(case))
    _contexts.move_to_end(key)
    return _contexts[key]


def _uniform(ctx, gen, level, count, scale):
    """`count` ciphertexts of uniform residues at `level`, one allocation."""
    buf = torch.empty((count, 2, level, ctx.n), dtype=torch.int64, device="cuda")
    for t in range(level):
        buf[:, :, t].random_(0, ctx.primes[t], generator=gen)
    return [he.Ciphertext(buf[i], level, level, scale) for i in range(count)]


def _outputs(ctx, level, count):
    buf = torch.empty((count, 2, level, ctx.n), dtype=torch.int64, device="cuda")
    return buf, [he.Ciphertext(buf[i], level) for i in range(count)]


def _values(case, seed):
    return np.random.default_rng(seed).uniform(-1.0, 1.0, 1 << (case["log_n"] - 1))


def _shares(case):
    """Sizes of the shards: uneven, in all `count` ciphertexts."""
    left, out = case["count"], []
    for k in range(case["shards"], 1, -1):
        n = max(1, min(left - (k - 1), (left * 2) // (k + 2)))
        out.append(n)
        left -= n
    return out + [left]


def prepare(case, seed):
    op, level, count = case["op"], case["level"], case["count"]
    ctx = _context(case)
    scale = 2.0 ** case["lscale"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = dict(case=case, ctx=ctx)
    if op == "encrypt":
        s["slots"] = _values(case, seed)
        s["buf"], s["out"] = _outputs(ctx, level, 1)
    elif op == "decrypt":
        s["a"] = ctx.new_ct(level)
        he.he_encode_encrypt(ctx, _values(case, seed), scale, level, s["a"], cid=seed & 0xFFFFFF)
    elif op == "affine":
        s["a"] = _uniform(ctx, gen, level, 1, scale)[0]
        s["weights"] = np.random.default_rng(seed).integers(-(1 << 30), 1 << 30, size=ctx.n, dtype=np.int64)
        s["mid"] = _outputs(ctx, level, 1)[1][0]
        s["buf"], s["out"] = _outputs(ctx, level - 1, 1)
    elif op == "mul":
        s["a"] = _uniform(ctx, gen, level, count, scale)
        s["b"] = _uniform(ctx, gen, level, count, scale)
        s["buf"], s["out"] = _outputs(ctx, level - 1, count)
    elif op in ("rotate", "rotsum"):
        s["a"] = _uniform(ctx, gen, level, count, scale)
        s["steps"] = list(_rot_steps(case))
        s["buf"], s["out"] = _outputs(ctx, level, count)
    else:
        s["cfg"] = he.lr_config(POLY, 1.0 / 4096, case["g"], 2.0 ** case["lmask"])
        s["shards"], s["bufs"] = [], []
        for n in _shares(case):
            Z = _uniform(ctx, gen, level, n, scale)
            W = _uniform(ctx, gen, case["w_level"], 1, scale)[0]
            buf, out = _outputs(ctx, case["w_level"] - (3 if op == "infer" else 5), n if op == "infer" else 1)
            s["shards"].append((Z, W, out if op == "infer" else out[0]))
            s["bufs"].append(buf)
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    op, level, count = case["op"], case["level"], case["count"]
    scale = 2.0 ** case["lscale"]
    if op == "encrypt":
        he.he_encode_encrypt(ctx, s["slots"], scale, level, s["out"][0], cid=7)
    elif op == "decrypt":
        return he.he_decrypt_decode(ctx, s["a"])
    elif op == "affine":
        he.he_mul_plain(ctx, s["a"], s["weights"], 2.0 ** 30, s["mid"])
        he.he_rescale(ctx, s["mid"], s["out"][0])
        he.he_add_const(ctx, s["out"][0], 0.25, s["out"][0])
    elif op == "mul":
        if count == 1:
            he.he_mul_relin_rescale(ctx, s["a"][0], s["b"][0], s["out"][0])
        else:
            he.he_mul_relin_rescale_batch(ctx, s["a"], s["b"], s["out"])
    elif op == "rotate":
        if count == 1:
            he.he_rotate(ctx, s["a"][0], s["steps"][0], s["out"][0])
        else:
            he.he_rotate_batch(ctx, s["a"], s["steps"][0], s["out"])
    elif op == "rotsum":
        if count == 1:
            he.he_rotate_sum(ctx, s["a"][0], s["steps"], s["out"][0])
        else:
            he.he_rotate_sum_batch(ctx, s["a"], s["steps"], s["out"])
    elif op == "infer":
        he.he_lr_inference_workers(ctx, s["shards"], s["cfg"])
        return s["bufs"]
    elif case["shards"] == 1:
        Z, W, out = s["shards"][0]
        he.he_lr_gradient_step(ctx, Z, W, s["cfg"], out)
        return s["bufs"]
    else:
        he.he_lr_gradient_step_workers(ctx, s["shards"], s["cfg"])
        return s["bufs"]
    return s["buf"]


class _Count:
    """Modular products of the operations a pass cannot do without (a
    butterfly is one), and the switching keys it reads."""

    def __init__(self, case):
        self.n, self.log_n, self.alpha = 1 << case["log_n"], case["log_n"], case["special"]
        self.mul, self.keys = 0.0, 0

    def ntt(self, polys):
        self.mul += polys * self.n / 2 * self.log_n

    def keyswitch(self, level, nrot=1, drop=0):
        """One decomposition, nrot key products, one division by P (and by `drop` limbs)."""
        a = self.alpha
        beta, nt = -(-level // a), level + a
        conv = beta * nt - level
        self.ntt(level + conv)
        self.mul += self.n * (level + sum(min(a, level - j * a) * (nt - min(a, level - j * a)) for j in range(beta)))
        self.mul += self.n * 2.0 * nrot * beta * nt
        out = level - drop
        self.ntt(2 * (a + drop + out))
        self.mul += self.n * 2.0 * (a + drop) * (out + 1) + self.n * 2.0 * out

    def key_words(self, level, nrot=1):
        self.keys += nrot * 2 * -(-level // self.alpha) * (level + self.alpha) * self.n

    def product(self, level):
        self.mul += 4.0 * level * self.n

    def rescale(self, level):
        self.ntt(2 * level)
        self.mul += self.n * 4.0 * (level - 1)


def work(case):
    op, level, count = case["op"], case["level"], case["count"]
    c = _Count(case)
    ct = 2 * c.n  # words of one limb of a ciphertext
    if op == "encrypt":
        c.ntt(3 * level)
        c.mul += 2.0 * level * c.n
        return {"bytes": 8 * (c.n // 2 + 2 * level * c.n + level * ct), "flops": c.mul + 5 * c.n * c.log_n}
    if op == "decrypt":
        c.ntt(level)
        c.mul += c.n * (level + level * (level - 1) / 2)
        return {"bytes": 8 * (level * ct + level * c.n + c.n // 2), "flops": c.mul + 5 * c.n * c.log_n}
    if op == "affine":
        c.ntt(level)
        c.mul += 2.0 * level * c.n
        c.rescale(level)
        return {"bytes": 8 * (level * ct + c.n + (level - 1) * ct), "flops": c.mul}
    if op == "mul":
        c.product(level)
        c.keyswitch(level, drop=1)
        c.key_words(level)
        return {"bytes": 8 * (count * (3 * level - 1) * ct + c.keys), "flops": count * c.mul}
    if op in ("rotate", "rotsum"):
        nrot = case.get("nrot", 1)
        c.keyswitch(level, nrot)
        c.key_words(level, nrot)
        return {"bytes": 8 * (2 * count * level * ct + c.keys), "flops": count * c.mul}
    l, slots, g = case["w_level"], c.n // 2, case["g"]
    stages = [len(st) for st in he.rotsum_stages(g, (slots // g).bit_length() - 1)]
    c.product(l)
    c.keyswitch(l, drop=1)
    for r in stages:
        c.keyswitch(l - 1, r)
        c.key_words(l - 1, r)
    for lv in (l - 1, l - 2):
        c.product(lv)
        c.keyswitch(lv, drop=1)
    c.mul += 4.0 * (l - 1) * c.n
    c.rescale(l - 1)
    c.rescale(l - 1)
    c.key_words(l)
    mul = c.mul * count
    z_words = count * level * ct + case["shards"] * l * ct
    if op == "infer":
        return {"bytes": 8 * (z_words + count * (l - 3) * ct + c.keys), "flops": mul}
    mul += count * 4.0 * (l - 3) * c.n
    c.mul = 0.0
    c.keyswitch(l - 3, drop=1)
    for lv, step in ((l - 4, 1), (l - 5, -1)):
        for st in he.rotsum_stages(step, g.bit_length() - 1):
            c.keyswitch(lv, len(st))
            c.key_words(lv, len(st))
    c.rescale(l - 4)
    return {"bytes": 8 * (z_words + case["shards"] * (l - 5) * ct + c.keys), "flops": mul + case["shards"] * c.mul}


def exact(case, seed):
    """Residues are whole numbers; only decrypted slots have a real value: the
    slots that were encrypted."""
    return _values(case, seed) if case["op"] == "decrypt" else None
