"""A batch's residues do not depend on its size: the conversion kernels split
target limbs over several CTAs when the batch leaves CTAs free, finish the
inverse transform themselves or not, and the key-product kernel takes several
ciphertexts per CTA; every route gives the residues of the others (small
batches are compared with the oracle in the parity tests)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def uniform(ctx, torch, level, count, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    cts = ctx.new_ct(level, count)
    for c in cts:
        for t in range(level):
            c.tensor[:, t].random_(0, ctx.primes[t], generator=gen)
        c.level, c.scale = level, 2.0 ** 40
    return cts


# (log_n, limbs, bits, special, special bits, level, batch): one limb per digit, a last digit that is not full,
# digits of four limbs, wide special primes; batches on both sides of one wave of CTAs
CASES = [(12, 4, 40, 1, 60, 4, 90), (12, 7, 45, 3, 59, 7, 70), (13, 9, 50, 4, 60, 6, 90), (14, 5, 40, 2, 59, 5, 61)]


@pytest.mark.parametrize("log_n,limbs,bits,special,sbits,level,batch", CASES)
def test_residues_do_not_depend_on_the_batch(log_n, limbs, bits, special, sbits, level, batch):
    import torch
    import paper_2006_10091_gb300 as he
    ctx = he.Context(log_n, limbs, bits, special, sbits, 2.0 ** 40, seed=5, rot_steps=[3, 64])
    A, B = uniform(ctx, torch, level, batch, 1), uniform(ctx, torch, level, batch, 2)
    ops = {
        "mul": lambda x, y, o: he.he_mul_relin_rescale_batch(ctx, x, y, o),
        "rotate": lambda x, y, o: he.he_rotate_batch(ctx, x, 3, o),
        "rotsum": lambda x, y, o: he.he_rotate_sum_batch(ctx, x, [3, 64], o),
        "rotsum_closed": lambda x, y, o: he.he_rotate_sum_batch(ctx, x, [64], o),
    }
    for name, op in ops.items():
        want = ctx.new_ct(level, batch)
        op(A, B, want)
        for first, count in ((0, 1), (batch - 1, 1), (7, 5), (3, 24)):
            got = ctx.new_ct(level, count)
            op(A[first:first + count], B[first:first + count], got)
            for i in range(count):
                assert np.array_equal(got[i].residues(), want[first + i].residues()), (name, first, count, i)


# stages that move rows between tiles (unit steps) and closed ones; 40-bit limbs (split sums), 58-bit limbs with 61-bit
# special primes and 75 products per residue (128-bit sums reduced after each rotation); one ciphertext and an odd count
@pytest.mark.parametrize("bits,special,sbits", [(40, 2, 59), (50, 4, 60), (58, 1, 61)])
@pytest.mark.parametrize("first,nrot", [(1, 15), (-1, 3), (64, 15)])
def test_rotation_stages_match_the_separate_kernels(bits, special, sbits, first, nrot):
    import torch
    import paper_2006_10091_gb300 as he
    steps = [first * m for m in range(1, nrot + 1)]
    ctx = he.Context(12, 5, bits, special, sbits, 2.0 ** 40, seed=6, rot_steps=steps)
    for count in (1, 3):
        A = uniform(ctx, torch, 5, count, 9)
        want, got = ctx.new_ct(5, count), ctx.new_ct(5, count)
        he.he_set_tuning(ctx, "ntt_generic", 1)
        he.he_rotate_sum_batch(ctx, A, steps, want)
        he.he_set_tuning(ctx, "ntt_generic", 0)
        for shape in (0, 1, 2):
            he.he_set_tuning(ctx, "ntt_shape", shape)
            he.he_rotate_sum_batch(ctx, A, steps, got)
            for i in range(count):
                assert np.array_equal(got[i].residues(), want[i].residues()), (shape, i)
        he.he_set_tuning(ctx, "ntt_shape", 0)


# the conversions' sums for one to five sources, prime sizes on both sides of what they take (30-bit limbs and 61-bit
# special primes keep the Shoup products), a last digit that is not full, inputs random and all q - 1
@pytest.mark.parametrize("limbs,bits,special,sbits", [(5, 30, 2, 45), (4, 34, 1, 40), (7, 40, 3, 59), (9, 45, 4, 60),
                                                      (6, 50, 5, 60), (5, 57, 2, 60), (5, 58, 2, 61), (4, 60, 3, 60)])
def test_conversions_match_the_separate_kernels(limbs, bits, special, sbits):
    import torch
    import paper_2006_10091_gb300 as he
    ctx = he.Context(12, limbs, bits, special, sbits, 2.0 ** 25, seed=7, rot_steps=[1])
    A, B = uniform(ctx, torch, limbs, 3, 3), uniform(ctx, torch, limbs, 3, 4)
    for t in range(limbs):
        A[2].tensor[:, t] = ctx.primes[t] - 1
        B[2].tensor[:, t] = ctx.primes[t] - 1
    res = {}
    for generic in (1, 0):
        he.he_set_tuning(ctx, "ntt_generic", generic)
        mul, rot, low = ctx.new_ct(limbs, 3), ctx.new_ct(limbs, 3), ctx.new_ct(limbs, 3)
        he.he_mul_relin_rescale_batch(ctx, A, B, mul)
        he.he_rotate_batch(ctx, A, 1, rot)
        for a, o in zip(A, low):
            he.he_rescale(ctx, a, o)
        res[generic] = [c.residues() for c in mul + rot + low]
    for got, want in zip(res[0], res[1]):
        assert np.array_equal(got, want)


def test_gradient_sum_over_more_ciphertexts_than_a_split_sum_takes():
    """600 data ciphertexts in one tensor accumulation (split sums of 512 at
    most) give the residues of accumulations of 100."""
    import torch
    import paper_2006_10091_gb300 as he
    g = 64
    ctx = he.Context(12, 6, 40, 2, 59, 2.0 ** 40, seed=8, rot_steps=he.lr_rot_steps(1 << 11, g))
    Z, W = uniform(ctx, torch, 6, 600, 5), uniform(ctx, torch, 6, 1, 6)[0]
    cfg = he.lr_config((0.5, -0.0843, 0.0, 0.0002), 1.0 / 4096, g, 2.0 ** 27)
    res = []
    for chunk in (0, 100):
        he.he_set_tuning(ctx, "lr_chunk", chunk)
        out = ctx.new_ct(1)
        he.he_lr_gradient_step(ctx, Z, W, cfg, out)
        res.append(out.residues())
    assert np.array_equal(res[0], res[1])


@pytest.mark.parametrize("chunk", [0, 4, 1])
def test_shards_in_pieces_give_the_residues_of_each_alone(chunk):
    """Chunks that span shards (data in order, out of order and backwards, one
    level above the weights) against each shard by itself."""
    import torch
    import paper_2006_10091_gb300 as he
    g = 64
    ctx = he.Context(12, 7, 40, 2, 59, 2.0 ** 40, seed=9, rot_steps=he.lr_rot_steps(1 << 11, g))
    Z, W = uniform(ctx, torch, 7, 12, 7), uniform(ctx, torch, 6, 4, 8)
    cfg = he.lr_config((0.5, -0.0843, 0.0, 0.0002), 1.0 / 16, g, 2.0 ** 27)
    data = [Z[:3], [Z[5], Z[3], Z[9]], Z[8:5:-1], Z[10:11]]

    def run(shards):
        grads, sums = ctx.new_ct(1, len(shards)), [ctx.new_ct(3, len(z)) for z, _ in shards]
        he.he_lr_gradient_step_workers(ctx, [(z, w, o) for (z, w), o in zip(shards, grads)], cfg)
        he.he_lr_inference_workers(ctx, [(z, w, o) for (z, w), o in zip(shards, sums)], cfg)
        return [[o.residues()] + [s.residues() for s in so] for o, so in zip(grads, sums)]

    alone = [run([(z, w)])[0] for z, w in zip(data, W)]
    he.he_set_tuning(ctx, "lr_chunk", chunk)
    for a, b in zip(alone, run(list(zip(data, W)))):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
