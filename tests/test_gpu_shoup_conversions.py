"""Conversions to primes that the folded sums turn down (below 33 bits, 61 bits)
run as Shoup products with a compile-time number of sources up to five and a
runtime one beyond; the residues are those of the separate kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# digits of one to six limbs, the last one not full, so ModUp takes 1 .. 6 sources, ModDown as many, and the ModDown
# merged with the rescale one more; inputs random and all q - 1
@pytest.mark.parametrize("log_n,limbs,bits,special,sbits", [(12, 4, 30, 1, 45), (12, 5, 30, 2, 45), (13, 7, 30, 3, 45),
                                                            (12, 9, 61, 4, 61), (14, 6, 58, 5, 61), (12, 13, 30, 6, 59)])
def test_shoup_conversions_match_the_separate_kernels(log_n, limbs, bits, special, sbits):
    import torch
    import paper_2006_10091_gb300 as he
    ctx = he.Context(log_n, limbs, bits, special, sbits, 2.0 ** 25, seed=7, rot_steps=[1])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    A, B = ctx.new_ct(limbs, 3), ctx.new_ct(limbs, 3)
    for c in A + B:
        for t in range(limbs):
            c.tensor[:, t].random_(0, ctx.primes[t], generator=gen)
        c.level, c.scale = limbs, 2.0 ** 25
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
