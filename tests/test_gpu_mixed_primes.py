"""Parameter sets whose limbs take the folds only in part (the first primes below
2^bits do, later ones are too far from it): split and lazy butterflies, both ends
of a split sum and Shoup conversions side by side in one launch give the residues
of the separate kernels, from one ciphertext to a few."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def folds(q):
    k = q.bit_length()
    return 33 <= k <= 60 and (1 << k) - q < 1 << min(28, (2 * k - 4) // 3)


@pytest.mark.parametrize("log_n,limbs,bits,special,sbits", [(12, 16, 33, 3, 59), (14, 16, 36, 2, 59),
                                                            (16, 23, 40, 4, 59)])
def test_mixed_limbs_match_the_separate_kernels(log_n, limbs, bits, special, sbits):
    import torch
    import paper_2006_10091_gb300 as he
    steps = [1, 2, 64, 128]
    ctx = he.Context(log_n, limbs, bits, special, sbits, 2.0 ** 30, seed=7, rot_steps=steps)
    assert len({folds(q) for q in ctx.primes[:limbs]}) == 2
    gen = torch.Generator(device="cuda")
    gen.manual_seed(13)
    A, B = ctx.new_ct(limbs, 3), ctx.new_ct(limbs, 3)
    for c in A + B:
        for t in range(limbs):
            c.tensor[:, t].random_(0, ctx.primes[t], generator=gen)
        c.level, c.scale = limbs, 2.0 ** 30
    for t in range(limbs):
        A[2].tensor[:, t] = ctx.primes[t] - 1
        B[2].tensor[:, t] = ctx.primes[t] - 1
    ops = [lambda n, o: he.he_mul_relin_rescale_batch(ctx, A[:n], B[:n], o),
           lambda n, o: he.he_rotate_batch(ctx, A[:n], 1, o),
           lambda n, o: he.he_rotate_sum_batch(ctx, A[:n], [1, 2], o),
           lambda n, o: he.he_rotate_sum_batch(ctx, A[:n], [64, 128], o),
           lambda n, o: [he.he_rescale(ctx, a, x) for a, x in zip(A[:n], o)]]
    for k, op in enumerate(ops):
        he.he_set_tuning(ctx, "ntt_generic", 1)
        want = ctx.new_ct(limbs, 3)
        op(3, want)
        he.he_set_tuning(ctx, "ntt_generic", 0)
        for n in (1, 3):
            got = ctx.new_ct(limbs, n)
            op(n, got)
            for i in range(n):
                assert np.array_equal(got[i].residues(), want[i].residues()), (k, n, i)
