"""The runtime-shaped transforms on both sides of the ring size from which 40-bit
primes take split butterflies, beside a wide prime in the same launch."""
import numpy as np
import pytest

import oracle
from paper_2006_10091_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", [4, 10, 11, 12])
@pytest.mark.parametrize("bits", [36, 40, 50])
def test_generic_ntt_matches_oracle(log_n, bits):
    import torch
    import paper_2006_10091_gb300 as he
    limbs, n = 2, 1 << log_n
    ctx = he.Context(log_n, limbs, bits, 1, 59, 2.0 ** 30, seed=1)
    he.he_set_tuning(ctx, "ntt_generic", 1)
    data = workloads.residues(log_n + bits, ctx.primes, n, parts=2)  # [2][limbs + 1][n]
    data[1] = (np.array(ctx.primes, dtype=np.uint64) - 1)[:, None]
    t = torch.from_numpy(data.view(np.int64).copy()).cuda()
    he.he_ntt(ctx, t, 2, (limbs + 1) * n, limbs + 1, 0, False)
    got = t.cpu().numpy().view(np.uint64)
    for p in range(2):
        for limb, q in enumerate(ctx.primes):
            want = oracle.ntt_r2(data[p, limb], log_n, q, oracle.min_root(q, log_n))
            assert np.array_equal(got[p, limb], want), (p, limb)
    he.he_ntt(ctx, t, 2, (limbs + 1) * n, limbs + 1, 0, True)
    assert np.array_equal(t.cpu().numpy().view(np.uint64), data)
