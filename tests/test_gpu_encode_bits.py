"""Encodings are pinned bit for bit.  Which product a fused multiply-add of the
encoder's butterflies rounds decides last bits of the coefficients before they
are rounded, and so, at large scales, coefficients: the digests are those of the
transform with one launch per stage, which every later form has to repeat."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# log2 N -> the first 16 hex digits of SHA-256 over the little-endian int64 coefficients at scales 2^40 and 2^52
DIGESTS = {4: ("0ff94ef605bae090", "d6863639864b6e16"), 8: ("24e6a3d99778e643", "39dbb8b41c9c3e47"),
           12: ("c303cd951f3e1c34", "f48e902f55d81986"), 14: ("f6401c867e31de9c", "da4ca3157ae44eba"),
           16: ("42abb0eed98e7cb8", "182c9d0dbf2f31a0")}


@pytest.mark.parametrize("log_n", sorted(DIGESTS))
def test_encoded_coefficients(log_n):
    import paper_2006_10091_gb300 as he
    ctx = he.Context(log_n, 2, 50, 1, 60, 2.0 ** 40, seed=1)
    i = np.arange(1 << (log_n - 1), dtype=np.uint64)
    z = ((i * np.uint64(2654435761) + np.uint64(12345)) % np.uint64(1 << 32)).astype(np.float64) / 2.0 ** 31 - 1.0
    got = tuple(hashlib.sha256(np.ascontiguousarray(he.he_encode(ctx, z, s)).astype("<i8").tobytes()).hexdigest()[:16]
                for s in (2.0 ** 40, 2.0 ** 52))
    assert got == DIGESTS[log_n]
