"""The rules that admit a prime or a sum to the folded and split arithmetic
(csrc/fold_rules.h, compiled here as they are) against the bounds that the
kernels' arithmetic needs, restated on Python integers at the ends of its
ranges: no intermediate leaves its register and every result is the right
residue within the range the next step takes."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2006_10091_gb300", "csrc")
M64, M32, SPLIT_VALUE = (1 << 64) - 1, (1 << 32) - 1, 1 << 46  # a split butterfly's values stay below 2^46
STAGES, ROUND = 16, 3                                          # transforms of up to 2^16 points, radix-8 rounds

SOURCE = """
#include "fold_rules.h"
extern "C" {
uint32_t delta(uint64_t q) { return fold_delta(q); }
int conv(uint64_t q, uint32_t cnt, uint32_t src) { return conv_split_ok(q, cnt, src); }
int split3(uint32_t k, uint32_t n) { return split3_fits(k, n); }
uint32_t split3_terms() { return kSplit3Terms; }
uint32_t split_bits() { return kSplitMaxBits; }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "rules.so"),
                    str(d / "rules.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "rules.so"))
    lib.delta.argtypes = [ctypes.c_uint64]
    lib.delta.restype = ctypes.c_uint32
    lib.conv.argtypes = [ctypes.c_uint64, ctypes.c_uint32, ctypes.c_uint32]
    lib.split3.argtypes = [ctypes.c_uint32, ctypes.c_uint32]
    return lib


def widest_delta(rules, k):
    """The largest delta of k bits that the rule takes (any odd modulus: the bounds do not need a prime)."""
    lo, hi = 1, 1 << (k - 1)
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if rules.delta((1 << k) - mid) else (lo, mid)
    return lo


def moduli(rules, k):
    top = widest_delta(rules, k)
    return [(1 << k) - d for d in (1, 3, top // 1000 | 1, top // 7 | 1, top - 1 + top % 2)]


def fold_bound(most, q):
    """The largest value of fold(x) for x <= most."""
    k = q.bit_length()
    assert most <= M64 and most >> k <= M32
    return (1 << k) - 1 + (most >> k) * ((1 << k) - q)


def conv_value(q, cnt, src):
    """The largest value that the conversion leaves in the tile, each of its sums inside 64 bits."""
    k = q.bit_length()
    e, d = (k + 1) // 2, (1 << k) - q
    half, rho = (1 << 30) - 1, d << (2 * e - k)  # source halves; the upper one has src - 30 bits
    assert src <= 60
    most = (1 << src) - 1
    if cnt > 1:
        a = cnt * 2 * half * ((1 << e) - 1)
        b = cnt * 2 * half * ((1 << (k - e)) - 1)
        assert a <= M64 and b <= M64 and ((b >> e) >> 32) * rho < 1 << 32
        most = a + (((1 << e) - 1) << e) + (b >> e) * rho
    return fold_bound(most + 2 * q, q)  # minus v P and h of ModDown's lift: at most 2q is added


def transform_takes(q, start, split_bits):
    """Whether a forward transform may start below `start`."""
    k = q.bit_length()
    if k <= split_bits:  # each stage adds at most 3q; the final fold leaves one correction
        end = start + STAGES * 3 * q
        return end <= SPLIT_VALUE and fold_bound(end, q) < 2 * q
    if q < 1 << 58:      # at most 2q a stage
        end = start + STAGES * 2 * q
        return end <= M64 and fold_bound(end, q) < 2 * q
    return start < 4 * q and 8 * q <= M64  # Harvey's corrected butterflies


@pytest.mark.parametrize("k", range(33, 61))
def test_conversions_the_rule_takes_stay_in_the_transforms_range(rules, k):
    split_bits = rules.split_bits()
    taken = 0
    for q in moduli(rules, k):
        for cnt in range(1, 7):
            for src in range(20, 62):
                if rules.conv(q, cnt, src):
                    taken += 1
                    assert transform_takes(q, conv_value(q, cnt, src), split_bits), (q, cnt, src)
    assert taken


def test_a_looser_rule_would_overflow_the_split_butterflies(rules):
    """Conversions left below 2^(k+5), which the lazy transforms take, are too large for split ones: at 40 bits the
    growth from there leaves 2^46.  The compiled rule refuses every such combination."""
    loose = 0
    for q in moduli(rules, 40):
        for cnt in range(1, 6):
            for src in range(20, 61):
                v = conv_value(q, cnt, src)
                if v <= 1 << 45 and not transform_takes(q, v, 40):
                    loose += 1
                    assert not rules.conv(q, cnt, src)
    assert loose


@pytest.mark.parametrize("k", [33, 34, 36, 39, 40])
def test_split_products(rules, k):
    """mul_split for any value below 2^46 and any twiddle: the sum fits 64 bits, the result is below 3q."""
    rng = random.Random(k)
    for q in moduli(rules, k):
        mu, neg = (1 << 64) // q, (1 << 64) - q
        assert mu <= M32
        for trial in range(2000):
            y = SPLIT_VALUE - 1 if trial < 20 else rng.randrange(SPLIT_VALUE)
            w = q - 1 - trial if trial < 20 else rng.randrange(q)
            w2 = (w << 23) % q
            y0, y1 = y & ((1 << 23) - 1), y >> 23
            s = y0 * w + y1 * w2
            assert y1 < 1 << 23 and s <= M64
            a = y1 * (w2 & M32) + y0 * (w & M32)
            h = ((a >> 32) + y0 * (w >> 32) + y1 * (w2 >> 32)) & M32
            qe = (h * mu) >> 32
            t = qe * (neg & M32) + ((a & M32) | h << 32) & M64
            r = (t & M32) | ((t >> 32) + qe * (neg >> 32) & M32) << 32
            assert r == s - qe * q and (r - y * w) % q == 0 and 0 <= r < 3 * q
            assert s < (qe + 2) * q + (1 << 32)  # the quotient falls short of s / q by less than 2 + 2^32 / q
        assert 1 << 32 < q


@pytest.mark.parametrize("k", [33, 36, 40])
def test_split_inverse_round(rules, k):
    """An inverse round starts below 3q; its sums double a stage, its differences get 3q 2^stage added."""
    for q in moduli(rules, k):
        top = 3 * q
        for stage in range(ROUND):
            assert top <= (3 * q) << stage              # so x + (3q << stage) - y is not negative
            assert top + ((3 * q) << stage) <= SPLIT_VALUE
            top *= 2
        assert fold_bound(top, q) < 3 * q               # the next round's start


@pytest.mark.parametrize("k", range(50, 61))
def test_low_word_of_a_128_bit_sum(rules, k):
    """reduce128_any: any 64-bit word folds below 2q, so that with the high part's [0, 2q) two corrections do."""
    for q in moduli(rules, k):
        assert fold_bound(M64, q) < 2 * q and 4 * q <= M64


def split_sum_residue_holds(q, terms):
    """split3_residue of `terms` products of residues below 2^k and of part 0's term (a folded sum below 1.01 times as
    much), every intermediate at its largest."""
    k = q.bit_length()
    sb, d = (k + 1) // 2, (1 << k) - q
    rho, low, high = d << (2 * sb - k), (1 << sb) - 1, (1 << (k - sb)) - 1  # the halves of a residue
    part0 = (101 << k) // 100 >> sb                                         # the upper half of part 0's term
    ll, hh = (terms + 1) * low * low, (terms * high + part0) * high
    mid = terms * 2 * low * high + low * high + part0 * low
    if (terms * (low + high) + low + part0) * (low + high) > M64:  # ss
        return False
    h = fold_bound(hh + (mid >> sb), q)
    if h >= 5 << (k - 2) or h * rho >> 32 > M64 or h * rho >> k > M32:
        return False
    r = (h * rho >> k) * d + (1 << k) - 1 + (low << sb) + ll
    return r <= M64 and fold_bound(r, q) < 2 * q


@pytest.mark.parametrize("k", range(33, 61))
def test_split_sums_the_rule_takes_reduce_to_residues(rules, k):
    lo, hi = 0, rules.split3_terms() + 1  # the most terms the rule takes
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if rules.split3(k, mid) else (lo, mid)
    for q in moduli(rules, k):
        for terms in {1, lo // 3, lo - 1, lo} - {0, -1}:
            assert split_sum_residue_holds(q, terms), (q, terms)
