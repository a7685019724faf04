"""The folded reductions of the conversion and key-product kernels (primes q =
2^k - delta), restated on Python integers: every intermediate fits its
register at the extremes of its range and the result has the right residue
and bound, over the prime sizes the kernels take."""
import random

import pytest

M64 = (1 << 64) - 1


def is_prime(n):
    if n % 2 == 0:
        return n == 2
    d, r = n - 1, 0
    while d % 2 == 0:
        d, r = d // 2, r + 1
    for a in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37):
        x = pow(a, d, n)
        if x in (1, n - 1):
            continue
        for _ in range(r - 1):
            x = x * x % n
            if x == n - 1:
                break
        else:
            return False
    return True


def scan(bits, log_n, count):
    step, out = 2 << log_n, []
    k = ((1 << bits) - 2) // step
    while len(out) < count:
        if is_prime(k * step + 1):
            out.append(k * step + 1)
        k -= 1
    return out


def delta_of(q):
    k = q.bit_length()
    d = (1 << k) - q
    return d if 33 <= k <= 60 and d < 1 << min(28, k - 11, (2 * k - 4) // 3) else 0


def fold(x, q):
    k = q.bit_length()
    assert 0 <= x <= M64 and x >> k < 1 << 32
    r = (x & ((1 << k) - 1)) + (x >> k) * delta_of(q)
    assert r <= M64
    return r


def conv_ok(q, cnt, src):
    k = q.bit_length()
    e = (k + 1) // 2
    if not 33 <= k <= 60 or not 1 <= cnt <= 5 or src > 60 or not delta_of(q):
        return False
    d = delta_of(q)
    most = 1 << src
    if cnt > 1:
        a, b = (2 * cnt) << (30 + e), (2 * cnt) << (30 + k - e)
        if b >> 64:
            return False
        most = a + (1 << 2 * e) + ((b >> e) + 1) * (d << (2 * e - k))
    most += 3 * q
    if most >> 64:
        return False
    f = (1 << k) + (most >> k) * d
    return f <= (1 << (k + 5) if q < 1 << 58 else 2 * q)


def conv(vs, cs, q, minus):
    k = q.bit_length()
    e = (k + 1) // 2
    mask, rho = (1 << e) - 1, delta_of(q) << (2 * e - k)
    a = b = 0
    if len(vs) == 1:
        a = vs[0]
    else:
        for v, c in zip(vs, cs):
            c2 = (c << 30) % q
            v0, v1 = v & ((1 << 30) - 1), v >> 30
            for x, w in ((v0, c), (v1, c2)):
                assert x < 1 << 32 and w & mask < 1 << 32 and w >> e < 1 << 32
                a, b = a + x * (w & mask), b + x * (w >> e)
        assert a <= M64 and b <= M64
        a += (b & mask) << e
        h = b >> e
        assert (h >> 32) * rho < 1 << 32
        a += h * rho
    a += minus
    assert a <= M64
    return fold(a, q)


@pytest.mark.parametrize("bits", [33, 34, 37, 40, 41, 45, 50, 55, 57, 58, 59, 60])
def test_conversion_sums(bits):
    rng = random.Random(bits)
    ran = 0
    for log_n in (12, 14, 16):
        for q in scan(bits, log_n, 8)[::7]:
            for cnt in range(1, 6):
                for src in (30, 40, 50, 59, 60):
                    if not conv_ok(q, cnt, src):
                        continue
                    ran += 1
                    top = (1 << src) - 1
                    for trial in range(4):
                        vs = [top if trial == 0 else rng.randrange(top + 1) for _ in range(cnt)]
                        cs = [1] if cnt == 1 else [q - 1 if trial < 2 else rng.randrange(q) for _ in range(cnt)]
                        sub = rng.randrange(2 * q)
                        r = conv(vs, cs, q, sub)
                        assert (r - sum(v * c for v, c in zip(vs, cs)) - sub) % q == 0
                        assert r < (2 * q if q >= 1 << 58 else 1 << (q.bit_length() + 5)) + 1
    assert ran or bits < 38  # (the smallest primes are too dense below a power of two)


@pytest.mark.parametrize("bits", [33, 36, 40, 41, 45, 50, 55, 56])
def test_split_sum_residue(bits):
    rng = random.Random(bits)
    for log_n in (12, 14, 16):
        for q in scan(bits, log_n, 8)[::7]:
            if not delta_of(q):
                continue
            k = q.bit_length()
            sb = (k + 1) // 2
            terms = 128
            while 2 * sb + 2 + (terms + 2).bit_length() > 64:
                terms //= 2
            for trial in range(4):
                xs = [(q - 1, q - 1) if trial == 0 else (rng.randrange(q), rng.randrange(q)) for _ in range(terms)]
                xs.append((min(int(1.01 * q), 2 * q - 1), q - 1))  # part 0's folded sum
                ll = hh = ss = 0
                for x, w in xs:
                    xl, xh, wl, wh = x & ((1 << sb) - 1), x >> sb, w & ((1 << sb) - 1), w >> sb
                    assert max(xl + xh, wl + wh) < 1 << 32
                    ll, hh, ss = ll + xl * wl, hh + xh * wh, ss + (xl + xh) * (wl + wh)
                assert ss <= M64
                mid, rho = ss - ll - hh, delta_of(q) << (2 * sb - k)
                h = fold(hh + (mid >> sb), q)
                t = (h * rho) >> 32
                assert t <= M64 and t >> (k - 32) < 1 << 32
                r = (t >> (k - 32)) * delta_of(q) + (h * rho) % (1 << k) + ll + ((mid & ((1 << sb) - 1)) << sb)
                assert r <= M64
                r = fold(r, q)
                assert r < 2 * q and (r - sum(x * w for x, w in xs)) % q == 0
