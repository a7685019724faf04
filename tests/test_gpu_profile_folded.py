"""The profile counts split butterflies and folded products where they run, and
their chains are faster than the ones they replace."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,special,sbits,level,sbfly,folds", [
    # a rotation of one ciphertext, level limbs in digits of two, two special primes.  Forward column passes: ModUp
    # 4 digits x 10 targets - 8 own = 32 limbs, 24 of them on 40-bit primes; products: 4 x 8 targets x 2 sources
    (40, 2, 59, 8, 24 / 32, 64), (50, 2, 59, 8, 0.0, 64), (50, 2, 61, 8, 0.0, 0)])
def test_a_rotation_counts_what_it_runs(bits, special, sbits, level, sbfly, folds):
    import paper_2006_10091_gb300 as he
    ctx = he.Context(12, level, bits, special, sbits, 2.0 ** 40, seed=1, rot_steps=[1])
    he.he_set_tuning(ctx, "ntt_pb_max", 1)
    a, out = ctx.new_ct(level), ctx.new_ct(level)
    a.tensor.zero_()
    a.level, a.scale = level, 2.0 ** 40
    he.he_rotate(ctx, a, 1, out)
    he.he_profile_enable(ctx, True)
    he.he_rotate(ctx, a, 1, out)
    p = {k: he.he_profile_read(ctx, k) for k in he.he_profile_names(ctx)}
    he.he_profile_enable(ctx, False)
    rows = p["ks_ntt_rot_products"]
    assert rows["sbfly"] == pytest.approx(sbfly * rows["bfly"])
    assert p["ks_modup_ntt"]["folds"] == folds * ctx.n
    assert p["moddown_ntt"]["folds"] == (2 * level * special * ctx.n if folds else 0)
    assert p["moddown_ntt_combine"]["sbfly"] == (p["moddown_ntt_combine"]["bfly"] if sbfly else 0)
    for v in p.values():
        assert v["sbfly"] <= v["bfly"] and v["folds"] <= v["work"] - v["bfly"] - v["mac"] - v["mac3"]


def test_the_chains_rates():
    import paper_2006_10091_gb300 as he
    r = [he.he_probe_alu(k)["per_clock_per_sm"] for k in range(7)]
    assert r[5] > r[2] and r[6] > r[1]
