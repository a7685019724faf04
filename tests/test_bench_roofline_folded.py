"""Roofline arithmetic of the narrow primes' work (no GPU): split butterflies and
folded conversion products are weighed at their own chains' rates, as parts of
the butterflies and of the other products."""
import pytest

import bench

RATES = {"per_second": 1.0e12, "mac_per_second": 2.0e12, "mac3_per_second": 4.0e12, "butterfly_per_second": 0.5e12,
         "split_butterfly_per_second": 0.8e12, "folded_per_second": 2.5e12}


@pytest.fixture(autouse=True)
def fixed_rates(monkeypatch):
    for k, v in RATES.items():
        monkeypatch.setitem(bench.ALU_PEAK, k, v)


def prof(ms, bfly=0.0, sbfly=0.0, products=0.0, folds=0.0):
    return {"ms": ms, "work": bfly + products, "bfly": bfly, "sbfly": sbfly, "folds": folds, "mac": 0.0, "mac3": 0.0,
            "bytes": 0.0, "launches": 1}


def test_parts_at_their_own_rates():
    # butterflies: 1e9 lazy (2 ms) and 0.8e9 split (1 ms); products: 1e9 Shoup (1 ms) and 2.5e9 folded (1 ms)
    p = prof(10.0, bfly=1.8e9, sbfly=0.8e9, products=3.5e9, folds=2.5e9)
    r = bench.class_roof(p, hbm_peak=1000.0, peak_kind="test", name="ks_modup_ntt")
    assert r["bound"] == "alu" and r["frac"] == pytest.approx(0.5)
    assert r["work_mix"] == pytest.approx({"butterflies": 1.0e9, "split_butterflies": 0.8e9, "shoup_products": 1.0e9,
                                           "folded_products": 2.5e9, "macs": 0.0, "split_macs": 0.0})
    assert bench.roof_time(p, 1000.0) == pytest.approx(5e-3)


def test_chain_fraction_weighs_both_butterflies():
    p = prof(4.0, bfly=1.8e9, sbfly=0.8e9, products=0.1e9)
    r = bench.class_roof(p, hbm_peak=1e6, peak_kind="test", name="ntt")
    assert r["butterfly_chain_frac"] == pytest.approx(3.0 / 4.0)


def test_without_the_chains_the_wide_primes_rates_hold(monkeypatch):
    monkeypatch.setitem(bench.ALU_PEAK, "split_butterfly_per_second", None)
    monkeypatch.setitem(bench.ALU_PEAK, "folded_per_second", None)
    assert bench.roof_time(prof(1.0, bfly=1e9, sbfly=1e9, products=1e9, folds=1e9), 1000.0) == pytest.approx(3e-3)
