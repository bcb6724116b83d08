"""The bytes that bench.py counts for stencil sweeps (host logic, no GPU): p and x
pass through memory every second iteration wherever the sweep takes its steps in
pairs, and DRAM traffic is taken from an ncu record of the same size only."""
import json

import pytest

import bench

N256 = 256 ** 3


@pytest.mark.parametrize("l,prec,nx,passes", [(1, "fp64", 256, 10), (2, "fp64", 256, 11), (3, "fp64", 255, 14),
                                              (4, "fp64", 256, 18), (4, "fp64", 255, 20), (1, "fp32", 256, 8),
                                              (1, "fp32", 254, 8), (2, "fp32", 256, 11), (4, "fp32", 254, 20)])
def test_passes(l, prec, nx, passes):
    r = bench.stencil_roofline(n=N256, nx=nx, l=l, prec=prec, iters=500, seconds=0.1, hbm_peak=6792.7, hbm_src="measured",
                               dp_peak_tf=1.2552, dp_src="measured", paired=bench.pairs_px(l, prec, nx))
    hbm = r if r["bound"] == "hbm" else r["hbm"]
    assert hbm["bytes_per_iter"] == passes * (8 if prec == "fp64" else 4) * N256


def test_fp32_headline_stays_below_the_roof():
    r = bench.stencil_roofline(n=N256, nx=256, l=1, prec="fp32", iters=538, seconds=0.0475, hbm_peak=6785.9,
                               hbm_src="measured", dp_peak_tf=1.2552, dp_src="measured",
                               paired=bench.pairs_px(1, "fp32", 256))
    assert r["bound"] == "hbm" and 0.85 < r["frac"] < 1.0


def test_traffic_of_another_size_is_not_used(tmp_path, monkeypatch):
    (tmp_path / "profiles").mkdir()
    rec = {"source_hash": bench.kernel_source_hash(), "n": 160 ** 3, "dram_bytes_per_point_iter": 21.4}
    (tmp_path / "profiles" / "r.json").write_text(json.dumps(rec))
    monkeypatch.setattr(bench, "kernel_source_hash", lambda: rec["source_hash"])
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.profiled_record("r.json", 160 ** 3) == rec
    assert bench.profiled_record("r.json", N256) is None
