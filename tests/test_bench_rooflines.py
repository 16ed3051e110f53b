"""The rooflines of bench.py: a kernel's share of the memory rate is by the bytes
that kernel takes, not by those of a search it does without."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

INFO = dict(edges_scanned=10_000_000, sigma_adds=2_000_000, frontier_vertices=300_000, edges_expanded=0,
            states_new=1_500_000, alg_bytes=24 * 10_000_000 + 8 * 300_000 + 12 * 1_500_000, kernel_ms=2.0,
            search_launches=3)


def test_rooflines_by_the_kernels_own_bytes(monkeypatch):
    import bench
    monkeypatch.delenv("MANTRA_PFM_KERNEL", raising=False)
    hop = bench.kernel_rooflines(INFO, "sfm", 6000.0)["k_hop"]
    assert hop["achieved"] == pytest.approx((12 * 2_000_000 + 40 * 300_000) / 2e-3 / 1e9)
    assert hop["frac"] == pytest.approx(hop["achieved"] / 6000.0) and hop["alg_gbps"] > 3 * hop["achieved"]
    scan = bench.kernel_rooflines(dict(INFO, edges_expanded=500), "pfm", 6000.0)     # a few samples re-run by the search
    assert list(scan) == ["k_scan"]
    assert scan["k_scan"]["own_model_bytes"] == 12 * 10_000_000 + 8 * 2_000_000
    assert bench.own_model_bytes("k_sweep", INFO) is None
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "cta")
    assert list(bench.kernel_rooflines(INFO, "pfm", 6000.0)) == ["k_pfm_cta"]
