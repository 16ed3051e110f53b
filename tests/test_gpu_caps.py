"""Samples past a per-sample cap of k_sweep (path vertices, vertices that lead to
z), k_scan (vertices that lead to z) or k_hop (events, states on optimal paths) are
re-run by the 64-bit searches without caps: results and work counters equal the
oracle's, the search's own counter shows that it ran, and no sample is counted as
a 128-bit one.  Counts past 64 bits still take the 128-bit kernels."""
import numpy as np
import pytest

from oracle import oracle as O
from test_gpu_hop import COUNTERS as HOP_COUNTERS, _combs, _hub
from test_gpu_sweep import COUNTERS, _chain, _layers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_2304_08356_gb300 import build as B
    B.build()
    from paper_2304_08356_gb300 import mantra
    return mantra


def _both(a, na, b, nb):
    """Two graphs side by side, without an edge between them."""
    return tuple(np.concatenate([x, y + (na if k < 2 else 0)]).astype(np.uint32)
                 for k, (x, y) in enumerate(zip(a, b))), na + nb


PFM = {
    "path past 2,048": ("sweep", lambda: _chain(3000, False)),
    "set past 1,024": ("sweep", lambda: _chain(1500, True)),
    "set past 2,048": ("scan", lambda: _chain(5000, True)),
    "set at 2,048": ("scan", lambda: _chain(2040, True)),
}


@pytest.mark.parametrize("name", list(PFM))
def test_pfm_caps(M, monkeypatch, name):
    kernel, make = PFM[name]
    monkeypatch.setenv("MANTRA_PFM_KERNEL", kernel)
    (u, v, t), n = make()
    g, o = M.Graph(u, v, t, n=n), O.Graph(u, v, t, n=n)
    for target in (0, 2):
        _, hits, info = g.estimate(2, 0.05, 0.1, 3, fixed_r=400, target=target)
        _, ohits, oinfo = o.estimate(2, 0.05, 0.1, 3, fixed_r=400, target=target)
        assert np.array_equal(hits, ohits)
        for k in COUNTERS:
            assert info[k] == oinfo[k], k
        assert info["wide_samples"] == 0
        assert (info["edges_expanded"] > 0) == (name != "set at 2,048")     # only the search expands edges
    assert g.sample_paths(2, 8, 5, 60, edges=True, cap=n + 1) == o.samples(2, 8, 5, 60, edges=True, cap=n + 1)
    g.free()


@pytest.mark.parametrize("kernel", ["sweep", "scan"])
def test_caps_and_64_bits_in_one_call(M, monkeypatch, kernel):
    """Both lists of a call: long sets on one part of the graph, counts past 64 bits
    on the other."""
    monkeypatch.setenv("MANTRA_PFM_KERNEL", kernel)
    (a, na), (b, nb) = _chain(2600, True), _layers(22, 28)          # up to 22^27 paths, steps of 484 edges
    tri, n = _both(a, na, b, nb)
    g, o = M.Graph(*tri, n=n), O.Graph(*tri, n=n)
    _, hits, info = g.estimate(2, 0.05, 0.1, 4, fixed_r=2500)
    _, ohits, oinfo = o.estimate(2, 0.05, 0.1, 4, fixed_r=2500)
    assert np.array_equal(hits, ohits)
    for k in COUNTERS:
        assert info[k] == oinfo[k], k
    assert info["wide_samples"] > 0 and info["edges_expanded"] > 0
    assert g.sample_paths(2, 8, 5, 300, cap=n + 1) == o.samples(2, 8, 5, 300, cap=n + 1)
    g.free()


@pytest.mark.parametrize("name,est", [("states", 0), ("states", 1), ("events", 0), ("events", 1)])
def test_hop_caps(M, name, est):
    (u, v, t), n = _hub(75100) if name == "states" else _combs(800, 400)
    r, paths = ((12 if est else 24), 12) if name == "states" else (60, 40)
    g, o = M.Graph(u, v, t, n=n), O.Graph(u, v, t, n=n)
    for opt in (0, 1):
        _, hits, info = g.estimate(opt, 0.05, 0.1, 3, fixed_r=r, estimator=est)
        _, ohits, oinfo = o.estimate(opt, 0.05, 0.1, 3, fixed_r=r, estimator=est)
        assert np.array_equal(hits, ohits)
        for k in HOP_COUNTERS:
            assert info[k] == oinfo[k], k
        assert info["wide_samples"] == 0
        if est == 0:
            assert info["search_launches"] == 2          # the caps were passed
            assert g.sample_paths(opt, 8, 5, paths, edges=True) == o.samples(opt, 8, 5, paths, edges=True)
    g.free()
