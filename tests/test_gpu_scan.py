"""k_scan (pfm, a CTA per sample over chunks of the time-sorted edges) equals the
oracle: at the edges of a chunk, with steps that fill one, with several ways back,
and with either CTA size.  All results are whole numbers or sums of the same
doubles in the same order, so the comparisons are exact."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_08356_gb300 import synth
from test_gpu_sweep import COUNTERS, _chain, _layers

pytestmark = pytest.mark.gpu

SMALL = 2048            # edges a CTA of 512 threads holds; chunks are cut every 1,536


@pytest.fixture()
def M(monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2304_08356_gb300 import build as B
    from paper_2304_08356_gb300 import mantra
    B.build()
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "scan")
    return mantra


def _random(n, m, t_hi, seed=3):
    return synth.uniform_small(n=n, m=m, t_lo=1, t_hi=t_hi, seed=seed), n


CASES = {
    "one edge": lambda: ((np.zeros(1, np.uint32), np.ones(1, np.uint32), np.ones(1, np.uint32)), 2),
    "below a chunk": lambda: _random(200, 1535, 900),
    "a chunk": lambda: _random(200, 1536, 1536),
    "past a chunk": lambda: _random(200, 1537, 5000),
    "chunks of an odd count": lambda: _random(500, 3 * 1536 + 1, 2000),
    "bursty": lambda: (synth.chung_lu_bursty(n=2500, m=60000, seed=9), 2500),
    "spread": lambda: (synth.chung_lu_uniform_t(n=3000, m=70000, seed=2), 3000),
    "bits past 2^16": lambda: (synth.chung_lu_uniform_t(n=70001, m=90007, seed=5), 70001),
    "steps within a chunk": lambda: _layers(22, 8),
    "steps of most of a chunk": lambda: _layers(32, 6),
    "steps past a chunk": lambda: _layers(46, 3),
    "past 64 bits": lambda: _layers(5, 40),
    "long path": lambda: _chain(3000, False),
    "long path with a choice": lambda: _chain(1500, True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_scan_equals_oracle(M, name):
    (u, v, t), n = CASES[name]()
    g, o = M.Graph(u, v, t, n=n), O.Graph(u, v, t, n=n)
    on_scan = name != "steps past a chunk"      # those stay with the CTA search
    assert (np.unique(t, return_counts=True)[1].max() <= SMALL) == on_scan
    for r in (1, 300, 700):                     # 1,024 threads up to two samples per SM, then 512
        for target in (0, 1, 2):
            est, hits, info = g.estimate(2, 0.05, 0.1, 3, fixed_r=r, target=target)
            oest, ohits, oinfo = o.estimate(2, 0.05, 0.1, 3, fixed_r=r, target=target)
            assert np.array_equal(hits, ohits) and np.array_equal(est, oest), (r, target)
            for k in COUNTERS:
                assert info[k] == oinfo[k], (r, target, k)
            if r == 700 and name != "past 64 bits":     # (whose 128-bit re-runs expand edges)
                assert (info["edges_expanded"] == 0) == on_scan
    assert g.sample_paths(2, 8, 5, 100, edges=True, cap=n + 1) == o.samples(2, 8, 5, 100, edges=True, cap=n + 1)
    g.free()


def test_scan_in_uneven_batch(M):
    """Graphs of many sizes in one launch, with rounds that share its workspace."""
    tris = [CASES[k]() for k in ("below a chunk", "bursty", "past a chunk", "long path", "spread")]
    probs = [dict(graph=M.Graph(*tri, n=n), opt=2, eps=0.05, delta=0.1, seed=7 + x)
             for x, (tri, n) in enumerate(tris)]
    for x, (est, hits, info, status) in enumerate(M.estimate_batch(probs)):
        tri, n = tris[x]
        oest, ohits, oinfo = O.Graph(*tri, n=n).estimate(2, 0.05, 0.1, 7 + x)
        assert status == 0 and np.array_equal(hits, ohits) and np.array_equal(est, oest)
        for k in COUNTERS:
            assert info[k] == oinfo[k], k
