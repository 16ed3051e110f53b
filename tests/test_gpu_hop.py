"""The hop-level search kernel (csrc/k_hop.cu) at the sizes where its parts
change: levels of more vertices than a CTA has threads, several-in-edge slots,
hubs whose slots span many tiles of the backward collection, path counts past
64 bits, and the two per-sample caps (events, states on optimal paths) past
which a sample takes the 128-bit kernel.  Every result and work counter equals
the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_08356_gb300 import synth

pytestmark = pytest.mark.gpu

COUNTERS = ("edges_scanned", "sigma_adds", "states_new", "frontier_vertices", "sum_int_len", "rade_num", "max_hits")


@pytest.fixture(scope="module")
def M():
    from paper_2304_08356_gb300 import build as B
    B.build()
    from paper_2304_08356_gb300 import mantra
    return mantra


def _cat(*parts):
    return tuple(np.concatenate([np.asarray(p[k]) for p in parts]).astype(np.uint32) for k in range(3))


def _star(width, ties):
    """width sources -> hub 0 -> width others -> hub 1 -> width sinks: a level of
    width vertices, and hub 1 with as many states (few with ties)."""
    src = 2 + np.arange(width)
    mid, out = src + width, src + 2 * width
    late = np.arange(width) % 5 if ties else np.arange(width)
    zero, one = np.zeros(width), np.ones(width)
    return _cat((src, zero, 1 + np.arange(width) % 7), (zero, mid, 10 + late), (mid, one, 10 + width + late),
                (one, out, 9 * width + late)), 3 * width + 2


def _hub(k):
    """0 -> 1 at k times, 1 -> 2 once later: k states of one vertex on the optimal paths."""
    return _cat((np.zeros(k), np.ones(k), 1 + np.arange(k)), ([1, 2], [2, 0], [k + 5, k + 9])), 3


def _combs(levels, leaves):
    """A chain with an edge from every chain vertex to every leaf, at times that
    fall along the chain: every leaf gets a new, earlier state on every level."""
    c = np.arange(levels)
    chain = (c[:-1], c[1:], c[:-1] + 1)
    u, w = np.meshgrid(c, np.arange(leaves), indexing="ij")
    comb = (u.ravel(), levels + w.ravel(), 3 * levels - u.ravel())
    far = levels + leaves + np.arange(leaves)     # reached from nowhere, with late in-edges
    return _cat(chain, comb, (far[:-1], far[1:], np.full(leaves - 1, 9 * levels))), levels + 2 * leaves


CASES = {
    "toy": lambda: (synth.uniform_small(n=60, m=900, t_lo=1, t_hi=8, seed=4), 60),
    "ties": lambda: (synth.uniform_small(n=700, m=30000, t_lo=1, t_hi=40, seed=6), 700),
    "bursty": lambda: (synth.chung_lu_bursty(n=2500, m=60000, seed=9), 2500),
    "spread": lambda: (synth.chung_lu_uniform_t(n=3000, m=70000, seed=2), 3000),
    "star 255": lambda: _star(255, True),
    "star 256": lambda: _star(256, False),
    "star 257": lambda: _star(257, True),
    "star 3000": lambda: _star(3000, True),
    "hub 257": lambda: _hub(257),
    "hub 9000": lambda: _hub(9000),
    "past the path-state cap": lambda: _hub(80000),
    "past the event cap": lambda: _combs(150, 100),
}


@pytest.mark.parametrize("smem", ["0", "1"])
@pytest.mark.parametrize("name", list(CASES))
def test_hop_equals_oracle(M, monkeypatch, name, smem):
    monkeypatch.setenv("MANTRA_BFS_SMEM", smem)
    (u, v, t), n = CASES[name]()
    g, o = M.Graph(u, v, t, n=n), O.Graph(u, v, t, n=n)
    few = name in ("hub 9000", "past the path-state cap", "past the event cap", "star 3000")
    r = 60 if few else 120
    for opt in (0, 1):
        for est in (0, 1):
            _, hits, info = g.estimate(opt, 0.05, 0.1, 3, fixed_r=r, estimator=est)
            _, ohits, oinfo = o.estimate(opt, 0.05, 0.1, 3, fixed_r=r, estimator=est)
            assert np.array_equal(hits, ohits), (opt, est)
            for k in COUNTERS:
                assert info[k] == oinfo[k], (opt, est, k)
        assert g.sample_paths(opt, 8, 5, 40, edges=True) == o.samples(opt, 8, 5, 40, edges=True)
    g.free()


@pytest.mark.parametrize("nt", ["256", "512", "1024"])
@pytest.mark.parametrize("name", ["ties", "bursty", "star 257"])
def test_hop_full_searches_equal_oracle(M, monkeypatch, name, nt):
    monkeypatch.setenv("MANTRA_BFS_NT", nt)
    (u, v, t), n = CASES[name]()
    g, o = M.Graph(u, v, t, n=n), O.Graph(u, v, t, n=n)
    st, reach = g.temporal_stats(0, 0.1, 5, r_override=50)
    oreach, odlb = o.stats_counts(0, 5, 50)
    assert st["d_lb"] == odlb and np.array_equal(reach, oreach)
    assert np.array_equal(g.temporal_closeness(1, 0.1, 5, r_override=50)[0], o.closeness(1, 5, 50)[0])
    g.free()
