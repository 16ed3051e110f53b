"""The pfm sweep (csrc/k_sweep.cu: 32 samples per warp over the stream's waves)
against the oracle: ragged sample counts, several edges per time step (arrivals
with several in-edges, so that paths are counted and drawn), path counts past
64 bits, and paths and path sets past its per-sample caps (both re-run by the
128-bit kernel).  Paths, hits, Rademacher sums and work counters are equal."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_08356_gb300 import synth

pytestmark = pytest.mark.gpu

COUNTERS = ("edges_scanned", "sigma_adds", "sum_int_len", "rade_num", "max_hits")


@pytest.fixture(scope="module")
def M():
    from paper_2304_08356_gb300 import build as B
    B.build()
    from paper_2304_08356_gb300 import mantra
    return mantra


@pytest.fixture(autouse=True)
def force(monkeypatch):
    """The sweep on every graph: set before the loads, so that small graphs get waves."""
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "sweep")


def _layers(width, depth):
    """Complete bipartite steps: width^2 edges per time step, width^k paths."""
    a, b = np.meshgrid(np.arange(width), np.arange(width), indexing="ij")
    k = np.repeat(np.arange(depth), width * width)
    return (tuple(np.asarray(x, np.uint32) for x in (k * width + np.tile(a.ravel(), depth),
                                                     (k + 1) * width + np.tile(b.ravel(), depth), k + 1)),
            width * (depth + 1))


def _chain(length, diamond):
    """A path of the given length; with diamond, two ways over a step in its middle."""
    c = np.arange(length)
    u, v, t = c, c + 1, 3 * c + 5
    n = length + 1
    if diamond:                                  # k -> n -> k + 2 beside k -> k + 1 -> k + 2, at the same times
        k = length // 2
        u, v, t = np.r_[u, k, n], np.r_[v, n, k + 2], np.r_[t, 3 * k + 5, 3 * k + 8]
        n += 1
    return tuple(x.astype(np.uint32) for x in (u, v, t)), n


CASES = {
    "toy": lambda: (synth.uniform_small(n=60, m=900, t_lo=1, t_hi=300, seed=4), 60),
    "few times": lambda: (synth.uniform_small(n=300, m=6000, t_lo=1, t_hi=1200, seed=6), 300),
    "bursty": lambda: (synth.chung_lu_bursty(n=2500, m=60000, seed=9), 2500),
    "spread": lambda: (synth.chung_lu_uniform_t(n=3000, m=70000, seed=2), 3000),
    "layers": lambda: _layers(4, 9),
    "past 64 bits": lambda: _layers(5, 40),
    "long path": lambda: _chain(3000, False),
    "long path with a choice": lambda: _chain(1500, True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_sweep_equals_oracle(M, name):
    (u, v, t), n = CASES[name]()
    g, o = M.Graph(u, v, t, n=n), O.Graph(u, v, t, n=n)
    for r in (1, 31, 33, 300):
        for target in (0, 1, 2):
            est, hits, info = g.estimate(2, 0.05, 0.1, 3, fixed_r=r, target=target)
            oest, ohits, oinfo = o.estimate(2, 0.05, 0.1, 3, fixed_r=r, target=target)
            assert np.array_equal(hits, ohits) and np.array_equal(est, oest), (r, target)
            for k in COUNTERS:
                assert info[k] == oinfo[k], (r, target, k)
    assert g.sample_paths(2, 8, 5, 100, edges=True, cap=n + 1) == o.samples(2, 8, 5, 100, edges=True, cap=n + 1)
    g.free()


def test_sweep_progressive_and_batch(M):
    """Bootstrap and rounds, and a batch of uneven graphs in one launch."""
    gs = [synth.chung_lu_bursty(n=k, m=20 * k, seed=k) for k in (40, 700, 2000, 333)]
    probs, want = [], []
    for x, tri in enumerate(gs):
        o = O.Graph(*tri)
        probs.append(dict(graph=M.Graph(*tri), opt=2, eps=0.05, delta=0.1, seed=x))
        want.append(o.estimate(2, 0.05, 0.1, x))
    for (est, hits, info, status), (oest, ohits, oinfo) in zip(M.estimate_batch(probs), want):
        assert status == 0 and np.array_equal(hits, ohits) and np.array_equal(est, oest)
        assert info["r"] == oinfo["r"] and info["rounds"] == oinfo["rounds"]
        for k in COUNTERS:
            assert info[k] == oinfo[k], k
