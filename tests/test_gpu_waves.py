"""pfm on streams whose waves are hard to cut (csrc/waves.h, csrc/k_sweep.cu): a
hub with a run of single contacts and then a time step of several waves, at every
place of a part of the cut, and arrivals in every wave of a batch.  Hits, estimates
and work counters equal the oracle's, and edges_expanded (0 unless the
label-correcting search ran) shows that the sweep ran."""
import numpy as np
import pytest

from oracle import oracle as O
from test_gpu_sweep import COUNTERS, _layers
from test_wave_cut import PART, hub_stream

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_2304_08356_gb300 import build as B
    B.build()
    from paper_2304_08356_gb300 import mantra
    return mantra


def equal(M, tri, n, r, swept=True):
    g, o = M.Graph(*tri, n=n), O.Graph(*tri, n=n)
    _, hits, info = g.estimate(2, 0.05, 0.1, 3, fixed_r=r)
    _, ohits, oinfo = o.estimate(2, 0.05, 0.1, 3, fixed_r=r)
    assert np.array_equal(hits, ohits)
    for k in COUNTERS:
        assert info[k] == oinfo[k], k
    assert (info["edges_expanded"] == 0) == swept
    g.free()


@pytest.mark.parametrize("before,step,after,periods", [(127, 33, 160, 60), (150, 40, 177, 60), (300, 100, 301, 40)])
def test_hub_then_broadcast(M, monkeypatch, before, step, after, periods):
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "sweep")
    equal(M, hub_stream(before, step, after, periods), 1000, 600)


@pytest.mark.parametrize("lead", range(PART - 4, PART + 1))
def test_step_at_the_end_of_a_part(M, monkeypatch, lead):
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "sweep")
    equal(M, hub_stream(lead, 40, 300, 1, n=60), 60, 600)


def test_hub_then_broadcast_by_default(M, monkeypatch):
    """More than 2^16 edges and samples enough that the rules choose the sweep."""
    monkeypatch.delenv("MANTRA_PFM_KERNEL", raising=False)
    equal(M, hub_stream(127, 33, 160, 300), 1000, 40000)


def test_arrival_in_every_wave_of_a_batch(M, monkeypatch):
    """A chain has a wave per edge: with all pairs drawn, z is reached in the first
    to the last wave of a batch of eight, where the sample's last time is read back
    from the records just written."""
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "sweep")
    c = np.arange(40)
    tri = tuple(x.astype(np.uint32) for x in (c, c + 1, 3 * c + 5))
    equal(M, tri, 41, 6000)
    g, o = M.Graph(*tri, n=41), O.Graph(*tri, n=41)
    got = g.sample_paths(2, 8, 0, 3000, cap=42)
    assert got == o.samples(2, 8, 0, 3000, cap=42)
    g.free()


def _layered(width, depth, lead=0, extra=0):
    """Complete bipartite steps of width^2 edges after a chain of `lead` edges, which
    shifts them against the batches of waves; `extra` more edges in the second step."""
    (u, v, t), n = _layers(width, depth)
    c = np.arange(lead)
    u = np.r_[n + c, u.astype(np.int64)]
    v = np.r_[n + c + 1, v.astype(np.int64)]
    t = np.r_[c + 1, t.astype(np.int64) + lead]
    n += lead + 1
    if extra:
        u, v, t = np.r_[u, n + np.arange(extra)], np.r_[v, np.full(extra, n + extra)], np.r_[t, np.full(extra, 2 + lead)]
        n += extra + 1
    return tuple(x.astype(np.uint32) for x in (u, v, t)), n


@pytest.mark.parametrize("width,depth", [(6, 12), (8, 9), (17, 6), (46, 4), (128, 3)])
def test_steps_of_several_waves(M, monkeypatch, width, depth):
    """36 to 16,384 edges at one time (2 to 512 waves), every one with in-edges of the
    same slot: read before any of them is applied."""
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "sweep")
    tri, n = _layered(width, depth)
    for r in (33, 300):
        equal(M, tri, n, r)


@pytest.mark.parametrize("lead", range(9))
def test_steps_across_batches(M, monkeypatch, lead):
    """A step of ten waves that begins in the first to the last wave of a batch."""
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "sweep")
    tri, n = _layered(17, 5, lead=lead)
    equal(M, tri, n, 300)


def test_step_past_the_limit_is_searched(M, monkeypatch):
    """16,385 edges at one time: the graph has no waves."""
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "sweep")
    tri, n = _layered(128, 3, extra=1)
    assert np.unique(tri[2], return_counts=True)[1].max() == 16385
    equal(M, tri, n, 300, swept=False)
