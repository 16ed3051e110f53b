"""Launch shapes that mantra_tune chooses, read from the library's launch lines:
RTB and fsfm (k_bfs) run with the shape that was fastest for that kernel, large sh
rounds with k_hop's, and small ones with the default.  And the pfm search's shapes
and placements (k_pfm_cta) against the oracle with that kernel named."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

from oracle import oracle as O
from paper_2304_08356_gb300 import synth

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUN = """
import sys
from paper_2304_08356_gb300 import mantra as M, synth
g = M.Graph(*synth.chung_lu_bursty(n=4000, m=90000, seed=17))
def call(name, *a, **k):
    print("call", name, file=sys.stderr, flush=True)
    g.estimate(*a, **k)
call("small default", 0, 0.05, 0.1, 3, fixed_r=200)
print("call tune", file=sys.stderr, flush=True)
res = g.tune()
print("call none", res["bfs_threads"], res["bfs_bitmap_shared"], file=sys.stderr, flush=True)
call("fsfm", 3, 0.05, 0.1, 3, fixed_r=9000)
call("rtb", 0, 0.05, 0.1, 3, fixed_r=3000, estimator=2)
call("sh", 0, 0.05, 0.1, 3, fixed_r=9000)
call("small", 0, 0.05, 0.1, 3, fixed_r=200)
"""


def test_every_kernel_runs_its_own_choice():
    env = dict(os.environ, MANTRA_LOG_LAUNCHES="1")
    r = subprocess.run([sys.executable, "-c", RUN], capture_output=True, text=True, cwd=ROOT, env=env)
    assert r.returncode == 0, r.stderr
    lines, name, reported = {}, None, None
    for ln in r.stderr.splitlines():
        if ln.startswith("call "):
            name = ln[5:]
            if name.startswith("none"):
                reported = tuple(int(x) for x in name.split()[1:])
            continue
        m = re.match(r"mantra-launch kernel=(\S+) nt=(\d+) mode=(\d+) samples=(\d+) .* ms=([0-9.]+)$", ln)
        if m:
            lines.setdefault(name, []).append((m[1], (int(m[2]), int(m[3])), int(m[4]), float(m[5])))
    probes = [x for x in lines["tune"] if x[0] == "k_bfs"]
    r_max = max(x[2] for x in probes)
    best = {}
    for _, shape, n, ms in probes:
        if n == r_max:
            best[shape] = min(ms, best.get(shape, 1e9))
    assert len(best) == 6                              # three sizes, two placements
    for call in ("fsfm", "rtb"):
        (kernel, shape, _, _), = lines[call]
        assert kernel == "k_bfs" and best[shape] <= 1.03 * min(best.values()), (shape, best)
    (kernel, shape, _, _), = lines["sh"]
    assert kernel == "k_hop" and shape == reported
    assert lines["small"][0][:2] == lines["small default"][0][:2]


@pytest.mark.parametrize("nt", ["256", "512"])
@pytest.mark.parametrize("smem", ["0", "1", "16", "staged"])
def test_pfm_search_shapes_equal_oracle(monkeypatch, nt, smem):
    from paper_2304_08356_gb300 import build as B, mantra as M
    B.build()
    monkeypatch.setenv("MANTRA_PFM_KERNEL", "cta")
    monkeypatch.setenv("MANTRA_PFM_CTA_NT", nt)
    monkeypatch.setenv("MANTRA_PFM_CTA_SMEM", "0" if smem == "staged" else smem)
    monkeypatch.setenv("MANTRA_PFM_STAGE", "1" if smem == "staged" else "0")
    tri = synth.chung_lu_bursty(n=4000, m=90000, seed=17)
    g, o = M.Graph(*tri), O.Graph(*tri)
    _, hits, info = g.estimate(2, 0.05, 0.1, 3, fixed_r=2000)
    _, ohits, oinfo = o.estimate(2, 0.05, 0.1, 3, fixed_r=2000)
    assert info["edges_expanded"] > 0                  # the search ran
    assert np.array_equal(hits, ohits)
    assert info["rade_num"] == oinfo["rade_num"] and info["sigma_adds"] == oinfo["sigma_adds"]
    g.free()
