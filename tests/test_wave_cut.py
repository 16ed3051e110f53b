"""The cut of the edge stream into waves (csrc/waves.h), run without a GPU: every
edge is in exactly one wave of at most 32 consecutive edges, no wave has an edge
that depends on another time of the same wave, and the steps of several waves are
flagged, whatever stands before a long step and wherever in a part it begins."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_08356_gb300", "csrc")
PART, STEP, BIG, LAST = 128, 512, 1, 2      # edges per part, waves per step, flags


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("wave") / "wave_driver")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "wave_driver.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def hub_stream(before, step, after, periods, n=1000, lead=0, seed=0):
    """A hub 0 that gets `before` single contacts, then sends to `step` vertices at
    one time, then `after` single contacts out, over and over; `lead` contacts among
    others shift it against the parts."""
    rng = np.random.default_rng(seed)
    u, v, t, now = [], [], [], 0
    for k in range(lead):
        now += 1
        u.append(1 + k % (n - 2)); v.append(2 + k % (n - 2)); t.append(now)
    for _ in range(periods):
        for _ in range(before):
            now += 1
            u.append(int(rng.integers(1, n))); v.append(0); t.append(now)
        now += 1
        for w in rng.choice(np.arange(1, n), step, replace=False):
            u.append(0); v.append(int(w)); t.append(now)
        for _ in range(after):
            now += 1
            u.append(0); v.append(int(rng.integers(1, n))); t.append(now)
    return tuple(np.asarray(x, np.uint32) for x in (u, v, t))


def sorted_stream(u, v, t):
    o = np.lexsort((v, u, t))
    return u[o].tolist(), v[o].tolist(), t[o].tolist()


def dependencies(u, v, t):
    """One past the last earlier edge, of another time, into an end of the edge."""
    last, dep, i = {}, [0] * len(t), 0
    while i < len(t):
        e = i
        while e < len(t) and t[e] == t[i]:
            dep[e] = max(last.get(u[e], 0), last.get(v[e], 0))
            e += 1
        for k in range(i, e):
            last[v[k]] = k + 1
        i = e
    return dep


def cut(driver, tmp_path, t, dep):
    src, dst = str(tmp_path / "in.bin"), str(tmp_path / "out.bin")
    with open(src, "wb") as f:
        f.write(np.uint64(len(t)).tobytes() + np.asarray(t, np.uint32).tobytes() + np.asarray(dep, np.uint32).tobytes())
    subprocess.run([driver, src, dst], check=True)
    raw = np.fromfile(dst, np.uint32)
    k = int(raw[2])
    return bool(raw[0]), int(raw[1]), raw[3:3 + k].tolist(), raw[3 + k:].tolist()


def check(driver, tmp_path, u, v, t):
    u, v, t = sorted_stream(u, v, t)
    dep, m = dependencies(u, v, t), len(t)
    fit, marks, first, flags = cut(driver, tmp_path, t, dep)
    assert fit and marks == 1 and first[0] == 0
    times = np.unique(np.asarray(t), return_counts=True)
    long_steps = set(times[0][times[1] > 32].tolist())
    for w, (a, b) in enumerate(zip(first, first[1:] + [m])):
        assert 0 < b - a <= 32                        # so no edge is lost
        assert all(dep[i] <= a for i in range(a, b))  # read before the wave, applied together
        if t[a] in long_steps:
            assert t[a] == t[b - 1] and flags[w] & BIG
            assert bool(flags[w] & LAST) == (b == m or t[b] != t[a])
        else:
            assert flags[w] == 0
            assert (a == 0 or t[a - 1] != t[a]) and (b == m or t[b - 1] != t[b])   # whole steps
    return first


@pytest.mark.parametrize("before,step,after,periods", [(127, 33, 160, 30), (150, 40, 177, 60), (300, 100, 301, 40),
                                                       (127, 40, 5, 40), (126, 64, 200, 30), (90, 600, 90, 20)])
def test_every_edge_is_in_one_wave(driver, tmp_path, before, step, after, periods):
    check(driver, tmp_path, *hub_stream(before, step, after, periods))


@pytest.mark.parametrize("lead", range(PART - 6, PART + 2))
@pytest.mark.parametrize("step", [33, 64, 257])
def test_long_step_at_the_end_of_a_part(driver, tmp_path, lead, step):
    """One-edge waves up to the last places of the first part, then the step."""
    check(driver, tmp_path, *hub_stream(lead, step, 300, 1))
    check(driver, tmp_path, *hub_stream(40, step, 300, 2, lead=lead))


def test_random_streams(driver, tmp_path):
    for seed in range(40):
        rng = np.random.default_rng(seed)
        n, m = int(rng.integers(3, 200)), int(rng.integers(1, 3000))
        u = rng.integers(0, n, m).astype(np.uint32)
        v = ((u + 1 + rng.integers(0, n - 1, m)) % n).astype(np.uint32)
        t = rng.integers(0, int(rng.integers(1, 2 * m + 2)), m).astype(np.uint32)
        check(driver, tmp_path, u, v, t)


@pytest.mark.parametrize("edges", [32 * STEP, 32 * STEP + 1])
def test_longest_step(driver, tmp_path, edges):
    t = [1] + [2] * edges + [3] * 5
    fit, marks, first, _ = cut(driver, tmp_path, t, [0] * len(t))
    assert fit == (edges <= 32 * STEP)
    if fit:
        assert marks == 1 and first == [0] + list(range(1, 1 + edges, 32)) + [1 + edges]


@pytest.mark.parametrize("waves", [0, 1, (1 << 27) - 8, (1 << 27) - 7, 1 << 27, (1 << 27) + 1, 1 << 31, (1 << 32) - 1])
def test_places_fit_in_32_bits(driver, waves):
    """A place is 32 * wave + lane; the last one of the last batch must not wrap."""
    last = (waves + 7) // 8 * 8 * 32 - 1
    r = subprocess.run([driver, "--indexable", str(waves)], capture_output=True, text=True, check=True)
    assert int(r.stdout) == (1 if last < 1 << 32 else 0)
