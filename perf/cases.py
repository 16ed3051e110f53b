"""The work that a user of the library has it do, as cases that can be timed.

A case is one pass through the public calls of ``paper_2304_08356_gb300.mantra``:
Algorithm 1 on one graph, on a batch of graphs, with the graph load in front
of it, or Algorithm 2.  Graphs are seeded stand-ins of the paper's data sets
(power-law degrees, bursty contacts or uniform times), drawn on the GPU and
handed to the library as host arrays, as a user has them.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the loaded graphs (or the host arrays) and the arguments
    run(state)          one pass
    work(case)          bytes that a pass cannot do without
    exact(case, seed)   the results from plain Python / torch, where that is quick
"""
import math

import numpy as np
import torch

import paper_2304_08356_gb300.mantra as M

# graph shapes: "bursty" Chung-Lu skeleton with bursts of contacts (gamma 2.3),
# "spread" Chung-Lu pairs with uniform times over [0, 2^24) (gamma 2.1),
# "ties" uniform pairs over few time steps (many equal times)


def listed():
    return [
        # the smallest call in use: a toy graph, a fixed number of samples (launches and latency count)
        dict(name="toy_sh", kind="estimate", graph="ties", n=100, m=2000, opt="sh", r=1000),
        # a small resident graph asked for a quick answer, as a serving process gets it
        dict(name="small_pfm", kind="estimate", graph="bursty", n=1000, m=25000, opt="pfm", eps=0.05),
        # a mid-size graph of odd sizes, moderate accuracy
        dict(name="mid_sfm", kind="estimate", graph="bursty", n=5003, m=125077, opt="sfm", eps=0.02),
        # the ordinary run: a 20,000-node graph at eps = 0.01, shortest paths
        dict(name="run_sh", kind="estimate", graph="bursty", n=20000, m=500000, opt="sh", eps=0.01),
        # the ordinary run, prefix-foremost paths
        dict(name="run_pfm", kind="estimate", graph="bursty", n=20000, m=500000, opt="pfm", eps=0.01),
        # end to end: host triples in, the graph loaded, sh + sfm + pfm as one batch, host results out
        dict(name="load_and_run3", kind="load", graph="bursty", n=20000, m=500000, eps=0.01),
        # many uneven graphs in one batch (ragged sizes, mixed optimalities)
        dict(name="batch_uneven", kind="batch", graph="bursty", count=96, n=500, n_hi=20000, deg=20, eps=0.02),
        # a large graph: one round's worth of samples of a high-accuracy run, both search kernels
        dict(name="large_sfm", kind="estimate", graph="spread", n=1000000, m=20000000, opt="sfm", r=4096),
        dict(name="large_pfm", kind="estimate", graph="spread", n=1000000, m=20000000, opt="pfm", r=3001),
        # temporal-edge betweenness (App. A) on a graph of odd sizes
        dict(name="edges_sfm", kind="estimate", graph="spread", n=50021, m=1000423, opt="sfm", eps=0.02, target=2),
        # the overlap (ob) estimator: every optimal path's internal vertices counted
        dict(name="ob_sh", kind="estimate", graph="bursty", n=20000, m=500000, opt="sh", eps=0.02, estimator=1),
        # Algorithm 2 and closeness: full searches from sampled sources
        dict(name="stats_sfm", kind="stats", graph="bursty", n=20000, m=500000, opt="sfm", r=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["estimate"] * 6 + ["eps"] * 4 + ["load", "batch", "stats", "ob", "rtb"])
    shape = rng.choice(["bursty", "bursty", "spread", "ties"])
    opt = rng.choice(["sh", "sfm", "pfm", "pfm", "sh", "sfm", "fsfm"])
    deg = rng.uniform(8.0, 30.0)
    if kind == "estimate":        # a fixed number of samples, any size
        n = _log(rng, 100, 500000)
        m = int(n * deg)
        r = min(_log(rng, 100, 20000), max(64, int(2e10 / m)))
        return dict(kind="estimate", graph=shape, n=n, m=m, opt=opt, r=r, target=rng.choice([0, 0, 0, 1, 2] if shape != "ties" else [0, 0, 1]))
    if kind == "eps":             # progressive sampling to an accuracy
        n = _log(rng, 300, 50000)
        eps = rng.choice([0.05, 0.03, 0.02, 0.01]) if n < 25000 else rng.choice([0.05, 0.03, 0.02])
        return dict(kind="estimate", graph=shape, n=n, m=int(n * deg), opt=opt, eps=eps)
    if kind == "load":
        n = _log(rng, 500, 50000)
        return dict(kind="load", graph=shape, n=n, m=int(n * deg), eps=rng.choice([0.05, 0.02]))
    if kind == "batch":
        return dict(kind="batch", graph=shape, count=rng.randint(5, 60), n=_log(rng, 200, 1000),
                    n_hi=_log(rng, 3000, 20000), deg=rng.randint(8, 25), eps=rng.choice([0.05, 0.02]))
    if kind == "stats":
        n = _log(rng, 300, 50000)
        return dict(kind="stats", graph=shape, n=n, m=int(n * deg), opt=opt, r=rng.randint(20, 300))
    n = _log(rng, 100, 20000 if kind == "ob" else 5000)
    return dict(kind="estimate", graph=shape, n=n, m=int(n * deg), opt=opt, r=_log(rng, 100, 3000),
                estimator=1 if kind == "ob" else 2)


# ---------------------------------------------------------------- inputs

def _pairs(n, gamma, k, gen):
    """k ordered pairs u != v, both ends drawn by power-law weights under a random id permutation."""
    dev = gen.device
    w = torch.arange(1, n + 1, device=dev, dtype=torch.float64) ** (-1.0 / (gamma - 1.0))
    p = torch.empty_like(w)
    p[torch.randperm(n, device=dev, generator=gen)] = w / w.sum()
    cdf = torch.cumsum(p, 0)
    cdf[-1] = 1.0

    def ends(c):
        return torch.searchsorted(cdf, torch.rand(c, device=dev, dtype=torch.float64, generator=gen),
                                  right=True).clamp_(max=n - 1)
    u, v = ends(k), ends(k)
    for _ in range(64):
        bad = (u == v).nonzero().flatten()
        if not bad.numel():
            break
        v[bad] = ends(bad.numel())
    v = torch.where(u == v, (u + 1) % n, v)
    return u, v


def _triples(shape, n, m, seed, distinct=False):
    """Host uint32 arrays u, v, t of m temporal edges on n nodes (distinct: no triple twice)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dev = gen.device
    asked = m
    if distinct:
        m = m + m // 16 + 64
    if shape == "ties":
        u = torch.randint(0, n, (m,), device=dev, generator=gen)
        v = torch.randint(0, n - 1, (m,), device=dev, generator=gen)
        v = v + (v >= u)
        t = torch.randint(1, max(200, m // 40) + 1, (m,), device=dev, generator=gen)
    elif shape == "spread":
        u, v = _pairs(n, 2.1, m, gen)
        t = torch.randint(0, 1 << 24, (m,), device=dev, generator=gen)
    else:
        k = m                                     # bursts of K ~ Geometric(0.3) contacts, the last one truncated
        K = 1 + torch.floor(torch.log1p(-torch.rand(k, device=dev, dtype=torch.float64, generator=gen))
                            / math.log(0.7)).long()
        k = int(torch.searchsorted(torch.cumsum(K, 0), m)) + 1
        K = K[:k]
        u, v = _pairs(n, 2.3, k, gen)
        centre = torch.rand(k, device=dev, dtype=torch.float64, generator=gen) * 1e6
        owner = torch.repeat_interleave(torch.arange(k, device=dev), K)[:m]
        gap = -1000.0 * torch.log1p(-torch.rand(m, device=dev, dtype=torch.float64, generator=gen))
        first = torch.ones(m, device=dev, dtype=torch.bool)
        first[1:] = owner[1:] != owner[:-1]
        gap[first] = 0.0
        c = torch.cumsum(gap, 0)
        start = first.nonzero().flatten()
        base = c[start][owner]
        t = torch.round(centre[owner] + c - base).clamp_(0, 1e6).long()
        u, v = u[owner], v[owner]
    if distinct:
        key = torch.unique((t * n + u) * n + v)
        key = key[torch.randperm(key.numel(), device=dev, generator=gen)[:asked]]
        if key.numel() < asked:
            raise ValueError("fewer than %d distinct edges" % asked)
        t, u, v = key // (n * n), key // n % n, key % n
    return tuple(x.to(torch.int32).cpu().numpy().view(np.uint32) for x in (u, v, t))


def _batch_sizes(case):
    """Log-uniform sizes (the same for every seed: the shapes belong to the case)."""
    rng = np.random.default_rng(case["count"])
    return np.exp(rng.uniform(math.log(case["n"]), math.log(case["n_hi"]), case["count"])).astype(int)


# ---------------------------------------------------------------- passes

def prepare(case, seed):
    kind, shape = case["kind"], case["graph"]
    state = dict(case=case, seed=seed & 0xFFFFFFFF)
    if kind == "batch":
        state["problems"] = [
            dict(graph=M.Graph(*_triples(shape, int(n), case["deg"] * int(n), seed * 1000 + k), n=int(n)),
                 opt=("sh", "sfm", "pfm")[k % 3], eps=case["eps"], delta=0.1, seed=state["seed"] + k)
            for k, n in enumerate(_batch_sizes(case))]
    elif kind == "load":
        state["triples"] = _triples(shape, case["n"], case["m"], seed)
    else:
        g = M.Graph(*_triples(shape, case["n"], case["m"], seed, case.get("target") == 2), n=case["n"])
        g.family_size(case.get("target", 0))      # the edge ids, which a program asks for once
        state["graph"] = g
    return state


_COUNTS = ("r", "rounds", "omega", "s1", "bootstrap", "sum_int_len", "max_hits", "rade_num", "edges_scanned",
           "sigma_adds", "states_new", "frontier_vertices")


def _filled(x, size):
    """x with zeros up to a size that does not depend on the graph drawn (its own size where that is fixed)."""
    return x if x.size == size else np.concatenate([x, np.zeros(size - x.size, x.dtype)])


def _outputs(est, hits, info, size):
    est, hits = _filled(est, size), _filled(hits, size)
    return dict(est=est, hits=hits, counts=np.array([info[k] for k in _COUNTS], dtype=np.int64),
                bounds=np.array([info["xi"], info["vhat"], info["rho_hat"]]))


def _joined(results):
    """The results of a batch, one after another."""
    if any(status for _, _, _, status in results):
        raise RuntimeError("a problem of the batch failed: %s" % [s for _, _, _, s in results])
    outs = [_outputs(e, h, i, e.size) for e, h, i, _ in results]
    return {k: np.concatenate([o[k] for o in outs]) for k in outs[0]}


def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "estimate":
        return _outputs(*state["graph"].estimate(case["opt"], case.get("eps", 0.05), 0.1, seed,
                                                 fixed_r=case.get("r", 0), target=case.get("target", 0),
                                                 estimator=case.get("estimator", 0)),
                        size=case["m"] if case.get("target", 0) else case["n"])
    if kind == "batch":
        return _joined(M.estimate_batch(state["problems"]))
    if kind == "load":
        g = M.Graph(*state["triples"], n=case["n"])
        out = _joined(M.estimate_batch([dict(graph=g, opt=opt, eps=case["eps"], delta=0.1, seed=seed)
                                        for opt in ("sh", "sfm", "pfm")]))
        g.free()
        return out
    g = state["graph"]
    st, reach = g.temporal_stats(case["opt"], 0.05, seed, r_override=case["r"])
    sums, closeness, _ = g.temporal_closeness(case["opt"], 0.05, seed, r_override=case["r"])
    return dict(reach=_filled(reach, case["n"]), sums=sums, closeness=closeness, d=np.array([st["d_lb"], st["d_tau"]], dtype=np.int64),
                averages=np.array([st["zeta"], st["psi"], st["rho"]]))


def work(case):
    """The edge triples (12 B) read once, the results (16 B an entry) written once."""
    kind = case["kind"]
    if kind == "batch":
        n = case["count"] * (case["n"] + case["n_hi"]) / 2.0
        return dict(bytes=(12.0 * case["deg"] + 16.0) * n, flops=0.0)
    entries = case["m"] if case.get("target", 0) else case["n"]
    return dict(bytes=12.0 * case["m"] + 16.0 * entries * (3 if kind == "load" else 1), flops=0.0)


# ---------------------------------------------------------------- plain 64-bit results

def _philox(seed, i, dom, att):
    x = [i & 0xFFFFFFFF, i >> 32, dom, att]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = 0xD2511F53 * x[0], 0xCD9E8D57 * x[2]
        x = [(b >> 32) ^ x[1] ^ k0, b & 0xFFFFFFFF, (a >> 32) ^ x[3] ^ k1, a & 0xFFFFFFFF]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x


def _below(N, seed, i, dom, bits):
    """Uniform in [0, N): the block masked to the bits of N - 1, rejected when N or more."""
    mask = (1 << (N - 1).bit_length()) - 1
    for att in range(1 << 16):
        w = _philox(seed, i, dom, att)
        x = (sum(v << (32 * k) for k, v in enumerate(w)) & ((1 << bits) - 1)) & mask
        if x < N:
            return x
    raise RuntimeError("no draw")


class _Plain:
    """Optimal temporal paths by dictionaries: the problem statement on a small graph."""

    def __init__(self, triples):
        edges = sorted({(t, u, v) for u, v, t in zip(*(x.tolist() for x in triples)) if u != v})
        self.edges, self.out, self.inn, self.last = edges, {}, {}, {}
        for t, u, v in edges:
            self.out.setdefault(u, []).append((t, v))
            self.inn.setdefault((v, t), []).append(u)
            self.last[v] = t

    def levels(self, s, z):
        """Levels of {(v, t): paths from s}; the last one holds z's appearances."""
        tz = self.last.get(z)
        lev, seen = [{(s, -1): 1}], set()
        while tz is not None and lev[-1]:
            new = {}
            for (u, tu), c in lev[-1].items():
                for t, v in self.out.get(u, ()):
                    if t > tu and (t < tz or (t == tz and v == z)) and (v, t) not in seen:
                        new[(v, t)] = new.get((v, t), 0) + c
            ends = {a: c for a, c in new.items() if a[0] == z}
            if ends:
                return lev + [ends]
            seen.update(new)
            lev.append(new)
        return None

    def draw(self, opt, s, z, pick):
        """The vertices of one optimal s-z path (pick(N): uniform in [0, N)), or []."""
        if opt == "pfm":
            fa, cnt = {s: -1}, {s: 1}
            for t, u, v in self.edges:
                if u in fa and fa[u] < t and v != s and fa.get(v, t) == t:
                    fa[v] = t
                    cnt[v] = cnt.get(v, 0) + cnt[u]
            if z not in fa:
                return []
            x, path = pick(cnt[z]), [z]
            while path[-1] != s:
                v = path[-1]
                for w in self.inn[(v, fa[v])]:
                    if w in fa and fa[w] < fa[v]:
                        if x < cnt[w]:
                            path.append(w)
                            break
                        x -= cnt[w]
            return path[::-1]
        lev = self.levels(s, z)
        if lev is None:
            return []
        ends = sorted(lev[-1], key=lambda a: a[1])
        ends = ends[:1] if opt == "sfm" else ends
        x = pick(sum(lev[-1][a] for a in ends))
        for cur in ends:
            if x < lev[-1][cur]:
                break
            x -= lev[-1][cur]
        path = [z]
        for k in range(len(lev) - 2, -1, -1):
            at = {}
            for w, tw in lev[k]:
                at.setdefault(w, []).append(tw)
            done = False
            for w in self.inn[cur]:
                for tw in sorted(at.get(w, ())):
                    if tw < cur[1] and not done:
                        if x < lev[k][(w, tw)]:
                            nxt, done = (w, tw), True
                        else:
                            x -= lev[k][(w, tw)]
            cur = nxt
            path.append(cur[0])
        return path[::-1]


def _exact_estimate(case, seed):
    n, r, c = case["n"], case["r"], 25
    g = _Plain(_triples(case["graph"], n, case["m"], seed))
    seed &= 0xFFFFFFFF
    hits, S = np.zeros(n, dtype=np.int64), np.zeros((c, n), dtype=np.int64)
    for i in range(r):
        a, b = divmod(_below(n * (n - 1), seed, i, 0, 64), n - 1)
        s, z = a, b + (b >= a)
        path = g.draw(case["opt"], s, z, lambda N: _below(N, seed, i, 1, 128))
        if len(path) > 2:
            lam = _philox(seed, i, 2, 0)[0]
            sign = np.array([1 if (lam >> j) & 1 else -1 for j in range(c)])
            for v in path[1:-1]:
                hits[v] += 1
                S[:, v] += sign
    W, L = hits.max() / r, math.log(4.0 / (0.1 / 4.0))
    Rc = S.max(axis=1).sum() / (c * r)
    Rt = Rc + math.sqrt(4.0 * W * L / (c * r))
    R = Rt + L / r + math.sqrt((L / r) ** 2 + 2.0 * L * Rt / r)
    xi = 2.0 * R + math.sqrt(2.0 * L * (W + 4.0 * R) / r) + L / (3.0 * r)
    return dict(est=hits / r, hits=hits.astype(np.uint64), counts=None, bounds=np.array([xi, W, 0.0]))


def _exact_stats(case, seed):
    n, rs = case["n"], case["r"]
    u, v, t = (torch.from_numpy(x.view(np.int32)).cuda().long() for x in _triples(case["graph"], n, case["m"], seed))
    keep = u != v
    u, v, t = u[keep], v[keep], t[keep]
    far = 1 << 40
    close = torch.zeros(n, dtype=torch.float64, device="cuda")
    count = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    for i in range(rs):
        s = _below(n, seed & 0xFFFFFFFF, i, 5, 64)
        arr = torch.full((n,), far, dtype=torch.int64, device="cuda")   # earliest arrival over paths of at most k edges
        arr[s] = -1
        dist = torch.zeros(n, dtype=torch.int64, device="cuda")
        for k in range(1, n + 1):
            cand = torch.where(t > arr[u], t, far)
            new = arr.scatter_reduce(0, v, cand, "amin")
            if torch.equal(new, arr):
                break
            dist[(arr == far) & (new < far)] = k
            arr = new
        got = dist > 0
        close[got] += 1.0 / dist[got].double()
        count += torch.bincount(dist[got], minlength=n + 1)
    h = torch.arange(n + 1, device="cuda", dtype=torch.float64)
    pairs = float(count.sum()) * n / rs
    psi = float((count * h).sum()) / max(1.0, float(count.sum()))
    zeta = pairs / (float(n) * (n - 1))
    return dict(reach=None, sums=None, closeness=(close * n / (float(rs) * (n - 1))).cpu().numpy(), d=None,
                averages=np.array([zeta, psi, zeta * (psi - 1.0)]))


def exact(case, seed):
    if case["kind"] == "stats" and case["opt"] in ("sh", "sfm") and case["r"] * case["m"] <= 2e8:
        return _exact_stats(case, seed)
    if (case["kind"] == "estimate" and case.get("r") and not case.get("estimator") and not case.get("target")
            and case["opt"] in ("sh", "sfm", "pfm") and case["r"] * case["m"] <= 4e6):
        return _exact_estimate(case, seed)
    return None
