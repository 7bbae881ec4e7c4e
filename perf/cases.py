"""The calls that are timed: what a user of this framework has it do.

Graphs are seeded synthetic bipartite graphs of the shapes that the benchmark
and the tests use: uniform ones, Chung-Lu power laws (expected degree of the
i-th vertex ~ (i + i0)^(-1/(exponent - 1)), the heaviest one a tenth of the
other layer unless stated) and the shopping shape (many users, few items).
Everything is drawn on the GPU, so a 300M-edge graph takes about a second.

A case's `kind` is the call that it makes:

  total     ButterflyGraph(...) then count(): one new graph, its total
  all       ButterflyGraph(...) then count_all(): every output of one new graph
  host_all  bfc_count_all_host: page-locked host arrays in and out
  vertices  count_vertices() on a prepared graph that the program keeps
  edges     count_edges() on a prepared graph that the program keeps
  noalloc   bfc_count_small_noalloc: a small graph, no allocation
  batch     bfc_prepare_batch then bfc_count_batch: many graphs, a total each
  plan      bfc_batch_plan_run: batches of one shape, no synchronisation
  estimate  estimate_butterflies: edge-sparsified samples and their estimate
"""
import math
import random

import numpy as np
import torch

import paper_1812_00283_gb300 as pkg
from paper_1812_00283_gb300 import ButterflyGraph, estimate_butterflies

SINGLE = ("total", "all", "host_all", "vertices", "edges", "noalloc", "estimate")


def _single(name, kind, num_u, num_l, edges, gamma_u, gamma_l, top_u=0.1, top_l=0.1, shuffled=False, **more):
    """A case on one graph.  gamma 0: uniform endpoints; top_u / top_l: the
    heaviest U / L vertex's expected degree as a share of the other layer;
    shuffled: neighbours in no order (lists as they arrive from an edge
    stream), else ascending."""
    c = dict(kind=kind, num_u=num_u, num_l=num_l, edges=edges, gamma_u=gamma_u, gamma_l=gamma_l,
             top_u=top_u, top_l=top_l, shuffled=shuffled, **more)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest calls: one little graph at a time, bound by launches and
        # host round trips (the uniform 2,000 x 3,000 graph of the tests)
        _single("small_total", "total", 2000, 3000, 20_000, 0.0, 0.0),
        # a caller that may not allocate (a real-time loop) on a small graph
        _single("small_noalloc", "noalloc", 12_007, 8_001, 150_001, 2.2, 2.1),
        # one graph of the batched workload's sizes counted by itself with all
        # outputs (per-vertex and per-edge features of a medium graph)
        _single("medium_all", "all", 20_011, 9_973, 300_007, 2.1, 2.3, shuffled=True),
        # a large graph of that range, total only (the per-graph arm of the batch)
        _single("medium_total", "total", 48_611, 31_013, 2_000_003, 2.0, 2.4),
        # the plain power-law benchmark: 20M edges, total
        _single("powerlaw_total", "total", 1_000_000, 500_000, 20_000_000, 2.1, 2.1),
        # a large request of the served stream, from host arrays into host arrays
        _single("large_host_all", "host_all", 1_000_000, 500_000, 5_000_000, 2.0, 2.0),
        # a kept graph whose per-vertex counts are asked for (ranking, anomaly scores)
        _single("kept_vertices", "vertices", 301_007, 152_003, 6_000_001, 2.2, 2.0),
        # a kept shopping graph whose per-edge counts are asked for (k-wing's first step)
        _single("kept_edges", "edges", 1_000_000, 10_000, 30_000_000, 2.5, 1.8, top_u=0.1, top_l=0.1),
        # the benchmark's headline: 300M edges, 10M users, 100k items, all outputs
        _single("shopping_all", "all", 10_000_000, 100_000, 300_000_000, 2.5, 1.8, top_u=0.1, top_l=0.1),
        # approximate counting of the power-law graph from 16 sparse samples
        _single("sparse_estimate", "estimate", 1_000_000, 500_000, 20_000_000, 2.1, 2.1, p=0.1, samples=16),
        # the batched workload: an eighth of its 4,096 graphs, prepared and counted
        dict(name="batch_512", kind="batch", graphs=512, sizes=4000),
        # a fixed-shape batch step, as a serving loop replays it
        dict(name="plan_64", kind="plan", graphs=64, sizes=5001),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["total", "total", "all", "all", "host_all", "vertices", "edges", "noalloc", "batch",
                       "plan", "estimate"])
    if kind in ("batch", "plan"):
        return dict(kind=kind, graphs=_log(rng, 16, 512), sizes=rng.randrange(1, 1 << 30))
    gu = 0.0 if rng.random() < 0.15 else rng.uniform(1.8, 2.6)
    gl = 0.0 if gu == 0.0 else rng.uniform(1.8, 2.6)
    if kind == "noalloc":
        edges = _log(rng, 5_000, 600_000)
        r = min(49_000, max(500, int(edges / rng.uniform(3, 40))))
        l = min(65_000 - r, 49_000, max(500, int(edges / rng.uniform(3, 40))))
    elif kind == "estimate":
        edges = _log(rng, 500_000, 20_000_000)
        r, l = int(edges / rng.uniform(5, 40)), int(edges / rng.uniform(5, 60))
    else:
        edges = _log(rng, 20_000, 20_000_000)
        r, l = max(300, int(edges / rng.uniform(3, 40))), max(300, int(edges / rng.uniform(3, 300)))
    edges = min(edges, r * l // 4)
    c = _single("", kind, r, l, edges, gu, gl, shuffled=rng.random() < 0.3)
    if kind == "estimate":
        c.update(p=round(rng.uniform(0.03, 0.2), 3), samples=rng.choice([4, 9, 16, 20]))
    return c


def _batch_sizes(case):
    """Per graph |U|, |L| log-uniform in [100, 50,000], edges log-uniform in
    [1,000, 2,000,000] clamped to half the pairs, exponents in [1.8, 2.6]."""
    rng = random.Random(case["sizes"])
    out = []
    for _ in range(case["graphs"]):
        r, l, m = _log(rng, 100, 50_000), _log(rng, 100, 50_000), _log(rng, 1_000, 2_000_000)
        out.append((r, l, min(m, r * l // 2), rng.uniform(1.8, 2.6), rng.uniform(1.8, 2.6), 0.1, 0.1))
    return out


def _sizes(case):
    if case["kind"] in SINGLE:
        return [tuple(case[k] for k in ("num_u", "num_l", "edges", "gamma_u", "gamma_l", "top_u", "top_l"))]
    return _batch_sizes(case)


def work(case):
    sizes = _sizes(case)
    r, l, m, kind = sum(s[0] for s in sizes), sum(s[1] for s in sizes), sum(s[2] for s in sizes), case["kind"]
    out = {"all": 8 * (m + r + l), "host_all": 8 * (m + r + l), "vertices": 8 * (r + l), "edges": 8 * m,
           "batch": 8 * len(sizes), "plan": 8 * len(sizes), "estimate": 8 * case.get("samples", 0) + 16}
    return {"bytes": 4 * (r + 1) + 4 * m + out.get(kind, 8), "flops": 0}


# ---- inputs -------------------------------------------------------------------

class _Layer:
    """Endpoint sampling of one layer of every graph: the inverse of the
    cumulative expected degree, then a random relabelling of the ids."""

    def __init__(self, n, m, gamma, top, gen):
        n, m, gamma, top = (np.asarray(a, dtype=np.float64) for a in (n, m, gamma, top))
        self.uniform = torch.tensor(gamma == 0.0, device="cuda")
        a = 1.0 / (np.where(gamma == 0.0, 2.5, gamma) - 1.0)
        b = 1.0 - np.where(np.abs(a - 1.0) < 1e-6, 1.0 + 1e-6, a)   # exponent of the cumulative weight
        lo, hi = np.full_like(n, 1e-6), np.full_like(n, 1e12)
        for _ in range(120):   # i0 so that the heaviest vertex expects `top` edges
            mid = np.sqrt(lo * hi)
            share = ((1 + mid) ** b - mid ** b) / ((n + mid) ** b - mid ** b)
            lo, hi = np.where(m * share > top, mid, lo), np.where(m * share > top, hi, mid)
        i0 = np.sqrt(lo * hi)
        dev = dict(device="cuda", dtype=torch.float64)
        self.i0, self.b = torch.tensor(i0, **dev), torch.tensor(b, **dev)
        self.c0, self.c1 = torch.tensor(i0 ** b, **dev), torch.tensor((n + i0) ** b - i0 ** b, **dev)
        self.n = torch.tensor(n, **dev)
        base = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
        self.total = int(base[-1])
        self.start = torch.tensor(base, device="cuda")
        if len(n) == 1:
            self.ids = torch.randperm(self.total, device="cuda", generator=gen)
        else:   # a permutation of each graph's ids: sort by (graph, random)
            g = torch.repeat_interleave(torch.arange(len(n), device="cuda"), torch.tensor(n, device="cuda").long())
            x = g.double() + torch.rand(self.total, device="cuda", dtype=torch.float64, generator=gen)
            self.ids = torch.argsort(x)

    def sample(self, g, k, gen, flat):
        """k endpoints; g: their graph (an index array, or 0 when there is one)."""
        x = torch.rand(k, device="cuda", dtype=torch.float64, generator=gen)
        if flat or (isinstance(g, int) and bool(self.uniform[0])):
            x.mul_(self.n[g])
        else:
            x.mul_(self.c1[g]).add_(self.c0[g]).pow_(1.0 / self.b[g]).sub_(self.i0[g])
        x = x.long()
        x.clamp_(min=0)
        x = torch.minimum(x, self.n[g].long() - 1)
        return self.ids[x.add_(self.start[g])]


def _graph(case, seed):
    """The union's edges as U-side CSR (int32 CUDA tensors) and layer starts."""
    sizes = _sizes(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r, l, m, gu, gl, tu, tl = (np.array(x) for x in zip(*sizes))
    U, L = _Layer(r, m, gu, tu * l, gen), _Layer(l, m, gl, tl * r, gen)
    total, one = int(m.sum()), len(sizes) == 1
    want = torch.tensor(m, device="cuda").long()
    keys = torch.zeros(0, dtype=torch.int64, device="cuda")
    for rnd in range(60):
        if one:
            k = int((total - keys.numel()) * (1.12 if rnd == 0 else 1.5)) + 1024
            g = 0
        else:
            have = torch.bincount(torch.searchsorted(U.start, keys // L.total, right=True) - 1,
                                  minlength=len(sizes)) if keys.numel() else torch.zeros_like(want)
            need = ((want - have).clamp(min=0).double() * 1.3).long() + 8
            g = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), need)
            k = g.numel()
        flat = rnd >= 6   # near-saturated skewed graphs are topped up uniformly
        new = U.sample(g, k, gen, flat).mul_(L.total).add_(L.sample(g, k, gen, flat))
        keys = torch.unique(torch.cat([keys, new]) if keys.numel() else new)
        del new, g
        if keys.numel() >= total:
            break
    # exactly `total` edges: the surplus is dropped at even distances
    n = keys.numel()
    if n > total:
        i = torch.arange(n, device="cuda")
        i.mul_(total)
        before = torch.div(i, n, rounding_mode="floor")
        keys = keys[torch.div(i.add_(total), n, rounding_mode="floor") > before]
        del i, before
    u = torch.div(keys, L.total, rounding_mode="floor")
    adj = keys.sub_(u * L.total).int()
    off = torch.searchsorted(u, torch.arange(U.total + 1, device="cuda")).int()
    if case.get("shuffled"):
        o = torch.randperm(adj.numel(), device="cuda", generator=gen)
        adj = adj[o][torch.argsort(u[o], stable=True)]
    return off, adj.contiguous(), U.total, L.total, U.start.int(), L.start.int()


class _State:
    def __init__(self, case, seed):
        self.kind, self.case = case["kind"], case
        self.off, self.adj, self.r, self.l, self.us, self.ls = _graph(case, seed)
        self.m = self.adj.numel()
        self.graph = self.plan = None
        dev = dict(device="cuda")
        if self.kind in ("vertices", "edges"):
            self.graph = ButterflyGraph(self.off, self.adj, self.r, self.l)
        elif self.kind == "plan":
            top = max(max(s[0], s[1]) for s in _sizes(case))
            self.plan = pkg.bfc.bfc_batch_plan_create(self.r, self.l, self.m, case["graphs"], top, None, _stream())
            self.totals = torch.zeros(case["graphs"], dtype=torch.int64, **dev)
            self.status = torch.zeros(1, dtype=torch.int32, **dev)
        elif self.kind == "noalloc":
            self.totals = torch.zeros(1, dtype=torch.int64, **dev)
            self.status = torch.zeros(1, dtype=torch.int32, **dev)
        elif self.kind == "host_all":
            self.off, self.adj = (t.cpu().pin_memory() for t in (self.off, self.adj))
            self.out = [torch.empty(max(k, 1), dtype=torch.int64, pin_memory=True) for k in (self.r, self.l, self.m)]
        elif self.kind == "estimate":
            self.sample_seed = seed * 2 + 1

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if self.graph is not None:
                self.graph.release()
            if self.plan is not None:
                pkg.bfc.bfc_batch_plan_destroy(self.plan)
        except Exception:
            pass


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    bfc = pkg.bfc
    if s.kind == "total":
        g = ButterflyGraph(s.off, s.adj, s.r, s.l)
        out = dict(total=g.count(), wedges=g.info()["wedges"])
        g.release()
    elif s.kind == "all":
        g = ButterflyGraph(s.off, s.adj, s.r, s.l)
        pu, pl, pe, total = g.count_all()
        out = dict(total=total, wedges=g.info()["wedges"], per_u=pu, per_l=pl, per_edge=pe)
        g.release()
    elif s.kind == "host_all":
        total, wedges = bfc.bfc_count_all_host(s.r, s.l, s.m, s.off.data_ptr(), s.adj.data_ptr(), None, _stream(),
                                               *(t.data_ptr() for t in s.out))
        out = dict(total=total, wedges=wedges, per_u=s.out[0], per_l=s.out[1], per_edge=s.out[2])
    elif s.kind == "vertices":
        pu, pl, total = s.graph.count_vertices()
        out = dict(total=total, per_u=pu, per_l=pl)
    elif s.kind == "edges":
        pe, total = s.graph.count_edges()
        out = dict(total=total, per_edge=pe)
    elif s.kind == "noalloc":
        bfc.bfc_count_small_noalloc(s.r, s.l, s.m, s.off.data_ptr(), s.adj.data_ptr(), _stream(),
                                    s.totals.data_ptr(), s.status.data_ptr())
        out = dict(total=s.totals, status=s.status)
    elif s.kind == "batch":
        totals = torch.empty(s.case["graphs"], dtype=torch.int64, device="cuda")
        h = bfc.bfc_prepare_batch(s.r, s.l, s.m, s.off.data_ptr(), s.adj.data_ptr(), s.case["graphs"],
                                  s.us.data_ptr(), s.ls.data_ptr(), None, _stream())
        bfc.bfc_count_batch(h, _stream(), totals.data_ptr())
        bfc.bfc_sync(h, _stream())
        bfc.bfc_release(h)
        out = dict(totals=totals)
    elif s.kind == "plan":
        bfc.bfc_batch_plan_run(s.plan, s.off.data_ptr(), s.adj.data_ptr(), s.us.data_ptr(), s.ls.data_ptr(),
                               _stream(), s.totals.data_ptr(), s.status.data_ptr())
        out = dict(totals=s.totals, status=s.status)
    else:
        e = estimate_butterflies(s.off, s.adj, s.r, s.l, s.case["p"], s.case["samples"], seed=s.sample_seed)
        out = dict(counts=e["counts"], estimate=e["estimate"], std_error=e["std_error"])
    return out


# ---- the same outputs in plain torch --------------------------------------------

_MOST_WEDGES = 700_000_000   # above this, the expansion below would take too long


def _by_hand(u, v, r, l, graph_of_u=None, graphs=1, parts=True):
    """Counts by expanding every wedge whose first end has the highest priority
    (degree, then id with U above L): None where there are too many."""
    m = u.numel()
    a, b = torch.cat([v, l + u]), torch.cat([l + u, v])   # every edge from both sides, L ids first
    deg = torch.bincount(a, minlength=r + l)
    order = torch.argsort(deg, stable=True)
    pri = torch.empty_like(order)
    pri[order] = torch.arange(r + l, device="cuda")
    e = torch.argsort(a * (r + l) + pri[b])               # lists of a in ascending priority of b
    a, b, edge = a[e], b[e], torch.arange(m, device="cuda").repeat(2)[e]
    first = torch.cumsum(deg, 0) - deg
    pos = torch.arange(2 * m, device="cuda") - first[a]
    starts = torch.nonzero((pri[b] > pri[a]) & (pos > 0)).flatten()   # slots (middle a, start b)
    n = pos[starts]
    wedges = int(n.sum())
    if wedges > _MOST_WEDGES:
        return None
    slot = torch.repeat_interleave(starts, n)
    end = torch.arange(wedges, device="cuda") - torch.repeat_interleave(torch.cumsum(n, 0) - n, n) + first[a[slot]]
    key = b[slot] * (r + l) + b[end]
    if parts:
        pair, inv, c = torch.unique(key, return_inverse=True, return_counts=True)
    else:
        pair, c = torch.unique(key, return_counts=True)
    x, w = pair // (r + l), pair % (r + l)
    c2 = c * (c - 1) // 2
    out = dict(total=int(c2.sum()), wedges=wedges)
    if graph_of_u is not None:   # any vertex names its graph; starts and ends share it
        out["totals"] = torch.zeros(graphs, dtype=torch.int64, device="cuda").index_add_(0, graph_of_u[x], c2)
    if parts:
        per = torch.zeros(r + l, dtype=torch.int64, device="cuda").index_add_(0, x, c2).index_add_(0, w, c2)
        d = c[inv] - 1
        per.index_add_(0, a[slot], d)
        pe = torch.zeros(m, dtype=torch.int64, device="cuda").index_add_(0, edge[slot], d).index_add_(0, edge[end], d)
        out.update(per_u=per[l:], per_l=per[:l], per_edge=pe)
    return out


def _draws(seed, k):
    """Outputs number k of SplitMix64 from `seed` (int64 bit patterns)."""
    def c(x):
        x &= (1 << 64) - 1
        return x - (1 << 64) if x >> 63 else x

    def shr(z, n):
        return (z >> n) & ((1 << (64 - n)) - 1)

    z = k * c(0x9E3779B97F4A7C15) + c(seed)
    z = (z ^ shr(z, 30)) * c(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * c(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def exact(case, seed):
    kind = case["kind"]
    off, adj, r, l, us, ls = _graph(case, seed)
    m, v = adj.numel(), adj.long()
    u = torch.repeat_interleave(torch.arange(r, device="cuda"), off.long().diff())
    if kind == "estimate":
        counts, p = [], case["p"]
        top = int(p * 2.0 ** 64) - (1 << 63)     # unsigned order, moved to signed
        e = torch.arange(m, device="cuda")
        for j in range(case["samples"]):
            keep = (_draws(seed * 2 + 1, e + (j * m + 1)) ^ (-(1 << 63))) < top
            got = _by_hand(u[keep], v[keep], r, l, parts=False)
            if got is None:
                return None
            counts.append(got["total"])
        n, mean = len(counts), sum(counts) / len(counts)
        err = math.sqrt(sum((c - mean) ** 2 for c in counts) / (n - 1) / n) / p ** 4
        return dict(counts=torch.tensor(counts), estimate=sum(counts) / (n * p ** 4), std_error=err)
    if kind in ("batch", "plan"):
        ids = torch.arange(r + l, device="cuda")
        g = torch.where(ids < l, torch.searchsorted(ls, ids.int(), right=True) - 1,
                        torch.searchsorted(us, (ids - l).clamp(min=0).int(), right=True) - 1)
        got = _by_hand(u, v, r, l, g, case["graphs"], parts=False)
        if got is None:
            return None
        return dict(totals=got["totals"], status=torch.zeros(1, dtype=torch.int32)) if kind == "plan" \
            else dict(totals=got["totals"])
    got = _by_hand(u, v, r, l, parts=kind in ("all", "host_all", "vertices", "edges"))
    if got is None:
        return None
    if kind == "noalloc":
        return dict(total=torch.tensor([got["total"]]), status=torch.zeros(1, dtype=torch.int32))
    keys = {"total": ("total", "wedges"), "vertices": ("total", "per_u", "per_l"), "edges": ("total", "per_edge")}
    return {k: got[k] for k in keys.get(kind, ("total", "wedges", "per_u", "per_l", "per_edge"))}
