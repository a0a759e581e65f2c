"""The workloads of the matching library that its speed is measured on.

Every case goes through the public binding as a program would call it: a
context, device graphs and result buffers are prepared once, and one pass is
one call (or one chain of calls) of the form the case names:

* ``match``    lm_match of one resident graph into a device buffer
* ``noalloc``  lm_match_small_noalloc of a device edge list
* ``batch``    lm_batch_match of many resident graphs
* ``served``   lm_submit of a burst of requests, then lm_wait / lm_poll of each
* ``host``     lm_graph_create from pinned host arrays, lm_match into a host
               buffer, lm_graph_destroy: one graph that is matched once
* ``contract`` lm_contract of a matching, through the C entry point into the
               caller's own arrays
* ``coarsen``  levels of lm_graph_create (device arrays), lm_match,
               lm_contract and lm_graph_destroy: multilevel coarsening

Graphs are drawn on the GPU from the seed: random graphs with m distinct pairs
(``er``), 2D grids with 5% long-range edges (``grid``) and R-MAT with
(.57, .19, .19, .05), random relabelling, loops and duplicates dropped
(``rmat``); weights are uniform multiples of 2^-24 in [0, 1) or all one
(``unit``, where the seeded permutation decides every comparison).
"""
import ctypes
import math
import random

import numpy as np
import torch

import paper_1302_4587_gb300 as lm

M32 = 0xFFFFFFFF


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one small edge list matched under a fixed device footprint
        {"name": "noalloc_er_10k", "form": "noalloc", "family": "er", "n": 10_000, "m": 50_000, "unit": False},
        # the smallest resident graph: latency of one call
        {"name": "match_er_10k", "form": "match", "family": "er", "n": 10_000, "m": 50_000, "unit": False,
         "renew": False},
        # a mesh whose weights all tie
        {"name": "match_grid_1024_unit", "form": "match", "family": "grid", "rows": 1024, "cols": 1024, "unit": True,
         "renew": False},
        # a random graph of average degree 32, odd sizes
        {"name": "match_er_100003_a16", "form": "match", "family": "er", "n": 100_003, "m": 1_600_047, "unit": False,
         "renew": False},
        # the flagship: a large skewed graph, far beyond L2
        {"name": "match_rmat23", "form": "match", "family": "rmat", "scale": 23, "ef": 16, "unit": False,
         "renew": False},
        # ties broken anew every round
        {"name": "match_rmat20_unit_renew", "form": "match", "family": "rmat", "scale": 20, "ef": 16, "unit": True,
         "renew": True},
        # thousands of uneven graphs in one call
        {"name": "batch_4096", "form": "batch", "count": 4096, "n_lo": 64, "n_hi": 65536, "shape": 4},
        # a few dozen graphs in one call
        {"name": "batch_48", "form": "batch", "count": 48, "n_lo": 64, "n_hi": 65536, "shape": 7},
        # a burst of requests to the serving loop
        {"name": "served_48", "form": "served", "count": 48, "m_lo": 1_000, "m_hi": 4_000_000, "shape": 5},
        # a graph that arrives in host memory and is matched once
        {"name": "host_rmat21", "form": "host", "family": "rmat", "scale": 21, "ef": 16, "unit": False},
        # one contraction of a matching, the step of multilevel partitioning
        {"name": "contract_rmat22", "form": "contract", "family": "rmat", "scale": 22, "ef": 16, "unit": False},
        # the multilevel chain itself, on the device throughout
        {"name": "coarsen_rmat20_x5", "form": "coarsen", "family": "rmat", "scale": 20, "ef": 16, "unit": False,
         "levels": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, m_lo, m_hi, scale_hi):
    """A graph of one family with about m_lo to m_hi edges."""
    m = _log_int(rng, m_lo, m_hi)
    family = rng.choice(["er", "er", "grid", "rmat"])
    unit = rng.random() < 0.3
    if family == "grid":
        side = max(8, math.sqrt(m / 2.1))
        rows = max(3, int(side * rng.uniform(0.4, 1.0)))
        return {"family": "grid", "rows": rows, "cols": max(3, int(side * side / rows)), "unit": unit}
    if family == "rmat" and m > 4 * 2**10:
        ef = rng.choice([4, 8, 16])
        scale = min(scale_hi, max(8, int(math.log2(m / ef))))
        return {"family": "rmat", "scale": scale, "ef": ef, "unit": unit}
    alpha = rng.choice([2, 4, 16, 64]) * rng.uniform(0.8, 1.2)
    n = max(64, int(m / alpha))
    return {"family": "er", "n": n, "m": min(m, n * (n - 1) // 8), "unit": unit}


def draw(rng):
    form = rng.choice(["noalloc", "match", "match", "match", "match", "batch", "served", "host", "contract", "coarsen"])
    if form == "noalloc":
        n = _log_int(rng, 500, 60_000)
        m = min(_log_int(rng, 2_000, 250_000), n * (n - 1) // 8)
        return {"form": form, "family": "er", "n": n, "m": m, "unit": rng.random() < 0.3}
    if form == "match":
        return dict({"form": form, "renew": rng.random() < 0.15}, **_draw_graph(rng, 20_000, 60_000_000, 22))
    if form == "batch":
        return {"form": form, "count": _log_int(rng, 4, 2500), "n_lo": 64, "n_hi": _log_int(rng, 2_000, 65_536),
                "shape": rng.randrange(1 << 20)}
    if form == "served":
        return {"form": form, "count": rng.randrange(8, 49), "m_lo": 1_000, "m_hi": _log_int(rng, 100_000, 4_000_000),
                "shape": rng.randrange(1 << 20)}
    if form == "host":
        return dict({"form": form}, **_draw_graph(rng, 100_000, 30_000_000, 20))
    if form == "contract":
        return dict({"form": form}, **_draw_graph(rng, 100_000, 40_000_000, 21))
    return dict({"form": form, "levels": rng.randrange(2, 6)}, **_draw_graph(rng, 50_000, 8_000_000, 19))


# ------------------------------------------------------------------ the graphs
def _generator(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1_000_003 + tag) & 0x7FFFFFFFFFFF)
    return g


def _weights(m, unit, gen):
    if unit:
        return torch.ones(m, dtype=torch.float32, device="cuda")
    return torch.randint(0, 1 << 24, (m,), generator=gen, device="cuda", dtype=torch.int32).float() * 2.0**-24


def _rmat_pairs(count, levels, gen):
    """(u, v) of `count` R-MAT draws with 2^levels vertices; `levels` a number or a tensor of one per draw."""
    u = torch.zeros(count, dtype=torch.int32, device="cuda")
    v = torch.zeros(count, dtype=torch.int32, device="cuda")
    top = levels if isinstance(levels, int) else int(levels.max()) if count else 0
    for k in range(top):
        r = torch.rand(count, generator=gen, device="cuda")
        bu = (r >= 0.76).to(torch.int32)
        bv = (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).to(torch.int32)
        if not isinstance(levels, int):
            on = (levels > k).to(torch.int32)
            bu, bv = bu * on, bv * on
        u |= bu << k
        v |= bv << k
    return u, v


def _graph(case, seed):
    """(n, eu, ev, w) of a single-graph case, on the device."""
    gen = _generator(seed, 1)
    if case["family"] == "er":
        n, m = case["n"], case["m"]
        a = torch.randint(0, n, (m + m // 4 + 64,), generator=gen, device="cuda")
        b = torch.randint(0, n, (m + m // 4 + 64,), generator=gen, device="cuda")
        key = torch.unique((torch.minimum(a, b) * n + torch.maximum(a, b))[a != b])
        key = key[torch.randperm(key.numel(), generator=gen, device="cuda")[:m]]
        swap = torch.rand(key.numel(), generator=gen, device="cuda") < 0.5
        lo, hi = key // n, key % n
        eu, ev = torch.where(swap, hi, lo), torch.where(swap, lo, hi)
    elif case["family"] == "grid":
        rows, cols = case["rows"], case["cols"]
        n = rows * cols
        i = torch.arange(n, device="cuda")
        right, down = i[i % cols != cols - 1], i[i < n - cols]
        edges = right.numel() + down.numel()
        a = torch.randint(0, n, (edges // 20,), generator=gen, device="cuda")
        b = torch.randint(0, n, (edges // 20,), generator=gen, device="cuda")
        far = torch.unique((torch.minimum(a, b) * n + torch.maximum(a, b))[(a - b).abs() > 1])
        eu = torch.cat([right, down, far // n])
        ev = torch.cat([right + 1, down + cols, far % n])
    else:
        scale = case["scale"]
        n = 1 << scale
        u, v = _rmat_pairs(case["ef"] << scale, scale, gen)
        relabel = torch.randperm(n, generator=gen, device="cuda")
        u, v = relabel[u.long()], relabel[v.long()]
        key = torch.unique(((torch.minimum(u, v) << scale) | torch.maximum(u, v))[u != v])
        eu, ev = key >> scale, key & (n - 1)
    eu, ev = eu.to(torch.int32), ev.to(torch.int32)
    return n, eu, ev, _weights(eu.numel(), case["unit"], gen)


def _shapes(case):
    """(kind, n, m) of the graphs of a batch or of a burst of requests: their sizes are the case's, their
    edges and weights the seed's."""
    rng = random.Random(case["shape"])
    out = []
    for _ in range(case["count"]):
        if case["form"] == "batch":
            n = max(2, _log_int(rng, case["n_lo"], case["n_hi"]))
            m = int(n * rng.uniform(4.0, 16.0) / 2)
        else:
            m = _log_int(rng, case["m_lo"], case["m_hi"])
            n = max(64, int(m / rng.uniform(2.0, 8.0)))
        out.append((rng.randrange(3), n, min(m, n * (n - 1) // 4)))
    return out


def _many(case, seed):
    """The graphs of _shapes(case) as a list of (n, eu, ev, w), drawn together."""
    gen = _generator(seed, 2)
    shapes = _shapes(case)
    kind, n, m = (torch.tensor(x, dtype=torch.int64, device="cuda") for x in zip(*shapes))
    count = len(shapes)
    ids = torch.arange(count, device="cuda")
    base = torch.cumsum(n, 0) - n
    # mesh edges of the grid graphs: side x side meshes cut to n vertices, at most m edges kept
    vg = torch.repeat_interleave(ids, n * (kind == 1))
    vi = torch.arange(vg.numel(), device="cuda") - torch.repeat_interleave(
        torch.cumsum(n * (kind == 1), 0) - n * (kind == 1), n * (kind == 1))
    side = torch.ceil(torch.sqrt(n.double())).long()[vg]
    right = (vi % side != side - 1) & (vi + 1 < n[vg])
    down = vi + side < n[vg]
    mg = torch.cat([vg[right], vg[down]])
    mu = torch.cat([vi[right], vi[down]])
    mv = torch.cat([vi[right] + 1, vi[down] + side[down]])
    have = torch.bincount(mg, minlength=count)
    # random pairs: all edges of the random and R-MAT graphs, the long-range ones of the grids
    want = torch.where(kind == 1, torch.clamp(m - have, min=0), m + m // 16)
    pg = torch.repeat_interleave(ids, want)
    pn = n[pg]
    pu = torch.minimum((torch.rand(pg.numel(), generator=gen, device="cuda", dtype=torch.float64) * pn).long(), pn - 1)
    pv = torch.minimum((torch.rand(pg.numel(), generator=gen, device="cuda", dtype=torch.float64) * pn).long(), pn - 1)
    skew = (kind == 2)[pg]
    levels = torch.ceil(torch.log2(n.double())).to(torch.int32)[pg[skew]]
    ru, rv = _rmat_pairs(int(skew.sum()), levels, gen)
    # relabelled by a multiplier prime to every n
    pu[skew] = (ru.long() % pn[skew]) * 1_000_003 % pn[skew]
    pv[skew] = (rv.long() % pn[skew]) * 1_000_003 % pn[skew]
    g, u, v = torch.cat([mg, pg]), torch.cat([mu, pu]), torch.cat([mv, pv])
    ok = u != v
    g, u, v = g[ok], u[ok], v[ok]
    nb = max(1, int(n.max()) - 1).bit_length()
    key = torch.unique((g << (2 * nb)) | (torch.minimum(u, v) << nb) | torch.maximum(u, v))
    g = key >> (2 * nb)
    eu = ((key >> nb) & ((1 << nb) - 1)).to(torch.int32)
    ev = (key & ((1 << nb) - 1)).to(torch.int32)
    w = _weights(eu.numel(), False, gen)
    cut = np.concatenate([[0], np.cumsum(torch.bincount(g, minlength=count).cpu().numpy())])
    return [(shapes[i][1], eu[cut[i]:cut[i + 1]], ev[cut[i]:cut[i + 1]], w[cut[i]:cut[i + 1]]) for i in range(count)]


# ------------------------------------------------------------------ one pass
class State:
    """What a program keeps between calls; the library's handles are given back with it."""

    def __init__(self, case, seed):
        self.case = case
        self.seed = 1000 + seed
        self.ctx = None
        self.graphs = []

    def graph(self, n, eu, ev, w):
        g = lm.lm_graph_create(self.ctx, n, eu, ev, w)
        self.graphs.append(g)
        return g

    def __del__(self):
        for g in self.graphs:
            lm.lm_graph_destroy(g)
        if self.ctx is not None:
            lm.lm_destroy(self.ctx)


def _mate(n):
    return torch.empty(n, dtype=torch.int32, device="cuda")


def _capacity(case):
    """(vertices, edges) that fit every seed's graph of a single-graph case."""
    if case["family"] == "er":
        return case["n"], case["m"]
    if case["family"] == "grid":
        return case["rows"] * case["cols"], (2 * case["rows"] * case["cols"]) * 21 // 20
    return 1 << case["scale"], case["ef"] << case["scale"]


def _coarse(case):
    """The caller's arrays of one contraction: cmap, cvw, ceu, cev, cw (zero where nothing is written)."""
    n, m = _capacity(case)
    return [torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"),
            torch.zeros(m, dtype=torch.int32, device="cuda"), torch.zeros(m, dtype=torch.int32, device="cuda"),
            torch.zeros(m, dtype=torch.float32, device="cuda")]


def _contract(ctx, n, m, eu, ev, w, vw, mate, out):
    """lm_contract of include/lm.h into the arrays `out`; returns the coarse vertex and edge counts."""
    nc, mc = ctypes.c_uint32(), ctypes.c_uint32()
    at = lambda t: ctypes.c_void_p(t.data_ptr()) if t is not None else None
    rc = lm.load().lm_contract(ctx, n, m, at(eu), at(ev), at(w), at(vw), at(mate), *[at(t) for t in out],
                               ctypes.byref(nc), ctypes.byref(mc))
    if rc != lm.LM_OK:
        raise lm.LmError(rc, lm.lm_strerror(rc))
    return int(nc.value), int(mc.value)


def prepare(case, seed):
    s = State(case, seed)
    form = case["form"]
    if form == "noalloc":
        s.n, s.eu, s.ev, s.w = _graph(case, seed)
        s.mate, s.status = _mate(s.n), torch.empty(1, dtype=torch.int32, device="cuda")
        return s
    if form == "served":
        s.ctx = lm.lm_create(torch.cuda.current_device(), hbm_budget_bytes=8 << 30)
    else:
        s.ctx = lm.lm_create(torch.cuda.current_device(), flags=lm.LM_F_RENEW if case.get("renew") else 0)
    if form in ("batch", "served"):
        many = _many(case, seed)
        handles = [s.graph(*g) for g in many]
        s.all = _mate(sum(g[0] for g in many))
        s.mates = list(torch.split(s.all, [g[0] for g in many]))
        s.seeds = [s.seed + i for i in range(len(many))]
        if form == "batch":
            s.args = lm.BatchArgs(handles, s.seeds, s.mates)
        return s
    s.n, s.eu, s.ev, s.w = _graph(case, seed)
    if form == "match":
        s.graph(s.n, s.eu, s.ev, s.w)
        s.mate = _mate(s.n)
        del s.eu, s.ev, s.w
    elif form == "host":
        s.eu, s.ev, s.w = (x.cpu().pin_memory() for x in (s.eu, s.ev, s.w))
        s.mate = torch.empty(s.n, dtype=torch.int32, pin_memory=True)
    elif form == "contract":
        g = s.graph(s.n, s.eu, s.ev, s.w)
        s.mate = lm.lm_match(s.ctx, g, s.seed, _mate(s.n))
        s.out = _coarse(case)
    else:
        s.mates = [torch.full((s.n,), -1, dtype=torch.int32, device="cuda") for _ in range(case["levels"])]
        s.out = [_coarse(case) for _ in range(case["levels"])]
    return s


def run(s):
    form = s.case["form"]
    if form == "match":
        return lm.lm_match(s.ctx, s.graphs[0], s.seed, s.mate)
    if form == "noalloc":
        lm.lm_match_small_noalloc(s.n, s.eu, s.ev, s.w, s.seed, s.mate, s.status,
                                  torch.cuda.current_stream().cuda_stream)
        return [s.mate, s.status]
    if form == "batch":
        lm.lm_batch_match(s.ctx, s.args)
        return s.all
    if form == "served":
        tickets = [lm.lm_submit(s.ctx, g, seed, mate) for g, seed, mate in zip(s.graphs, s.seeds, s.mates)]
        for t in tickets:
            lm.lm_wait(s.ctx, t, 60_000)
            lm.lm_poll(s.ctx, t)
        return s.all
    if form == "host":
        g = lm.lm_graph_create(s.ctx, s.n, s.eu, s.ev, s.w)
        lm.lm_match(s.ctx, g, s.seed, s.mate)
        lm.lm_graph_destroy(g)
        return s.mate
    if form == "contract":
        return s.out + list(_contract(s.ctx, s.n, s.eu.numel(), s.eu, s.ev, s.w, None, s.mate, s.out))
    n, m, eu, ev, w, vw = s.n, s.eu.numel(), s.eu, s.ev, s.w, None
    counts = []
    for level in range(s.case["levels"]):
        g = lm.lm_graph_create(s.ctx, n, eu[:m], ev[:m], w[:m])
        lm.lm_match(s.ctx, g, s.seed + level, s.mates[level])
        lm.lm_graph_destroy(g)
        out = s.out[level]
        n, m = _contract(s.ctx, n, m, eu, ev, w, vw, s.mates[level], out)
        vw, eu, ev, w = out[1:]
        counts += [n, m]
        if m == 0:
            break
    return s.mates + [t for out in s.out for t in out] + counts


# ------------------------------------------------------------------ what a pass cannot do without
def _size(case):
    """(n, m) of a single-graph case (R-MAT: about m, after duplicates are dropped)."""
    if case["family"] == "er":
        return case["n"], case["m"]
    if case["family"] == "grid":
        r, c = case["rows"], case["cols"]
        return r * c, (2 * r * c - r - c) * 21 // 20
    return 1 << case["scale"], int(0.95 * (case["ef"] << case["scale"]))


def work(case):
    """Each edge (two ends and a weight, 12 bytes) read once, each vertex's result written once, and the two
    comparisons an edge takes part in."""
    if case["form"] in ("batch", "served"):
        shapes = _shapes(case)
        n, m = sum(x[1] for x in shapes), sum(x[2] for x in shapes)
    else:
        n, m = _size(case)
    moved = 12 * m + 4 * n
    if case["form"] == "contract":
        moved += 12 * m + 8 * n          # the coarse edges; the matching in, the coarse map and weights out
    elif case["form"] == "coarsen":
        # every level reads its edges and writes the next ones (about 0.8 of them)
        moved = sum((24 * m + 12 * n) * 0.8**k for k in range(case["levels"]))
    return {"bytes": int(moved), "flops": int(2 * m)}


# ------------------------------------------------------------------ the definition, in plain torch
def _fmix32(h):
    h = h ^ (h >> 16)
    h = (h * 0x85EBCA6B) & M32
    h = h ^ (h >> 13)
    h = (h * 0xC2B2AE35) & M32
    return h ^ (h >> 16)


def _keys(w, seed, rnd):
    """The order of the edges in round `rnd` as int64: ord(w) above the seeded permutation of the edge index."""
    z = (seed + (rnd + 1) * 0x9E3779B97F4A7C15) & (2**64 - 1)
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & (2**64 - 1)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & (2**64 - 1)
    z ^= z >> 31
    e = torch.arange(w.numel(), device=w.device)
    p = _fmix32(_fmix32(e ^ (z & M32)) ^ (z >> 32))
    return (w.view(torch.int32).long() << 32) | p      # weights here are not negative: their bits are ordered


def _local_max(n, eu, ev, w, seed, renew=False):
    eu, ev = eu.long(), ev.long()
    mate = torch.full((n,), -1, dtype=torch.int32, device=w.device)
    live = torch.arange(w.numel(), device=w.device)
    key = _keys(w, seed, 0)
    rnd = 0
    while live.numel():
        u, v, k = eu[live], ev[live], key[live]
        best = torch.full((n,), -1, dtype=torch.int64, device=w.device)
        best.scatter_reduce_(0, u, k, "amax")
        best.scatter_reduce_(0, v, k, "amax")
        hit = (best[u] == k) & (best[v] == k)
        mate[u[hit]] = v[hit].to(torch.int32)
        mate[v[hit]] = u[hit].to(torch.int32)
        live = live[(mate[u] < 0) & (mate[v] < 0)]
        rnd += 1
        if renew:
            key = _keys(w, seed, rnd)
    return mate


def _contraction(n, eu, ev, w, mate, vw):
    me = torch.arange(n, device=w.device)
    other = torch.where(mate < 0, me, mate.long())
    rep = me <= other
    rank = torch.cumsum(rep.long(), 0) - 1
    cmap = rank[torch.minimum(me, other)]
    nc = int(rep.sum())
    cvw = torch.zeros(nc, dtype=torch.int64, device=w.device)
    cvw.index_add_(0, cmap, torch.ones(n, dtype=torch.int64, device=w.device) if vw is None else vw.long())
    a, b = cmap[eu.long()], cmap[ev.long()]
    e = torch.nonzero(a != b).flatten()
    pair = torch.minimum(a[e], b[e]) * max(nc, 1) + torch.maximum(a[e], b[e])
    groups, inv = torch.unique(pair, return_inverse=True)
    lead = torch.full((groups.numel(),), w.numel(), dtype=torch.int64, device=w.device)
    lead.scatter_reduce_(0, inv, e, "amin")
    total = torch.zeros(groups.numel(), dtype=torch.float64, device=w.device)
    total.index_add_(0, inv, w[e].double())
    order = torch.argsort(lead)
    lead = lead[order]
    return (cmap.to(torch.int32), cvw.to(torch.int32), a[lead].to(torch.int32), b[lead].to(torch.int32), total[order])


def _pad(t, count, fill=0):
    return torch.cat([t, torch.full((count - t.numel(),), fill, dtype=t.dtype, device=t.device)])


def _padded(coarse, case):
    n, m = _capacity(case)
    return [_pad(t, c) for t, c in zip(coarse, (n, n, m, m, m))]


def exact(case, seed):
    form, match_seed = case["form"], 1000 + seed
    if form in ("batch", "served"):
        # graph by graph, each with its own edge indices and seed: only where they are few
        if case["count"] > 64:
            return None
        return torch.cat([_local_max(n, eu, ev, w, match_seed + i)
                          for i, (n, eu, ev, w) in enumerate(_many(case, seed))])
    n, eu, ev, w = _graph(case, seed)
    if form == "coarsen":
        mates, out, counts, vw = [], [], [], None
        size = _capacity(case)[0]
        for level in range(case["levels"]):
            mates.append(_local_max(n, eu, ev, w, match_seed + level))
            cmap, vw, eu, ev, total = _contraction(n, eu, ev, w, mates[-1], vw)
            out += _padded((cmap, vw, eu, ev, total), case)
            w = total.float()           # the next level's weights are rounded once, by definition
            n = int(vw.numel())
            counts += [n, eu.numel()]
            if not eu.numel():
                break
        for _ in range(case["levels"] - len(mates)):
            mates.append(mates[-1][:0])
            out += _padded((cmap[:0], cmap[:0], cmap[:0], cmap[:0], total[:0]), case)
        return [_pad(t, size, -1) for t in mates] + out + counts
    mate = _local_max(n, eu, ev, w, match_seed, bool(case.get("renew")))
    if form == "contract":
        coarse = _contraction(n, eu, ev, w, mate, None)
        return _padded(coarse, case) + [coarse[1].numel(), coarse[2].numel()]
    if form == "noalloc":
        return [mate, torch.zeros(1, dtype=torch.int32, device=w.device)]
    return mate.cpu() if form == "host" else mate
