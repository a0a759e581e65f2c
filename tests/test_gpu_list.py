"""The list path of the matching (lm_match / lm_batch_match without a renewed
order): rows around every size at which a row changes hands (a thread, eight
lanes, a warp, a warp's loop, a block, chunks), weights that are distinct, few
or all equal (the lists then order by the permutation), and every way of asking:
without statistics, with them (exact rounds and per-round counts), batched,
queued.  Results are whole numbers: they equal the oracle's."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_util import Lm, to_u32

pytestmark = pytest.mark.gpu

# a row's sizes: 1 .. 5 (four are kept), then both sides of 16, 32, 64, 256, 1024, 2048 and two chunks
DEGREES = [1, 2, 3, 4, 5, 8, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025,
           2047, 2048, 2049, 4095, 4096, 4097, 6151]


def _weights(m, kind, seed):
    w = synth.weights(m, seed, unit=kind == "unit")
    if kind == "few":
        w = (np.floor(w * 8.0) / 8.0).astype(np.float32)
    elif kind == "ulp":     # neighbouring floats: equal in all but the lowest bits
        w = (np.float32(1.0).view(np.int32) + (w * 64).astype(np.int32)).view(np.float32)
    elif kind == "signed":
        w = (w * 2.0 - 1.0).astype(np.float32)
        w[:: 7] = np.float32("inf")
        w[3:: 11] = np.float32("-inf")
    return w


def _hubs(kind, seed, shuffle):
    """A hub of every size in DEGREES over shared leaves (so that hubs lose their heaviest neighbours to
    one another and scan their rows again), hubs joined in a path."""
    k = len(DEGREES)
    leaves = 6200
    rng = np.random.default_rng(seed)
    eu, ev = [], []
    for h, d in enumerate(DEGREES):
        eu.append(np.full(d, h, np.uint32))
        ev.append((k + rng.permutation(leaves)[:d]).astype(np.uint32))
    eu.append(np.arange(k - 1, dtype=np.uint32))
    ev.append(np.arange(1, k, dtype=np.uint32))
    eu, ev = np.concatenate(eu), np.concatenate(ev)
    if shuffle:
        p = rng.permutation(eu.size)
        eu, ev = eu[p], ev[p]
    return synth.Graph(k + leaves, eu, ev, _weights(eu.size, kind, seed), f"hubs_{kind}_{seed}")


def _few_leaves(kind, seed):
    """Hubs that share few leaves by parallel edges: most of a row dies before its hub is matched."""
    rng = np.random.default_rng(seed)
    eu, ev = [], []
    for h, d in enumerate([40, 70, 300, 1100, 2100, 5000] * 3):
        eu.append(np.full(d, h, np.uint32))
        ev.append((18 + rng.integers(0, 24, d)).astype(np.uint32))
    eu, ev = np.concatenate(eu), np.concatenate(ev)
    return synth.Graph(18 + 24, eu, ev, _weights(eu.size, kind, seed), f"few_{kind}_{seed}")


def _check(L, g, seed):
    lm, torch = L.lm, L.torch
    want = oracle.greedy(g.n, g.eu, g.ev, g.w, seed)
    _, r, rm, rn = oracle.seq_local_max(g.n, g.eu, g.ev, g.w, seed)
    h = L.graph(g)
    try:
        mate = torch.full((g.n,), -7, dtype=torch.int32, device="cuda")
        lm.lm_match(L.ctx, h, seed, mate)
        assert np.array_equal(to_u32(mate), want), g.name
        got, st = L.match(g, seed, handle=h)
        assert np.array_equal(got, want), g.name
        k = min(r, 64)
        assert st["rounds"] == r and st["matched"] == int((want != 0xFFFFFFFF).sum()) // 2
        assert st["round_m"][:k] == [int(x) for x in rm[:k]]
        assert st["round_n"][:k] == [int(x) for x in rn[:k]]
    finally:
        lm.lm_graph_destroy(h)


@pytest.fixture(scope="module")
def L():
    x = Lm()
    yield x
    x.close()


@pytest.mark.parametrize("kind", ["uniform", "unit", "few", "ulp", "signed"])
@pytest.mark.parametrize("shape", ["hubs", "hubs_shuffled", "few_leaves"])
def test_rows_of_every_size(L, shape, kind):
    for seed in (1, 2):
        g = _few_leaves(kind, seed) if shape == "few_leaves" else _hubs(kind, seed, shape == "hubs_shuffled")
        _check(L, g, 10 + seed)


@pytest.mark.parametrize("n,m,unit", [(255, 900, False), (257, 900, True), (511, 4000, False), (70_001, 300_007, False),
                                      (70_001, 300_007, True), (300_001, 2_400_011, False)])
def test_parts_of_several_blocks(L, n, m, unit):
    _check(L, synth.er(n, m, seed=n, unit=unit), 5)


def test_a_long_chain_of_dependent_rows(L):
    """A path with monotone weights through many blocks' rows: each match waits for the previous one."""
    n = 30_001
    eu = np.arange(n - 1, dtype=np.uint32)
    g = synth.Graph(n, eu, eu + 1, (np.arange(n - 1) + 1).astype(np.float32), "chain")
    mate = L.torch.full((n,), -7, dtype=L.torch.int32, device="cuda")
    h = L.graph(g)
    try:
        L.lm.lm_match(L.ctx, h, 1, mate)
        assert np.array_equal(to_u32(mate), oracle.greedy(n, g.eu, g.ev, g.w, 1))
        _, st = L.match(g, 1, handle=h)
        assert st["rounds"] == (n - 1 + 1) // 2
    finally:
        L.lm.lm_graph_destroy(h)


def test_batches_queued_matches_and_host_results(L):
    lm, torch = L.lm, L.torch
    gs = [_hubs("uniform", 3, True), synth.er(10_000, 50_000, 4), _few_leaves("unit", 5),
          synth.Graph(5, np.zeros(0, np.uint32), np.zeros(0, np.uint32), np.zeros(0, np.float32), "edgeless"),
          synth.grid(90, 70, 0.05, seed=6, unit=True), synth.rmat(scale=13, edge_factor=16, seed=7)]
    want = [oracle.greedy(g.n, g.eu, g.ev, g.w, 20 + i) for i, g in enumerate(gs)]
    hs = [L.graph(g) for g in gs]
    actx = lm.lm_create(0, None, flags=lm.LM_F_ASYNC)
    try:
        mates = [np.empty(g.n, np.uint32) if i % 2 else torch.empty(g.n, dtype=torch.int32, device="cuda")
                 for i, g in enumerate(gs)]
        for stats in (False, True):
            out = lm.lm_batch_match(L.ctx, hs, [20 + i for i in range(len(gs))], mates, stats=stats)
            for g, a, b in zip(gs, out[0] if stats else out, want):
                assert np.array_equal(to_u32(a), b), g.name
            if stats:
                for g, st, i in zip(gs, out[1], range(len(gs))):
                    assert st["rounds"] == oracle.seq_local_max(g.n, g.eu, g.ev, g.w, 20 + i)[1], g.name
        qs = [torch.full((max(g.n, 1),), -7, dtype=torch.int32, device="cuda")[: g.n] for g in gs]
        for _ in range(3):
            for i, (h, q) in enumerate(zip(hs, qs)):
                lm.lm_match(actx, h, 20 + i, q)
        lm.lm_sync(actx)
        for g, q, b in zip(gs, qs, want):
            assert np.array_equal(to_u32(q), b), g.name
    finally:
        lm.lm_destroy(actx)
        for h in hs:
            lm.lm_graph_destroy(h)


@pytest.mark.parametrize("n", [4095, 4096, 4097, 100_000, 5_000_001])
def test_few_edges_among_many_vertices(n):
    # the vertices without edges have blocks of their own that clear their results; alone, in a
    # batch between others, and with rounds wanted
    import paper_1302_4587_gb300 as lm
    L = Lm()
    torch = L.torch
    try:
        rng = np.random.default_rng(n)
        eu = rng.permutation(n)[:120].astype(np.uint32)
        ev = np.concatenate([eu[1:], eu[:1]])
        g = synth.Graph(n, eu, ev, rng.random(120, dtype=np.float32), f"sparse{n}")
        want = oracle.greedy(n, g.eu, g.ev, g.w, 3)
        other = synth.er(500, 2000, seed=4)
        h, ho = L.graph(g), L.graph(other)
        for stats in (False, True):
            mate = torch.full((n,), 7, dtype=torch.int32, device="cuda")
            lm.lm_match(L.ctx, h, 3, mate, stats=stats)
            assert np.array_equal(mate.cpu().numpy().view(np.uint32), want)
            mates = [torch.full((k,), 7, dtype=torch.int32, device="cuda") for k in (500, n, 500)]
            lm.lm_batch_match(L.ctx, [ho, h, ho], [3, 3, 3], mates, stats=stats)
            assert np.array_equal(mates[1].cpu().numpy().view(np.uint32), want)
            assert np.array_equal(mates[2].cpu().numpy().view(np.uint32),
                                  oracle.greedy(500, other.eu, other.ev, other.w, 3))
        lm.lm_graph_destroy(h)
        lm.lm_graph_destroy(ho)
    finally:
        L.close()
