"""The renewed order's kernel at the edges of its kinds of row (a thread's, half a warp's,
a warp's, chunks), of its hand-over to one block, with parallel edges, long chains of
rounds, and queued without the host: identical to the oracle's rounds."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_util import NIL, Lm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rn():
    c = Lm(renew=True)
    yield c
    c.close()


def _check(L, g, seed):
    mate, st = L.match(g, seed)
    want, r, rm, rn_ = oracle.seq_local_max(g.n, g.eu, g.ev, g.w, seed, renew=True)
    assert np.array_equal(mate, want), g.name
    assert st["rounds"] == r and st["matched"] == int((want != NIL).sum()) // 2
    k = min(r, 64)
    assert st["round_m"][:k] == [int(x) for x in rm[:k]]
    assert st["round_n"][:k] == [int(x) for x in rn_[:k]]


def _hubs(rng, hub_rows, n, levels):
    """hubs with rows of the given lengths into n other vertices, plus a sparse rest"""
    eu, ev = [], []
    for i, d in enumerate(hub_rows):
        eu.append(np.full(d, n + i, np.uint32))
        ev.append(rng.integers(0, n, d, dtype=np.uint32))
    a = rng.integers(0, n, n, dtype=np.uint32)
    eu.append(a)
    ev.append(((a + rng.integers(1, n, n, dtype=np.uint32)) % n).astype(np.uint32))
    eu, ev = np.concatenate(eu), np.concatenate(ev)
    w = rng.integers(1, levels + 1, eu.shape[0]).astype(np.float32)
    return synth.Graph(n + len(hub_rows), eu, ev, w, f"hubs_{levels}")


@pytest.mark.parametrize("levels", [1, 3, 1 << 20])
@pytest.mark.parametrize("n", [40, 700, 9000])   # (few vertices: parallel edges, dead neighbours early)
def test_row_kinds(rn, n, levels):
    rng = np.random.default_rng(n + levels)
    g = _hubs(rng, [1, 3, 4, 5, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 2047, 2048, 2049, 4096, 4097,
                    66_000], n, levels)
    for seed in (1, 77):
        _check(rn, g, seed)


@pytest.mark.parametrize("n", [2, 3, 33, 511, 512, 513, 1200])
def test_chain_of_rounds(rn, n):
    # weights rising along a path: a matched edge a round, from many live rows down to none
    e = np.arange(n - 1, dtype=np.uint32)
    g = synth.Graph(n, e, e + 1, (e + 1).astype(np.float32), "path")
    _check(rn, g, 9)


def test_queued(rn):
    lm, torch = rn.lm, rn.torch
    ctx = lm.lm_create(0, flags=lm.LM_F_RENEW | lm.LM_F_ASYNC)
    try:
        gs = [synth.er(3000, 20_000, seed=4, unit=True), synth.rmat(scale=12, edge_factor=16, seed=5)]
        hs = [lm.lm_graph_create(ctx, g.n, *(torch.from_numpy(np.ascontiguousarray(x).view(t)).cuda()
                                             for x, t in ((g.eu, np.int32), (g.ev, np.int32), (g.w, np.float32))))
              for g in gs]
        jobs = [(i, s, torch.empty(gs[i].n, dtype=torch.int32, device="cuda")) for s in range(4) for i in range(2)]
        for i, s, mate in jobs:
            lm.lm_match(ctx, hs[i], s, mate)
        lm.lm_sync(ctx)
        for i, s, mate in jobs:
            g = gs[i]
            want = oracle.seq_local_max(g.n, g.eu, g.ev, g.w, s, renew=True)[0]
            assert np.array_equal(mate.cpu().numpy().view(np.uint32), want)
        for h in hs:
            lm.lm_graph_destroy(h)
    finally:
        lm.lm_destroy(ctx)


@pytest.mark.parametrize("n", [16_383, 16_384, 40_000, 5_000_001])
def test_few_edges_among_many_vertices(rn, n):
    # blocks beyond those that the rows need clear the result
    rng = np.random.default_rng(n)
    eu = rng.permutation(n)[:300].astype(np.uint32)
    ev = np.concatenate([eu[1:], eu[:1]])
    w = rng.integers(1, 3, 300).astype(np.float32)
    _check(rn, synth.Graph(n, eu, ev, w, f"sparse{n}"), 5)
