"""Dense graphs whose vertices agree on their heaviest neighbours: every row passes over its
list many times and scans its entries again, by a warp (129 entries and more), a block
(1025) or in chunks at first (2049), looking only at entries no heavier than its last list's."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_util import NIL, Lm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    c = Lm()
    yield c
    c.close()


@pytest.mark.parametrize("kind", ["distinct", "levels", "negative", "unit"])
@pytest.mark.parametrize("n", [66, 129, 130, 300, 1025, 1026, 2050])
def test_rows_that_agree(L, n, kind):
    rng = np.random.default_rng(n)
    eu, ev = (x.astype(np.uint32) for x in np.triu_indices(n, 1))
    p = rng.permutation(eu.shape[0])
    eu, ev = eu[p], ev[p]
    f = rng.permutation(n).astype(np.float32)
    w = f[eu] + f[ev] + rng.random(eu.shape[0], dtype=np.float32)
    if kind == "levels":
        w = np.floor(w / 16).astype(np.float32)
    elif kind == "negative":
        w = -w
    elif kind == "unit":
        w = np.ones_like(w)
    g = synth.Graph(n, eu, ev, w.astype(np.float32), f"dense_{kind}")
    want, r, rm, rn = oracle.seq_local_max(g.n, g.eu, g.ev, g.w, 3)
    h = L.graph(g)
    try:
        out = L.torch.empty(n, dtype=L.torch.int32, device="cuda")
        L.lm.lm_match(L.ctx, h, 3, out)   # without rounds
        assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
        mate, st = L.match(g, 3, handle=h)
        assert np.array_equal(mate, want) and st["rounds"] == r
        assert st["matched"] == int((want != NIL).sum()) // 2
        k = min(r, 64)
        assert st["round_m"][:k] == [int(x) for x in rm[:k]] and st["round_n"][:k] == [int(x) for x in rn[:k]]
    finally:
        L.lm.lm_graph_destroy(h)
