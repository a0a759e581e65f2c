"""lm_match_small_noalloc at the sizes where its kernels change hands: one block or a
cluster (8192 vertices, 4096 edges), edges in registers or lists (65,536 edges with
eight blocks, 131,072 with sixteen), the smallest graphs, and weights that are
distinct, few or all equal (the second maximum then decides).  Equal to the
oracle's greedy matching."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_util import to_u32

pytestmark = pytest.mark.gpu

SIZES = [(2, 1), (3, 2), (100, 99), (8192, 4096), (8193, 4096), (8192, 4097), (5000, 65_536), (5000, 65_537),
         (20_001, 131_072), (20_001, 131_073), (65_536, 40_000), (600, 100_000)]


@pytest.mark.parametrize("kind", ["uniform", "few", "unit", "inf"])
@pytest.mark.parametrize("n,m", SIZES)
def test_small_graphs_equal_the_oracle(n, m, kind):
    import torch
    import paper_1302_4587_gb300 as lm
    rng = np.random.default_rng(n * 31 + m)
    eu = rng.integers(0, n, m).astype(np.uint32)
    ev = ((eu + 1 + rng.integers(0, n - 1, m)) % n).astype(np.uint32)   # never a loop; parallel edges occur
    w = synth.weights(m, n + m, unit=kind == "unit")
    if kind == "few":
        w = (np.floor(w * 4.0) / 4.0).astype(np.float32)
    elif kind == "inf":
        w[::3] = np.inf
        w[1::5] = -np.inf
    mate = torch.full((n,), 12345, dtype=torch.int32, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    lm.lm_match_small_noalloc(n, torch.from_numpy(eu.view(np.int32)).cuda(), torch.from_numpy(ev.view(np.int32)).cuda(),
                              torch.from_numpy(w).cuda(), 7, mate, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert np.array_equal(to_u32(mate), oracle.greedy(n, eu, ev, w, 7))
