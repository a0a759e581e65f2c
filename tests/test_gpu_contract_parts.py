"""Contraction by partitions of the hash: sizes at the edges of its tiles and of the rule
that counts its partitions, groups beyond what one partition takes at once (passes by
residue), a residue beyond that (the pair sort), and a pair that outgrows a partition's
room (the hash sort instead), each identical to the oracle's contraction."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gpu_util import NIL, Lm
from test_gpu_contract import _contract, _same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lmc():
    c = Lm()
    yield c
    c.close()


def _edges(rng, n, m):
    eu = rng.integers(0, n, m, dtype=np.uint32)
    ev = ((eu + rng.integers(1, n, m, dtype=np.uint32)) % n).astype(np.uint32)
    return eu, ev, rng.standard_normal(m).astype(np.float32)


@pytest.mark.parametrize("m", [1, 2, 3, 31, 33, 8191, 8192, 8193, 16383, 16384, 16385, 32769, 40001, 262147])
def test_sizes(lmc, m):
    # about one edge in four in a group of several, orientations mixed, some pairs matched
    rng = np.random.default_rng(m)
    n = max(3, int(1.2 * m ** 0.5))
    eu, ev, w = _edges(rng, n, m)
    mate = oracle.greedy(n, eu, ev, w, 7) if m & 1 else np.full(n, NIL, np.uint32)
    _same(_contract(lmc, n, eu, ev, w, mate), oracle.contract(n, eu, ev, w, mate))


@pytest.mark.parametrize("kind", ["every_pair_twice", "one_pair_7000", "one_pair_40000", "pairs_of_500"])
def test_groups_beyond_a_partition(lmc, kind):
    # 64 partitions of about 8000 items, 16000 at most, 6144 of them at once
    rng = np.random.default_rng(5)
    n, m = 100_000, 512_000
    eu, ev, w = _edges(rng, n, m)
    if kind == "every_pair_twice":
        eu[m // 2:], ev[m // 2:] = ev[: m // 2], eu[: m // 2]
    elif kind == "pairs_of_500":
        eu[:], ev[:] = eu[np.arange(m) % (m // 500)], ev[np.arange(m) % (m // 500)]
    else:
        k = rng.permutation(m)[: int(kind.rsplit("_", 1)[1])]
        eu[k], ev[k] = 17, 4711
    p = rng.permutation(m)
    eu, ev = eu[p], ev[p]
    mate = np.full(n, NIL, np.uint32)
    _same(_contract(lmc, n, eu, ev, w, mate), oracle.contract(n, eu, ev, w, mate))


@pytest.mark.parametrize("n,m", [(64, 4_000_000), (12, 400_000)])
def test_few_pairs_outgrow_their_partitions(lmc, n, m):
    # 2016 and 66 pairs over 512 and 64 partitions: some get more than twice the average of 4
    # and 1, so the list is sorted
    rng = np.random.default_rng(n)
    eu, ev, w = _edges(rng, n, m)
    for mate in (np.full(n, NIL, np.uint32), oracle.greedy(n, eu, ev, w, 7)):
        _same(_contract(lmc, n, eu, ev, w, mate), oracle.contract(n, eu, ev, w, mate))


@pytest.mark.parametrize("bits", [0, 8], ids=["partitions", "sort"])
@pytest.mark.parametrize("length", [2, 8, 9, 31, 32, 33, 63, 64, 65, 200])
def test_runs_of_every_length(lmc, length, bits):
    # runs put in order by a thread (up to 8), by a warp (up to 64), or left to the pair sort;
    # a few longer and shorter ones among them, all shuffled, orientations mixed
    lm, rng = lmc.lm, np.random.default_rng(length)
    n = 5000
    pairs = 12_000 // length
    times = np.full(pairs, length)
    times[::7] = rng.integers(1, 2 * length + 2, times[::7].size)
    u = rng.integers(0, n, pairs, dtype=np.uint32)
    v = ((u + rng.integers(1, n, pairs, dtype=np.uint32)) % n).astype(np.uint32)
    eu, ev = np.repeat(u, times), np.repeat(v, times)
    p = rng.permutation(eu.size)
    eu, ev = eu[p], ev[p]
    flip = rng.random(eu.size) < 0.5
    eu, ev = np.where(flip, ev, eu), np.where(flip, eu, ev)
    w = rng.standard_normal(eu.size).astype(np.float32)
    mate = np.full(n, NIL, np.uint32)
    keep = lm.lm_get_tuning(lmc.ctx)
    tune = {x: keep[x] for x in ("rmax", "chunk", "sweep_ctas_per_sm", "vertex_ctas_per_sm", "batch")}
    try:
        lm.lm_set_tuning(lmc.ctx, **tune, contract_bits=bits)
        _same(_contract(lmc, n, eu, ev, w, mate), oracle.contract(n, eu, ev, w, mate))
    finally:
        lm.lm_set_tuning(lmc.ctx, **tune, contract_bits=keep["contract_bits"])


@pytest.mark.parametrize("m", [66_000_001, 70_000_000, 135_000_003])
def test_many_partitions(lmc, m):
    # 1024, 2048 and 4096 partitions, against the sort (which the smaller sizes tie to the
    # oracle); a twentieth of the edges repeated, in the other orientation
    torch, lm = lmc.torch, lmc.lm
    n = 3_000_000
    gen = torch.Generator(device="cuda").manual_seed(m)
    eu = torch.randint(0, n, (m,), generator=gen, device="cuda", dtype=torch.int32)
    ev = torch.randint(0, n, (m,), generator=gen, device="cuda", dtype=torch.int32)
    ev = torch.where(ev == eu, (ev + 1) % n, ev)
    k = m // 20
    eu[-k:], ev[-k:] = ev[:k].clone(), eu[:k].clone()
    w = torch.rand(m, generator=gen, device="cuda")
    mate = torch.arange(n, device="cuda", dtype=torch.int32) ^ 1   # pairs (2 i, 2 i + 1)
    keep = lm.lm_get_tuning(lmc.ctx)
    tune = {x: keep[x] for x in ("rmax", "chunk", "sweep_ctas_per_sm", "vertex_ctas_per_sm", "batch")}
    got = lm.lm_contract(lmc.ctx, n, eu, ev, w, mate)
    try:
        lm.lm_set_tuning(lmc.ctx, **tune, contract_bits=16)
        want = lm.lm_contract(lmc.ctx, n, eu, ev, w, mate)
    finally:
        lm.lm_set_tuning(lmc.ctx, **tune, contract_bits=keep["contract_bits"])
    for a, b in zip(got, want):
        assert torch.equal(a, b)
