"""The served form's contract through the C ABI: admission limits, unknown
tickets, empty graphs, the same graph in flight many times with different
seeds, and shutdown with requests in flight."""
from __future__ import annotations

import time

import numpy as np
import pytest

import oracle
import synth
from gpu_util import NIL, Lm, to_u32

pytestmark = pytest.mark.gpu


def test_request_larger_than_the_budget_is_refused():
    import paper_1302_4587_gb300 as lm
    srv = Lm(budget=1 << 20)  # room for about 33 thousand entries
    try:
        g = synth.er(20_000, 40_000, seed=3)
        h = srv.graph(g)
        mate = np.empty(g.n, np.uint32)
        with pytest.raises(lm.LmError) as ei:
            lm.lm_submit(srv.ctx, h, 1, mate)
        assert ei.value.code == lm.LM_ENOMEM
        small = synth.er(200, 600, seed=4)
        hs = srv.graph(small)
        ms = np.empty(small.n, np.uint32)
        t = lm.lm_submit(srv.ctx, hs, 2, ms)  # a request that fits is still served
        assert lm.lm_wait(srv.ctx, t, 60_000)
        assert lm.lm_poll(srv.ctx, t)[0]
        assert np.array_equal(ms, oracle.greedy(small.n, small.eu, small.ev, small.w, 2))
        lm.lm_graph_destroy(h)
        lm.lm_graph_destroy(hs)
    finally:
        srv.close()


def test_unknown_tickets():
    import paper_1302_4587_gb300 as lm
    srv = Lm()
    try:
        for fn in (lambda: lm.lm_poll(srv.ctx, 123456), lambda: lm.lm_wait(srv.ctx, 123456, 10)):
            with pytest.raises(lm.LmError) as ei:
                fn()
            assert ei.value.code == lm.LM_ENOTFOUND
    finally:
        srv.close()


def test_empty_graphs_are_served():
    import paper_1302_4587_gb300 as lm
    srv = Lm()
    try:
        cases = [synth.Graph(7, np.zeros(0, np.uint32), np.zeros(0, np.uint32), np.zeros(0, np.float32), "edgeless"),
                 synth.Graph(0, np.zeros(0, np.uint32), np.zeros(0, np.uint32), np.zeros(0, np.float32), "empty")]
        for g in cases:
            h = srv.graph(g, device=False)
            mate = np.full(max(g.n, 1), 5, np.uint32)[: g.n]
            t = lm.lm_submit(srv.ctx, h, 1, mate)
            assert lm.lm_wait(srv.ctx, t, 60_000)
            done, st = lm.lm_poll(srv.ctx, t)
            assert done and st["rounds"] == 0 and st["matched"] == 0
            assert (mate == NIL).all()
            lm.lm_graph_destroy(h)
    finally:
        srv.close()


def test_one_graph_many_seeds_in_flight():
    import paper_1302_4587_gb300 as lm
    srv = Lm()
    try:
        g = synth.grid(128, 128, 0.05, seed=12, unit=True)  # unit weights: the seed decides
        h = srv.graph(g)
        mates = [srv.torch.empty(g.n, dtype=srv.torch.int32, device="cuda") for _ in range(16)]
        tickets = [lm.lm_submit(srv.ctx, h, 900 + i, m) for i, m in enumerate(mates)]
        for i, t in enumerate(tickets):
            assert lm.lm_wait(srv.ctx, t, 60_000)
            assert lm.lm_poll(srv.ctx, t)[0]
            assert np.array_equal(to_u32(mates[i]), oracle.greedy(g.n, g.eu, g.ev, g.w, 900 + i))
        lm.lm_graph_destroy(h)
    finally:
        srv.close()


def test_destroy_with_requests_in_flight_returns():
    import paper_1302_4587_gb300 as lm
    srv = Lm()
    g = synth.grid(256, 256, 0.05, seed=13)
    h = srv.graph(g)
    mates = [srv.torch.empty(g.n, dtype=srv.torch.int32, device="cuda") for _ in range(8)]
    for i, m in enumerate(mates):
        lm.lm_submit(srv.ctx, h, i, m)
    t0 = time.perf_counter()
    srv.close()  # stops the scheduler; must not hang on the requests in flight
    assert time.perf_counter() - t0 < 30
    # (the graph belonged to the destroyed context: its handle is abandoned, not destroyed)


def _mono_path(n):
    eu = np.arange(n - 1, dtype=np.uint32)
    return synth.Graph(n, eu, eu + 1, (np.arange(n - 1) + 1).astype(np.float32), f"mono{n}")


def test_a_request_beyond_a_limit_fails_alone():
    # the path needs 1500 rounds, the others at most 40; all of them wait together behind
    # two larger graphs, so that they are taken as groups
    import paper_1302_4587_gb300 as lm
    srv = Lm()
    try:
        lm.lm_set_limits(srv.ctx, 40, 0)
        big = [synth.er(1_000_000, 4_000_000, seed=s) for s in (1, 2)]
        small = [synth.er(300 + 10 * i, 900 + 50 * i, seed=20 + i) for i in range(12)]
        order = big + small[:6] + [_mono_path(3001)] + small[6:]
        hs = [srv.graph(g) for g in order]
        want = [oracle.greedy(g.n, g.eu, g.ev, g.w, 5) for g in order]
        for _ in range(5):
            mates = [srv.torch.empty(g.n, dtype=srv.torch.int32, device="cuda") for g in order]
            tickets = [lm.lm_submit(srv.ctx, h, 5, m) for h, m in zip(hs, mates)]
            for g, t, m, x in zip(order, tickets, mates, want):
                assert lm.lm_wait(srv.ctx, t, 60_000)
                if g.name.startswith("mono"):
                    with pytest.raises(lm.LmError) as ei:
                        lm.lm_poll(srv.ctx, t)
                    assert ei.value.code == lm.LM_ETIMEOUT
                else:
                    done, st = lm.lm_poll(srv.ctx, t)
                    assert done and st["rounds"] <= 40 and st["matched"] == int((x != NIL).sum()) // 2
                    assert np.array_equal(to_u32(m), x)
        for h in hs:
            lm.lm_graph_destroy(h)
    finally:
        srv.close()


def _serve(srv, handles, mates, seed=5):
    import paper_1302_4587_gb300 as lm
    return [lm.lm_submit(srv.ctx, h, seed, m) for h, m in zip(handles, mates)]


def _finish(srv, g, ticket, mate, want):
    import paper_1302_4587_gb300 as lm
    assert lm.lm_wait(srv.ctx, ticket, 60_000)
    done, st = lm.lm_poll(srv.ctx, ticket)
    assert done and st["matched"] == int((want != NIL).sum()) // 2
    assert np.array_equal(to_u32(mate) if not isinstance(mate, np.ndarray) else mate, want), g.name


@pytest.mark.parametrize("host", [False, True], ids=["device", "host"])
def test_short_requests_leave_before_a_long_one(host):
    # the path needs 100,000 rounds (half a second), the others a handful; two larger graphs
    # keep both lanes busy while the others arrive, so that they are taken together
    import paper_1302_4587_gb300 as lm
    srv = Lm()
    try:
        big = [synth.er(1_000_000, 4_000_000, seed=s) for s in (1, 2)]
        path = _mono_path(200_001)
        small = [synth.er(300 + 10 * i, 900 + 50 * i, seed=20 + i) for i in range(12)]
        order = big + small[:6] + [path] + small[6:]
        hs = [srv.graph(g) for g in order]
        want = [oracle.greedy(g.n, g.eu, g.ev, g.w, 5) for g in order]
        mates = [np.zeros(g.n, np.uint32) if host else srv.torch.empty(g.n, dtype=srv.torch.int32, device="cuda")
                 for g in order]
        tickets = _serve(srv, hs, mates)
        for g, t, m, x in zip(order, tickets, mates, want):
            if g is not path:
                _finish(srv, g, t, m, x)
        assert not lm.lm_poll(srv.ctx, tickets[8])[0]   # still on its way
        _finish(srv, path, tickets[8], mates[8], want[8])
        for h in hs:
            lm.lm_graph_destroy(h)
    finally:
        srv.close()


def test_arrivals_pass_groups_of_many_rounds():
    # both lanes are busy with paths of half a second and more when the others arrive
    import paper_1302_4587_gb300 as lm
    srv = Lm()
    try:
        paths = [_mono_path(200_001 + 2 * i) for i in range(4)]
        small = [synth.er(300 + 10 * i, 900 + 50 * i, seed=20 + i) for i in range(4)] + [synth.grid(300, 300, 0.05, seed=3)]
        hp, hs = [srv.graph(g) for g in paths], [srv.graph(g) for g in small]
        wp, ws = ([oracle.greedy(g.n, g.eu, g.ev, g.w, 5) for g in gs] for gs in (paths, small))
        new = lambda gs: [srv.torch.empty(g.n, dtype=srv.torch.int32, device="cuda") for g in gs]
        mp, ms = new(paths), new(small)
        tp = []
        for h, m in zip(hp, mp):      # one by one, so that both lanes have some
            tp += _serve(srv, [h], [m])
            time.sleep(0.01)
        for _ in range(3):
            ts = _serve(srv, hs, ms)
            for g, t, m, x in zip(small, ts, ms, ws):
                _finish(srv, g, t, m, x)
        assert not any(lm.lm_poll(srv.ctx, t)[0] for t in tp)
        for g, t, m, x in zip(paths, tp, mp, wp):
            _finish(srv, g, t, m, x)
        for h in hp + hs:
            lm.lm_graph_destroy(h)
    finally:
        srv.close()


def test_destroy_with_a_request_of_many_rounds_in_flight():
    import paper_1302_4587_gb300 as lm
    srv = Lm()
    g = _mono_path(2_000_001)   # a million rounds
    h = srv.graph(g)
    mate = srv.torch.empty(g.n, dtype=srv.torch.int32, device="cuda")
    lm.lm_submit(srv.ctx, h, 1, mate)
    time.sleep(0.05)
    t0 = time.perf_counter()
    srv.close()   # at the next slice, not after all rounds
    assert time.perf_counter() - t0 < 2
