"""The largest vertex counts (2^32 - 2), where vertex numbers of a grid's next step and a
rounded-up tile count do not fit 32 bits: graph creation and contraction with few edges."""
import numpy as np
import pytest

from gpu_util import Lm

pytestmark = pytest.mark.gpu

N = (1 << 32) - 2
CHUNK = 1 << 27


def _need(torch, gib):
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < gib << 30:
        pytest.skip(f"needs {gib} GiB of free device memory")


def _i32(xs):
    return np.array(xs, np.uint32)


def test_graph_creation_with_the_most_vertices():
    import paper_1302_4587_gb300 as lm
    L = Lm()
    try:
        _need(L.torch, 80)
        eu, ev = _i32([0, N - 1, 5]), _i32([N - 1, N - 2, N - 2])
        h = lm.lm_graph_create(L.ctx, N, eu, ev, np.array([1, 2, 3], np.float32))
        assert lm.lm_graph_info(h)[:2] == (N, 3)
        lm.lm_graph_destroy(h)
        with pytest.raises(lm.LmError) as ei:   # the last id is n - 1
            lm.lm_graph_create(L.ctx, N, _i32([0]), _i32([N]), np.ones(1, np.float32))
        assert ei.value.code == lm.LM_EINVAL
    finally:
        L.close()


def test_contraction_with_the_most_vertices():
    import paper_1302_4587_gb300 as lm
    L = Lm()
    torch = L.torch
    try:
        _need(torch, 100)
        mate = torch.empty(N, dtype=torch.int32, device="cuda")   # 2k and 2k + 1 are a pair
        for a in range(0, N, CHUNK):
            b = min(a + CHUNK, N)
            mate[a:b] = torch.arange(a, b, device="cuda").bitwise_xor_(1).to(torch.int32)
        eu, ev = _i32([0, N - 1, 4, 6]), _i32([N - 1, 1, 5, N - 2])
        w = np.array([1, 2, 4, 8], np.float32)
        dev = [torch.from_numpy(x.view(np.int32) if x.dtype == np.uint32 else x).cuda() for x in (eu, ev, w)]
        cmap, cvw, ceu, cev, cw = lm.lm_contract(L.ctx, N, *dev, mate)
        assert cvw.numel() == N // 2
        for a in range(0, N, CHUNK):
            b = min(a + CHUNK, N)
            assert bool((cmap[a:b] == (torch.arange(a, b, device="cuda") >> 1)).all()), a
        for a in range(0, N // 2, CHUNK):
            assert bool((cvw[a:a + CHUNK] == 2).all()), a
        # (0, n - 1) and (n - 1, 1) are one coarse edge, (4, 5) is inside a pair
        assert ceu.tolist() == [0, 3] and cev.tolist() == [N // 2 - 1] * 2 and cw.tolist() == [3.0, 8.0]
    finally:
        L.close()
        torch.cuda.empty_cache()
