"""The memory of a batch in the marching form: a batch whose states exceed the limit runs in
parts, with the same results, and a limit below one problem leaves it to the grouped path."""
import numpy as np
import pytest

from paper_1712_10279_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")


@pytest.fixture(autouse=True)
def _restore_limit():
    yield
    if torch.cuda.is_available():
        V.set_memory_limit()


def _batch(shapes, seed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    probs, r0, r1 = [], [], []
    for q, (n, k) in enumerate(shapes):
        a, b = S.blob_pair(n, k, seed=seed + q)
        probs.append(dict(n=n, k=k, edges=S.complete_graph(k) if k > 1 else [], alpha=0.2 + 0.1 * (q % 4),
                          tau=0.003 * k * n * n))
        r0.append(a.astype(np.float32))
        r1.append(b.astype(np.float32))
    return V.Batch(probs, r0, r1)


SHAPES = [(128, 5), (64, 5)] * 12 + [(100, 3)] * 4       # 94 MiB of states


@pytest.mark.parametrize("kw", [dict(max_iters=60, check_every=20),
                                dict(max_iters=900, check_every=20, tol_gap=0.3, tol_res=0.3)])
@pytest.mark.parametrize("warm", [False, True])
def test_parts_give_the_same_results(kw, warm):
    whole, parts = _batch(SHAPES, 1), _batch(SHAPES, 1)
    for batch, limit in ((whole, 1 << 30), (parts, 30 << 20)):
        V.set_memory_limit(limit)
        batch.solve(**kw)
        assert V.last_form() == "batch march"
        if warm:
            batch.solve(warm_start=True, **kw)
            assert V.last_form() == "batch march"
    for q in range(len(SHAPES)):
        x, y = whole.results[q], parts.results[q]
        assert (x["iters"], x["status"], x["checks"]) == (y["iters"], y["status"], y["checks"])
        assert x["primal"] == pytest.approx(y["primal"], rel=1e-6)
    assert torch.equal(whole.arena, parts.arena)


def test_the_limit_bounds_the_memory():
    batch = _batch(SHAPES, 1)
    V.set_memory_limit(0)
    batch.solve(max_iters=20, check_every=20)
    assert V.last_form() == "batch grouped"
    torch.cuda.synchronize()
    used = {}
    for limit in (30 << 20, 1 << 30):
        V.set_memory_limit(limit)
        free = torch.cuda.mem_get_info()[0]
        batch.solve(max_iters=20, check_every=20)
        assert V.last_form() == "batch march"
        used[limit] = free - torch.cuda.mem_get_info()[0]
        V.set_memory_limit(0)
        assert torch.cuda.mem_get_info()[0] - free > -(4 << 20)
    assert used[30 << 20] <= 40 << 20 and used[1 << 30] >= 90 << 20
