"""Marching solves that stop at a tolerance: few launches past the deciding check, the iterate
of that check, and the same stop as the engines that stop inside their kernel."""
import numpy as np
import pytest

from paper_1712_10279_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")

ANY = dict(tol_gap=1e9, tol_res=1e9)      # met by the first check
FOREVER = 10 ** 6


def _t(x):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


def _pair(n, k, seed):
    return tuple(_t(x) for x in S.blob_pair(n, k, seed=seed))


def _edges(k):
    return S.complete_graph(k) if k > 1 else []


@pytest.mark.parametrize("n,k,check", [(352, 3, 100), (444, 3, 12), (400, 1, 200), (512, 3, 8), (200, 8, 50),
                                       (768, 3, 100)])
def test_few_launches_follow_the_deciding_check(n, k, check):
    """An interval launches at most `check` passes and two check kernels; what is queued beyond
    the first stays within two polls of about 150 us, at least 2 us a launch each."""
    r0, r1 = _pair(n, k, n)
    kw = dict(tau=0.003 * k * n * n, check_every=check)
    a = V.solve(r0, r1, _edges(k), 0.3, max_iters=FOREVER, **kw, **ANY)
    assert V.last_form() == "march"
    assert a.result["iters"] == check and a.result["checks"] == 1 and a.result["status"] == 0
    assert a.result["launches"] <= 10 + 2 * max(check + 2, 150 // 2)
    fixed = V.solve(r0, r1, _edges(k), 0.3, max_iters=check, **kw)
    assert torch.equal(a.u, fixed.u) and torch.equal(a.w, fixed.w) and torch.equal(a.phi, fixed.phi)
    assert a.result["primal"] == fixed.result["primal"]


@pytest.mark.parametrize("n,k,check", [(352, 3, 20), (352, 3, 100), (440, 1, 50)])
def test_stops_where_the_resident_engine_stops(n, k, check):
    r0, r1 = _pair(n, k, n + 1)
    kw = dict(tau=0.003 * k * n * n, check_every=check, max_iters=40000, tol_gap=0.2, tol_res=0.2)
    a = V.solve(r0, r1, _edges(k), 0.3, **kw)
    assert V.last_form() == "march"
    b = V.solve(r0, r1, _edges(k), 0.3, engine="resident", **kw)
    assert 1 < a.result["checks"] == b.result["checks"] and a.result["iters"] == b.result["iters"]
    assert torch.equal(a.u, b.u) and torch.equal(a.w, b.w) and torch.equal(a.phi, b.phi)
    assert len(V.history()) == b.result["checks"]


@pytest.mark.parametrize("check", [2 ** 31 - 1, 2 ** 31 - 2048, 2000])
@pytest.mark.parametrize("tol", [0.0, 1e-30])
def test_an_interval_beyond_the_cap_checks_once(check, tol):
    r0, r1 = _pair(352, 3, 3)
    a = V.solve(r0, r1, _edges(3), 0.3, tau=1000.0, max_iters=37, check_every=check, tol_gap=tol, tol_res=tol)
    assert V.last_form() == "march"
    assert a.result["iters"] == 37 and a.result["checks"] == 1 and a.result["status"] == (1 if tol else 0)
