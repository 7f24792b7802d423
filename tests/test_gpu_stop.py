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


def _batch(shapes, moving, seed):
    """Problems of the given (n, k); those not in `moving` have equal densities and stop at
    their first check."""
    probs, r0, r1 = [], [], []
    for q, (n, k) in enumerate(shapes):
        a, b = S.blob_pair(n, k, seed=seed + q)
        probs.append(dict(n=n, k=k, edges=_edges(k), alpha=0.2 + 0.1 * (q % 4), tau=0.003 * k * n * n))
        r0.append(a.astype(np.float32))
        r1.append((b if q in moving else a).astype(np.float32))
    return V.Batch(probs, r0, r1), V.Batch(probs, r0, r1)


def _same(a, b, count):
    for q in range(count):
        x, y = a.results[q], b.results[q]
        assert (x["iters"], x["status"], x["checks"]) == (y["iters"], y["status"], y["checks"])
        assert torch.equal(a.phi(q), b.phi(q)) and torch.equal(a.u(q), b.u(q)) and torch.equal(a.w(q), b.w(q))


@pytest.mark.parametrize("shapes,moving", [
    ([(256, 3)] * 8, (2,)),
    ([(256, 3)] * 6 + [(200, 5)] * 4 + [(128, 1)] * 3, (0, 4, 11)),         # every five-channel problem stops
    ([(255, 5), (97, 5), (256, 3), (33, 1), (256, 3), (250, 5), (2, 1), (9, 3)], (1, 2, 5)),
])
@pytest.mark.parametrize("kw", [dict(max_iters=500, check_every=20, tol_gap=1e-6, tol_res=1e-6),
                                dict(max_iters=1500, check_every=50, tol_gap=0.3, tol_res=0.3),
                                dict(max_iters=90, check_every=4, tol_gap=1e-6, tol_res=1e-6)])
def test_batches_go_on_with_the_problems_left(shapes, moving, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    auto, grouped = _batch(shapes, moving, 7)
    auto.solve(**kw)
    assert V.last_form() == "batch march"
    grouped.solve(path="grouped", **kw)
    _same(auto, grouped, len(shapes))
    stopped = [q for q in range(len(shapes)) if q not in moving]
    assert all(auto.results[q]["checks"] == 1 for q in stopped)
    if kw["tol_gap"] < 1e-3:                   # the passes were planned again: more blocks for those left
        assert all(auto.results[q]["iters"] == kw["max_iters"] for q in moving)
        pairs = [(q, s) for q in moving for s in stopped if shapes[q] == shapes[s]]
        assert pairs and all(auto.results[q]["blocks"] > auto.results[s]["blocks"] for q, s in pairs)


@pytest.mark.parametrize("shapes", [[(256, 3)] * 6, [(64, 5)] * 40, [(200, 4), (160, 2)] * 6])
def test_few_batch_launches_follow_the_deciding_check(shapes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    auto, grouped = _batch(shapes, range(len(shapes)), 3)
    auto.solve(max_iters=200000, check_every=100, **ANY)
    assert V.last_form() == "batch march"
    grouped.solve(max_iters=200000, check_every=100, path="grouped", **ANY)
    _same(auto, grouped, len(shapes))
    groups = len({k for _, k in shapes})
    assert all(r["checks"] == 1 for r in auto.results)
    assert auto.results[0]["launches"] <= 10 + groups * 2 * 102
