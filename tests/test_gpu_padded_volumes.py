"""Volumes whose rows are no multiple of 16 bytes: the TMA form on padded rows against the FP64
oracle at remainders 1, 2 and 3, up to six channels, every norm, several z chunks, and against
the per-thread form, which takes over where the padding does not fit the memory limit.

Tolerances of test_gpu_3d.py and test_gpu_momt3d.py; the two GPU forms round every value alike,
so their fields are equal bit for bit.
"""
import numpy as np
import pytest

import oracle
from paper_1712_10279_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")


def _t(x):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


@pytest.fixture(autouse=True)
def _restore_limit():
    yield
    if torch.cuda.is_available():
        V.set_memory_limit()


def _rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / (nb if nb > 0 else 1.0)


def _f64(x):
    return np.asarray(x, np.float32).astype(np.float64)


def _edges(k):
    return [] if k == 1 else (S.complete_graph(k) if k <= 5 else [(c, c + 1) for c in range(k - 1)])


@pytest.mark.parametrize("n,k,zc", [(41, 1, 0), (42, 2, 7), (43, 3, 1), (45, 4, 0), (47, 5, 5), (41, 6, 3), (75, 3, 0)])
@pytest.mark.parametrize("norms", [(0, 0), (1, 1), (2, 0)])
def test_vector_volumes_match_oracle_and_the_per_thread_form(n, k, zc, norms):
    un, wn = norms
    if k == 1 and wn:
        pytest.skip("no edges at k = 1")
    r0, r1 = (x * x.size for x in S.blob_pair3(n, k, seed=n + k))
    kw = dict(u_norm=un, w_norm=wn, max_iters=40, check_every=20, zc=zc)
    V.set_memory_limit()
    a = V.solve3d(_t(r0), _t(r1), _edges(k), 0.7, **kw)
    assert V.last_form() == "step3 padded"
    V.set_memory_limit(0)
    b = V.solve3d(_t(r0), _t(r1), _edges(k), 0.7, **kw)
    assert V.last_form() == "step3"
    assert torch.equal(a.phi, b.phi) and torch.equal(a.u, b.u) and torch.equal(a.w, b.w)
    r = a.result
    o = oracle.vomt3_solve(_f64(r0), _f64(r1), _edges(k), 0.7, tau=r["tau"], mu=r["mu"], nu=r["nu"], u_norm=un,
                           w_norm=wn, max_iters=40, check_every=20)
    assert _rel(a.phi.cpu().numpy(), o["phi"]) <= 1e-3
    assert _rel(a.u.cpu().numpy(), np.stack([o["ux"], o["uy"], o["uz"]])) <= 1e-3
    if k > 1:
        assert _rel(a.w.cpu().numpy(), o["w"]) <= 1e-3
    for x in (r, b.result):
        assert x["primal"] == pytest.approx(o["metrics"]["primal"], rel=1e-4)


@pytest.mark.parametrize("n,k,zc", [(41, 2, 0), (42, 3, 5), (43, 3, 0)])
@pytest.mark.parametrize("norms", [(V.U_L2, V.W_L1), (V.U_L1, V.W_L2), (V.U_NUC, V.W_L1), (V.U_NUC, V.W_NUC)])
def test_tensor_volumes_match_oracle_and_the_per_thread_form(n, k, zc, norms):
    un, wn = norms
    L0, L1 = (x * n ** 3 for x in S.tensor_field_pair3(n, k, seed=n))
    L = S.random_L(k, 3, seed=31 + k)
    kw = dict(u_norm=un, w_norm=wn, max_iters=30, check_every=15, zc=zc)
    V.set_memory_limit()
    a = V.momt_solve3d(_t(L0), _t(L1), L, 0.7, **kw)
    assert V.last_form() == "step3 padded"
    V.set_memory_limit(0)
    b = V.momt_solve3d(_t(L0), _t(L1), L, 0.7, **kw)
    assert V.last_form() == "step3"
    for x, y in ((a.Phi, b.Phi), (a.U, b.U), (a.W, b.W)):
        assert _rel(x.cpu().numpy().astype(np.float64), y.cpu().numpy().astype(np.float64)) <= 1e-6
    r = a.result
    o = oracle.momt3_solve(_f64(L0), _f64(L1), L, 0.7, tau=r["tau"], mu=r["mu"], nu=r["nu"], u_norm=un, w_norm=wn,
                           max_iters=30, check_every=15)
    assert _rel(a.Phi.cpu().numpy(), o["Phi"]) <= 1e-3
    assert _rel(a.U.cpu().numpy(), np.stack([o["Ux"], o["Uy"], o["Uz"]])) <= 1e-3
    assert _rel(a.W.cpu().numpy().reshape(o["W"].shape), o["W"]) <= 1e-3
    assert r["primal"] == pytest.approx(o["metrics"]["primal"], rel=1e-4)


def test_warm_start_and_stop_on_padded_rows():
    n, k = 43, 2
    r0, r1 = (_t(x * x.size) for x in S.blob_pair3(n, k, seed=9))
    whole = V.solve3d(r0, r1, _edges(k), 0.7, max_iters=60, check_every=10)
    half = V.solve3d(r0, r1, _edges(k), 0.7, max_iters=30, check_every=10)
    rest = V.solve3d(r0, r1, _edges(k), 0.7, max_iters=30, check_every=10, init=(half.u, half.w, half.phi))
    assert V.last_form() == "step3 padded"
    assert torch.equal(rest.phi, whole.phi) and torch.equal(rest.u, whole.u) and torch.equal(rest.w, whole.w)
    met = V.solve3d(r0, r1, _edges(k), 0.7, max_iters=60, check_every=10, tol_gap=1e9, tol_res=1e9)
    assert met.result["iters"] == 10 and met.result["checks"] == 1
