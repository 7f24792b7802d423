"""The marching form of the streaming engine (several iterations per pass) against the FP64
oracle where it can go wrong: grids at the edges of the strips (24, 28, 30 columns), of the
32-column layout blocks and of the chunks, check intervals that leave passes of fewer
iterations, edges in any order and missing pairs, warm starts and early stops.

Tolerances: each iteration rounds every field a few times in FP32 (6e-8), so tens of
iterations leave well under 1e-4 of a field's norm; w is zero except where a threshold is
passed, so its error is bounded against the threshold it cancels with: 1e-3 of its norm.
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


def _rel(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(a - b) / (nb if nb > 0 else 1.0)


def _fields(n, k, seed):
    """Cell masses of order one with equal totals: the fluxes are active at once."""
    rng = np.random.default_rng(seed)
    out = rng.uniform(0.2, 1.0, (2, k, n, n))
    out /= out.mean(axis=(1, 2, 3), keepdims=True)
    return out.astype(np.float32)


def _check(sol, ref):
    u = sol.u.cpu().numpy().astype(np.float64)
    assert _rel(u, np.stack([ref["ux"], ref["uy"]])) < 1e-4
    assert _rel(sol.phi.cpu().numpy().astype(np.float64), ref["phi"]) < 1e-4
    if ref["w"].size:
        assert _rel(sol.w.cpu().numpy().astype(np.float64), ref["w"]) < 1e-3
    assert abs(sol.result["primal"] - ref["metrics"]["primal"]) <= 1e-4 * abs(ref["metrics"]["primal"])
    assert np.all(u[0, :, :, -1] == 0) and np.all(u[1, :, -1, :] == 0)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n", [2, 3, 23, 25, 28, 31, 32, 33, 48, 61, 97])
def test_sizes_and_passes_match_oracle(n, k):
    rng = np.random.default_rng(100 * n + k)
    edges = [e[::rng.choice([-1, 1])] for e in S.random_connected_graph(rng, k, 0.5)]
    rng.shuffle(edges)
    edges = [tuple(int(a) for a in e) for e in edges]
    cost = rng.uniform(0.5, 2.0, len(edges)) if edges else None
    r0, r1 = _fields(n, k, n + 7 * k)
    kw = dict(max_iters=24, check_every=11, tau=0.7, cost=cost)      # passes of 1, 2 and 4 iterations
    sol = V.solve(_t(r0), _t(r1), edges, 0.6, engine="stream", **kw)
    assert sol.result["engine"] == "stream" and sol.result["iters"] == 24 and sol.result["checks"] == 3
    ref = oracle.vomt_solve(r0.astype(np.float64), r1.astype(np.float64), edges, 0.6, history=True, **kw)
    _check(sol, ref)
    h = V.history()
    np.testing.assert_allclose(h[:, 6], ref["history"][:, 6])
    np.testing.assert_allclose(h[:, 0], ref["history"][:, 0], rtol=1e-4)
    np.testing.assert_allclose(h[:, 3], ref["history"][:, 3], rtol=1e-3)
    np.testing.assert_allclose(h[:, 4], ref["history"][:, 4], rtol=5e-2, atol=1e-6 * ref["history"][0, 4])
    np.testing.assert_allclose(h[:, 5], ref["history"][:, 5], rtol=1e-3, atol=1e-4)


@pytest.mark.parametrize("u_norm,w_norm", [(0, 0), (1, 0), (2, 0), (0, 1), (1, 1), (2, 1)])
@pytest.mark.parametrize("eps", [0.0, 0.3])
def test_norms_and_regularisation_match_oracle(u_norm, w_norm, eps):
    n, k, edges = 53, 3, [(1, 2), (0, 1)]
    r0, r1 = _fields(n, k, 5)
    kw = dict(max_iters=20, check_every=10, tau=0.7, u_norm=u_norm, w_norm=w_norm, eps=eps)
    sol = V.solve(_t(r0), _t(r1), edges, 0.6, engine="stream", **kw)
    _check(sol, oracle.vomt_solve(r0.astype(np.float64), r1.astype(np.float64), edges, 0.6, **kw))


def test_chunks_of_a_larger_grid_match_the_resident_engine():
    """Several chunks of rows per strip and more blocks than one wave; the resident engine
    (pinned against the oracle elsewhere) holds the same iterate."""
    n, k, edges = 300, 3, S.COMPLETE_K3
    r0, r1 = _fields(n, k, 9)
    kw = dict(max_iters=43, check_every=20, tau=0.7)
    a = V.solve(_t(r0), _t(r1), edges, 0.6, engine="stream", **kw)
    b = V.solve(_t(r0), _t(r1), edges, 0.6, engine="resident", **kw)
    for x, y, tol in ((a.u, b.u, 1e-4), (a.phi, b.phi, 1e-4), (a.w, b.w, 1e-3)):
        assert _rel(x.double().cpu().numpy(), y.double().cpu().numpy()) < tol


def test_warm_start_continues_and_a_met_tolerance_stops():
    n, k, edges = 40, 3, S.COMPLETE_K3
    r0, r1 = S.blob_pair(n, k, seed=3)
    kw = dict(tau=10.0, check_every=50, engine="stream")
    whole = V.solve(_t(r0), _t(r1), edges, 1.0, max_iters=400, **kw)
    half = V.solve(_t(r0), _t(r1), edges, 1.0, max_iters=200, **kw)
    rest = V.solve(_t(r0), _t(r1), edges, 1.0, max_iters=200, init=(half.u, half.w, half.phi), **kw)
    assert _rel(rest.phi.double().cpu().numpy(), whole.phi.double().cpu().numpy()) < 1e-4
    tol = dict(max_iters=200000, tol_gap=1e-3, tol_res=1e-3)
    a = V.solve(_t(r0), _t(r1), edges, 1.0, **tol, **kw)
    b = V.solve(_t(r0), _t(r1), edges, 1.0, tau=10.0, check_every=50, engine="resident", **tol)
    assert a.result["status"] == 0 and a.result["iters"] % 50 == 0
    assert abs(a.result["iters"] - b.result["iters"]) <= 50
    assert a.result["rel_gap"] <= 1e-3 and a.result["rel_res"] <= 1e-3
    fixed = V.solve(_t(r0), _t(r1), edges, 1.0, max_iters=a.result["iters"], **kw)
    assert torch.equal(fixed.u, a.u) and torch.equal(fixed.phi, a.phi) and torch.equal(fixed.w, a.w)


def _batch(shapes, seed, turn=False):
    rng = np.random.default_rng(seed)
    probs, r0, r1 = [], [], []
    for n, k in shapes:
        edges = S.random_connected_graph(rng, k, 0.6)
        edges = edges[::-1] if turn else edges
        a, b = S.blob_pair(n, k, seed=int(rng.integers(1 << 30)))
        probs.append(dict(n=n, k=k, edges=edges, alpha=float(rng.uniform(0.1, 1.0)), tau=0.003 * k * n * n,
                          cost=rng.uniform(0.5, 2.0, len(edges)) if edges else None))
        r0.append(a.astype(np.float32))
        r1.append(b.astype(np.float32))
    return V.Batch(probs, r0, r1), V.Batch(probs, r0, r1)


@pytest.mark.parametrize("shapes", [
    [(256, 3)] * 6,
    [(256, 1), (255, 3), (192, 5), (97, 5), (256, 3), (33, 1), (128, 3), (250, 5), (200, 2), (180, 4), (2, 1), (9, 3)],
])
@pytest.mark.parametrize("kw", [dict(max_iters=57, check_every=20), dict(max_iters=6, check_every=6),
                                dict(max_iters=2400, check_every=100, tol_gap=3e-2, tol_res=3e-2)])
def test_marching_batch_equals_the_grouped_batch(shapes, kw):
    """AUTO's marching form of a batch against the grouped resident form: the same iterates
    bit for bit (the kernels round alike), each problem stopped at the same check."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    auto, grouped = _batch(shapes, 5)
    auto.solve(**kw)
    grouped.solve(path="grouped", **kw)
    assert all(r["variant"] == 0 and r["blocks"] >= 1 for r in auto.results)      # the marching form ran
    assert all(r["variant"] == 1 for r in grouped.results)
    if "tol_gap" in kw:
        assert len({r["iters"] for r in grouped.results}) > 1 or len(set(shapes)) == 1
    for q in range(len(shapes)):
        a, g = auto.results[q], grouped.results[q]
        assert a["iters"] == g["iters"] and a["status"] == g["status"] and a["checks"] == g["checks"]
        assert torch.equal(auto.phi(q), grouped.phi(q)) and torch.equal(auto.u(q), grouped.u(q))
        assert torch.equal(auto.w(q), grouped.w(q))
        for key in ("primal", "dual", "rel_res"):
            assert a[key] == pytest.approx(g[key], rel=1e-5)
    auto.solve(warm_start=True, **kw)
    grouped.solve(path="grouped", warm_start=True, **kw)
    for q in range(len(shapes)):
        assert torch.equal(auto.phi(q), grouped.phi(q)) and torch.equal(auto.w(q), grouped.w(q))


def test_edges_out_of_order_keep_the_listed_sums():
    """Edges that are not listed in the order of the pairs: the kernels that sum as listed."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    kw = dict(max_iters=57, check_every=20)
    auto, grouped = _batch([(256, 3)] * 4 + [(128, 4)], 7, turn=True)
    auto.solve(**kw)
    grouped.solve(path="grouped", **kw)
    assert all(r["variant"] == 1 for r in auto.results)
    for q in range(5):
        assert torch.equal(auto.phi(q), grouped.phi(q)) and torch.equal(auto.w(q), grouped.w(q))
    r0, r1 = _fields(80, 4, 8)
    a, b = (V.solve(_t(r0), _t(r1), S.complete_graph(4)[::-1], 0.6, engine="stream", max_iters=40, check_every=c,
                    tau=0.7) for c in (2, 20))
    assert torch.equal(a.u, b.u) and torch.equal(a.w, b.w) and torch.equal(a.phi, b.phi)


@pytest.mark.parametrize("n,k", [(352, 3), (330, 4), (256, 5), (200, 8), (400, 1)])
def test_auto_keeps_the_resident_results(n, k):
    """Where AUTO leaves the resident engine for the marching form, the iterates are the
    resident engine's bit for bit."""
    edges = S.complete_graph(k) if k > 1 else []
    r0, r1 = _fields(n, k, n)
    kw = dict(max_iters=47, check_every=20, tau=0.7)
    a = V.solve(_t(r0), _t(r1), edges, 0.6, **kw)
    b = V.solve(_t(r0), _t(r1), edges, 0.6, engine="resident", **kw)
    assert a.result["engine"] == "stream" and b.result["engine"] == "resident"
    assert torch.equal(a.u, b.u) and torch.equal(a.w, b.w) and torch.equal(a.phi, b.phi)


def test_marching_keeps_the_one_iteration_results():
    """check_every = 2 takes the one-iteration kernels, 20 the marching form: the same
    iterates bit for bit, for every norm pair and with eps (three channels)."""
    n, k = 75, 3
    r0, r1 = _fields(n, k, 4)
    for un, wn, eps in ((0, 0, 0.0), (1, 1, 0.0), (2, 0, 0.0), (0, 1, 0.4)):
        a, b = (V.solve(_t(r0), _t(r1), S.COMPLETE_K3, 0.6, engine="stream", max_iters=40, check_every=c, tau=0.7,
                        u_norm=un, w_norm=wn, eps=eps) for c in (2, 20))
        assert torch.equal(a.u, b.u) and torch.equal(a.w, b.w) and torch.equal(a.phi, b.phi)
