"""The marching kernels of every channel count, norm pair and order of operations against the
FP64 oracle, each test asserting that the marching form is what ran: edges listed in the order
of their pairs (either orientation, some pairs without an edge) take it, others keep the
kernels that sum as listed.

Tolerances are those of test_gpu_march.py: tens of iterations, each rounding every field a few
times in FP32 (6e-8), leave well under 1e-4 of a field's norm; w is zero except where a
threshold is passed, so its error is bounded against the threshold it cancels with: 1e-3.
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


def _graph(rng, k):
    """A connected graph's edges in the order of their pairs, turned at random, and costs."""
    edges = sorted(tuple(sorted(int(a) for a in e)) for e in S.random_connected_graph(rng, k, 0.5))
    return ([(b, a) if rng.random() < 0.5 else (a, b) for a, b in edges],
            rng.uniform(0.5, 2.0, len(edges)) if edges else None)


def _check(sol, ref):
    u = sol.u.cpu().numpy().astype(np.float64)
    assert _rel(u, np.stack([ref["ux"], ref["uy"]])) < 1e-4
    assert _rel(sol.phi.cpu().numpy().astype(np.float64), ref["phi"]) < 1e-4
    if ref["w"].size:
        assert u.shape[-1] < 23 or np.abs(ref["w"]).max() > 0
        assert _rel(sol.w.cpu().numpy().astype(np.float64), ref["w"]) < 1e-3
    assert abs(sol.result["primal"] - ref["metrics"]["primal"]) <= 1e-4 * abs(ref["metrics"]["primal"])
    assert np.all(u[0, :, :, -1] == 0) and np.all(u[1, :, -1, :] == 0)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n", [2, 3, 23, 25, 28, 31, 32, 33, 48, 61, 97])
def test_sizes_and_passes_match_oracle(n, k):
    edges, cost = _graph(np.random.default_rng(100 * n + k), k)
    r0, r1 = _fields(n, k, n + 7 * k)
    kw = dict(max_iters=24, check_every=11, tau=0.7, cost=cost)      # passes of 1, 2 and 4 iterations
    sol = V.solve(_t(r0), _t(r1), edges, 0.6, engine="stream", **kw)
    assert V.last_form() == "march"
    ref = oracle.vomt_solve(r0.astype(np.float64), r1.astype(np.float64), edges, 0.6, history=True, **kw)
    _check(sol, ref)
    h = V.history()
    np.testing.assert_allclose(h[:, 6], ref["history"][:, 6])
    np.testing.assert_allclose(h[:, 0], ref["history"][:, 0], rtol=1e-4)
    np.testing.assert_allclose(h[:, 3], ref["history"][:, 3], rtol=1e-3)


@pytest.mark.parametrize("k", [1, 2, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("u_norm,w_norm", [(0, 0), (1, 0), (2, 0), (0, 1), (1, 1), (2, 1)])
@pytest.mark.parametrize("eps", [0.0, 0.3])
def test_norms_and_regularisation_match_oracle(u_norm, w_norm, eps, k):
    n = {1: 53, 2: 47, 4: 45, 5: 43, 6: 41, 7: 39, 8: 37}[k]
    if k == 1 and w_norm:
        pytest.skip("no edges at k = 1")
    edges, cost = _graph(np.random.default_rng(k), k)
    r0, r1 = _fields(n, k, 5)
    kw = dict(max_iters=20, check_every=10, tau=0.7, u_norm=u_norm, w_norm=w_norm, eps=eps, cost=cost)
    sol = V.solve(_t(r0), _t(r1), edges, 0.6, engine="stream", **kw)
    assert V.last_form() == "march"
    _check(sol, oracle.vomt_solve(r0.astype(np.float64), r1.astype(np.float64), edges, 0.6, **kw))


@pytest.mark.parametrize("u_norm,w_norm", [(0, 0), (1, 1), (2, 0)])
def test_three_channels_with_a_missing_pair(u_norm, w_norm):
    r0, r1 = _fields(53, 3, 5)
    kw = dict(max_iters=20, check_every=10, tau=0.7, u_norm=u_norm, w_norm=w_norm, cost=[0.7, 1.9])
    for edges in ([(0, 1), (1, 2)], [(2, 0), (1, 2)], [(0, 1), (2, 0)]):
        sol = V.solve(_t(r0), _t(r1), edges, 0.6, engine="stream", **kw)
        assert V.last_form() == "march"
        _check(sol, oracle.vomt_solve(r0.astype(np.float64), r1.astype(np.float64), edges, 0.6, **kw))


@pytest.mark.parametrize("k", [3, 5, 8])
def test_edges_out_of_order_run_the_one_iteration_kernels(k):
    edges, cost = _graph(np.random.default_rng(k), k)
    edges, cost = edges[::-1], cost[::-1]
    r0, r1 = _fields(33, k, 5)
    kw = dict(max_iters=20, check_every=10, tau=0.7, cost=cost)
    sol = V.solve(_t(r0), _t(r1), edges, 0.6, engine="stream", **kw)
    assert V.last_form() == "step"
    _check(sol, oracle.vomt_solve(r0.astype(np.float64), r1.astype(np.float64), edges, 0.6, **kw))


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8])
def test_auto_marches_with_the_resident_results(k):
    """Past the sizes that the resident engine is good at, AUTO's marching form (in the resident
    engine's order of operations) returns that engine's iterates bit for bit, with costs and
    missing pairs too."""
    n = {1: 400, 2: 352, 3: 340, 4: 322, 5: 260, 6: 256, 7: 256, 8: 200}[k]
    edges, cost = _graph(np.random.default_rng(k + 40), k)
    r0, r1 = _fields(n, k, n)
    kw = dict(max_iters=47, check_every=20, tau=0.7, cost=cost)
    a = V.solve(_t(r0), _t(r1), edges, 0.6, **kw)
    assert V.last_form() == "march"
    b = V.solve(_t(r0), _t(r1), edges, 0.6, engine="resident", **kw)
    assert V.last_form() == "resident"
    assert torch.equal(a.u, b.u) and torch.equal(a.w, b.w) and torch.equal(a.phi, b.phi)
