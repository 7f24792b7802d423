"""The unrolled gradient's two forms (every iterate kept; checkpoints and recomputed segments)
against each other, bit for bit, and its reverse step against the FP64 oracle for every kind of
graph: one to eight channels, missing pairs, edges in any order and orientation, costs, both w
norms, at sides around the strips of 30 columns.

The oracle cases are chosen (on the CPU) so that no shrink argument comes within 5e-5 of its
threshold, relatively, while FP32 moves arguments by about 1e-6; the bars are then those of
test_gpu_grad.py away from kinks.
"""
import numpy as np
import pytest

import oracle
from paper_1712_10279_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")
A = pytest.importorskip("paper_1712_10279_gb300.autograd")

FORMS = {"kept": 1 << 30, "checkpoints": 0}


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


def _graph(k, kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "complete":
        e = S.complete_graph(k)
    elif kind == "path":
        e = [(a, a + 1) for a in range(k - 1)]
    else:
        e = [tuple(map(int, x)) for x in S.random_connected_graph(rng, k, 0.5)]
        e = [(b, a) if rng.random() < .5 else (a, b) for a, b in e]
        rng.shuffle(e)
        e = [tuple(map(int, x)) for x in e]
    return e, (rng.uniform(0.5, 2.0, len(e)) if kind != "path" and e else None)


def _pair(n, k, seed):
    return tuple((x * x[0].size).astype(np.float32) for x in S.blob_pair(n, k, seed=seed))


def _grad(form, r0, r1, edges, **kw):
    V.set_memory_limit(FORMS[form])
    out = A.unrolled_grad(_t(r0), _t(r1), edges, 0.3, **kw)
    assert V.last_form() == "unrolled " + form
    return out


@pytest.mark.parametrize("T,ckpt", [(1, 1), (1, 7), (2, 1), (20, 1), (20, 2), (20, 5), (20, 20), (20, 21), (20, 1000),
                                    (23, 5), (21, 20), (29, 7)])
@pytest.mark.parametrize("n,k", [(31, 1), (33, 3), (20, 6)])
def test_checkpoints_give_the_gradients_of_the_kept_iterates(n, k, T, ckpt):
    edges = _graph(k, "complete", 0)[0] if k > 1 else []
    r0, r1 = _pair(n, k, n)
    kw = dict(T=T, ckpt=ckpt, tau=0.7)
    a, b = (_grad(form, r0, r1, edges, **kw) for form in FORMS)
    assert a[0] == b[0] and a[3] == b[3]
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    assert T == 1 or float(a[2].abs().max()) > 0


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("n,k,kind,T,w_norm,seed", [
    (2, 1, "path", 5, 0, 0), (3, 2, "path", 7, 0, 0), (29, 1, "path", 12, 0, 0), (30, 2, "complete", 9, 0, 0),
    (31, 3, "path", 9, 0, 1), (31, 3, "turned", 9, 1, 1), (59, 3, "turned", 6, 0, 7), (60, 4, "path", 6, 1, 1),
    (61, 2, "path", 6, 1, 5), (30, 5, "turned", 6, 0, 1), (29, 5, "complete", 6, 1, 7), (31, 6, "path", 6, 0, 5),
    (29, 7, "turned", 5, 0, 3), (30, 8, "complete", 4, 0, 0), (33, 8, "turned", 4, 1, 0)])
def test_every_graph_matches_oracle(form, n, k, kind, T, w_norm, seed):
    edges, cost = _graph(k, kind, seed)
    r0, r1 = _pair(n, k, seed)
    J, d0, d1, da = _grad(form, r0, r1, edges, T=T, ckpt=4, tau=0.7, w_norm=w_norm, cost=cost)
    Jo, g1, g0, gao = oracle.unrolled_grad(r0.astype(np.float64), r1.astype(np.float64), edges, 0.3, T, tau=0.7,
                                           w_norm=w_norm, cost=cost)
    assert J == pytest.approx(Jo, rel=1e-5)
    assert _rel(d1.cpu().numpy().astype(np.float64), g1) < 1e-3
    assert _rel(d0.cpu().numpy().astype(np.float64), g0) < 1e-3
    assert da == pytest.approx(gao, rel=1e-3)


def test_the_limit_bounds_the_memory_and_lowering_it_gives_memory_back():
    """256^2, three channels, 100 iterations: 312 MB of iterates, or ten checkpoints and a
    segment of ten (66 MB) within any limit below that."""
    n, k, T = 256, 3, 100
    r0, r1 = _pair(n, k, 1)
    d0, d1 = _t(r0), _t(r1)
    V.set_memory_limit(0)
    torch.cuda.synchronize()

    def used(limit):
        V.set_memory_limit(limit)
        before = torch.cuda.mem_get_info()[0]
        A.unrolled_grad(d0, d1, S.COMPLETE_K3, 0.3, T=T, ckpt=10, tau=100.0)
        torch.cuda.synchronize()
        return before - torch.cuda.mem_get_info()[0], V.last_form()

    A.unrolled_grad(d0, d1, S.COMPLETE_K3, 0.3, T=1, ckpt=1, tau=100.0)       # what every call allocates
    small, form = used(100 << 20)
    assert form == "unrolled checkpoints" and small < 100 << 20
    large, form = used(1 << 30)
    assert form == "unrolled kept" and large > 150 << 20
    free = torch.cuda.mem_get_info()[0]
    V.set_memory_limit(100 << 20)
    assert torch.cuda.mem_get_info()[0] - free > 150 << 20
