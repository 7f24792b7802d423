"""The batch tuner and the marching form: what was timed faster for a batch runs for batches of
its shapes, and other batches keep their choice by estimate."""
import numpy as np
import pytest

from paper_1712_10279_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")


def _batch(shapes, seed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    probs, r0, r1 = [], [], []
    for q, (n, k) in enumerate(shapes):
        a, b = S.blob_pair(n, k, seed=seed + q)
        probs.append(dict(n=n, k=k, edges=S.complete_graph(k) if k > 1 else [], alpha=0.3, tau=0.003 * k * n * n))
        r0.append(a.astype(np.float32))
        r1.append(b.astype(np.float32))
    return V.Batch(probs, r0, r1)


def test_a_tuned_batch_takes_the_form_timed_fastest():
    """32 problems of 64^2 and 128^2 with five channels: the marching form takes a third of the
    grouped path's time.  With a check every 3 iterations it does not apply, and a batch of other
    shapes is not held to its timing."""
    kw = dict(max_iters=40, check_every=20)
    shapes = [(64, 5), (128, 5)] * 16
    batch, other = _batch(shapes, 1), _batch([(256, 3)] * 6, 2)
    other.solve(**kw)
    before = V.last_form()
    best, times = batch.tune(sample_iters=40)
    assert best in (128, 256, 512) and all(t > 0 for t in times.values())
    batch.solve(**kw)
    assert V.last_form() == "batch march"
    grouped = _batch(shapes, 1)
    grouped.solve(path="grouped", **kw)
    assert V.last_form() == "batch grouped" and torch.equal(batch.arena, grouped.arena)
    batch.solve(max_iters=40, check_every=3)
    assert V.last_form() in ("batch grouped", "batch queue")
    other.solve(**kw)
    assert V.last_form() in (before, "batch queue")
    queue = _batch(shapes, 1)
    queue.solve(path="queue", **kw)
    assert V.last_form() == "batch queue"


def test_a_batch_that_the_marching_form_does_not_take_can_be_tuned():
    """Six channels (no grouped kernel) and edges out of pair order."""
    six = _batch([(20, 6), (33, 2)], 3)
    six.tune(sample_iters=20)
    six.solve(max_iters=20, check_every=20)
    assert V.last_form() == "batch queue"
    turned = _batch([(64, 3)] * 8, 4)
    probs = [dict(p, edges=p["edges"][::-1]) for p in turned.problems]
    turned = V.Batch(probs, [S.blob_pair(64, 3, seed=q)[0] for q in range(8)], [S.blob_pair(64, 3, seed=q)[1] for q in range(8)])
    turned.tune(sample_iters=20)
    turned.solve(max_iters=20, check_every=20)
    assert V.last_form() in ("batch grouped", "batch queue")
