"""AUTO's choice between the resident engine and the marching form: it depends on how many
iterations a check serves, and both return the same iterates."""
import numpy as np
import pytest

from paper_1712_10279_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")


@pytest.mark.parametrize("n,k,below,at", [
    (400, 1, 19, 20), (470, 1, 49, 50), (500, 1, 7, 8), (352, 2, 19, 20), (500, 2, 7, 8),
    (336, 3, 99, 100), (352, 3, 7, 8), (362, 3, 3, 4), (336, 4, 15, 16), (352, 4, 3, 4),
    (240, 5, 100, None), (256, 5, 19, 20), (280, 5, 11, 12), (300, 5, None, 1), (200, 6, 49, 50), (256, 6, 7, 8),
    (280, 6, 3, 4), (230, 7, 100, None), (256, 7, None, 1), (161, 8, None, 1), (160, 8, 100, None),
])
def test_auto_marches_from_the_interval_at_which_it_is_faster(n, k, below, at):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    edges = S.complete_graph(k) if k > 1 else []
    r0, r1 = (torch.from_numpy(x.astype(np.float32)).cuda() for x in S.blob_pair(n, k, seed=n))
    for check, form in ((below, "resident"), (at, "march")):
        if check is None:
            continue
        kw = dict(max_iters=100, check_every=check, tau=0.003 * k * n * n)
        a = V.solve(r0, r1, edges, 0.3, **kw)
        assert V.last_form() == form
        assert a.result["engine"] == ("stream" if form == "march" else "resident")
        b = V.solve(r0, r1, edges, 0.3, engine="resident" if form == "march" else "stream", **kw)
        if form == "march":
            assert torch.equal(a.u, b.u) and torch.equal(a.w, b.w) and torch.equal(a.phi, b.phi)
        assert a.result["iters"] == b.result["iters"] == 100
