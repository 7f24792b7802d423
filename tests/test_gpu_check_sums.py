"""The constraint residual of the streaming engine's checks: its per-point values cancel, so they
are formed to more than FP32 precision.  Densities are small whole numbers, so that
rho1 - rho0 and its squares are exact in FP32 and, with one channel, the reported relative
residual depends on nothing rounded to FP32: it equals 64-bit arithmetic on the returned flux to
the FP32 pairs' 2^-48 times the hundred additions of a thread, well within 1e-12.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")


@pytest.mark.parametrize("n", [3, 31, 61, 300, 700])
@pytest.mark.parametrize("u_norm", [V.U_L12, V.U_L2, V.U_L1])
@pytest.mark.parametrize("iters", [4, 60])
def test_relative_residual_is_that_of_the_returned_flux(n, u_norm, iters):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n)
    a = rng.integers(0, 64, (1, n, n)).astype(np.float32)
    b = rng.permutation(a.reshape(-1)).reshape(a.shape)
    sol = V.solve(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), [], 1.0, max_iters=iters, check_every=iters,
                  tau=0.05, u_norm=u_norm, engine="stream")
    assert V.last_form() == "march"
    u = sol.u.double().cpu().numpy()
    r = (b - a).astype(np.float64)
    ux, uy = u[0], u[1]
    dx, dy = ux.copy(), uy.copy()
    dx[:, :, 1:] -= ux[:, :, :-1]
    dy[:, 1:, :] -= uy[:, :-1, :]
    res = (n - 1.0) * (dx + dy) + r
    expected = np.sqrt((res * res).sum()) / np.sqrt((r * r).sum())
    assert np.abs(u).max() > 0
    assert sol.result["rel_res"] == pytest.approx(expected, rel=1e-12)
