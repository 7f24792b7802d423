"""The envelope gradient's kernel against the same formula in exact and 64-bit arithmetic:
phi less its mean, and the sum of ||w||, over sizes and batches that take every number of
blocks per problem, row pitches, and values near the ends of FP32's range.

phi - mean is FP64's difference rounded to FP32, so it is within half a unit in the last place
(0.51 with the rounding of the mean and of the difference); sum ||w|| likewise.
"""
import ctypes
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")
N = V._native


def _backward(phi, w, w_norm, scale=None, pitch=0):
    """phi [B, k, n, pitch or n], w [B, l, n, ...]: (d_rho0, d_rho1, d_alpha)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B, k, n = phi.shape[:3]
    l = w.shape[1]
    p, x = torch.from_numpy(phi).cuda(), torch.from_numpy(w).cuda()
    g = None if scale is None else torch.full((B,), scale, device="cuda")
    d0, d1, da = torch.full_like(p, 7.0), torch.full_like(p, 7.0), torch.empty(B, device="cuda")
    ctx = N.context(0)
    N.check(N.load().vomt_backward(ctx, B, n, pitch, k, l, w_norm, p.data_ptr(), x.data_ptr() if l else None,
                                   None if g is None else g.data_ptr(), d0.data_ptr(), d1.data_ptr(), da.data_ptr(),
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), ctx)
    torch.cuda.synchronize()
    return tuple(t.cpu().numpy() for t in (d0, d1, da))


def _check(phi, w, w_norm, out, n):
    d0, d1, da = out
    for q in range(phi.shape[0]):
        x = phi[q, :, :, :n].astype(np.float64)
        mean = math.fsum(x.reshape(-1).tolist()) / x.size
        ref = x - mean
        got = d1[q, :, :, :n].astype(np.float64)
        ulp = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
        assert np.all(np.abs(got - ref) <= 0.51 * ulp + 2.0 ** -52 * abs(mean))
        assert np.array_equal(d0[q, :, :, :n], -d1[q, :, :, :n])
        v = w[q, :, :, :n].astype(np.float64)
        total = np.abs(v).sum() if w_norm == V.W_L1 else np.sqrt((v * v).sum(0)).sum()
        assert abs(float(da[q]) - total) <= 0.51 * float(np.spacing(np.float32(total)))


SHAPES = [(1, 2, 1), (1, 7, 3), (2, 33, 1), (3, 64, 2), (1, 75, 3), (1, 128, 3), (2, 181, 1), (1, 256, 5), (40, 129, 1),
          (64, 64, 3), (200, 60, 2), (500, 33, 1), (1500, 16, 1)]


@pytest.mark.parametrize("B,n,k", SHAPES)
@pytest.mark.parametrize("w_norm", [0, 1])
def test_centred_potential_and_dalpha(B, n, k, w_norm):
    rng = np.random.default_rng(B + n)
    l = k * (k - 1) // 2
    phi = (rng.normal(0, 1, (B, k, n, n)) + rng.choice([0.0, 3.0, -1000.0], (B, 1, 1, 1))).astype(np.float32)
    w = (rng.normal(0, 1, (B, l, n, n)) * (rng.random((B, l, n, n)) < 0.3)).astype(np.float32)
    _check(phi, w, w_norm, _backward(phi, w, w_norm), n)


@pytest.mark.parametrize("w_norm", [0, 1])
def test_row_pitch_leaves_the_padding(w_norm):
    rng = np.random.default_rng(5)
    phi = rng.normal(2, 1, (3, 2, 41, 48)).astype(np.float32)
    w = rng.normal(0, 1, (3, 1, 41, 48)).astype(np.float32)
    out = _backward(phi, w, w_norm, pitch=48)
    _check(phi, w, w_norm, out, 41)
    assert np.all(out[0][..., 41:] == 7.0) and np.all(out[1][..., 41:] == 7.0)


@pytest.mark.parametrize("B,n", [(1, 40), (1, 300), (400, 24)])
@pytest.mark.parametrize("exponent", [126, -140, -70])
@pytest.mark.parametrize("w_norm", [0, 1])
def test_values_near_the_ends_of_the_range(B, n, exponent, w_norm):
    """Sums and squares beyond FP32's range (or below it) do not show in the gradient."""
    rng = np.random.default_rng(6)
    f = 2.0 ** exponent
    phi = (rng.uniform(0.5, 1.0, (B, 3, n, n)) * f).astype(np.float32)
    w = (rng.uniform(-1.0, 1.0, (B, 3, n, n)) * f).astype(np.float32)
    d0, d1, da = _backward(phi, w, w_norm, scale=2.0 ** -30 if exponent > 0 else None)
    if exponent > 0:
        for q in range(B):
            x = phi[q].astype(np.float64)
            ref = (x - math.fsum(x.reshape(-1).tolist()) / x.size) * 2.0 ** -30
            assert np.all(np.abs(d1[q] - ref) <= 0.51 * np.spacing(np.abs(ref).astype(np.float32)) + 2.0 ** -82 * f)
            v = w[q].astype(np.float64)
            total = 2.0 ** -30 * (np.abs(v).sum() if w_norm == V.W_L1 else np.sqrt((v * v).sum(0)).sum())
            assert abs(float(da[q]) - total) <= 0.51 * float(np.spacing(np.float32(total)))
    else:
        _check(phi, w, w_norm, (d0, d1, da), n)


def test_non_finite_potentials_stay_visible():
    phi = np.ones((2, 1, 9, 9), np.float32)
    phi[1, 0, 3, 3] = np.nan
    d0, d1, _ = _backward(phi, np.zeros((2, 0, 9, 9), np.float32), 0)
    assert np.all(d1[0] == 0.0) and np.all(np.isnan(d1[1])) and np.all(np.isnan(d0[1]))
