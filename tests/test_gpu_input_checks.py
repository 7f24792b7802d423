"""The density checks of every entry point: masses beyond FP32's range, values of very
different size, and mismatches on either side of the 1e-6 bound.

The totals are compared in FP64 from sums no less accurate than FP64's, so a mismatch 1e-12 of
the total away from the bound is decided right.
"""
import numpy as np
import pytest

from paper_1712_10279_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
V = pytest.importorskip("paper_1712_10279_gb300")


def _t(x):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _call(kind, r0, r1):
    """One iteration-free solve with densities r0, r1 [2, n, n] through an entry point."""
    edges, kw = [(0, 1)], dict(tau=1.0, max_iters=0)
    n = r0.shape[-1]
    if kind == "solve":
        V.solve(_t(r0), _t(r1), edges, 1.0, **kw)
    elif kind == "batch":
        ok = np.ones((2, 5, 5), np.float32)
        V.Batch([dict(n=5, k=2, edges=edges), dict(n=n, k=2, edges=edges), dict(n=5, k=2, edges=edges)],
                [_t(ok), _t(r0), _t(ok)], [_t(ok), _t(r1), _t(ok)]).solve(max_iters=0, tau=1.0)
    elif kind == "volume":
        m = round((n * n) ** (1 / 3))
        assert m ** 3 == n * n
        V.solve3d(_t(r0.reshape(2, m, m, m)), _t(r1.reshape(2, m, m, m)), edges, 1.0, **kw)
    else:
        z = np.zeros((n, n), np.float32)
        full = [np.stack([r[0], z, z, r[1]]) for r in (r0, r1)]
        if kind == "matrix":
            V.momt_solve(_t(full[0]), _t(full[1]), S.random_L(2, 2, seed=1), 1.0, **kw)
        else:
            V.momt_solve_complex(*(_t(x.astype(np.complex64)) for x in full), S.random_hermitian_L(2, 2, seed=1), 1.0,
                                 **kw)


KINDS = ["solve", "batch", "volume", "matrix", "complex"]


def _status(kind, r0, r1):
    try:
        _call(kind, r0.astype(np.float32), r1.astype(np.float32))
    except V.VomtError as e:
        return e.status
    return 0


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 105, 2.0 ** -120])
def test_equal_masses_pass_and_unequal_ones_do_not(kind, scale):
    """scale 2^105: 1458 cells of up to 2^20 sum to more than FP32 holds (and the check of the
    iterate, which squares their differences, then reports a non-finite value)."""
    rng = np.random.default_rng(3)
    a = rng.integers(1, 1 << 20, (2, 27, 27)).astype(np.float64)
    b = rng.permutation(a.reshape(-1)).reshape(a.shape)
    accepted = (0, -7) if scale > 1.0 else (0,)

    def shift(by):                       # b with its total larger by `by`, every entry below 2^24
        c = b.copy().reshape(-1)
        each, rest = divmod(by, c.size)
        c += each
        c[:rest] += 1
        return c.reshape(b.shape)

    assert _status(kind, a * scale, a * scale) == 0
    assert _status(kind, a * scale, b * scale) in accepted
    # |difference| against 1e-6 of the larger total: the last whole number below it and the next
    by = int(np.floor(1e-6 * a.sum() / (1.0 - 1e-6)))
    assert _status(kind, a * scale, shift(by) * scale) in accepted
    assert _status(kind, a * scale, shift(by + 1) * scale) == -2
    assert _status(kind, shift(by + 1) * scale, a * scale) == -2


@pytest.mark.parametrize("kind", KINDS)
def test_one_large_cell_does_not_hide_the_others(kind):
    """A cell of 2^60 beside many of about one: the totals differ by 1e-6 of the sum only if the
    large cells do, and a single negative or NaN cell is found wherever it is."""
    rng = np.random.default_rng(4)
    a = rng.uniform(0.5, 1.0, (2, 27, 27)).astype(np.float32)
    b = rng.uniform(0.5, 1.0, (2, 27, 27)).astype(np.float32)
    a[0, 3, 5] = b[1, 20, 7] = 2.0 ** 60
    _call(kind, a, b)
    for at in ((0, 0, 0), (1, 26, 26), (0, 13, 7)):
        for value, status in ((-1.0, -3), (np.nan, -7), (np.inf, -7)):
            for bad in (0, 1):
                pair = [a.copy(), b.copy()]
                pair[bad][at] = value
                with pytest.raises(V.VomtError) as e:
                    _call(kind, *pair)
                assert e.value.status == status
