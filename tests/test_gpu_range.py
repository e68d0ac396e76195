"""Vectors whose squared length leaves the normal range: matrices far from 1 in size, and graded
ones, keep their singular values (absolute error relative to sigma_1, as everywhere)."""
import numpy as np
import pytest

from _util import err_rel, to_device_colmajor, tol_for

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nla():
    from paper_2608_21227_gb300 import nla as _nla

    _nla.lib()
    return _nla


def _values(A):
    """Singular values by LAPACK on the matrix brought to size 1 by an exact power of two."""
    e = int(np.floor(np.log2(np.abs(A).max())))
    return np.linalg.svd(np.ldexp(A, -e), compute_uv=False), e


def _check(S, info, A, tol):
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    ref, e = _values(A)
    assert err_rel(np.ldexp(S.double().cpu().numpy(), -e), ref) <= tol


def _graded(n, low, rows, seed):
    """n x n Gaussian whose columns (or rows) fall from 1 to 10^low."""
    A = np.random.default_rng(seed).standard_normal((n, n))
    f = 10.0 ** np.linspace(0.0, low, n)
    return A * (f[:, None] if rows else f[None, :])


# 2^-518 = 1.2e-156: squares are subnormal (about 2^-1030, 44 bits left of 52: norms to 2e-13);
# 2^505: squares are the largest that stay finite
@pytest.mark.parametrize("scale", [-518, 505])
@pytest.mark.parametrize("b", [8, 16, 32, 64])
def test_fp64_far_from_one(nla, scale, b):
    A = np.ldexp(np.random.default_rng(b).standard_normal((120, 100)), scale)
    S, info = nla.gesvd_vals(to_device_colmajor(A, torch.float64), cfg=nla.Cfg.make(band=b))
    _check(S, info, A, tol_for(0, 120))


@pytest.mark.parametrize("b", [8, 16, 32, 64])
@pytest.mark.parametrize("rows", [False, True])
@pytest.mark.parametrize("low", [-170.0, -200.0, -300.0])
def test_fp64_graded(nla, b, rows, low):
    A = _graded(150, low, rows, b)
    S, info = nla.gesvd_vals(to_device_colmajor(A, torch.float64), cfg=nla.Cfg.make(band=b))
    _check(S, info, A, tol_for(0, 150))


@pytest.mark.parametrize("update,u", [(1, 2.0 ** -11), (2, 2.0 ** -8), (3, 2.0 ** -20), (4, 2.0 ** -15)])
def test_mixed_graded(nla, update, u):
    # the first-order model of the mixed update, 10 u sqrt(n / b)
    A = _graded(150, -200.0, False, update)
    S, info = nla.gesvd_vals(to_device_colmajor(A, torch.float64), update=update, cfg=nla.Cfg.make(band=16))
    _check(S, info, A, 10.0 * u * np.sqrt(150 / 16))


@pytest.mark.parametrize("b", [8, 16, 32, 64])
@pytest.mark.parametrize("low", [-160.0, -250.0])
def test_band_fp64_graded(nla, b, low):
    # the chase alone: a block of tiny rows inside a band of size 1, rows that decay, all tiny
    n = 200
    i, j = np.indices((n, n))
    D = np.where((j - i >= 0) & (j - i <= b), np.random.default_rng(b).standard_normal((n, n)), 0.0)
    tiny = D.copy()
    tiny[60:90] *= 10.0 ** low
    graded = D * (10.0 ** np.linspace(0.0, low, n))[:, None]
    for M in (tiny, graded, D * 10.0 ** low):
        ABt = nla.band_extract(to_device_colmajor(M, torch.float64), b)
        d, e, info = nla.band2bd(ABt, b)
        S, info2 = nla.bdsvd_vals(d, e)
        assert int(info2.item()) == 0
        _check(S, info, M, tol_for(0, n))


@pytest.mark.parametrize("dt,tiny,big,medium", [(0, 4e-156, 8e153, 1e100)])
@pytest.mark.parametrize("m,band", [(40, 16), (40, 32), (3000, 16), (3000, 32)])
def test_panel_quotient_of_column_sizes_overflows(nla, dt, tiny, big, medium, m, band):
    # columns 0 and 1: one entry of size tiny, two of size big, whose quotient overflows while no square does
    n = 40
    A = np.random.default_rng(m).standard_normal((m, n)) * medium
    A[:, :2] = 0.0
    A[1, 0] = tiny
    A[0, 1] = A[1, 1] = big
    t = to_device_colmajor(A, torch.float32 if dt else torch.float64)
    A = t.double().cpu().numpy().T
    _, _, info = nla.gebrd_band(t, band)
    D = np.triu(t.double().cpu().numpy().T[:n, :n])
    D = np.where(np.subtract.outer(np.arange(n), np.arange(n)) >= -band, D, 0.0)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    s1 = np.hypot(big, big)
    ref = np.linalg.svd(A / s1, compute_uv=False)
    assert err_rel(np.linalg.svd(D / s1, compute_uv=False), ref) <= tol_for(dt, m)


@pytest.mark.parametrize("b", [8, 16, 32, 64])
def test_band_quotient_overflows(nla, b):
    # rows of size 1e-156 beside rows of size 1e152
    n = 150
    i, j = np.indices((n, n))
    D = np.where((j - i >= 0) & (j - i <= b), np.random.default_rng(b).uniform(0.5, 1.0, (n, n)), 0.0)
    D *= np.where(np.arange(n) % 3 == 0, 2e-156, 4e153 / (2 * b))[:, None]
    d, e, info = nla.band2bd(nla.band_extract(to_device_colmajor(D, torch.float64), b), b)
    S, info2 = nla.bdsvd_vals(d, e)
    torch.cuda.synchronize()
    assert int(info2.item()) == 0
    _check(S, info, D, tol_for(0, n))


@pytest.mark.parametrize("dt", [0, 1])
def test_band_zero_blocks(nla, dt):
    # zero vectors take no reflector: diagonal parts, zero rows and columns
    n, b = 200, 16
    i, j = np.indices((n, n))
    D = np.where((j - i >= 0) & (j - i <= b), np.random.default_rng(7).standard_normal((n, n)), 0.0)
    D[50:90][:, 50:] = np.where(np.eye(n)[50:90][:, 50:] > 0, D[50:90][:, 50:], 0.0)
    D[120:140] = 0.0
    D[:, 160:180] = 0.0
    tdt = torch.float32 if dt else torch.float64
    d, e, info = nla.band2bd(nla.band_extract(to_device_colmajor(D, tdt), b), b)
    S, _ = nla.bdsvd_vals(d, e, dtype=tdt)
    _check(S, info, D, tol_for(dt, n))
