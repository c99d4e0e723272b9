"""The spectral kernels at the edges of their size classes (32, 64, 128) and
of their thread mapping (four lanes per eigenvalue, two per eigenvector): the
quadrature against a dense eigendecomposition, and the bounds of Theorem 4.4
against the oracle's evaluation of the same g_m."""
import numpy as np
import pytest

from oracle import bounds
from paper_2212_09642_gb300 import vne

pytestmark = pytest.mark.gpu


def _tridiagonals(m, count, seed):
    """Positive definite, well separated: diagonally dominant with a graded diagonal."""
    rng = np.random.default_rng(seed)
    a = 1.0 + np.arange(m)[None, :] / m + 0.3 * rng.random((count, m))
    b = 0.05 + 0.2 * rng.random((count, m))
    return a, b


@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128])
def test_quadrature_at_size_classes(vctx, m):
    a, b = _tridiagonals(m, 5, 10 + m)
    norm2 = 1.0 + np.arange(5.0)
    got = vne.vne_tridiag_quadrature(vctx, a, b, norm2, 0.01)
    for i in range(5):
        T = np.diag(a[i]) + np.diag(b[i, :m - 1], 1) + np.diag(b[i, :m - 1], -1)
        th, U = np.linalg.eigh(T)
        x = 0.01 * th
        ref = norm2[i] * np.sum(U[0] ** 2 * np.where(x > 0, -x * np.log(np.maximum(x, 1e-300)), 0.0))
        assert abs(got[i] - ref) <= 1e-12 * abs(ref)


@pytest.mark.parametrize("m", [1, 3, 8, 9, 12])
@pytest.mark.parametrize("grid", [1, 16, 257])
def test_bounds_at_thread_mapping_edges(vctx, m, grid):
    a, b = _tridiagonals(m, 3, 40 + m)
    lam = 0.2, 3.0
    lo, hi, est = vne.vne_quadrature_bounds(vctx, a, b, np.ones(3), 1.0, lam[0], lam[1], grid)
    for i in range(3):
        rlo, rhi, rest = bounds.posterior_bounds(a[i], b[i], 1.0, lam[0], lam[1], grid=grid)
        # terms of g_m cancel as m grows: two correct evaluations agree to 1e-6 of the maximum
        assert abs(hi[i] - rhi) <= 1e-6 * rhi and abs(lo[i] - rlo) <= 1e-6 * rhi
        assert abs(est[i] - np.sqrt(lo[i] * hi[i])) <= 1e-12 * est[i]
