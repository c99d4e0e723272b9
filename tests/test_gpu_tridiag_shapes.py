"""The spectral kernels at the edges of their size classes (32, 64, 128) and
of their thread mapping (four lanes per eigenvalue, two per eigenvector): the
quadrature against a dense eigendecomposition."""
import numpy as np
import pytest

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
