"""Bounds of Theorem 4.4 at the edges of the kernel's thread mapping (four lanes
per Ritz value, single points, points beyond one pass of the CTA) against the
oracle's evaluation of the same g_m.  Tolerances of the bounds tests: 1e-6 of
the maximum (the terms of g_m cancel as m grows), and 1e-12 of the quadrature,
below which both sides are rounding."""
import numpy as np
import pytest

from oracle import bounds, krylov
from paper_2212_09642_gb300 import vne

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 3, 8, 9, 12])
@pytest.mark.parametrize("grid", [1, 16, 257])
def test_bounds_at_thread_mapping_edges(vctx, m, grid):
    r = np.random.default_rng(40 + m)
    a = 1.0 + np.arange(m)[None, :] / m + 0.3 * r.random((3, m))  # positive definite, well separated
    b = 0.05 + 0.2 * r.random((3, m))
    lam = 0.2, 3.0
    lo, hi, est = vne.vne_quadrature_bounds(vctx, a, b, np.ones(3), 1.0, lam[0], lam[1], grid)
    for i in range(3):
        rlo, rhi, _ = bounds.posterior_bounds(a[i], b[i], 1.0, lam[0], lam[1], grid=grid)
        floor = 1e-12 * abs(krylov.gauss_quadrature(a[i], b[i, :-1], 1.0))
        assert abs(hi[i] - rhi) <= 1e-6 * rhi + floor, (hi[i], rhi)
        assert abs(lo[i] - rlo) <= 1e-6 * rhi + floor, (lo[i], rlo)
        assert abs(est[i] - np.sqrt(lo[i] * hi[i])) <= 1e-12 * est[i]
