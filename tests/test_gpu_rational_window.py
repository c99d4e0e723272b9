"""Multi-shift CG with the shifted iterates formed from windows of residuals:
row counts around the flush kernel's 1024-row CTAs, every panel width, one to
eight shifts (more than four take a second group) and solves of one partial
window up to many, against the oracle's direct solves.  Tolerances of the
rational tests: 1e-10 relative (FP64, CG to 1e-13), 1e-5 (FP32, CG to 1e-8)."""
import numpy as np
import pytest

from oracle import density, rational, rng
from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp64,panel", [(True, 4), (True, 8), (True, 16), (False, 8), (False, 16), (False, 32)])
@pytest.mark.parametrize("n,shifts,k", [(1023, 1, 3), (1024, 4, 9), (1025, 5, 17), (2049, 8, 5)])
def test_windowed_shifts(vctx, fp64, panel, n, shifts, k):
    g = graphs.watts_strogatz(n, 6, 0.2, n)
    A, _ = density.density_matrix(g)
    sh = rational.default_shifts(A)[:shifts]
    X = rng.rademacher(5, g.n, 0, k)
    mat = vne.matrix_from_graph(vctx, g, fp64=fp64)
    tol_cg = 1e-13 if fp64 else 1e-8
    try:
        psi, its, res = vne.vne_quadform_rational(vctx, mat, X, sh, opt=vne.options(cg_tol=tol_cg, panel=panel))
    finally:
        vne.vne_matrix_destroy(mat)
    ref = np.array([rational.rational_quadform(A, X[:, j], sh) for j in range(k)])
    assert np.max(np.abs(psi - ref) / np.abs(ref)) <= (1e-10 if fp64 else 1e-5)
    assert np.all(res <= tol_cg * 1.0000001)


@pytest.mark.parametrize("n", [303 * 1024 + 1, 305 * 1024])
def test_update_over_several_tiles(vctx, n):
    """FP32 blocks of many row tiles take three of them per CTA of the update
    (64 columns of 304 or 305 tiles, one or two tiles in the last CTA); eight of
    the columns alone take one.  Each is within 1e-5 of the exact value."""
    g = graphs.watts_strogatz(n, 6, 0.2, 3)
    sh = np.array([1e-6, 1e-5])
    X = rng.rademacher(5, g.n, 0, 64)
    mat = vne.matrix_from_graph(vctx, g, fp64=False)
    opt = vne.options(cg_tol=1e-8, panel=8)
    try:
        psi, its, res = vne.vne_quadform_rational(vctx, mat, X, sh, opt=opt)
        alone, _, _ = vne.vne_quadform_rational(vctx, mat, X[:, 24:32], sh, opt=opt)
    finally:
        vne.vne_matrix_destroy(mat)
    assert np.all(res <= 1e-8 * 1.0000001)
    assert np.max(np.abs(psi[24:32] - alone) / np.abs(alone)) <= 2e-5
