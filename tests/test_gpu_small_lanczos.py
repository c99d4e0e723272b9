"""Quadratic forms of small graphs on a CTA per column (automatic schedule)
against the oracle: row counts around the kernel's 1024 threads, rows longer
than 64 (whole warps), weighted entries, more columns than SMs, breakdown, and
the alpha / beta of both routes.  Tolerances of the Lanczos tests: 1e-10 (FP64,
full reorthogonalisation), 1e-5 (FP32, none)."""
import numpy as np
import pytest

from oracle import density, estimators, rng
from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu


def _graphs():
    hub = graphs.from_edges(900, np.r_[np.arange(1, 900), np.arange(2, 900)], np.r_[np.zeros(899, int), np.arange(1, 899)],
                            "hub with a path")  # one row of 899 entries
    return [("ER3", graphs.erdos_renyi(40, 0.2, 3)), ("WS1023", graphs.watts_strogatz(1023, 6, 0.2, 1)),
            ("BA1025", graphs.barabasi_albert(1025, 4, 2)), ("hub900", hub)]


@pytest.mark.parametrize("name,g", _graphs())
@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("k", [1, 9, 160])
def test_small_route_matches_oracle(vctx, name, g, fp64, k):
    m = 18
    A, _ = density.density_matrix(g)
    X = rng.rademacher(11, g.n, 0, k)
    mat = vne.matrix_from_graph(vctx, g, fp64=fp64)
    try:
        psi, ab = vne.vne_quadform_batch(vctx, mat, X, m, want_alpha_beta=True)
        # an explicit schedule takes the multi-CTA kernels
        ref2, ab2 = vne.vne_quadform_batch(vctx, mat, X, m, opt=vne.options(panel=8), want_alpha_beta=True)
    finally:
        vne.vne_matrix_destroy(mat)
    tol = 1e-10 if fp64 else 1e-5
    ref = estimators.quadforms(A, X, m, reorth="full" if fp64 else "none")
    assert np.max(np.abs(psi - ref) / np.abs(ref)) <= tol
    assert np.max(np.abs(psi - ref2) / np.abs(ref2)) <= tol
    # the first steps' coefficients agree to the vectors' rounding
    assert np.max(np.abs(ab[:, :4] - ab2[:, :4])) <= (1e-12 if fp64 else 1e-4) * np.max(np.abs(ab2[:, :4]))


@pytest.mark.parametrize("fp64", [True, False])
def test_small_route_breakdown(vctx, fp64):
    g = graphs.complete(30)  # invariant after one step
    X = rng.rademacher(2, g.n, 0, 5)
    mat = vne.matrix_from_graph(vctx, g, fp64=fp64)
    try:
        psi, ab = vne.vne_quadform_batch(vctx, mat, X, 10, want_alpha_beta=True)
    finally:
        vne.vne_matrix_destroy(mat)
    c2 = np.sum((X - X.mean(0)) ** 2, axis=0)
    lam = 1.0 / 29
    assert np.max(np.abs(psi - c2 * -lam * np.log(lam)) / np.abs(psi)) <= (1e-10 if fp64 else 1e-5)
    if fp64:  # an FP32 beta of rounding size (6e-8 ||A||) lies above the breakdown threshold (1e-10 ||A||)
        assert np.all(ab[:, 10:] == 0.0)
