"""Which kernels vne_quadform_batch takes for a small FP64 graph: a CTA per column
in one launch, or the multi-CTA kernels, whose launches grow with the steps.
Each is taken where it is the faster one, also with few steps."""
import numpy as np
import pytest

from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,m,small", [(12000, 8, 2, False), (12000, 1, 1, False), (8000, 33, 3, False),
                                         (8000, 8, 5, False), (700, 5, 20, True), (700, 8, 2, True),
                                         (3000, 64, 8, True), (3000, 150, 20, True)])
def test_route_of_small_fp64_graphs(vctx, n, k, m, small):
    g = graphs.watts_strogatz(n, 6, 0.1, 1)
    X = np.random.default_rng(2).standard_normal((n, k))
    mat = vne.matrix_from_graph(vctx, g, fp64=True)

    def launches(**kw):
        vne.vne_quadform_batch(vctx, mat, X, m, opt=vne.options(**kw))
        before = vne.vne_ctx_stats(vctx)[0]
        psi = vne.vne_quadform_batch(vctx, mat, X, m, opt=vne.options(**kw))
        return vne.vne_ctx_stats(vctx)[0] - before, psi

    try:
        auto, psi = launches()
        panels, ref = launches(panel=8)
    finally:
        vne.vne_matrix_destroy(mat)
    assert auto < panels if small else auto == panels
    assert np.max(np.abs(psi - ref) / np.abs(ref)) <= 1e-10
