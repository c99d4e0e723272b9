"""Captured step loops run their panels in two groups on parallel branches of
the graph: the quadratic forms equal those of direct launches bit for bit,
for even and odd numbers of panels, both precisions, with and without full
reorthogonalisation, and for a graph with long rows."""
import numpy as np
import pytest

from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp64,reorth,n,k", [(False, 0, 20011, 48), (False, 0, 33000, 32), (False, 1, 12000, 80),
                                             (True, 1, 9001, 40), (True, 0, 17000, 16)])
def test_branches_equal_direct_launches(vctx, fp64, reorth, n, k):
    g = graphs.barabasi_albert(n, 4, n)
    mat = vne.matrix_from_graph(vctx, g, fp64=fp64)
    try:
        ref = vne.vne_entropy_hutchinson(vctx, mat, k, 12, 3, opt=vne.options(reorth=reorth, graphs=0), want_psi=True)[2]
        c0 = vne.vne_ctx_graph_stats(vctx)[0]
        for _ in range(4):  # direct, then captured and replayed
            psi = vne.vne_entropy_hutchinson(vctx, mat, k, 12, 3, opt=vne.options(reorth=reorth), want_psi=True)[2]
            assert np.array_equal(psi, ref)
        assert vne.vne_ctx_graph_stats(vctx)[0] == c0 + 1
    finally:
        vne.vne_matrix_destroy(mat)
