"""FP32 reorthogonalisation whose inner products take four row tiles per CTA (from
2048 tiles times basis vectors on): one to four tiles in the last group, full and
partial policy, against FP64 vectors; and a range of the columns gives the
bits of the whole."""
import numpy as np
import pytest

from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reorth", [1, 2])
@pytest.mark.parametrize("n", [256 * 1024 + 1, 258 * 1024, 259 * 1024 - 5, 260 * 1024])
def test_groups_of_row_tiles(vctx, n, reorth):
    """256 to 260 tiles: groups from the eighth basis vector on, 24 steps."""
    g = graphs.barabasi_albert(n, 4, 6)
    out = []
    for fp64 in (False, True):
        mat = vne.matrix_from_graph(vctx, g, fp64=fp64)
        try:
            opt = vne.options(reorth=reorth if not fp64 else 1)
            out.append(vne.vne_entropy_hutchinson(vctx, mat, 20, 24, 3, opt=opt, want_psi=True)[2])
            if not fp64:
                part = vne.vne_entropy_hutchinson(vctx, mat, 8, 24, 3, opt=opt, want_psi=True)[2]
                assert np.array_equal(part, out[0][:8])
        finally:
            vne.vne_matrix_destroy(mat)
    assert np.max(np.abs(out[0] - out[1]) / np.abs(out[1])) <= 1e-5
