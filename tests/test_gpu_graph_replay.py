"""Captured step loops and what their launches depend on beside sizes and
buffers: the breakdown threshold and the norm of the matrix.  A call that
replays a graph equals direct launches bit for bit after the threshold changed
or after a matrix took the place of another of the same shape (whose buffers
usually come back at the same addresses), and a captured batch on two branches
equals direct launches."""
import numpy as np
import pytest

from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu


def _psi(ctx, mat, graphs_on, **kw):
    opt = vne.options(graphs=graphs_on, **kw)
    return vne.vne_entropy_hutchinson(ctx, mat, 24, 12, 3, opt=opt, want_psi=True)[2]


@pytest.mark.parametrize("first", [0.0, 0.2])
def test_changed_breakdown_tol(first):
    """tol = 0.2 is above every beta_j / ||A||_G of this graph (columns end after
    one step), the default below all of them."""
    g = graphs.erdos_renyi(3000, 8.0 / 2999, 5)
    ctx = vne.vne_ctx_create(0)
    try:
        mat = vne.matrix_from_graph(ctx, g, fp64=True)
        ref = {tol: _psi(ctx, mat, 0, breakdown_tol=tol) for tol in (0.0, 0.2)}
        assert np.all(np.abs(ref[0.2] - ref[0.0]) > 1e-3 * np.abs(ref[0.0]))
        for tol in (first, 0.2 - first, first):
            for _ in range(4):  # direct, then captured and replayed
                assert np.array_equal(_psi(ctx, mat, -1, breakdown_tol=tol), ref[tol]), tol
        assert vne.vne_ctx_graph_stats(ctx)[1] >= 3
        vne.vne_matrix_destroy(mat)
    finally:
        vne.vne_ctx_destroy(ctx)


@pytest.mark.parametrize("reorth", [1, 2])
def test_matrix_replaced_by_one_of_another_scale(reorth):
    """A weighted Laplacian and the same with its entries scaled by 2^-44, made one
    after the other in the same place: the threshold (reorth 1) and the norm in
    the estimate of the loss of orthogonality (reorth 2) are each matrix's own."""
    g = graphs.watts_strogatz(3000, 6, 0.2, 7)
    rows = np.repeat(np.arange(g.n), np.diff(g.rowptr))
    col = np.asarray(g.col, dtype=np.int64)
    w = 0.5 + ((rows + col) % 97) / 97.0
    r = np.concatenate([rows, np.arange(g.n)])
    c = np.concatenate([col, np.arange(g.n)])
    v = np.concatenate([-w, np.bincount(rows, weights=w, minlength=g.n)])
    order = np.lexsort((c, r))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=g.n))])
    flags = vne.VNE_FP64 | vne.VNE_NORMALIZE_TRACE | vne.VNE_IS_LAPLACIAN
    ctx = vne.vne_ctx_create(0)
    try:
        for scale in (1.0, 2.0 ** -44, 1.0):
            mat = vne.vne_create_density_matrix(ctx, g.n, rowptr, c[order], scale * v[order], flags)
            got = [_psi(ctx, mat, -1, reorth=reorth) for _ in range(4)]
            ref = _psi(ctx, mat, 0, reorth=reorth)
            for x in got:
                assert np.array_equal(x, ref), scale
            vne.vne_matrix_destroy(mat)
        assert vne.vne_ctx_graph_stats(ctx)[1] >= 3
    finally:
        vne.vne_ctx_destroy(ctx)


def test_captured_batch_on_two_branches():
    """Three graphs of 39,000 rows in all and five panels (above the 2 MB at which
    a captured loop takes two branches)."""
    gs = [graphs.barabasi_albert(30000, 4, 1), graphs.erdos_renyi(1500, 8.0 / 1499, 2),
          graphs.watts_strogatz(7500, 6, 0.1, 3)]
    ctx = vne.vne_ctx_create(0)
    try:
        mats = [vne.matrix_from_graph(ctx, g, fp64=False) for g in gs]
        ref = vne.vne_batch_hutchinson(ctx, mats, 80, 15, 9, opt=vne.options(graphs=0))
        for _ in range(4):
            got = vne.vne_batch_hutchinson(ctx, mats, 80, 15, 9)
            assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
        assert vne.vne_ctx_graph_stats(ctx) == (1, 3)
        for mat in mats:
            vne.vne_matrix_destroy(mat)
    finally:
        vne.vne_ctx_destroy(ctx)
