"""Work on streams beside the call's own: what it uses is made before the streams
fork, and the call's stream continues after all of them."""
import numpy as np
import pytest

from oracle import rng
from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp64", [False, True])
def test_first_rational_call_of_a_context(fp64):
    """Conjugate gradients of a small block run their panels in two groups.  The
    first call of a context, and a later one whose workspace grows, equal the
    same calls on one stream (a profiled context) bit for bit: three and seven
    panels of 8, a graph with rows of several work items."""
    g = graphs.barabasi_albert(30000, 4, 5)
    assert g.degrees.max() > 2 * 256
    X = rng.rademacher(7, g.n, 0, 56)
    out = []
    for profiled in (False, True):
        ctx = vne.vne_ctx_create(0)
        try:
            vne.vne_ctx_profile(ctx, profiled)
            mat = vne.matrix_from_graph(ctx, g, fp64=fp64)
            out.append([vne.vne_quadform_rational(ctx, mat, X[:, :k], None, num_shifts=5, opt=vne.options(panel=8))
                        for k in (24, 56)])
            vne.vne_matrix_destroy(mat)
        finally:
            vne.vne_ctx_destroy(ctx)
    for two, one in zip(*out):
        for a, b in zip(two, one):
            assert np.array_equal(a, b)


def test_first_colourings_of_a_context():
    """The three colourings of the probing method run on a stream each.  On a fresh
    context, and after its workspace grew, the colour counts and T values are
    those of one colouring at a time."""
    ctx = vne.vne_ctx_create(0)
    try:
        for n in (5000, 40000):
            g = graphs.random_geometric(n, graphs.rgg_radius_for_degree(n, 6.0), 3)
            mat = vne.matrix_from_graph(ctx, g, fp64=True, reorder="rcm")
            est, rep = vne.vne_entropy_probing_auto(ctx, mat, 1e-3, 40)
            one = {d: vne.vne_matrix_coloring(ctx, mat, g.n, d) for d in {1, 2, 3, rep["d"]}}
            assert [one[d][1] for d in (1, 2, 3)] == rep["colors_d"]
            # the same colours handed in, so that no colouring runs on the device
            est1, rep1 = vne.vne_entropy_probing_auto(ctx, mat, 1e-3, 40, coloring=lambda d: one[d][0])
            assert np.array_equal(rep["T"], rep1["T"]) and est == est1
            vne.vne_matrix_destroy(mat)
    finally:
        vne.vne_ctx_destroy(ctx)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("max_iter", [4, 7, 36, 37, 38, 39])
def test_solve_after_one_that_was_stopped(fp64, max_iter):
    """A solve that cg_max_iter ends with a copy of its activity flags under way,
    followed at once by a full one: equal to the full one alone."""
    g = graphs.watts_strogatz(20000, 6, 0.1, 2)
    X = rng.rademacher(3, g.n, 0, 32)
    opt = vne.options(panel=8)
    ctx = vne.vne_ctx_create(0)
    try:
        mat = vne.matrix_from_graph(ctx, g, fp64=fp64)
        want = vne.vne_quadform_rational(ctx, mat, X, None, num_shifts=4, opt=opt)
        for _ in range(3):
            _, its, _ = vne.vne_quadform_rational(ctx, mat, X, None, num_shifts=4,
                                                  opt=vne.options(panel=8, cg_max_iter=max_iter))
            assert its.max() == max_iter
            got = vne.vne_quadform_rational(ctx, mat, X, None, num_shifts=4, opt=opt)
            for a, b in zip(got, want):
                assert np.array_equal(a, b)
        vne.vne_matrix_destroy(mat)
    finally:
        vne.vne_ctx_destroy(ctx)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("tol", [1e-2, 1e-3, 1e-4, 1e-6, 1e-8])
def test_short_solves_stop_at_the_next_look(fp64, tol):
    """The conjugate gradients ask for the activity flags every four iterations (of
    the first 64) and look at them four later: a short solve makes as many
    launches as with cg_max_iter set to that iteration."""
    g = graphs.watts_strogatz(3000, 6, 0.1, 2)
    X = rng.rademacher(3, g.n, 0, 5)
    ctx = vne.vne_ctx_create(0)

    def launches(**kw):
        before = vne.vne_ctx_stats(ctx)[0]
        out = vne.vne_quadform_rational(ctx, mat, X, None, num_shifts=1, opt=vne.options(cg_tol=tol, **kw))
        return vne.vne_ctx_stats(ctx)[0] - before, out

    try:
        mat = vne.matrix_from_graph(ctx, g, fp64=fp64)
        launches()
        n, (psi, its, _) = launches()
        assert its.max() < 60
        want, (ref, _, _) = launches(cg_max_iter=(int(its.max()) + 3) // 4 * 4 + 4)
        assert n == want
        assert np.array_equal(psi, ref)
        vne.vne_matrix_destroy(mat)
    finally:
        vne.vne_ctx_destroy(ctx)
