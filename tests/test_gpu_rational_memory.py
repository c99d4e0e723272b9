"""Rational quadratic forms when memory is short: a solve that cannot have the
long window of residuals takes the shortest one, whose residuals fit the room of
the basis that the solve needs in any case."""
import numpy as np
import pytest

from oracle import rng
from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp64", [False, True])
def test_solve_without_room_for_the_long_window(fp64):
    """One allocation of the solve after the other fails once; the call gives the
    undisturbed result with FP32's tolerance 1e-5 (FP64: 1e-10)."""
    g = graphs.watts_strogatz(100_000, 6, 0.1, 3)
    X = rng.rademacher(5, g.n, 0, 16)

    def prepared():
        ctx = vne.vne_ctx_create(0)
        mat = vne.matrix_from_graph(ctx, g, fp64=fp64)
        vne.vne_quadform_batch(ctx, mat, X, 2, opt=vne.options(panel=16))  # schedule and input buffer
        return ctx, mat

    def solve(ctx, mat):
        return vne.vne_quadform_rational(ctx, mat, X, None, num_shifts=3)

    ctx, mat = prepared()
    base = sum(vne.vne_debug_live_allocations())
    want, _, _ = solve(ctx, mat)
    count = sum(vne.vne_debug_live_allocations()) - base
    vne.vne_matrix_destroy(mat)
    vne.vne_ctx_destroy(ctx)
    assert count >= 10
    for k in range(1, count + 1):
        ctx, mat = prepared()
        try:
            vne.vne_debug_fail_allocation(k)
            psi, _, res = solve(ctx, mat)
            vne.vne_debug_fail_allocation(0)
            assert np.max(np.abs(psi - want) / want) <= (1e-10 if fp64 else 1e-5), k
            assert np.all(res <= 1e-8 * 1.0000001), k
        finally:
            vne.vne_debug_fail_allocation(0)
            vne.vne_matrix_destroy(mat)
            vne.vne_ctx_destroy(ctx)
