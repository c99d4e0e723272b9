"""The FP32 update over several row tiles per CTA: 64 columns of at least two
tiles per SM and panel, one or two tiles in the last CTA of a panel, every
column against the 64-bit value (shifted systems by CG to 1e-13)."""
import numpy as np
import pytest
import torch

from oracle import rng
from paper_2212_09642_gb300 import graphs, vne

pytestmark = pytest.mark.gpu

SHIFTS = (1e-6, 1e-5)


def _reference(g, X):
    n, tr = g.n, float(g.nnz)
    M = torch.sparse_csr_tensor(torch.from_numpy(np.asarray(g.rowptr, dtype=np.int64)),
                                torch.from_numpy(np.asarray(g.col, dtype=np.int64)),
                                torch.ones(g.nnz, dtype=torch.float64), size=(n, n)).cuda()
    deg = torch.from_numpy(np.asarray(g.degrees, dtype=np.float64)).cuda()[:, None]

    def A(x):
        return (deg * x - M @ x) / tr

    C = torch.from_numpy(np.asarray(X, dtype=np.float64)).cuda()
    C = C - C.mean(0)
    W = [C, A(C)]
    W.append(A(W[1]))
    for s in SHIFTS:
        x, r, p = torch.zeros_like(C), C.clone(), C.clone()
        rho = rho0 = (r * r).sum(0)
        for _ in range(2000):
            q = A(p) + s * p
            a = rho / (p * q).sum(0)
            x, r = x + a * p, r - a * q
            new = (r * r).sum(0)
            if bool((new <= 1e-26 * rho0).all()):
                break
            p, rho = r + (new / rho) * p, new
        W.append(x)
    out = np.zeros(C.shape[1])
    for j in range(C.shape[1]):
        Q = torch.linalg.qr(torch.stack([w[:, j] / w[:, j].norm() for w in W], 1))[0]
        H = Q.T @ A(Q)
        th, U = torch.linalg.eigh(((H + H.T) / 2).cpu())
        f = torch.where(th > 0, -th * torch.log(th.clamp(min=1e-300)), torch.zeros_like(th))
        out[j] = float(C[:, j] @ C[:, j]) * float((U[0] ** 2 * f).sum())
    return out


@pytest.mark.parametrize("last", [1, 2])
def test_update_over_several_tiles(vctx, last):
    tiles = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    while tiles % 3 != last:
        tiles += 1
    n = (tiles - 1) * 1024 + (1 if last == 1 else 1024)
    g = graphs.watts_strogatz(n, 6, 0.2, 3)
    X = rng.rademacher(5, g.n, 0, 64)
    mat = vne.matrix_from_graph(vctx, g, fp64=False)
    try:
        psi, _, res = vne.vne_quadform_rational(vctx, mat, X, np.array(SHIFTS),
                                                opt=vne.options(cg_tol=1e-8, panel=8))
    finally:
        vne.vne_matrix_destroy(mat)
    ref = _reference(g, X)
    assert np.all(res <= 1e-8 * 1.0000001)
    assert np.max(np.abs(psi - ref) / ref) <= 1e-5
