"""Performance cases of the library: what they stand for, their inputs, one pass of each, its necessary work and its 64-bit value.

Every case goes through the calls of ``paper_2212_09642_gb300.vne`` (the binding of the C ABI) with default schedules, as a program
does that creates a matrix and asks for an estimate.  A case is a dict of plain values; ``op`` names the call:

* ``quadform``      quadratic forms of vectors the caller holds (host or device), pattern or valued matrices
* ``rational``      the same by rational Krylov spaces (8 poles, multi-shift CG)
* ``hutchinson``    seeded Hutchinson estimates
* ``build_hutchpp`` a graph that is used once: matrix from host arrays, Hutch++ estimate, matrix freed
* ``hutchpp``       Hutch++ on a resident matrix
* ``batch``         Hutchinson estimates of many uneven graphs in one call
* ``probing``       probing by distance-2 colouring with rational quadratic forms
* ``probing_auto``  probing with the choice of the distance
* ``serve``         a saturated server that answers a set of entropy queries

Results of FP32 matrices (the mixed path: FP32 vectors, FP64 scalars) are returned as float32, the precision that path carries;
results of FP64 matrices as float64.
"""
import math

import numpy as np
import torch

from paper_2212_09642_gb300 import graphs, vne


def listed():
    return [
        # the smallest call: a handful of host vectors on a graph of a few hundred nodes; launches and copies are its cost
        dict(name="quadform_host_small_fp32", op="quadform", family="er", n=700, k=5, m=20, fp64=False, valued=False, device=False,
             reorder=False),
        # the plain FP64 method at the size of the test configuration: G(2000, 0.005), 100 vectors, 50 steps, full reorthogonalisation
        dict(name="hutchinson_er2000_fp64", op="hutchinson", family="er", deg=10.0, n=2000, k=100, m=50, fp64=True, gaussian=False,
             reorder=False),
        # an ordinary FP64 call with device vectors, an odd number of columns and a weighted Laplacian given by its entries
        dict(name="quadform_weighted_fp64", op="quadform", family="ws", n=60001, k=33, m=30, fp64=True, valued=True, device=True,
             reorder=False),
        # an ordinary FP32 Hutchinson estimate on a small-world graph with the paper's Gaussian probes
        dict(name="hutchinson_ws_gauss_fp32", op="hutchinson", family="ws", n=150000, k=64, m=40, fp64=False, gaussian=True,
             reorder=False),
        # rational quadratic forms in FP64 (accuracy studies): basis orthonormalised vector by vector
        dict(name="rational_rgg_fp64", op="rational", family="rgg", n=30011, k=12, fp64=True, poles=8, reorder=False),
        # a graph seen once: assembly, estimate and release all count
        dict(name="build_hutchpp_ba_fp32", op="build_hutchpp", family="ba", n=200003, nr=40, nh=60, m=30, fp64=False, reorder=True),
        # the headline: Barabasi-Albert graph of a million nodes, 100 sketch columns, 100 Hutchinson vectors, 60 steps
        dict(name="hutchpp_ba1e6_fp32", op="hutchpp", family="ba", n=1000000, nr=100, nh=100, m=60, fp64=False, reorder=True),
        # many uneven graphs at once, three families, n log-uniform in [1e3, 2e5]
        dict(name="batch_uneven_fp32", op="batch", count=48, n_min=1000, n_max=200000, k=64, m=40, fp64=False),
        # a large road-network-like graph: device colouring, multi-shift CG with 8 poles on every colour class
        dict(name="probing_rational_rgg1e6_fp32", op="probing", family="rgg", n=1000003, poles=8, fp64=False, reorder="rcm"),
        # the same kind of graph by the method that chooses the distance itself (three colourings, few Lanczos steps)
        dict(name="probing_auto_rgg1e6_fp32", op="probing_auto", family="rgg", n=1000003, eps=1e-3, m=60, fp64=False, reorder="rcm"),
        # a server with every query waiting: uneven graphs, relative accuracy 1e-3, blocks of 64 probes
        dict(name="serve_mix_fp32", op="serve", count=24, n_min=1000, n_max=200000, queries=32, fp64=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["quadform", "quadform", "hutchinson", "hutchinson", "rational", "build_hutchpp", "hutchpp", "batch", "probing",
                     "probing_auto", "serve"])
    fp64 = rng.random() < 0.35
    family = rng.choice(["er", "ba", "ws"])
    if op == "quadform":
        n = _log_int(rng, 300, 80000)
        return dict(op=op, family=family, n=n, k=_log_int(rng, 1, 64), m=rng.randint(10, 40), fp64=fp64,
                    valued=rng.random() < 0.5, device=rng.random() < 0.5, reorder=rng.random() < 0.5)
    if op == "hutchinson":
        n = _log_int(rng, 500, 60000 if fp64 else 400000)
        return dict(op=op, family=family, n=n, k=_log_int(rng, 8, 128), m=rng.randint(15, 50), fp64=fp64,
                    gaussian=rng.random() < 0.3, reorder=rng.random() < 0.5)
    if op == "rational":
        return dict(op=op, family="rgg", n=_log_int(rng, 1000, 50000), k=_log_int(rng, 1, 24), fp64=fp64, poles=rng.randint(3, 8),
                    reorder=rng.choice([False, "rcm"]))
    if op in ("build_hutchpp", "hutchpp"):
        n = _log_int(rng, 2000, 15000 if fp64 else 500000)
        return dict(op=op, family=family, n=n, nr=rng.randint(10, 100), nh=rng.randint(10, 100), m=rng.randint(20, 60), fp64=fp64,
                    reorder=rng.random() < 0.7)
    if op == "batch":
        return dict(op=op, count=rng.randint(3, 40), n_min=1000, n_max=_log_int(rng, 5000, 200000), k=_log_int(rng, 8, 100),
                    m=rng.randint(15, 50), fp64=False)
    if op == "probing":
        return dict(op=op, family="rgg", n=_log_int(rng, 5000, 800000), poles=rng.randint(4, 8), fp64=False, reorder="rcm")
    if op == "probing_auto":
        return dict(op=op, family="rgg", n=_log_int(rng, 5000, 1000000), eps=1e-3, m=60, fp64=False,
                    reorder=rng.choice([False, "rcm"]))
    return dict(op=op, count=rng.randint(3, 20), n_min=1000, n_max=_log_int(rng, 3000, 200000), queries=rng.randint(4, 32), fp64=False)


# ---------------------------------------------------------------------------------------------------------------- inputs

def _graph(family, n, seed, deg=8.0):
    if family == "er":
        return graphs.erdos_renyi(n, deg / (n - 1), seed)
    if family == "ba":
        return graphs.barabasi_albert(n, 4, seed)
    if family == "ws":
        return graphs.watts_strogatz(n, 6, 0.1, seed)
    return graphs.random_geometric(n, graphs.rgg_radius_for_degree(n, 6.0), seed)


def _uneven(case, seed):
    """Graphs of three families, n log-uniform in [n_min, n_max], in the proportions of the batched configuration."""
    rng = np.random.default_rng(seed)
    # spread the sizes evenly over the range, so that the work hardly depends on the seed
    q = (np.arange(case["count"]) + rng.uniform(0.3, 0.7, size=case["count"])) / case["count"]
    sizes = np.rint(case["n_min"] * (case["n_max"] / case["n_min"]) ** q).astype(int)
    out = []
    for i, n in enumerate(sizes):
        n = int(n)
        if i % 3 == 0:
            out.append(graphs.erdos_renyi(n, 8.0 / (n - 1), seed * 64 + i))
        elif i % 3 == 1:
            out.append(graphs.barabasi_albert(n, 3, seed * 64 + i))
        else:
            out.append(graphs.watts_strogatz(n, 6, 0.1, seed * 64 + i))
    return out


def _weighted(g, seed):
    """CSR (rowptr, col, vals) of a weighted Laplacian on the graph g: weights in [0.5, 1.5), diagonal stored."""
    rows = np.repeat(np.arange(g.n, dtype=np.int64), g.degrees)
    col = g.col.astype(np.int64)
    lo, hi = np.minimum(rows, col), np.maximum(rows, col)
    h = (lo * 1000003 + hi * 7919 + seed) & 0xFFFFF  # one weight per edge, the same seen from both ends
    w = 0.5 + h.astype(np.float64) / float(1 << 20)
    diag = np.bincount(rows, weights=w, minlength=g.n)
    r = np.concatenate([rows, np.arange(g.n, dtype=np.int64)])
    c = np.concatenate([col, np.arange(g.n, dtype=np.int64)])
    v = np.concatenate([-w, diag])
    order = np.argsort(r * g.n + c, kind="stable")
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=g.n))]).astype(np.int64)
    return rowptr, c[order].astype(np.int32), v[order]


def _vectors(n, k, seed):
    """Start vectors of a caller: standard normal entries, FP64, host."""
    return np.random.default_rng(seed + 17).standard_normal((n, k))


class State:
    """A context with the matrices (and the server) of one program."""

    def __init__(self, case, seed):
        self.case, self.seed, self.mats, self.srv = case, seed, [], None
        self.ctx = vne.vne_ctx_create(torch.cuda.current_device())
        vne.vne_ctx_set_stream(self.ctx, torch.cuda.current_stream())

    def __del__(self):
        if self.srv is not None:
            vne.vne_server_destroy(self.srv)
        for m in self.mats:
            vne.vne_matrix_destroy(m)
        vne.vne_ctx_destroy(self.ctx)


def _flags(case):
    f = vne.VNE_FP64 if case["fp64"] else vne.VNE_FP32
    if case.get("reorder"):
        f |= vne.VNE_REORDER_RCM if case["reorder"] == "rcm" else vne.VNE_REORDER
    return f


def prepare(case, seed):
    s = State(case, seed)
    op = case["op"]
    if op in ("batch", "serve"):
        for g in _uneven(case, seed):
            s.mats.append(vne.matrix_from_graph(s.ctx, g, fp64=case["fp64"], reorder=op == "serve"))
        if op == "serve":
            s.srv = vne.vne_server_create(s.ctx, 16 << 30, max_active=64, krylov_steps=40, block_vectors=64,
                                          opt=vne.options(reorth=0, quad_tol=-1.0, check_every=3, sketch_steps=10))
        return s
    g = s.graph = _graph(case["family"], case["n"], seed, case.get("deg", 8.0))
    if op == "build_hutchpp":
        return s
    if case.get("valued"):
        rowptr, col, vals = _weighted(g, seed)
        s.mats.append(vne.vne_create_density_matrix(s.ctx, g.n, rowptr, col, vals,
                                                    _flags(case) | vne.VNE_NORMALIZE_TRACE | vne.VNE_IS_LAPLACIAN))
    else:
        s.mats.append(vne.matrix_from_graph(s.ctx, g, fp64=case["fp64"], reorder=case.get("reorder", False)))
    if op in ("quadform", "rational"):
        v = _vectors(g.n, case["k"], seed)
        s.vectors = torch.from_numpy(v).cuda() if case.get("device") else v
    return s


# ------------------------------------------------------------------------------------------------------------- one pass

def run(s):
    c, op, ctx = s.case, s.case["op"], s.ctx
    ft = np.float64 if c["fp64"] else np.float32
    if op == "quadform":
        psi = vne.vne_quadform_batch(ctx, s.mats[0], s.vectors, c["m"], device=bool(c["device"]), k=c["k"])
        return ft(psi)
    if op == "rational":
        psi, its, _ = vne.vne_quadform_rational(ctx, s.mats[0], s.vectors, num_shifts=c["poles"])
        # the iteration counts of an FP32 recurrence depend on its rounding; those of the FP64 one do not
        return {"psi": ft(psi), "iterations": its} if c["fp64"] else {"psi": ft(psi)}
    if op == "hutchinson":
        est, se, psi = vne.vne_entropy_hutchinson(ctx, s.mats[0], c["k"], c["m"], s.seed,
                                                  opt=vne.options(gaussian_probes=int(c["gaussian"])), want_psi=True)
        return {"estimate": ft(est), "std_error": ft(se), "psi": ft(psi)}
    if op == "build_hutchpp":
        g = s.graph
        mat = vne.vne_create_density_matrix(ctx, g.n, g.rowptr, g.col, None, _flags(c))
        try:
            est, parts = vne.vne_entropy_hutchpp(ctx, mat, c["nr"], c["nh"], c["m"], s.seed)
        finally:
            vne.vne_matrix_destroy(mat)
        return {"estimate": ft(est), "parts": ft(parts)}
    if op == "hutchpp":
        est, parts = vne.vne_entropy_hutchpp(ctx, s.mats[0], c["nr"], c["nh"], c["m"], s.seed)
        return {"estimate": ft(est), "parts": ft(parts)}
    if op == "batch":
        est, se = vne.vne_batch_hutchinson(ctx, s.mats, c["k"], c["m"], s.seed)
        return {"estimates": ft(est), "std_errors": ft(se)}
    if op == "probing":
        est, colors = vne.vne_entropy_probing(ctx, s.mats[0], None, 2, 0, num_shifts=c["poles"])
        return {"estimate": ft(est), "colors": colors}
    if op == "probing_auto":
        est, rep = vne.vne_entropy_probing_auto(ctx, s.mats[0], c["eps"], c["m"], opt=vne.options(check_every=2))
        return {"estimate": ft(est), "T": ft(rep["T"]), "d": rep["d"], "colors": rep["colors_d"], "steps": rep["steps_d"]}
    tickets = [vne.vne_server_submit(ctx, s.srv, s.mats[i % len(s.mats)], 1e-3, s.seed * 1000 + i, 8192)
               for i in range(c["queries"])]
    active = 1
    while active or vne.vne_server_info(s.srv)[:2] != (0, 0):
        _, active = vne.vne_server_step(ctx, s.srv)
    res = [vne.vne_server_result(s.srv, t) for t in tickets]
    return {"estimates": ft([r["estimate"] for r in res]), "std_errors": ft([r["std_error"] for r in res]),
            "vectors": np.array([r["vectors"] for r in res])}


# --------------------------------------------------------------------------------------------------------- necessary work

def _size(case):
    """(rows, nonzeros) of a case's graphs, from the families' mean degrees."""
    if case["op"] in ("batch", "serve"):
        r = case["n_max"] / case["n_min"]
        n = case["count"] * case["n_min"] * (r - 1) / math.log(r)
        return n, n * 20.0 / 3.0
    deg = {"er": case.get("deg", 8.0), "ba": 8.0, "ws": 6.0, "rgg": 6.0}[case["family"]]
    return float(case["n"]), case["n"] * (deg + (1.0 if case.get("valued") else 0.0))


def work(case):
    """Bytes: the CSR read once (int32 indices, values if there are any), the caller's vectors read once, the results written.
    Operations: the sparse products, inner products and vector updates of every Krylov step (and of the full
    reorthogonalisation that is the FP64 default), the sketch's products; for adaptive calls the least they run."""
    op, (n, nnz) = case["op"], _size(case)
    es = 8.0 if case["fp64"] else 4.0
    by = 4.0 * (n + 1) + 4.0 * nnz + (es * nnz if case.get("valued") else 0.0)

    def lanczos(k, m):
        f = k * m * (2.0 * nnz + 8.0 * n)
        return f + (4.0 * k * n * m * (m + 1) if case["fp64"] else 0.0)

    if op in ("quadform", "hutchinson", "batch"):
        k, m = case["k"], case["m"]
        return {"bytes": by + (8.0 * n * k if op == "quadform" else 0.0) + 8.0 * k, "flops": lanczos(k, m)}
    if op in ("hutchpp", "build_hutchpp"):
        nr, nh, m = case["nr"], case["nh"], case["m"]
        dense = 2.0 * n * nr * (3.0 * nr + 2.0 * nh) + 2.0 * n * nr * m
        return {"bytes": by + 32.0, "flops": lanczos(nr, m) + lanczos(nr + nh, m) + dense}
    if op in ("rational", "probing"):
        k = case["k"] if op == "rational" else 20
        its, nb = 60.0, case["poles"] + 3.0  # CG iterations of the smallest shift (condition 1e4), basis size
        flops = k * its * (2.0 * nnz + n * (8.0 + 4.0 * case["poles"])) + 2.0 * k * n * nb * nb + k * nb * 2.0 * nnz
        return {"bytes": by + (8.0 * n * k if op == "rational" else 0.0) + 8.0 * k, "flops": flops}
    if op == "probing_auto":
        return {"bytes": by + 64.0, "flops": lanczos(60, 2)}
    per = case["queries"] / case["count"]
    return {"bytes": by + 32.0 * case["queries"], "flops": per * lanczos(4, 10) + per * lanczos(128 + 4, 3)}


# ------------------------------------------------------------------------------------------- 64-bit values (torch, numpy)

_G = 0x9E3779B97F4A7C15


def _i64(x):
    return x - (1 << 64) if x >= (1 << 63) else x


def _shr(z, b):
    return (z >> b) & ((1 << (64 - b)) - 1)


def _mix(z):
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _probes(seed, n, col0, k, gaussian=False):
    """The seeded probe columns that the header documents, float64 [n, k]."""
    t = torch.tensor
    s = _mix(t(_i64((seed + _G) & ((1 << 64) - 1)), device="cuda"))
    key = (torch.arange(col0, col0 + k, device="cuda")[None, :] << 32) | torch.arange(n, device="cuda")[:, None]
    h = _mix((key ^ s) + _i64(_G))
    if not gaussian:
        return 1.0 - 2.0 * _shr(h, 63).double()
    u1 = (_shr(h, 11).double() + 0.5) * 2.0 ** -53
    u2 = _shr(_mix(h + _i64(_G)), 11).double() * 2.0 ** -53
    return torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2)


class _Operator:
    """A = M / tr M in float64: M the graph Laplacian of g, or the matrix of the given entries."""

    def __init__(self, g, entries=None):
        rowptr, col, vals = entries if entries is not None else (g.rowptr, g.col, np.ones(g.nnz))
        self.n = g.n
        self.M = torch.sparse_csr_tensor(torch.from_numpy(rowptr).cuda(), torch.from_numpy(col.astype(np.int64)).cuda(),
                                         torch.from_numpy(vals).cuda(), size=(g.n, g.n))
        rows = np.repeat(np.arange(g.n), np.diff(rowptr))
        self.deg = None if entries is not None else torch.from_numpy(np.diff(rowptr).astype(np.float64)).cuda()[:, None]
        self.trace = float(vals[rows == col].sum()) if entries is not None else float(g.nnz)
        off = np.bincount(rows, weights=np.abs(vals), minlength=g.n)
        self.norm = float(off.max() if entries is not None else 2.0 * np.diff(rowptr).max()) / self.trace

    def __call__(self, x):
        y = self.M @ x
        return (y if self.deg is None else self.deg * x - y) / self.trace


def _f(x):
    return torch.where(x > 0, -x * torch.log(x.clamp(min=1e-300)), torch.zeros_like(x))


def _lanczos(A, X, m, full, keep=False):
    """alpha [k, m], beta [k, m], ||c||, basis (None unless kept) of the centred columns of X."""
    X = X - X.mean(0)
    nrm = X.norm(dim=0)
    v, prev = X / nrm, torch.zeros_like(X)
    beta = torch.zeros(X.shape[1], device=X.device, dtype=X.dtype)
    V, al, be = [v], [], []
    for _ in range(m):
        w = A(v) - beta * prev
        a = (v * w).sum(0)
        w = w - a * v
        if full:
            for _ in range(2):
                for q in V:
                    w = w - (q * w).sum(0) * q
        beta = w.norm(dim=0)
        al.append(a)
        be.append(beta)
        prev, v = v, w / beta
        if full or keep:
            V.append(v)
    return torch.stack(al, 1), torch.stack(be, 1), nrm, V if keep else None


def _tridiag(al, be):
    T = torch.diag_embed(al) + torch.diag_embed(be[:, :-1], 1) + torch.diag_embed(be[:, :-1], -1)
    return torch.linalg.eigh(T.cpu())


def _quad(A, X, m, full):
    al, be, nrm, _ = _lanczos(A, X, m, full)
    th, U = _tridiag(al, be)
    return (nrm.cpu() ** 2 * (U[:, 0, :] ** 2 * _f(th)).sum(1)).numpy()


def _pivoted_q(Y):
    """Q of the column-pivoted QR factorisation, R with a positive diagonal."""
    G = (Y.T @ Y).cpu().numpy()
    k = G.shape[0]
    d, R, piv, left = np.diag(G).copy(), np.zeros((k, k)), [], list(range(k))
    for i in range(k):
        p = max(left, key=lambda j: d[j])
        left.remove(p)
        piv.append(p)
        r = np.sqrt(d[p])
        row = (G[p] - R[:i, p] @ R[:i]) / r
        R[i, left], R[i, p] = row[left], r
        d[left] -= row[left] ** 2
    Q = Y[:, piv] @ torch.from_numpy(np.linalg.inv(R[:, piv])).cuda()
    L = torch.linalg.cholesky(Q.T @ Q)
    return torch.linalg.solve_triangular(L, Q.T, upper=False).T.contiguous()


def _hutchpp(A, nr, nh, m, seed, full):
    al, be, nrm, V = _lanczos(A, _probes(seed, A.n, 0, nr), m, full, keep=True)
    th, U = _tridiag(al, be)
    z = torch.einsum("kij,kj->ki", U, U[:, 0, :] * _f(th)).cuda() * nrm[:, None]
    Y = sum(z[:, j] * V[j] for j in range(m))
    del V
    Q = _pivoted_q(Y)
    G = _probes(seed, A.n, nr, nh)
    psi = _quad(A, torch.cat([Q, G - Q @ (Q.T @ G)], 1), m, full)
    low, res = psi[:nr].sum(), psi[nr:].mean()
    return {"estimate": low + res, "parts": np.array([low, res, nr])}


def _rational(A, B, num_shifts):
    """psi and None for the iterations: span{c, Ac, A^2 c, (A + s)^{-1} c}, shifted systems by CG to 1e-13."""
    C = B - B.mean(0)
    x, W = C, [C]
    for _ in range(2):
        x = A(x)
        W.append(x)
    for i in range(num_shifts):
        s = A.norm * 10.0 ** (-4.0 * i / (num_shifts - 1) if num_shifts > 1 else 0.0)
        x, r, p = torch.zeros_like(C), C.clone(), C.clone()
        rho = rho0 = (r * r).sum(0)
        for it in range(4000):
            q = A(p) + s * p
            a = rho / (p * q).sum(0)
            x, r = x + a * p, r - a * q
            new = (r * r).sum(0)
            if it % 8 == 0 and bool((new <= 1e-26 * rho0).all()):
                break
            p, rho = r + (new / rho) * p, new
        W.append(x)
    out = []
    for j in range(C.shape[1]):
        w = torch.stack([v[:, j] / v[:, j].norm() for v in W], 1)
        Q, R = torch.linalg.qr(w)
        keep = R.diag().abs() > 1e-12
        Q = Q[:, keep]
        H = Q.T @ A(Q)
        th, U = torch.linalg.eigh(((H + H.T) / 2).cpu())
        out.append(float(C[:, j] @ C[:, j]) * float((U[0] ** 2 * _f(th)).sum()))
    return {"psi": np.array(out), "iterations": None}


def exact(case, seed):
    op = case["op"]
    full = case["fp64"]
    if op == "batch":
        est, se = [], []
        for g in _uneven(case, seed):
            p = _quad(_Operator(g), _probes(seed, g.n, 0, case["k"]), case["m"], False)
            est.append(p.mean())
            se.append(p.std(ddof=1) / math.sqrt(len(p)))
        return {"estimates": np.array(est), "std_errors": np.array(se)}
    if op in ("probing", "probing_auto", "serve"):
        # the sequential greedy colouring takes minutes in plain Python; a served or adaptive estimate stops by its own error
        return None
    g = _graph(case["family"], case["n"], seed, case.get("deg", 8.0))
    A = _Operator(g, _weighted(g, seed) if case.get("valued") else None)
    if op == "quadform":
        return _quad(A, torch.from_numpy(_vectors(g.n, case["k"], seed)).cuda(), case["m"], full)
    if op == "rational":
        r = _rational(A, torch.from_numpy(_vectors(g.n, case["k"], seed)).cuda(), case["poles"])
        return r if case["fp64"] else {"psi": r["psi"]}
    if op == "hutchinson":
        p = _quad(A, _probes(seed, g.n, 0, case["k"], case["gaussian"]), case["m"], full)
        return {"estimate": p.mean(), "std_error": p.std(ddof=1) / math.sqrt(len(p)), "psi": p}
    return _hutchpp(A, case["nr"], case["nh"], case["m"], seed, full)
