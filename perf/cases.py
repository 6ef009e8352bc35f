"""The work that a user of this library has it do, as cases that can be timed and compared.

`listed()` names the cases, `draw(rng)` gives more of the same ranges, `prepare(case, seed)` makes what a user's
program holds before the call (matrices, start blocks, a context), `run(state)` is one pass through the public entry
points, `work(case)` the bytes and flops it cannot do without and `exact(case, seed)` its outputs in 64 bits.

Eigenpairs come back from the library in the order of their residuals and with the phase of their largest entry, which
rounding decides when two entries or two residuals tie (the grid operators here have mirror symmetry).  A program that
uses the pairs sorts them by eigenvalue and fixes their phase against a vector of its own; `run` does the same on the
device.
"""
import math

import numpy as np
import torch

from paper_1506_04463_gb300 import feast_nh as F
from paper_1506_04463_gb300 import workloads as wl

PREC = {"fp64": F.PREC_FP64, "fp32_ir": F.PREC_FP32_IR}
NET_LAYERS, NET_CH = 4, 32


def listed():
    return [
        # A small interactive problem: a full solve whose kernels are all short, so launches, reads of the status and
        # the one-block dense kernels count.
        {"name": "solve_grid10", "kind": "solve", "N": 10, "beta": 10.0, "m": 6, "m0": 12, "ne": 8,
         "precision": "fp32_ir"},
        # The default options (FP64 throughout) on the convection-diffusion test problem.
        {"name": "solve_grid40_fp64", "kind": "solve", "N": 40, "beta": 10.0, "m": 30, "m0": 48, "ne": 16,
         "precision": "fp64"},
        # An ordinary solve: 10 000 unknowns, FP32 factors inside FP64 refinement.
        {"name": "solve_grid100", "kind": "solve", "N": 100, "beta": 10.0, "m": 24, "m0": 40, "ne": 16,
         "precision": "fp32_ir"},
        # The benchmark: 90 000 unknowns, 30 interior eigenvalues, 64 columns, 16 nodes.
        {"name": "solve_grid300", "kind": "solve", "N": 300, "beta": 10.0, "m": 30, "m0": 64, "ne": 16,
         "precision": "fp32_ir"},
        # The contour filter alone on the tridiagonal problem in FP64, factors kept from call to call (a program with
        # its own outer iteration).
        {"name": "filter_tridiag1000", "kind": "filter_tridiag", "n": 1000, "m0": 40, "ne": 8, "precision": "fp64"},
        # The filter on the generalized complex-symmetric problem (diagonal B, complex A, half-bandwidth 256).
        {"name": "filter_cube16", "kind": "filter_cube", "L": 16, "layers": 2, "m0": 32, "ne": 16,
         "precision": "fp32_ir"},
        # The filter with the Krylov inner solver (FGMRES, Jacobi) on a random sparse matrix that has no band.
        {"name": "filter_sparse3000_fgmres", "kind": "filter_sparse", "n": 3000, "m0": 32, "ne": 8, "inside": 24},
        # One Rayleigh-Ritz step at the benchmark's size (projections, dense eigenproblems, residuals).
        {"name": "rr_grid300", "kind": "rr", "N": 300, "beta": 10.0, "m": 64, "ne": 16},
        # The FP64 residual of every shifted system: the check that ends each refinement step, odd sizes.
        {"name": "residual_grid211", "kind": "residual", "N": 211, "beta": 10.0, "m": 45, "ne": 15},
        # The FP32 operator of the Krylov sweeps for every node at once, nine entries a row at random columns.
        {"name": "spmm_sparse50021", "kind": "spmm", "n": 50021, "m": 48, "ne": 8, "inside": 24, "side": 0},
        # Many independent sparse problems of different sizes solved together.
        {"name": "batch6_sparse", "kind": "batch", "nprob": 6, "nmin": 1000, "nmax": 6000, "m0": 32, "ne": 8,
         "inside": 20},
        # One training pass of the learned preconditioner's network: forward, loss, gradient of every weight.
        {"name": "net_train64", "kind": "net", "N": 64, "images": 48},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "filter_tridiag", "filter_cube", "filter_sparse", "rr", "residual",
                       "spmm", "batch", "net"])
    if kind == "solve":
        prec = rng.choice(["fp32_ir", "fp32_ir", "fp64"])
        N = _log(rng, 9, 60 if prec == "fp64" else 260)
        m = min(rng.randint(4, 30), N * N // 12)
        return {"kind": kind, "N": N, "beta": round(rng.uniform(7.0, 12.0), 2), "m": m,
                "m0": min(64, 2 * m + rng.randint(0, 6)), "ne": rng.choice([8, 12, 16]), "precision": prec}
    if kind == "filter_tridiag":
        return {"kind": kind, "n": _log(rng, 150, 4000), "m0": rng.randint(5, 64), "ne": rng.choice([4, 6, 8, 16]),
                "precision": rng.choice(["fp64", "fp32_ir"])}
    if kind == "filter_cube":
        L = rng.randint(6, 16)
        return {"kind": kind, "L": L, "layers": rng.randint(1, max(1, L // 8)), "m0": rng.randint(7, 32),
                "ne": rng.choice([6, 8, 16]), "precision": "fp32_ir"}
    if kind == "filter_sparse":
        m0 = rng.randint(9, 32)
        return {"kind": kind, "n": _log(rng, 400, 3000), "m0": m0, "ne": rng.choice([4, 8]), "inside": m0 // 2}
    if kind == "rr":
        N = _log(rng, 24, 300)
        return {"kind": kind, "N": N, "beta": round(rng.uniform(7.0, 12.0), 2), "m": rng.randint(9, 64), "ne": 16}
    if kind == "residual":
        return {"kind": kind, "N": _log(rng, 16, 211), "beta": round(rng.uniform(2.0, 20.0), 2),
                "m": rng.randint(5, 64), "ne": rng.choice([6, 8, 15, 16])}
    if kind == "spmm":
        m = rng.randint(9, 64)
        return {"kind": kind, "n": _log(rng, 700, 50000), "m": m, "ne": rng.choice([4, 8, 16] if m < 25 else [4, 8]),
                "inside": 16, "side": rng.randint(0, 1)}
    if kind == "batch":
        lo = _log(rng, 500, 2000)
        m0 = rng.randint(20, 32)
        return {"kind": kind, "nprob": rng.randint(2, 6), "nmin": lo, "nmax": lo * rng.randint(2, 3), "m0": m0,
                "ne": 8, "inside": rng.randint(10, 5 * m0 // 8)}
    return {"kind": "net", "N": _log(rng, 17, 64), "images": rng.randint(5, 48)}


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------
def _normal(seed, *shape, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


def _beta(case, seed):
    """The case's Peclet number, within two percent: every seed is another operator."""
    return case["beta"] * (1.0 + 0.02 * (2.0 * np.random.default_rng(seed).random() - 1.0))


def _grid_modes(N, beta, first, m):
    """(eigenvalue, k, l) of the m eigenvalues from index `first` of the closed form, increasing."""
    h = 1.0 / (N + 1)
    g = beta * h
    k = np.arange(1, N + 1)
    lx = (2 + g) - 2 * np.sqrt(1 + g) * np.cos(k * np.pi * h)
    ly = 2 - 2 * np.cos(k * np.pi * h)
    lam = lx[:, None] + ly[None, :]
    order = np.argsort(lam.ravel(), kind="stable")[first:first + m]
    return lam.ravel()[order], order // N + 1, order % N + 1


def _grid_vectors(N, beta, k, l):
    """Closed-form right and left eigenvectors (N*N x m, x fastest): ||x|| = 1 and x^^H x = 1."""
    i = torch.arange(1, N + 1, device="cuda", dtype=torch.float64)
    k, l = (torch.as_tensor(v, device="cuda", dtype=torch.float64) for v in (k, l))
    sx, sy = (torch.sin(i[:, None] * v[None, :] * (math.pi / (N + 1))) for v in (k, l))
    d = torch.exp(0.5 * i * math.log1p(beta / (N + 1)))[:, None]
    X = (sy[:, None, :] * (sx * d)[None, :, :]).reshape(N * N, -1)
    Xh = (sy[:, None, :] * (sx / d)[None, :, :]).reshape(N * N, -1)
    X = X / torch.linalg.vector_norm(X, dim=0)
    Xh = Xh / (Xh * X).sum(0)
    return X.to(torch.complex128), Xh.to(torch.complex128)


def _grid_first(N):
    return 300 if N * N > 4000 else max(1, N * N // 4)


def _grid_contour(case, beta):
    """The benchmark's contour: an ellipse around m consecutive eigenvalues, placed where the gaps around them are
    widest.  Returns (contour, index of the first eigenvalue inside)."""
    N, m = case["N"], case["m"]
    lam = wl.convdiff2d_eigs(N, beta)
    lo = _grid_first(N)
    s = max(range(lo, min(lo + 100, N * N - m - 1)),
            key=lambda i: min(lam[i] - lam[i - 1], lam[i + m] - lam[i + m - 1]))
    gap = min(lam[s] - lam[s - 1], lam[s + m] - lam[s + m - 1])
    a = 0.5 * (lam[s + m - 1] - lam[s]) + 0.5 * gap
    return wl.Contour(1, complex(0.5 * (lam[s] + lam[s + m - 1])), float(a), ratio=0.5, ne=case["ne"]), s


def _sparse_csr(n, inside, seed):
    """A matrix of the many-problem family: the diagonal and eight more distinct columns a row, N(0, 1/9), the
    diagonal shifted by U(0, 4); `inside` rows are shifted to the right of that, 5.7 to 8.3, so that a circle at the
    spectrum's right edge holds their eigenvalues.  Returns rowptr, colind, val (numpy) and the shifted diagonals."""
    rng = np.random.default_rng(seed)
    i = np.arange(n)[:, None]
    step = 1 + np.floor((np.arange(8) + rng.random((n, 8))) * ((n - 1) / 8.0)).astype(np.int64)
    cols = np.concatenate([i, (i + step) % n], axis=1)
    vals = rng.normal(0.0, 1.0 / 3.0, (n, 9))
    vals[:, 0] += rng.uniform(0.0, 4.0, n)
    rows = rng.choice(n, size=inside, replace=False)
    at = 5.8 + 2.4 * (np.arange(inside) + 0.5) / inside
    vals[rows, 0] = at
    order = np.argsort(cols, axis=1)
    cols, vals = np.take_along_axis(cols, order, 1), np.take_along_axis(vals, order, 1)
    return (9 * np.arange(n + 1)).astype(np.int32), cols.astype(np.int32).ravel(), vals.ravel(), at


def _sparse_contour(ne):
    return wl.Contour(0, 7.0 + 0j, 1.5, ne=ne)


def _csr_tuple(rp, ci, val):
    return (torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), torch.from_numpy(val).cuda(), F.R64,
            rp.size - 1, ci.size)


def _sizes(case, seed):
    rng = np.random.default_rng(case["nmin"] * 7 + case["nprob"])
    u = np.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["nprob"]))
    return [int(v) for v in np.round(u)]


def _cube(case, seed):
    A, B = wl.laplace3d_cap(case["L"], case["layers"], seed_cap=2 * seed, seed_b=2 * seed + 1)
    return A, B, wl.Contour(0, 0.35 - 0.1j, 0.12, ne=case["ne"])


def _tridiag(case):
    A, _ = wl.symmetrized_tridiag(case["n"], 1.0, 2.0, 0.5)
    return A, wl.Contour(0, 2.0 + 0j, 0.08, ne=case["ne"])


def _start(n, m, seed, complex_=False):
    Y = _normal(2 * seed, n, m)
    Yh = _normal(2 * seed + 1, n, m)
    if complex_:
        return torch.complex(Y, Yh) / math.sqrt(2.0)
    return Y.to(torch.complex128), Yh.to(torch.complex128)


def _rr_blocks(case, seed):
    """Filtered blocks: m eigenvectors of each side, mixed by well-conditioned matrices (what a late outer iteration
    hands to the Rayleigh-Ritz step)."""
    N, m = case["N"], case["m"]
    beta = _beta(case, seed)
    lam, k, l = _grid_modes(N, beta, _grid_first(N), m)
    X, Xh = _grid_vectors(N, beta, k, l)
    eye = torch.eye(m, device="cuda", dtype=torch.complex128)
    C = eye + 0.5 / math.sqrt(m) * torch.complex(_normal(4 * seed, m, m), _normal(4 * seed + 1, m, m))
    Ch = eye + 0.5 / math.sqrt(m) * torch.complex(_normal(4 * seed + 2, m, m), _normal(4 * seed + 3, m, m))
    return beta, lam, X, Xh, X @ C, Xh @ Ch


def _net_data(case, seed):
    N, S = case["N"], case["images"]
    rng = np.random.default_rng(seed)
    p = []
    for _ in range(NET_LAYERS):
        p.append(rng.standard_normal(9 * NET_CH * NET_CH) * math.sqrt(2.0 / (9 * NET_CH)))
        p.append(0.05 * rng.standard_normal(NET_CH))
    x = torch.zeros(S, N, N, NET_CH, device="cuda")
    x[..., :2] = _normal(2 * seed, S, N, N, 2, dtype=torch.float32)  # the residual, scaled to unit size
    x[..., 2:4] = _normal(2 * seed + 1, S, 1, 1, 2, dtype=torch.float32)  # the node
    x[..., 4] = 0.3
    t = _normal(2 * seed + 5, S, N, N, 2, dtype=torch.float32)
    return np.concatenate(p).astype(np.float32), x, t


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind in ("solve", "rr", "residual"):
        N = case["N"]
        beta = _beta(case, seed)
        A = wl.convdiff2d(N, beta)
        st["ref"] = _normal(17, N * N).to(torch.complex128)
    if kind == "solve":
        con, _ = _grid_contour(case, beta)
        st["ctx"] = F.FeastNH(A, None, con, case["m0"], precision=PREC[case["precision"]])
        st["Y"], st["Yh"] = _start(N * N, case["m0"], seed)
    elif kind == "rr":
        _, lam, _, _, st["Q"], st["Qh"] = _rr_blocks(case, seed)
        con = wl.Contour(1, complex(0.5 * (lam[0] + lam[-1])), float(0.6 * (lam[-1] - lam[0])), ratio=0.5,
                         ne=case["ne"])
        st["ctx"] = F.FeastNH(A, None, con, case["m"], precision=F.PREC_FP32_IR)
    elif kind == "residual":
        con = wl.Contour(1, 0.5 + 0j, 0.1, ratio=0.5, ne=case["ne"])
        st["ctx"] = F.FeastNH(A, None, con, case["m"], precision=F.PREC_FP32_IR)
        sh = (case["ne"], N * N, case["m"])
        st["X"] = torch.complex(_normal(4 * seed, *sh), _normal(4 * seed + 1, *sh))
        st["BY"] = torch.complex(_normal(4 * seed + 2, *sh[1:]), _normal(4 * seed + 3, *sh[1:]))
    elif kind == "filter_tridiag":
        A, con = _tridiag(case)
        st["ctx"] = F.FeastNH(A, None, con, case["m0"], precision=PREC[case["precision"]])
        st["Y"], st["Yh"] = _start(case["n"], case["m0"], seed)
    elif kind == "filter_cube":
        A, B, con = _cube(case, seed)
        st["ctx"] = F.FeastNH(A, B, con, case["m0"], precision=PREC[case["precision"]],
                              problem=F.PROBLEM_COMPLEX_SYMMETRIC)
        st["Y"] = _start(case["L"] ** 3, case["m0"], seed, True)
        st["Yh"] = None
    elif kind == "filter_sparse":
        A = _csr_tuple(*_sparse_csr(case["n"], case["inside"], seed)[:3])
        st["ctx"] = F.FeastNH(A, None, _sparse_contour(case["ne"]), case["m0"], precision=F.PREC_FP32_IR,
                              inner_kind=F.INNER_FGMRES)
        st["Y"], st["Yh"] = _start(case["n"], case["m0"], seed)
    elif kind == "spmm":
        A = _csr_tuple(*_sparse_csr(case["n"], case["inside"], seed)[:3])
        st["ctx"] = F.FeastNH(A, None, _sparse_contour(case["ne"]), case["m"], precision=F.PREC_FP32_IR,
                              inner_kind=F.INNER_FGMRES, krylov_restart=1)
        sh = (case["ne"], case["n"], case["m"])
        st["P"] = torch.complex(_normal(2 * seed, *sh, dtype=torch.float32),
                                _normal(2 * seed + 1, *sh, dtype=torch.float32))
        st["side"] = case["side"]
    elif kind == "batch":
        sizes = _sizes(case, seed)
        A = [_csr_tuple(*_sparse_csr(n, case["inside"], 100 * seed + p)[:3]) for p, n in enumerate(sizes)]
        # the shifted systems two digits below the eigenpairs' tolerance, so that the outer iteration ends by
        # converging and not at the noise of its inner solves
        st["ctx"] = F.FeastBatch(A, [_sparse_contour(case["ne"])] * len(A), case["m0"], precision=F.PREC_FP32_IR,
                                 inner_tol=1e-12, inner_max=8, max_iter=30)
        st["Y"], st["Yh"] = _start(sum(sizes), case["m0"], seed)
        st["ref"] = [_normal(17, n).to(torch.complex128) for n in sizes]
    else:
        p, st["x"], st["t"] = _net_data(case, seed)
        st["net"] = F.Net(NET_LAYERS, case["N"], case["images"])
        st["net"].set_params(p)
    return st


def _sorted_pairs(lam, X, Xh, ref):
    """Eigenpairs by increasing real part, with ref^H x real and positive (x^^H B x is unchanged)."""
    order = torch.argsort(lam.real)
    X, Xh = X[:, order], Xh[:, order]
    ph = torch.conj(torch.sgn(torch.mv(X.t(), ref)))
    return {"lam": lam[order], "X": X * ph, "Xh": Xh * ph}


def run(st):
    kind = st["kind"]
    if kind == "solve":
        out = st["ctx"].solve(st["Y"], st["Yh"])
        return _sorted_pairs(out["lam"], out["X"], out["Xh"], st["ref"])
    if kind == "rr":
        lam, Y, Yh, _ = st["ctx"].rr(st["Q"], st["Qh"])
        return _sorted_pairs(lam, Y, Yh, st["ref"])
    if kind == "residual":
        R, Q = st["ctx"].multishift_residual(st["X"], st["BY"])
        return {"R": R, "Q": Q}
    if kind == "spmm":
        return {"V": st["ctx"].multishift_spmm(st["P"], st["side"])}
    if kind == "batch":
        out = st["ctx"].solve(st["Y"], st["Yh"])
        return [_sorted_pairs(p["lam"], p["X"], p["Xh"], r) for p, r in zip(out["problems"], st["ref"])]
    if kind == "net":
        loss, grad = st["net"].train_step(st["x"], st["t"], 0.0, want_grad=True)
        return {"loss": loss, "grad": grad}
    Q, Qh = st["ctx"].filter(st["Y"], st["Yh"])
    return {"Q": Q, "Qh": Qh}


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("solve", "rr", "residual"):
        n = case["N"] ** 2
        csr = 12 * (5 * n - 4 * case["N"]) + 4 * (n + 1)
    if kind == "solve":
        # one factorisation of each conjugate pair of nodes; two filters (the first, and the one that converges), each
        # with one forward and one backward substitution for both sides; the tall products of the two Rayleigh-Ritz
        # steps (three projections and four updates of n x m0 blocks)
        m0, ne, bw = case["m0"], case["ne"], case["N"]
        flops = 8.0 * (ne // 2) * n * bw * bw + 2 * 2 * ne * m0 * 16.0 * n * bw + 2 * 7 * 8.0 * n * m0 * m0
        return {"bytes": csr + 16.0 * n * (2 * m0 + 2 * case["m"]), "flops": flops}
    if kind == "rr":
        m = case["m"]
        return {"bytes": 2 * csr + 16.0 * n * 4 * m, "flops": 7 * 8.0 * n * m * m + 2 * 8.0 * 5 * n * m}
    if kind == "residual":
        m, ne = case["m"], case["ne"]
        return {"bytes": csr + 16.0 * n * m * (2 * ne + 2), "flops": float(ne) * m * n * (8 + 4 * 5 + 8)}
    if kind == "filter_tridiag":
        n, m, ne = case["n"], case["m0"], case["ne"]
        return {"bytes": 16.0 * n * 4 * m + 48.0 * n, "flops": 2.0 * ne * m * n * (16 + 16)}
    if kind == "filter_cube":
        n, m, ne, bw = case["L"] ** 3, case["m0"], case["ne"], case["L"] ** 2
        return {"bytes": 16.0 * n * 3 * m + 20.0 * 8 * n, "flops": 16.0 * ne * m * n * bw + ne * m * n * 70.0}
    if kind == "filter_sparse":
        # each side's systems need at least one application of the operator for every digit or so: ten applications
        n, m, ne = case["n"], case["m0"], case["ne"]
        return {"bytes": 16.0 * n * 4 * m + 12.0 * 9 * n, "flops": 2 * 10.0 * ne * m * n * (8 + 4 * 9)}
    if kind == "spmm":
        n, m, ne = case["n"], case["m"], case["ne"]
        return {"bytes": 16.0 * n * m * ne + 12.0 * 9 * n, "flops": float(ne) * m * n * (8 + 4 * 9)}
    if kind == "batch":
        n, m, ne = sum(_sizes(case, 0)), case["m0"], case["ne"]
        return {"bytes": 16.0 * n * 4 * m + 12.0 * 9 * n, "flops": 3 * 2 * 10.0 * ne * m * n * (8 + 4 * 9)}
    pix = case["images"] * case["N"] ** 2
    conv = 2.0 * pix * 9 * NET_CH * NET_CH
    return {"bytes": 4.0 * pix * (NET_CH + 2), "flops": conv * (3 * NET_LAYERS - 1)}


# ---------------------------------------------------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------------------------------------------------
def _nodes(con):
    """Half-offset trapezoidal nodes and weights on a circle or an ellipse whose axes are parallel to the axes."""
    t = math.pi * (2 * np.arange(con.ne) + 1) / con.ne
    a, b = con.r, con.r * (con.ratio if con.kind == 1 else 1.0)
    z = con.center + a * np.cos(t) + 1j * b * np.sin(t)
    return z, (b * np.cos(t) + 1j * a * np.sin(t)) / con.ne


def _dense(rp, ci, val):
    n = rp.size - 1
    A = torch.zeros(n, n, dtype=torch.complex128, device="cuda")
    rows = torch.from_numpy(np.repeat(np.arange(n), np.diff(rp))).cuda()
    A.index_put_((rows, torch.from_numpy(ci.astype(np.int64)).cuda()),
                 torch.from_numpy(val.astype(np.complex128)).cuda(), accumulate=True)
    return A


def _filter_dense(A, B, con, Y, Yh):
    Q, Qh = torch.zeros_like(Y), torch.zeros_like(Y)
    z, w = _nodes(con)
    BY, BhYh = (Y, Yh) if B is None else (B @ Y, B.mH @ Yh)
    eye = torch.eye(A.shape[0], device="cuda", dtype=A.dtype) if B is None else B
    for zj, wj in zip(z, w):
        M = complex(zj) * eye - A
        Q += complex(wj) * torch.linalg.solve(M, BY)
        Qh += complex(wj).conjugate() * torch.linalg.solve(M.mH, BhYh)
    return {"Q": Q, "Qh": Qh}


def _shift_apply(rp, ci, val, z, X):
    """z_j X_j - A X_j for every node j."""
    out = torch.from_numpy(np.asarray(z)).cuda()[:, None, None] * X
    rows = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    at = np.arange(ci.size) - rp[rows]
    for k in range(int(at.max()) + 1):
        sel = at == k
        r = torch.from_numpy(rows[sel]).cuda()
        c = torch.from_numpy(ci[sel].astype(np.int64)).cuda()
        v = torch.from_numpy(val[sel]).cuda()[None, :, None]
        for j in range(X.shape[0]):
            out[j].index_add_(0, r, -(v[0] * X[j, c]))
    return out


def _transpose(rp, ci, val):
    rows = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    order = np.argsort(ci, kind="stable")
    cnt = np.bincount(ci, minlength=rp.size - 1)
    return np.concatenate(([0], np.cumsum(cnt))).astype(np.int32), rows[order].astype(np.int32), val[order]


def _inverse_iteration(A, guess):
    """The eigenpairs of a dense A nearest to well separated guesses."""
    n = A.shape[0]
    eye = torch.eye(n, device="cuda", dtype=A.dtype)
    lam, X, Xh = [], [], []
    for g in guess:
        mu = complex(g)
        x, y = _normal(1, n, 1).to(A.dtype), _normal(2, n, 1).to(A.dtype)
        for it in range(6):
            lu, piv = torch.linalg.lu_factor(A - mu * (1 + 1e-14) * eye)
            for _ in range(2):
                x = torch.linalg.lu_solve(lu, piv, x)
                x = x / torch.linalg.vector_norm(x)
                y = torch.linalg.lu_solve(lu, piv, y, adjoint=True)
                y = y / torch.linalg.vector_norm(y)
            new = complex(((y.mH @ (A @ x)) / (y.mH @ x)).item())
            done = abs(new - mu) <= 1e-14 * abs(mu)
            mu = new
            if done:
                break
        lam.append(mu)
        X.append(x)
        Xh.append(y / torch.conj(y.mH @ x))
    return torch.tensor(lam, dtype=A.dtype, device="cuda"), torch.cat(X, 1), torch.cat(Xh, 1)


def _net_exact(case, seed):
    p, x, t = _net_data(case, seed)
    p = torch.from_numpy(p).cuda().double()
    per = 9 * NET_CH * NET_CH + NET_CH
    params = [p[k * per:(k + 1) * per].clone().requires_grad_() for k in range(NET_LAYERS)]
    S = case["images"]
    count = t.numel()
    loss = 0.0
    for s in range(0, S, 8):  # images are independent: a few at a time
        a = x[s:s + 8].double().permute(0, 3, 1, 2)
        for k, q in enumerate(params):
            W = q[:9 * NET_CH * NET_CH].view(3, 3, NET_CH, NET_CH).permute(3, 2, 0, 1)
            a = torch.nn.functional.conv2d(a, W, q[9 * NET_CH * NET_CH:], padding=1)
            if k + 1 < NET_LAYERS:
                a = torch.relu(a)
        part = (a[:, :2].permute(0, 2, 3, 1) - t[s:s + 8].double()).square().sum() / count
        part.backward()
        loss += float(part.detach())
    return {"loss": loss, "grad": torch.cat([q.grad for q in params])}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "rr"):
        N, beta = case["N"], _beta(case, seed)
        if kind == "solve":
            _, first = _grid_contour(case, beta)
            lam, k, l = _grid_modes(N, beta, first, case["m"])
        else:
            lam, k, l = _grid_modes(N, beta, _grid_first(N), case["m"])
        X, Xh = _grid_vectors(N, beta, k, l)
        ref = _normal(17, N * N).to(torch.complex128)
        return _sorted_pairs(torch.from_numpy(lam).cuda().to(torch.complex128), X, Xh, ref)
    if kind == "residual":
        st = {}
        A = wl.convdiff2d(case["N"], _beta(case, seed))
        con = wl.Contour(1, 0.5 + 0j, 0.1, ratio=0.5, ne=case["ne"])
        sh = (case["ne"], case["N"] ** 2, case["m"])
        X = torch.complex(_normal(4 * seed, *sh), _normal(4 * seed + 1, *sh))
        BY = torch.complex(_normal(4 * seed + 2, *sh[1:]), _normal(4 * seed + 3, *sh[1:]))
        z, w = _nodes(con)
        st["R"] = BY[None] - _shift_apply(A.indptr, A.indices, A.data, z, X)
        st["Q"] = torch.einsum("j,jnm->nm", torch.from_numpy(w).cuda(), X)
        return st
    if kind == "spmm":
        rp, ci, val, _ = _sparse_csr(case["n"], case["inside"], seed)
        sh = (case["ne"], case["n"], case["m"])
        P = torch.complex(_normal(2 * seed, *sh, dtype=torch.float32), _normal(2 * seed + 1, *sh, dtype=torch.float32))
        z, _ = _nodes(_sparse_contour(case["ne"]))
        if case["side"]:
            rp, ci, val = _transpose(rp, ci, val)
            z = z.conj()
        return {"V": _shift_apply(rp, ci, val, z, P.to(torch.complex128))}
    if kind == "filter_tridiag":
        A, con = _tridiag(case)
        return _filter_dense(torch.from_numpy(A.toarray()).cuda().to(torch.complex128), None, con,
                             *_start(case["n"], case["m0"], seed))
    if kind == "filter_cube":
        A, B, con = _cube(case, seed)
        Y = _start(case["L"] ** 3, case["m0"], seed, True)
        A, B = (torch.from_numpy(M.toarray()).cuda() for M in (A, B))
        z, w = _nodes(con)
        BY = B @ Y
        Q = torch.zeros_like(Y)
        for zj, wj in zip(z, w):
            Q += complex(wj) * torch.linalg.solve(complex(zj) * B - A, BY)
        return {"Q": Q, "Qh": Q.conj().resolve_conj()}
    if kind == "filter_sparse":
        A = _dense(*_sparse_csr(case["n"], case["inside"], seed)[:3])
        return _filter_dense(A, None, _sparse_contour(case["ne"]), *_start(case["n"], case["m0"], seed))
    if kind == "batch":
        out = []
        sizes = _sizes(case, seed)
        for p, n in enumerate(sizes):
            if n > 2500:  # the dense eigenproblem of a larger one takes too long
                out.append({"lam": None, "X": None, "Xh": None})
                continue
            rp, ci, val, at = _sparse_csr(n, case["inside"], 100 * seed + p)
            lam, X, Xh = _inverse_iteration(_dense(rp, ci, val), at)
            out.append(_sorted_pairs(lam, X, Xh, _normal(17, n).to(torch.complex128)))
        return out
    return _net_exact(case, seed)
