"""Shifted solves by chunked tridiagonal recurrences (csrc/tri.cu) and by inverted diagonal blocks
(csrc/blocksolve.cu), and the way back to the triangular factors, against dense solves.

Bound: every node's system is solved to a column residual of inner_tol * ||B y||, so column c of Q is off by at most
sum_j |w_j| ||M_j^{-1}|| inner_tol ||B y_c||, and by 1e-13 of the same sum without inner_tol for the rest."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from paper_1506_04463_gb300 import workloads as wl  # noqa: E402
from gpu_helpers import dev, host  # noqa: E402

TOL = 1e-10


def _band(n, kl, ku, seed, cplx, per_row=3):
    """Band edges filled, a few entries a row in between, diagonally dominant by rows and columns."""
    rng = np.random.default_rng(seed)
    offs = sorted({-kl, ku} | set(rng.integers(-kl, ku + 1, per_row)) - {0})
    val = lambda k: rng.standard_normal(k) + (1j * rng.standard_normal(k) if cplx else 0)  # noqa: E731
    return sp.diags([val(n - abs(o)) for o in offs], offs, shape=(n, n)).tocsr() + 8 * sp.eye(n)


def _run(A, B, con, m, prec, opts, tol):
    n = A.shape[0]
    rng = np.random.default_rng(n + m)
    Y = [rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m)) for _ in range(2)]
    ctx = F.FeastNH(A, B, con, m, precision=prec, **opts)
    out = [torch.empty((n, m), dtype=torch.complex128, device="cuda") for _ in range(2)]
    yd = [dev(y) for y in Y]
    st = F.lib().feast_nh_filter(ctx.h, *(F._ptr(t) for t in yd + out), m)
    z, w = F.nodes(con)
    Ad, Bd = A.toarray().astype(complex), np.eye(n) if B is None else B.toarray()
    for side in range(2):
        C = (lambda M: M.conj().T) if side else (lambda M: M)
        R = C(Bd) @ Y[side]
        ref, amp = np.zeros_like(R), 0.0
        for zj, wj in zip(z, w):
            inv = np.linalg.inv(C(zj * Bd - Ad))
            wj = np.conj(wj) if side else wj
            ref += wj * (inv @ R)
            amp += abs(wj) * np.linalg.norm(inv, 2)
        err = np.linalg.norm(host(out[side]) - ref, axis=0)
        assert np.all(err <= (tol + 1e-13) * amp * np.linalg.norm(R, axis=0)), (side, err.max())
    return st


@pytest.mark.parametrize("prec", [F.PREC_FP32_IR, F.PREC_FP64])
@pytest.mark.parametrize("n,m,kl,ku,cplx,withB", [
    (1, 1, 0, 0, True, False), (2, 2, 1, 1, False, False), (31, 3, 1, 1, True, True), (32, 4, 1, 0, False, False),
    (33, 5, 1, 1, False, True), (65, 1, 0, 1, True, False), (1000, 7, 1, 1, False, False)])
def test_tridiagonal(prec, n, m, kl, ku, cplx, withB):
    if kl + ku == 0:
        A = sp.csr_matrix(np.array([[0.3 + 0.2j]]))
    else:
        A = _band(n, kl, ku, n, cplx)
    B = (sp.eye(n) + 0.1 * _band(n, kl, ku, n + 1, cplx) / 8).tocsr() if withB else None
    con = wl.Contour(1, 8 + 0j, 1.0, ratio=0.7, ne=6) if cplx else wl.Contour(0, 5 + 0j, 1.0, ne=8)
    assert _run(A, B, con, m, prec, dict(inner_tol=TOL), TOL) == F.OK


@pytest.mark.parametrize("prec", [F.PREC_FP32_IR, F.PREC_FP64])
@pytest.mark.parametrize("n,m,kl,ku,cplx,withB", [
    (3, 1, 2, 2, False, False),       # one block, mostly padding
    (16, 3, 2, 1, True, False),       # one block, full
    (17, 17, 2, 2, False, True),      # a second block of one row
    (64, 5, 16, 3, True, False),      # block = kl, whole blocks
    (49, 9, 3, 17, False, False),     # blocks of 32, ku > kl
    (300, 33, 40, 40, True, True),    # columns beyond a CTA's
    (385, 4, 128, 100, False, False),  # last block of one row, largest of one row group
    (400, 20, 130, 129, True, False),  # two row groups, some past the end
    (600, 12, 256, 250, False, True)])  # largest block
def test_blocks(prec, n, m, kl, ku, cplx, withB):
    A = _band(n, kl, ku, n, cplx)
    B = (sp.eye(n) + 0.1 * _band(n, kl, ku, n + 1, cplx) / 8).tocsr() if withB else None
    con = wl.Contour(1, 8 + 0j, 1.0, ratio=0.7, ne=6) if cplx else wl.Contour(0, 4 + 0j, 1.0, ne=8)
    assert _run(A, B, con, m, prec, dict(inner_tol=TOL), TOL) == F.OK


@pytest.mark.parametrize("prec,inner_max,tol", [(F.PREC_FP64, 1, 1e-12), (F.PREC_FP32_IR, 5, 1e-12)])
@pytest.mark.parametrize("bw", [1, 20])
def test_steps_used_up(prec, inner_max, tol, bw):
    """A tolerance that nothing reaches: the triangular factors take over and give their own best, EINNER as before."""
    A = _band(200, bw, bw, 3, False)
    con = wl.Contour(0, 4 + 0j, 1.0, ne=8)
    assert _run(A, None, con, 6, prec, dict(inner_tol=1e-30, inner_max=inner_max), tol) == F.EINNER


def test_many_entries_a_row():
    """More entries a row than the block form takes: triangular factors."""
    A = _band(150, 30, 30, 5, False, per_row=40)
    con = wl.Contour(0, 4 + 0j, 1.0, ne=8)
    assert _run(A, None, con, 6, F.PREC_FP32_IR, dict(inner_tol=TOL), TOL) == F.OK
