"""Batched FGMRES (csrc/fgmres.cu) over its passes: row blocks with a remainder, several blocks a CTA, more systems than
a CTA's threads, several restart cycles.  The refinement ends at a column residual of inner_tol * ||y||, so column c of
Q is off by at most sum_j |w_j| ||M_j^{-1}|| inner_tol ||y_c||; M_j is diagonally dominant by rows and columns, with
||M_j^{-1}|| <= 1 / gap."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from paper_1506_04463_gb300 import workloads as wl  # noqa: E402
from gpu_helpers import dev, host  # noqa: E402

TOL = 1e-10


@pytest.mark.parametrize("n,m,ne,restart", [(7, 1, 2, 5), (8, 3, 4, 20), (9, 2, 4, 3), (333, 20, 16, 2), (1001, 12, 8, 30),
                                            (9737, 2, 2, 6)])
def test_filter(n, m, ne, restart):
    rng = np.random.default_rng(n)
    k = 3 * n
    i = rng.integers(0, n, k)
    A = sp.coo_matrix((rng.uniform(-1, 1, k) / 12, (i, (i + rng.integers(-4, 5, k)) % n)), shape=(n, n)).tocsr()
    off = max(abs(A).sum(0).max(), abs(A).sum(1).max())
    A = (A + sp.diags(rng.uniform(3, 6, n))).tocsr()
    con = wl.Contour(0, 0.0 + 0.2j, 1.0, ne=ne)
    ctx = F.FeastNH(A, None, con, m, precision=F.PREC_FP32_IR, inner_kind=F.INNER_FGMRES, inner_tol=TOL,
                    krylov_restart=restart)
    Y = [rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m)) for _ in range(2)]
    out = ctx.filter(dev(Y[0]), dev(Y[1]))
    z, w = F.nodes(con)
    gap = np.min(3 - abs(z)) - off
    assert gap > 0.3
    for side in range(2):
        ref = np.zeros((n, m), complex)
        for zj, wj in zip(z, w):
            M = (zj * sp.eye(n) - A).tocsc()
            lu = spl.splu(M if side == 0 else M.conj().T.tocsc())
            ref += (wj if side == 0 else np.conj(wj)) * lu.solve(Y[side])
        err = np.linalg.norm(host(out[side]) - ref, axis=0)
        assert np.all(err <= (TOL + 1e-13) * np.sum(abs(w)) / gap * np.linalg.norm(Y[side], axis=0)), side
