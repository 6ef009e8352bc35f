"""The banded factorisation's panel steps in FP64 (csrc/band.cu) over the tiles of the trailing update and the columns
of U12: filters against dense solves.  Bound: the solves are refined to inner_tol, so column c of Q is off by at most
sum_j |w_j| ||M_j^{-1}|| inner_tol ||y_c||; the pivots are those of diagonally dominant matrices."""
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

TOL = 1e-12


@pytest.mark.parametrize("n,kl,ku,ne", [(18, 2, 2, 2), (33, 16, 15, 2), (50, 17, 33, 4), (200, 63, 70, 4), (330, 130, 100, 16),
                                        (450, 200, 220, 32)])
def test_filter(n, kl, ku, ne):
    rng = np.random.default_rng(n)
    A = np.triu(np.tril(rng.uniform(-1, 1, (n, n)), ku), -kl) / (kl + ku) + np.diag(rng.uniform(3, 5, n))
    con = wl.Contour(0, 0.1 + 0.2j, 1.0, ne=ne)
    ctx = F.FeastNH(sp.csr_matrix(A), None, con, 3, precision=F.PREC_FP64, inner_tol=TOL)
    Y = [rng.standard_normal((n, 3)) + 1j * rng.standard_normal((n, 3)) for _ in range(2)]
    out = ctx.filter(dev(Y[0]), dev(Y[1]))
    z, w = F.nodes(con)
    for side in range(2):
        ref, amp = np.zeros((n, 3), complex), 0.0
        for zj, wj in zip(z, w):
            inv = np.linalg.inv(zj * np.eye(n) - A)
            inv, wj = (inv, wj) if side == 0 else (inv.conj().T, np.conj(wj))
            ref += wj * (inv @ Y[side])
            amp += abs(wj) * np.linalg.norm(inv, 2)
        err = np.linalg.norm(host(out[side]) - ref, axis=0)
        assert np.all(err <= (TOL + 1e-13) * amp * np.linalg.norm(Y[side], axis=0)), side
