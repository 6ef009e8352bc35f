"""The single-precision multi-shift operator (csrc/spmm.cu) over its row groups: lanes a row, rows longer than a group,
empty rows, odd columns, nodes in several turns; bound by the rounding of FP32 sums."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from paper_1506_04463_gb300 import workloads as wl  # noqa: E402
from gpu_helpers import host  # noqa: E402


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("n,m,ne,per_row,cplx,withB", [
    (1, 1, 2, 1, False, False), (40, 2, 3, 2, True, False), (41, 7, 3, 30, False, False), (100, 8, 4, 4, False, True),
    (101, 10, 3, 4, True, True), (130, 16, 2, 6, False, False), (131, 17, 2, 12, True, False),
    (200, 33, 2, 70, False, True), (201, 34, 3, 40, True, False), (300, 66, 2, 5, False, False),
    (150, 40, 3, 3, True, False), (56000, 96, 3, 3, False, False), (56000, 96, 3, 7, False, False)])
def test_operator(side, n, m, ne, per_row, cplx, withB):
    rng = np.random.default_rng(n + m)

    def mat():
        k = n * per_row
        v = rng.standard_normal(k) + (1j * rng.standard_normal(k) if cplx else 0)
        M = sp.coo_matrix((v, (rng.integers(0, n, k), rng.integers(0, n, k))), shape=(n, n)).tocsr()
        M.sum_duplicates()
        return M

    A, B = mat(), (mat() if withB else None)
    con = wl.Contour(0, 0.3 + 0.1j, 1.5, ne=ne)
    ctx = F.FeastNH(A, B, con, m, precision=F.PREC_FP32_IR, inner_kind=F.INNER_FGMRES, krylov_restart=1)
    P = (rng.standard_normal((ne, n, m)) + 1j * rng.standard_normal((ne, n, m))).astype(np.complex64)
    V = host(ctx.multishift_spmm(torch.from_numpy(P).cuda(), side))
    z, _ = F.nodes(con)
    Ah, Bh = (A, B) if side == 0 else (A.conj().T.tocsr(), None if B is None else B.conj().T.tocsr())
    terms = 6 + np.max(np.diff(Ah.indptr)) + (np.max(np.diff(Bh.indptr)) if withB else 0)
    for j in range(ne):
        zj = z[j] if side == 0 else np.conj(z[j])
        Pj = P[j].astype(complex)
        bp, bm = (Bh @ Pj, abs(Bh) @ abs(Pj)) if withB else (Pj, abs(Pj))
        ref, mag = zj * bp - Ah @ Pj, abs(zj) * bm + abs(Ah) @ abs(Pj)
        assert np.all(abs(V[j] - ref) <= 4 * terms * 2.0 ** -24 * mag)
