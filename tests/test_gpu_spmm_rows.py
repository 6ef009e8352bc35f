"""The single-precision multi-shift operator with a warp a row (csrc/spmm.cu): rows of up to seven and of ten to sixteen
entries, more than 32 columns, even and odd, all nodes at once and in turns; bound by the rounding of FP32 sums."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from paper_1506_04463_gb300 import workloads as wl  # noqa: E402
import test_gpu_spmm_groups  # noqa: E402
from gpu_helpers import host  # noqa: E402


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("n,m,ne,per_row,span,cplx", [
    (34, 33, 2, 6, 5, False), (41, 34, 3, 7, 9, True), (90, 65, 2, 6, 10, False), (91, 35, 2, 7, 20, True),
    (67, 66, 3, 12, 12, False), (51, 47, 2, 16, 18, True), (130, 128, 2, 14, 30, True), (70, 63, 4, 16, 17, False),
    (20000, 49, 8, 7, 8000, False), (20000, 48, 8, 13, 8000, False), (20000, 35, 8, 16, 8000, True), (60000, 64, 2, 14, 20000, False),
    (60000, 65, 2, 14, 20000, False), (60000, 96, 2, 7, 20000, False)])
def test_rows(side, n, m, ne, per_row, span, cplx):
    rng = np.random.default_rng(n + m)
    # every row and every column has per_row entries but at the ends of the band
    offs = np.unique(np.r_[-span, span, 0, rng.choice(np.arange(1, span), max(0, per_row - 3), replace=False)])[:per_row]
    val = lambda k: rng.standard_normal(k) + (1j * rng.standard_normal(k) if cplx else 0)  # noqa: E731
    A = sp.diags([val(n - abs(o)) for o in offs], offs, shape=(n, n)).tocsr()
    m0 = min(m, n)
    con = wl.Contour(0, 0.3 + 0.1j, 1.5, ne=ne)
    ctx = F.FeastNH(A, None, con, m0, precision=F.PREC_FP32_IR, inner_kind=F.INNER_FGMRES, krylov_restart=1)
    P = (rng.standard_normal((ne, n, m0)) + 1j * rng.standard_normal((ne, n, m0))).astype(np.complex64)
    V = host(ctx.multishift_spmm(torch.from_numpy(P).cuda(), side))
    z, _ = F.nodes(con)
    Ah = A if side == 0 else A.conj().T.tocsr()
    for j in range(ne):
        zj = z[j] if side == 0 else np.conj(z[j])
        Pj = P[j].astype(complex)
        ref, mag = zj * Pj - Ah @ Pj, abs(zj) * abs(Pj) + abs(Ah) @ abs(Pj)
        assert np.all(abs(V[j] - ref) <= 4 * (6 + per_row) * 2.0 ** -24 * mag)
    ctx.close()


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("n,m,ne,per_row,cplx,withB", [
    (300, 1, 2, 60, False, False), (301, 8, 3, 200, True, False), (300, 13, 2, 90, False, True), (3648, 7, 2, 18, False, False),
    (3649, 7, 2, 18, False, False)])
def test_few_long_rows(side, n, m, ne, per_row, cplx, withB):
    """Sixteen lanes a row for few columns."""
    test_gpu_spmm_groups.test_operator(side, n, m, ne, per_row, cplx, withB)
