"""The multi-shift residual (csrc/spmm.cu) where its row chunks change: one row, chunk ends, rows too long to be staged,
rows without a diagonal entry; bound by the rounding of the sums in FP64 (and of the result in FP32)."""
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


@pytest.mark.parametrize("single", [False, True])
@pytest.mark.parametrize("n,m,ne,density,cplx,withB,diag", [
    (1, 1, 1, 1.0, False, False, True), (7, 3, 4, 0.4, True, False, True), (8, 8, 40, 0.5, False, False, False),
    (9, 5, 3, 0.9, True, True, True), (60, 60, 32, 0.6, False, False, True), (61, 33, 15, 0.9, True, False, False),
    (2500, 6, 8, 0.002, False, True, True), (2503, 11, 8, 0.002, True, False, False)])
def test_residual(single, n, m, ne, density, cplx, withB, diag):
    rng = np.random.default_rng(n * 7 + m)

    def mat():
        M = sp.random(n, n, density, random_state=rng, data_rvs=rng.standard_normal).tocsr()
        if cplx:
            M = (M + 1j * M.multiply(M)).tocsr()
        return (M + 3 * sp.eye(n)).tocsr() if diag else (M - sp.diags(M.diagonal())).tocsr()

    A, B = mat(), (mat() if withB else None)
    if A.nnz == 0:
        A = sp.eye(n).tocsr()
    A.eliminate_zeros()
    con = wl.Contour(0, 0.3 + 0.1j, 1.5, ne=ne)
    ctx = F.FeastNH(A, B, con, m, precision=F.PREC_FP32_IR, inner_kind=F.INNER_FGMRES, krylov_restart=1)
    X = rng.standard_normal((ne, n, m)) + 1j * rng.standard_normal((ne, n, m))
    BY = rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m))
    R, Q = ctx.multishift_residual(dev(X), dev(BY), True, single)
    R, Q = host(R).reshape(ne, n, m), host(Q)
    z, w = F.nodes(con)
    terms = 8 + np.max(np.diff(A.indptr)) + (np.max(np.diff(B.indptr)) if withB else 0)
    eps = np.finfo(float).eps
    qref, qabs = np.zeros((n, m), complex), np.zeros((n, m))
    for j in range(ne):
        bx = B @ X[j] if withB else X[j]
        babs = abs(B) @ abs(X[j]) if withB else abs(X[j])
        ref = BY - z[j] * bx + A @ X[j]
        mag = abs(BY) + abs(z[j]) * babs + abs(A) @ abs(X[j])
        bound = 4 * terms * eps * mag + (2.0 ** -23 * abs(ref) if single else 0)
        assert np.all(abs(R[j] - ref) <= bound)
        qref += w[j] * X[j]
        qabs += abs(w[j] * X[j])
    assert np.all(abs(Q - qref) <= 4 * (ne + 2) * eps * qabs)
