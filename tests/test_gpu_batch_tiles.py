"""Batched contour integration (csrc/batch.cu): rows that fit the staged tiles and rows that do not (one dense row), real
and complex values, problem sizes that leave ragged tiles, both sweep precisions."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from paper_1506_04463_gb300 import workloads as wl  # noqa: E402
from gpu_helpers import dev, host, match_rel  # noqa: E402


def _problem(n, seed, cplx, dense_row):
    rng = np.random.default_rng(seed)
    A = sp.random(n, n, density=4.0 / n, random_state=rng, format="lil", data_rvs=lambda k: 0.2 * rng.standard_normal(k))
    if cplx:
        A = (A + 0.1j * sp.random(n, n, density=2.0 / n, random_state=rng, format="lil")).tolil()
    if dense_row:
        A[n // 2, :] = 0.01 * rng.standard_normal(n)
    d = rng.uniform(0.0, 3.0, n)
    d[rng.choice(n, 6, replace=False)] = 6.0 + 0.3 * np.arange(6)
    A.setdiag(d)
    return A.tocsr()


@pytest.mark.parametrize("prec", [F.PREC_FP32_IR, F.PREC_FP64])
@pytest.mark.parametrize("cplx,dense_row", [(False, False), (False, True), (True, False), (True, True)])
def test_eigenvalues(prec, cplx, dense_row):
    sizes = [61, 256, 415]
    A = [_problem(n, n + 7 * cplx, cplx, dense_row) for n in sizes]
    con = wl.Contour(0, 6.75 + 0j, 1.4, ne=8)
    m0 = 11
    ctx = F.FeastBatch(A, [con] * 3, m0, precision=prec, inner_tol=1e-12, krylov_max=500)
    n = sum(sizes)
    out = ctx.solve(dev(wl.start_block(n, m0, 0)), dev(wl.start_block(n, m0, 1)))
    assert out["status"] == F.OK
    for Ap, p in zip(A, out["problems"]):
        ev = np.linalg.eigvals(Ap.toarray())
        inside = ev[np.abs(ev - con.center) <= con.r]
        assert p["m"] == inside.size == 6
        # residuals below 1e-10 of well-conditioned eigenvalues
        assert match_rel(host(p["lam"]), inside, 1.0) < 1e-9
        assert float(p["res"].max()) < 1e-10
    ctx.close()
