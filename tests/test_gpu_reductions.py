"""Sums of per-CTA partials (csrc/reduce.cuh) and the Jacobi quotients, at the sizes where a loop or a tile ends:
one partial, fewer than the threads of an output, and several rounds of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from oracle import feast_nh as OF  # noqa: E402
from oracle.contour import contour_nodes  # noqa: E402
from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from paper_1506_04463_gb300 import workloads as wl  # noqa: E402
from gpu_helpers import dev, host  # noqa: E402


@pytest.mark.parametrize("n,m", [(1, 1), (63, 3), (65, 4), (4097, 5), (40000, 7)])
def test_residual_norms(n, m):
    # ||R_jc|| / ||BY_c|| against the definition; the sums have at most 608 partials of FP64 terms
    ne = 3
    A = wl.tridiag_toeplitz(n, 1.0, 2.0, 0.5) if n > 1 else wl.sp.csr_matrix(np.array([[2.0]]))
    con = wl.Contour(0, 2.0 + 0.1j, 0.3, ne=ne)
    rng = np.random.default_rng(n)
    X = rng.standard_normal((ne, n, m)) + 1j * rng.standard_normal((ne, n, m))
    BY = rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m))
    R, _, rel = F.multishift_residual_noalloc(F.csr_to_device(A), None, con, dev(X), dev(BY))
    z, w = contour_nodes(con)
    Ro, _ = OF.shifted_residuals(A, None, z, w, X, BY)
    ref = np.linalg.norm(Ro, axis=1) / np.linalg.norm(BY, axis=0)[None, :]
    assert np.max(np.abs(host(rel) - ref) / ref) < 1e-13


@pytest.mark.parametrize("n,m0", [(40, 3), (700, 11)])
def test_fgmres_filter(n, m0):
    # the filter through the batched dots and Jacobi quotients, against exact node solves
    A = wl.random_sparse(n, 5)
    con = wl.Contour(0, 9.0 + 0j, 1.5, ne=4)
    Y, Yh = wl.start_block(n, m0, 0), wl.start_block(n, m0, 1)
    ctx = F.FeastNH(A, None, con, m0, precision=F.PREC_FP32_IR, inner_kind=F.INNER_FGMRES)
    Q, Qh = ctx.filter(dev(Y), dev(Yh))
    z, w = contour_nodes(con)
    Qo, Qho = OF.contour_integration(A, None, OF.node_solvers(A, None, z), z, w, Y, Yh)
    # every system is solved to a relative residual of 1e-10 and |z - lambda| > 1 on this contour
    assert np.max(np.abs(host(Q) - Qo)) < 1e-8 * np.max(np.abs(Qo))
    assert np.max(np.abs(host(Qh) - Qho)) < 1e-8 * np.max(np.abs(Qho))
    ctx.close()
