"""V^{-1} of the refined small eigensolver (csrc/eig.cu), which the left Ritz vectors are formed with."""
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


@pytest.mark.parametrize("m", [32, 64])
def test_left_vectors_of_ill_conditioned_pairs(m):
    """Eigenvectors of condition 4000: Yh^H B Y = W X of the reduced problem, where W is refined towards X^{-1}.  An
    entry is a sum over a row of W and a unit column of X, rounded to eps |W| <= eps cond(X); four times that.  (From
    the right defect I - X W the remainder is 8 to 12 eps cond in a numpy
    emulation, from the left one 0.1, with an FP64 inverse 0.4.)"""
    rng = np.random.default_rng(m)
    Q1, Q2 = (np.linalg.qr(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)))[0] for _ in range(2))
    X = Q1 @ np.diag(4000.0 ** -np.linspace(0, 1, m)) @ Q2
    X /= np.linalg.norm(X, axis=0)
    lam = rng.standard_normal(m) + 1j * rng.standard_normal(m)
    A = sp.csr_matrix(X @ np.diag(lam) @ np.linalg.inv(X))
    ctx = F.FeastNH(A, None, wl.Contour(0, 0j, 4.0, ne=4), m, projection=F.PROJ_FP64)
    eye = dev(np.eye(m))
    _, Y, Yh, _ = ctx.rr(eye, eye)
    assert ctx.forms() & F.FORM_EIG_REFINED
    ctx.close()
    cond = np.linalg.cond(np.linalg.eig(A.toarray())[1])
    assert np.max(np.abs(host(Yh).conj().T @ host(Y) - np.eye(m))) < 4 * 2.3e-16 * cond
