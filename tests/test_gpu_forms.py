"""The fast forms that fall back to a general one where they fail (csrc/blocksolve.cu, csrc/tri.cu, csrc/eig.cu) were
really in use at the sizes where they can go wrong, and were left where they have to be: the results alone do not show
it.  Blocks of 160 and 176 rows split unevenly over the row groups of a product."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import scipy.sparse as sp  # noqa: E402

from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from paper_1506_04463_gb300 import workloads as wl  # noqa: E402
from gpu_helpers import dev, host, make_ctx  # noqa: E402
import test_gpu_small_eig  # noqa: E402
from test_gpu_solve_forms import TOL, _band, _run  # noqa: E402

SOLVES = F.FORM_TRIDIAGONAL | F.FORM_BLOCKS


@pytest.fixture
def made(monkeypatch):
    """The contexts that a helper creates."""
    ctxs = []

    class Recorded(F.FeastNH):
        def __init__(self, *a, **k):
            super().__init__(*a, **k)
            ctxs.append(self)

    monkeypatch.setattr(F, "FeastNH", Recorded)
    return ctxs


@pytest.mark.parametrize("prec", [F.PREC_FP32_IR, F.PREC_FP64])
@pytest.mark.parametrize("center", [4, 8])
@pytest.mark.parametrize("n,m,kl,ku,cplx,withB", [
    (2, 2, 1, 1, False, False), (31, 3, 1, 1, True, True), (65, 1, 0, 1, True, False), (1000, 7, 1, 1, False, False),
    (3, 1, 2, 2, False, False), (17, 17, 2, 2, False, True), (49, 9, 3, 17, False, False), (300, 33, 40, 40, True, True),
    (385, 4, 128, 100, False, False), (400, 20, 130, 129, True, False), (401, 3, 160, 150, False, False),
    (530, 18, 170, 176, True, True), (600, 12, 256, 250, False, True)])
def test_solves(made, prec, n, m, kl, ku, cplx, withB, center):
    """Nodes around 4, where the pencils are diagonally dominant; for the complex ones also around 8, their diagonal,
    as elsewhere: there a numpy emulation of the FP32 form has a first residual of 0.7 and 2.2 at the two sizes below
    (the triangular factors 0.8 and 0.2), above the 0.2 at which it is left."""
    if center == 8 and not cplx:
        pytest.skip("nodes on the real spectrum")
    A = _band(n, kl, ku, n, cplx)
    B = (sp.eye(n) + 0.1 * _band(n, kl, ku, n + 1, cplx) / 8).tocsr() if withB else None
    con = wl.Contour(1, 8 + 0j, 1.0, ratio=0.7, ne=6) if center == 8 else wl.Contour(0, 4 + 0j, 1.0, ne=8)
    assert _run(A, B, con, m, prec, dict(inner_tol=TOL), TOL) == F.OK
    left = prec == F.PREC_FP32_IR and center == 8 and (n, kl) in [(400, 130), (530, 170)]
    form = F.FORM_TRIDIAGONAL if max(kl, ku) <= 1 else F.FORM_BLOCKS
    assert made[0].forms() & SOLVES == (0 if left else form)


@pytest.mark.parametrize("prec,inner_max", [(F.PREC_FP64, 1), (F.PREC_FP64, 4), (F.PREC_FP32_IR, 5)])
@pytest.mark.parametrize("bw", [1, 20])
def test_solves_left(made, prec, inner_max, bw):
    con = wl.Contour(0, 4 + 0j, 1.0, ne=8)
    opts = dict(inner_tol=1e-30, inner_max=inner_max)
    assert _run(_band(200, bw, bw, 3, False), None, con, 6, prec, opts, 1e-12) == F.EINNER
    assert made[0].forms() & SOLVES == 0


def test_solves_not_taken(made):
    con = wl.Contour(0, 4 + 0j, 1.0, ne=8)
    assert _run(_band(150, 30, 30, 5, False, per_row=40), None, con, 6, F.PREC_FP32_IR, dict(inner_tol=TOL), TOL) == F.OK
    assert made[0].forms() & SOLVES == 0


@pytest.mark.parametrize("kind,m,refined", [
    ("random", 3, False), ("random", 4, True), ("random", 31, True), ("random", 65, True), ("random", 97, True),
    ("random", 112, True), ("random", 113, True), ("diagonal", 40, True), ("clustered", 32, False),
    ("graded", 48, False), ("random", 4, True)])
def test_small_eigenproblem(kind, m, refined):
    ctx = make_ctx(wl.pencil_workload(40, 3, ne=8, m0=8))
    ctx.small_eig(dev(test_gpu_small_eig._matrix(kind, m)))
    assert bool(ctx.forms() & F.FORM_EIG_REFINED) == refined
    ctx.close()


@pytest.mark.parametrize("m", [1, 7, 8, 9, 33, 64])
def test_rayleigh_ritz(made, monkeypatch, m):
    monkeypatch.setattr(F.FeastNH, "close", lambda self: None)  # still open for the query
    test_gpu_small_eig.test_rayleigh_ritz_sizes(m)
    small = F.FORM_ELIMINATION | F.FORM_NEAR_IDENTITY | (F.FORM_EIG_REFINED if m >= 4 else 0)
    assert made[0].forms() & ~SOLVES == small


@pytest.mark.parametrize("bw,m,ne,blocks", [(4, 64, 14, True), (4, 64, 15, False), (90, 24, 25, True), (96, 32, 28, True),
                                            (97, 32, 19, True), (97, 32, 20, False), (256, 128, 16, False)])
def test_fp64_blocks_by_rounds(bw, m, ne, blocks):
    """The FP64 rule at its line on a chip of 152 SMs: CTAs of four columns, two sides, three rounds for blocks of up to
    96 rows and two for larger ones; the filter is right either way."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line depends on the number of SMs")
    n = 700
    A = _band(n, bw, bw, bw, False)
    con = wl.Contour(0, 4 + 0.1j, 1.0, ne=ne)
    ctx = F.FeastNH(A, None, con, m, precision=F.PREC_FP64, inner_tol=TOL)
    Y = np.random.default_rng(1).standard_normal((n, m))
    Q, _ = ctx.filter(dev(Y), dev(Y))
    assert (ctx.forms() & SOLVES == F.FORM_BLOCKS) == blocks
    ctx.close()
    z, w = F.nodes(con)
    ref, amp = 0, 0.0
    for zj, wj in zip(z, w):
        inv = np.linalg.inv(zj * np.eye(n) - A.toarray())
        ref, amp = ref + wj * (inv @ Y), amp + abs(wj) * np.linalg.norm(inv, 2)
    err = np.linalg.norm(host(Q) - ref, axis=0)
    assert np.all(err <= (TOL + 1e-13) * amp * np.linalg.norm(Y, axis=0))
