"""Shifted solves at the ends of what the block form accepts (csrc/blocksolve.cu)."""
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


@pytest.mark.parametrize("prec", [F.PREC_FP32_IR, F.PREC_FP64])
def test_more_blocks_than_a_grid_has_rows(prec):
    """Blocks of 16 rows, 65537 of them: more than the y and z extents of a grid take.  Entries below 0.2 off a
    diagonal of 8, nodes at distance one from 4: ||M^{-1}|| <= 1 / (8 - 4 - 1 - 0.8) by rows and by columns, and the
    two weights have modulus 1/2."""
    n, m = 16 * 65536 + 1, 1
    rng = np.random.default_rng(5)
    A = (sp.diags([0.2 * rng.uniform(-1, 1, n - abs(o)) for o in (-2, -1, 1, 2)], (-2, -1, 1, 2)) + 8 * sp.eye(n)).tocsr()
    con = wl.Contour(0, 4 + 0j, 1.0, ne=2)
    Y = [rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m)) for _ in range(2)]
    ctx = F.FeastNH(A, None, con, m, precision=prec, inner_tol=TOL)
    out = [host(t) for t in ctx.filter(*(dev(y) for y in Y))]
    ctx.close()
    z, w = F.nodes(con)
    lu = [spl.splu((zj * sp.eye(n) - A).tocsc()) for zj in z]
    for side in range(2):
        ref = sum((np.conj(wj) if side else wj) * f.solve(Y[side], trans="H" if side else "N") for f, wj in zip(lu, w))
        err = np.linalg.norm(out[side] - ref, axis=0)
        assert np.all(err <= (TOL + 1e-13) / 2.2 * np.linalg.norm(Y[side], axis=0)), (side, err.max())


@pytest.mark.parametrize("prec", [F.PREC_FP32_IR, F.PREC_FP64])
@pytest.mark.parametrize("bw", [1, 20])
def test_no_memory_for_the_triangular_factors(prec, bw):
    """A tolerance that nothing reaches sends a filter back to the triangular factors; their workspace fails.  The call
    says so, and the next one asks for it again and gives the filter (||M^{-1}|| <= 1 as the bands below are diagonally
    dominant: 8 - 5 - 2)."""
    n, m = 200, 6
    rng = np.random.default_rng(bw)
    A = (sp.diags([rng.uniform(-1, 1, n - bw) for _ in range(2)], (-bw, bw)) + 8 * sp.eye(n)).tocsr()
    con = wl.Contour(0, 4 + 0j, 1.0, ne=8)
    Y = [rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m)) for _ in range(2)]
    ctx = F.FeastNH(A, None, con, m, precision=prec, inner_tol=1e-30, inner_max=5)
    out = [torch.empty((n, m), dtype=torch.complex128, device="cuda") for _ in range(2)]
    blocks = [dev(y) for y in Y] + out
    ptrs = [F._ptr(t) for t in blocks]
    assert F.lib().feast_nh_inject_device_error(ctx.h, F.INJECT_NOMEM) == F.OK
    assert F.lib().feast_nh_filter(ctx.h, *ptrs, m) == F.ENOMEM
    z, w = F.nodes(con)
    for _ in range(2):
        assert F.lib().feast_nh_filter(ctx.h, *ptrs, m) == F.EINNER
        for side in range(2):
            ref = 0
            for zj, wj in zip(z, w):
                M = zj * np.eye(n) - A.toarray()
                ref = ref + (np.conj(wj) * np.linalg.solve(M.conj().T, Y[1]) if side else wj * np.linalg.solve(M, Y[0]))
            err = np.linalg.norm(host(out[side]) - ref, axis=0)
            assert np.all(err <= 1e-12 * np.linalg.norm(Y[side], axis=0) * np.sum(np.abs(w)))
    ctx.close()



@pytest.mark.parametrize("inner_max", [1, 12])
def test_tridiagonal_fp64_residual(inner_max):
    """Three pivots of 1e-5, so that the chunked recurrences alone leave a residual of 5e-13 to 2e-12 (emulated in
    numpy): below inner_tol, but far above a refined solve's, eps (|M| |x| + |y|) / |y| = 1e-15 here.  One node with
    weight one: Q is the solution itself.  With a single step the triangular factors are taken, whose growth by the
    small pivots is eps / 1e-5."""
    n, m = 500, 3
    rng = np.random.default_rng(2)
    lo, up, di = rng.uniform(0.5, 1, n), rng.uniform(0.5, 1, n), 4 + rng.uniform(0, 1, n)
    d = di[0]
    for r in range(1, n):
        d = di[r] - lo[r] / d * up[r - 1]
        if r in (100, 250, 400):
            di[r] += 1e-5 - d
            d = 1e-5
    A = sp.diags([lo[1:], di, up[:-1]], [-1, 0, 1]).tocsr()
    con = wl.Contour(2, 0j, 1.0, z=np.array([0j]), w=np.array([1 + 0j]))
    Y = [rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m)) for _ in range(2)]
    ctx = F.FeastNH(A, None, con, m, precision=F.PREC_FP64, inner_tol=TOL, inner_max=inner_max)
    Q = [host(t) for t in ctx.filter(*(dev(y) for y in Y))]
    assert bool(ctx.forms() & F.FORM_TRIDIAGONAL) == (inner_max > 1)
    ctx.close()
    for C, y, q in zip((A, A.T), Y, Q):
        res = np.linalg.norm(y + C @ q, axis=0) / np.linalg.norm(y, axis=0)
        assert np.all(res <= (5e-15 if inner_max > 1 else 2.3e-11)), res


def test_single_step_fp64_blocks():
    """No step left to refine solves by inverted blocks: triangular factors."""
    n, m = 200, 4
    rng = np.random.default_rng(3)
    A = (sp.diags([rng.uniform(-1, 1, n - 20) for _ in range(2)], (-20, 20)) + 8 * sp.eye(n)).tocsr()
    ctx = F.FeastNH(A, None, wl.Contour(0, 4 + 0j, 1.0, ne=4), m, precision=F.PREC_FP64, inner_tol=TOL, inner_max=1)
    ctx.filter(*(dev(rng.standard_normal((n, m))) for _ in range(2)))
    assert ctx.forms() & (F.FORM_TRIDIAGONAL | F.FORM_BLOCKS) == 0
    ctx.close()


def test_no_room_for_the_inverses():
    """Memory for the factors and all other workspace, but not for the inverted blocks: the context is created all the
    same, with the triangular factors, and filters like one that has them (both to TOL; ||M^{-1}|| <= 1 / (8 - 5 - 2),
    the sum of the weights' moduli is 1).  In FP64 they come on top of all that the triangular factors need."""
    n, m, bw, ne = 40000, 4, 64, 8
    rng = np.random.default_rng(9)
    A = (sp.diags([rng.uniform(-1, 1, n - bw) for _ in range(2)], (-bw, bw)) + (8 + 0j) * sp.eye(n)).tocsr()
    con = wl.Contour(0, 4 + 0j, 1.0, ne=ne)
    Y = [dev(rng.standard_normal((n, m))) for _ in range(2)]
    inverse = ne * n * bw * 16  # one of the two copies

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        F.release_memory()
        return torch.cuda.mem_get_info()[0]

    before = free()
    ctx = F.FeastNH(A, None, con, m, precision=F.PREC_FP64, inner_tol=TOL)
    assert ctx.forms() & F.FORM_BLOCKS
    ref = [host(q) for q in ctx.filter(*Y)]
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    ctx.close()
    filler = torch.empty(free() - (used - inverse), dtype=torch.uint8, device="cuda")
    try:
        ctx = F.FeastNH(A, None, con, m, precision=F.PREC_FP64, inner_tol=TOL)
        assert ctx.forms() & F.FORM_BLOCKS == 0
        out = [host(q) for q in ctx.filter(*Y)]
        ctx.close()
    finally:
        del filler
        free()
    for a, b, y in zip(out, ref, Y):
        assert np.all(np.linalg.norm(a - b, axis=0) <= 2 * (TOL + 1e-13) * np.linalg.norm(host(y), axis=0))


@pytest.mark.parametrize("prec,n,bw,m,ne,far", [
    (F.PREC_FP64, 8000, 208, 8, 4, 1), (F.PREC_FP64, 8000, 224, 8, 4, 1), (F.PREC_FP64, 8000, 112, 16, 8, 1),
    (F.PREC_FP64, 4000, 48, 32, 8, 1), (F.PREC_FP32_IR, 5000, 240, 64, 8, 8)])
def test_odd_number_of_stages(prec, n, bw, m, ne, far):
    """Three stages (FP64) and five (FP32, blocks of 240 with eight entries towards a neighbour), which the two groups
    of a product use in turns, some warps without rows of their own: bit-identical results, filter after filter, by a
    solve that needs no other form."""
    rng = np.random.default_rng(bw)
    offs = [o for k in range(far) for o in (bw - k, k - bw)] + ([1, -7] if far < 7 else [])  # at most eight either way
    A = (sp.diags([rng.uniform(-1, 1, n - abs(o)) for o in offs], offs) + (6 + len(offs)) * sp.eye(n)).tocsr()
    con = wl.Contour(0, 4 + 0.1j, 1.0, ne=ne)
    Y = [dev(rng.standard_normal((n, m))) for _ in range(2)]
    ctx = F.FeastNH(A, None, con, m, precision=prec, inner_tol=TOL)
    ref = [q.clone() for q in ctx.filter(*Y)]
    for _ in range(6):
        assert all(torch.equal(a, b) for a, b in zip(ctx.filter(*Y), ref))
    assert ctx.forms() & F.FORM_BLOCKS
    ctx.close()
