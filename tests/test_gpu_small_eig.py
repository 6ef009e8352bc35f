"""The refined small eigensolver (csrc/eig.cu) where its rules change route: the smallest sizes, the ends of the lanes'
columns, Z in and out of shared memory, and spectra that the refinement does not separate (FP64 QR)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from paper_1506_04463_gb300 import workloads as wl  # noqa: E402
from gpu_helpers import dev, host, make_ctx, match_rel  # noqa: E402


def _matrix(kind, m):
    rng = np.random.default_rng(m)
    R = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    if kind == "random":
        return R
    if kind == "diagonal":
        return np.diag(np.arange(m) + 1.0).astype(complex)
    if kind == "scaled":  # rows and columns over 16 orders
        s = 10.0 ** np.linspace(-8, 8, m)
        return R * s[:, None] / s[None, :]
    X = np.linalg.qr(R)[0]
    if kind == "close":  # gaps of 1e-4 of the spectrum's position
        d = 0.02 * (1 + 1e-4 * np.arange(m))
    elif kind == "clustered":
        d = np.r_[np.ones(m // 2), np.linspace(0.1, 0.5, m - m // 2)]
    else:  # graded
        d = 10.0 ** -np.linspace(0, 12, m)
    return X @ np.diag(d) @ X.conj().T


@pytest.mark.parametrize("kind,m", [("random", 3), ("random", 4), ("random", 31), ("random", 65), ("random", 97),
                                    ("random", 112), ("random", 113), ("diagonal", 40), ("scaled", 33), ("close", 64),
                                    ("clustered", 32), ("graded", 48), ("random", 1), ("random", 2)])
def test_pairs(kind, m):
    M = _matrix(kind, m)
    ctx = make_ctx(wl.pencil_workload(40, 3, ne=8, m0=8))
    lam, V = (host(t) for t in ctx.small_eig(dev(M)))
    nrm = np.linalg.norm(M, 2)
    # the residual of a backward-stable solver is a small multiple of m eps ||M||
    assert np.max(np.linalg.norm(M @ V - V * lam, axis=0)) < 20 * m * 2.3e-16 * nrm
    assert np.max(np.abs(np.linalg.norm(V, axis=0) - 1)) < 1e-14
    if kind != "scaled":
        assert match_rel(lam, np.linalg.eigvals(M), nrm) < 1e-12
    else:  # eigenvalues of the balanced matrix
        s = 10.0 ** np.linspace(-8, 8, m)
        assert match_rel(lam, np.linalg.eigvals(M / s[:, None] * s[None, :]), m) < 1e-12
    ctx.close()


@pytest.mark.parametrize("m", [1, 7, 8, 9, 33, 64])
def test_rayleigh_ritz_sizes(m):
    # B_Q eliminated on a cluster of eight CTAs: fewer columns than CTAs, ragged and full ones
    N = 12
    A = wl.convdiff2d(N)
    lam = wl.convdiff2d_eigs(N)
    con = wl.Contour(1, complex(0.5 * (lam[0] + lam[m - 1])), 0.6 * (lam[m - 1] - lam[0]) + 0.01, ratio=0.5, ne=8)
    ctx = F.FeastNH(A, None, con, m)
    w, X = np.linalg.eig(A.toarray())
    o = np.argsort(w.real)[:m]
    X = X[:, o]
    Xh = np.linalg.inv(np.linalg.eig(A.toarray())[1]).conj().T[:, o]
    rng = np.random.default_rng(m)
    C, Ch = (np.eye(m) + 0.3 / np.sqrt(m) * rng.standard_normal((m, m)) for _ in range(2))
    ritz, Y, Yh, info = ctx.rr(dev(X @ C), dev(Xh @ Ch))
    assert info["m_tilde"] == m
    assert match_rel(host(ritz), w[o], 1.0) < 1e-12
    assert np.max(np.abs(host(Yh).conj().T @ host(Y) - np.eye(m))) < 1e-11
    ctx.close()
