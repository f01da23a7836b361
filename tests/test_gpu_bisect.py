"""Eigenvalues by bisection and eigenvectors by twisted factorisations (inverse
iteration for the ones these leave).  Bisection: the bracket's points are placed by
an FP32 estimate, by a secant or evenly.  Vectors: 4 to 16 per block, in shared or
global memory, alone or in groups.  Spectra with repeated and nearly repeated
eigenvalues, a diagonal K (a tridiagonal form that decouples), a graded one,
and warps at the edges of a block.

Both sides are stable eigensolvers, so the eigenvalues agree within a few
n eps ||K||: 1e-13 ||K|| at these sizes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2307_04508_gb300 import ltgw
    c = ltgw.Context(0)
    yield c
    c.close()


def _spectrum(kind, n):
    i = np.arange(n)
    return {"decay": np.exp(-6.0 * i / n), "repeated": np.where(i % 3 == 0, 1.0, 0.5),
            "close": np.where(i % 3 == 0, 1.0, 0.5) + 1e-10 * i, "low_rank": (i < max(1, n // 3)) * (1.0 + i),
            "equal": np.ones(n), "graded": 10.0 ** (-12.0 * i / n), "scaled": 1e30 * np.exp(-3.0 * i / n)}[kind]


@pytest.mark.parametrize("n", [1, 2, 5, 33, 153, 264])
@pytest.mark.parametrize("kind", ["decay", "repeated", "close", "low_rank", "equal", "graded", "scaled"])
@pytest.mark.parametrize("diagonal", [False, True])
def test_eigenvalues_and_vectors(ctx, kind, n, diagonal):
    w = _spectrum(kind, n)
    Q = np.eye(n) if diagonal else np.linalg.qr(np.random.default_rng(n).standard_normal((n, n)))[0]
    B = np.ascontiguousarray(Q * np.sqrt(w)[None, :])
    K = B @ B.T
    ref = np.sort(np.linalg.eigvalsh(K))[::-1]
    srt = np.sort(w)[::-1]
    gap = int(np.argmax(srt[:-1] - srt[1:])) if n > 1 and srt[0] > srt[-1] else n - 1
    thr = 0.5 * (srt[gap] + srt[gap + 1]) if gap + 1 < n else 0.5 * srt[-1]
    Ut = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    k = ctx.naf_basis(torch.from_numpy(B).cuda(), n, n, thr, Ut, lam)
    assert k == gap + 1
    g, U = lam[:k].cpu().numpy(), Ut[:k].cpu().numpy()
    assert np.all(np.diff(g) <= 1e-13 * ref[0])
    assert np.abs(g - ref[:k]).max() <= 1e-13 * ref[0]
    assert np.linalg.norm(K @ U.T - U.T * g[None, :], axis=0).max() <= 1e-12 * ref[0]
    assert np.abs(U @ U.T - np.eye(k)).max() <= 1e-12


@pytest.mark.parametrize("n", [620, 1300])   # 8 vectors per block in shared memory, 16 in global
def test_all_vectors_kept(ctx, n):
    w = _spectrum("decay", n)
    Q = np.linalg.qr(np.random.default_rng(n).standard_normal((n, n)))[0]
    B = np.ascontiguousarray(Q * np.sqrt(w)[None, :])
    K = B @ B.T
    Ut = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    assert ctx.naf_basis(torch.from_numpy(B).cuda(), n, n, 1e-4, Ut, lam) == n
    g, U = lam.cpu().numpy(), Ut.cpu().numpy()
    assert np.abs(g - np.sort(np.linalg.eigvalsh(K))[::-1]).max() <= 1e-13 * g[0]
    assert np.linalg.norm(K @ U.T - U.T * g[None, :], axis=0).max() <= 1e-12 * g[0]
    assert np.abs(U @ U.T - np.eye(n)).max() <= 1e-12


@pytest.mark.parametrize("n", [33, 153, 264])
def test_small_eigenvalues_of_a_graded_matrix(ctx, n):
    """A diagonal K graded over twelve decades: the tridiagonal form is exact, so each
    eigenvalue, and not only the largest, is the diagonal entry to the rounding of
    the metric (2^-54 in digits, 2^-53 in FP64) and half a bracket of 2 eps: 4 eps."""
    b = np.sqrt(_spectrum("graded", n))
    Ut = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    assert ctx.naf_basis(torch.from_numpy(np.diag(b)).cuda(), n, n, 1e-14, Ut, lam) == n
    ref = b.astype(np.longdouble) ** 2
    assert np.abs((lam.cpu().numpy() - ref) / ref).max() <= 4 * 2.0 ** -52
