"""FP64 contractions on the tensor cores from base-256 digits (slice_gemm.cu),
reached through the FP64 polarisability, against the exact sum in extended
precision.

Bound per entry (i, j) of M = sum_k A_ik B_jk with A = B = R~ diag(sqrt|f|)
(the sign of f with A), K pairs and row scales 2^(e_i) > max_k |A_ik|: the
digits hold each entry to 2^-56 2^(e_i) (two operands: 2 * 2^-56), the dropped
levels i + j >= 9 are at most 6 * 2^14 * 2^-72 * 4 (1 + 2^-7) < 6.1 * 2^-56 per
pair, so K 2^(e_i + e_j) 2^-53 in all; the roots, their products with R~ and the
factor itself add 8 * 2^-53 of sum_k |A_ik B_jk|, and the final rounding and the
sums over K splits and chunks another 8 * 2^-53 of it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = U_ROUND = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2307_04508_gb300 import ltgw
    c = ltgw.Context(0)
    yield c
    c.close()


def _pi(ctx, R, delta, omegas, **kw):
    N, J = R.shape[0], len(omegas)
    out = torch.full((J, N, N), float("nan"), dtype=torch.float64, device="cuda")
    ctx.polarizability(torch.from_numpy(R).cuda(), torch.from_numpy(delta).cuda(), omegas, out, **kw)
    return out.cpu().numpy()


def _check(got, R, f, alpha):
    """got ~ alpha R diag(f) R^T within the bound of the module docstring."""
    N = R.shape[0]
    pick = np.unique(np.array([0, 1, 31, 63, 64, 65, 127, 128, N // 2, N - 2, N - 1]).clip(0, N - 1))
    g = np.sqrt(np.abs(f))
    A = R * g[None, :]   # sizes only; the reference sums R_i f R_j in extended precision
    Rl, fl = R.astype(np.longdouble), f.astype(np.longdouble)
    e = np.frexp(np.maximum(np.abs(A).max(axis=1), 1e-320))[1]
    size = np.abs(A) @ np.abs(A).T
    for i in pick:   # whole rows, chosen at the edges of the tiles
        ref = alpha * (Rl * (Rl[i] * fl)[None, :]).sum(axis=1)
        bound = abs(alpha) * (R.shape[1] * np.exp2((e + e[i]).astype(np.float64)) * U + 16 * U * size[i])
        err = np.abs((got[i] - ref).astype(np.float64))
        assert np.all(err <= bound), (i, (err / np.maximum(bound, 1e-300)).max())
    assert np.array_equal(got, got.T)


# one tile and its edges (64 / 128 rows, 16 k), one warp-held row (512) and past
# it, drains of 144 k, K splits, ragged tails
@pytest.mark.parametrize("N,K", [(400, 128), (63, 5200), (64, 4880), (65, 4800), (128, 1296), (129, 1297), (257, 512),
                                 (257, 513), (192, 2049), (321, 20000)])
def test_pi_matches_exact_sum(ctx, N, K):
    rng = np.random.default_rng(N * 7 + K)
    R = rng.standard_normal((N, K)) * np.exp2(rng.integers(-40, 40, N))[:, None]
    R[N // 2] = 0.0
    delta = 0.3 + 3.0 * rng.random(K)
    om = np.array([0.02, 1.7])
    got = _pi(ctx, R, delta, om)
    for j, w in enumerate(om):
        f = delta / (w * w + delta * delta)
        _check(got[j], R, f, -4.0)


def test_pi_moments_negative_weights_and_gaps(ctx):
    """Negative factors (the sign goes with one operand only), a factor that
    singles out the smallest gaps, spin 1, and the recombination."""
    rng = np.random.default_rng(3)
    N, K = 150, 3001
    R = rng.standard_normal((N, K))
    delta = 0.3 + 3.0 * rng.random(K)
    delta[::5] *= -1.0
    x, w = np.array([0.5, 40.0]), np.array([-0.7, 2.0])
    om = np.array([0.0])   # exp(-w^2 x) = 1: Pi = -2 (M^0 + M^1)
    got = _pi(ctx, R, delta, om, x=x, w=w, spin=1)[0]
    f = [w[k] * delta * np.exp(-delta * delta * x[k]) for k in range(2)]
    Rl = R.astype(np.longdouble)
    ref = sum(-2.0 * np.stack([(Rl * (Rl[i] * fk)[None, :]).sum(axis=1) for i in range(N)]) for fk in f)
    size = sum(2.0 * ((np.abs(R) * np.abs(fk)[None, :]) @ np.abs(R).T) for fk in f)
    scale = sum(2.0 * K * np.exp2(2.0 * np.frexp((np.abs(R) * np.sqrt(np.abs(fk))[None, :]).max())[1]) for fk in f)
    # the factor's own exponent argument d^2 x carries a relative rounding of
    # 2 u, an error of up to 2 u d^2 x <= 900 u in exp where it still matters
    assert np.all(np.abs((got - ref).astype(np.float64)) <= U * scale + 1000 * U * size)


def test_pi_nonfinite_rows_stay_in_their_rows(ctx):
    rng = np.random.default_rng(5)
    N, K = 140, 4000
    R = rng.standard_normal((N, K))
    R[7, 11], R[130, 3999] = np.nan, np.inf
    delta = 0.3 + rng.random(K)
    om = np.array([0.1])
    got = _pi(ctx, R, delta, om)[0]
    bad = np.zeros(N, dtype=bool)
    bad[[7, 130]] = True
    assert not np.isfinite(got[bad]).any() and not np.isfinite(got[:, bad]).any()
    keep = np.ix_(~bad, ~bad)
    f = delta / (om[0] ** 2 + delta * delta)
    _check(got[keep], R[~bad], f, -4.0)


# one block and a remainder of 16, both sides of a block's edge, a ragged last
# block shorter than a 16-k step; one and several frequencies
@pytest.mark.parametrize("N,J", [(144, 3), (255, 1), (256, 2), (257, 2), (393, 2)])
def test_screen_digits_matches_inverse(ctx, N, J):
    """C = (1 - Pi)^-1 - 1 by the digit sweep: (1 - Pi)(C + 1) = 1 to a backward
    error of N steps' roundings, 8 N u of |1 - Pi||C + 1| (a sweep of an SPD
    matrix with eigenvalues >= 1 is stable; the digits' error per update is
    below N u of the rows' scales), symmetric bit for bit, and a matrix that is
    not positive definite is reported."""
    from paper_2307_04508_gb300 import ltgw
    rng = np.random.default_rng(N)
    R = rng.standard_normal((J, N, 2 * N)) * (0.6 / np.sqrt(N)) * np.exp(-2.0 * np.arange(N) / N)[None, :, None]
    Pi = -4.0 * R @ R.transpose(0, 2, 1)
    Pi = 0.5 * (Pi + Pi.transpose(0, 2, 1))
    C = torch.empty((J, N, N), dtype=torch.float64, device="cuda")
    ctx.screen(torch.from_numpy(Pi).cuda(), C)
    got = C.cpu().numpy()
    eye = np.eye(N)
    for j in range(J):
        assert np.array_equal(got[j], got[j].T)
        A, X = eye - Pi[j], got[j] + eye
        res = np.abs(A @ X - eye)
        assert res.max() <= 8 * N * U * np.linalg.norm(A, 2) * np.linalg.norm(X, 2)
    Pi[J - 1, N - 1, N - 1] = 50.0   # the last pivot turns negative
    with pytest.raises(ltgw.LtgwError) as e:
        ctx.screen(torch.from_numpy(Pi).cuda(), C)
    assert e.value.status == ltgw.LTGW_ERR_NOT_SPD


# the vectors' products from digits: their smallest size, five whole blocks of
# 64 reflectors and one more; the blocked reduction: its smallest size, one
# panel and several, remainders on both sides of a panel; a metric of rank 70
# (reflectors of a zero column)
@pytest.mark.parametrize("n,pairs", [(200, 600), (322, 644), (323, 646), (1000, 3000), (1001, 2002), (1063, 2126), (1129, 2258), (1003, 70)])
def test_naf_from_digits(ctx, n, pairs):
    """Residual, orthonormality and eigenvalues of the kept pairs: the reduction
    and the vectors are backward stable to n u |K| each (32 n u with the
    constants of two-sided reflectors and the panel's sums)."""
    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, pairs)) / np.sqrt(pairs) * np.exp(-3.0 * np.arange(n) / n)[:, None]
    K = B @ B.T
    ref = np.sort(np.linalg.eigvalsh(K))[::-1]
    m = int(np.argmax(ref[20:60] - ref[21:61])) + 20
    thr = 0.5 * (ref[m] + ref[m + 1])
    Ut = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    k = ctx.naf_basis(torch.from_numpy(B).cuda(), pairs, pairs, thr, Ut, lam)
    assert k == m + 1
    U, lg = Ut[:k].cpu().numpy().T, lam[:k].cpu().numpy()
    tol = 32 * n * U_ROUND * ref[0]
    assert np.abs(lg - ref[:k]).max() <= tol
    assert np.linalg.norm(K @ U - U * lg[None, :], axis=0).max() <= tol
    assert np.abs(U.T @ U - np.eye(k)).max() <= 32 * n * U_ROUND


def _weak_rows(rng, N, K, odd, tail):
    """Gaussian rows, large on the first half of the pairs and `tail` times smaller on
    the second; the rows `odd` the other way round, so that every term of their
    products with the others is small beside the rows' largest entries."""
    R = rng.standard_normal((N, K))
    head = np.arange(K) < K // 2
    R[:, ~head] *= tail
    R[odd] = rng.standard_normal((len(odd), K)) * np.where(head, tail, 1.0)
    return R


# few weak entries per tile (one pass of 128 and several), most of a tile, whole
# tiles; eight and seven levels; a tail that the digits hold in part and not at all
@pytest.mark.parametrize("N,K,odd,tail", [(150, 3001, [5, 77], 1e-9), (150, 3001, [3, 4, 70, 71, 149], 1e-20),
                                          (130, 5200, list(range(0, 130, 2)), 1e-9), (70, 5200, [69], 1e-6),
                                          (64, 700, list(range(20, 64)), 1e-12), (40, 500001, [7, 8], 1e-9)])
def test_pi_weakly_coupled_rows(ctx, N, K, odd, tail):
    """Componentwise: an entry is off by no more than an FP64 sum's bound, K u of
    sum |a||b| (1.04 K u where the leading digits have just passed it) and the 16 u of
    the module docstring."""
    rng = np.random.default_rng(N + K)
    R = _weak_rows(rng, N, K, odd, tail)
    delta = 0.3 + 3.0 * rng.random(K)
    om = np.array([0.4])
    got = _pi(ctx, R, delta, om)[0]
    f = delta / (om[0] ** 2 + delta * delta)
    size = 4.0 * ((np.abs(R) * f[None, :]) @ np.abs(R).T)
    Rl, fl = R.astype(np.longdouble), f.astype(np.longdouble)
    for i in sorted({0, N // 2, N - 1, odd[0], odd[-1]}):
        ref = -4.0 * (Rl * (Rl[i] * fl)[None, :]).sum(axis=1)
        err = np.abs((got[i] - ref).astype(np.float64))
        assert np.all(err <= (1.04 * K + 16) * U * size[i]), (i, (err / size[i]).max())
    assert np.array_equal(got, got.T)


def test_pi_infinite_entries_as_an_fp64_sum(ctx):
    rng = np.random.default_rng(8)
    N, K = 140, 4000
    R = rng.standard_normal((N, K))
    R[130, 3999] = np.inf
    R[2, 3999] = 0.0
    got = _pi(ctx, R, 0.3 + rng.random(K), np.array([0.1]))[0]
    want = np.where(R[:, 3999] == 0.0, np.nan, -np.inf * np.sign(R[:, 3999]))
    assert np.array_equal(got[130], want, equal_nan=True) and np.array_equal(got[:, 130], want, equal_nan=True)
