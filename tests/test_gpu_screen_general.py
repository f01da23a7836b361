"""ltgw_screen of a Pi that is not symmetric bit for bit: what lies in the lower
triangle counts.  A NaN there is reported, a matrix of one pivot block (N <= 64)
is inverted whole, a larger one goes to the form that reads both triangles, and
asymmetry of a product's rounding changes the result by no more than that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2307_04508_gb300 import ltgw
    c = ltgw.Context(0)
    yield c
    c.close()


def _pi(N, J, seed):
    R = np.random.default_rng(seed).standard_normal((J, N, 2 * N)) * (0.5 / np.sqrt(N))
    P = -4.0 * R @ R.transpose(0, 2, 1)
    return 0.5 * (P + P.transpose(0, 2, 1))


def _screen(ctx, Pi):
    C = torch.empty(Pi.shape, dtype=torch.float64, device="cuda")
    ctx.screen(torch.from_numpy(Pi).cuda(), C)
    return C.cpu().numpy()


@pytest.mark.parametrize("N,i,j", [(40, 30, 2), (100, 99, 0), (200, 199, 0), (200, 150, 140), (300, 40, 33)])
def test_nan_below_the_diagonal_is_reported(ctx, N, i, j):
    from paper_2307_04508_gb300 import ltgw
    Pi = _pi(N, 2, N)
    Pi[1, i, j] = np.nan
    with pytest.raises(ltgw.LtgwError) as e:
        _screen(ctx, Pi)
    assert e.value.status == ltgw.LTGW_ERR_NOT_SPD


@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 40, 64])
def test_one_block_is_inverted_whole(ctx, N):
    """I - Pi + (a skew part of 0.1): its symmetric part's eigenvalues are >= 1, so
    every pivot is positive and the sweep stable: 64 N u of the two norms."""
    Pi = _pi(N, 2, N + 7)
    S = np.random.default_rng(N).standard_normal(Pi.shape) * 0.1 / np.sqrt(N)
    Pi = Pi + np.tril(S, -1) - np.tril(S, -1).transpose(0, 2, 1)
    got, eye = _screen(ctx, Pi), np.eye(N)
    for p, c in zip(Pi, got):
        A, X = eye - p, c + eye
        assert np.abs(A @ X - eye).max() <= 64 * N * 2.0 ** -53 * np.linalg.norm(A, 2) * np.linalg.norm(X, 2)


@pytest.mark.parametrize("N", [144, 257])
def test_asymmetric_matrix_takes_the_general_form(ctx, N):
    from paper_2307_04508_gb300 import ltgw
    Pi = _pi(N, 3, N)
    Pi[2, N - 1, 5] += 1e-3
    got = _screen(ctx, Pi)
    c = ltgw.Context(0)
    c.set_digit_memory(0)   # the FP64 tiles throughout
    ref = _screen(c, Pi)
    c.close()
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("N", [144, 257])
def test_asymmetry_of_rounding(ctx, N):
    """Entries off by 2 u of the rows' scales: the inverse moves by |X|^2 times
    that, |X| <= 1 here: N 4 u in norm, beside the sweep's own 8 N u |A||X|."""
    Pi = _pi(N, 2, N)
    noise = np.random.default_rng(1).integers(-2, 3, Pi.shape) * 2.0 ** -53
    got, ref = _screen(ctx, Pi + np.tril(noise, -1)), _screen(ctx, Pi)
    A = np.eye(N) - Pi
    tol = 16 * N * 2.0 ** -53 * np.linalg.norm(A, 2, axis=(1, 2)).max()
    assert np.abs(got - ref).max() <= tol
    assert np.array_equal(got, got.transpose(0, 2, 1))
