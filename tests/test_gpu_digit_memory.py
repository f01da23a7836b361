"""The digits' memory: a product that runs in pieces (frequencies, moments,
columns) gives the same bits as the whole one, one whose smallest piece does not
fit runs on the FP64 tiles, and the chunks of a long sum add up.

Bounds: the FP64 tiles against the digits, both within K u sum |a||b| of the exact
sum with Gaussian rows (their scales are below a few sum |a||b|): 1e-12 of the
largest entry at these lengths; chunked sums as in test_gpu_slices.py."""
import numpy as np
import pytest

from paper_2307_04508_gb300 import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53
MB = 1 << 20


def _ctx(limit=None):
    from paper_2307_04508_gb300 import ltgw
    c = ltgw.Context(0)
    if limit is not None:
        c.set_digit_memory(limit)
    return c


def _pi(limit, emu, n_tau):
    rng = np.random.default_rng(2)
    R = torch.from_numpy(rng.standard_normal((150, 3001))).cuda()
    delta = torch.from_numpy(0.3 + 3.0 * rng.random(3001)).cuda()
    om = np.linspace(0.02, 2.0, 7)
    kw = dict(x=np.array([0.1, 0.5, 2.0]), w=np.array([-0.3, 0.7, 1.1])) if n_tau else {}
    out = torch.full((7, 150, 150), float("nan"), dtype=torch.float64, device="cuda")
    c = _ctx(limit)
    (c.polarizability_emulated if emu else c.polarizability)(R, delta, om, out, **kw)
    held = c.workspace_bytes()
    c.close()
    return out.cpu().numpy(), held


# one frequency's digits: 2 x 256 x 3008 x 14 bytes = 21 MB (emulated 9.2 and the
# shared operand's 9.2)
@pytest.mark.parametrize("emu,n_tau", [(False, 0), (False, 3), (True, 0), (True, 3)])
def test_pi_in_pieces_has_the_same_bits(emu, n_tau):
    whole, held = _pi(None, emu, n_tau)
    for limit in (80 * MB, 48 * MB, 24 * MB):
        part, h = _pi(limit, emu, n_tau)
        assert np.array_equal(part, whole)
        assert h <= min(held, limit + 8 * MB)   # 8 MB: the arrays that are not digits
    low, _ = _pi(MB, emu, n_tau)   # below the smallest piece
    if emu:
        assert np.array_equal(low, whole)
    else:
        assert np.abs(low - whole).max() <= 1e-12 * np.abs(whole).max()


def test_screening_in_pieces_has_the_same_bits():
    rng = np.random.default_rng(4)
    R = rng.standard_normal((5, 200, 300)) * 0.03
    Pi = torch.from_numpy(-4.0 * R @ R.transpose(0, 2, 1)).cuda()
    Pi = 0.5 * (Pi + Pi.transpose(1, 2))
    got = []
    for limit in (None, 3 * MB, 0):   # 1.4 MB per frequency: five at once, two, the FP64 tiles
        C = torch.empty_like(Pi)
        c = _ctx(limit)
        c.screen(Pi, C)
        c.close()
        got.append(C.cpu().numpy())
    assert np.array_equal(got[0], got[1])
    assert np.abs(got[2] - got[0]).max() <= 1e-12 * np.abs(got[0]).max()


def _solve(prec, limit, sizes=(12, 100, 300), n_tgt=3, naf=1e-2, held=None):
    from paper_2307_04508_gb300 import ltgw
    p = S.make_problem(*sizes, n_frozen=2, seed=5, n_targets=n_tgt)
    q = ltgw.make_params(*sizes, 2, 16, 6, 0.5, naf, 2, True, prec)
    T = len(p.targets)
    sig, e, st = np.zeros((T, 16, 2)), np.zeros(T), np.zeros(T, dtype=np.int32)
    c = _ctx(limit)
    c.solve(q, p.eps, p.B_ov, p.B_tgt, p.targets.astype(np.int32), p.shift, sig, e, st)
    if held is not None:
        held.append(c.workspace_bytes())
    c.close()
    return sig


# metric 320 x 1008 x 14 bytes = 4.5 MB, the projection of 1000 columns 4.7
# beside 0.9, W_nm's frequencies 0.4 each, Pi's moments 4 each
@pytest.mark.parametrize("emu", [False, True])
def test_solve_in_pieces_has_the_same_bits(emu):
    from paper_2307_04508_gb300 import ltgw
    prec = ltgw.LTGW_FP64_EMU if emu else ltgw.LTGW_FP64
    whole = _solve(prec, None)
    assert np.array_equal(_solve(prec, 14 * MB), whole)
    low = _solve(prec, 0)
    assert np.array_equal(low, whole) if emu else np.abs(low - whole).max() <= 1e-9 * np.abs(whole).max()


@pytest.mark.parametrize("emu", [False, True])
@pytest.mark.parametrize("naf", [1e-2, -1.0])
def test_many_targets_in_pieces_have_the_same_bits(emu, naf):
    """64 targets of 74 orbitals: 24 MB of digits in the projection, 14 MB in W_nm
    without NAF (a seventh less emulated), above the limit, which the other
    products keep to in pieces of one moment; the targets run in pieces too."""
    from paper_2307_04508_gb300 import ltgw
    prec = ltgw.LTGW_FP64_EMU if emu else ltgw.LTGW_FP64
    args, held = ((36, 40, 200), 64, naf), []
    whole = _solve(prec, None, *args)
    assert np.array_equal(_solve(prec, 13 * MB, *args, held), whole)
    _solve(prec, 0, *args, held)
    assert held[0] <= held[1] + 13 * MB


def test_pi_chunks_of_a_long_sum():
    """512,001 pairs of 100 rows: 2 x 128 x 14 bytes a pair, two chunks of at most
    1.5 GiB, the last one ragged."""
    rng = np.random.default_rng(6)
    N, K = 100, 512001
    R = rng.standard_normal((N, K))
    delta = 0.3 + 3.0 * rng.random(K)
    om = np.array([0.1, 1.0])
    out = torch.empty((2, N, N), dtype=torch.float64, device="cuda")
    c = _ctx()
    c.polarizability(torch.from_numpy(R).cuda(), torch.from_numpy(delta).cuda(), om, out)
    c.close()
    got = out.cpu().numpy()
    for j, w in enumerate(om):
        f = delta / (w * w + delta * delta)
        A = np.abs(R) * np.sqrt(f)[None, :]
        e = np.frexp(A.max(axis=1))[1]
        size = A @ A.T
        for i in (0, 63, 64, 99):
            ref = -4.0 * (R.astype(np.longdouble) * (R[i].astype(np.longdouble) * f)[None, :]).sum(axis=1)
            bound = 4.0 * U * (K * np.exp2((e + e[i]).astype(np.float64)) + 16 * size[i])
            assert np.all(np.abs((got[j, i] - ref).astype(np.float64)) <= bound)


def test_metric_chunks_of_a_long_sum():
    """1,000,003 pairs of 48 rows (two chunks of 128 x 14 bytes a pair) through the
    NAF eigenvalues: K to K u of the rows' scales, the eigensolver to n u |K|."""
    rng = np.random.default_rng(7)
    n, K = 48, 1000003
    B = rng.standard_normal((n, K)) * np.exp(-0.05 * np.arange(n))[:, None] / 1000.0
    Ut = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    c = _ctx()
    assert c.naf_basis(torch.from_numpy(B).cuda(), K, K, 1e-9, Ut, lam) == n
    c.close()
    ref = np.sort(np.linalg.eigvalsh(B @ B.T))[::-1]
    assert np.abs(lam.cpu().numpy() - ref).max() <= 1e-12 * ref[0]
