"""Sums of the tensor-core partial tiles into both triangles, at sizes around the
64-entry quarters and 128-entry tiles that the reduction walks.

An entry's error is at most 2^-15 of the Cauchy-Schwarz product of its rows
(operands kept to 16 bits, three products), which no diagonal entry exceeds:
1e-4 of the largest entry, so that one misplaced entry fails.
"""
import numpy as np
import pytest

from oracle import ltgw_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [2, 63, 64, 65, 127, 128, 129, 192, 193, 257])
def test_both_triangles(N):
    from paper_2307_04508_gb300 import ltgw
    rng = np.random.default_rng(N)
    Bt = rng.standard_normal((N, 500)) * 0.05
    delta = rng.uniform(0.3, 4.0, 500)
    om, _ = O.gl_grid(3, 0.5)
    Pi = torch.full((3, N, N), float("nan"), dtype=torch.float64, device="cuda")
    ctx = ltgw.Context(0)
    ctx.polarizability_mixed(torch.from_numpy(Bt).cuda(), torch.from_numpy(delta).cuda(), om, Pi, spin=2)
    got, ref = Pi.cpu().numpy(), O.polarizability_direct(Bt, delta, om, 2)
    ctx.close()
    assert np.array_equal(got, np.swapaxes(got, 1, 2))
    for j in range(3):
        assert np.abs(got[j] - ref[j]).max() <= 1e-4 * np.abs(ref[j]).max()


@pytest.mark.parametrize("N", [159, 160, 321])
def test_both_kernels_many_splits(N):
    """The last size of one thread per element and the first ones of the strips,
    with several K splits per entry (20,000 pairs) and Laplace moments."""
    from paper_2307_04508_gb300 import ltgw
    rng = np.random.default_rng(N)
    Bt = rng.standard_normal((N, 20000)) * 0.01
    delta = rng.uniform(0.3, 4.0, 20000)
    om, _ = O.gl_grid(3, 0.5)
    x, w = np.array([0.1, 1.0, 3.0]), np.array([0.3, 0.7, 1.1])
    Pi = torch.full((3, N, N), float("nan"), dtype=torch.float64, device="cuda")
    ctx = ltgw.Context(0)
    ctx.polarizability_mixed(torch.from_numpy(Bt).cuda(), torch.from_numpy(delta).cuda(), om, Pi, x=x, w=w, spin=2)
    got = Pi.cpu().numpy()
    ctx.close()
    M = [(Bt * (w[k] * delta * np.exp(-delta * delta * x[k]))[None, :]) @ Bt.T for k in range(3)]
    assert np.array_equal(got, np.swapaxes(got, 1, 2))
    for j in range(3):
        ref = -4.0 * sum(np.exp(-om[j] ** 2 * x[k]) * M[k] for k in range(3))
        assert np.abs(got[j] - ref).max() <= 1e-4 * np.abs(ref).max()
