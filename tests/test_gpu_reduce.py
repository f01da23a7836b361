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
