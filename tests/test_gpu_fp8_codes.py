"""Every route of the FP8 quantisation (a block per row with up to 8 and up to 12
factor rows; two kernels with two and with eight factor rows per block) against
the oracle's FP8 definition: the same codes, so only the FP32 accumulation
differs, 2e-5 relative Frobenius as in test_gpu_fp8.py."""
import numpy as np
import pytest

from oracle import ltgw_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,P,n_om", [(70, 700, 8), (130, 12300, 9), (70, 700, 12), (129, 12289, 12), (70, 13000, 5),
                                      (70, 700, 13), (500, 13000, 20)])
def test_codes_on_every_route(N, P, n_om):
    from paper_2307_04508_gb300 import ltgw
    rng = np.random.default_rng(N + P + n_om)
    Bt = rng.standard_normal((N, P)) * 0.05
    Bt[N // 2] = 0.0
    delta = rng.uniform(0.3, 4.0, P)
    om, _ = O.gl_grid(n_om, 0.5)
    Pi = torch.empty((n_om, N, N), dtype=torch.float64, device="cuda")
    ctx = ltgw.Context(0)
    ctx.polarizability_fp8(torch.from_numpy(Bt).cuda(), torch.from_numpy(delta).cuda(), om, Pi, spin=2)
    ctx.close()
    got, ref = Pi.cpu().numpy(), O.polarizability_fp8(Bt, delta, om, 2)
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
    assert np.array_equal(got, np.swapaxes(got, 1, 2))
