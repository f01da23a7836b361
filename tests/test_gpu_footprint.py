"""What a solve holds on the device stays within ltgw_request_footprint, by which
the server admits requests: the serving law's sizes, with and without NAF, in
every form (contexts as the server sets them up: digit workspace of 640 MiB)."""
import numpy as np
import pytest

from paper_2307_04508_gb300.synthetic.device import DeviceLaw

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_occ", [8, 20, 40])
@pytest.mark.parametrize("naf,n_tau", [(1e-2, 8), (-1.0, 8), (-1.0, 0)])
@pytest.mark.parametrize("prec", [0, 1, 2, 4])
def test_workspace_within_the_footprint(n_occ, naf, n_tau, prec):
    from paper_2307_04508_gb300 import ltgw
    n_virt, n_aux, nf = 10 * n_occ, 33 * n_occ, n_occ // 6
    law = DeviceLaw(n_occ, n_virt, n_aux, nf, 3, 4, gemm="tf32")
    p = ltgw.make_params(n_occ, n_virt, n_aux, nf, 32, n_tau, 0.5, naf, 2, bool(n_tau), prec)
    sig, e, st = np.zeros((4, 32, 2)), np.zeros(4), np.zeros(4, dtype=np.int32)
    c = ltgw.Context(0)
    c.set_digit_memory(640 << 20)
    # inputs from the host: the estimate counts their staged copies
    c.solve(p, law.eps, law.b_ov().cpu().numpy(), law.b_tgt().cpu().numpy(), law.targets.astype(np.int32), law.shift,
            sig, e, st)
    held = c.workspace_bytes()
    c.close()
    assert held <= ltgw.request_footprint(p, 4)


def test_many_kept_functions_stay_on_the_digits():
    """A threshold that keeps nearly every auxiliary function: the digits of the
    server's contexts still hold a piece, so the solve in the server has the bits of
    the one alone (the FP64 tiles round differently)."""
    from paper_2307_04508_gb300 import ltgw
    n_occ, n_virt, n_aux, nf = 60, 600, 1980, 10
    law = DeviceLaw(n_occ, n_virt, n_aux, nf, 3, 2, gemm="tf32")
    p = ltgw.make_params(n_occ, n_virt, n_aux, nf, 8, 2, 0.5, 1e-9, 2, True, 0)
    B, Bt, tg = law.b_ov(), law.b_tgt(), law.targets.astype(np.int32)
    outs = []
    c = ltgw.Context(0)
    srv = ltgw.Server(0, 1, 64 << 30)
    for run in (c.solve, srv.submit):
        outs.append((np.zeros((2, 8, 2)), np.zeros(2), np.zeros(2, dtype=np.int32)))
        run(p, law.eps, B, Bt, tg, law.shift, *outs[-1])
    srv.wait_all()
    kept = c.stats()["n_naf"]
    c.close()
    srv.close()
    assert kept > 0.9 * n_aux
    assert np.array_equal(outs[0][0], outs[1][0])
