"""The third-order reciprocal and the reflector's scalars (fast_fp64.cuh) against
extended precision over the exponent range, on both sides of the range beyond
which IEEE operations take over.  Bounds, u = 2^-53, as derived in the header:
reciprocal 1.01 u; given s = alpha^2 + sigma rounded once (s off by u: 1/2 u more
in its root), tau 3.1 u, beta 3.1 u, sc 5.2 u.  The extended format adds 2^-11 u."""
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53

SRC = r"""
#include "fast_fp64.cuh"
__global__ void k_recip(const double *q, double *r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = ltgw::recip_cubic(q[i]);
}
__global__ void k_refl(const double *a, const double *s, double *t, double *b, double *c, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) ltgw::reflector_scalars(a[i], s[i], t + i, b + i, c + i);
}
extern "C" int run(const double *q, double *r, const double *a, const double *s, double *t, double *b, double *c, int n) {
  k_recip<<<(n + 255) / 256, 256>>>(q, r, n);
  k_refl<<<(n + 255) / 256, 256>>>(a, s, t, b, c, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_against_extended_precision(tmp_path):
    import ctypes
    from paper_2307_04508_gb300 import build
    src, lib = tmp_path / "fast.cu", tmp_path / "fast.so"
    src.write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2307_04508_gb300", "csrc")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", csrc,
                           str(src), "-o", str(lib)])
    n = 1 << 20
    rng = np.random.default_rng(11)
    q = (1.0 + rng.random(n)) * np.exp2(rng.integers(-1000, 1000, n)) * rng.choice([-1.0, 1.0], n)
    # alpha and sigma around one scale, and alpha far below or above |x'|; the last
    # eighth beyond 2^+-800 for s
    ex = np.where(np.arange(n) < 7 * n // 8, rng.integers(-395, 396, n),
                  rng.choice([-1.0, 1.0], n) * rng.integers(402, 480, n))
    alpha = rng.standard_normal(n) * np.exp2(ex) * np.exp2(rng.choice([0.0, -20.0, -60.0, 4.0], n))
    sigma = rng.random(n) * np.exp2(2.0 * ex) + np.exp2(2.0 * ex - 40.0)
    d = [torch.from_numpy(x).cuda() for x in (q, alpha, sigma)]
    o = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(4)]
    run = ctypes.CDLL(str(lib)).run
    P = [ctypes.c_void_p(x.data_ptr()) for x in (d[0], o[0], d[1], d[2], o[1], o[2], o[3])]
    torch.cuda.synchronize()
    assert run(*P, ctypes.c_int(n)) == 0
    r, tau, beta, sc = (x.cpu().numpy().astype(np.longdouble) for x in o)
    a, s, ql = (x.astype(np.longdouble) for x in (alpha, sigma, q))
    nrm = np.sqrt(a * a + s)
    want_b = np.where(alpha < 0, nrm, -nrm)
    for got, ref, tol in ((r, 1 / ql, 1.01), (beta, want_b, 3.1), (tau, (want_b - a) / want_b, 3.1),
                          (sc, 1 / (a - want_b), 5.2)):
        assert np.abs((got - ref) / ref).max() <= tol * U
