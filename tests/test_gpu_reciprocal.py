"""The FP64 reciprocal of the WENO weights against IEEE division.

rcp_newton refines the hardware's approximation r, of relative error e, to r (1 + e + e^2): the
third-order member of the hyperpower iterations for an inverse (Altman 1960; Householder's method
for 1/r - x).  Its error is e^3 of the result plus one rounding: with e of 2^-20 less than 0.51
units in the last place, so the result is the correctly rounded reciprocal or its neighbour.
The quotient num rcp_newton(den) adds one rounding to that: at most two units from num / den.
The denominators of the weights start at 10 (3/4 1e-6)^4 = 3.2e-24 (WENO5) and grow as the eighth
power of the differences of c; 1e60 is differences of some 1e7."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include "weno.cuh"
__global__ void k(const double* num, const double* den, double* r, double* q, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = lw::rcp_newton(den[i]);
  q[i] = num[i] * lw::rcp_newton(den[i]);
}
extern "C" int run(const double* num, const double* den, double* r, double* q, int n) {
  k<<<(n + 255) / 256, 256>>>(num, den, r, q, n);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
"""


def _ordered(x):
    """Integers in the order of the doubles: neighbours differ by one."""
    b = x.view(np.int64)
    return np.where(b < 0, np.int64(-2**63) - b, b)


def test_reciprocal_is_within_a_unit_of_ieee_division(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_07694_gb300 import build
    src, lib = tmp_path / "rcp.cu", tmp_path / "rcp.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc()] + build.NVCC_FLAGS + ["-I" + build.CSRC, "-o", str(lib), str(src)], check=True)
    L = ctypes.CDLL(os.fspath(lib))
    rng = np.random.default_rng(81)
    n = 1 << 22
    den = 10.0 ** rng.uniform(np.log10(3.2e-24), 60, n)
    # mantissas at both ends of a binade, where a unit of the reciprocal changes size
    edge = np.ldexp(1.0, rng.integers(-78, 199, 1 << 16))
    den[:3 << 16] = np.concatenate([edge, np.nextafter(edge, np.inf), np.nextafter(edge, 0)])
    num = rng.normal(size=n) * den * 10.0 ** rng.uniform(-6, 0, n)
    d = [torch.from_numpy(a).cuda() for a in (num, den)]
    out = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    assert L.run(*(ctypes.c_void_p(t.data_ptr()) for t in d + out), n) == 0
    r, q = (t.cpu().numpy() for t in out)
    assert np.abs(_ordered(r) - _ordered(1.0 / den)).max() <= 1
    assert np.abs(_ordered(q) - _ordered(num / den)).max() <= 2
