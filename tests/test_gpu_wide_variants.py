"""The scheme variants and the sugar scalar on the four-column stage kernels against the
one-column ones, and the FP32 adjoint's tile kernels at the edges of their tiles.

The four-column kernels compute every face with the one-column kernels' arithmetic in the same
order, so c, u, rho and S agree bit for bit; the deposit's FP64 partial sums are grouped per
strip, so it agrees to rounding.  The adjoint works on 32 x 32 tiles in FP32 while the FP64
build keeps the per-face records: the two gradients agree to FP32 accuracy, 1e-3 relative L2 as
for the whole-lattice comparisons (a node's derivative sums some twenty rounded terms whose
weights carry a relative error of a few 1e-6 each where differences are near sqrt(eps))."""
import numpy as np
import pytest

from paper_2106_07694_gb300 import workloads
from tests.helpers import PHYS, rel_l2, to_np

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_07694_gb300 import build
    build.build()


SUGAR = dict(sugar=True, sugar_contrast=0.5, sugar_diffusivity=0.02, phi0=0.05, vs_sugar=0.3)
VARIANTS = {
    "weno3": dict(weno3=True), "sign": dict(sign_split=True), "weno3_sign": dict(weno3=True, sign_split=True),
    "sugar": SUGAR, "sugar_weno3": dict(SUGAR, weno3=True), "sugar_sign": dict(SUGAR, sign_split=True),
}


def _run(shape, variant, one):
    from paper_2106_07694_gb300 import lbm_wenoc as lw
    s = lw.Simulation(shape, one_column=one, **dict(PHYS, gravity=5e-4, settling_velocity=3e-3), **VARIANTS[variant])
    s.init(workloads.interface_field(shape, interface_frac=0.6, amplitude=0.03, seed=31))
    if "sugar" in variant:
        s.set_sugar(1.0 - workloads.interface_field(shape, interface_frac=0.5, amplitude=0.02, seed=32))
    s.step(7)
    out = [to_np(t) for t in s.fields()] + ([to_np(s.sugar())] if "sugar" in variant else [])
    return out, s.deposit


@pytest.mark.parametrize("variant", sorted(VARIANTS))
@pytest.mark.parametrize("shape", [(4, 5), (260, 33), (1028, 18), (36, 20, 9), (68, 17, 25)])
def test_four_column_variants_bitwise_equal_to_one_column(shape, variant):
    wide, dw = _run(shape, variant, False)
    narrow, dn = _run(shape, variant, True)
    for a, b in zip(wide, narrow):
        assert np.array_equal(a, b)
    assert abs(dw - dn) <= 1e-12 * abs(dn)


@pytest.mark.parametrize("shape", [(4, 4), (12, 31), (32, 32), (36, 33), (60, 34), (132, 65), (64, 130)])
def test_adjoint_tiles_match_fp64(shape):
    from paper_2106_07694_gb300.lbm_wenoc import Simulation
    kw = dict(tau=0.6, gravity=2e-3, density_contrast=1.0, settling_velocity=0.05, diffusivity=0.02, lf_alpha=0.25,
              u_cap=0.2)
    c0 = (0.5 + 0.4 * np.random.default_rng(33).uniform(-1, 1, (shape[1], shape[0]))).astype(np.float32).astype(float)
    out = []
    for fp64 in (False, True):
        J, g, dvs = Simulation(shape, fp64=fp64, **kw).deposit_gradient(c0, 12, 5)
        out.append((J, to_np(g), dvs))
    (J, g, v), (J64, g64, v64) = out
    assert J == pytest.approx(J64, rel=1e-5)
    assert rel_l2(g, g64) <= 1e-3
    assert v == pytest.approx(v64, rel=1e-3)
