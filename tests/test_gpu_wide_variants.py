"""The scheme variants and the sugar scalar on the four-column stage kernels against the
one-column ones.

The four-column kernels compute every face with the one-column kernels' arithmetic in the same
order, so c, u, rho and S agree bit for bit; the deposit's FP64 partial sums are grouped per
strip, so it agrees to rounding."""
import numpy as np
import pytest

from paper_2106_07694_gb300 import workloads
from tests.helpers import PHYS, to_np

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
