"""dJ/dVs of the FP32 gradient: its terms, which cancel, are summed well beyond FP32.

With the fluid at rest and Vs and the split speed far below FP32 resolution a step leaves c as it
is, so dJ/dVs is the sum of c over the floor, c (1/6 + 1/6 + 2/3) a node, up to terms of relative
size Vs and alpha: at most ten of 1e-11 each.  In FP32 the weights alone would be off by 3e-8 and
the sum of a tile's columns, which have both signs here, by some 1e-7 of their size."""
import math

import numpy as np
import pytest

from tests.helpers import rel_l2, to_np

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_07694_gb300 import build
    build.build()


@pytest.mark.parametrize("shape", [(4, 4), (100, 33), (2048, 4), (64, 70)])
@pytest.mark.parametrize("signs", [False, True])
def test_terms_that_cancel_are_summed_beyond_fp32(shape, signs):
    from paper_2106_07694_gb300.lbm_wenoc import Simulation
    rng = np.random.default_rng(61)
    c0 = rng.uniform(0.5, 1.5, shape[::-1])
    if signs:
        c0[:, 1::2] *= -1
    c0 = c0.astype(np.float32)
    s = Simulation(shape, tau=0.6, gravity=0.0, settling_velocity=1e-12, diffusivity=0.0, lf_alpha=1e-11, u_cap=0.2)
    _, _, dvs = s.deposit_gradient(c0, 1, 1)
    floor = [float(v) for v in c0[0]]
    assert abs(dvs - math.fsum(floor)) <= 1e-10 * math.fsum(map(abs, floor))


@pytest.mark.parametrize("rough", [False, True])
def test_lambda_does_not_drift_with_the_steps(rough):
    """The reverse stages' weights 1/3 and 2/3 of lambda sum to one.  Rounded to FP32 one by one they
    sum to 1 + 3e-8, which over the deposits of 100 steps, 50 steps back on average, is 1.5e-6 on the
    gradient; the roundings themselves, of 1e-7 or so a step and of both signs, stay well below half
    of that, which is the bound."""
    from paper_2106_07694_gb300 import workloads
    from paper_2106_07694_gb300.lbm_wenoc import Simulation
    shape, steps = (200, 160), 100
    rng = np.random.default_rng(62)
    if rough:
        c0 = 0.5 + 0.4 * rng.uniform(-1, 1, shape[::-1])
    else:
        c0 = workloads.interface_field(shape, interface_frac=0.6, amplitude=1e-3, seed=62, lower=0.05)
    c0 = c0.astype(np.float32)
    kw = dict(tau=0.6, gravity=2e-3, density_contrast=1.0, settling_velocity=0.05, diffusivity=0.02, lf_alpha=0.25, u_cap=0.2)
    g32, g64 = (to_np(Simulation(shape, fp64=f, **kw).deposit_gradient(c0, steps, 10)[1]) for f in (False, True))
    err = rel_l2(g32, g64)
    print(f"gradient of {steps} steps: {err:.2e}")
    assert err <= 0.75e-6
