"""dJ/dVs of the FP32 gradient: its terms, which cancel, are summed well beyond FP32.

With the fluid at rest and Vs and the split speed far below FP32 resolution a step leaves c as it
is, so dJ/dVs is the sum of c over the floor, c (1/6 + 1/6 + 2/3) a node, up to terms of relative
size Vs and alpha: at most ten of 1e-11 each.  In FP32 the weights alone would be off by 3e-8 and
the sum of a tile's columns, which have both signs here, by some 1e-7 of their size."""
import math

import numpy as np
import pytest

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
