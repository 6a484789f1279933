"""On tiles the deposit of a step is folded by the next step, or before it is read.

When it is folded must not show: a run read after every step, one read at the end, one resumed
from a state saved in between and one whose total mass is read in between (the reductions share
the scratch) give the same bits, and instances stepped alone hand over to the batch."""
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


KW = dict(PHYS, gravity=5e-4, settling_velocity=3e-3)
SUGAR = dict(sugar=True, sugar_contrast=0.5, sugar_diffusivity=0.02, phi0=0.05, vs_sugar=0.3)


# one tile, several, ragged; more than eight strips of 256 columns; the row sweep (over 3.5 M nodes)
@pytest.mark.parametrize("shape,extra", [((32, 20), {}), ((100, 33), {}), ((260, 18), SUGAR), ((2308, 16), {}),
                                         ((4096, 900), {})])
def test_deposit_does_not_depend_on_when_it_is_read(shape, extra):
    from paper_2106_07694_gb300.lbm_wenoc import Simulation
    c0 = workloads.interface_field(shape, interface_frac=0.3, amplitude=0.03, seed=41, lower=0.2)
    sims = [Simulation(shape, **KW, **extra) for _ in range(4)]
    end, each, mass, saved = sims
    for s in sims:
        s.init(c0)
    for k in range(5):
        for s in sims:
            s.step(1)
        first = each.deposit
        assert first == each.deposit and first > 0
        assert mass.total_mass > 0
        if k == 2:
            state = saved.save_state()
            saved.step(3)
            saved.load_state(state)
    want = end.deposit
    assert [s.deposit for s in sims] == [want] * 4
    for s in sims[1:]:
        for a, b in zip(s.fields(), end.fields()):
            assert np.array_equal(to_np(a), to_np(b))


def test_steps_replayed_from_a_callers_graph():
    # an even number of steps (the population layout is back where it was), replayed twice
    from paper_2106_07694_gb300.lbm_wenoc import Simulation
    shape = (100, 33)
    c0 = workloads.interface_field(shape, interface_frac=0.3, amplitude=0.03, seed=43, lower=0.2)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        s, ref = (Simulation(shape, graphs=False, **KW) for _ in range(2))
        for k in (s, ref):
            k.init(torch.from_numpy(c0.astype(np.float32)).cuda())
        stream.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            s.step(2)
        for n in range(3):
            g.replay()
            ref.step(2)
            assert s.deposit == ref.deposit
        for a, b in zip(s.fields(), ref.fields()):
            assert np.array_equal(to_np(a), to_np(b))


def test_instances_stepped_alone_then_together():
    from paper_2106_07694_gb300 import lbm_wenoc as lw
    from paper_2106_07694_gb300.lbm_wenoc import Batch, Simulation
    specs = [dict(shape=(96, 40), **KW), dict(shape=(260, 24), **KW)]
    c0 = [workloads.interface_field(sp["shape"], interface_frac=0.3, amplitude=0.03, seed=42, lower=0.2) for sp in specs]
    b = Batch(specs)
    for inst, c in zip(b.instances, c0):
        inst.init(c)
        lw.lbm_wenoc_step(inst.handle, 2)
    b.step(2)
    for inst in b.instances:
        lw.lbm_wenoc_step(inst.handle, 2)
    for inst, c, sp in zip(b.instances, c0, specs):
        s = Simulation(sp["shape"], **KW)
        s.init(c)
        s.step(6)
        assert inst.deposit == s.deposit
