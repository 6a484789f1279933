"""A segment height selects the row sweep on lattices that otherwise run on tiles.

The row sweep, its scheme variants and the sugar scalar included, gives the bits of the one-column
kernel at every height: one row, odd ones, the longest segment (64) and past it; on a strip narrower
than a warp, ragged strips (256 columns) and several.  Switching between steps carries the deposit
that a step on tiles leaves to the next one."""
import ctypes

import numpy as np
import pytest

from paper_2106_07694_gb300 import lbm_wenoc as lw, workloads
from tests.helpers import PHYS, to_np

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KW = dict(PHYS, gravity=5e-4, settling_velocity=3e-3)
SUGAR = dict(sugar=True, sugar_contrast=0.5, sugar_diffusivity=0.02, phi0=0.05, vs_sugar=0.3)
VARIANTS = {
    "plain": {}, "weno3": dict(weno3=True), "sign": dict(sign_split=True), "weno3_sign": dict(weno3=True, sign_split=True),
    "sugar": SUGAR, "sugar_weno3": dict(SUGAR, weno3=True), "sugar_sign": dict(SUGAR, sign_split=True),
    "sugar_weno3_sign": dict(SUGAR, weno3=True, sign_split=True), "classes": dict(class_vs=(1e-3, 4e-3)),
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_07694_gb300 import build
    build.build()


def _init(s, shape, kw):
    s.init(workloads.interface_field(shape, interface_frac=0.6, amplitude=0.03, seed=31, lower=0.2))
    if "sugar" in kw:
        s.set_sugar(1.0 - workloads.interface_field(shape, interface_frac=0.5, amplitude=0.02, seed=32))
    if "class_vs" in kw:
        s.set_class(1, workloads.interface_field(shape, interface_frac=0.4, amplitude=0.02, seed=33, lower=0.1))


def _fields(s, kw):
    return [to_np(t) for t in s.fields()] + ([to_np(s.sugar())] if "sugar" in kw else [])


@pytest.mark.parametrize("variant", sorted(VARIANTS))
@pytest.mark.parametrize("shape", [(4, 5), (260, 33), (520, 90)])
def test_row_sweep_at_every_height_bitwise_equal_to_one_column(shape, variant):
    kw = VARIANTS[variant]
    one = lw.Simulation(shape, one_column=True, **KW, **kw)
    _init(one, shape, kw)
    one.step(6)
    want, dep = _fields(one, kw), None
    for rows in (0, 1, 7, 64, 200):
        s = lw.Simulation(shape, **KW, **kw)
        lw.lbm_wenoc_set_segment_rows(s.handle, rows)
        _init(s, shape, kw)
        s.step(6)
        for a, b in zip(_fields(s, kw), want):
            assert np.array_equal(a, b), rows
        dep = s.deposit if dep is None else dep
        assert s.deposit == dep, rows
    assert abs(dep - one.deposit) <= 1e-12 * abs(one.deposit)


class _KernelNode(ctypes.Structure):  # cudaKernelNodeParams
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p)]


def _block_sizes(s):
    """Threads a block of the kernels of a captured step."""
    rt, vp = ctypes.CDLL("libcudart.so.13"), ctypes.c_void_p
    stream, graph, count = vp(s.stream.cuda_stream), vp(), ctypes.c_size_t()
    assert rt.cudaStreamBeginCapture(stream, 2) == 0  # relaxed
    s.step(1)
    assert rt.cudaStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes = (vp * count.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    out = []
    for n in nodes:
        k = _KernelNode()
        assert rt.cudaGraphKernelNodeGetParams(vp(n), ctypes.byref(k)) == 0
        out.append(k.block[0] * k.block[1] * k.block[2])
    assert rt.cudaGraphDestroy(graph) == 0
    return out


# the fluid kernel and three stages: tiles of 32 x 16 nodes with four nodes a thread, or strips of
# 256 columns with four a thread
@pytest.mark.parametrize("rows,threads", [(0, 128), (9, 64)])
def test_a_height_selects_the_row_sweep(rows, threads):
    shape = (100, 33)
    s = lw.Simulation(shape, stream=torch.cuda.Stream(), graphs=False, **KW)
    with torch.cuda.stream(s.stream):
        lw.lbm_wenoc_set_segment_rows(s.handle, rows)
        _init(s, shape, {})
    s.stream.synchronize()
    assert sorted(_block_sizes(s)) == sorted([128] + 3 * [threads])


@pytest.mark.parametrize("extra", [{}, SUGAR])
def test_switching_between_steps_keeps_the_deposit(extra):
    shape = (260, 40)
    s, ref = (lw.Simulation(shape, **KW, **extra) for _ in range(2))
    for k in (s, ref):
        _init(k, shape, extra)
    for rows in (0, 5, 0, 0, 64, 64, 0):
        lw.lbm_wenoc_set_segment_rows(s.handle, rows)
        s.step(3)
        ref.step(3)
    assert s.deposit == ref.deposit > 0
    for a, b in zip(_fields(s, extra), _fields(ref, extra)):
        assert np.array_equal(a, b)


def test_replayed_tile_steps_count_after_a_switch():
    # steps on tiles that a caller captured leave their deposit also when the handle has moved on
    shape = (100, 33)
    s, ref = (lw.Simulation(shape, stream=torch.cuda.Stream(), graphs=False, **KW) for _ in range(2))
    g = torch.cuda.CUDAGraph()
    for k in (s, ref):
        with torch.cuda.stream(k.stream):
            _init(k, shape, {})
            k.stream.synchronize()
    with torch.cuda.stream(s.stream):
        with torch.cuda.graph(g, stream=s.stream):
            s.step(2)
        lw.lbm_wenoc_set_segment_rows(s.handle, 6)
        g.replay()
    with torch.cuda.stream(ref.stream):
        ref.step(2)
    assert s.deposit == ref.deposit > 0


@pytest.mark.parametrize("shape,rows", [((4, 8), 0), ((260, 40), 0), ((260, 40), 6), ((2308, 16), 0)])
def test_a_fresh_state_drops_what_a_step_left(shape, rows):
    s, ref = (lw.Simulation(shape, **KW) for _ in range(2))
    _init(s, shape, {})
    s.step(5)
    lw.lbm_wenoc_set_segment_rows(s.handle, rows)
    for k in (s, ref):
        _init(k, shape, {})
    assert s.deposit == 0.0
    for k in (s, ref):
        k.step(3)
    assert s.deposit == ref.deposit > 0
