"""Device buffers that a caller hands to init and fields: kernels use them in place only where they
are long enough and apart from the handle's workspace.  One too short is refused by the copy it
goes through, as any buffer was before kernels used them in place."""
import ctypes

import numpy as np
import pytest

from paper_2106_07694_gb300 import lbm_wenoc as lw, workloads
from tests.helpers import PHYS, to_np

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPE = (128, 128)
N = SHAPE[0] * SHAPE[1]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_07694_gb300 import build
    build.build()


@pytest.fixture()
def cudart():
    lw.load()  # brings the process's libcudart
    rt = ctypes.CDLL("libcudart.so.13")
    rt.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
    rt.cudaFree.argtypes = [ctypes.c_void_p]
    return rt


def _sim():
    s = lw.Simulation(SHAPE, **PHYS)
    c0 = torch.from_numpy(workloads.interface_field(SHAPE, seed=51).astype(np.float32)).cuda()
    return s, c0


def test_a_short_buffer_is_refused(cudart):
    s, c0 = _sim()
    torch.cuda.synchronize()
    p = ctypes.c_void_p()
    assert cudart.cudaMalloc(ctypes.byref(p), 4 * N) == 0  # a scalar field fits, a vector field does not
    L = lw.load()
    try:
        assert L.lbm_wenoc_init(s.handle, c0.data_ptr(), p.value) == lw.LW_ECUDA
        cudart.cudaGetLastError()
        assert L.lbm_wenoc_init(s.handle, c0.data_ptr(), None) == lw.LW_OK
        s.step(2)
        assert L.lbm_wenoc_fields(s.handle, None, p.value, None) == lw.LW_ECUDA
        cudart.cudaGetLastError()
        assert L.lbm_wenoc_fields(s.handle, p.value + 4096, None, None) == lw.LW_ECUDA
        cudart.cudaGetLastError()
        assert L.lbm_wenoc_fields(s.handle, p.value, None, None) == lw.LW_OK
    finally:
        torch.cuda.synchronize()
        cudart.cudaFree(p)


def test_a_velocity_inside_the_workspace_is_copied_first():
    s, c0 = _sim()
    rng = np.random.default_rng(52)
    u0 = torch.from_numpy((0.02 * rng.uniform(-1, 1, (2,) + SHAPE[::-1])).astype(np.float32)).cuda()
    s.workspace[:u0.numel() * 4].copy_(u0.reshape(-1).view(torch.uint8))
    torch.cuda.synchronize()
    assert lw.load().lbm_wenoc_init(s.handle, c0.data_ptr(), s.workspace.data_ptr()) == lw.LW_OK
    t = lw.Simulation(SHAPE, **PHYS)
    t.init(c0, u0)
    for a, b in zip(s.fields(), t.fields()):
        assert np.array_equal(to_np(a), to_np(b))
