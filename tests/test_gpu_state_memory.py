"""States given with on_device = 1 in memory that the library copies instead of
reading or writing it with its own kernels: a device buffer off the 8-byte
boundary, managed memory and page-locked host memory.  set_state, get_state and
residual give the same numbers as with a host array, whole numbers of doubles
moved by the same copies, so the comparison is exact.
"""
import ctypes

import numpy as np
import pytest

from paper_1908_03972_gb300 import workloads as W

pytestmark = pytest.mark.gpu
MA = 0.05


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_03972_gb300 import build, pmgfr
    build.build()
    pmgfr.load()


class _Managed:
    def __init__(self, nbytes):
        self.cu = ctypes.CDLL("libcuda.so.1")
        p = ctypes.c_uint64()
        assert self.cu.cuMemAllocManaged(ctypes.byref(p), ctypes.c_size_t(nbytes), ctypes.c_uint(1)) == 0
        self.ptr = p.value
        self.host = np.ctypeslib.as_array((ctypes.c_ubyte * nbytes).from_address(self.ptr))

    def write(self, x):
        self.host[:] = np.frombuffer(x.tobytes(), np.uint8)

    def read(self, shape):
        return np.frombuffer(self.host.tobytes(), np.float64).reshape(shape)

    def close(self):
        self.host = None
        self.cu.cuMemFree_v2(ctypes.c_uint64(self.ptr))


class _Tensor:
    """Bytes of a torch buffer from an offset on (device memory) or of a page-locked one."""

    def __init__(self, nbytes, offset=0, pinned=False):
        import torch
        self.torch = torch
        self.t = (torch.zeros(nbytes, dtype=torch.uint8, pin_memory=True) if pinned
                  else torch.zeros(nbytes + offset, dtype=torch.uint8, device="cuda")[offset:])
        self.ptr = self.t.data_ptr()

    def write(self, x):
        self.t.copy_(self.torch.frombuffer(bytearray(x.tobytes()), dtype=self.torch.uint8))
        self.torch.cuda.synchronize()

    def read(self, shape):
        self.torch.cuda.synchronize()
        return np.frombuffer(self.t.cpu().numpy().tobytes(), np.float64).reshape(shape)

    def close(self):
        self.t = None


KINDS = {"device": lambda n: _Tensor(n), "device+4": lambda n: _Tensor(n, 4), "device+1": lambda n: _Tensor(n, 1),
         "managed": lambda n: _Managed(n), "pinned": lambda n: _Tensor(n, pinned=True)}


@pytest.mark.parametrize("gauge", [False, True])
@pytest.mark.parametrize("kind", list(KINDS))
def test_states_in_other_memory(kind, gauge):
    from paper_1908_03972_gb300 import pmgfr
    nodes, nbr = W.periodic_box(5, 4, Ng=1)
    s = pmgfr.Solver(nodes, nbr, [2], [1], Ma_inf=MA, p_gauge=W.freestream_T(MA) if gauge else 0.0)
    lib = pmgfr.load()
    q = np.ascontiguousarray(W.isentropic_vortex(s.coords(), Ma_inf=MA, center=(4.0, 6.0)))
    buf = KINDS[kind](q.nbytes)
    out = _Tensor(q.nbytes)
    try:
        assert kind in ("device", "device+4", "device+1") or buf.ptr % 8 == 0
        buf.write(q)
        assert lib.pmg_set_state(s.h, 0, ctypes.c_void_p(buf.ptr), 1) == 0
        ref = np.empty_like(q)
        pmgfr.pmg_get_state(s.h, 0, ref)
        pmgfr.pmg_set_state(s.h, 0, q)
        host = np.empty_like(q)
        pmgfr.pmg_get_state(s.h, 0, host)
        assert np.array_equal(ref, host)
        buf.write(np.full_like(q, np.nan))
        assert lib.pmg_get_state(s.h, 0, ctypes.c_void_p(buf.ptr), 1) == 0
        assert np.array_equal(buf.read(q.shape), host)
        buf.write(q)
        assert lib.pmg_residual(s.h, 0, ctypes.c_void_p(buf.ptr), ctypes.c_void_p(out.ptr), 1) == 0
        R = np.empty_like(q)
        pmgfr.pmg_residual(s.h, 0, q, R)
        assert np.array_equal(out.read(q.shape), R)
    finally:
        buf.close()
        out.close()
        s.close()
