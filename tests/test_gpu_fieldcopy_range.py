"""Device field copies refuse an array that its allocation does not hold, and take one that it just
holds.  (The refusal comes before any device work.)"""
import ctypes as C
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2206_00638_gb300 import sbpsat  # noqa: E402


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP64, sbpsat.FP32_FP16STORE])
def test_short_allocation(precision):
    s = sbpsat.Sim((12, 9, 11), (1e-3,) * 3, (sbpsat.PEC,) * 6, precision=precision)
    L, esize = sbpsat.lib(), np.dtype(s.dtype).itemsize
    shape = s.shape(sbpsat.EY)
    size = int(np.prod(shape)) * esize
    cuda = C.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    mem = C.c_void_p()
    assert cuda.cudaMalloc(C.byref(mem), C.c_size_t(size)) == 0
    try:
        values = np.arange(np.prod(shape), dtype=s.dtype).reshape(shape)
        s.set_field(sbpsat.EY, values)
        assert L.sbp_get_field(s.handle, sbpsat.EY, mem.value, 1) == 0
        s.set_field(sbpsat.EY, np.zeros(shape, dtype=s.dtype))
        assert L.sbp_set_field(s.handle, sbpsat.EY, mem.value, 1) == 0
        assert np.array_equal(s.field(sbpsat.EY), values)
        for past in (esize, size // 2 // esize * esize):      # ends one element, then half the array, too late
            assert L.sbp_get_field(s.handle, sbpsat.EY, mem.value + past, 1) < 0
            assert L.sbp_set_field(s.handle, sbpsat.EY, mem.value + past, 1) < 0
        assert np.array_equal(s.field(sbpsat.EY), values)     # and the simulation goes on
    finally:
        torch.cuda.synchronize()
        cuda.cudaFree(mem)


@pytest.mark.parametrize("precision", [sbpsat.FP32, sbpsat.FP32_FP16STORE])
def test_first_cuda_call_of_a_thread(precision):
    """The allocation is looked up in a thread that has made no CUDA call yet, too."""
    s = sbpsat.Sim((12, 9, 11), (1e-3,) * 3, (sbpsat.PEC,) * 6, precision=precision)
    shape = s.shape(sbpsat.EZ)
    size = int(np.prod(shape)) * 4
    cuda = C.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    mem = C.c_void_p()
    assert cuda.cudaMalloc(C.byref(mem), C.c_size_t(size)) == 0
    got = []
    for past in (4, 0):
        th = threading.Thread(target=lambda: got.append(sbpsat.lib().sbp_get_field(s.handle, sbpsat.EZ, mem.value + past, 1)))
        th.start()
        th.join()
    torch.cuda.synchronize()
    cuda.cudaFree(mem)
    assert got[0] < 0 and got[1] == 0
