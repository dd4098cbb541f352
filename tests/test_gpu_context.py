"""Fields made in a thread whose caller has a context of its own current: it stays current."""
import ctypes
import threading

import pytest

pytestmark = pytest.mark.gpu


def test_a_callers_context_stays_current(gpu_lib):
    su3s = gpu_lib
    lat = su3s.Lattice((4, 4, 4, 4))
    f = su3s.Field(lat)             # in the device's primary context, as the buffer below
    L, cu = su3s.load(), ctypes.CDLL("libcuda.so.1")
    P = ctypes.c_void_p
    cu.cuCtxCreate_v2.argtypes = [ctypes.POINTER(P), ctypes.c_uint, ctypes.c_int]
    cu.cuCtxGetCurrent.argtypes = [ctypes.POINTER(P)]
    cu.cuCtxDestroy_v2.argtypes = [P]
    seen = {}

    def work():
        own, now, h = P(), P(), P()
        seen["create"] = cu.cuCtxCreate_v2(ctypes.byref(own), 0, 0)
        if seen["create"]:
            return
        # the field's description only: nothing is launched
        seen["wrap"] = L.su3s_field_wrap(lat._h, su3s.MATRIX, 1, su3s.F64, su3s.SOA, 0, f.tensor.data_ptr(),
                                         f.tensor.numel() * 8, ctypes.byref(h))
        cu.cuCtxGetCurrent(ctypes.byref(now))
        seen["own"], seen["now"] = own.value, now.value
        L.su3s_field_destroy(h)
        seen["destroy"] = cu.cuCtxDestroy_v2(own)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert seen["create"] == 0 and seen["wrap"] == 0 and seen["destroy"] == 0
    assert seen["own"] and seen["now"] == seen["own"]
