"""The rule that takes small 2D images to the multi-step kernel: its lines lie at a
number of tiles per SM, whatever the device's number of SMs."""
import ctypes as C
import os

import pytest

from paper_2201_04565_gb300 import lsm


class _Plan(C.Structure):
    _fields_ = [("shape", C.c_int), ("halo", C.c_int), ("tiles", C.c_int64)]


@pytest.mark.parametrize("sms", [152, 160, 76, 20])
def test_lines_follow_the_device(sms):
    if not os.path.exists(lsm.LIB_PATH):
        pytest.skip("liblsm.so is not built")
    f = C.CDLL(lsm.LIB_PATH)._ZN3lsm11multi_shapeEiiii
    f.restype, f.argtypes = _Plan, [C.c_int] * 4
    exact, f32, df = (lsm.PRECISIONS[p] for p in ("exact64", "f32", "df64"))
    none, s16x4, s32x8, e16x4, e32x4 = range(5)

    def plan(prec, nx, ny):
        p = f(prec, nx, ny, sms)
        return p.shape, p.halo, p.tiles

    for prec in (f32, df):
        n = sms + sms // 16
        assert plan(prec, 16 * n, 4) == (s16x4, 3, n)
        assert plan(prec, 16 * n + 1, 4) == (s32x8, 2, (16 * n + 32) // 32)
        assert plan(prec, 64 * sms, 8) == (s32x8, 2, 2 * sms)
        assert plan(prec, 64 * sms + 1, 8)[0] == none
    assert plan(exact, 16 * (sms // 2), 4) == (e16x4, 1, sms // 2)
    assert plan(exact, 16 * (sms // 2) + 1, 4)[0] == e32x4
    assert plan(exact, 32 * sms, 4) == (e32x4, 1, sms)
    assert plan(exact, 32 * sms + 1, 4)[0] == none
