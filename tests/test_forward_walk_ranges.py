"""The host plans the forward projector's warps (which rays walk which rows, and
whether several angles per warp stay inside the staged image) from the range
that each ray's lane forms on the device, so both must be the same number: at
an angle almost parallel to the walk a last bit of the ray's position decides
between no row and all rows.  CPU only: the device's FP32 arithmetic is
restated (one rounding per multiply-add), the plan is the library's own."""
import ctypes
import math
import platform

import numpy as np
import pytest

FX = 2.0 ** 32
f32 = np.float32


class FwdAngle(ctypes.Structure):
    _fields_ = [("P", ctypes.c_longlong), ("Q", ctypes.c_longlong), ("D", ctypes.c_longlong), ("pf", ctypes.c_float),
                ("qf", ctypes.c_float), ("df", ctypes.c_float), ("scale", ctypes.c_float),
                ("row_group8", ctypes.c_uint), ("group4", ctypes.c_uint)]


@pytest.fixture(scope="module")
def ranges():
    if platform.machine() != "x86_64":
        pytest.skip("calls a C++ function that returns a vector, by this machine's convention")
    from paper_2110_01481_gb300 import _native, build
    build.build()
    f = ctypes.CDLL(_native.LIB_PATH)["_Z18ctg_forward_rangesPK8FwdAngleiii"]
    f.restype = ctypes.c_void_p

    def call(tab, N, n_det):
        vec = (ctypes.c_void_p * 3)()                       # begin, end, capacity; its memory is not given back
        f(vec, tab, ctypes.c_int(N), ctypes.c_int(len(tab)), ctypes.c_int(n_det))
        n = (vec[1] - vec[0]) // 8
        return np.ctypeslib.as_array((ctypes.c_int * (2 * n)).from_address(vec[0])).reshape(len(tab), -1, 2).copy()

    return call


def _table(N, n_angles, n_det, ds):
    """A 180-degree scan's forward angles."""
    h, hd = 0.5 * (N - 1), 0.5 * (n_det - 1)
    tab = (FwdAngle * n_angles)()
    for a in range(n_angles):
        th = a / n_angles * math.pi
        c, s = {0.0: (1.0, 0.0), 0.5: (0.0, 1.0)}.get(a / n_angles, (math.cos(th), math.sin(th)))
        row = 4 * a <= n_angles or 4 * a >= 3 * n_angles
        if not row:
            c, s = s, c
        P, Q, D = ds / c, (h * s - hd * ds) / c + h, -s / c
        tab[a] = FwdAngle(round(P * FX), round(Q * FX), round(D * FX), P, Q, D, 1 / abs(c), int(row), 0)
    return tab


def _device_range(t, N, d):
    """A lane's rows [lo, hi] (N, -1: none)."""
    u0 = f32(np.longdouble(d) * np.longdouble(t.pf) + np.longdouble(t.qf))
    if abs(t.df) <= 1e-20:
        return (0, N - 1) if -2.0 < u0 < N + 1.0 else (N, -1)
    r1, r2 = f32(f32(-1) - u0) / f32(t.df), f32(f32(N) - u0) / f32(t.df)
    lo = max(0, math.floor(min(max(min(r1, r2), f32(-2)), f32(2 * N))) - 1)
    hi = min(N - 1, math.ceil(max(min(max(r1, r2), f32(N + 1)), f32(-2 * N))) + 1)
    return (lo, hi) if lo <= hi else (N, -1)


# detector pitches that put a ray of the first angle, or of one near it, within rounding of the image's edge
@pytest.mark.parametrize("N,n_angles,n_det,ds", [
    (64, 8, 114, 0.99999997), (64, 90, 92, 1.0), (33, 48, 64, 17 / 31.5 * (1 - 1e-8)), (128, 2000, 215, 64.5 / 77),
    (100, 60, 181, 50.5 / 69 * (1 + 3e-8))])
def test_planned_ranges_are_the_device_ranges(ranges, N, n_angles, n_det, ds):
    tab = _table(N, n_angles, n_det, ds)
    got = ranges(tab, N, n_det)
    for a in range(n_angles):
        r = np.array([_device_range(tab[a], N, d) for d in range(n_det)])
        for g in range((n_det + 7) // 8):
            want = (r[8 * g:8 * g + 8, 0].min(), r[8 * g:8 * g + 8, 1].max())
            assert tuple(got[a, g]) == want, (a, g)
