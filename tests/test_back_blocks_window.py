"""The 2 x 2 block back projector stages a window of detector bins per angle
and tile and tests no bound when it reads it: for every geometry that the
library gives to that kernel, each index it forms lies inside the window.  CPU
only: the index arithmetic is restated, the rule is the library's own."""
import ctypes
import itertools
import math

import numpy as np
import pytest

# rows of a tile: (window entry of the bin at the tile's centre, entries)
WINDOWS = {32: (24, 52), 64: (37, 78)}
FX = 40


class BackAngle(ctypes.Structure):
    _fields_ = [("C", ctypes.c_longlong), ("COS", ctypes.c_longlong), ("SIN", ctypes.c_longlong),
                ("cf", ctypes.c_float), ("sf", ctypes.c_float)]


@pytest.fixture(scope="module")
def blocks_ok():
    from paper_2110_01481_gb300 import _native, build
    build.build()
    f = ctypes.CDLL(_native.LIB_PATH)["_Z18ctg_back_blocks_okPK9BackAnglei"]    # ctg_back_blocks_ok(table, angles)
    f.restype = ctypes.c_bool
    f.argtypes = [ctypes.POINTER(BackAngle), ctypes.c_int]
    return f


def _table(N, n_angles, n_det, start, range_, ds):
    tab = (BackAngle * n_angles)()
    h, hd = 0.5 * (N - 1), 0.5 * (n_det - 1)
    for a in range(n_angles):
        num = start * n_angles + a * range_
        if num % (90 * n_angles) == 0:
            c, s = ((1.0, 0.0), (0.0, 1.0), (-1.0, 0.0), (0.0, -1.0))[num // (90 * n_angles) % 4]
        else:
            th = num / (180 * n_angles) * math.pi
            c, s = math.cos(th), math.sin(th)
        tab[a] = BackAngle(round((hd - h * (c + s) / ds) * 2.0 ** FX), round(c / ds * 2.0 ** FX),
                           round(s / ds * 2.0 ** FX), c / ds, s / ds)
    return tab


def _index_range(tab, N, n_det, rows):
    """Least and greatest window entry that the kernel reads, over all angles, tiles and threads."""
    centre, _ = WINDOWS[rows]
    least, most = 10 ** 9, -10 ** 9
    f32 = np.float32
    # the lowest corner's offset from the tile's centre, columns and rows: its extremes over the blocks
    offs_j = np.array([-15.5, 14.5], f32)
    offs_i = np.array([-0.5 * (rows - 1), 0.5 * (rows - 1) - 1.0], f32)
    for t in tab:
        C, COS, SIN, cf, sf = t.C, t.COS, t.SIN, f32(t.cf), f32(t.sf)
        for bx, by in itertools.product(range((N + 31) // 32), range(((N + 1) // 2 + rows - 1) // rows)):
            U = C + 32 * bx * COS + rows * by * SIN + ((31 * COS + (rows - 1) * SIN) >> 1)
            c, s = cf, sf
            if SIN < 0:
                U, c, s = ((n_det - 1) << FX) - U, -c, -s
            phase = f32(((U >> (FX - 24)) & 0xFFFFFF) / 16777216.0)
            u = phase + s * offs_i[:, None] + abs(c) * offs_j[None, :]
            least = min(least, math.floor(u.min()) + centre)
            most = max(most, math.floor(u.max()) + centre + 3)
    return least, most


# pitches about and below one pixel; scans about the diagonals, where both |cos| and |sin| are below such a pitch
SCANS = [(0, 180, 30), (40, 10, 12), (42, 6, 12), (45, 360, 4), (45, 90, 2), (30, 30, 15), (35, 20, 10), (133, 4, 5),
         (-47, 4, 4), (225, 1, 1), (0, 90, 7)]
PITCHES = [0.7, 0.71, 0.72, 0.75, 0.8, 0.85, 0.9, 0.93, 0.95, 0.96, 0.98, 0.999, 1.0, 1.001, 1.01, 1.5]


@pytest.mark.parametrize("ds", PITCHES)
@pytest.mark.parametrize("N", [64, 131])
def test_every_index_lies_in_the_staged_window(blocks_ok, N, ds):
    n_det = math.ceil(math.sqrt(2) * N / ds)
    admitted = 0
    for start, range_, n_angles in SCANS:
        for nd in (n_det, n_det + 1):
            tab = _table(N, n_angles, nd, start, range_, ds)
            if not blocks_ok(tab, n_angles):
                continue
            admitted += 1
            for t in tab:                                   # a pixel step moves at most one bin
                assert abs(t.cf) <= 1.0 and abs(t.sf) <= 1.0
            for rows, (_, window) in WINDOWS.items():
                least, most = _index_range(tab, N, nd, rows)
                assert least >= 0 and most < window, (start, range_, n_angles, nd, rows, least, most)
    if ds >= 1.0:
        assert admitted == 2 * len(SCANS)                   # every scan at a pitch of a pixel or more


def test_far_corner_rule(blocks_ok):
    """Where the far corner takes three bins (one bin or more beyond the lowest
    corner), its distance f + (oB - 1) + (oC - 1) from the middle one of them,
    formed in FP32, lies in [-1, 1] for every fraction f in [0, 1)."""
    from paper_2110_01481_gb300 import _native
    unit = ctypes.CDLL(_native.LIB_PATH)["_Z20ctg_back_blocks_unitPK9BackAnglei"]     # ctg_back_blocks_unit(table, angles)
    unit.restype, unit.argtypes = ctypes.c_bool, [ctypes.POINTER(BackAngle), ctypes.c_int]
    f32 = np.float32
    seen = set()
    for ds, (start, range_, n_angles) in itertools.product(PITCHES + [1.2, 1.4, 1.0000001, 2.0], SCANS + [(0, 360, 100000)]):
        tab = _table(64, n_angles, 91, start, range_, ds)
        if not blocks_ok(tab, n_angles):
            continue
        is_unit = unit(tab, n_angles)
        seen.add((ds > 1.0, is_unit))
        if is_unit:
            for t in tab:
                oB, oC = abs(f32(t.cf)), abs(f32(t.sf))
                o = f32(f32(oB - f32(1)) + f32(oC - f32(1)))
                assert f32(f32(0) + o) >= -1.0 and f32(f32(1 - 2.0 ** -24) + o) <= 1.0
        elif ds == 1.0:
            raise AssertionError((start, range_, n_angles))
    assert seen == {(False, True), (True, True), (True, False)}
