"""Which kernels a length runs on, from the library's own rule (no GPU): the steps of
the tile kernels, their Bluestein form, or the Stockham stages."""
import ctypes

import pytest

from paper_1211_5244_gb300 import build as _build
from paper_1211_5244_gb300 import psolver as ps

# products of 2, 3, 5, 7 that need a fourth radix up to 16, and the lengths too short for two steps
STOCKHAM = [2, 3, 5, 7, 625, 875, 1029, 1225, 1250, 1323, 1458, 1701, 1715, 1750, 1875, 1944, 2000, 2058, 2187, 2205,
            2268, 2401, 2430, 2450, 2500, 2592, 2625, 2646, 2800, 2835, 2916, 3000, 3024, 3087, 3125, 3200, 3240, 3402,
            3430, 3456, 3500, 3528, 3645, 3675, 3750, 3780, 3888, 3920, 3969, 4000, 4032, 4050]
MAX_M = {True: 4096, False: 3200}  # convolution points of a Bluestein line, FP32 and FP64


class Radix(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("Ra", "Rm", "Rl", "cls")]


@pytest.fixture(scope="module")
def rule():
    _build.build()
    lib = ps.load_library()
    radix, blue = lib._ZN2ps10tile_radixEibbPNS_9TileRadixEPd, lib._ZN2ps16tile_blue_lengthEibi
    radix.argtypes = [ctypes.c_int, ctypes.c_bool, ctypes.c_bool, ctypes.POINTER(Radix), ctypes.c_void_p]
    radix.restype = ctypes.c_bool
    blue.argtypes = [ctypes.c_int, ctypes.c_bool, ctypes.c_int]
    blue.restype = ctypes.c_int

    def steps(N, f32, even_first=False):
        r = Radix()
        return (r.Ra, r.Rm, r.Rl, r.cls) if radix(N, even_first, f32, ctypes.byref(r), None) else None

    def length(N, f32):
        return blue(N, f32, MAX_M[f32])

    return steps, length


def _big_prime(N):
    big, p = 1, 2
    while N > 1:
        while N % p == 0:
            N, big = N // p, p
        p += 1
    return big


@pytest.mark.parametrize("f32", [True, False])
def test_steps_of_every_length(rule, f32):
    steps, length = rule
    smooth_without, blue_without = [], []
    for N in range(2, 4097):
        for even_first in ([False, True] if N % 2 == 0 else [False]):
            r = steps(N, f32, even_first)
            if r is None:
                continue
            Ra, Rm, Rl, cls = r
            assert Ra * Rm * Rl == N
            assert not (even_first and Ra % 2)
            if cls == 2:
                assert Rl in (17, 19, 23, 29, 31) and max(Ra, Rm) <= 16 and (Ra >= 2 or N == Rl)
            else:
                assert min(Ra, Rl) >= 2 and max(r[:3]) <= (16 if cls else 8)
        if N % 2 == 0:  # an even first step costs no length its form
            assert (steps(N, f32, True) is None) == (steps(N, f32) is None), N
        if steps(N, f32) is None:
            if _big_prime(N) < 11:
                smooth_without.append(N)
            elif length(N, f32) == 0:
                blue_without.append(N)
            else:
                M = length(N, f32)
                assert 2 * N <= M <= 4 * N and M % 2 == 0 and steps(M, f32, True)[3] != 2
    assert smooth_without == STOCKHAM
    assert min(blue_without) == (2049 if f32 else 1576)


def test_families_of_known_lengths(rule):
    steps, length = rule
    for f32 in (True, False):
        assert all(steps(N, f32)[1] == 1 for N in (36, 100, 180))              # two steps
        assert all(steps(N, f32)[1] > 1 for N in (343, 1000, 1920, 2048, 4096))  # three
        assert steps(2000, f32) is None and _big_prime(2000) < 11               # Stockham
        for N in (11, 13, 37, 289, 1031):                                      # Bluestein
            assert steps(N, f32) is None and length(N, f32) > 0
