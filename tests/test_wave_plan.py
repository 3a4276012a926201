"""The cut of a frame into waves, and the band that the autotuner times: a wave size is timed only in waves of that
size (the code compiled with the host compiler)."""
import ctypes as C

import pytest

from tests.native import load

LANES = 4


def _lib():
    lib = load("plan")
    for f in (lib.waves, lib.full):
        f.argtypes = [C.c_longlong, C.c_int, C.c_int, C.c_int]
    return lib


@pytest.mark.parametrize("W,H,nl,spp", [(1920, 1080, 3, 64), (3840, 2160, 3, 256), (960, 540, 3, 128), (8192, 4096, 1, 1),
                                        (1917, 1003, 2, 31)])
def test_the_band_fills_every_candidate(W, H, nl, spp):
    lib = _lib()
    h = lib.rows(W, H, nl, spp, LANES)
    assert 1 <= h <= H
    want = 2 * LANES * lib.tune_wave(3)                          # two waves a lane
    if W * H * nl * spp < want:
        assert h == H
        return
    total = W * h * nl * spp
    assert want <= total < want + W * nl * spp                   # and no more rows than that takes
    for i in range(4):
        for lanes in range(1, LANES + 1):
            assert lib.full(total, spp, lanes, lib.tune_wave(i))


def test_wave_sizes_that_a_small_frame_cannot_fill_are_no_candidates():
    lib = _lib()
    total = 320 * 180 * 3 * 8
    for i in range(4):
        assert not lib.full(total, 8, 3, lib.tune_wave(i))
        assert lib.waves(total, 8, 3, lib.tune_wave(i)) == lib.waves(total, 8, 3, lib.tune_wave(0))


@pytest.mark.parametrize("total,spp,lanes,cap", [(5 * 3 * 3, 1, 3, 1 << 23), (1 << 20, 64, 3, 1 << 23), (1 << 20, 1 << 19, 4, 1 << 21),
                                                 (1 << 26, 16, 4, 1 << 24), (1 << 33, 16, 4, 1 << 24), (1 << 18, 3, 1, 4096)])
def test_waves_are_within_the_capacity_and_hold_a_pixel(total, spp, lanes, cap):
    n = _lib().waves(total, spp, lanes, cap)
    assert spp <= n <= cap
    # one wave per lane at the most below the capacity: a wave holds whole pixels, n // spp of them
    assert n == cap or n // spp * spp * lanes >= total
