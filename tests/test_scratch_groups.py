"""Groups of fields or maps in the wave-optics calls: as many as their spectra may take, halved while the device has
no room for their scratch, and an error only when one is too many (the code compiled with the host compiler)."""
import ctypes as C

import pytest

from tests.native import load

OK, INVALID, NO_MEMORY = 0, 1, 2


def test_group_items():
    lib = load("scratch")
    lib.items.argtypes = [C.c_longlong, C.c_size_t, C.c_size_t]
    assert lib.items(24, 35 << 20, 300 << 20) == 8
    assert lib.items(3, 35 << 20, 300 << 20) == 3
    assert lib.items(8, 400 << 20, 300 << 20) == 1
    assert lib.items(6 << 30, 32, 300 << 20) == (300 << 20) // 32


def _shrink(G, room, other=0):
    lib = load("scratch")
    st, n, asked = C.c_int(), C.c_int(), (C.c_int * 64)()
    return lib.shrink(G, room, other, C.byref(st), asked, C.byref(n)), st.value, list(asked[:n.value])


@pytest.mark.parametrize("G,room,want", [(8, 8, [8]), (8, 5, [8, 4]), (75, 3, [75, 38, 19, 10, 5, 3]), (7, 1, [7, 4, 2, 1]),
                                         (1, 1, [1])])
def test_groups_shrink_to_what_fits(G, room, want):
    assert _shrink(G, room) == (want[-1], OK, want)


def test_no_room_for_one_item_is_the_allocators_error():
    assert _shrink(5, 0) == (1, NO_MEMORY, [5, 3, 2, 1])
    assert _shrink(5, 5, other=1) == (5, INVALID, [5])      # another error is not a matter of size


@pytest.mark.parametrize("total,G", [(1, 1), (24, 8), (25, 8), (2 ** 31 - 1, 9830400), (3 * (2 ** 31 - 1), 9830400)])
def test_groups_cover_every_item(total, G):
    lib = load("scratch")
    n, last, items = C.c_longlong(), C.c_longlong(), C.c_longlong()
    lib.walk.argtypes = [C.c_longlong, C.c_int] + [C.POINTER(C.c_longlong)] * 3
    lib.walk(total, G, C.byref(n), C.byref(last), C.byref(items))
    assert (n.value, last.value, items.value) == (-(-total // G), (total - 1) // G * G, total)


@pytest.mark.parametrize("per", [1, 8, 11, 2 ** 30, 2 ** 31 - 1])
def test_wavelength_of_a_field(per):
    lib = load("scratch")
    lib.lambda_at.argtypes = [C.c_longlong, C.c_int, C.c_int]
    for first in {0, per - 1, per, 2 * per - 1, 2 * per + per // 2}:
        for f in {0, 1, min(per, 9830399)}:
            assert lib.lambda_at(first, f, per) == (first + f) // per
