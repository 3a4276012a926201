"""The multiplier and shift that the host gives the kernels for a division (the code compiled with the host
compiler): (n mul) >> (31 + shift), by a 32-bit high product, is n // d for every n below 2^31."""
import ctypes as C

import numpy as np

from tests.native import load


def test_constants_divide():
    lib = load("fastdiv")
    rng = np.random.default_rng(3)
    mul, shift = C.c_uint(), C.c_int()
    ds = {1, 2, 3, 5, 7, 31, 32, 33, 240, 641, 65535, 65537, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, (1 << 31) - 1}
    ds |= {int(x) for x in np.exp(rng.uniform(0, np.log(2.0 ** 31 - 1), 400))}
    for d in sorted(ds):
        lib.constants(d, C.byref(mul), C.byref(shift))
        ns = np.concatenate([rng.integers(0, 1 << 31, 500), [0, 1, d - 1, d, d + 1, (1 << 31) - 1],
                             d * rng.integers(1, (1 << 31) // d + 1, 50) - 1]).astype(np.uint64)
        ns = ns[ns < 1 << 31]
        if d == 1:
            assert shift.value < 0
            continue
        assert shift.value >= 1
        q = (ns * np.uint64(mul.value)) >> np.uint64(32) >> np.uint64(shift.value - 1)
        assert (q == ns // np.uint64(d)).all(), d
