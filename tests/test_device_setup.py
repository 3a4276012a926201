"""Set-up that belongs to a device (shared-memory limits of kernels, tables in the module) is done once for each
device, under a lock: a second device gets its own, two threads do it once, and a failure is tried again."""
import ctypes as C
import os
import re

from tests.native import ROOT, load


def _calls(devs, bad=-1):
    lib = load("once")
    st = (C.c_int * len(devs))()
    return lib.calls(len(devs), (C.c_int * len(devs))(*devs), bad, st), list(st)


def test_once_for_each_device():
    assert _calls([0, 0, 1, 0, 1, 5]) == (3, [0] * 6)


def test_a_failed_setup_is_tried_again():
    assert _calls([0, 1, 1, 1, 0], bad=1) == (3, [0, 1, 0, 0, 0])


def test_threads_wait_for_the_one_that_sets_up():
    lib = load("once")
    early = C.c_int()
    assert lib.together(8, C.byref(early)) == 1 and early.value == 0


def test_no_unguarded_flag_stands_for_a_devices_setup():
    """cudaFuncSetAttribute holds for the current device: no process-wide 'done' flag decides about it."""
    csrc = os.path.join(ROOT, "paper_2606_14173_gb300", "csrc")
    for f in sorted(os.listdir(csrc)):
        with open(os.path.join(csrc, f), encoding="utf-8") as fh:
            assert not re.search(r"\bstatic\s+bool\s+\w+\s*=", fh.read()), f
