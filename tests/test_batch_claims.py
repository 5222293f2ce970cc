"""The batched sweep's claim counter after a sweep that gave up: a CTA that gives up a bounded wait claims
nothing more, so the counter does not return to zero by itself.  The next propagation, or tuning, starts its
claims at zero all the same.  Host code on a runtime without a GPU, on which the test sets the counter as
such a sweep leaves it."""
import ctypes

import numpy as np
import pytest

from tests import _fake


class SweepArgs(ctypes.Structure):  # BatchSweepArgs
    _fields_ = [("sp", ctypes.c_void_p), ("maps", ctypes.c_void_p), ("term", ctypes.c_int),
                ("begin", ctypes.c_void_p), ("n_sys", ctypes.c_int), ("total", ctypes.c_long),
                ("work", ctypes.POINTER(ctypes.c_uint)), ("item_sys", ctypes.c_void_p)]


@pytest.mark.parametrize("again", ["propagate", "autotune"])
def test_claims_start_at_zero(tmp_path, again):
    lib = _fake.load(tmp_path)
    systems = []
    for n in (9, 11):
        s = _fake.create(lib, n, n, n)
        assert lib.tdks_set_orbitals(s, np.zeros(2 * n ** 3).ctypes.data) == 0
        assert lib.tdks_set_clock(s, 0.0, 0.001, 1) == 0
        systems.append(s)
    b = ctypes.c_void_p()
    arr = (ctypes.c_void_p * 2)(*[s.value for s in systems])
    assert lib.tdks_batch_create(arr, 2, None, ctypes.byref(b)) == 0
    starts = []

    def launch(name, grid, block, args):
        if b"ws_sweep_batch_kernel" in name:
            a = ctypes.cast(args[0], ctypes.POINTER(SweepArgs)).contents
            starts.append(a.work[0])
            a.work[0] = 3 if len(starts) == 4 else 0  # the first step's last sweep gives up
        return 1.0

    cb = _fake.HOOK(launch)
    lib.fake_set_hook(cb)
    assert lib.tdks_batch_propagate(b, 1, 0) == 0
    assert (lib.tdks_batch_propagate(b, 1, 0) if again == "propagate" else lib.tdks_batch_autotune(b, 1, None)) == 0
    assert len(starts) > 4 and not any(starts)
    lib.tdks_batch_destroy(b)
    for s in systems:
        lib.tdks_destroy(s)
