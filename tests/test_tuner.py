"""The tuners keep the fastest shape of short sweeps too, of which a single launch between two events seems
longer than one of many, and time shapes that are far behind with one launch.  Host code on a runtime without
a GPU, with the kernels' times given, 5 us of host work a launch and 2.5 us between an event and a kernel (a
24^3 box on a GB300: 8.9 us alone, 6.3 among others)."""
import ctypes
import re

import numpy as np
import pytest

from paper_1912_07921_gb300 import inputs as I
from tests import _fake

REPS = 10


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    lib = _fake.load(tmp_path_factory.mktemp("fake"))
    lib.fake_times(5.0, 2.5)
    return lib


def _system(lib, prec, n=12):
    s = _fake.create(lib, n, n, n, order=8, prec=prec, n_orb=3)
    assert lib.tdks_set_orbitals(s, np.zeros(2 * 3 * n ** 3).ctypes.data) == 0
    assert lib.tdks_set_clock(s, 0.0, 0.001, 1) == 0
    return s


def _tune(lib, prec, batch, us):
    """Shapes kept and launches of each kernel, (mode, its tile and block): number."""
    systems = [_system(lib, prec) for _ in range(2 if batch else 1)]
    count = {}

    def launch(name, grid, block, args):
        m = re.search(rb"ws_sweep_(?:batch_)?kernelI((?:Li\d+E)+)E", name)
        if not m:
            return 0.0
        v = tuple(int(x) for x in re.findall(rb"Li(\d+)E", m.group(1)))
        mode, kernel = v[2], v[3:8]  # (M, precision, mode, TX, TY, R, RX, planes[, periodic])
        count[mode, kernel] = count.get((mode, kernel), 0) + 1
        return us(mode, kernel)

    cb = _fake.HOOK(launch)
    lib.fake_set_hook(cb)
    got, kept = ctypes.c_int(), []
    if batch:
        b = ctypes.c_void_p()
        assert lib.tdks_batch_create((ctypes.c_void_p * 2)(*[s.value for s in systems]), 2, None, ctypes.byref(b)) == 0
        assert lib.tdks_batch_autotune(b, REPS, None) == 0
    else:
        assert lib.tdks_autotune(systems[0], REPS, None) == 0
    for k in range(4):
        rc = lib.tdks_batch_get_shape(b, k, ctypes.byref(got)) if batch else \
            lib.tdks_get_sweep_shape(systems[0], k, ctypes.byref(got))
        assert rc == 0
        kept.append(got.value)
    if batch:
        lib.tdks_batch_destroy(b)
    for s in systems:
        lib.tdks_destroy(s)
    lib.fake_set_hook(_fake.HOOK())
    return kept, count


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("base", [6.0, 12.0, 40.0])
def test_short_sweeps(lib, batch, base):
    # complex64: shape 8's kernel for terms 1 to 3, shape 4's for the last, are the fastest by a twentieth
    best = {0: (16, 12, 2, 2, 2), 1: (16, 12, 2, 2, 2), 2: (14, 8, 2, 1, 1)}
    kept, _ = _tune(lib, I.PREC_C64, batch, lambda mode, k: base * (0.95 if k == best[mode] else 1.0))
    assert kept == [8, 8, 8, 4]
    # complex128: shape 3's
    kept, _ = _tune(lib, I.PREC_C128, batch, lambda mode, k: base * (0.95 if k == (16, 8, 1, 1, 1) else 1.0))
    assert kept == [3, 3, 3, 3]


@pytest.mark.parametrize("batch", [False, True])
def test_long_sweeps_that_are_behind_are_launched_twice(lib, batch):
    slow = (16, 8, 1, 1, 1)
    kept, count = _tune(lib, I.PREC_C128, batch, lambda mode, k: 1500.0 if k == slow else 1000.0 + k[1] * 10 + k[4])
    assert kept == [0, 0, 0, 0]
    assert all(n == (2 if k == slow else 2 + REPS) * (2 if mode == 1 else 1) for (mode, k), n in count.items())
