"""How the batched potential kernel is split over the systems: no slot of the GPU (four CTAs on each of 152
SMs) gets much more than its share of the work, whatever the number of systems.  A point's work: in complex64
the 4 values that do not depend on the orbitals and one per batch of them, as it is bound by the loads; in
complex128 the same for every point, bound by the cube root's FP64 instructions.  Host code on a runtime without a GPU."""
import ctypes
import heapq

import numpy as np
import pytest

from paper_1912_07921_gb300 import inputs as I
from tests import _fake


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _fake.load(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("prec", [I.PREC_C64, I.PREC_C128])
@pytest.mark.parametrize("n", [1, 2, 12, 24, 64, 96, 128, 256])
def test_no_slot_has_a_fifth_more_than_its_share(lib, n, prec):
    specs, systems = I.batched_systems(n), []
    host = np.zeros(2 * max(s.n_points * s.n_orb for s in specs))
    for sp in specs:
        s = _fake.create(lib, sp.nx, sp.ny, sp.nz, h=sp.h, order=sp.fd_order, prec=prec, n_orb=sp.n_orb)
        assert lib.tdks_set_orbitals(s, host.ctypes.data) == 0
        assert lib.tdks_set_clock(s, 0.0, sp.dt, 1) == 0
        systems.append(s)
    b = ctypes.c_void_p()
    assert lib.tdks_batch_create((ctypes.c_void_p * n)(*[s.value for s in systems]), n, None, ctypes.byref(b)) == 0
    ctas = []

    def launch(name, grid, block, args):
        if b"lda_batch_kernel" in name:  # (aux, clocks, first CTA of each system, n)
            begin = ctypes.cast(args[2], ctypes.POINTER(ctypes.POINTER(ctypes.c_long)))[0][:n + 1]
            assert begin[0] == 0 and begin[n] == grid[0]
            ctas.append([begin[i + 1] - begin[i] for i in range(n)])
        return 0.0

    cb = _fake.HOOK(launch)
    lib.fake_set_hook(cb)
    assert lib.tdks_batch_propagate(b, 1, 0) == 0
    lib.fake_set_hook(_fake.HOOK())
    lib.tdks_batch_destroy(b)
    for s in systems:
        lib.tdks_destroy(s)
    work = [sp.n_points * (4 + -(-sp.n_orb // 8) if prec == I.PREC_C64 else 1) for sp in specs]
    slots = [0.0] * (152 * 4)
    for w, k in zip(work, ctas[0]):
        assert k >= 1
        for _ in range(k):  # CTAs start in order, each on the slot that is free first
            heapq.heapreplace(slots, slots[0] + w / k)
    assert max(slots) < 1.2 * sum(work) / len(slots)
