"""Tables and fills of a set-up are in place for the kernels of a system on a stream of its own, which nothing
orders after the default stream: every kind of set-up, then the kernels that read it.  Host code on a runtime
without a GPU."""
import ctypes

import numpy as np
import pytest

from tests import _fake

HARTREE, C64, STREAM = 2, 1, 0x10  # (any handle but the default stream's)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _fake.load(tmp_path_factory.mktemp("fake"))


def _system(lib, bc, prec, n=12):
    s = _fake.create(lib, n, n, n, bc=bc, prec=prec, stream=STREAM)
    pos, D = np.array([0.4, 0.3, 0.5]), np.ones(4)
    assert lib.tdks_set_atoms_projectors(s, 1, pos.ctypes.data, D.ctypes.data, 0.6, 1.0) == 0
    assert lib.tdks_set_local_potential(s, np.zeros(n ** 3).ctypes.data) == 0
    assert lib.tdks_set_orbitals(s, np.zeros(2 * n ** 3).ctypes.data) == 0
    return s


@pytest.mark.parametrize("prec", [0, C64])
@pytest.mark.parametrize("bc", [0, 1])
def test_one_system(lib, bc, prec):
    s = _system(lib, bc, prec)
    assert lib.tdks_propagate_n(s, 0.0, 0.001, 1, 1) == 0
    assert lib.tdks_set_xc(s, HARTREE, 2.0) == 0
    assert lib.tdks_propagate_n(s, 0.001, 0.001, 1, 1) == 0
    if bc == 0:
        box, p = np.array([3, 8, 3, 8, 3, 8], dtype=np.int32), np.ones((5, 3))
        assert lib.tdks_set_tsurff(s, box.ctypes.data, 5, p.ctypes.data) == 0
        assert lib.tdks_propagate_n(s, 0.002, 0.001, 1, 1) == 0
    assert lib.tdks_autotune(s, 1, None) == 0
    lib.tdks_destroy(s)
    assert lib.fake_unordered_launches() == 0


def test_a_batch(lib):
    systems = [_system(lib, 0, C64, n) for n in (12, 14)]
    for s in systems:
        assert lib.tdks_set_clock(s, 0.0, 0.001, 1) == 0
    b = ctypes.c_void_p()
    arr = (ctypes.c_void_p * 2)(*[s.value for s in systems])
    assert lib.tdks_batch_create(arr, 2, STREAM, ctypes.byref(b)) == 0
    assert lib.tdks_batch_propagate(b, 1, 0) == 0
    assert lib.tdks_batch_set_shape(b, -1, 3) == 0
    assert lib.tdks_batch_propagate(b, 1, 0) == 0
    assert lib.tdks_batch_autotune(b, 1, None) == 0
    lib.tdks_batch_destroy(b)
    for s in systems:
        lib.tdks_destroy(s)
    assert lib.fake_unordered_launches() == 0
