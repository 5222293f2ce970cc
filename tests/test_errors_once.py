"""A failed CUDA call is reported by the library call that made it, not by the next one as well.  Host code
on a runtime without a GPU."""
import ctypes

import numpy as np
import pytest

from tests import _fake

ENOMEM, EDEVICE, CFM4 = 2, 5, 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _fake.load(tmp_path_factory.mktemp("fake"))


def _system(lib):
    s = _fake.create(lib, 9, 8, 7)
    pos, D = np.array([0.1, 0.0, -0.1]), np.ones(4)
    assert lib.tdks_set_atoms_projectors(s, 1, pos.ctypes.data, D.ctypes.data, 0.6, 1.0) == 0
    psi = np.zeros(2 * 9 * 8 * 7)
    assert lib.tdks_set_orbitals(s, psi.ctypes.data) == 0
    return s


def _observe(lib, s):
    out = np.zeros(8)
    return lib.tdks_observe(s, 0.0, 0.0, out.ctypes.data)


def test_an_allocation(lib):
    s = _system(lib)
    lib.fake_fail_malloc(1)
    assert lib.tdks_set_propagator(s, CFM4) == ENOMEM
    assert _observe(lib, s) == 0, lib.tdks_last_error()
    lib.tdks_destroy(s)


def test_every_launch_of_an_observation(lib):
    s = _system(lib)
    names = []
    cb = _fake.HOOK(lambda name, g, b, a: names.append(name) or 0.0)
    lib.fake_set_hook(cb)
    assert _observe(lib, s) == 0
    lib.fake_set_hook(_fake.HOOK())
    assert len(names) == 5  # potential, projections, their term, sweep, record
    for n in range(1, len(names) + 1):
        lib.fake_fail_launch(n)
        assert _observe(lib, s) == EDEVICE, names[n - 1]
        assert _observe(lib, s) == 0, (names[n - 1], lib.tdks_last_error())
    lib.tdks_destroy(s)
