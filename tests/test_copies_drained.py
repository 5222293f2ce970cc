"""A call that copies to or from the caller's buffer and fails half-way has waited for its copies when it
returns: the caller may free the buffer.  Host code on a runtime without a GPU."""
import numpy as np
import pytest

from tests import _fake

EDEVICE = 5


@pytest.mark.parametrize("call", ["get", "set"])
def test_failing_launches(tmp_path, call):
    lib = _fake.load(tmp_path)
    s = _fake.create(lib, 96, 96, 96)
    host = np.zeros(2 * 96 ** 3)
    assert lib.tdks_set_orbitals(s, host.ctypes.data) == 0
    assert lib.tdks_get_orbitals(s, host.ctypes.data) == 0
    run = lib.tdks_get_orbitals if call == "get" else lib.tdks_set_orbitals
    for n in (1, 2, 3):  # (four chunks down, eight up)
        lib.fake_fail_launch(n)
        assert run(s, host.ctypes.data) == EDEVICE
        assert lib.fake_copies_in_flight() == 0
    assert run(s, host.ctypes.data) == 0 and lib.fake_copies_in_flight() == 0
    lib.tdks_destroy(s)
