"""Set-ups of several allocations, the n-th of which fails: the next call of the same kind completes what is
missing (no kernel gets a null pointer) and keeps what is there (nothing is allocated twice).  Host code on a
runtime without a GPU."""
import numpy as np
import pytest

from tests import _fake

ENOMEM, CFM4, ETRS, C64 = 2, 1, 5, 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _fake.load(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("what,blocks", [("cfm4", 4), ("etrs", 6), ("upload", 3)])
def test_every_allocation_failing_in_turn(lib, what, blocks):
    call = {"cfm4": lambda s: lib.tdks_set_propagator(s, CFM4), "etrs": lambda s: lib.tdks_set_propagator(s, ETRS),
            "upload": lambda s: lib.tdks_set_upload_buffers(s, 2)}[what]
    for n in range(1, blocks + 1):
        s = _fake.create(lib, 9, 8, 7, prec=C64)
        assert lib.tdks_set_orbitals(s, np.zeros(2 * 9 * 8 * 7).ctypes.data) == 0
        before = lib.fake_live_blocks()
        lib.fake_fail_malloc(n)
        assert call(s) == ENOMEM
        lib.fake_fail_malloc(0)
        assert call(s) == 0, lib.tdks_last_error()
        assert lib.fake_live_blocks() == before + blocks
        lib.tdks_destroy(s)
