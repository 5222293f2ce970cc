"""Setting up the Hartree term when it cannot be: device memory that runs out in any of its allocations,
and cell edges whose transforms are refused.  Host code on a runtime without a GPU."""
import pytest

from tests import _fake

EINVAL, ENOMEM, HARTREE, LDA = 1, 2, 2, 1


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _fake.load(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("bc", [0, 1])
def test_a_setup_that_ran_out_of_memory_is_done_again(lib, bc):
    s = _fake.create(lib, 12, 10, 9, bc=bc)
    free = lib.fake_live_blocks()
    n = 0
    while True:
        n += 1
        lib.fake_fail_malloc(n)
        rc = lib.tdks_set_xc(s, HARTREE, 2.0)
        lib.fake_fail_malloc(0)
        if rc == 0:
            break
        assert rc == ENOMEM, lib.tdks_last_error()
        assert lib.fake_live_blocks() == free          # nothing half-made is kept
        assert lib.tdks_set_xc(s, LDA, 2.0) == 0       # the system goes on without it
        # the next attempt allocates everything: it fails where it did, not later and not never
        lib.fake_fail_malloc(n)
        assert lib.tdks_set_xc(s, HARTREE, 2.0) == ENOMEM
        lib.fake_fail_malloc(0)
    # the twiddles, the spectrum, the kernel, v_H, the density; a box's kernel transform takes two more
    assert n - 1 == (7 if bc == 0 else 5)
    lib.tdks_destroy(s)
