"""Setting up the Hartree term when it cannot be: device memory that runs out in any of its allocations,
and cell edges whose transforms are refused.  Host code on a runtime without a GPU."""
import os
import subprocess
import sys

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


# edges with more radices than a plan has room for (3^17 on the last axis: seventeen), and just past 1024
LONG = """
import sys
from tests import _fake
lib = _fake.load(sys.argv[1])
for n in (3 ** 7, 1025, 2 ** 20, 3 ** 13, 3 ** 17):
    for dims in ((n, 2, 2), (2, n, 2), (2, 2, n)):
        s = _fake.create(lib, *dims, bc=1)
        assert lib.tdks_set_xc(s, 2, 2.0) == 1, dims
        lib.tdks_destroy(s)
s = _fake.create(lib, 4, 1024, 2, bc=1)
assert lib.tdks_set_xc(s, 2, 2.0) == 0
"""


def test_edges_that_are_too_long_are_refused(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    # (a process of its own: an overrun of the plan ends it)
    r = subprocess.run([sys.executable, "-c", LONG, str(tmp_path)], cwd=root, capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
