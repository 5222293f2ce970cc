"""The exchange hook of a state-parallel system gets device buffers whatever was set up before it: a system
that has the Hartree term's density buffer already, and one whose first attempt ran out of memory.  Host
code on a runtime without a GPU."""
import ctypes

import numpy as np
import pytest

from paper_1912_07921_gb300 import _lib
from tests import _fake

ENOMEM, LDA, HARTREE = 2, 1, 2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _fake.load(tmp_path_factory.mktemp("fake"))


def _buffers_of_a_step(lib, s, n):
    seen = []
    hook = _lib.EXCHANGE_FN(lambda ptr, n, stream, ctx: seen.append((ptr, n)) or 0)
    sums = []

    def launch(name, grid, block, args):
        if b"finalize_kernel" in name:
            # (obs_part, n_items, lda_part, n_lda, sums, rec, ...)
            sums.append(ctypes.cast(args[4], ctypes.POINTER(ctypes.c_void_p))[0])
        return 0.0

    cb = _fake.HOOK(launch)
    lib.fake_set_hook(cb)
    rc = lib.tdks_set_exchange(s, ctypes.cast(hook, ctypes.c_void_p), None)
    if rc == 0:
        psi = np.zeros(2 * n)
        assert lib.tdks_set_orbitals(s, psi.ctypes.data) == 0
        assert lib.tdks_propagate_n(s, 0.0, 0.001, 1, 1) == 0, lib.tdks_last_error()
    lib.fake_set_hook(_fake.HOOK())
    return rc, seen, sums


@pytest.mark.parametrize("xc", [LDA, HARTREE])
def test_buffers(lib, xc):
    s = _fake.create(lib, 9, 8, 7)
    assert lib.tdks_set_xc(s, xc, 2.0) == 0
    rc, seen, sums = _buffers_of_a_step(lib, s, 9 * 8 * 7)
    assert rc == 0
    assert [n for _, n in seen] == [9 * 8 * 7, 4] and all(p for p, _ in seen)
    assert sums == [seen[1][0]]
    lib.tdks_destroy(s)


@pytest.mark.parametrize("fails", [1, 2])
def test_buffers_after_a_failure(lib, fails):
    s = _fake.create(lib, 9, 8, 7)
    lib.fake_fail_malloc(fails)
    assert _buffers_of_a_step(lib, s, 9 * 8 * 7)[0] == ENOMEM
    lib.fake_fail_malloc(0)
    rc, seen, sums = _buffers_of_a_step(lib, s, 9 * 8 * 7)
    assert rc == 0 and len(seen) == 2 and all(p for p, _ in seen) and sums == [seen[1][0]]
    lib.tdks_destroy(s)
