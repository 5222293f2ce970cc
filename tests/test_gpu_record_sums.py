"""The record's sums over the grid meet in FP64 in complex64 systems too: a density whose sum needs more
bits than a pair of FP32 numbers has, and fewer than FP64 has, is counted exactly.

Every value of the density is p^2 2^-50 with an odd p of at most 12 bits, except for one point of 1: each is
an FP32 number, so what a point adds is exact, every partial sum is a multiple of 2^-50 below 2, exact in
FP64 in any order, and the electron count has to be equal to the sum.  (As pairs of FP32 numbers, one of which
is 1, sums round at 2^-47 and above.)
"""
import ctypes

import numpy as np
import pytest

from paper_1912_07921_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# grids of the launch's CTAs of 32, 64, 128 and 256 threads
@pytest.mark.parametrize("grid", [(8, 8, 8), (27, 30, 25), (33, 30, 32), (40, 50, 40), (60, 56, 50)])
def test_electron_count_is_exact(grid):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import System
    nx, ny, nz = grid
    spec = I.SystemSpec(nx=nx, ny=ny, nz=nz, h=1.0, fd_order=4, prec=I.PREC_C64, n_orb=1, n_atoms=0, wells=False,
                        occ=1.0, xc=I.XC_NONE, gauge=I.GAUGE_NONE)
    rng = np.random.default_rng(nx)
    p = 2 * rng.integers(0, 2048, nx * ny * nz) + 1
    big = int(rng.integers(0, p.size))
    psi = p * 2.0 ** -25
    psi[big] = 1.0
    want = 2 ** 50 + sum(int(v) ** 2 for i, v in enumerate(p) if i != big)
    assert want < 2 ** 52
    s = System(spec, None, stream=torch.cuda.current_stream().cuda_stream,
               orbitals=psi.reshape(1, nz, ny, nx, 1).astype(np.complex128))
    rec = s.observe(0.0, 0.0)
    s.close()
    assert rec[1] == want * 2.0 ** -50
