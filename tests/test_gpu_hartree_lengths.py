"""The Hartree transforms at line lengths that take every radix, odd lengths and odd numbers of
lines, against the FP64 oracle: the recorded energy with Hartree minus the one without is E_H, and a
complex128 propagation follows the oracle's.

Tolerance: FP64 transforms of up to 100 points, 1e-12 relative as for the other complex128 paths.
"""
import numpy as np
import pytest

import oracle
from paper_1912_07921_gb300 import inputs as I
from tests._util import bloch_cell, bloch_inputs, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# cells transform n points (radices 2, 3, 4, 5, 7, 8, 11, 13); boxes the smallest 2^a 3^b >= 2n - 1
CELLS = [(8, 7, 5), (16, 9, 11), (13, 4, 6), (22, 10, 14), (3, 32, 2)]
BOXES = [(5, 9, 14), (7, 3, 24), (17, 16, 13)]


def _check(spec, inp):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import System
    s = System(spec, inp, stream=torch.cuda.current_stream().cuda_stream)
    s.propagate(0.0, spec.dt, 2, 1)
    rec, psi = s.reductions(0, 2), s.get_orbitals()
    s.close()
    psi_o, rec_o = oracle.System(spec, inp).propagate(inp.psi0, 0.0, spec.dt, 2, 1)
    assert rel_err(psi, psi_o) < 1e-12
    assert np.max(np.abs(rec - rec_o)) < 1e-12 * max(1.0, np.max(np.abs(rec_o)))


@pytest.mark.parametrize("grid", CELLS)
def test_cell(grid):
    nx, ny, nz = grid
    spec = bloch_cell(I.PREC_C128, nx=nx, ny=ny, nz=nz, n_orb=2, n_k=1, n_atoms=0, projectors=False,
                      gauge=I.GAUGE_NONE, xc=I.XC_LDA_X_HARTREE, dt=0.01)
    _check(spec, bloch_inputs(spec))


@pytest.mark.parametrize("grid", BOXES)
def test_box(grid):
    nx, ny, nz = grid
    spec = I.SystemSpec(nx=nx, ny=ny, nz=nz, h=0.4, fd_order=4, n_orb=2, n_atoms=1, gauge=I.GAUGE_LENGTH, amp=0.05,
                        omega=0.3, dt=0.01, xc=I.XC_LDA_X_HARTREE, seed=12)
    _check(spec, I.make_inputs(spec))
