"""Sweep shapes that take two planes at a time or blocks of 2 x 2 points, and every shape in cells of order
8 (where some run another's kernel), against the FP64 oracle where blocks, tiles and periodic images can
go wrong: odd edges (blocks half outside a box), edges below and just past a tile, cells smaller
than the tile, odd cells (which run another shape), spheres across the faces, the velocity gauge
with all three components and the current's gradients.

Tolerances: one H application in FP32, 5e-6 of the largest value; two steps of a few
applications each, 2e-5 (the complex64 tolerances of the other parity tests).
"""
import numpy as np
import pytest

import oracle
from paper_1912_07921_gb300 import inputs as I
from tests._util import bloch_cell, bloch_inputs, ragged_molecule, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOXES = [(37, 21, 19), (16, 12, 9), (17, 25, 6), (5, 5, 5)]
CELLS = [(18, 14, 9), (34, 26, 5), (2, 2, 2), (16, 24, 7), (13, 12, 10)]


def _check(spec, inp, shape):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import System
    s = System(spec, inp, stream=torch.cuda.current_stream().cuda_stream)
    s.set_sweep_shape(-1, shape)
    o = oracle.System(spec, inp)
    psi = I.random_orbitals(spec, 33).astype(np.complex64).astype(np.complex128)
    packed = s.pack(psi)
    x = torch.from_numpy(packed.view(np.float32)).cuda()
    y = torch.empty_like(x)
    s.apply_H(0.4, x.data_ptr(), y.data_ptr())
    got = s.unpack(y.cpu().numpy().view(np.complex64).reshape(packed.shape))
    assert rel_err(got, o.apply_H(psi, 0.4, o.vx_of(inp.psi0))) < 5e-6
    s.propagate(0.0, spec.dt, 2, 2)
    rec, out = s.reductions(0, 2), s.get_orbitals()
    s.close()
    psi_o, rec_o = o.propagate(inp.psi0, 0.0, spec.dt, 2, 2)
    assert rel_err(out, psi_o) < 2e-5
    assert np.max(np.abs(rec - rec_o)) < 2e-5 * max(1.0, np.max(np.abs(rec_o)))


@pytest.mark.parametrize("shape", [6, 7, 8])
@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("grid", BOXES)
def test_blocks_in_a_box(shape, order, grid):
    nx, ny, nz = grid
    spec = ragged_molecule(I.PREC_C64, fd_order=order, n_orb=11, nx=nx, ny=ny, nz=nz, n_atoms=3)
    _check(spec, I.make_inputs(spec), shape)


@pytest.mark.parametrize("shape", [6, 7, 8])
@pytest.mark.parametrize("grid", CELLS)
def test_blocks_in_a_cell(shape, grid):
    nx, ny, nz = grid
    spec = bloch_cell(I.PREC_C64, n_orb=2 if nx == 2 else 5, n_k=2, nx=nx, ny=ny, nz=nz)
    _check(spec, bloch_inputs(spec), shape)


@pytest.mark.parametrize("shape", range(9))
@pytest.mark.parametrize("order,grid", [(4, (18, 14, 9)), (8, (18, 14, 9)), (8, (17, 25, 10))])
def test_every_shape_in_a_cell(shape, order, grid):
    nx, ny, nz = grid
    spec = bloch_cell(I.PREC_C64, n_orb=5, n_k=2, nx=nx, ny=ny, nz=nz, fd_order=order)
    _check(spec, bloch_inputs(spec), shape)
