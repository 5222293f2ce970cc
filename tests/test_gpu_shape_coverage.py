"""Sweep kernels that only a default, or a tuner's choice, would run: the default shapes of cells above their
size thresholds (both precisions and orders), complex128 sweeps that take two planes at a time (first term
with records, middle terms), and every such shape in batches of both orders.

Tolerances of the other parity tests: complex128 1e-12 against the oracle and 1e-13 against the system alone,
complex64 2e-5 after two steps and 1e-6 against the system alone.
"""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1912_07921_gb300 import inputs as I
from tests._util import bloch_cell, bloch_inputs, ragged_molecule, rel_err, small_uneven_batch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _system(spec, inp):
    from paper_1912_07921_gb300.system import System
    return System(spec, inp, stream=torch.cuda.current_stream().cuda_stream)


def _two_steps(s, spec, inp, tol):
    s.propagate(0.0, spec.dt, 2, 2)
    rec, psi = s.reductions(0, 2), s.get_orbitals()
    s.close()
    psi_o, rec_o = oracle.System(spec, inp).propagate(inp.psi0, 0.0, spec.dt, 2, 2)
    assert rel_err(psi, psi_o) < tol
    assert np.max(np.abs(rec - rec_o)) < tol * max(1.0, np.max(np.abs(rec_o)))


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("prec,shapes,tol", [(I.PREC_C128, [2, 2, 2, 2], 1e-12), (I.PREC_C64, [6, 6, 6, 3], 2e-5)])
def test_default_shapes_of_a_cell(prec, shapes, tol, order):
    # (12 rows: one tile of 16 x 12, two of 16 x 8; 103 680 or 69 120 points with their orbital batches)
    spec = bloch_cell(prec, fd_order=order, nx=40, ny=12, nz=24, n_orb=10, n_k=3)
    inp = bloch_inputs(spec)
    s = _system(spec, inp)
    assert s.sweep_shapes() == shapes
    _two_steps(s, spec, inp, tol)


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("grid", [(37, 21, 19), (16, 12, 9), (17, 25, 6), (5, 5, 5)])
def test_two_planes_in_complex128(grid, order):
    nx, ny, nz = grid
    spec = ragged_molecule(I.PREC_C128, fd_order=order, n_orb=7, nx=nx, ny=ny, nz=nz, n_atoms=3)
    inp = I.make_inputs(spec)
    s = _system(spec, inp)
    s.set_sweep_shape(-1, 6)
    _two_steps(s, spec, inp, 1e-12)


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("prec,shape", [(I.PREC_C64, 6), (I.PREC_C64, 7), (I.PREC_C64, 8), (I.PREC_C128, 6)])
def test_shapes_in_a_batch(prec, shape, order):
    from paper_1912_07921_gb300.system import Batch
    specs = [dataclasses.replace(s, fd_order=order, dt=0.0125) for s in small_uneven_batch(prec, n=3, seed=17)]
    inps = [I.make_inputs(s) for s in specs]
    alone, systems = [], []
    for spec, inp in zip(specs, inps):
        s = _system(spec, inp)
        s.set_sweep_shape(-1, shape)
        s.propagate(0.0, spec.dt, 2, 1)
        alone.append((s.get_orbitals(), s.reductions(0, 2)))
        s.close()
        systems.append(_system(spec, inp))
        systems[-1].set_clock(0.0, spec.dt, 1)
    b = Batch(systems, stream=torch.cuda.current_stream().cuda_stream)
    b.set_shape(-1, shape)
    b.propagate(2)
    tol = 1e-13 if prec == I.PREC_C128 else 1e-6
    for s, (psi, rec) in zip(systems, alone):
        assert rel_err(s.get_orbitals(), psi) < tol
        assert rel_err(s.reductions(0, 2), rec) < tol
    b.close()
    for s in systems:
        s.close()
