"""Runs of the same work give the same bits.  The sweeps' rings are refilled by copies of the asynchronous proxy
while warps still read other slots: where a copy is not ordered after the reads of the slot it overwrites, a
value in some 10^12 is wrong, now and then.  Sweeps whose centre slots are handed back long before their
values are used (two planes at a time, few slots), over a few hundred sub-steps, three times each."""
import dataclasses

import numpy as np
import pytest

from paper_1912_07921_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _inputs(spec):
    inp = I.make_inputs(dataclasses.replace(spec, n_orb=1, n_k=1))
    rng = np.random.default_rng(spec.seed)
    shape = (spec.n_k, spec.nz, spec.ny, spec.nx, spec.n_orb)
    inp.psi0 = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / np.sqrt(spec.n_points * spec.h ** 3)
    return inp


@pytest.mark.parametrize("what", ["batch", "box"])
def test_three_runs(what):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import Batch, System
    stream = torch.cuda.current_stream().cuda_stream
    specs = I.batched_systems(24) if what == "batch" else [I.medium_molecule(n_orb=16)]
    inps = [_inputs(s) for s in specs]
    systems = [System(s, i, stream=stream) for s, i in zip(specs, inps)]
    for s, sp in zip(systems, specs):
        s.set_clock(0.0, sp.dt, sp.substeps)
    b = Batch(systems, stream=stream)
    for k, shape in enumerate((6, 8, 8, 2)):
        b.set_shape(k, shape)
    first = None
    for _ in range(3):
        for s, i, sp in zip(systems, inps, specs):
            s.set_orbitals(i.psi0)
            s.set_clock(0.0, sp.dt, sp.substeps)
        b.propagate(200 if what == "batch" else 50)
        out = [(s.get_orbitals(), s.reductions(s.step_count() - 5, 5)) for s in systems]
        first = first or out
        for (psi, rec), (psi1, rec1) in zip(out, first):
            assert np.array_equal(psi, psi1) and np.array_equal(rec, rec1)
    b.close()
    for s in systems:
        s.close()
