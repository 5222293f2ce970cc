"""A batch of more systems than the batched potential kernel gives 8 CTAs each in one round (two rounds, one CTA
for the smallest), some with projectors: every system as alone."""
import numpy as np
import pytest

from paper_1912_07921_gb300 import inputs as I
from tests._util import rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(I.PREC_C64, 1e-6), (I.PREC_C128, 1e-13)])
def test_a_hundred_systems(prec, tol):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import Batch, System
    stream = torch.cuda.current_stream().cuda_stream
    rng = np.random.default_rng(19)
    specs = []
    for i in range(100):
        nx, ny, nz = (int(v) for v in rng.integers(6, 26 if i % 9 == 0 else 12, 3))
        specs.append(I.SystemSpec(nx=nx, ny=ny, nz=nz, h=0.3, fd_order=4, prec=prec, n_orb=int(rng.integers(1, 4)),
                                  n_atoms=i % 3, projectors=i % 3 > 0, gauge=I.GAUGE_LENGTH, amp=0.05, omega=0.3,
                                  r_cut=1.0, dt=0.015, seed=900 + i))
    inps = [I.make_inputs(s) for s in specs]
    systems, alone = ([System(s, i, stream=stream) for s, i in zip(specs, inps)] for _ in range(2))
    for s, sp in zip(systems, specs):
        s.set_clock(0.0, sp.dt, 1)
    b = Batch(systems, stream=stream)
    b.propagate(3)
    for s, a, sp in zip(systems, alone, specs):
        a.propagate(0.0, sp.dt, 3, 1)
        assert rel_err(s.get_orbitals(), a.get_orbitals()) < tol
        assert rel_err(s.reductions(0, 3), a.reductions(0, 3)) < tol
    b.close()
    for s in systems + alone:
        s.close()
