"""The t-SURFF flux where its (momentum, orbital) pairs and entry splits can go wrong: one orbital and
more momenta than a CTA has threads, orbital counts that do not divide a CTA, a single momentum.
complex128 against the oracle to 1e-12 of the largest amplitude."""
import numpy as np
import pytest

import oracle
from paper_1912_07921_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orb,n_p", [(1, 300), (17, 31), (5, 1), (3, 171)])
def test_flux_pairs(n_orb, n_p):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import System
    spec = I.SystemSpec(nx=18, ny=15, nz=20, h=0.3, fd_order=4, n_orb=n_orb, n_atoms=1, gauge=I.GAUGE_LENGTH, amp=0.2,
                        omega=0.7, pol=(0.3, -0.2, 0.9), dt=0.02, seed=17)
    inp = I.make_inputs(spec)
    p = np.random.default_rng(n_p).normal(0.0, 1.0, (n_p, 3))
    box = (4, 13, 2, 11, 5, 16)
    s = System(spec, inp, stream=torch.cuda.current_stream().cuda_stream)
    s.set_tsurff(box, p)
    s.propagate(0.0, spec.dt, 3, 1)
    b, _ = s.tsurff()
    s.close()
    b_o = oracle.System(spec, inp).propagate_tsurff(inp.psi0, 0.0, spec.dt, 3, 1, box, p)[2]
    assert np.max(np.abs(b - b_o)) < 1e-12 * np.max(np.abs(b_o))


