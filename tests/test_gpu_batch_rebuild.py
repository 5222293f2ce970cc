"""A batch whose tables are rebuilt between propagations (every shape in turn, the new tensor maps where the old
ones were) gives each system what it gives alone with the same shapes."""
import numpy as np
import pytest

from paper_1912_07921_gb300 import inputs as I
from tests._util import rel_err, small_uneven_batch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(I.PREC_C64, 1e-6), (I.PREC_C128, 1e-13)])
def test_every_shape_in_turn(prec, tol):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import Batch, System, shape_count
    stream = torch.cuda.current_stream().cuda_stream
    specs = small_uneven_batch(prec, n=4, seed=23)
    inps = [I.make_inputs(s) for s in specs]
    systems, alone = ([System(s, i, stream=stream) for s, i in zip(specs, inps)] for _ in range(2))
    for s, sp in zip(systems, specs):
        s.set_clock(0.0, sp.dt, 1)
    b = Batch(systems, stream=stream)
    for n in range(2 * shape_count()):
        shape = (4 * n + 1) % shape_count()
        b.set_shape(-1, shape)
        b.propagate(1, use_graph=n % 2 == 0)
        for s, sp in zip(alone, specs):
            s.set_sweep_shape(-1, shape)
            s.propagate(n * sp.dt, sp.dt, 1, 1)
    for s, a in zip(systems, alone):
        assert rel_err(s.get_orbitals(), a.get_orbitals()) < tol
    b.close()
    for s in systems + alone:
        s.close()
