"""A cell's propagation captured into a CUDA graph: the first work of a new system, and a replay after other
calls have formed the projectors' phases of another vector potential.  The replay and uncaptured calls after it
give what an uncaptured system gives, bit for bit."""
import numpy as np
import pytest

from paper_1912_07921_gb300 import inputs as I
from tests._util import bloch_cell, bloch_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [I.PREC_C128, I.PREC_C64])
@pytest.mark.parametrize("before", ["nothing", "a step", "an observation"])
def test_replay(prec, before):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import System
    spec = bloch_cell(prec, dt=0.01)
    inp = bloch_inputs(spec)
    st = torch.cuda.Stream()
    s, ref = System(spec, inp, stream=st.cuda_stream), System(spec, inp, stream=st.cuda_stream)
    if before == "a step":  # leaves the phases of the captured step's vector potential
        for x in (s, ref):
            x.propagate(0.0, spec.dt, 1, 1)
            x.set_orbitals(inp.psi0)
    elif before == "an observation":
        s.observe(0.0, 0.5 * spec.dt)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
        s.propagate(0.0, spec.dt, 1, 1)
    s.observe(0.0, 7.0)  # the phases of another vector potential
    s.set_orbitals(inp.psi0)
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        g.replay()
    st.synchronize()
    ref.propagate(0.0, spec.dt, 1, 1)
    assert np.array_equal(s.get_orbitals(), ref.get_orbitals())
    # the graph's phases are in the table now, whatever the calls before it left
    assert np.array_equal(s.observe(0.0, 7.0), ref.observe(0.0, 7.0))
    s.propagate(spec.dt, spec.dt, 2, 2)
    ref.propagate(spec.dt, spec.dt, 2, 2)
    assert np.array_equal(s.get_orbitals(), ref.get_orbitals())
    s.close()
    ref.close()
