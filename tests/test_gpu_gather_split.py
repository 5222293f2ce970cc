"""The projector gather of a system alone, over the splits that its number of (atom, k-batch) units
selects: 16 shares of a unit on 8 CTAs down to one share on one CTA, shares that straddle CTAs (5, 3),
atoms whose spheres leave some shares empty.  One H application against the FP64 oracle; complex64
5e-6 of the largest value, complex128 1e-12 (the tolerances of the other parity tests).
"""
import numpy as np
import pytest

import oracle
from paper_1912_07921_gb300 import inputs as I
from tests._util import ragged_molecule, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(I.PREC_C64, 5e-6), (I.PREC_C128, 1e-12)])
@pytest.mark.parametrize("n_atoms", [1, 10, 16, 20, 30, 38, 76])  # c64: 16, 8, 5, 4, 3, 2, 1 shares
def test_gather_splits(prec, tol, n_atoms):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1912_07921_gb300.system import System
    spec = ragged_molecule(prec, n_orb=64 if prec == I.PREC_C64 else 8, nx=13, ny=11, nz=9, n_atoms=n_atoms)
    inp = I.make_inputs(spec)
    s = System(spec, inp, stream=torch.cuda.current_stream().cuda_stream)
    real, cplx = (np.float32, np.complex64) if prec == I.PREC_C64 else (np.float64, np.complex128)
    psi = I.random_orbitals(spec, 35).astype(cplx).astype(np.complex128)
    packed = s.pack(psi)
    x = torch.from_numpy(packed.view(real)).cuda()
    y = torch.empty_like(x)
    s.apply_H(0.4, x.data_ptr(), y.data_ptr())
    got = s.unpack(y.cpu().numpy().view(cplx).reshape(packed.shape))
    s.close()
    o = oracle.System(spec, inp)
    assert rel_err(got, o.apply_H(psi, 0.4, o.vx_of(inp.psi0))) < tol
