"""The triangular pair contraction of the U vector at sizes where a batch of 256 pairs starts or ends inside an
orbital's pairs (17 orbitals: one batch; 23 and 24: two): forces against the oracle, to the plain path's target of
1e-7 Ha/bohr in FP64 and the FP32 grids' 1e-5 in the mixed form."""
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_occ", [17, 23, 24])
def test_forces(n_occ):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    from oracle import forces
    spec = replace(bi.small16(), n_occ=n_occ)
    ref = forces.bse_forces(spec, tol=1e-11)
    for precision, tol_w, tol_f in ((0, 1e-9, 1e-7), (1, 1e-6, 1e-5)):
        s = p.BSESystem(spec, gs_tol=1e-11, precision=precision)
        try:
            w = s.davidson(1, tol=1e-9 if precision == 0 else 1e-6)[0]
            F = np.asarray(s.forces(0))
        finally:
            s.close()
        assert abs(float(w[0]) - ref.omega[0]) < tol_w
        assert np.abs(F - ref.F).max() < tol_f
