"""The FP64 K1d kernel's bounded waits that run out inside the U vector: the call reports it, in both launch shapes
(eight and sixteen consumer warps; 17 orbitals and 101), all warps leave, and the context computes the same
excitation and forces afterwards as before."""
import time
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_occ", [17, 101])
def test_uvector_reports_a_stalled_k1d(n_occ):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    s = p.BSESystem(replace(bi.small16(), n_occ=n_occ), gs_tol=1e-9)
    lib = p.load_library()
    try:
        assert lib.bse_selftest_uvector_stall(s.ctx, 0) == 7  # BSE_ERR_STATE: no roots yet
        s.davidson(1, tol=1e-6)
        before = np.asarray(s.forces(0))
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        st = lib.bse_selftest_uvector_stall(s.ctx, 0)
        dt = time.perf_counter() - t0
        assert st == 6, p.STATUS.get(st, st)                  # BSE_ERR_TIMEOUT
        assert 0.5 < dt < 60.0
        s.zvector(0, tol=1e-10)                               # the flag does not fail the next call
        after = np.asarray(s.forces(0))
        assert np.abs(after - before).max() <= 1e-8 * max(1.0, np.abs(before).max())
    finally:
        s.close()
