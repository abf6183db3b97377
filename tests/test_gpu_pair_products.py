"""Pair densities multiplied as the plane passes load them: root and forces by the density-sphere transforms
against the full-grid path, which multiplies them in a pass of its own, for one pair, an odd number of pairs
(the last packed grid holds one) and more than one batch of 256, on a grid with three different axes.
Tolerances: Davidson and Z-vector at 1e-9 and the batch-of-systems bounds for FP32 grids (1e-6 Ha, 1e-5 Ha/bohr)."""
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol_w,tol_f", [(0, 1e-9, 1e-7), (1, 1e-6, 1e-5)])
@pytest.mark.parametrize("n_occ", [1, 2, 23])
def test_both_paths(n_occ, precision, tol_w, tol_f):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    spec = replace(bi.small16(), n_occ=n_occ, grid=(24, 25, 27))
    out = []
    for flags in (0, p.FLAG_FULL_GRID_FFT):
        s = p.BSESystem(spec, flags=flags, gs_tol=1e-11, precision=precision)
        try:
            w = s.davidson(1, tol=1e-9 if precision == 0 else 1e-6)[0]
            s.zvector(0, tol=1e-10)
            out.append((np.asarray(w.cpu() if hasattr(w, "cpu") else w).ravel()[0], np.asarray(s.forces(0))))
        finally:
            s.close()
    assert abs(out[0][0] - out[1][0]) < tol_w
    assert np.abs(out[0][1] - out[1][1]).max() < tol_f
