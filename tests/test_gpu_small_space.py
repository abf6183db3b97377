"""Ground states of a cell so small that the Davidson subspace may span everything (123 plane waves, blocks of up to
96): relaxations of six copies side by side, whose host eigensolves share a thread pool and so round differently
from run to run, all converge.  (With a restart whenever a block might not fit, about one relaxation in sixty ended
in a ground state that stood still: 48 of them find that with a probability of one half, and in the loop that
counted them, 0 of 600 failed afterwards.)"""
import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_relaxations_side_by_side():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    h = bi.hartree_model(bi.micro())
    for _ in range(8):
        b = p.BSEBatch([h] * 6, n_workers=6, precision=0, gs_tol=1e-12)
        try:
            def gs(system, pos):
                d = pos - h.pos
                return 0.1 * float((d * d).sum()), -0.2 * d

            out, E, w, evals, st = b.relax(gs, fmax=2e-5, max_steps=400, davidson_tol=1e-10, zvector_tol=1e-11)
            assert st == 0, [b.error(i) for i in range(6)]
            assert np.ptp(w) < 1e-6
        finally:
            b.close()
