"""The streamed FP32 K1d contraction on shapes that 16-orbital blocks and 32-point tiles do not divide:
mixed-precision rows of one to four vectors against the oracle, for a last block of 1, 3, 8 and 15 orbitals,
an odd number of orbitals (packed partners change parity from vector to vector) and a ragged last tile.
FP32 grid products summed over N_occ terms: 2e-5 of the largest entry, as in the mid-size parity tests."""
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    return p


@pytest.mark.parametrize("n_occ,grid", [(17, 24), (19, 25), (24, 24), (31, 25), (33, 24)])
def test_rows(pkg, n_occ, grid):
    from oracle import liouville, model
    spec = replace(bi.small16(), n_occ=n_occ, grid=(grid,) * 3)
    o = liouville.Liouville(spec, gs=model.GroundState(spec, all_states=True))
    s = pkg.BSESystem(spec, gs_tol=1e-11, precision=1)
    try:
        g = bi.gauge_vector(spec.lattice, spec.ecut)
        P = s.ground_state()[1].cpu().numpy()
        sg = np.sign(P @ g)

        def trials(X):
            out = []
            for i in range(4):
                A = X * bi.covariant_weights(spec.lattice, spec.ecut, i % 3)[None, :] * (1 + 0.1 * i)
                out.append(A - (A @ X.T) @ X)
            return np.stack(out)

        A = trials(P)
        ref = np.stack([o.basis.full_to_real(o.apply(o.basis.real_to_full(t))) for t in trials(o.gs.X)])
        for nb in (1, 2, 3, 4):
            got = s.apply(torch.tensor(A[:nb], device="cuda")).cpu().numpy() * sg[None, :, None]
            assert np.abs(got - ref[:nb]).max() < 2e-5 * np.abs(ref).max(), nb
    finally:
        s.close()


def test_sizes_side_by_side(pkg):
    """Systems that take the same kernels with different shared-memory sizes, launched by four threads at once:
    every launch is accepted, whichever size another thread asked for last."""
    specs = [replace(bi.small16(), n_occ=n) for n in (17, 33, 49, 65)]
    b = pkg.BSEBatch(specs, n_workers=4, precision=1, gs_tol=1e-9, flags=pkg.FLAG_NO_GRAPHS)
    try:
        assert b.setup_status == 0
        for _ in range(16):
            assert b.solve(davidson_tol=1e-5, zvector_tol=1e-5)[2] == 0
    finally:
        b.close()
