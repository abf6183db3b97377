"""The FP64 K1d contraction in fixed point (16 orbitals and more) against the oracle, at the sizes where its
tiling can go wrong: one, two and three 8-orbital columns with a last column of 1..8 orbitals, an odd number
of columns (the 8-row chunk) and an even one, an odd number of orbitals (packed partners change parity
from vector to vector), a ragged last 32-point tile, one to three vectors per call.

The oracle's orbitals and the library's carry a rotation within the occupied space of the ground-state
residual (3e-13) over the smallest occupied level spacing; rows are compared to 2e-9 of their largest
entry, as in the mid-size parity tests, and the contraction itself to 1e-13 by its symmetry:
<b, K1d a> = <a, K1d b> for any two vectors (exact up to the rounding of the sums and transforms).
"""
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NO_K1E, NO_K1D = 1, 2


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    return p


def _spec(n_occ, grid):
    return replace(bi.small16(), n_occ=n_occ, grid=(grid,) * 3)


@pytest.mark.parametrize("n_occ,grid", [(16, 24), (17, 25), (19, 24), (24, 25), (31, 24), (33, 25)])
def test_rows_and_symmetry(pkg, n_occ, grid):
    from oracle import liouville, model
    spec = _spec(n_occ, grid)
    o = liouville.Liouville(spec, gs=model.GroundState(spec, all_states=True))
    s = pkg.BSESystem(spec, gs_tol=3e-13)
    d = pkg.BSESystem(spec, gs_tol=3e-13, flags=NO_K1E | NO_K1D)
    k = pkg.BSESystem(spec, gs_tol=3e-13, flags=NO_K1E)
    try:
        g = bi.gauge_vector(spec.lattice, spec.ecut)
        P = s.ground_state()[1].cpu().numpy()
        sg = np.sign(P @ g)

        def trials(X):
            out = []
            for i in range(3):
                A = X * bi.covariant_weights(spec.lattice, spec.ecut, i)[None, :]
                out.append(A - (A @ X.T) @ X)
            return np.stack(out)

        A = trials(P)
        ref = np.stack([o.basis.full_to_real(o.apply(o.basis.real_to_full(t))) for t in trials(o.gs.X)])
        for nb in (1, 2, 3):
            got = s.apply(torch.tensor(A[:nb], device="cuda")).cpu().numpy() * sg[None, :, None]
            assert np.abs(got - ref[:nb]).max() < 2e-9 * np.abs(ref).max(), nb
        At = torch.tensor(A, device="cuda")
        K = (d.apply(At) - k.apply(At)).reshape(3, -1)      # K1d A
        G = At.reshape(3, -1) @ K.T
        assert (G - G.T).abs().max().item() < 1e-13 * G.abs().max().item()
    finally:
        for x in (s, d, k):
            x.close()


def test_non_finite_point_stays_a_nan(pkg):
    """A NaN in a trial vector is not swallowed by the integer sums."""
    s = pkg.BSESystem(_spec(16, 24), gs_tol=1e-10)
    try:
        A = torch.randn(1, 16, s.n_pw, dtype=torch.float64, device="cuda")
        A[0, 3, 5] = float("nan")
        torch.cuda.synchronize()
        assert torch.isnan(s.apply(A)[0, 7]).any()
    finally:
        s.close()
