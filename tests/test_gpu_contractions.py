"""The density and pair contractions of the operators at the sizes where their indexing can go wrong: odd
and even orbital counts, blocks of one to five vectors (four, two and one at a time), pair batches that
start and end inside an orbital's pairs (more than 256 pairs, not a multiple).

The exchange term K1e A (Eq. 2b) and the coupling block (Sec. SI) against the oracle, FP64: the orbitals'
residual rotation (3e-13 over the smallest level spacing) allows 2e-9 of the largest entry; the forces,
which run the triangular pair contraction of the U vector, to 1e-7 Ha/bohr, the plain path's target."""
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NO_K1D = 2


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    return p


@pytest.mark.parametrize("n_occ", [4, 17, 24])
def test_exchange_and_coupling(pkg, n_occ):
    from oracle import liouville, model
    spec = replace(bi.small16(), n_occ=n_occ)
    gs = model.GroundState(spec, all_states=True)
    g = bi.gauge_vector(spec.lattice, spec.ecut)
    for k1d in (False, True):
        o = liouville.Liouville(spec, gs=gs, k1d=k1d)
        s = pkg.BSESystem(spec, gs_tol=3e-13, flags=0 if k1d else NO_K1D)
        try:
            P = s.ground_state()[1].cpu().numpy()
            sg = np.sign(P @ g)

            def trials(X):
                out = []
                for i in range(5):
                    A = X * bi.covariant_weights(spec.lattice, spec.ecut, i % 3)[None, :] * (1 + 0.1 * i)
                    out.append(A - (A @ X.T) @ X)
                return np.stack(out)

            A, Ao = trials(P), trials(o.gs.X)
            if k1d:
                ref = np.stack([o.basis.full_to_real(o.apply_B(o.basis.real_to_full(t))) for t in Ao[:2]])
                got = s.apply(torch.tensor(A[:2], device="cuda"), op=3).cpu().numpy() * sg[None, :, None]
                assert np.abs(got - ref).max() < 2e-9 * np.abs(ref).max()
                continue
            ref = np.stack([o.basis.full_to_real(o.apply(o.basis.real_to_full(t))) for t in Ao])
            for nb in (1, 3, 5):
                got = s.apply(torch.tensor(A[:nb], device="cuda")).cpu().numpy() * sg[None, :, None]
                assert np.abs(got - ref[:nb]).max() < 2e-9 * np.abs(ref).max(), nb
        finally:
            s.close()
