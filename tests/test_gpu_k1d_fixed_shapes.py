"""The FP64 K1d contraction in the launch shapes of larger cells: sixteen consumer warps (one vector from 98 orbitals
on, two from 49), tau with one bit less (from 129 orbitals), two vectors that no longer fit one launch (from 131),
ragged last columns, odd orbital counts and a ragged last tile of 32 points.

Reference: -sum_v' W*(phi_v' phi_v) a_v' by torch FFTs in FP64 from the library's own orbitals.  The library's term is
the difference of two applies, each good to a few 1e-15 of its largest row entry (transforms and sums), which is at
most about fifty times the term's: 1e-12 of the term's largest entry."""
import math
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NO_K1E, NO_K1D = 1, 2


class _Torch:
    def __init__(self, spec):
        self.spec = spec
        n1, n2, n3 = spec.grid
        self.shape, self.nr = (n3, n2, n1), n1 * n2 * n3
        rec = bi.reciprocal_rows(spec.lattice)
        self.omega = abs(np.linalg.det(spec.lattice))
        mill = np.concatenate([np.zeros((1, 3), int), bi.half_sphere_miller(spec.lattice, spec.ecut)])
        g2 = ((mill @ rec) ** 2).sum(1)
        N = np.array(spec.grid)

        def place(m):
            j = np.mod(m, N)
            return torch.tensor(j[:, 0] + n1 * (j[:, 1] + n2 * j[:, 2]), device="cuda")
        self.ip, self.im = place(mill), place(-mill)
        root_vc = np.where(g2 > 0, np.sqrt(4 * math.pi / np.where(g2 > 0, g2, 1.0)), 0.0)
        self.P = torch.tensor(spec.pdep_coef * np.concatenate([root_vc[:1], np.repeat(root_vc[1:], 2)]), device="cuda")
        lam = torch.tensor(spec.pdep_lambda, device="cuda")
        self.c = lam / (1 - lam)
        f = [np.where(np.arange(m) <= m // 2, np.arange(m), np.arange(m) - m) for m in (n1, n2, n3)]
        m3, m2, m1 = np.meshgrid(f[2], f[1], f[0], indexing="ij")
        q2 = ((np.stack([m1.ravel(), m2.ravel(), m3.ravel()], 1) @ rec) ** 2).sum(1)
        inside = (q2 <= 4 * spec.ecut) & (q2 > 0)
        self.vc = torch.tensor(np.where(inside, 4 * math.pi / np.where(q2 > 0, q2, 1.0), 0.0), device="cuda")

    def spread(self, X):
        c = torch.zeros(X.shape[0], self.nr, dtype=torch.complex128, device="cuda")
        z = torch.complex(X[:, 1::2], X[:, 2::2]) / math.sqrt(2.0)
        c[:, self.ip[1:]], c[:, self.im[1:]] = z, z.conj()
        c[:, self.ip[0]] = X[:, 0].to(torch.complex128)
        return c

    def collect(self, c):
        z = c[:, self.ip[1:]] * math.sqrt(2.0)
        X = torch.empty(c.shape[0], 2 * len(self.ip) - 1, dtype=torch.float64, device="cuda")
        X[:, 0], X[:, 1::2], X[:, 2::2] = c[:, self.ip[0]].real, z.real, z.imag
        return X

    def fft(self, f):
        return torch.fft.fftn(f.reshape(-1, *self.shape), dim=(1, 2, 3)).reshape(f.shape[0], -1) / self.nr

    def ifft(self, c):
        return (torch.fft.ifftn(c.reshape(-1, *self.shape), dim=(1, 2, 3)) * self.nr).real.reshape(c.shape[0], -1)

    def to_grid(self, X):
        return self.ifft(self.spread(X)) / math.sqrt(self.omega)

    def k1d(self, phi, A):
        """P_c of the term for trial vectors A [nb][n_occ][n_pw]."""
        ph, ar = self.to_grid(phi), torch.stack([self.to_grid(a) for a in A])
        y = torch.zeros_like(ar)
        for v in range(self.spec.n_occ):
            d = self.fft(ph * ph[v])
            tau = self.ifft(d * self.vc + self.spread(((self.collect(d) @ self.P.T) * self.c) @ self.P))
            y[:, v] = -(tau * ar).sum(1)
        r = torch.stack([self.collect(self.fft(b)) for b in y]) * math.sqrt(self.omega)
        return r - (r @ phi.T) @ phi


@pytest.mark.parametrize("n_occ,grid", [(50, 25), (65, 24), (101, 25), (129, 24), (140, 25)])
def test_term(n_occ, grid):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    spec = replace(bi.small16(), n_occ=n_occ, grid=(grid,) * 3)
    d = p.BSESystem(spec, gs_tol=1e-9, flags=NO_K1E | NO_K1D)
    k = p.BSESystem(spec, gs_tol=1e-9, flags=NO_K1E)
    try:
        phi = k.ground_state()[1]
        assert torch.equal(phi, d.ground_state()[1])  # the difference of the applies is the term
        A = torch.stack([phi * torch.tensor(bi.covariant_weights(spec.lattice, spec.ecut, i), device="cuda")
                         for i in range(3)])
        A -= (A @ phi.T) @ phi
        ref = _Torch(spec).k1d(phi, A)
        torch.cuda.synchronize()  # the contexts run on streams of their own
        for nb in (1, 2, 3):
            got = k.apply(A[:nb]) - d.apply(A[:nb])
            torch.cuda.synchronize()
            assert (got - ref[:nb]).abs().max().item() < 1e-12 * ref.abs().max().item(), nb
    finally:
        for s in (d, k):
            s.close()
