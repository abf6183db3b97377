"""FP64 sphere transforms on planes of 64 x 72 points and more, which have an SM to themselves and the most threads,
against extended-precision discrete Fourier transforms; as on small grids (test_gpu_fixed_fft.py) the bound is
2e-15 of the 2-norm (6 roundings of the z pass at FP64, everything else below)."""
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LD, CL = np.longdouble, np.clongdouble


def _dft(c, sg):
    for ax, n in enumerate(c.shape):
        k = np.arange(n)
        a = (np.outer(k, k) % n).astype(LD) * (LD("6.28318530717958647692528676655900576") / LD(n))
        m = np.cos(a) + CL(1j) * sg * np.sin(a)
        c = np.moveaxis(np.tensordot(m, c, axes=(1, ax)), 0, ax)
    return c


@pytest.mark.parametrize("grid", [(72, 64, 16), (64, 75, 16), (80, 72, 16)])
def test_large_planes(grid):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    spec = replace(bi.micro(), grid=grid)
    s = p.BSESystem(spec, gs_tol=1e-6)
    n1, n2, n3 = grid
    half = bi.half_sphere_miller(spec.lattice, spec.ecut)
    om = LD(abs(np.linalg.det(spec.lattice)))
    at = (half[:, 2] % n3, half[:, 1] % n2, half[:, 0] % n1)
    am = (-half[:, 2] % n3, -half[:, 1] % n2, -half[:, 0] % n1)
    rng = np.random.default_rng(sum(grid))
    try:
        X = rng.standard_normal((1, s.n_pw))
        G = s.sphere_to_grid(torch.tensor(X, device="cuda")).cpu().numpy()[0]
        c = np.zeros((n3, n2, n1), CL)
        z = (X[0, 1::2].astype(LD) + CL(1j) * X[0, 2::2]) / np.sqrt(LD(2))
        c[0, 0, 0], c[at], c[am] = X[0, 0], z, np.conj(z)
        E = _dft(c, 1) / np.sqrt(om)
        assert np.linalg.norm(np.abs(G.astype(CL) - E).astype(float)) < 2e-15 * np.linalg.norm(np.abs(E).astype(float))
        H = rng.standard_normal((1, n3, n2, n1)) + 1j * rng.standard_normal((1, n3, n2, n1))
        Y = s.grid_to_sphere(torch.tensor(H, device="cuda"), 2).cpu().numpy()
        F = _dft(H[0].astype(CL), -1) * np.sqrt(om) / LD(n1 * n2 * n3)
        r2 = 1 / np.sqrt(LD(2))
        R = np.zeros((2, s.n_pw), LD)
        R[0, 0], R[1, 0] = F[0, 0, 0].real, F[0, 0, 0].imag
        R[0, 1::2], R[0, 2::2] = (F[at].real + F[am].real) * r2, (F[at].imag - F[am].imag) * r2
        R[1, 1::2], R[1, 2::2] = (F[at].imag + F[am].imag) * r2, (F[am].real - F[at].real) * r2
        assert np.linalg.norm((Y - R).astype(float)) < 2e-15 * np.linalg.norm(R.astype(float))
    finally:
        s.close()
