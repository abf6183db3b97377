"""FP64 sphere transforms on 64-bit fixed point against extended-precision discrete Fourier transforms.

Grids take every radix (2, 3, 4, 5, 8, 9) and odd and even numbers of stages per axis; data range from flat
to strongly decaying coefficients, from smooth to spiked grids, and over sizes near the ends of the FP64
range.  The FP64 pass these replaced has a relative error of about 5e-16 (2-norm) on such data; the bound
is 2e-15 of the 2-norm (6 roundings of the z pass at FP64, everything else below).
"""
from dataclasses import replace

import numpy as np
import pytest

import bse_inputs as bi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LD, CL = np.longdouble, np.clongdouble


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    return p


def _dft(c, sg):
    for ax, n in enumerate(c.shape):
        k = np.arange(n)
        a = (np.outer(k, k) % n).astype(LD) * (LD("6.28318530717958647692528676655900576") / LD(n))
        m = np.cos(a) + CL(1j) * sg * np.sin(a)
        c = np.moveaxis(np.tensordot(m, c, axes=(1, ax)), 0, ax)
    return c


@pytest.mark.parametrize("grid", [(16, 18, 20), (20, 16, 25), (27, 24, 16), (30, 45, 32), (25, 20, 18)])
def test_transforms(pkg, grid):
    spec = replace(bi.micro(), grid=grid)
    s = pkg.BSESystem(spec, gs_tol=1e-6)
    n1, n2, n3 = grid
    half = bi.half_sphere_miller(spec.lattice, spec.ecut)
    g2 = np.repeat(((half @ bi.reciprocal_rows(spec.lattice)) ** 2).sum(1), 2)
    om = LD(abs(np.linalg.det(spec.lattice)))
    at = (half[:, 2] % n3, half[:, 1] % n2, half[:, 0] % n1)
    am = (-half[:, 2] % n3, -half[:, 1] % n2, -half[:, 0] % n1)
    rng = np.random.default_rng(sum(grid))
    try:
        for size in (1.0, 1e-290, 1e290):
            for decay in (0.0, 3.0):
                X = rng.standard_normal((3, s.n_pw)) * size
                X[:, 1:] /= (1 + g2) ** decay
                G = s.sphere_to_grid(torch.tensor(X, device="cuda")).cpu().numpy()
                for q in range(2):
                    c = np.zeros((n3, n2, n1), CL)
                    for f, ph in ((2 * q, CL(1)), (2 * q + 1, CL(1j))):
                        if f < 3:
                            x = X[f].astype(LD)
                            z = (x[1::2] + CL(1j) * x[2::2]) / np.sqrt(LD(2))
                            c[0, 0, 0] += ph * x[0]
                            c[at] += ph * z
                            c[am] += ph * np.conj(z)
                    E = _dft(c, 1) / np.sqrt(om)
                    d = np.abs(G[q].astype(CL) - E) / LD(size)
                    assert np.linalg.norm(d.astype(float)) < 2e-15 * np.linalg.norm(np.abs(E / LD(size)).astype(float))
            for spike in (0.0, 300.0):
                H = rng.standard_normal((1, n3, n2, n1)) + 1j * rng.standard_normal((1, n3, n2, n1))
                H[0, 1, 2, 3] += spike
                H *= size
                Y = s.grid_to_sphere(torch.tensor(H, device="cuda"), 2).cpu().numpy()
                F = _dft(H[0].astype(CL), -1) * np.sqrt(om) / LD(n1 * n2 * n3)
                r2 = 1 / np.sqrt(LD(2))
                R = np.zeros((2, s.n_pw), LD)
                R[0, 0], R[1, 0] = F[0, 0, 0].real, F[0, 0, 0].imag
                R[0, 1::2], R[0, 2::2] = (F[at].real + F[am].real) * r2, (F[at].imag - F[am].imag) * r2
                R[1, 1::2], R[1, 2::2] = (F[at].imag + F[am].imag) * r2, (F[am].real - F[at].real) * r2
                d = (Y.astype(LD) - R) / LD(size)
                assert np.linalg.norm(d.astype(float)) < 2e-15 * np.linalg.norm((R / LD(size)).astype(float))
    finally:
        s.close()


def test_zeros_and_non_finite_planes(pkg):
    """All-zero input gives zeros; a NaN or infinity spoils its own packed grid and no other."""
    spec = bi.micro()
    s = pkg.BSESystem(spec, gs_tol=1e-6)
    try:
        X = torch.zeros(4, s.n_pw, dtype=torch.float64, device="cuda")
        X[2, 5], X[3, 7] = float("nan"), 1.0
        torch.cuda.synchronize()
        P = s.sphere_to_grid(X)
        assert (P[0] == 0).all() and torch.isnan(P[1].real).all()
        H = torch.ones(2, 16, 16, 16, dtype=torch.complex128, device="cuda")
        H[1, 3, 2, 1] = float("inf")
        torch.cuda.synchronize()
        Y = s.grid_to_sphere(H, 4)
        assert torch.isfinite(Y[:2]).all() and torch.isnan(Y[2]).all()
    finally:
        s.close()
