"""FP64 products from exact BF16 digit products (bse_gemm) against extended-precision products.

Every row of op(A) and column of op(B) is rounded once to 56 bits below its largest entry, the digit
products left out are below 2^-62 of the largest product, sums are exact, and each K slice is rounded
once.  So with a = max |op(A)_i|, b = max |op(B)_j| the error of one output is at most
2^-56 (a sum_k |B_kj| + b sum_k |A_ik|) + 8 * 2^-62 K a b + 2^-50 |A| |B| (rounding of the slice sums,
alpha and beta; the reference product itself is exact to 2^-60).
"""
import numpy as np
import pytest

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


def _operands(kind, M, N, K, rng):
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    if kind == "decay":          # plane-wave coefficients: a few large entries, a long tail
        w = (1 + 0.05 * np.arange(K)) ** -1.5
        A, B = A * w, B * w[:, None]
    elif kind == "scales":       # rows and columns of very different size, zeros, denormals
        A *= 10.0 ** rng.integers(-300, 200, (M, 1))
        B *= 10.0 ** rng.integers(-4, 100, (1, N))
        A[0] = 0.0
        A[-1] = 5e-324 * np.arange(K)
    return A, B


@pytest.mark.parametrize("kind", ["randn", "decay", "scales"])
@pytest.mark.parametrize("ta,tb,M,N,K", [
    ("N", "N", 1, 1, 1), ("N", "T", 5, 5, 31), ("T", "N", 16, 16, 32), ("N", "T", 17, 33, 33),
    ("T", "T", 65, 20, 127), ("N", "N", 80, 48, 129), ("N", "T", 44, 81, 922), ("T", "N", 7, 130, 257)])
def test_against_extended_precision(pkg, kind, ta, tb, M, N, K):
    rng = np.random.default_rng(M + 10 * N + 100 * K)
    A, B = _operands(kind, M, N, K, rng)
    E = A.astype(np.longdouble) @ B.astype(np.longdouble)
    a = torch.tensor(A.T.copy() if ta == "T" else A, device="cuda")
    b = torch.tensor(B.T.copy() if tb == "T" else B, device="cuda")
    c = torch.ones(M, N, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    pkg.bse_gemm(ta, tb, 1.0, a, b, 0.0, c)
    aA, aB = np.abs(A), np.abs(B)
    am, bm = aA.max(1)[:, None], aB.max(0)[None]
    tol = (2.0 ** -56 * (am * aB.sum(0)[None] + bm * aA.sum(1)[:, None]) + 8 * 2.0 ** -62 * K * am * bm
           + 2.0 ** -50 * (aA @ aB) + 5e-324 * K)
    assert (np.abs((c.cpu().numpy() - E).astype(np.float64)) <= tol).all()


def test_infinities_and_nan(pkg):
    """Rows and columns with non-finite entries follow the plain sum; the others are untouched."""
    rng = np.random.default_rng(1)
    A, B = rng.standard_normal((20, 70)), rng.standard_normal((70, 40))
    A[3, 5], A[7, 0], A[9, 69], B[11, 2], B[6, 39] = np.inf, np.nan, -np.inf, np.inf, np.nan
    with np.errstate(invalid="ignore"):
        E = A @ B
    c = torch.zeros(20, 40, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    pkg.bse_gemm("N", "N", 1.0, torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda"), 0.0, c)
    got = c.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(E))
    assert np.array_equal(got[np.isinf(E)], E[np.isinf(E)])
    ok = np.isfinite(E)
    assert np.abs(got[ok] - E[ok]).max() < 1e-13


def test_long_sum(pkg):
    """Slices of thousands of chunks: entries at the largest digits, exact result."""
    K = 300000
    a = torch.full((2, K), 0.9999, dtype=torch.float64, device="cuda")
    b = torch.full((5, K), -0.9999, dtype=torch.float64, device="cuda")
    a[1] = 1.0
    b[1] = 1.0
    c = torch.zeros(5, 2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    pkg.bse_gemm("N", "T", 1.0, b, a, 0.0, c)
    assert c[1, 1].item() == K
    assert abs(c[0, 0].item() + K * 0.9999 * 0.9999) < 1e-10 * K
