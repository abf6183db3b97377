"""bse_gemm on rows and columns whose entries span many decades: every output within the bound of an FP64 sum,
(K + 8) 2^-53 sum_k |A_ik| |B_kj| (K roundings of products and sums, alpha and beta), against extended precision.

Data: A diag(s) and diag(1/s) B with s between 10^-r and 10^r, disjoint supports (the bound is 0), rotations close
to the identity, a huge entry per row that meets a zero.  Shapes with one K slice and with many, every
orientation, sizes that 16-row strips do not divide, few rows on both sides of the streaming kernel's rule, and
long rows whose largest entry and sum are found in slices (1025 and more across the memory, 16384 along it)."""
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
    if kind.startswith("graded"):
        s = 10.0 ** rng.uniform(-float(kind[6:]), float(kind[6:]), K)
        A, B = A * s, B / s[:, None]
    elif kind == "disjoint":
        A[:, K // 2:] = 0.0
        B[:K // 2] = 0.0
    elif kind == "rotation":
        A *= 1e-6
        A[np.arange(M), np.arange(M) % K] += 1.0
        B *= 10.0 ** rng.uniform(-12, 0, (K, 1))
    elif kind == "spike":
        A[:, 0] = 1e20
        B[0] = 0.0
    return A, B


@pytest.mark.parametrize("kind", ["randn", "graded1", "graded2", "graded4", "graded6", "graded18", "disjoint", "rotation",
                                  "spike"])
@pytest.mark.parametrize("ta,tb,M,N,K", [
    ("N", "T", 1, 1, 2), ("N", "T", 5, 5, 31), ("N", "N", 40, 301, 48), ("T", "N", 33, 130, 257), ("T", "T", 65, 20, 500),
    ("N", "N", 4, 4100, 68), ("N", "N", 4, 4100, 69), ("T", "N", 2, 4111, 276), ("N", "N", 9, 5000, 5),
    ("N", "N", 60, 1500, 130), ("N", "T", 17, 33, 900), ("N", "T", 80, 70, 3001),
    ("N", "N", 8, 33, 6859), ("T", "N", 5, 40, 5000), ("T", "T", 33, 7, 1025), ("N", "T", 5, 6, 20000)])
def test_entrywise_bound(pkg, kind, ta, tb, M, N, K):
    rng = np.random.default_rng(M + 10 * N + 100 * K)
    A, B = _operands(kind, M, N, K, rng)
    E = A.astype(np.longdouble) @ B.astype(np.longdouble)
    tol = (K + 8) * 2.0 ** -53 * (np.abs(A) @ np.abs(B))
    a = torch.tensor(A.T.copy() if ta == "T" else A, device="cuda")
    b = torch.tensor(B.T.copy() if tb == "T" else B, device="cuda")
    c = torch.ones(M, N, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    pkg.bse_gemm(ta, tb, 1.0, a, b, 0.0, c)
    assert (np.abs((c.cpu().numpy() - E).astype(np.float64)) <= tol).all()


def test_alpha_and_beta(pkg):
    """The outputs that are summed anew take alpha and beta like the others."""
    rng = np.random.default_rng(5)
    for M, N, K in ((40, 301, 48), (17, 33, 900)):
        A, B = _operands("graded4", M, N, K, rng)
        C = rng.standard_normal((M, N))
        E = C.astype(np.longdouble) - 3 * (A.astype(np.longdouble) @ B.astype(np.longdouble))
        tol = (K + 8) * 2.0 ** -53 * (3 * np.abs(A) @ np.abs(B) + np.abs(C))
        c = torch.tensor(C, device="cuda")
        torch.cuda.synchronize()
        pkg.bse_gemm("N", "N", -3.0, torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda"), 1.0, c)
        assert (np.abs((c.cpu().numpy() - E).astype(np.float64)) <= tol).all()


def test_non_finite_long_rows(pkg):
    """A NaN or infinity in any slice of a long row or column reaches its outputs and no others."""
    rng = np.random.default_rng(2)
    K = 20000
    A, B = rng.standard_normal((6, K)), rng.standard_normal((K, 40))
    A[1, 3], A[4, K - 1], B[K // 2, 7], B[K - 2, 33] = np.inf, np.nan, -np.inf, np.nan
    with np.errstate(invalid="ignore"):
        E = A @ B
    for ta, tb in (("N", "N"), ("T", "T")):
        c = torch.zeros(6, 40, dtype=torch.float64, device="cuda")
        a, b = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
        a, b = (a.T.contiguous(), b.T.contiguous()) if ta == "T" else (a, b)
        torch.cuda.synchronize()
        pkg.bse_gemm(ta, tb, 1.0, a, b, 0.0, c)
        got = c.cpu().numpy()
        assert np.array_equal(np.isnan(got), np.isnan(E))
        assert np.array_equal(got[np.isinf(E)], E[np.isinf(E)])
        ok = np.isfinite(E)
        assert np.abs(got[ok] - E[ok]).max() < 1e-10
