"""Inner products of a few rows over a long K (bse_gemm N, T), which stream in FP64 in groups of four rows: row
counts that four does not divide, a single row of B, odd K (rows off 16 bytes), both sides of the rule's limits,
against torch within the bound of two FP64 sums, 2 (K + 8) 2^-53 (|A||B| + |C|)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 32768), (3, 17, 40001), (5, 32, 32768), (5, 33, 32768), (8, 1, 65537),
                                   (13, 1, 32770), (7, 7, 70000), (9, 64, 65536), (9, 65, 65536), (16, 48, 65537),
                                   (1, 9, 100001)])
def test_long_rows(M, N, K):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(N, K, dtype=torch.float64, device="cuda", generator=g)
    C = torch.randn(M, N, dtype=torch.float64, device="cuda", generator=g)
    D = C.clone()
    torch.cuda.synchronize()
    p.bse_gemm("N", "T", -2.0, A, B, 0.5, D)
    E = 0.5 * C - 2.0 * (A @ B.T)
    mag = 2.0 * (A.abs() @ B.abs().T) + 0.5 * C.abs()
    assert ((D - E).abs() <= 2 * (K + 8) * 2.0 ** -53 * mag).all()
