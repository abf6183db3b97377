"""bse_gemm on millions of rows, where tiles of 32 or 48 rows are more than 65535: A (M x 2) times B (2 x N) against
torch, to the bound of two FP64 sums, 2 (K + 8) 2^-53 |A| |B|."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(2200000, 97), (3200000, 65)])
def test_tall_product(M, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20728_gb300 as p
    K = 2
    g = torch.Generator(device="cuda").manual_seed(7)
    A = torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(K, N, dtype=torch.float64, device="cuda", generator=g)
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p.bse_gemm("N", "N", 1.0, A, B, 0.0, C)
    C -= A @ B
    assert (C.abs_() <= 2 * (K + 8) * 2.0 ** -53 * (A.abs() @ B.abs())).all()
