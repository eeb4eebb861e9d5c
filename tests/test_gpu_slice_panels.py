"""FP64 products whose digit planes exceed the slice workspace: panels of rows and of K (csrc/slice_panels.h)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lnocc():
    from paper_2407_11258_gb300 import build
    from paper_2407_11258_gb300 import lnocc as m
    build.build()
    m.load()
    return m


# a small A panel beside a B kept whole, K panels, row panels of B, of A, and of both
@pytest.mark.parametrize("M,N,K", [(100, 260, 47040), (130, 290, 42000), (520, 300, 30000), (600, 3000, 8200), (3000, 600, 8200),
                                   (1100, 2900, 16500)])
def test_panel_products_are_exact(lnocc, M, N, K):
    """Integers of 16 bits: every sum is an integer below 2^53, so the FP64 result is exact in any order."""
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A, B = (torch.randint(-2 ** 15, 2 ** 15, (r, K), generator=g, device="cuda").double() for r in (M, N))
    C = torch.full((M, N), float("nan"), dtype=torch.float64, device="cuda")
    lnocc.lnocc_debug_gemm(0, A, B, C)
    assert torch.equal(C, A @ B.T)
