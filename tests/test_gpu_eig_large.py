"""The Jacobi eigensolver where its form changes: blocks per SM above order 400, two launches per round above 1024."""
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


@pytest.mark.parametrize("n", [400, 401, 1023, 1024, 1025, 1026])
def test_eigenpairs(lnocc, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64)
    A = A @ A.T / n + torch.diag(torch.linspace(0, 1, n, device="cuda", dtype=torch.float64))
    A = 0.5 * (A + A.T)
    C, lam, keep = lnocc.lnocc_lno_select(A, None, 0.0)
    ref = torch.linalg.eigvalsh(A).flip(0)
    tol = 1e-14 * n * float(ref[0])  # a few roundings of every element per sweep
    assert keep == n and float((lam - ref).abs().max()) <= tol
    assert float((C.T @ C - torch.eye(n, device="cuda", dtype=torch.float64)).abs().max()) <= 1e-14 * n
    assert float((A @ C - C * lam).abs().max()) <= tol
