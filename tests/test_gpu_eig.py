"""The Jacobi eigensolver behind lnocc_lno_select at orders that exercise the tiling of its sweep kernel."""
import numpy as np
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


# one element, one pair, odd orders (a bye in every round), one block, several, more than one pass per thread
@pytest.mark.parametrize("n", [1, 2, 3, 7, 16, 65, 130, 333])
def test_eigenpairs(lnocc, n):
    g = np.random.default_rng(n)
    A = g.standard_normal((n, n))
    A = A @ A.T / n + np.diag(np.linspace(0.0, 1.0, n))
    C, lam, keep = lnocc.lnocc_lno_select(torch.tensor(A, device="cuda"), None, 0.0)
    C, lam = C.cpu().numpy(), lam.cpu().numpy()
    ref = np.linalg.eigvalsh(A)[::-1]
    tol = 1e-14 * n * ref[0]  # a few roundings of every element per sweep
    assert keep == n and np.abs(lam - ref).max() <= tol
    assert np.abs(C.T @ C - np.eye(n)).max() <= 1e-14 * n + 1e-14
    assert np.abs(A @ C - C * lam).max() <= tol
