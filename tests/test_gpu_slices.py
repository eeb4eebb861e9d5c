"""FP64 contractions formed from BF16 digit planes on the tensor pipe (csrc/gemm_slices.cu)."""
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


def product(lnocc, A, B, fn="lnocc_debug_gemm"):
    C = torch.full((A.shape[0], B.shape[0]), float("nan"), dtype=torch.float64, device="cuda")
    getattr(lnocc, fn)(0, A.cuda().contiguous(), B.cuda().contiguous(), C)
    return C.cpu()


# tiles are 128 x 64, a chunk of one exponent is 512 columns: one element, full and ragged tiles, one
# column beyond a chunk, split K with one tile
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (128, 64, 512), (130, 70, 64), (129, 65, 513), (64, 64, 1024), (257, 300, 700),
                                   (20, 16, 14400)])
def test_integer_products_are_exact(lnocc, M, N, K):
    """Integers of 20 bits: every product and sum is an integer below 2^53, so the FP64 result is exact."""
    g = torch.Generator().manual_seed(M + N + K)
    A = torch.randint(-2 ** 19, 2 ** 19, (M, K), generator=g).double()
    B = torch.randint(-2 ** 19, 2 ** 19, (N, K), generator=g).double()
    ref = (A.long().numpy() @ B.long().numpy().T).astype(np.float64)
    assert np.array_equal(product(lnocc, A, B).numpy(), ref)


def test_largest_digits_accumulate_exactly(lnocc):
    """All digits 64 with one sign over a whole chunk: the largest partial sums an accumulator can hold."""
    x = sum(64 * 2.0 ** (-7 * i) for i in range(7))
    A = torch.full((128, 512), x, dtype=torch.float64)
    C = product(lnocc, A, A[:64])
    assert torch.equal(C, torch.full_like(C, float(np.longdouble(x) ** 2 * 512)))


@pytest.mark.parametrize("K", [8, 24, 100, 240, 960])
@pytest.mark.parametrize("kind", ["gauss", "decay"])
def test_error_is_not_larger_than_that_of_the_fp64_kernel(lnocc, kind, K):
    """Against an extended-precision sum, on entries like those of B (Gaussian, decaying from the diagonal)."""
    g = torch.Generator().manual_seed(K)
    A, B = (torch.randn(r, K, generator=g, dtype=torch.float64) for r in (70, 60))
    if kind == "decay":
        k = torch.arange(K).double()
        A, B = (X * torch.exp(-(k[None, :] - torch.arange(X.shape[0])[:, None]).abs() / 20.0) for X in (A, B))
    a, b = A.numpy().astype(np.longdouble), B.numpy().astype(np.longdouble)
    ref = np.zeros((70, 60), np.longdouble)
    for k in range(K):
        ref += np.outer(a[:, k], b[:, k])
    err = {fn: float(np.linalg.norm((product(lnocc, A, B, fn).numpy() - ref).astype(np.float64)))
           for fn in ("lnocc_debug_gemm", "lnocc_gemm_noalloc")}  # digit planes; FP64 FMA chain
    assert err["lnocc_debug_gemm"] <= err["lnocc_gemm_noalloc"], err


def test_non_finite_and_extreme_elements(lnocc):
    g = torch.Generator().manual_seed(5)
    A, B = (torch.randn(r, 80, generator=g, dtype=torch.float64) for r in (130, 70))
    A[3, 5], A[129, 1], B[69, 0] = float("inf"), float("nan"), -float("inf")
    A[7, :], B[5, :] = 5e-310, 1e200  # subnormal row; results 4e-108
    A[11, :], B[6, :] = 0.0, 0.0
    C, ref = product(lnocc, A, B), A @ B.T
    assert torch.equal(C.isnan(), ref.isnan()) and torch.equal(C.isinf(), ref.isinf())
    assert torch.equal(C[C.isinf()], ref[ref.isinf()])
    ok = ref.isfinite()
    assert ((C - ref)[ok].abs() <= 1e-14 * (A.abs() @ B.abs().T)[ok]).all()
    assert (C[11][:69] == 0).all() and (C[12:129, 6] == 0).all()
    # results in the subnormal range and beyond the largest double
    tiny = product(lnocc, 1e-200 * A[20:24], 1e-110 * B[20:24])
    assert (tiny - (1e-200 * A[20:24]) @ (1e-110 * B[20:24]).T).abs().max() <= 3e-323
    big = product(lnocc, 1e200 * A[20:24].abs(), 1e200 * B[20:24].abs())
    assert big.isinf().all()
