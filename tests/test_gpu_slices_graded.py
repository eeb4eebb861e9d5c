"""FP64 products of graded operands: no element may be less exact than by an FP64 FMA chain (csrc/gemm_slices.cu)."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def lnocc():
    from paper_2407_11258_gb300 import build
    from paper_2407_11258_gb300 import lnocc as m
    build.build()
    m.load()
    return m


def product(lnocc, A, B, fn="lnocc_debug_gemm"):
    A, B = (torch.as_tensor(np.ascontiguousarray(X)) for X in (A, B))
    C = torch.full((A.shape[0], B.shape[0]), float("nan"), dtype=torch.float64, device="cuda")
    getattr(lnocc, fn)(0, A.cuda(), B.cuda(), C)
    return C.cpu().numpy()


def reference(A, B):
    """(C, sum |a||b|) in extended precision."""
    a, b = A.astype(np.longdouble), B.astype(np.longdouble)
    C, T = np.zeros((len(A), len(B)), np.longdouble), np.zeros((len(A), len(B)), np.longdouble)
    for k in range(A.shape[1]):
        t = np.outer(a[:, k], b[:, k])
        C += t
        T += np.abs(t)
    return C, T


def operands(kind, M, N, K, seed):
    g = np.random.default_rng(seed)
    A, B = g.standard_normal((M, K)), g.standard_normal((N, K))
    if kind == "graded":  # every element its own order of magnitude
        A *= 10.0 ** -g.uniform(0, 30, (M, K))
        B *= 10.0 ** -g.uniform(0, 30, (N, K))
    elif kind == "local":  # rows decay from a centre of their own: far pairs have only small terms
        k = np.arange(K)
        A *= np.exp(-np.abs(k[None, :] - g.uniform(0, K, M)[:, None]) / 3.0)
        B *= np.exp(-np.abs(k[None, :] - g.uniform(0, K, N)[:, None]) / 3.0)
    elif kind == "opposed":  # the large columns of one operand are the small ones of the other
        w = 10.0 ** -np.linspace(0, 40, K)
        A *= w
        B *= w[::-1]
    elif kind == "sparse":  # mostly zeros: many elements have no term at all
        A *= g.random((M, K)) < 0.05
        B *= g.random((N, K)) < 0.05
    return A, B


# a single element, tiles of 128 x 48 with every remainder kind, one chunk of 512 columns and two and a half, split K
SHAPES = [(1, 1, 1), (17, 9, 3), (70, 60, 24), (129, 49, 100), (128, 48, 512), (131, 100, 513), (40, 100, 1300)]


@pytest.mark.parametrize("kind", ["gauss", "graded", "local", "opposed", "sparse"])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_every_element_is_within_the_bound_of_an_fma_chain(lnocc, kind, M, N, K):
    A, B = operands(kind, M, N, K, M + N + K)
    C, T = reference(A, B)
    err = np.abs(product(lnocc, A, B) - C)
    # K roundings of partial sums below T; one rounding of the exact product at K = 1 (near a tie by the dropped digits)
    assert (err <= max(K, 1.01) * U * T).all(), float((err / np.where(T > 0, T, 1)).max() / U)
    assert (product(lnocc, A, B)[np.asarray(T == 0)] == 0).all()


@pytest.mark.parametrize("kind", ["graded", "local", "opposed"])
@pytest.mark.parametrize("K", [100, 512])
def test_errors_relative_to_the_terms_are_not_larger_than_those_of_the_fp64_kernel(lnocc, kind, K):
    A, B = operands(kind, 140, 100, K, 7 + K)
    C, T = reference(A, B)
    rms = {fn: float(np.sqrt(np.mean((((product(lnocc, A, B, fn) - C) / T) ** 2).astype(np.float64))))
           for fn in ("lnocc_debug_gemm", "lnocc_gemm_noalloc")}  # digit planes with FP64 sums; FP64 FMA chain
    assert rms["lnocc_debug_gemm"] <= rms["lnocc_gemm_noalloc"], rms


def test_small_elements_beside_large_ones_keep_their_own_53_bits(lnocc):
    x = 1.0 + 2.0 ** -52
    for e in (10, 40, 57, 80, 300, 600):
        A = np.array([[1.0, x * 2.0 ** -e], [x * 2.0 ** -e, 3.0]])
        B = np.array([[0.0, x], [x, 0.0]])
        want = [[float(Fraction(A[i, 0]) * Fraction(B[j, 0]) + Fraction(A[i, 1]) * Fraction(B[j, 1])) for j in range(2)]
                for i in range(2)]
        assert np.array_equal(product(lnocc, A, B), np.array(want)), e


def test_marked_rows_and_fp64_sums_in_one_unit(lnocc):
    """Infinities and NaN beside elements that fall back for their size, and ordinary ones."""
    A, B = operands("local", 130, 50, 96, 3)
    A[5, 7], A[129, 0], B[49, 95] = np.inf, np.nan, -np.inf
    A[8, :] = 5e-310
    got, ref = product(lnocc, A, B), (torch.as_tensor(A) @ torch.as_tensor(B).T).numpy()
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    ok = np.isfinite(ref)
    T = np.abs(np.where(np.isfinite(A), A, 0)) @ np.abs(np.where(np.isfinite(B), B, 0)).T
    assert (np.abs(got - ref)[ok] <= 2 * 96 * U * T[ok] + 1e-323 * 96).all()


def test_digits_of_63_accumulate_exactly(lnocc):
    """x has seven digits of 63 (exponent 6). Half of a chunk adds x x, half takes it away but for one unit of the last
    digit: every accumulator up to the seventh climbs to g 256 63^2 units (2^22.8 at g = 7) and returns, so a
    lost bit on the way would stay in the result. That is what the pairs i + j <= 10 of the unit (j = 7) give: the first three
    digits of x, times 2^-42; the rest of x 2^-42 is dropped, 2^-63 of the largest terms. (1300 x 800: enough tiles that K is not split over work
    items, whose FP64 partials would round.)"""
    x = sum(63 * 2.0 ** (-7 * i) for i in range(7))
    r, digits = Fraction(x) / 64, []  # the recurrence of the cut: balanced radix-128 digits
    for i in range(9):
        d = int(np.floor(r * 2 ** (6 + 7 * i) + Fraction(1, 2)))
        digits.append(d)
        r -= Fraction(d, 2 ** (6 + 7 * i))
    assert digits == [63] * 7 + [0, 0] and r == 0
    A = np.full((1300, 512), x)
    B = np.full((800, 512), x)
    B[:, 256:] = -x
    B[:, 300] += 2.0 ** -42
    assert np.array_equal(product(lnocc, A, B), np.full((1300, 800), 63 * (1 + 2.0 ** -7 + 2.0 ** -14) * 2.0 ** -42))
