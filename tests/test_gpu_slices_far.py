"""FP64 products with twelve digits (csrc/gemm_slices.cu): exactness, graded operands, and the terms that take them."""
import importlib.util
import os

import numpy as np
import pytest

from oracle import ccsd as occ
from oracle import triples as otr
from paper_2407_11258_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53

spec = importlib.util.spec_from_file_location("graded", os.path.join(os.path.dirname(__file__), "test_gpu_slices_graded.py"))
graded = importlib.util.module_from_spec(spec)
spec.loader.exec_module(graded)


@pytest.fixture(scope="module")
def lnocc():
    from paper_2407_11258_gb300 import build
    from paper_2407_11258_gb300 import lnocc as m
    build.build()
    m.load()
    return m


def product(lnocc, A, B, precision=2):
    A, B = (torch.as_tensor(np.ascontiguousarray(X)).cuda() for X in (A, B))
    C = torch.full((A.shape[0], B.shape[0]), float("nan"), dtype=torch.float64, device="cuda")
    lnocc.lnocc_debug_gemm(precision, A, B, C)
    return C.cpu().numpy()


# tiles of 128 x 32, K blocks of 16, chunks of 512 columns, split K, panels beyond the workspace
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (128, 32, 512), (130, 70, 64), (129, 33, 513), (257, 300, 700), (20, 16, 14400),
                                   (1300, 800, 1040)])
def test_integer_products_are_exact(lnocc, M, N, K):
    g = np.random.default_rng(M + N + K)
    A, B = (g.integers(-2 ** 19, 2 ** 19, (r, K)).astype(np.float64) for r in (M, N))
    ref = (A.astype(np.int64) @ B.astype(np.int64).T).astype(np.float64)
    assert np.array_equal(product(lnocc, A, B), ref)


@pytest.mark.parametrize("M,N,K", [(100, 260, 40000), (520, 300, 30000), (600, 2900, 8200)])
def test_panel_products_are_exact(lnocc, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A, B = (torch.randint(-2 ** 15, 2 ** 15, (r, K), generator=g, device="cuda").double() for r in (M, N))
    C = torch.full((M, N), float("nan"), dtype=torch.float64, device="cuda")
    lnocc.lnocc_debug_gemm(2, A, B, C)
    assert torch.equal(C, A @ B.T)


@pytest.mark.parametrize("kind", ["gauss", "graded", "local", "opposed", "sparse"])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (17, 9, 3), (129, 49, 100), (128, 48, 512), (40, 100, 1300)])
def test_every_element_is_within_the_bound_of_an_fma_chain(lnocc, kind, M, N, K):
    A, B = graded.operands(kind, M, N, K, M + N + K)
    C, T = graded.reference(A, B)
    got = product(lnocc, A, B)
    err = np.abs(got - C)
    assert (err <= max(K, 1.01) * U * T).all(), float((err / np.where(T > 0, T, 1)).max() / U)
    assert (got[np.asarray(T == 0)] == 0).all()


def test_terms_between_the_two_lines_come_from_the_digits_and_are_rounded_once(lnocc):
    """Sums 2^-17 of the product of their rows' largest elements (2^10 each, which meet zeros): nine digits fall back to
    FP64 sums, twelve do not, and each element is the nearest double but for the dropped digits (2^-64 of T)."""
    g = np.random.default_rng(11)
    A, B = g.standard_normal((64, 40)), g.standard_normal((48, 40))
    A[:, 0], B[:, 0], A[:, 1], B[:, 1] = 2.0 ** 10, 0.0, 0.0, 2.0 ** 10
    C, T = graded.reference(A, B)
    assert (np.abs(product(lnocc, A, B) - C) <= (0.501 * np.abs(C) * 2 * U + 2.0 ** -60 * T)).all()


# both sides of the line in nvir, K = nvir not a multiple of 64; decay 3: virtuals far apart have only tiny terms.
# One iteration: the extrapolation of two nearly parallel ones would amplify any rounding a hundredfold.
@pytest.mark.parametrize("o,v,q", [(2, 100, 50), (2, 129, 50), (3, 150, 40)])
@pytest.mark.parametrize("decay", [20.0, 3.0])
def test_fp64_iteration_and_triples_match_the_oracle(lnocc, o, v, q, decay):
    fr = synth.make_fragment(o, v, q, 8100 + v, decay=decay, frag=(0,))
    ref = occ.ccsd(fr.eps, fr.B, o, max_iter=1)
    eps, B = torch.tensor(fr.eps, device="cuda"), torch.tensor(fr.B, device="cuda")
    t1 = torch.empty(o, v, dtype=torch.float64, device="cuda")
    t2 = torch.empty(o, o, v, v, dtype=torch.float64, device="cuda")
    f = lnocc.lnocc_build_ints(o, v, q, eps, B, lnocc.default_opts(precision=0, max_iter=1))
    try:
        lnocc.lnocc_ccsd(f, t1_out=t1, t2_out=t2, allow_noconv=True)
        e_t, _ = lnocc.lnocc_triples(f, None)
    finally:
        f.free()
    tol = 1e-12 * max(np.abs(ref["t2"]).max(), np.abs(ref["t1"]).max())  # rounding of sums of at most q v terms
    assert np.abs(t2.cpu().numpy() - ref["t2"]).max() <= tol
    assert np.abs(t1.cpu().numpy() - ref["t1"]).max() <= tol
    want = otr.pair_matrix(t1.cpu().numpy(), t2.cpu().numpy(), fr.eps, fr.B, o)
    assert abs(e_t - np.trace(want)) <= 1e-11 * np.abs(np.diag(want)).sum()
