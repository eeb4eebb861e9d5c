"""The doubles update on the GPU: one evaluation serves (i,j,a,b) and (j,i,b,a)."""
import numpy as np
import pytest

from oracle import ccsd as occ
from paper_2407_11258_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lnocc():
    from paper_2407_11258_gb300 import build
    from paper_2407_11258_gb300 import lnocc as m
    build.build()
    m.load()
    return m


def solve(lnocc, fr, t_in=None, allow_noconv=True, **opts):
    f = lnocc.lnocc_build_ints(fr.nocc, fr.nvir, fr.naux, torch.tensor(fr.eps, device="cuda"),
                               torch.tensor(fr.B, device="cuda"), lnocc.default_opts(**opts))
    t1 = torch.empty(fr.nocc, fr.nvir, dtype=torch.float64, device="cuda")
    t2 = torch.empty(fr.nocc, fr.nocc, fr.nvir, fr.nvir, dtype=torch.float64, device="cuda")
    try:
        if t_in is None:
            e, _, _ = lnocc.lnocc_ccsd(f, t1_out=t1, t2_out=t2, allow_noconv=allow_noconv)
        else:
            e, _, _ = lnocc.lnocc_ccsd(f, *t_in, lnocc.LNOCC_GUESS_GIVEN, t1, t2, allow_noconv=allow_noconv)
    finally:
        f.free()
    return e, t1, t2


# edges of the 32 x 32 tiles, a single occupied orbital (diagonal pairs only), a single virtual one
@pytest.mark.parametrize("shape", [(1, 1, 3), (1, 33, 40), (2, 32, 40), (3, 31, 50), (4, 1, 9), (5, 65, 70)])
def test_two_iterations_match_the_oracle_and_are_symmetric(lnocc, shape):
    o, v, q = shape
    fr = synth.make_fragment(o, v, q, 4400 + o, decay=20.0)
    ref = occ.ccsd(fr.eps, fr.B, o, max_iter=2)
    for prec in (0, 1):
        _, t1, t2 = solve(lnocc, fr, precision=prec, max_iter=2)
        assert torch.equal(t2, t2.permute(1, 0, 3, 2))
        # FP64: rounding of sums of at most q v terms; mixed: BF16x3 products, 2^-16 each
        tol = (1e-12 if prec == 0 else 1e-4) * max(np.abs(ref["t2"]).max(), np.abs(ref["t1"]).max())
        assert np.abs(t2.cpu().numpy() - ref["t2"]).max() <= tol
        assert np.abs(t1.cpu().numpy() - ref["t1"]).max() <= tol


@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 1e-6)])
def test_a_guess_without_the_symmetry_converges_to_the_same_energy(lnocc, prec, tol):
    fr = synth.make_fragment(4, 24, 96, 4500, decay=20.0)
    e0, t1, t2 = solve(lnocc, fr, precision=0, allow_noconv=False)
    g = torch.Generator(device="cpu").manual_seed(1)
    noisy = t2 + 1e-3 * torch.randn(t2.shape, generator=g, dtype=torch.float64).cuda()
    e1, _, s2 = solve(lnocc, fr, (t1, noisy), allow_noconv=False, precision=prec)
    assert abs(e1 - e0) <= tol
    assert torch.equal(s2, s2.permute(1, 0, 3, 2))
