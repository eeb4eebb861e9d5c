"""Digit planes of FP64 products are optional: whole solves when their allocations fail (SIMT products)."""
import pytest

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


def solve(lnocc, fr, prec, **opts):
    eps, B, U = (torch.tensor(x, device="cuda") for x in (fr.eps, fr.B, fr.U_frag))
    f = lnocc.lnocc_build_ints(fr.nocc, fr.nvir, fr.naux, eps, B, lnocc.default_opts(precision=prec, **opts))
    try:
        info = f.info()
        e = lnocc.lnocc_ccsd(f)[0]
        return [info.e_mp2, e, *lnocc.lnocc_fragment_energy(f, U), *lnocc.lnocc_triples(f, U)], info.device_bytes
    finally:
        f.free()


@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (1, 1e-9)])
@pytest.mark.parametrize("shape", [(3, 20, 70), (6, 40, 160)])
def test_solve_without_digit_planes(lnocc, shape, prec, tol):
    """FP64: sums of other order; mixed: (ia|jb) and h alone, a rounding that nine iterations carry on."""
    o, v, q = shape
    fr = synth.make_fragment(o, v, q, 6100 + o, decay=20.0, frag=(0, 1))
    ref, full = solve(lnocc, fr, prec)
    got, less = solve(lnocc, fr, prec, fault_inject=lnocc.LNOCC_FAULT_NO_PLANES)
    assert less < full
    assert all(abs(a - b) <= tol for a, b in zip(got, ref)), (got, ref)
