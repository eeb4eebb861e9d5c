"""The FP32 block-energy kernels of (T) at the limits of their ranges, against the oracle."""
import numpy as np
import pytest

from oracle import ccsd as occ
from oracle import fragment as ofr
from oracle import triples as otr
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


# one thread round per pair up to nocc 22, two up to 28; w and v staged together up to 28, one at a time up to
# 37, nothing beyond; nvir small: every kind of block (a < b < c, a = b, b = c, a = b = c) carries weight
@pytest.mark.parametrize("nocc,nvir", [(1, 4), (2, 5), (5, 9), (22, 4), (23, 4), (28, 4), (29, 4), (37, 3), (38, 3)])
def test_block_energies_against_the_oracle(lnocc, nocc, nvir):
    fr = synth.make_fragment(nocc, nvir, 3 * nvir + 5, 7300 + nocc, decay=20.0)
    t2 = occ.mp2_amplitudes(fr.eps, fr.B, nocc)
    t1 = 0.02 * synth.Stream(7400 + nocc, 1).normal(nocc * nvir).reshape(nocc, nvir)
    E = otr.pair_matrix(t1, t2, fr.eps, fr.B, nocc)
    dev = {k: torch.tensor(x, device="cuda") for k, x in (("eps", fr.eps), ("B", fr.B), ("t1", t1), ("t2", t2))}
    f = lnocc.lnocc_build_ints(nocc, nvir, fr.naux, dev["eps"], dev["B"], lnocc.default_opts(precision=1, max_iter=0))
    try:
        lnocc.lnocc_ccsd(f, dev["t1"], dev["t2"], lnocc.LNOCC_GUESS_GIVEN, allow_noconv=True)
        # BF16x3 products keep about 16 bits of W, and the terms of the sum exceed its value a few times
        tol = 2e-4 * np.abs(np.diag(E)).sum()
        for nlo in (0, 1, 2, 3):
            if nlo > nocc:
                continue
            U = np.ascontiguousarray(fr.U[:, :nlo])
            e_t, e_f = lnocc.lnocc_triples(f, torch.tensor(U, device="cuda") if nlo else None)
            if nocc == 1:  # every W is symmetric in its virtual labels: exactly zero (the oracle leaves 1e-37)
                assert e_t == 0.0 and e_f == 0.0
                continue
            assert abs(e_t - np.trace(E)) <= tol
            assert abs(e_f - (ofr.project(E, U) if nlo else 0.0)) <= tol
    finally:
        f.free()
