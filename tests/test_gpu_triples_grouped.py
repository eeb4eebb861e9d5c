"""Grouped (T) contraction launches at any nocc from 4 to 32 against the per-term launches and the oracle."""
import numpy as np
import pytest

from oracle import ccsd as occ
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


def energies(lnocc, fr, t1, t2, **opts):
    dev = [torch.tensor(x, device="cuda") for x in (fr.eps, fr.B, t1, t2)]
    f = lnocc.lnocc_build_ints(fr.nocc, fr.nvir, fr.naux, dev[0], dev[1],
                               lnocc.default_opts(precision=1, max_iter=0, **opts))
    try:
        lnocc.lnocc_ccsd(f, dev[2], dev[3], lnocc.LNOCC_GUESS_GIVEN, allow_noconv=True)
        return lnocc.lnocc_triples(f, torch.tensor(fr.U_frag, device="cuda"))
    finally:
        f.free()


# rows of W padded or not (nocc mod 4), one and several column tiles per plane, tiles whose 128 rows hold a
# whole number of a values or leave some over, nvir that leaves partial row tiles and partial blocks of c, and
# several W chunks per slab (triples_chunk_mb = 1)
@pytest.mark.parametrize("nocc,nvir", [(3, 20), (4, 33), (5, 30), (8, 45), (13, 24), (15, 17), (17, 21), (23, 13), (24, 12),
                                       (31, 9)])
def test_grouped_matches_per_term_and_oracle(lnocc, nocc, nvir):
    fr = synth.make_fragment(nocc, nvir, 3 * nvir, 8800 + nocc, decay=20.0, frag=(0,))
    t2 = occ.mp2_amplitudes(fr.eps, fr.B, nocc)
    t1 = 0.01 * synth.Stream(8900 + nocc, 1).normal(nocc * nvir).reshape(nocc, nvir)
    per_term = energies(lnocc, fr, t1, t2, triples_kernel=lnocc.LNOCC_TK_PER_TERM)
    # the same BF16x3 products summed in another order of FP32 additions into W: 2^-23 of the terms
    for opts in ({}, {"triples_kernel": lnocc.LNOCC_TK_GROUPED, "triples_chunk_mb": 1}):
        got = energies(lnocc, fr, t1, t2, **opts)
        assert np.allclose(got, per_term, rtol=1e-5, atol=0.0), (opts, got, per_term)
    if nocc * nvir <= 400:
        E = otr.pair_matrix(t1, t2, fr.eps, fr.B, nocc)
        assert abs(per_term[0] - np.trace(E)) <= 2e-4 * np.abs(np.diag(E)).sum()
        assert abs(got[0] - np.trace(E)) <= 2e-4 * np.abs(np.diag(E)).sum()
