"""lnocc_mp2_energy in FP64: the digit planes lie in the workspace of the plain product (csrc/mp2.cu, mp2_plan)."""
import numpy as np
import pytest

from oracle import mp2 as omp2
from paper_2407_11258_gb300 import lnocc as binding
from paper_2407_11258_gb300 import synth

torch = pytest.importorskip("torch")


def plain_bytes(o, v, q, prec):
    def al(x):
        return (x + 255) // 256 * 256

    ov, kp, t = o * v, (q + 63) // 64 * 64, (v + 31) // 32
    ni = max(1, min(o, 2 ** 29 // (ov * v * 8)))
    return 256 + al(ov * kp * (4 if prec else 8)) + al(ni * ov * v * 8) + al(t * (t + 1) // 2 * o * ni * 8 + 8)


@pytest.mark.parametrize("o,v,q", [(1, 50, 200), (4, 24, 96), (8, 60, 240), (12, 200, 800), (16, 240, 960), (30, 200, 640)])
@pytest.mark.parametrize("prec", [0, 1])
def test_size_is_that_of_the_plain_product(o, v, q, prec):
    binding.load()
    assert binding.lnocc_mp2_workspace_bytes(prec, o, v, q) == plain_bytes(o, v, q, prec)


@pytest.mark.parametrize("o,v,q", [(10, 3000, 9000), (60, 500, 9000)])
def test_only_large_systems_ask_for_more(o, v, q):
    """Their X chunk has no room: one occupied row, or planes far wider than it."""
    binding.load()
    assert 0 < binding.lnocc_mp2_workspace_bytes(0, o, v, q) - plain_bytes(o, v, q, 0) <= 2 ** 28


@pytest.fixture(scope="module")
def lnocc():
    from paper_2407_11258_gb300 import build
    build.build()
    binding.load()
    return binding


# planes whole (one and several X chunks), in two, three and four K panels (the last of another width), none
@pytest.mark.gpu
@pytest.mark.parametrize("o,v,q", [(25, 40, 100), (16, 70, 280), (9, 61, 250), (8, 60, 240), (6, 80, 330), (5, 90, 500), (3, 40, 160),
                                   (1, 50, 200), (14, 33, 600)])
def test_energy_and_memory_behind_the_workspace(lnocc, o, v, q):
    fr = synth.make_fragment(o, v, q, 7200 + o, decay=20.0, frag=tuple(range(o)))
    Bov = np.ascontiguousarray(fr.B[:, :o, o:])
    eps, Bd = torch.tensor(fr.eps, device="cuda"), torch.tensor(Bov, device="cuda")
    nb = lnocc.lnocc_mp2_workspace_bytes(0, o, v, q)
    ws = torch.full((nb + 4096,), 171, dtype=torch.uint8, device="cuda")
    got = lnocc.lnocc_mp2_energy(0, o, v, q, eps, Bd, workspace=ws[:nb])
    assert abs(got - omp2.full_mp2_energy(fr.eps, Bov, o)) <= 1e-11
    assert bool((ws[nb:] == 171).all())
    assert lnocc.lnocc_mp2_energy(0, o, v, q, eps, Bd) == got


@pytest.mark.gpu
def test_large_system_with_no_more_than_the_plain_product_needs(lnocc):
    """naux far above nocc nvir: no panel of planes fits the X chunk, so more is asked for, and done without."""
    o, v, q = 4, 600, 9000
    g = torch.Generator(device="cuda").manual_seed(4)
    Bd = 0.02 * torch.randn(q, o, v, generator=g, device="cuda", dtype=torch.float64)
    eps = torch.cat([torch.linspace(-1.2, -0.5, o), torch.linspace(0.3, 4.0, v)]).double().cuda()
    nb, plain = lnocc.lnocc_mp2_workspace_bytes(0, o, v, q), plain_bytes(o, v, q, 0)
    assert nb > plain
    full = lnocc.lnocc_mp2_energy(0, o, v, q, eps, Bd, workspace=torch.empty(nb, dtype=torch.uint8, device="cuda"))
    assert full == lnocc.lnocc_mp2_energy(0, o, v, q, eps, Bd)
    ws = torch.full((plain + 4096,), 171, dtype=torch.uint8, device="cuda")
    got = lnocc.lnocc_mp2_energy(0, o, v, q, eps, Bd, workspace=ws[:plain])
    assert bool((ws[plain:] == 171).all())
    assert abs(got - full) <= 1e-12 * abs(full)  # FP64 products of other order
    with pytest.raises(lnocc.LnoccError) as ei:
        lnocc.lnocc_mp2_energy(0, o, v, q, eps, Bd, workspace=ws[:plain - 256])
    assert ei.value.code == lnocc.LNOCC_EINVAL
