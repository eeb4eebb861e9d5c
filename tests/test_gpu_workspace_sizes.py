"""Attached (T) workspaces: what is optional (digit planes, padded rows of W) never decides whether one is large enough."""
import numpy as np
import pytest

from paper_2407_11258_gb300 import lnocc as binding
from paper_2407_11258_gb300 import synth

torch = pytest.importorskip("torch")


def plain_bytes(o, v, q, prec, chunk_mb=768):
    """The temporaries without planes and padding, in allocation order, 256-byte aligned."""
    esz = 4 if prec else 8

    def al(x):
        return (max(x, 256) + 255) // 256 * 256

    def packed(rows, k):
        return rows * ((max(k, 1) + 63) // 64 * 64) * esz

    slab = max((b + 1) * (v - b) for b in range(v)) * o ** 3
    w = max(min(chunk_mb * 2 ** 20 // esz, slab), v * o ** 3) * esz
    bc = max(1, min(v, 2 ** 26 // (o * v * v)))
    nblk = sum((b + 1) * (v - b) for b in range(v))
    return (2 * al(packed(v * v * o, v + o)) + 2 * al(packed(v * o * o, v + o)) + al(o ** 3 * v * 8) + al(packed(v * v, q)) +
            al(bc * o * v * v * 8) + al(w) + al((nblk + 256) * 16) + 2 * al(32 * max(1, v * v // 2 + v)) + al(o * 64) +
            (al(v * v * o * o * 4) if prec else 0))


@pytest.mark.parametrize("o,v,q", [(4, 24, 96), (5, 37, 150), (7, 40, 160), (13, 60, 240), (19, 125, 500), (30, 200, 800)])
@pytest.mark.parametrize("mb", [1, 64, 768])
def test_mixed_size_holds_the_padding_in_its_dead_temporaries(o, v, q, mb):
    binding.load()
    assert binding.lnocc_workspace_bytes(o, v, q, binding.default_opts(precision=1, triples_chunk_mb=mb)) == plain_bytes(
        o, v, q, 1, mb)


@pytest.fixture(scope="module")
def lnocc():
    from paper_2407_11258_gb300 import build
    build.build()
    binding.load()
    return binding


def energies(lnocc, fr, prec, nbytes=None, nlo=1, capture=False, **opts):
    dev = [torch.tensor(x, device="cuda") for x in (fr.eps, fr.B, np.ascontiguousarray(fr.U[:, :nlo]))]
    f = lnocc.lnocc_build_ints(fr.nocc, fr.nvir, fr.naux, dev[0], dev[1], lnocc.default_opts(precision=prec, **opts))
    try:
        lnocc.lnocc_ccsd(f, allow_noconv=True)
        if nbytes is None:
            return lnocc.lnocc_triples(f, dev[2])
        # the memory behind the workspace must stay as it is
        ws = torch.full((nbytes + 4096,), 171, dtype=torch.uint8, device="cuda")
        lnocc.lnocc_frag_set_workspace(f, ws[:nbytes])
        before = f.info().device_allocs
        got = lnocc.lnocc_triples(f, dev[2])
        if capture:
            e = torch.zeros(2, dtype=torch.float64, device="cuda")
            st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                lnocc.lnocc_triples_device(f, dev[2], e, st, stream=s)
            g.replay()
            torch.cuda.synchronize()
            assert tuple(e.tolist()) == tuple(got) and int(st.item()) == 0
        assert f.info().device_allocs == before
        assert bool((ws[nbytes:] == 171).all())
        with pytest.raises(lnocc.LnoccError) as ei:
            lnocc.lnocc_frag_set_workspace(f, ws[:plain_bytes(fr.nocc, fr.nvir, fr.naux, prec) - 256])
        assert ei.value.code == lnocc.LNOCC_EINVAL
        return got
    finally:
        f.free()


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(3, 10, 40), (4, 24, 96), (9, 40, 150)])
def test_fp64_without_room_for_the_digit_planes(lnocc, shape):
    """sigma3, 4 and 6 cut their operands per chunk, sigma1, 2 and 5 run on the SIMT kernel."""
    o, v, q = shape
    fr = synth.make_fragment(o, v, q, 5100 + o, decay=20.0, frag=(0,))
    size = plain_bytes(o, v, q, 0)
    assert size < lnocc.lnocc_workspace_bytes(o, v, q, lnocc.default_opts(precision=0))
    ref = energies(lnocc, fr, 0)
    got = energies(lnocc, fr, 0, size, capture=True)
    assert np.allclose(got, ref, rtol=1e-11, atol=0.0)  # FP64 sums of other order, a few 1e3 terms


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(4, 24, 96), (5, 37, 150), (7, 12, 50), (13, 20, 80), (16, 18, 72), (19, 17, 60)])
def test_mixed_with_the_padding_inside(lnocc, shape):
    o, v, q = shape
    fr = synth.make_fragment(o, v, q, 5200 + o, decay=20.0, frag=(0,))
    assert energies(lnocc, fr, 1, plain_bytes(o, v, q, 1), capture=True) == energies(lnocc, fr, 1)  # same kernels, same bits


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(1, 3, 12), (6, 1, 9), (9, 2, 16), (31, 4, 40), (37, 2, 30)])
def test_mixed_sizes_too_small_for_the_padding(lnocc, shape):
    o, v, q = shape
    fr = synth.make_fragment(o, v, q, 5300 + o, decay=20.0, frag=(0,))
    ref = energies(lnocc, fr, 1)
    got = energies(lnocc, fr, 1, plain_bytes(o, v, q, 1))
    # the same BF16x3 products of W, the energies in FP64 instead of FP32 sums: 2^-23 of the terms
    assert np.allclose(got, ref, rtol=1e-5, atol=1e-15)
