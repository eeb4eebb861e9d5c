"""lnocc_triples_device under capture on every launch form: per-term launches with device-built tables, and grouped ones."""
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


# per-term launches: below nocc 4, and by option with rows of W padded (5) and not (8); grouped at an odd nocc
@pytest.mark.parametrize("shape,kernel", [((3, 21, 80), "LNOCC_TK_AUTO"), ((5, 37, 150), "LNOCC_TK_PER_TERM"),
                                          ((8, 30, 120), "LNOCC_TK_PER_TERM"), ((5, 37, 150), "LNOCC_TK_GROUPED"),
                                          ((19, 18, 70), "LNOCC_TK_AUTO")])
def test_captured_triples_give_the_synchronous_energies(lnocc, shape, kernel):
    o, v, q = shape
    fr = synth.make_fragment(o, v, q, 1900 + o, decay=20.0, frag=(0, 1))
    eps, B, U = (torch.tensor(x, device="cuda") for x in (fr.eps, fr.B, fr.U_frag))
    opts = lnocc.default_opts(precision=1, triples_kernel=getattr(lnocc, kernel), triples_chunk_mb=1)  # several chunks per slab
    f = lnocc.lnocc_build_ints(o, v, q, eps, B, opts)
    try:
        lnocc.lnocc_ccsd(f)
        want = list(lnocc.lnocc_triples(f, U))
        ws = torch.empty(lnocc.lnocc_workspace_bytes(o, v, q, opts), dtype=torch.uint8, device="cuda")
        lnocc.lnocc_frag_set_workspace(f, ws)
        e = torch.zeros(2, dtype=torch.float64, device="cuda")
        st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        lnocc.lnocc_triples_device(f, U, e, st, stream=s)
        s.synchronize()
        assert e.tolist() == want and int(st.item()) == 0
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lnocc.lnocc_triples_device(f, U, e, st, stream=s)
        for _ in range(2):
            e.zero_()
            ws.fill_(255)  # the launch tables and operands are rebuilt by every replay
            g.replay()
            torch.cuda.synchronize()
            assert e.tolist() == want and int(st.item()) == 0
    finally:
        f.free()
