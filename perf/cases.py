"""What a user of lnocc has it do, as measurable cases.

A calculation with this library runs, for each fragment of a crystal: the local active space
(internal orbitals, MP2 densities, LNOs, semi-canonical DF factors), integral assembly, CCSD, the
projected fragment energies and (T); plus one full-system MP2 energy for the composite correction, and
batches of uneven fragments. Production runs use the mixed precision (BF16x3 products, FP64 update and
energies); plain FP64 is used for small fragments, for checks, and where an MP2 or LNO quantity has to be
good to better than 1e-6 Eh. Sizes are those of the library's own workloads (4/24/96; 16/240/960;
nocc 8..24 with nvir 120..360 and naux about 4 nvir; nocc 32; 12/96/320; 30/200/640) or lie between them.

Each case is a dict with a "kind" (what is called) and the sizes. `listed()` gives the fixed cases,
`draw(rng)` one more from the same ranges, `prepare` the inputs and handles a program holds before the
call, `run` one call (or the few calls that make up the step), `work` what that step cannot do without,
and `exact` the same results in plain 64-bit torch where that is affordable.

Inputs follow the library's synthetic fragments: sorted orbital energies (a 0.7 Eh gap, or a small gap of
0.04..0.2 Eh), B[Q,p,q] symmetric in (p, q) with entries N(0, 1/naux) 0.3 exp(-|p-q|/20), and orthonormal
LO columns; drawn with torch's generators on the device.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2407_11258_gb300 import lnocc

FP64, MIXED = lnocc.LNOCC_PREC_FP64, lnocc.LNOCC_PREC_MIXED
DIIS = 8  # the library's default subspace


# ------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # one small fragment, plain FP64, build to free: every kernel is tiny, so launches, graph capture
        # and host waits are what the user waits for
        dict(name="solve_small_fp64", kind="solve", prec="fp64", o=4, v=24, q=96, nlo=1),
        # the library's headline workload: the diamond-like fragment, build to free, mixed precision
        dict(name="solve_diamond_mixed", kind="solve", prec="mixed", o=16, v=240, q=960, nlo=2),
        # CCSD iterations of a ragged fragment with a small gap (no size a multiple of a tile), mixed
        dict(name="ccsd_ragged_mixed", kind="ccsd", prec="mixed", o=19, v=151, q=604, iters=4, small=True),
        # CCSD iterations in plain FP64 (checks, refinement of metallic fragments)
        dict(name="ccsd_fp64", kind="ccsd", prec="fp64", o=12, v=96, q=320, iters=3, small=False),
        # (T) of the smallest fragments of a batch
        dict(name="triples_small_mixed", kind="triples", prec="mixed", o=8, v=120, q=480, nlo=1),
        # (T) of a ragged mid-size fragment (batches draw nocc from 8..24, so most are like this one)
        dict(name="triples_ragged_mixed", kind="triples", prec="mixed", o=19, v=125, q=500, nlo=1),
        # (T) of a (T)-dominated fragment with many occupied orbitals
        dict(name="triples_wide_mixed", kind="triples", prec="mixed", o=32, v=200, q=800, nlo=1),
        # (T) in plain FP64
        dict(name="triples_fp64", kind="triples", prec="fp64", o=8, v=64, q=256, nlo=2),
        # integral assembly of a large fragment and its MP2 fragment energy (screening of fragments; also
        # the part of every solve that comes before CCSD)
        dict(name="screen_mp2_mixed", kind="screen", prec="mixed", o=24, v=300, q=1200, nlo=1),
        # a batch of uneven fragments through the batch runtime, the production mode
        dict(name="batch_uneven_mixed", kind="batch", prec="mixed", count=5, omin=8, omax=24, vmin=96, vmax=176,
             shapes=1),
        # full-system MP2 energy of the composite correction in FP64
        dict(name="mp2_system_fp64", kind="mp2", prec="fp64", o=30, v=200, q=640),
        # the local active space of one fragment: densities, LNOs and the active-space DF factors
        dict(name="lno_space_fp64", kind="lno", prec="fp64", o=16, v=160, q=640, nlo=2, keep=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind, prec = rng.choice([("solve", "fp64"), ("solve", "mixed"), ("ccsd", "mixed"), ("ccsd", "fp64"),
                             ("triples", "mixed"), ("triples", "mixed"), ("triples", "mixed"), ("triples", "fp64"),
                             ("screen", "mixed"), ("batch", "mixed"), ("mp2", "fp64"), ("mp2", "mixed"),
                             ("lno", "fp64")])
    mixed = prec == "mixed"

    def sizes(olo, ohi, vlo, vhi, cap):
        """nocc, nvir and naux of one draw, the model cost o^3 v^4 at most `cap`."""
        while True:
            o, v = rng.randint(olo, ohi), _log_int(rng, vlo, vhi)
            if float(o) ** 3 * float(v) ** 4 <= cap:
                return dict(o=o, v=v, q=int(v * rng.uniform(3.2, 4.2)))

    case = dict(kind=kind, prec=prec)
    if kind == "solve":
        case.update(sizes(8, 24, 96, 240, 16.0 ** 3 * 240.0 ** 4) if mixed else sizes(2, 5, 12, 28, 1e9),
                    nlo=rng.randint(1, 2))
    elif kind == "ccsd":
        case.update(sizes(8, 24, 96, 260, 24.0 ** 3 * 220.0 ** 4) if mixed else sizes(4, 12, 24, 96, 12.0 ** 3 * 96.0 ** 4),
                    iters=rng.randint(2, 5) if mixed else rng.randint(2, 3), small=rng.random() < 0.5)
    elif kind == "triples":
        case.update(sizes(8, 32, 96, 240, 32.0 ** 3 * 200.0 ** 4) if mixed else sizes(3, 9, 24, 72, 8.0 ** 3 * 64.0 ** 4),
                    nlo=rng.choice([0, 1, 1, 2, 3]))
    elif kind == "screen":
        case.update(sizes(8, 24, 120, 300, 1e30), nlo=rng.randint(1, 2))
    elif kind == "batch":
        case.update(count=rng.randint(3, 5), omin=8, omax=rng.randint(14, 24), vmin=96, vmax=rng.randint(120, 176),
                    shapes=rng.randint(2, 10 ** 6))
    elif kind == "mp2":
        case.update(sizes(8, 30, 60, 200, 1e30))
    else:
        case.update(sizes(8, 16, 60, 160, 1e30), nlo=rng.randint(1, 3))
        case.update(keep=int(case["v"] * rng.uniform(0.4, 0.7)))
    return case


def _batch_shapes(case):
    rng = random.Random(case["shapes"])
    out = []
    for _ in range(case["count"]):
        v = rng.randint(case["vmin"], case["vmax"])
        out.append((rng.randint(case["omin"], case["omax"]), v, 4 * v))
    return out


# ------------------------------------------------------------------------------------------ inputs
def _fragment(o, v, q, nlo, seed, small=False):
    """(eps [n], B [q][n][n], U [o][nlo]) on the device."""
    n = o + v
    host = torch.Generator().manual_seed(seed)

    def uniform(k, lo, hi):
        return lo + (hi - lo) * torch.rand(k, generator=host, dtype=torch.float64)

    if small:
        vmin = float(uniform(1, 0.02, 0.1))
        ev, eo = uniform(v, vmin, 4.0).sort().values, uniform(o, -0.8, 0.0).sort().values - vmin
        ev[0], eo[-1] = vmin, -vmin
    else:
        eo, ev = uniform(o, -1.2, -0.4).sort().values, uniform(v, 0.3, 4.0).sort().values
    U = torch.linalg.qr(torch.randn(o, o, generator=host, dtype=torch.float64))[0][:, :max(nlo, 1)]
    dev = torch.Generator(device="cuda").manual_seed(seed)
    B = torch.randn(q, n, n, generator=dev, device="cuda", dtype=torch.float64)
    B = torch.triu(B) + torch.triu(B, 1).transpose(1, 2)
    i = torch.arange(n, device="cuda", dtype=torch.float64)
    B *= 0.3 / math.sqrt(q) * torch.exp(-(i[:, None] - i[None, :]).abs() / 20.0)
    return torch.cat([eo, ev]).cuda(), B.contiguous(), U.contiguous().cuda()


def _mp2_t2(eps, B, o):
    """First-order doubles t[i][j][a][b]."""
    ovov = _ovov(B, o)
    e = eps
    D = e[:o, None, None, None] + e[None, :o, None, None] - e[None, None, o:, None] - e[None, None, None, o:]
    return ovov.permute(0, 2, 1, 3).div(D).contiguous()


def _ovov(B, o):
    q, n = B.shape[0], B.shape[1]
    M = B[:, :o, o:].reshape(q, -1)
    return (M.T @ M).reshape(o, n - o, o, n - o)


def _amplitudes(eps, B, o, seed):
    """Amplitudes as a converged solve leaves them, for (T): the first-order doubles and small singles."""
    dev = torch.Generator(device="cuda").manual_seed(seed + 1)
    t1 = 0.005 * torch.randn(o, B.shape[1] - o, generator=dev, device="cuda", dtype=torch.float64)
    return t1, _mp2_t2(eps, B, o)


def _opts(case, **kw):
    return lnocc.default_opts(precision=MIXED if case["prec"] == "mixed" else FP64, **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return dict(case=case, opts=_opts(case), frags=[(o, v, q, *_fragment(o, v, q, 1, 1000 * seed + k))
                                                       for k, (o, v, q) in enumerate(_batch_shapes(case))])
    o, v, q = case["o"], case["v"], case["q"]
    eps, B, U = _fragment(o, v, q, case.get("nlo", 1), seed, case.get("small", False))
    s = dict(case=case, o=o, v=v, q=q, eps=eps, U=U)
    if kind in ("solve", "screen"):
        s.update(B=B, opts=_opts(case))
    elif kind == "ccsd":
        # a fixed number of iterations from the MP2 guess; the amplitudes land in the program's buffers
        s.update(frag=lnocc.lnocc_build_ints(o, v, q, eps, B, _opts(case, max_iter=case["iters"])),
                 t1=torch.empty(o, v, dtype=torch.float64, device="cuda"),
                 t2=torch.empty(o, o, v, v, dtype=torch.float64, device="cuda"))
    elif kind == "triples":
        # (T) restarted from stored amplitudes: the handle takes them over without iterating
        s.update(frag=lnocc.lnocc_build_ints(o, v, q, eps, B, _opts(case, max_iter=0)))
        t1, t2 = _amplitudes(eps, B, o, seed)
        lnocc.lnocc_ccsd(s["frag"], t1, t2, lnocc.LNOCC_GUESS_GIVEN, allow_noconv=True)
    elif kind == "mp2":
        s.update(Bov=B[:, :o, o:].contiguous(), prec=MIXED if case["prec"] == "mixed" else FP64)
    else:
        s.update(B=B, Bov=B[:, :o, o:].contiguous(), prec=MIXED if case["prec"] == "mixed" else FP64)
    return s


# ------------------------------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        _, res = lnocc.lnocc_solve_batch(s["frags"], s["opts"], allow_noconv=True)
        return [dict(e_mp2=r.e_mp2, e_ccsd=r.e_ccsd, e_ccsd_frag=r.e_ccsd_frag, e_mp2_frag=r.e_mp2_frag, e_t=r.e_t,
                     e_t_frag=r.e_t_frag) for r in res]
    o, v, q, eps, U = s["o"], s["v"], s["q"], s["eps"], s["U"]
    if kind == "solve":
        f = lnocc.lnocc_build_ints(o, v, q, eps, s["B"], s["opts"])
        e_mp2 = f.info().e_mp2
        e_ccsd, _, _ = lnocc.lnocc_ccsd(f, allow_noconv=True)
        e_ccsd_frag, e_mp2_frag = lnocc.lnocc_fragment_energy(f, U)
        e_t, e_t_frag = lnocc.lnocc_triples(f, U)
        f.free()
        return dict(e_mp2=e_mp2, e_ccsd=e_ccsd, e_ccsd_frag=e_ccsd_frag, e_mp2_frag=e_mp2_frag, e_t=e_t,
                    e_t_frag=e_t_frag)
    if kind == "screen":
        f = lnocc.lnocc_build_ints(o, v, q, eps, s["B"], s["opts"])
        e_mp2 = f.info().e_mp2
        _, e_mp2_frag = lnocc.lnocc_fragment_energy(f, U, ccsd=False)
        f.free()
        return dict(e_mp2=e_mp2, e_mp2_frag=e_mp2_frag)
    if kind == "ccsd":
        e, _, _ = lnocc.lnocc_ccsd(s["frag"], t1_out=s["t1"], t2_out=s["t2"], allow_noconv=True)
        if case["prec"] == "mixed":
            # a restart file of a mixed-precision solve holds FP32 amplitudes: BF16x3 products leave no more
            return dict(e=e, t1=s["t1"].float(), t2=s["t2"].float())
        return dict(e=e, t1=s["t1"], t2=s["t2"])
    if kind == "triples":
        e_t, e_t_frag = lnocc.lnocc_triples(s["frag"], U if case["nlo"] > 0 else None)
        return dict(e_t=e_t, e_t_frag=e_t_frag)
    if kind == "mp2":
        return dict(e_mp2=lnocc.lnocc_mp2_energy(s["prec"], o, v, q, eps, s["Bov"]))
    # the local active space of the fragment whose LOs are the columns of U
    W, f_int, _ = lnocc.lnocc_lno_internal(U, eps[:o].contiguous())
    Do, Dv = lnocc.lnocc_lno_densities(s["prec"], lnocc.LNOCC_LNO_MP2, o, v, q, eps, s["Bov"], W, f_int)
    Co, lam_o, no = lnocc.lnocc_lno_select(Do, W, ETA)
    Cv, lam_v, nv = lnocc.lnocc_lno_select(Dv, None, 0.0)
    C_occ = torch.cat([W, Co], dim=1).contiguous()
    C_vir = Cv[:, :case["keep"]].contiguous()  # an active space of a set size: the leading LNOs
    eF, BF, _ = lnocc.lnocc_active_space(s["prec"], o, v, q, eps, s["B"], C_occ, C_vir)
    return dict(D_occ=Do, D_vir=Dv, lam_occ=lam_o, lam_vir=lam_v, no=no, nv=nv, eps_F=eF, B_F=BF)


ETA = 1e-10  # occupied LNOs: every external orbital of these systems lies above, the projected-out ones below


# ------------------------------------------------------------------------------------------ floors
def _flops_iter(o, v, q):
    """One CCSD iteration: the packed particle-particle ladder, the o^3 v^3 rings, the DF products."""
    return o * o * v ** 4 / 2 + 8 * o ** 3 * v ** 3 + 2 * q * (o * o * v * v * 2 + 3 * o * v * v)


def _flops_triples(o, v):
    return 2 * o ** 3 * v ** 4 + 2 * o ** 4 * v ** 3  # every sorted virtual triple once


def _flops_build(o, v, q):
    return q * (o * v) ** 2 + 2 * q * o * v ** 3 + q * v ** 4 / 2


def _solve_work(o, v, q, iters):
    return (8.0 * q * (o + v) ** 2,
            _flops_build(o, v, q) + iters * _flops_iter(o, v, q) + _flops_triples(o, v))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_solve_work(o, v, q, 8) for o, v, q in _batch_shapes(case)]
        return dict(bytes=sum(x[0] for x in w), flops=sum(x[1] for x in w))
    o, v, q = case["o"], case["v"], case["q"]
    n = o + v
    esz = 4.0 if case["prec"] == "mixed" else 8.0
    if kind == "solve":
        b, f = _solve_work(o, v, q, 8)
    elif kind == "screen":
        b, f = 8.0 * q * n * n, _flops_build(o, v, q)
    elif kind == "ccsd":  # the ladder integrals are read once per iteration
        b = case["iters"] * (esz * v ** 4 / 2 + 16.0 * (o * v) ** 2) + 8.0 * q * n * n
        f = case["iters"] * _flops_iter(o, v, q)
    elif kind == "triples":
        b, f = 8.0 * (q * n * v + (o * v) ** 2), _flops_triples(o, v)
    elif kind == "mp2":
        b, f = 8.0 * q * o * v, float(q) * (o * v) ** 2
    else:
        nlo = case["nlo"]
        b = 8.0 * (q * o * v + 2 * q * n * n)
        f = nlo * (2.0 * q * o * v * v + 6.0 * o * v ** 3 + 4.0 * o * o * v * v) + 4.0 * q * n ** 3
    return dict(bytes=float(b), flops=float(f))


# ------------------------------------------------------------------------------------------ 64 bits
def _pair_L(B, o):
    """L[i][j][a][b] = 2 (ia|jb) - (ib|ja)."""
    g = _ovov(B, o).permute(0, 2, 1, 3)
    return 2.0 * g - g.transpose(2, 3)


def _project(tau, L, U):
    """sum_alpha sum_ii' U_i U_i' sum_jab tau_ij^ab L_i'j^ab."""
    o = tau.shape[0]
    E = tau.reshape(o, -1) @ L.reshape(o, -1).T
    return float(torch.einsum("ia,ij,ja->", U, E, U))


def _exact_mp2(eps, B, U, o):
    t2, L = _mp2_t2(eps, B, o), _pair_L(B, o)
    return dict(e_mp2=float((t2 * L).sum()), e_mp2_frag=_project(t2, L, U))


def _exact_ccsd(eps, B, o, iters, best):
    """`iters` DIIS-accelerated Jacobi iterations of closed-shell CCSD from the MP2 guess (T1-transformed
    form: Koch et al., Chem. Phys. Lett. 228, 233 (1994)). `best`: return the iterate of the lowest
    update norm, as the mixed solver does when it stops early, else the last one."""
    q, n = B.shape[0], B.shape[1]
    v = n - o
    ein = torch.einsum
    e1 = eps[:o, None] - eps[None, o:]
    e2 = e1[:, None, :, None] + e1[None, :, None, :]
    Bo = B[:, :o, :]
    h = torch.diag(eps) - 2.0 * ein("Qpq,Q->pq", B, ein("Qkk->Q", Bo[:, :, :o]))
    h = h + Bo.reshape(q * o, n).T @ Bo.reshape(q * o, n)  # (pk|kq), B symmetric
    L = _pair_L(B, o)
    ovov = _ovov(B, o)
    t1, t2 = torch.zeros(o, v, dtype=B.dtype, device=B.device), _mp2_t2(eps, B, o)
    vecs, errs = [], []
    keep = None
    for _ in range(iters):
        T = torch.zeros(n, n, dtype=B.dtype, device=B.device)
        T[o:, :o] = t1.T
        one = torch.eye(n, dtype=B.dtype, device=B.device)
        Bh = (one - T) @ B @ (one + T)
        F = (one - T) @ h @ (one + T) + 2.0 * ein("Qpq,Q->pq", Bh, ein("Qkk->Q", Bh[:, :o, :o]))
        F = F - Bh[:, :, :o].transpose(0, 1).reshape(n, -1) @ Bh[:, :o, :].transpose(1, 2).permute(1, 0, 2).reshape(n, -1).T
        oo, ov, vo, vv = Bh[:, :o, :o], Bh[:, :o, o:], Bh[:, o:, :o], Bh[:, o:, o:]
        u = 2.0 * t2 - t2.transpose(0, 1)
        # P-symmetric part: (ai|bj), both ladders
        R = ein("Qai,Qbj->ijab", vo, vo)
        tf, vvf = t2.reshape(o * o, v * v), vv.reshape(q, v * v)
        for a in range(v):  # sum_cd t_ij^cd (ac|bd)
            g = (vv[:, a, :].T @ vvf).reshape(v, v, v)  # [c][b][d]
            R[:, :, a, :] += (tf @ g.transpose(1, 2).reshape(v * v, v)).reshape(o, o, v)
        W = ein("Qki,Qlj->klij", oo, oo) + ein("ijcd,kcld->klij", t2, ovov)
        R += ein("klab,klij->ijab", t2, W)
        # C2, D2, E2 with P(ij, ab)
        X = ein("Qki,Qac->kiac", oo, vv) - 0.5 * ein("liad,kdlc->kiac", t2, ovov)
        S = ein("kjbc,kiac->ijab", t2, X)
        S = -0.5 * S - S.transpose(0, 1)
        Lt = L.permute(0, 2, 1, 3)  # [k][c][l][d]
        Y = 2.0 * ein("Qai,Qkc->aikc", vo, ov) - ein("Qac,Qki->aikc", vv, oo) + 0.5 * ein("ilad,kcld->aikc", u, Lt)
        S += 0.5 * ein("jkbc,aikc->ijab", u, Y)
        Fvv = F[o:, o:] - ein("klbd,ldkc->bc", u, ovov)
        Foo = F[:o, :o] + ein("ljcd,kdlc->kj", u, ovov)
        S += ein("ijac,bc->ijab", t2, Fvv) - ein("ikab,kj->ijab", t2, Foo)
        R += S + S.permute(1, 0, 3, 2)
        R1 = ein("Qad,Qdi->ia", vv, ein("Qkc,kicd->Qdi", ov, u))
        R1 = R1 - ein("klac,kilc->ia", u, ein("Qki,Qlc->kilc", oo, ov)) + ein("ikac,kc->ia", u, F[:o, o:]) + F[o:, :o].T
        d = torch.cat([(R1 / e1).reshape(-1), (R / e2).reshape(-1)])
        vecs.append(torch.cat([t1.reshape(-1), t2.reshape(-1)]) + d)
        errs.append(d)
        vecs, errs = vecs[-DIIS:], errs[-DIIS:]
        m = len(vecs)
        G = torch.zeros(m + 1, m + 1, dtype=torch.float64)
        for i in range(m):
            for j in range(m):
                G[i, j] = float(errs[i] @ errs[j])
        G /= G.diagonal()[:m].max()
        G[m, :m] = G[:m, m] = -1.0
        G[m, m] = 0.0
        c = torch.linalg.solve(G, torch.cat([torch.zeros(m, dtype=torch.float64), torch.tensor([-1.0], dtype=torch.float64)]))
        x = sum(float(c[i]) * vecs[i] for i in range(m))
        t1, t2 = x[:o * v].reshape(o, v), x[o * v:].reshape(o, o, v, v)
        rms = float(d @ d)
        if keep is None or not best or rms < keep[0]:
            keep = (rms, t1, t2)
    _, t1, t2 = keep
    tau = t2 + t1[:, None, :, None] * t1[None, :, None, :]
    return dict(e=float((tau * L).sum()), t1=t1, t2=t2)


def _exact_triples(eps, B, U, o, nlo, t1, t2):
    """(T) energy and its projection (supplementary Sec. S1), one (j, k <= j) pair at a time."""
    v = B.shape[1] - o
    ov, vv = B[:, :o, o:], B[:, o:, o:]
    ovoo = torch.einsum("Qkc,Qjl->kcjl", ov, B[:, :o, :o])
    ovov = _ovov(B, o)
    ovvv = torch.einsum("Qia,Qbd->iabd", ov, vv)
    eo, ev = eps[:o], eps[o:]
    evs = ev[:, None, None] + ev[None, :, None] + ev[None, None, :]

    def X(i, j, k):
        """sum_d (ai|bd) t_kj^cd - sum_l (ck|jl) t_il^ab as [a][b][c]; i, j or k a list of all i."""
        x = torch.einsum("...abd,...cd->...abc", ovvv[i], t2[k, j])
        return x - torch.einsum("...cl,...lab->...abc", ovoo[k, :, j, :], t2[i])

    e_t = e_f = 0.0
    al = torch.arange(o, device=B.device)
    for j in range(o):
        for k in range(j + 1):
            J, K = torch.full_like(al, j), torch.full_like(al, k)
            W = X(al, J, K) + X(al, K, J).permute(0, 1, 3, 2) + X(J, al, K).permute(0, 2, 1, 3)
            W += X(J, K, al).permute(0, 3, 1, 2) + X(K, al, J).permute(0, 2, 3, 1) + X(K, J, al).permute(0, 3, 2, 1)
            V = W + ovov[:, :, j, :][..., None] * t1[k] + ovov[:, :, k, :][:, :, None, :] * t1[j][None, None, :, None]
            V += ovov[j, :, k, :][None, None] * t1[:, :, None, None]
            s = torch.rsqrt(evs[None] - eo[:, None, None, None] - eo[j] - eo[k])
            W *= s
            V *= s
            for w, y in ((W, V), (W.transpose(2, 3), V.transpose(2, 3)))[:1 if j == k else 2]:  # (j, k), (k, j)
                z = 4.0 * w + w.permute(0, 3, 1, 2) + w.permute(0, 2, 3, 1)
                y = y - y.permute(0, 3, 2, 1)
                e_t -= float((z * y).sum()) / 3.0
                if nlo > 0:
                    e_f -= float(((U.T @ z.reshape(o, -1)) * (U.T @ y.reshape(o, -1))).sum()) / 3.0
    return dict(e_t=e_t, e_t_frag=e_f)


def _exact_lno(eps, B, U, o, keep):
    v = B.shape[1] - o
    ov = B[:, :o, o:]
    f, R = torch.linalg.eigh(U.T @ (eps[:o, None] * U))
    W = U @ R
    t = torch.einsum("QIa,Qjb->Iajb", torch.einsum("iI,Qia->QIa", W, ov), ov)
    t = t / (f[:, None, None, None] + eps[None, None, :o, None] - eps[None, o:, None, None] - eps[None, None, None, o:])
    C, Cp = t.permute(2, 0, 1, 3).reshape(o, -1), t.permute(2, 0, 3, 1).reshape(o, -1)
    Do = 4.0 * C @ C.T - C @ Cp.T - Cp @ C.T
    A, Bm = t.permute(1, 0, 2, 3).reshape(v, -1), t.permute(3, 0, 2, 1).reshape(v, -1)
    Dv = 2.0 * (A @ A.T + Bm @ Bm.T) - A @ Bm.T - Bm @ A.T

    def kept(D, Win, eta):
        P = torch.eye(D.shape[0], dtype=D.dtype, device=D.device)
        if Win is not None:
            P = P - Win @ Win.T
        lam, C = torch.linalg.eigh(P @ D @ P)
        at = (lam.abs() >= eta).nonzero().reshape(-1).flip(0)
        return lam[at].contiguous(), C[:, at]

    lo, Co = kept(Do, W, ETA)
    lv, Cv = kept(Dv, None, 0.0)
    Co, Ck = torch.cat([W, Co], dim=1), Cv[:, :keep]
    eF = torch.cat([torch.linalg.eigvalsh(Co.T @ (eps[:o, None] * Co)), torch.linalg.eigvalsh(Ck.T @ (eps[o:, None] * Ck))])
    # B_F is fixed up to the signs of its orbitals: no one value
    return dict(D_occ=Do, D_vir=Dv, lam_occ=lo, lam_vir=lv, no=int(lo.numel()), nv=int(lv.numel()), eps_F=eF, B_F=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for k, (o, v, q) in enumerate(_batch_shapes(case)):
            eps, B, U = _fragment(o, v, q, 1, 1000 * seed + k)
            out.append(dict(_exact_mp2(eps, B, U, o), e_ccsd=None, e_ccsd_frag=None, e_t=None, e_t_frag=None))
        return out
    o, v, q = case["o"], case["v"], case["q"]
    eps, B, U = _fragment(o, v, q, case.get("nlo", 1), seed, case.get("small", False))
    if kind == "screen":
        return _exact_mp2(eps, B, U, o)
    if kind == "mp2":
        return dict(e_mp2=_exact_mp2(eps, B, U, o)["e_mp2"])
    if kind == "lno":
        return _exact_lno(eps, B, U, o, case["keep"])
    if kind == "ccsd":
        cost = case["iters"] * (2.0 * q * v ** 4 + 2.0 * o * o * v ** 4 + 20.0 * o ** 3 * v ** 3)
        return _exact_ccsd(eps, B, o, case["iters"], case["prec"] == "mixed") if cost < 1.2e13 else None
    if kind == "triples":
        if 6.0 * o ** 3 * v ** 4 > 1.2e13:
            return None
        return _exact_triples(eps, B, U, o, case["nlo"], *_amplitudes(eps, B, o, seed))
    out = dict(_exact_mp2(eps, B, U, o), e_ccsd=None, e_ccsd_frag=None, e_t=None, e_t_frag=None)
    if o * v <= 200:  # small enough to iterate to convergence
        c = _exact_ccsd(eps, B, o, 30, False)
        tau = c["t2"] + c["t1"][:, None, :, None] * c["t1"][None, :, None, :]
        out.update(e_ccsd=c["e"], e_ccsd_frag=_project(tau, _pair_L(B, o), U),
                   **_exact_triples(eps, B, U, o, case["nlo"], c["t1"], c["t2"]))
    return out
