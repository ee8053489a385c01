"""Performance cases: what a user of the library has it do, over the sizes it is used at.

Every case is one call, or one short sequence of calls, of the Python binding
(`paper_1702_00339_gb300.fock`) on seeded problems:

  plan       a device-resident batch executed and its results fetched (the benchmark's step)
  solve      the one-shot call on host problems: plan, run and fetch in one
  serve      a burst of requests submitted to the server and polled
  assemble   the generators of a chain, assembled and copied out
  matvec     the structured operator of an assembled chain applied to device vectors
  product    an FP64 matrix product on the tensor cores

Exponents are even-tempered series with a few per cent of jitter drawn from the
seed, as basis sets are built, so that every eigenvalue asked for is determined
by the problem to many more digits than FP64 rounding moves it.  Cells have no
mirror symmetry where the Fourier index of each eigenvalue is returned, so that
its order is determined too.
"""
import math

import numpy as np
import torch

import lattice_inputs as li
from paper_1702_00339_gb300 import fock

# nuclei of a cell, as fractions: one or two, at places without symmetry
PLACES = {1: [[0.3, 0.45, 0.6]], 2: [[0.25, 0.25, 0.25], [0.6875, 0.5, 0.625]]}


def listed():
    return [
        # the smallest call: one short ring (8 cells, the four s functions of the smallest workload)
        dict(name="ring_8", call="plan", kind="ring", count=1, L1=8, m0=4, n0=32, perp=256, R=24),
        # one application of a 64-cell chain's operator, as an outer iterative solver does it
        dict(name="matvec_1", call="matvec", L1=64, m0=8, n0=15, pad=32, perp=256, R=32, nvec=1, which=0),
        # a block of 72 vectors on the longest chain (512 cells of 32 functions)
        dict(name="matvec_72", call="matvec", L1=512, m0=32, n0=15, pad=256, perp=256, R=40, nvec=72, which=1),
        # the Gram matrix of a block iteration's basis on that chain: 216 columns of 16384
        dict(name="gram_216", call="product", M=216, N=216, K=16384, ksplit=32, sym=True),
        # assembly alone: the generators and wall blocks of a chain of 101 cells, 16 functions each
        dict(name="assemble_101", call="assemble", L1=101, m0=16, n0=16, pad=32, perp=256, R=32),
        # two lattices of 16^3 cells, two nuclei and 16 functions per cell: every eigenvalue
        dict(name="lattice_16", call="plan", kind="lattice", count=2, L1=16, L2=16, L3=16, m0=16, nuclei=2, n0=32, R=32),
        # the largest lattice: 32^3 cells of 32 functions on a grid too coarse for the core functions,
        # whose overlaps vanish and are cut
        dict(name="lattice_32", call="plan", kind="lattice", count=1, L1=32, L2=32, L3=32, m0=32, nuclei=2, n0=16, R=40),
        # one chain of the benchmark's shape (64 cells, 1024 x 256 x 256 nodes) in one call
        dict(name="chain_64", call="solve", kind="box", count=1, L1=64, m0=8, n0=15, pad=32, perp=256, R=32, k=16, defects=0, precision=0),
        # a batch of 32 such chains, each beside its periodic ring (box against supercell)
        dict(name="pairs_64", call="plan", kind="pair", count=32, L1=64, m0=8, n0=15, pad=32, perp=256, R=32, k=16, precision=0),
        # the largest chain (512 cells of 32 functions, 64 eigenpairs) in the mixed form
        dict(name="chain_512", call="plan", kind="box", count=1, L1=512, m0=32, n0=15, pad=256, perp=256, R=40, k=64, defects=0, precision=1),
        # substituted and missing nuclei: three rings of 61 cells, 16 functions each
        dict(name="defects_61", call="plan", kind="defect_ring", count=3, L1=61, m0=16, n0=16, perp=256, R=32, k=16, defects=2, precision=0),
        # a burst of twelve requests of the serving mix: chains and rings with and without defects, cubes
        dict(name="burst_12", call="serve", count=12, slots=2, mix=1, longest=96, largest=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["ring", "matvec", "matvec", "product", "assemble", "lattice", "lattice", "box", "box", "pair", "defect_ring", "serve"])
    m0 = rng.choice([4, 7, 8, 12, 16])
    n0 = rng.choice([12, 15, 16])
    if what == "ring":
        return dict(call="plan", kind="ring", count=_log(rng, 1, 24), L1=_log(rng, 4, 256), m0=m0, n0=n0, perp=256, R=rng.choice([24, 32]))
    if what == "matvec":
        L = _log(rng, 16, 512)
        nvec = _log(rng, 1, 72)
        return dict(call="matvec", L1=L, m0=rng.choice([4, 7, 8, 16, 32]), n0=15, pad=rng.choice([32, 64]), perp=256, R=32, nvec=nvec, which=rng.choice([0, 1]))
    if what == "product":
        sym = rng.random() < 0.5
        M = _log(rng, 20, 256)
        return dict(call="product", M=M, N=M if sym else _log(rng, 16, 1024), K=_log(rng, 15, 16384), ksplit=rng.choice([1, 4, 16, 32]), sym=sym)
    if what == "assemble":
        return dict(call="assemble", L1=_log(rng, 24, 128), m0=m0, n0=n0, pad=32, perp=256, R=32)
    if what == "lattice":
        Ls = [_log(rng, 6, 20) for _ in range(3)]
        m0 = rng.choice([8, 14, 16])
        return dict(call="plan", kind="lattice", count=_log(rng, 1, 4), L1=Ls[0], L2=Ls[1], L3=Ls[2], m0=m0, nuclei=rng.choice([1, 2]) if m0 == 8 else 2, n0=16, R=rng.choice([24, 32]))
    if what == "box":
        long = rng.random() < 0.4
        L = _log(rng, 128, 300) if long else _log(rng, 32, 128)
        return dict(call=rng.choice(["solve", "plan"]), kind="box", count=1 if long else _log(rng, 1, 8), L1=L, m0=rng.choice([8, 16]) if long else m0, n0=n0, pad=32, perp=256, R=32,
                    k=rng.choice([16, 24, 32]) if long else 16, defects=0, precision=rng.choice([0, 1]))
    if what == "pair":
        return dict(call="plan", kind="pair", count=_log(rng, 1, 32), L1=_log(rng, 32, 96), m0=8, n0=n0, pad=32, perp=256, R=32, k=16, precision=0)
    if what == "defect_ring":
        m0 = rng.choice([4, 8, 16])
        return dict(call="plan", kind="defect_ring", count=_log(rng, 1, 3), L1=_log(rng, 32, 61 if m0 == 16 else 100), m0=m0, n0=16, perp=256, R=32, k=16, defects=rng.choice([1, 2, 3]), precision=rng.choice([0, 1]))
    return dict(call="serve", count=rng.choice([6, 12, 16]), slots=rng.choice([1, 2, 3]), mix=rng.randrange(1000), longest=_log(rng, 48, 96), largest=rng.choice([8, 10, 12]))


# ---- problems ----

def _table(R, zmin, zmax):
    """A Gaussian-sum quadrature of 1/z on [zmin, zmax]: the trapezoid rule of
    (2/sqrt(pi)) int exp(u - z^2 e^(2u)) du with a node for its lower tail."""
    lo, hi = math.log(1.0 / zmax), math.log(2.5 / zmin)
    u = np.linspace(lo, hi, R - 1)
    s = 2.0 / math.sqrt(math.pi)
    c = s * np.exp(u) * (u[1] - u[0])
    c[0] *= 0.5
    c[-1] *= 0.5
    return np.append(math.exp(lo) / math.sqrt(3.0), np.exp(u)), np.append(s * math.exp(lo), c)


def _basis(rng, m0, nuclei, lowest, ratio):
    """m0 functions, shared evenly by the nuclei: s functions in an even-tempered
    series, and a set of three p functions for every 8 functions of a nucleus
    (six sets for 32 on one)."""
    exps, ang, cen = [], [], []
    for a in range(nuclei):
        own = m0 // nuclei + (1 if a < m0 % nuclei else 0)
        sets = {7: 1, 8: 1, 12: 2, 14: 2, 16: 3, 32: 6}.get(own, 0)
        ns = own - 3 * sets
        # (the most diffuse function, which sets how far cells reach, is the series' own)
        exps += list(lowest * ratio ** np.arange(ns) * np.exp(np.append(0.0, rng.uniform(-0.1, 0.1, ns - 1))))
        ang += [0] * ns
        for i in range(sets):
            exps += [lowest * ratio ** (i + 1) * math.exp(rng.uniform(-0.1, 0.1))] * 3
            ang += [1, 2, 3]
        cen += [a] * own
    return dict(exps=np.array(exps), ang=np.array(ang), centre=np.array(cen))


def _problem(rng, kind, case):
    L1, m0, n0, R = case["L1"], case["m0"], case["n0"], case["R"]
    if kind == "lattice":
        L = (L1, case["L2"], case["L3"])
        M0, b0 = case["nuclei"], 4.0
        p = li.Problem(L=L, periodic=(1, 1, 1), N=tuple(x * n0 for x in L), n0=n0, b0=b0, Z=np.array([1.0, 2.0])[:M0],
                       frac=np.array(PLACES[M0]), R=R, **_basis(rng, m0, M0, 0.25, 4.0 if m0 == 32 else 3.5))
        diam = b0 * math.sqrt(sum((x + 1) ** 2 for x in L))
    else:
        # chains: b0 = 2 bohr; 32 functions on one nucleus need a closer series
        # (off the axis, so that a ring's p_y and p_z bands differ)
        ratio = 1.8 if m0 == 32 else 2.5 if kind != "ring" else 3.0
        off = [[0.5, 0.45, 0.6]] if kind == "ring" else [[0.5, 0.5, 0.5]]
        box = kind == "box"
        p = li.Problem(L=(L1, 1, 1), periodic=(0 if box else 1, 0, 0), N=(L1 * n0 + (2 * case["pad"] if box else 0), case["perp"], case["perp"]),
                       n0=n0, b0=2.0, Z=np.array([1.0]), frac=np.array(off), R=R, k_eig=case.get("k", 16) if kind != "ring" else 0,
                       precision=case.get("precision", 0), **_basis(rng, m0, 1, 0.3 if kind == "ring" else 0.2, ratio))
        if case.get("defects"):
            p.defects = li.random_defects(rng, p.L, 1, case["defects"])
        diam = p.b0 * (L1 + 1) + case["perp"] * p.h
    return p.with_table(*_table(R, p.h / 4.0, diam))


def _problems(case, seed):
    rng = np.random.default_rng([abs(int(seed)), 17])
    if case["call"] == "serve":
        out, size = [], np.random.default_rng(case["mix"])   # the requests' sizes are the case's, the rest the seed's
        for i in range(case["count"]):
            kind = ["defect_ring", "lattice", "box", "lattice", "ring", "box"][i % 6]
            if kind == "lattice":
                L = [int(size.integers(6, case["largest"] + 1)) for _ in range(3)]
                m0 = int(size.choice([4, 8, 16]))
                c = dict(L1=L[0], L2=L[1], L3=L[2], m0=m0, nuclei=2 if m0 == 16 else 1, n0=16, R=32)
            else:
                c = dict(L1=int(size.integers(32, case["longest"] + 1)), m0=int(size.choice([4, 8])), n0=16, pad=32, perp=256, R=32, k=16,
                         defects=int(size.integers(1, 4)) if kind == "defect_ring" else int(size.integers(0, 2)) if kind == "box" else 0)
            out.append(_problem(rng, kind, c))
        return out
    kinds = {"pair": ["box", "ring"], None: ["box"]}.get(case.get("kind"), [case.get("kind")])
    return [_problem(rng, k, case) for _ in range(case.get("count", 1)) for k in kinds]


# ---- the calls ----

def _fetch(results):
    """The spectra one after another, and the Fourier index of each periodic eigenvalue."""
    blocks = [r["block_of"] for r in results if r["block_of"] is not None]
    out = {"evals": np.concatenate([r["evals"] for r in results])}
    if blocks:
        out["blocks"] = np.concatenate(blocks)
    return out


def prepare(case, seed):
    call = case["call"]
    if call == "product":
        A, B = _operands(case, seed)
        return dict(case=case, ctx=fock.Context(0), A=A, B=B, C=torch.zeros(case["N"], case["M"], device="cuda", dtype=torch.float64))
    ps = _problems(case, seed)
    if call == "serve":
        return dict(case=case, server=fock.Server(0, slots=case["slots"]), problems=ps)
    ctx = fock.Context(0)
    if call == "plan":
        return dict(case=case, ctx=ctx, plan=ctx.plan(ps))
    if call == "matvec":
        op = ctx.assemble(ps[0])
        return dict(case=case, ctx=ctx, op=op, x=_vectors(case, seed, ps[0].Nb), y=torch.zeros(case["nvec"], ps[0].Nb, device="cuda", dtype=torch.float64))
    return dict(case=case, ctx=ctx, problems=ps)


def _operands(case, seed):
    """A^T and B^T of a product, a row for each column: columns of a basis, about unit
    norm, the rows' sizes spread over two decades (wall to bulk); B is A in a Gram product."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 31))
    size = torch.exp(2.3 * torch.randn(1, case["K"], generator=g, device="cuda", dtype=torch.float64)).clamp(0.1, 10.0)
    A = size * torch.randn(case["M"], case["K"], generator=g, device="cuda", dtype=torch.float64) / math.sqrt(case["K"])
    return A, A if case["sym"] else torch.randn(case["N"], case["K"], generator=g, device="cuda", dtype=torch.float64)


def _vectors(case, seed, n):
    g = torch.Generator(device="cuda").manual_seed((int(seed) + 1) % (1 << 31))
    return torch.randn(case["nvec"], n, generator=g, device="cuda", dtype=torch.float64)


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "plan":
        state["plan"].execute()
        return _fetch(state["plan"].outputs())
    if call == "solve":
        return _fetch(state["ctx"].solve(state["problems"]))
    if call == "serve":
        tickets = [state["server"].submit(p) for p in state["problems"]]
        return _fetch([state["server"].poll(t) for t in tickets])
    if call == "matvec":
        state["op"].matvec_device(state["x"].data_ptr(), state["y"].data_ptr(), case["nvec"], case["which"])
        return state["y"]
    if call == "assemble":
        op = state["ctx"].assemble(state["problems"][0])
        out = op.generators()
        op.close()
        return dict(zip(("H", "S", "EH", "ES", "cells"), out))
    M, N, K = case["M"], case["N"], case["K"]
    A, B = state["A"], state["B"]
    # columns of A and B contiguous along the summation; C column-major
    state["ctx"].split_dgemm(M, N, K, A.data_ptr(), K, 1, B.data_ptr(), 1, K, state["C"].data_ptr(), 1, M, ksplit=case["ksplit"], sym=case["sym"])
    return state["C"]


# ---- what a pass cannot do without ----

def _reach(m0, kind):
    """Cells over which functions of a chain overlap (cut-off 1e-14, lowest exponent 0.2 or 0.3, b0 = 2)."""
    return int((2.0 * math.sqrt(math.log(1e14) / (0.3 if kind == "ring" else 0.2)) + 0.13) / 2.0)


def _spectrum_work(c, kind):
    """A periodic problem: its blocks (conjugate pairs once) formed, reduced and diagonalised; eigenvalues and indices written."""
    m, cells, nuc = c["m0"], c["L1"] * c.get("L2", 1) * c.get("L3", 1), c.get("nuclei", 1)
    per = 10.0 * (nuc * c["R"] + 3) * m * (m + 1) + (8.0 + 16.0 / 3.0) * m ** 3
    return cells * m * 12.0 + 8.0 * (m * 4 + 2 * c["R"]), (cells // 2 + 1) * per


def _chain_work(c):
    """A chain: ten steps of the block iteration (Gram products, basis products, banded solve and images) and the assembly."""
    m, L, k = c["m0"], c["L1"], c.get("k", 16)
    n, kb, D = L * m, k + max(4, k // 8), _reach(m, "box")
    step = 2.0 * n * (3 * kb) ** 2 + 4.0 * n * 3 * kb * 2 * kb + 4.0 * n * kb * kb + 2.0 * L * (2 * D + 1) * m * m * 6 * kb + 4.0 * L * (D + 1) * m * m * kb + 4.0 * (3 * kb) ** 3
    return 8.0 * (m * 4 + 2 * c["R"] + k), 10.0 * step + 6.0 * (2 * D + 1) * c["R"] * m * m


def work(case):
    call = case["call"]
    if call == "product":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8.0 * (K * M + (0 if case["sym"] else K * N) + M * N), "flops": 2.0 * M * N * K * (0.5 if case["sym"] else 1.0)}
    if call == "matvec":
        m, D = case["m0"], _reach(case["m0"], "box")
        n = case["L1"] * m
        return {"bytes": 8.0 * (2 * n * case["nvec"] + (D + 1) * m * m), "flops": 2.0 * n * (2 * D + 1) * m * case["nvec"]}
    if call == "assemble":
        m, D = case["m0"], _reach(case["m0"], "box")
        blocks = 2 * D + 1 + (D + 1) ** 2 // 2
        return {"bytes": 16.0 * blocks * m * m, "flops": blocks * case["R"] * m * m * (2.0 * case["n0"] + 6.0)}
    if call == "serve":
        half = case["count"] / 2.0
        L, w = case["longest"] * 0.7, case["largest"] * 0.75
        b1, f1 = _spectrum_work(dict(L1=w, L2=w, L3=w, m0=8, R=32), "lattice")
        b2, f2 = _chain_work(dict(L1=L, m0=6, R=32))
        return {"bytes": half * (b1 + b2), "flops": half * (f1 + f2)}
    b = f = 0.0
    for kind in {"pair": ["box", "ring"]}.get(case["kind"], [case["kind"]]):
        bb, ff = _spectrum_work(case, kind) if kind in ("ring", "lattice") else _chain_work(case)
        b, f = b + case["count"] * bb, f + case["count"] * ff
    return {"bytes": b, "flops": f}


# ---- the same results in 64 bits with plain torch ----

def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _t(x):
    return torch.as_tensor(np.asarray(x, float), dtype=torch.float64, device=_dev())


def _gauss(t, lo, hi):
    """int_lo^hi exp(-t^2 s^2) ds without cancellation in the tails."""
    a, b = t * lo, t * hi
    v = torch.where(a >= 0, torch.erfc(a) - torch.erfc(b), torch.where(b <= 0, torch.erfc(-b) - torch.erfc(-a), torch.erf(b) - torch.erf(a)))
    return v * (math.sqrt(math.pi) / 2.0) / t


def _functions(p, ax, rho, cells):
    """g[i, k, mu]: the 1D factor of function mu of cell k at node rho_i (positions (rho + 1/2) h)."""
    x = (_t(rho) + 0.5) * p.h
    al = _t(p.exps)
    f = _t(p.frac[np.asarray(p.centre), ax])
    d = x[:, None, None] - (_t(cells)[None, :, None] + f) * p.b0
    if p.periodic[ax]:
        per = p.N[ax] * p.h
        d = d - per * torch.floor(d / per + 0.5)
    isp = torch.as_tensor(np.asarray(p.ang) == ax + 1, device=d.device)
    v = (2.0 * al / math.pi) ** 0.25 * torch.where(isp, 2.0 * torch.sqrt(al), torch.ones_like(al)) * torch.exp(-al * d * d) * torch.where(isp, d, torch.ones_like(d))
    return torch.where(d.abs() <= torch.sqrt(math.log(1.0 / p.eps_support) / al), v, torch.zeros_like(v))


def _nodes(p, ax):
    pad = 0 if p.periodic[ax] else (p.N[ax] - p.L[ax] * p.n0) // 2
    return np.arange(p.N[ax]) - pad


def _reduced(p, ax, rho):
    """Nodes replicated into the reference cell (cell index clamped to the box)."""
    k = rho // p.n0
    return rho - (k if p.periodic[ax] else np.clip(k, 0, p.L[ax] - 1)) * p.n0


def _potential(p, ax, r):
    """The window-summed factors [nucleus, q, i] at reduced nodes r."""
    L, hw = p.L[ax], (0 if p.L[ax] == 1 else p.L[ax] // 2)
    x, t = _t(r) * p.h, _t(p.sinc_t)[:, None]
    out = []
    for nu in range(p.M0):
        s = 0.0
        for k in range(-hw, hw + 1):
            w = 0.5 if L > 1 and L % 2 == 0 and abs(k) == hw else 1.0
            u = (x - (k + p.frac[nu, ax]) * p.b0)[None, :]
            s = s + w * _gauss(t, u, u + p.h)
        out.append(s)
    return torch.stack(out)


def _mass_stiff(p, ax, ga, gb, ring):
    """<a, M b> and <a, K b> of P1 elements for node columns ga, gb (nodes, .)."""
    z = torch.zeros_like(gb[:1])
    lo = torch.cat([gb[-1:] if ring else z, gb[:-1]])
    hi = torch.cat([gb[1:], gb[:1] if ring else z])
    return ga.T @ (4.0 * gb + lo + hi) * (p.h / 6.0), ga.T @ (2.0 * gb - lo - hi) / p.h


def _weights(p):
    return torch.cat([_t(p.sinc_c) * float(z) for z in p.Z])


def _transverse(p):
    """Per transverse axis of a chain (one cell): mass, stiffness and the potential forms [term, mu, nu]."""
    out = []
    for ax in (1, 2):
        rho = _nodes(p, ax)
        g = _functions(p, ax, rho, [0])[:, 0]
        s, a = _mass_stiff(p, ax, g, g, False)
        out.append((s, a, torch.einsum("im,ti,in->tmn", g, _potential(p, ax, _reduced(p, ax, rho)).flatten(0, 1), g)))
    return out


def _chain_matrix(p, want="HS"):
    """Dense H and S of a chain or ring, defects included."""
    (s1, a1, y1), (s2, a2, y2) = _transverse(p)
    rho, ring, m, L = _nodes(p, 0), bool(p.periodic[0]), p.m0, p.L[0]
    g = _functions(p, 0, rho, range(L))
    G = g.reshape(len(rho), L * m)
    s0, a0 = _mass_stiff(p, 0, G, G, ring)
    per = lambda b: b.repeat(L, L)  # noqa: E731
    S = s0 * per(s1 * s2) if "S" in want else None
    if "H" not in want:
        return None, S
    H = 0.5 * (a0 * per(s1 * s2) + s0 * per(a1 * s2 + s1 * a2))
    del a0, s0
    w = _weights(p)[:, None, None]
    F = torch.einsum("ti,tmn->imn", _potential(p, 0, _reduced(p, 0, rho)).flatten(0, 1), w * y1 * y2)
    for d in p.defects:
        own = []
        for ax in range(3):
            u = (_t(_nodes(p, ax)) + 0.5 - p.frac[d.nucleus, ax] * p.n0 - d.cell[ax] * p.n0) * p.h
            if p.periodic[ax]:
                u = u - p.N[ax] * p.h * torch.floor(u / (p.N[ax] * p.h) + 0.5)
            own.append(_gauss(_t(p.sinc_t)[:, None], u[None] - 0.5 * p.h, u[None] + 0.5 * p.h))
        forms = [torch.einsum("im,qi,in->qmn", *(lambda q: (q, own[ax], q))(_functions(p, ax, _nodes(p, ax), [0])[:, 0])) for ax in (1, 2)]
        F = F + (d.newZ - p.Z[d.nucleus]) * torch.einsum("qi,qmn->imn", own[0], _t(p.sinc_c)[:, None, None] * forms[0] * forms[1])
    V = torch.empty(L, m, L, m, dtype=torch.float64, device=H.device)
    for mu in range(m):
        for nu in range(mu, m):
            b = (g[:, :, mu] * F[:, mu, nu][:, None]).T @ g[:, :, nu]
            V[:, mu, :, nu] = b
            V[:, nu, :, mu] = b.T
    H -= V.reshape(L * m, L * m)
    return H, S


def _chain_lowest(p):
    H, S = _chain_matrix(p)
    Li = torch.linalg.inv(torch.linalg.cholesky(0.5 * (S + S.T)))
    C = Li @ (0.5 * (H + H.T)) @ Li.T
    return torch.linalg.eigvalsh(0.5 * (C + C.T))[: p.k_eig or 16].cpu().numpy()


def _spectrum(p):
    """Every eigenvalue of a periodic problem, ascending (+inf for directions whose overlap is numerically zero)."""
    X, scale = [], 1.0
    for ax in range(3):
        rho, L, ring = _nodes(p, ax), p.L[ax], bool(p.periodic[ax])
        g = _functions(p, ax, rho, range(L) if ring else [0])
        P = _potential(p, ax, _reduced(p, ax, rho)).flatten(0, 1)
        g0 = g[:, 0]
        fs = []
        for d in range(L if ring else 1):   # block (cell d, cell 0)
            s, a = _mass_stiff(p, ax, g[:, d], g0, ring)
            fs.append(torch.cat([s[None], a[None], torch.einsum("im,ti,in->tmn", g[:, d], P, g0)]))
        x = torch.stack(fs)
        scale = scale * x[:, 0].abs().sum(0)
        X.append(torch.fft.fft(x.to(torch.complex128), dim=0))
    tau = float(torch.linalg.norm(scale)) * p.Nb * 2.0 ** -52
    w = _weights(p).to(torch.complex128)
    done = []
    n1, n2, n3 = (len(x) for x in X)
    for j1 in range(n1 // 2 + 1):
        times = 1 if j1 == 0 or 2 * j1 == n1 else 2   # the blocks at -j are the conjugates
        for j2 in range(n2):
            a, b, c = X[0][j1], X[1][j2], X[2]
            S = a[0] * b[0] * c[:, 0]
            H = 0.5 * (a[1] * b[0] * c[:, 0] + a[0] * b[1] * c[:, 0] + a[0] * b[0] * c[:, 1]) - torch.einsum("tmn,jtmn->jmn", w[:, None, None] * a[2:] * b[2:], c[:, 2:])
            done.append((times, H, S))
    H = torch.cat([h for _, h, _ in done])
    S = torch.cat([s for _, _, s in done])
    times = np.concatenate([np.full(len(h), t) for t, h, _ in done])
    s, Q = torch.linalg.eigh(0.5 * (S + S.mH))
    kept = (s > tau).sum(1).cpu().numpy()
    ev = np.full((len(times), p.m0), np.inf)
    for r in np.unique(kept):
        at = np.flatnonzero(kept == r)
        if r:
            i = torch.as_tensor(at, device=H.device)
            x = Q[i][:, :, p.m0 - r:] * s[i][:, None, p.m0 - r:] ** -0.5
            C = x.mH @ H[i] @ x
            ev[at[:, None], np.arange(r)] = torch.linalg.eigvalsh(0.5 * (C + C.mH)).cpu().numpy()
    return np.sort(np.concatenate([ev[times == 1].ravel(), np.repeat(ev[times == 2].ravel(), 2)]))


def _generators(p):
    """The blocks T_d (cell k + d, cell k) of a chain's interior, d = -D .. D."""
    (s1, a1, y1), (s2, a2, y2) = _transverse(p)
    reach = math.sqrt(math.log(1.0 / p.eps_support) / float(np.min(p.exps)))
    D = math.ceil((2.0 * reach + p.h) / p.b0)
    n = int(reach / p.h) + p.n0 * 2
    rho = np.arange(-n - D * p.n0, n + D * p.n0)
    g = _functions(p, 0, rho, range(-D, D + 1))
    w = _weights(p)[:, None, None]
    F = torch.einsum("ti,tmn->imn", _potential(p, 0, rho % p.n0).flatten(0, 1), w * y1 * y2)
    Hs, Ss = [], []
    for d in range(2 * D + 1):
        s0, a0 = _mass_stiff(p, 0, g[:, d], g[:, D], False)
        Ss.append(s0 * s1 * s2)
        Hs.append(0.5 * (a0 * s1 * s2 + s0 * a1 * s2 + s0 * s1 * a2) - torch.einsum("im,imn,in->mn", g[:, d], F, g[:, D]))
    return torch.stack(Hs).cpu().numpy(), torch.stack(Ss).cpu().numpy()


def exact(case, seed):
    call = case["call"]
    if call == "product":
        A, B = _operands(case, seed)
        return B @ A.T
    ps = _problems(case, seed)
    if call == "matvec":
        H, S = _chain_matrix(ps[0], "HS"[case["which"]])
        M = H if case["which"] == 0 else S
        return _vectors(case, seed, ps[0].Nb) @ (0.5 * (M + M.T))
    if call == "assemble":
        H, S = _generators(ps[0])
        return {"H": H, "S": S, "EH": None, "ES": None, "cells": None}
    if any(p.Nb > 6000 and (p.is_box or p.defects) for p in ps):
        return None   # a dense generalized eigenproblem of that order takes too long
    ev = [_chain_lowest(p) if p.is_box or p.defects else _spectrum(p) for p in ps]
    return {"evals": np.concatenate(ev), "blocks": None}
