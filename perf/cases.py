"""Workloads of the CS decomposition library that its speed is measured on.

Every case goes through the public entry points of
`paper_1804_09002_gb300.binding` and `.autograd`, on the engine that a user
chooses with `Context.set_tensor_cores` (the FP64 pipe is the default).

Inputs have a prescribed CS structure A1 = U1 C V^*, A2 = U2 S V^* with Haar
U1, U2, V, as in `paper_1804_09002_gb300.inputs`, built on the GPU.  The
angles are one per cell of an even grid on [0, pi/2], uniform inside the
middle half of their cell: like the angles of a random orthonormal matrix
they repel each other, so the factors are functions of the input (up to the
column signs, which `set_sign_convention` fixes) and can be compared.
"""
import math

import numpy as np
import torch

from paper_1804_09002_gb300 import autograd as G
from paper_1804_09002_gb300 import binding as B

HALF_PI = math.pi / 2
DEV = "cuda:0"


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest decomposition of the benchmark, where latency is all
        dict(name="csd_64", kind="csd", n=64, cplx=False, rank=64, tc=False),
        # the default engine (FP64 pipe) at an ordinary odd size
        dict(name="csd_fp64_201", kind="csd", n=201, cplx=False, rank=201, tc=False),
        # tensor-core products: ordinary, benchmark-sized and the largest
        # that stays within two seconds (not multiples of any tile)
        dict(name="csd_tc_500", kind="csd", n=500, cplx=False, rank=500, tc=True),
        dict(name="csd_tc_1024", kind="csd", n=1024, cplx=False, rank=1024, tc=True),
        dict(name="csd_tc_3000", kind="csd", n=3000, cplx=False, rank=3000, tc=True),
        # complex partial isometry with 3/4 of full rank (the shape of the
        # complex benchmark configuration at a quarter of its side)
        dict(name="csd_c128_rankdef_512", kind="csd", n=512, cplx=True, rank=384, tc=True),
        # blocks of different heights
        dict(name="csd_rect_900_700_450", kind="rect", m1=900, m2=700, n=450, cplx=False, tc=True),
        # the two building blocks called on their own
        dict(name="polar_2048", kind="polar", n=2048, cplx=False, tc=True),
        dict(name="heig_1500", kind="heig", n=1500, cplx=False, tc=True),
        # one training step: decomposition, a loss on angles and factors,
        # gradients of both blocks
        dict(name="grad_200", kind="grad", n=200),
        # many small decompositions of ragged sizes in one planned launch
        dict(name="batch_48", kind="batch", count=48, lo=16, hi=256, pick=5),
        # one FP64-accurate product C <- alpha A^T B + beta C
        dict(name="gemm_3001_2500_4096", kind="gemm", m=3001, n=2500, k=4096, opA=1, opB=0, engine=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["csd", "csd", "csd", "rankdef", "rect", "polar", "heig", "grad", "batch", "gemm"])
    if kind == "csd":
        tc = rng.random() < 0.7
        n = _log_int(rng, 200, 2800) if tc else _log_int(rng, 40, 400)
        return dict(kind="csd", n=n, cplx=False, rank=n, tc=tc)
    if kind == "rankdef":
        cplx = rng.random() < 0.5
        n = _log_int(rng, 64, 600 if cplx else 1200)
        return dict(kind="csd", n=n, cplx=cplx, rank=max(1, int(n * rng.uniform(0.5, 0.95))), tc=n >= 200)
    if kind == "rect":
        n = _log_int(rng, 64, 800)
        m1, m2 = (n + int(n * rng.uniform(0.0, 1.5)) for _ in range(2))
        return dict(kind="rect", m1=m1, m2=m2, n=n, cplx=False, tc=n >= 200)
    if kind in ("polar", "heig"):
        cplx = rng.random() < 0.25
        n = _log_int(rng, 64, 700 if cplx else 2500)
        return dict(kind=kind, n=n, cplx=cplx, tc=n >= 200)
    if kind == "grad":
        return dict(kind="grad", n=_log_int(rng, 32, 320))
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 8, 64), lo=16, hi=rng.randint(64, 256), pick=rng.randrange(1 << 20))
    return dict(kind="gemm", m=_log_int(rng, 100, 4096), n=_log_int(rng, 100, 4096), k=_log_int(rng, 100, 4096),
                opA=rng.randrange(2), opB=rng.randrange(2), engine=1)


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, m, n, cplx=False):
    return torch.randn(m, n, dtype=torch.complex128 if cplx else torch.float64, device=DEV, generator=g)


def _haar(g, m, n, cplx=False):
    """m x n, orthonormal columns, Haar distributed (phases of diag(R) moved into Q)."""
    q, r = torch.linalg.qr(_randn(g, m, n, cplx))
    return q * torch.sgn(torch.diagonal(r))[None, :]


def _grid(g, n, lo=0.0, hi=HALF_PI):
    u = torch.rand(n, dtype=torch.float64, device=DEV, generator=g)
    return lo + (torch.arange(n, dtype=torch.float64, device=DEV) + 0.25 + 0.5 * u) * ((hi - lo) / n)


def _col(x):
    """The same matrix stored column by column, as the library's arrays are."""
    return x.t().contiguous().t()


def _signed(V, *Us):
    """V's columns scaled so that their largest entry is real and positive, and the Us with them."""
    top = V.gather(0, V.abs().argmax(0, keepdim=True))
    ph = top.conj() / top.abs()
    return [V * ph] + [u * ph for u in Us]


def _csd_parts(case, seed):
    """(U1, U2, V, theta of the kept columns) with ascending theta."""
    g = _gen(seed)
    n, cplx = case["n"], case.get("cplx", False)
    m1, m2, k = case.get("m1", n), case.get("m2", n), case.get("rank", n)
    U1, U2, V = _haar(g, m1, n, cplx), _haar(g, m2, n, cplx), _haar(g, n, n, cplx)
    return U1[:, :k], U2[:, :k], V[:, :k], _grid(g, k)


def _csd_inputs(case, seed):
    U1, U2, V, th = _csd_parts(case, seed)
    return _col((U1 * torch.cos(th)) @ V.mH), _col((U2 * torch.sin(th)) @ V.mH)


def _polar_parts(case, seed):
    """Singular values spread evenly in their logarithm over [1e-4, 1]."""
    g = _gen(seed)
    n, cplx = case["n"], case["cplx"]
    s = torch.exp(_grid(g, n, math.log(1e-4), 0.0))
    return _haar(g, n, n, cplx), s, _haar(g, n, n, cplx)


def _heig_input(case, seed):
    X = _randn(_gen(seed), case["n"], case["n"], case["cplx"])
    return _col(X + X.mH)


def _batch_sizes(case):
    return np.random.default_rng(case["pick"]).integers(case["lo"], case["hi"] + 1, size=case["count"]).tolist()


def _batch_inputs(case, seed):
    return [_csd_inputs(dict(n=n), seed * 1000 + i) for i, n in enumerate(_batch_sizes(case))]


def _gemm_inputs(case, seed):
    g = _gen(seed)
    m, n, k = case["m"], case["n"], case["k"]
    A = _col(_randn(g, k, m) if case["opA"] else _randn(g, m, k))
    Bm = _col(_randn(g, n, k) if case["opB"] else _randn(g, k, n))
    return A, Bm, _col(_randn(g, m, n))


def _grad_inputs(case, seed):
    """The blocks and the loss's constants: weights of the angles, targets of U1 and V1."""
    A1, A2 = _csd_inputs(case, seed)
    g = _gen(seed + 1)
    n = case["n"]
    w = torch.randn(n, dtype=torch.float64, device=DEV, generator=g)
    return A1, A2, w, _haar(g, n, n), _haar(g, n, n)


# ---------------------------------------------------------------- what a program keeps
_contexts = {}
_plans = {}


def _context(tc):
    """One context per engine for the life of the process, with canonical column signs."""
    if tc not in _contexts:
        c = B.Context(0)
        c.set_tensor_cores(tc)
        c.set_sign_convention(1)
        _contexts[tc] = c
    return _contexts[tc]


def _plan(case, pairs):
    """One batch plan per set of sizes; its first run tunes and captures it."""
    key = tuple(_batch_sizes(case))
    if key not in _plans:
        if len(_plans) >= 2:
            _plans.pop(next(iter(_plans))).close()
        p = B.Batch(_context(False), list(key))
        p.load([a for a, _ in pairs], [b for _, b in pairs])
        p.run()
        _plans[key] = p
    return _plans[key]


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("csd", "rect"):
        st["ctx"], st["A"] = _context(case["tc"]), _csd_inputs(case, seed)
    elif kind == "polar":
        U, s, V = _polar_parts(case, seed)
        st["ctx"], st["A"] = _context(case["tc"]), _col((U * s) @ V.mH)
    elif kind == "heig":
        st["ctx"], st["A"] = _context(case["tc"]), _heig_input(case, seed)
    elif kind == "grad":
        st["A"] = _grad_inputs(case, seed)
    elif kind == "batch":
        pairs = _batch_inputs(case, seed)
        st["plan"] = _plan(case, pairs)
        st["A"] = [a for a, _ in pairs], [b for _, b in pairs]
    else:
        st["ctx"], st["A"] = _context(True), _gemm_inputs(case, seed)
    return st


def _loss(U1, U2, V1, th, w, T1, T2):
    return (w * th).sum() + ((U1 - T1) ** 2).sum() + (U2 * T2).sum() + ((V1 - T2) ** 2).sum()


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "csd":
        R = st["ctx"].csd_polar(*st["A"])
        r = R["rank"]  # columns and angles beyond the rank are not part of the result
        return dict(U1=R["U1"][:, :r], U2=R["U2"][:, :r], V1=R["V1"][:, :r], theta=R["theta"][:r], rank=r)
    if kind == "rect":
        # the blocks' own Q factors leave the column signs of U1 and U2 to V1's
        R = st["ctx"].csd_polar_rect(*st["A"])
        return dict(U1=R["U1"], U2=R["U2"], V1=R["V1"], theta=R["theta"], rank=R["rank"])
    if kind == "polar":
        W, H, _ = st["ctx"].polar(st["A"])
        return dict(W=W, H=H)
    if kind == "heig":
        # eigenvectors are defined up to a sign or phase; this program fixes it
        lam, V, _ = st["ctx"].heig(st["A"])
        return dict(lam=lam, V=_signed(V)[0])
    if kind == "grad":
        A1, A2, w, T1, T2 = st["A"]
        A1, A2 = A1.detach().requires_grad_(True), A2.detach().requires_grad_(True)
        U1, U2, V1, th = G.csd(A1, A2)
        loss = _loss(U1, U2, V1, th, w, T1, T2)
        g1, g2 = torch.autograd.grad(loss, (A1, A2))
        return dict(loss=loss.detach(), theta=th.detach(), V1=V1.detach(), gA1=g1, gA2=g2)
    if kind == "batch":
        p = st["plan"]
        p.load(*st["A"])
        status = p.run()
        # the planned launch leaves column signs open; this program fixes
        # them, all instances of the packed buffers at once
        out = dict(status=status.copy(), theta=p.theta)
        out["U1"], out["U2"], out["V1"] = _batch_signed(p)
        return out
    A, Bm, C = st["A"]
    # the product writes into its C: a program that keeps its C passes a copy
    out = st["ctx"].gemm(A, Bm, _col(C.clone()), alpha=-0.75, beta=0.5, opA=case["opA"], opB=case["opB"],
                         engine=case["engine"])
    return dict(C=out)


def _batch_index(p):
    """Column number of every entry of the packed buffers (kept with the plan)."""
    if not hasattr(p, "column_of"):
        n = torch.tensor(p.sizes, device=DEV)
        p.column_of = torch.repeat_interleave(torch.arange(int(n.sum()), device=DEV), torch.repeat_interleave(n, n))
    return p.column_of


def _batch_signed(p):
    col = _batch_index(p)
    cols = int(p.toff[-1])
    big = torch.zeros(cols, dtype=torch.float64, device=DEV).scatter_reduce_(0, col, p.V1.abs(), "amax")
    at = torch.where(p.V1.abs() == big[col], torch.sign(p.V1), 0.0)
    sign = torch.zeros(cols, dtype=torch.float64, device=DEV).scatter_reduce_(0, col, at, "sum")
    ph = torch.where(sign < 0, -1.0, 1.0).to(torch.float64)[col]
    return p.U1 * ph, p.U2 * ph, p.V1 * ph


# ---------------------------------------------------------------- cost and exact values
def work(case):
    """Inputs read once and outputs written once; flops of the classical dense
    algorithms (20 n^3 polar by an SVD, 9 n^3 symmetric eigenproblem, 8 n^3 for
    H_i and U_i), four times as many for complex data."""
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + 2 * m * n), "flops": 2.0 * m * n * k}
    if kind == "batch":
        s = _batch_sizes(case)
        return {"bytes": 8.0 * 5 * sum(v * v for v in s), "flops": 57.0 * sum(v ** 3 for v in s)}
    n, z = case["n"], 2.0 if case.get("cplx") else 1.0
    nn, n3 = 8.0 * z * n * n, z * z * float(n) ** 3
    if kind == "polar":
        return {"bytes": 3 * nn, "flops": 22 * n3}
    if kind == "heig":
        return {"bytes": 2 * nn + 8 * n, "flops": 9 * n3}
    if kind == "grad":
        return {"bytes": 12 * nn, "flops": 57 * n3 + 16 * n3}
    if kind == "rect":
        m = case["m1"] + case["m2"]
        return {"bytes": 8.0 * z * (2 * m * n + n * n), "flops": 57 * n3 + 6.0 * z * z * m * n * n}
    return {"bytes": 5 * nn, "flops": 57 * n3}


def _csd_exact(case, seed):
    """The factors that the inputs were made from, columns in the library's order and signs."""
    U1, U2, V, th = _csd_parts(case, seed)
    V, U1, U2 = _signed(V, U1, U2)
    return U1, U2, V, th


def exact(case, seed):
    kind = case["kind"]
    if kind in ("csd", "rect"):
        U1, U2, V, th = _csd_exact(case, seed)
        return dict(U1=U1, U2=U2, V1=V, theta=th, rank=None)
    if kind == "polar":
        U, s, V = _polar_parts(case, seed)
        return dict(W=U @ V.mH, H=(V * s) @ V.mH)
    if kind == "heig":
        lam, V = np.linalg.eigh(_heig_input(case, seed).cpu().numpy())
        return dict(lam=lam, V=_signed(torch.from_numpy(V))[0])
    if kind == "grad":
        return _grad_exact(*(x.cpu() for x in _grad_inputs(case, seed)))
    if kind == "batch":
        parts = [_csd_exact(dict(n=n), seed * 1000 + i) for i, n in enumerate(_batch_sizes(case))]
        flat = [torch.cat([q[j].t().reshape(-1) for q in parts]) for j in range(3)]
        return dict(status=None, theta=torch.cat([q[3] for q in parts]), U1=flat[0], U2=flat[1], V1=flat[2])
    A, Bm, C = _gemm_inputs(case, seed)
    return dict(C=-0.75 * ((A.t() if case["opA"] else A) @ (Bm.t() if case["opB"] else Bm)) + 0.5 * C)


def _grad_exact(A1, A2, w, T1, T2):
    """The same loss by differentiating the decomposition's definition: polar
    factors from singular value decompositions, V1 from the symmetric B."""
    A1, A2 = A1.detach().requires_grad_(True), A2.detach().requires_grad_(True)

    def polar(A):
        u, _, vh = torch.linalg.svd(A)
        W = u @ vh
        P = W.t() @ A
        return W, (P + P.t()) / 2

    W1, H1 = polar(A1)
    W2, H2 = polar(A2)
    V = torch.linalg.eigh(H2 - H1)[1]
    top = V.gather(0, V.abs().argmax(0, keepdim=True)).detach()
    V = V * torch.sign(top)
    c, s = ((V * (H @ V)).sum(0) for H in (H1, H2))
    th = torch.atan2(s, c)
    loss = _loss(W1 @ V, W2 @ V, V, th, w, T1, T2)
    g1, g2 = torch.autograd.grad(loss, (A1, A2))
    return dict(loss=loss.detach(), theta=th.detach(), V1=V.detach(), gA1=g1, gA2=g2)
