"""Measured workloads: the work that a program built on this library has it do.

A program that optimises or measures an infinite PEPS builds the site's double
layer, runs directional corner-transfer-matrix moves until the environment has
converged, and contracts block-sparse tensors with it.  The cases below are
those calls: single contractions of every size and arithmetic, a batch of
independent ones, a permutation, the SVD projector alone, directional and full
moves on the double layer, a move on the single-layer site, and the SU(2)
corner and move.  Sizes are those of the library's own configurations (bond
dimensions 3..8, environment bonds 12..256, SU(2) bonds up to 150 states) and
odd ones between them.

``exact`` recomputes the results densely in 64 bits with torch and numpy only.
"""
import functools
import itertools
import math
from fractions import Fraction

import numpy as np
import torch

from paper_1808_10804_gb300 import bst
from paper_1808_10804_gb300.ctmrg import Network

DEV = "cuda:0"
ROLES = ("C1", "C2", "C3", "C4", "T1", "T2", "T3", "T4")
RENEWED = {0: ("C1", "T4", "C4"), 1: ("C1", "T1", "C2"), 2: ("C2", "T2", "C3"), 3: ("C3", "T3", "C4"), 4: ROLES}
STREAM = {n: i for i, n in enumerate(("A", "R", "C1", "C2", "C3", "C4", "T1", "T2", "T3", "T4", "B", "X"))}


# ---- the cases ----------------------------------------------------------------

def listed():
    return [
        # the first contraction of a small move: latency and launches decide
        {"name": "edge_d4_fp64", "kind": "contract", "op": "edge", "group": "u1", "D": 4, "chi": 16, "prec": "fp64"},
        # the contraction that dominates an ordinary move, in the default mixed arithmetic
        {"name": "corner_d6_ozaki", "kind": "contract", "op": "corner", "group": "u1", "D": 6, "chi": 72,
         "prec": "ozaki"},
        # the same with ragged sectors, in plain FP64
        {"name": "corner_odd_fp64", "kind": "contract", "op": "corner", "group": "u1", "D": 5, "chi": 101,
         "prec": "fp64"},
        # joining two enlarged corners (large square sectors), in the cheaper arithmetic
        {"name": "half_d6_bf16x3", "kind": "contract", "op": "half", "group": "u1", "D": 6, "chi": 72,
         "prec": "bf16x3"},
        # many independent corner contractions of mixed sizes in one call
        {"name": "batch64_ozaki", "kind": "batch", "count": 64, "prec": "ozaki"},
        # reordering a large intermediate: bound by memory
        {"name": "permute_d8", "kind": "permute", "group": "u1", "D": 8, "chi": 256, "perm": "2031"},
        # the truncation step by itself, on the half systems of an ordinary move
        {"name": "projector_d6_ozaki", "kind": "projector", "D": 6, "chi": 72, "prec": "ozaki"},
        # a small move in FP64: every sector is decomposed directly
        {"name": "left_d4_fp64", "kind": "move", "D": 4, "chi": 16, "dir": 0, "prec": "fp64"},
        # the benchmark step: double layer and full move
        {"name": "full_d6_ozaki", "kind": "move", "D": 6, "chi": 72, "dir": 4, "prec": "ozaki"},
        # a large three-spin site: the double layer is never formed, wide sectors
        {"name": "single_d8_ozaki", "kind": "single", "D": 8, "chi": 192, "dir": 0, "prec": "ozaki"},
        # the non-abelian corner: pair products and recoupling
        {"name": "su2_corner_ozaki", "kind": "su2", "op": "corner", "size": "large", "prec": "ozaki"},
        # the non-abelian move
        {"name": "su2_left_ozaki", "kind": "su2", "op": "left", "size": "large", "prec": "ozaki"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("contract", "contract", "contract", "batch", "permute", "projector", "move", "move",
                       "single", "su2"))
    prec = rng.choice(("fp64", "ozaki", "ozaki", "bf16x3"))
    if kind == "contract":
        c = {"kind": kind, "op": rng.choice(("edge", "corner", "half")), "group": rng.choice(("u1", "u1", "u1", "z2")),
             "D": rng.randint(3, 8), "chi": _log_int(rng, 12, 256), "prec": prec}
        # the plain FP64 path runs near 1 TFLOP/s: keep a call within the large move's time
        while work(c)["flops"] > (8e10 if prec == "fp64" else 5e11):
            c["chi"] = max(12, int(c["chi"] * 0.8))
        return c
    if kind == "batch":
        return {"kind": kind, "count": _log_int(rng, 4, 16 if prec == "fp64" else 64), "prec": prec}
    if kind == "permute":
        perm = list("0123")
        while perm == list("0123"):
            rng.shuffle(perm)
        return {"kind": kind, "group": rng.choice(("u1", "z2")), "D": rng.randint(3, 8),
                "chi": _log_int(rng, 16, 256), "perm": "".join(perm)}
    if kind == "projector":
        return {"kind": kind, "D": rng.randint(4, 6), "chi": _log_int(rng, 16, 96),
                "prec": rng.choice(("fp64", "ozaki"))}
    if kind == "move":
        D, prec = rng.randint(3, 6), rng.choice(("fp64", "ozaki", "ozaki"))
        return {"kind": kind, "D": D, "chi": _log_int(rng, 12, 20 * D - 30),
                "dir": rng.randint(0, 3 if prec == "fp64" and D > 4 else 4), "prec": prec}
    if kind == "single":
        return {"kind": kind, "D": rng.randint(4, 7), "chi": _log_int(rng, 24, 128), "dir": rng.randint(0, 3),
                "prec": "ozaki"}
    return {"kind": "su2", "op": rng.choice(("corner", "left")), "size": rng.choice(("small", "medium", "middle")),
            "prec": rng.choice(("fp64", "ozaki"))}


# ---- legs -----------------------------------------------------------------------

def _bond(chi):
    """Environment bond: chi states over the even charges -Q..Q with Gaussian
    weights (sigma = Q/2), symmetric, rounded by largest remainder."""
    Q = 2 if chi < 8 else 4 if chi < 32 else 6 if chi < 160 else 8
    qs = list(range(-Q, Q + 1, 2))
    w = np.exp(-np.array(qs) ** 2 / (2.0 * (Q / 2.0) ** 2))
    ideal = dict(zip(qs, chi * w / w.sum()))
    n = {q: int(ideal[q]) for q in qs}
    left = chi - sum(n.values())
    for q in sorted((q for q in qs if q >= 0), key=lambda q: (n[q] - ideal[q], q)):
        cost = 2 if q else 1
        if cost <= left:
            n[q] += 1
            n[-q] = n[q]
            left -= cost
    n[0] += left
    return tuple(q for q in qs if n[q]), tuple(n[q] for q in qs if n[q])


def _legs(case):
    """(odd, even, physical, environment bond) as (charges, degeneracies)."""
    D, c = case["D"], max(1, case["D"] // 4)
    phys = ((-3, -1, 1, 3), (1, 3, 3, 1)) if case["kind"] == "single" else ((-1, 1), (1, 1))
    return ((-1, 1), (D // 2, D - D // 2)), ((-2, 0, 2), (c, D - 2 * c, c)), phys, _bond(case["chi"])


def _leg(flow, sectors):
    return bst.Leg(flow, tuple(sectors[0]), tuple(sectors[1]))


def _fused(sectors):
    """Sectors of a ket leg fused with its bra partner (charge ket - bra)."""
    n = {}
    for (q, d), (p, e) in itertools.product(list(zip(*sectors)), repeat=2):
        n[q - p] = n.get(q - p, 0) + d * e
    return tuple(sorted(n)), tuple(n[q] for q in sorted(n))


def _parity(sectors):
    n = {}
    for q, d in zip(*sectors):
        p = (q // 2) % 2  # every charge of a double-layer or environment leg is even
        n[p] = n.get(p, 0) + d
    return tuple(sorted(n)), tuple(n[q] for q in sorted(n))


def _operands(case):
    """Legs of A and B and the contracted pairs of a single contraction."""
    odd, even, _, x = _legs(case)
    kl, ku = _fused(odd), _fused(even)
    if case["group"] == "z2":
        kl, ku, x = _parity(kl), _parity(ku), _parity(x)
    if case["op"] == "edge":      # C1[R, D] . T1[L, D, R]
        return [_leg(-1, x), _leg(-1, x)], [_leg(1, x), _leg(-1, ku), _leg(-1, x)], (0,), (0,)
    if case["op"] == "corner":    # X2[T1.D, T1.R, T4.R, T4.D] . a[L, U, R, D]
        return ([_leg(-1, ku), _leg(-1, x), _leg(-1, kl), _leg(-1, x)],
                [_leg(1, kl), _leg(1, ku), _leg(-1, kl), _leg(-1, ku)], (0, 2), (1, 0))
    # Q1[T1.R, T4.D, a.R, a.D] . Q2[T1.L, T2.D, a.L, a.D]
    return ([_leg(-1, x), _leg(-1, x), _leg(-1, kl), _leg(-1, ku)],
            [_leg(1, x), _leg(-1, x), _leg(1, kl), _leg(-1, ku)], (0, 2), (0, 2))


def _permute_legs(case):
    odd, even, _, x = _legs(case)
    kl, ku = _fused(odd), _fused(even)
    if case["group"] == "z2":
        kl, ku, x = _parity(kl), _parity(ku), _parity(x)
    return [_leg(-1, ku), _leg(-1, x), _leg(-1, kl), _leg(-1, x)]


def _batch_recipe(case, i):
    """Leg lists of batch entry i: D in 4..8, an environment bond of 32..128,
    random splits of D over the charges of the odd and the even leg."""
    rng = np.random.default_rng([20, i])
    D, chi = int(rng.integers(4, 9)), int(rng.choice([32, 64, 96, 128]))
    a, c = int(rng.integers(1, D)), int(rng.integers(1, D - 1))
    odd = ((-1, 1), (a, D - a))
    ev = [(q, n) for q, n in ((-2, (D - c) // 2), (0, c), (2, D - c - (D - c) // 2)) if n]
    kl, ku, x = _fused(odd), _fused(tuple(zip(*ev))), _bond(chi)
    return ([_leg(-1, ku), _leg(-1, x), _leg(-1, kl), _leg(-1, x)],
            [_leg(1, kl), _leg(1, ku), _leg(-1, ku), _leg(-1, ku)])


SU2 = {"large": (((0, 1, 2, 3, 4), (11, 12, 12, 6, 1)), ((0, 1, 2, 3, 4, 5, 6), (11, 12, 10, 7, 5, 3, 2))),
       "middle": (((0, 1, 2, 3, 4), (5, 7, 6, 3, 1)), ((0, 1, 2, 3, 4), (7, 7, 6, 5, 3))),
       "medium": (((0, 1, 2, 3, 4), (3, 4, 4, 2, 1)), ((0, 1, 2, 3), (4, 4, 3, 2))),
       "small": (((0, 1, 2), (2, 2, 1)), ((0, 1, 2), (2, 2, 1)))}


def _su2_legs(case):
    k, x = SU2[case["size"]]
    K, X = (lambda f: _leg(f, k)), (lambda f: _leg(f, x))
    return {"C1": [X(-1), X(-1)], "C2": [X(1), X(-1)], "C3": [X(1), X(1)], "C4": [X(1), X(-1)],
            "T1": [X(1), K(-1), X(-1)], "T2": [X(1), K(1), X(-1)], "T3": [X(1), K(1), X(-1)],
            "T4": [X(1), K(-1), X(-1)], "A": [K(1), K(1), K(-1), K(-1)]}


def _su2_chi(case):
    """States kept by an SU(2) move: the total dimension of the bond."""
    return sum(d * (j + 1) for j, d in zip(*SU2[case["size"]][1]))


def _site_legs(case):
    odd, even, phys, _ = _legs(case)
    return {"A": [_leg(1, phys), _leg(1, odd), _leg(1, even), _leg(-1, even), _leg(-1, even)],
            "R": [_leg(1, even), _leg(-1, odd), _leg(-1, ((-1, 1), (1, 1)))]}


def _env_legs(case):
    odd, even, _, x = _legs(case)
    kl, ku = _fused(odd), _fused(even)
    X = lambda f: _leg(f, x)  # noqa: E731
    return {"C1": [X(-1), X(-1)], "C2": [X(1), X(-1)], "C3": [X(1), X(1)], "C4": [X(1), X(-1)],
            "T1": [X(1), _leg(-1, ku), X(-1)], "T2": [X(1), _leg(1, kl), X(-1)],
            "T3": [X(1), _leg(1, ku), X(-1)], "T4": [X(1), _leg(-1, kl), X(-1)],
            "a": [_leg(1, kl), _leg(1, ku), _leg(-1, kl), _leg(-1, ku)]}


# ---- inputs and passes -------------------------------------------------------------

_CTX = None


def _context():
    """A program keeps one context for all its tensors."""
    global _CTX
    if _CTX is None:
        _CTX = bst.Context(0)
    return _CTX


def _values(seed, name, n, extra=0):
    """N(0, 1) draws of one tensor, in its storage order."""
    g = torch.Generator(device=DEV).manual_seed((int(seed) * 1009 + STREAM[name]) * 4099 + extra)
    return torch.randn(max(n, 1), dtype=torch.float64, device=DEV, generator=g)[:n]


def _network(case, seed):
    legs = _site_legs(case)
    spec = {r: [{"flow": l.flow, "charges": l.charges, "degs": l.degs} for l in legs[r]] for r in legs}
    return Network(_context(), spec, _legs(case)[3], case["chi"], lambda n, k: _values(seed, n, k).cpu().numpy(),
                   device=DEV, single_layer=case["kind"] == "single")


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    if kind == "contract":
        la, lb, pa, pb = _operands(case)
        A, B = ctx.layout(la, case["group"]), ctx.layout(lb, case["group"])
        return {"case": case, "args": (A, _values(seed, "A", A.nnz), B, _values(seed, "B", B.nnz), pa, pb)}
    if kind == "batch":
        pairs = [_batch_recipe(case, i) for i in range(case["count"])]
        As, Bs = [ctx.layout(p[0]) for p in pairs], [ctx.layout(p[1]) for p in pairs]
        Cs = [ctx.contract_layout(A, B, (0, 2), (1, 0)) for A, B in zip(As, Bs)]
        out = torch.zeros(sum(C.nnz for C in Cs), dtype=torch.float64, device=DEV)
        return {"case": case, "out": out, "Cs": Cs, "cs": list(torch.split(out, [C.nnz for C in Cs])),
                "args": (As, [_values(seed, "A", A.nnz, i) for i, A in enumerate(As)],
                         Bs, [_values(seed, "B", B.nnz, i) for i, B in enumerate(Bs)], (0, 2), (1, 0))}
    if kind == "permute":
        L = ctx.layout(_permute_legs(case), case["group"])
        return {"case": case, "args": (L, _values(seed, "X", L.nnz), tuple(int(p) for p in case["perm"]))}
    if kind == "projector":
        return {"case": case, "args": _half_systems(ctx, _network(case, seed)), "cap": _cut_cap(case)}
    if kind in ("move", "single"):
        return {"case": case, "net": _network(case, seed)}
    legs = _su2_legs(case)
    L = {r: ctx.layout(legs[r], "su2") for r in legs}
    d = {r: _values(seed, r, L[r].nnz) for r in legs}
    if case["op"] == "corner":
        return {"case": case, "L": L, "d": d}
    env = bst.Env(ctx, {r: L[r] for r in ROLES}, {r: d[r] for r in ROLES},
                  {r: _env_cap(case, r, L[r].nnz) for r in ROLES})
    return {"case": case, "L": L, "d": d, "env": env, "start": {r: env.buf[r].clone() for r in ROLES}}


def _cut_cap(case):
    """Room for P or Pt whatever sectors the kept states fall into."""
    return _env_legs(case)["C1"][0].dim * _env_legs(case)["a"][1].dim * case["chi"]


def _env_cap(case, r, nnz):
    """Elements of the buffer of environment tensor r: its renewed form fits
    whatever sectors the kept states fall into."""
    if case["kind"] == "su2":
        return max(nnz, _su2_chi(case) ** 2 * (sum(SU2[case["size"]][0][1]) if r[0] == "T" else 1))
    site = _env_legs(case)[r][1].dim if r[0] == "T" else 1
    return max(nnz, case["chi"] ** 2 * site)


def _padded(x, n):
    """x in a buffer of n elements, zeros after it: which sectors the kept
    states fall into, and so the length of x, differs between inputs."""
    return torch.nn.functional.pad(x, (0, n - x.numel()))


def _half_systems(ctx, net):
    """Top and bottom half of the network, from the public contractions."""
    L, t = dict(net.env.L, a=net.aL), {r: net.env.data(r) for r in ROLES}
    t["a"] = net.a
    T = {r: (L[r], t[r]) for r in L}
    con = lambda a, b, i, j: ctx.contract(*a, *b, i, j)  # noqa: E731
    q1 = con(con(con(T["C1"], T["T1"], (0,), (0,)), T["T4"], (0,), (0,)), T["a"], (0, 2), (1, 0))
    q2 = con(con(con(T["T1"], T["C2"], (2,), (0,)), T["T2"], (2,), (0,)), T["a"], (1, 2), (1, 2))
    q4 = con(con(con(T["T4"], T["C4"], (2,), (0,)), T["T3"], (2,), (0,)), T["a"], (1, 2), (0, 3))
    q3 = con(con(con(T["T2"], T["C3"], (2,), (0,)), T["T3"], (2,), (2,)), T["a"], (1, 3), (2, 3))
    return con(q1, q2, (0, 2), (0, 2)) + con(q4, q3, (1, 3), (1, 2))


def run(state):
    ctx, case = _context(), state["case"]
    kind = case["kind"]
    if kind == "contract":
        return ctx.contract(*state["args"], prec=case["prec"])[1]
    if kind == "batch":
        ctx.contract_batched(*state["args"], prec=case["prec"], Cls=state["Cs"], cs=state["cs"])
        return state["out"]
    if kind == "permute":
        return ctx.permute(*state["args"])[1]
    if kind == "projector":
        _, p, _, pt, sv, _ = ctx.svd_projector(*state["args"], 2, case["chi"], prec=case["prec"])
        return {"p": _padded(p, state["cap"]), "pt": _padded(pt, state["cap"]), "sv": np.array(sv)}
    if kind in ("move", "single"):
        net = state["net"]
        net.reset()
        net.step(case["prec"], direction=case["dir"])
        return {r: net.env.buf[r] for r in RENEWED[case["dir"]]}
    L, d = state["L"], state["d"]
    if case["op"] == "corner":
        con = lambda a, b, i, j: ctx.contract(*a, L[b], d[b], i, j, prec=case["prec"])  # noqa: E731
        return con(con(con((L["C1"], d["C1"]), "T1", (0,), (0,)), "T4", (0,), (0,)), "A", (0, 2), (1, 0))[1]
    env = state["env"]
    for r in ROLES:
        env.buf[r].copy_(state["start"][r])
    env.L = {r: L[r] for r in ROLES}
    ctx.ctm_move(env, L["A"], d["A"], bst.LEFT, _su2_chi(case), prec=case["prec"])
    return {r: env.buf[r] for r in RENEWED[0]}


# ---- the work of a pass ---------------------------------------------------------------

def _hist(legs, sign, mod):
    h = {0: 1}
    for l in legs:
        n = {}
        for (t, m), (q, d) in itertools.product(h.items(), zip(l.charges, l.degs)):
            s = t + sign * l.flow * q
            s = s % mod if mod else s
            n[s] = n.get(s, 0) + m * d
        h = n
    return h


def _nnz(legs, mod=0):
    return _hist(legs, 1, mod).get(0, 0)


def _product(A, B, la, lb, mod=0):
    """(flops, output legs) of a contraction: 2 M K N per charge through the cut."""
    a = [l for i, l in enumerate(A) if i not in la]
    b = [l for i, l in enumerate(B) if i not in lb]
    m, k, n = _hist(a, -1, mod), _hist([A[i] for i in la], 1, mod), _hist(b, 1, mod)
    return 2.0 * sum(m.get(q, 0) * k[q] * n.get(q, 0) for q in k), a + b


def _move_work(legs, chi, single=None):
    """Flops of the contractions of one LEFT move; the truncated decomposition
    counted as one application of N and N^T to the kept states.  `single`: the
    legs of a single-layer site, absorbed ket and bra in turn."""
    total = 0.0

    def con(A, B, i, j):
        nonlocal total
        f, out = _product(A, B, i, j)
        total += f
        return out

    def absorb(X, i, j):
        """X times the site over X's legs i and the site's legs j."""
        if single is None:
            return con(X, legs["a"], i, j)
        keep = [l for p, l in enumerate(X) if p not in i]
        ket, bra = [single[q + 1].dual() for q in j], [single[q + 1] for q in j]
        half = con(keep + ket + bra, single, tuple(range(len(keep), len(keep) + len(j))), tuple(q + 1 for q in j))
        nb = len(keep)
        conj = [l.dual() for l in single]
        con(half, conj, tuple(range(nb, nb + len(j))) + (nb + len(j),), tuple(q + 1 for q in j) + (0,))
        return keep + [l for q, l in enumerate(legs["a"]) if q not in j]

    C, T = (lambda i: legs["C%d" % i]), (lambda i: legs["T%d" % i])
    x1 = con(C(1), T(1), (0,), (0,))
    q1 = absorb(con(x1, T(4), (0,), (0,)), (0, 2), (1, 0))
    q2 = absorb(con(con(T(1), C(2), (2,), (0,)), T(2), (2,), (0,)), (1, 2), (1, 2))
    y = con(C(4), T(3), (1,), (0,))
    q4 = absorb(con(con(T(4), C(4), (2,), (0,)), T(3), (2,), (0,)), (1, 2), (0, 3))
    q3 = absorb(con(con(T(2), C(3), (2,), (0,)), T(3), (2,), (2,)), (1, 3), (2, 3))
    rt, rb = con(q1, q2, (0, 2), (0, 2)), con(q4, q3, (1, 3), (1, 2))
    con(rt, rb, (0, 1), (0, 1))
    cut, new = _hist(rt[2:], -1, 0), _leg(-1, _bond(chi))
    total += sum(4.0 * n * n * dict(zip(*_bond(chi))).get(q, 0) for q, n in cut.items())
    p, pt = con(rb, [l.dual() for l in rb[2:]] + [new], (2, 3), (0, 1)), [new.dual()] + rt[:2]
    total += _product(rt, [l.dual() for l in rt[2:]] + [new], (2, 3), (0, 1))[0]
    con(x1, p, (0, 1), (0, 1))
    con(absorb(con(pt, T(4), (1,), (0,)), (1, 2), (1, 0)), p, (1, 3), (0, 1))
    con(pt, y, (1, 2), (0, 1))
    return total


def work(case):
    kind = case["kind"]
    if kind == "contract":
        a, b, la, lb = _operands(case)
        mod = 2 if case["group"] == "z2" else 0
        f, c = _product(a, b, la, lb, mod)
        return {"bytes": 8.0 * (_nnz(a, mod) + _nnz(b, mod) + _nnz(c, mod)), "flops": f}
    if kind == "batch":
        by = fl = 0.0
        for i in range(case["count"]):
            a, b = _batch_recipe(case, i)
            f, c = _product(a, b, (0, 2), (1, 0))
            by, fl = by + 8.0 * (_nnz(a) + _nnz(b) + _nnz(c)), fl + f
        return {"bytes": by, "flops": fl}
    if kind == "permute":
        return {"bytes": 16.0 * _nnz(_permute_legs(case), 2 if case["group"] == "z2" else 0), "flops": 0.0}
    if kind == "su2":
        return _su2_work(case)
    legs = _env_legs(case)
    x, k = legs["C1"][0], legs["a"]
    if kind == "projector":
        n = _hist([x, k[3]], 1, 0)
        kept = dict(zip(*_bond(case["chi"])))
        f = sum(2.0 * m ** 3 + 8.0 * m * m * kept.get(q, 0) for q, m in n.items())
        return {"bytes": 8.0 * (2 * sum(m * m for m in n.values()) + 2 * sum(m * kept.get(q, 0) for q, m in n.items())),
                "flops": f}
    site = _site_legs(case)
    single = None
    if kind == "single":  # A' = A with the remover's leg absorbed, (p, s) fused
        q = {}
        for (a, d), s in itertools.product(zip(site["A"][0].charges, site["A"][0].degs), (1, -1)):
            q[a - s] = q.get(a - s, 0) + d
        P = _leg(1, (tuple(sorted(q)), tuple(q[c] for c in sorted(q))))
        single = [P, site["A"][1], site["A"][2], site["A"][1].dual(), site["A"][4]]
    ins = sum(_nnz(legs[r]) for r in ROLES) + _nnz(site["A"]) + _nnz(site["R"])
    moves = 4 if case["dir"] == 4 else 1
    return {"bytes": 8.0 * (ins + sum(_nnz(legs[r]) for r in RENEWED[case["dir"]])),
            "flops": moves * _move_work(legs, case["chi"], single)}


# ---- SU(2): blocks, trees and coefficients ------------------------------------------------

def _couplings(spins):
    """Left-to-right coupling trees of doubled spins: (intermediates, J)."""
    if not spins:
        return [((), 0)]
    paths = [(spins[0],)]
    for s in spins[1:]:
        paths = [p + (k,) for p in paths for k in range(abs(p[-1] - s), p[-1] + s + 1, 2)]
    return [(p[1:-1], p[-1]) for p in paths]


@functools.lru_cache(maxsize=None)
def _trees(spins, flows):
    ins = _couplings([s for s, f in zip(spins, flows) if f == 1])
    outs = _couplings([s for s, f in zip(spins, flows) if f == -1])
    return tuple(sorted(a + (J,) + b for a, J in ins for b, K in outs if J == K))


def _su2_blocks(legs):
    """(sector tuple, spins, tree, shape) of every block in storage order."""
    flows = tuple(l.flow for l in legs)
    for s in itertools.product(*[range(len(l.charges)) for l in legs]):
        spins = tuple(l.charges[i] for l, i in zip(legs, s))
        shape = tuple(l.degs[i] for l, i in zip(legs, s))
        for t in _trees(spins, flows):
            yield s, spins, t, shape


def _su2_work(case):
    legs = _su2_legs(case)
    total = 0.0

    def nnz(L):
        return sum(math.prod(b[3]) for b in _su2_blocks(L))

    def con(A, B, la, lb):
        """Every pair of blocks that agree on the contracted sectors, once."""
        nonlocal total
        rows, cols, k = {}, {}, {}
        for s, _, _, sh in _su2_blocks(A):
            key = tuple(s[i] for i in la)
            k[key] = math.prod(sh[i] for i in la)
            rows[key] = rows.get(key, 0) + math.prod(sh) // k[key]
        for s, _, _, sh in _su2_blocks(B):
            key = tuple(s[i] for i in lb)
            cols[key] = cols.get(key, 0) + math.prod(sh) // math.prod(sh[i] for i in lb)
        total += sum(2.0 * m * k[q] * cols.get(q, 0) for q, m in rows.items())
        return [l for i, l in enumerate(A) if i not in la] + [l for i, l in enumerate(B) if i not in lb]

    x1 = con(legs["C1"], legs["T1"], (0,), (0,))
    q1 = con(con(x1, legs["T4"], (0,), (0,)), legs["A"], (0, 2), (1, 0))
    if case["op"] == "corner":
        return {"bytes": 8.0 * (sum(nnz(legs[r]) for r in ("C1", "T1", "T4", "A")) + nnz(q1)), "flops": total}
    corner = total
    n = {}  # reduced dimension of the cut per coupled spin
    for (i, d), (j, e) in itertools.product(zip(*SU2[case["size"]][1]), zip(*SU2[case["size"]][0])):
        for J in range(abs(i - j), i + j + 1, 2):
            n[J] = n.get(J, 0) + d * e
    kept = dict(zip(*SU2[case["size"]][1]))
    half = sum(2.0 * m ** 3 for m in n.values())
    total = 4 * corner + 3 * half + sum(8.0 * m * m * kept.get(J, 0) for J, m in n.items())
    return {"bytes": 8.0 * (sum(nnz(legs[r]) for r in legs) + sum(nnz(legs[r]) for r in RENEWED[0])), "flops": total}


@functools.lru_cache(maxsize=None)
def _cg(a, ma, b, mb, J, M):
    """Clebsch-Gordan coefficient, all arguments doubled (Racah's sum, exact
    rationals under one square root)."""
    if ma + mb != M or not abs(a - b) <= J <= a + b or abs(M) > J:
        return 0.0
    f = lambda n: math.factorial(n // 2)  # noqa: E731
    pre = Fraction((J + 1) * f(J + a - b) * f(J - a + b) * f(a + b - J), f(a + b + J + 2))
    pre *= f(J + M) * f(J - M) * f(a - ma) * f(a + ma) * f(b - mb) * f(b + mb)
    s = Fraction(0)
    for k in range(0, a + b + J + 1):
        den = (2 * k, a + b - J - 2 * k, a - ma - 2 * k, b + mb - 2 * k, J - b + ma + 2 * k, J - a - mb + 2 * k)
        if min(den) >= 0:
            s += Fraction((-1) ** k, math.prod(f(d) for d in den))
    return math.copysign(math.sqrt(float(s * s * pre)), s) if s else 0.0


@functools.lru_cache(maxsize=None)
def _couple(a, b, J):
    """<a m_a b m_b | J M> with every m descending."""
    w = np.zeros((a + 1, b + 1, J + 1))
    for i, j in itertools.product(range(a + 1), range(b + 1)):
        M = a - 2 * i + b - 2 * j
        if abs(M) <= J:
            w[i, j, (J - M) // 2] = _cg(a, a - 2 * i, b, b - 2 * j, J, M)
    return w


def _tree_tensor(spins, inter, J):
    if not spins:
        return np.ones(1)
    v, k = np.eye(spins[0] + 1), spins[0]
    for s, nxt in zip(spins[1:], list(inter) + [J]):
        v, k = np.tensordot(v, _couple(k, s, nxt), (v.ndim - 1, 0)), nxt
    return v


@functools.lru_cache(maxsize=None)
def _cgc(spins, flows, tree):
    """CGC tensor of a block over the magnetic numbers of its legs."""
    ins, outs = ([i for i, f in enumerate(flows) if f == s] for s in (1, -1))
    ni = max(len(ins) - 2, 0)
    u = _tree_tensor([spins[i] for i in ins], tree[:ni], tree[ni])
    v = _tree_tensor([spins[i] for i in outs], tree[ni + 1:], tree[ni])
    c = np.tensordot(u, v, (u.ndim - 1, v.ndim - 1))
    return torch.from_numpy(np.ascontiguousarray(np.transpose(c, np.argsort(ins + outs)))).to(DEV)


# ---- dense reference ------------------------------------------------------------------------

class _Dense:
    """A dense tensor with its legs; `charge(i)` is the conserved charge of
    every index of leg i (U(1): 2 S_z, Z2: parity, SU(2): 2m)."""

    def __init__(self, legs, t, group="u1"):
        self.legs, self.t, self.group = list(legs), t, group

    def charge(self, i):
        l = self.legs[i]
        if self.group == "su2":
            q = [j - 2 * m for j, d in zip(l.charges, l.degs) for _ in range(d) for m in range(j + 1)]
        else:
            q = [c for c, d in zip(l.charges, l.degs) for _ in range(d)]
        return torch.tensor(q, dtype=torch.int64, device=DEV)

    def key(self, which, sign):
        """Charge carried by the composite index of legs `which`."""
        tot = torch.zeros(1, dtype=torch.int64, device=DEV)
        for i in which:
            tot = (tot[:, None] + sign * self.legs[i].flow * self.charge(i)[None, :]).reshape(-1)
        return tot % 2 if self.group == "z2" else tot

    def permute(self, perm):
        return _Dense([self.legs[p] for p in perm], self.t.permute(*perm).contiguous(), self.group)


def _offsets(leg, group):
    return np.concatenate([[0], np.cumsum([d * (q + 1 if group == "su2" else 1) for q, d in zip(leg.charges, leg.degs)])])


def _block_list(legs, group):
    if group == "su2":
        yield from _su2_blocks(legs)
        return
    for s in itertools.product(*[range(len(l.charges)) for l in legs]):
        q = sum(l.flow * l.charges[i] for l, i in zip(legs, s))
        if (q % 2 if group == "z2" else q) == 0:
            yield s, None, None, tuple(l.degs[i] for l, i in zip(legs, s))


def _dense(legs, flat, group="u1"):
    offs = [_offsets(l, group) for l in legs]
    out = torch.zeros([int(o[-1]) for o in offs], dtype=torch.float64, device=DEV)
    flows, pos, R = tuple(l.flow for l in legs), 0, len(legs)
    for s, spins, tree, shape in _block_list(legs, group):
        b = flat[pos:pos + math.prod(shape)].reshape(shape)
        pos += math.prod(shape)
        at = tuple(slice(int(o[i]), int(o[i + 1])) for o, i in zip(offs, s))
        if group == "su2":
            c = _cgc(spins, flows, tree)
            inter = [x for d, m in zip(shape, c.shape) for x in (d, m)]
            b = (b.reshape([x for d in shape for x in (d, 1)]) * c.reshape([x for m in c.shape for x in (1, m)])).expand(inter)
            b = b.reshape([d * m for d, m in zip(shape, c.shape)])
        out[at] += b
    return _Dense(legs, out, group)


def _flat(T):
    """Stored values of a dense symmetric tensor, in storage order."""
    offs = [_offsets(l, T.group) for l in T.legs]
    flows, R, out = tuple(l.flow for l in T.legs), len(T.legs), []
    for s, spins, tree, shape in _block_list(T.legs, T.group):
        b = T.t[tuple(slice(int(o[i]), int(o[i + 1])) for o, i in zip(offs, s))]
        if T.group == "su2":
            c = _cgc(spins, flows, tree)
            b = b.reshape([x for d, m in zip(shape, c.shape) for x in (d, m)])
            b = torch.tensordot(b, c, (list(range(1, 2 * R, 2)), list(range(R)))) / c.square().sum()
        out.append(b.reshape(-1))
    return torch.cat(out) if out else torch.zeros(0, dtype=torch.float64, device=DEV)


def _contract(A, B, la, lb):
    """Dense contraction, one product per conserved charge."""
    oa = [i for i in range(len(A.legs)) if i not in la]
    ob = [i for i in range(len(B.legs)) if i not in lb]
    a = A.t.permute(*oa, *la).reshape(math.prod(A.t.shape[i] for i in oa), -1)
    b = B.t.permute(*lb, *ob).reshape(a.shape[1], -1)
    ka, kk, kb = A.key(oa, -1), A.key(la, 1), B.key(ob, 1)
    out = torch.zeros(a.shape[0], b.shape[1], dtype=torch.float64, device=DEV)
    for q in torch.unique(kk).tolist():
        i, k, j = ((x == q).nonzero()[:, 0] for x in (ka, kk, kb))
        if len(i) and len(j):
            out[i[:, None], j[None, :]] = a[i[:, None], k[None, :]] @ b[k[:, None], j[None, :]]
    shape = [A.t.shape[i] for i in oa] + [B.t.shape[j] for j in ob]
    return _Dense([A.legs[i] for i in oa] + [B.legs[j] for j in ob], out.reshape(shape), A.group)


def _fuse_order(leg):
    """Composite (ket, bra) index of a fused leg in its storage order."""
    q = np.repeat(leg.charges, leg.degs)
    sec = np.repeat(np.arange(len(leg.degs)), leg.degs)
    i, j = (x.reshape(-1) for x in np.indices((leg.dim, leg.dim)))
    return torch.from_numpy(np.lexsort((j, i, sec[j], sec[i], q[i] - q[j]))).to(DEV)


def _double_layer(case, seed):
    """a[L, U, R, D] = sum_{p,s} (A R)(A R)*, ket and bra legs fused."""
    legs = _site_legs(case)
    A, R = (_dense(legs[r], _values(seed, r, _nnz(legs[r]))) for r in ("A", "R"))
    B = torch.einsum("plurd,rms->pslumd", A.t, R.t)
    B = B.reshape((-1,) + B.shape[2:])
    t = torch.einsum("plumd,pabce->laubmcde", B, B)
    out = [legs["A"][1], legs["A"][2], legs["A"][1], legs["A"][4]]
    t = t.reshape([l.dim ** 2 for l in out])
    for ax, l in enumerate(out):
        t = t.index_select(ax, _fuse_order(l))
    return _Dense(_env_legs(case)["a"], t)


def _dense_network(case, seed):
    if case["kind"] == "su2":
        legs = _su2_legs(case)
        net = {r: _dense(legs[r], _values(seed, r, _su2_nnz(legs[r])), "su2") for r in legs}
        net["a"] = net.pop("A")
        return net
    legs = _env_legs(case)
    net = {r: _dense(legs[r], _values(seed, r, _nnz(legs[r]))) for r in ROLES}
    net["a"] = _double_layer(case, seed)
    return net


def _su2_nnz(legs):
    return sum(math.prod(b[3]) for b in _su2_blocks(legs))


DIRS = {"C1": "RD", "C2": "LD", "C3": "UL", "C4": "UR", "T1": "LDR", "T2": "ULD", "T3": "LUR", "T4": "URD", "a": "LURD"}
TURN = {"U": "L", "L": "D", "D": "R", "R": "U"}


def _turn(net, times):
    """The network after counter-clockwise quarter turns."""
    for _ in range(times % 4):
        new = {}
        for r, T in net.items():
            to = r if r == "a" else "%s%d" % (r[0], (int(r[1]) + 2) % 4 + 1)
            now = [TURN[d] for d in DIRS[r]]
            new[to] = T.permute([now.index(d) for d in DIRS[to]])
        net = new
    return net


def _halves(net):
    con = lambda a, b, i, j: _contract(a, b, i, j)  # noqa: E731
    n = net
    x1 = con(n["C1"], n["T1"], (0,), (0,))
    q1 = con(con(x1, n["T4"], (0,), (0,)), n["a"], (0, 2), (1, 0))
    q2 = con(con(con(n["T1"], n["C2"], (2,), (0,)), n["T2"], (2,), (0,)), n["a"], (1, 2), (1, 2))
    rt = con(q1, q2, (0, 2), (0, 2))
    del q1, q2
    q4 = con(con(con(n["T4"], n["C4"], (2,), (0,)), n["T3"], (2,), (0,)), n["a"], (1, 2), (0, 3))
    q3 = con(con(con(n["T2"], n["C3"], (2,), (0,)), n["T3"], (2,), (2,)), n["a"], (1, 3), (2, 3))
    return x1, rt, con(q4, q3, (1, 3), (1, 2))


def _svd(m):
    """Singular triplets with the largest entry of each left vector positive."""
    scale = np.abs(m).max() or 1.0
    try:
        U, S, Vt = np.linalg.svd(m / scale, full_matrices=False)
    except np.linalg.LinAlgError:  # the divide-and-conquer driver gave up: QR iteration instead
        U, S, Vt = (x.cpu().numpy() for x in torch.linalg.svd(torch.from_numpy(m / scale).to(DEV), full_matrices=False,
                                                             driver="gesvd" if DEV != "cpu" else None))
    S = S * scale
    sign = np.sign(U[np.argmax(np.abs(U), axis=0), np.arange(U.shape[1])])
    return U * sign, S, Vt.T * sign


def _projectors(rt, rb, chi, flow):
    """P, Pt and the kept singular values (new leg: ascending charge)."""
    N = _contract(rt, rb, (0, 1), (0, 1))
    n = rt.t.shape[2] * rt.t.shape[3]
    m = N.t.reshape(n, -1)
    kr, kc = N.key((0, 1), -1), N.key((2, 3), 1)
    sec, cand = {}, []
    for q in sorted(set(kr.tolist()) & set(kc.tolist())):
        i, j = (kr == q).nonzero()[:, 0], (kc == q).nonzero()[:, 0]
        sec[q] = (i, j) + _svd(m[i[:, None], j[None, :]].cpu().numpy())
        cand += [(-s, abs(q), flow * q, c) for c, s in enumerate(sec[q][3])]
    cand = [c for c in sorted(cand)[:chi] if -c[0] > -1e-14 * min(cand)[0]]
    kept = {}
    for c in cand:
        kept[c[2]] = kept.get(c[2], 0) + 1
    new = _leg(flow, (tuple(sorted(kept)), tuple(kept[q] for q in sorted(kept))))
    P, Pt, sv = [], [], []
    for q in new.charges:
        i, j, U, S, V = sec[flow * q]
        k = kept[q]
        s = 1.0 / np.sqrt(S[:k])
        V, U = (torch.from_numpy(x[:, :k] * s).to(DEV) for x in (V, U))
        P.append(rb.t.reshape(-1, n)[:, j] @ V)
        Pt.append(U.T @ rt.t.reshape(-1, n)[:, i].T)
        sv += S[:k].tolist()
    P = torch.cat(P, 1).reshape(rb.t.shape[:2] + (-1,))
    Pt = torch.cat(Pt, 0).reshape((-1,) + rt.t.shape[:2])
    return (_Dense(rb.legs[:2] + [new], P), _Dense([new.dual()] + rt.legs[:2], Pt), np.array(sv))


def _su2_projectors(rt, rb, chi):
    """The same per coupled spin on reduced matrices; whole multiplets are
    kept by descending value while the total dimension fits chi."""
    N = _contract(rt, rb, (0, 1), (0, 1))
    flat, pos, mats = _flat(N).cpu().numpy(), 0, {}
    place = [{}, {}]
    for s, spins, tree, sh in _su2_blocks(N.legs):
        for side, (key, size) in enumerate(((s[:2], sh[0] * sh[1]), (s[2:], sh[2] * sh[3]))):
            place[side].setdefault(tree[0], {})[key] = size
    start = [{J: dict(zip(sorted(p), np.concatenate([[0], np.cumsum([p[k] for k in sorted(p)])]))) for J, p in side.items()}
             for side in place]
    for J in place[0]:
        mats[J] = np.zeros((sum(place[0][J].values()), sum(place[1][J].values())))
    for s, spins, tree, sh in _su2_blocks(N.legs):
        n, J = math.prod(sh), tree[0]
        r, c = int(start[0][J][s[:2]]), int(start[1][J][s[2:]])
        mats[J][r:r + sh[0] * sh[1], c:c + sh[2] * sh[3]] = flat[pos:pos + n].reshape(sh[0] * sh[1], -1)
        pos += n
    sec = {J: _svd(m) for J, m in mats.items()}
    kept, dim = {J: 0 for J in sec}, 0
    top = max(S[0] for _, S, _ in sec.values())
    for s, J, j in sorted((-s, J, j) for J, (_, S, _) in sec.items() for j, s in enumerate(S)):
        if -s > 1e-14 * top and kept[J] == j and dim + J + 1 <= chi:
            kept[J] += 1
            dim += J + 1
    Js = [J for J in sorted(kept) if kept[J]]
    new = _leg(1, (tuple(Js), tuple(kept[J] for J in Js)))
    vl, ul = [l.dual() for l in N.legs[2:]] + [new], [new.dual()] + [l.dual() for l in N.legs[:2]]
    v, u = [], []
    for s, spins, _, sh in _su2_blocks(vl):
        U, S, V = sec[spins[2]]
        r = int(start[1][spins[2]][s[:2]])
        v.append((V[r:r + sh[0] * sh[1], :sh[2]] / np.sqrt(S[:sh[2]])).reshape(-1))
    for s, spins, _, sh in _su2_blocks(ul):
        U, S, V = sec[spins[0]]
        r = int(start[0][spins[0]][s[1:]])
        u.append((U[r:r + sh[1] * sh[2], :sh[0]] / np.sqrt(S[:sh[0]])).T.reshape(-1))
    up = lambda x: torch.from_numpy(np.concatenate(x)).to(DEV)  # noqa: E731
    P = _contract(rb, _dense(vl, up(v), "su2"), (2, 3), (0, 1))
    return P, _contract(_dense(ul, up(u), "su2"), rt, (1, 2), (2, 3))


def _left(net, chi):
    x1, rt, rb = _halves(net)
    if rt.group == "su2":
        P, Pt = _su2_projectors(rt, rb, chi)
    else:
        P, Pt, _ = _projectors(rt, rb, chi, net["C1"].legs[1].flow)
    del rt, rb
    w = _contract(_contract(Pt, net["T4"], (1,), (0,)), net["a"], (1, 2), (1, 0))   # [new, T4.D, a.R, a.D]
    new = {"C1": _contract(x1, P, (0, 1), (0, 1)), "T4": _contract(w, P, (1, 3), (0, 1)),
           "C4": _contract(Pt, _contract(net["C4"], net["T3"], (1,), (0,)), (1, 2), (0, 1))}
    out = dict(net)
    for r, T in new.items():
        out[r] = _Dense(T.legs, T.t / T.t.norm(), T.group)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "contract":
        a, b, la, lb = _operands(case)
        g = case["group"]
        A, B = (_dense(l, _values(seed, n, _nnz(l, 2 if g == "z2" else 0)), g) for l, n in ((a, "A"), (b, "B")))
        return _flat(_contract(A, B, la, lb))
    if kind == "batch":
        out = []
        for i in range(case["count"]):
            a, b = _batch_recipe(case, i)
            A, B = _dense(a, _values(seed, "A", _nnz(a), i)), _dense(b, _values(seed, "B", _nnz(b), i))
            out.append(_flat(_contract(A, B, (0, 2), (1, 0))))
        return torch.cat(out)
    if kind == "permute":
        legs, g = _permute_legs(case), case["group"]
        T = _dense(legs, _values(seed, "X", _nnz(legs, 2 if g == "z2" else 0)), g)
        return _flat(T.permute([int(p) for p in case["perm"]]))
    if kind == "su2" and case["op"] == "corner":
        n = _dense_network(case, seed)
        x2 = _contract(_contract(n["C1"], n["T1"], (0,), (0,)), n["T4"], (0,), (0,))
        return _flat(_contract(x2, n["a"], (0, 2), (1, 0)))
    if kind != "su2" and max(_hist([_env_legs(case)["C1"][0], _env_legs(case)["a"][3]], 1, 0).values()) > 1500:
        return None  # dense decompositions of that size take minutes
    net = _dense_network(case, seed)
    if kind == "projector":
        _, rt, rb = _halves(net)
        P, Pt, sv = _projectors(rt, rb, case["chi"], -1)
        return {"p": _padded(_flat(P), _cut_cap(case)), "pt": _padded(_flat(Pt), _cut_cap(case)), "sv": sv}
    chi = _su2_chi(case) if kind == "su2" else case["chi"]
    which = case.get("dir", 0)
    buf = {}
    for r in ROLES:  # the environment's buffers: a renewed tensor overwrites the front of its own
        x = _flat(net[r])
        buf[r] = _padded(x, _env_cap(case, r, x.numel()))
    for d in ((0, 2, 1, 3) if which == 4 else (which,)):
        net = _turn(_left(_turn(net, d), chi), -d)
        for r in RENEWED[d]:
            x = _flat(net[r])
            buf[r][:x.numel()] = x
    return {r: buf[r] for r in RENEWED[which]}
