"""Performance cases: the calls that programs built on this library spend their time in.

The library's users contract abelian-symmetric tensors of iPEPS / MPS codes. The cases
follow such a program from its smallest calls (an MPS bond, a Z2 site) over the ordinary
ones (one request of a served U(1) run, a CTM step at D = 12, the enlarged corner as a
network, a batch of served requests) to the largest environment contraction (D = 20,
chi = 400), in FP64 and in split precision at the tolerances in use, real and complex,
together with the calls around the contractions: conjugation, swap gates, fuse and
unfuse, norms and traces.

Every tensor is fully populated (every block that charge conservation allows) with
N(0, 1) elements. Structures depend on the case alone, data on the seed alone. The
``exact`` values are per-sector dense products (and plain block copies) in 64 bits.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2405_12196_gb300 import ytn

DEV = "cuda:0"


# --------------------------------------------------------------------------- cases

def listed():
    return [
        # one bond of a U(1) MPS sweep: five sectors of a few elements, all latency
        {"name": "mps_u1_fp64", "op": "mps", "sizes": "3,6,8,6,3", "prec": "fp64"},
        # the double layer of a Z2 iPEPS site (D = 8): conj, A . conj(A), fuse
        {"name": "site_z2_double_layer", "op": "double_layer", "dh0": 4, "dh1": 4, "prec": "fp64"},
        # a Z2 CTM edge (chi = 64) times the double layer: two wide sectors with K = 32,
        # an output of gigabytes
        {"name": "edge_z2_split", "op": "edge", "dh0": 4, "dh1": 4, "ch0": 32, "ch1": 32, "prec": "split",
         "rtol": 1e-10},
        # a served U(1) run at small D in the reference precision; ragged sector sizes
        {"name": "run_u1_d6_fp64", "op": "x2a", "sym": "u1", "D": 6, "chi": 37, "layout": 11, "prec": "fp64"},
        # a served U(1) run at ordinary D, split precision
        {"name": "run_u1_d10_split", "op": "x2a", "sym": "u1", "D": 10, "chi": 63, "layout": 12, "prec": "split",
         "rtol": 1e-10},
        # complex tensors (real-time evolution, magnetic fields) at a tighter tolerance
        {"name": "run_u1_d8_c128", "op": "x2a", "sym": "u1", "D": 8, "chi": 45, "layout": 13, "prec": "split",
         "rtol": 2e-11, "dtype": "c128"},
        # the dominant contraction of a U(1)xU(1) CTM step, D = 12, chi = 144: 7225 blocks
        {"name": "ctm_u1u1_d12_split", "op": "x2a", "sym": "u1u1", "D": 12, "layout": 0, "prec": "split",
         "rtol": 1e-10},
        # the enlarged corner of the same step as one network call
        {"name": "corner_u1u1_d12", "op": "corner", "D": 12, "layout": 0, "prec": "split", "rtol": 1e-10},
        # the largest environment contraction, D = 20, chi = 400: 1e5 blocks, 225 sectors
        {"name": "env_u1u1_d20_split", "op": "x2a", "sym": "u1u1", "D": 20, "layout": 0, "prec": "split",
         "rtol": 1e-10},
        # around the contractions: a fermionic swap gate, then the matrix form for a
        # decomposition and back; many small blocks
        {"name": "swap_fuse_unfuse_d16", "op": "moves", "sym": "u1u1", "D": 16, "layout": 0},
        # scalars of an environment: the overlap of two tensors and a partial trace
        {"name": "overlap_trace_d16", "op": "scalars", "sym": "u1u1", "D": 16, "layout": 0},
        # requests of independent U(1) runs through the serving loop
        {"name": "serving_u1_16", "op": "serving", "requests": 16, "layout": 5, "prec": "split", "rtol": 1e-10},
    ]


def draw(rng):
    op = rng.choice(["mps", "double_layer", "edge", "x2a_u1", "x2a_u1", "x2a_u1", "x2a_u1u1", "x2a_u1u1", "corner",
                     "moves", "scalars", "serving"])
    layout = rng.randrange(1, 1 << 20)
    split = {"prec": "split", "rtol": rng.choice([1e-10, 1e-10, 1e-10, 2e-11, 1e-8])}
    logint = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if op == "mps":
        sizes = ",".join(str(logint(2, 300)) for _ in range(5))
        return {"op": "mps", "sizes": sizes, **rng.choice([{"prec": "fp64"}, split])}
    if op == "double_layer":
        return {"op": op, "dh0": rng.randint(1, 4), "dh1": rng.randint(1, 4), "prec": "fp64"}
    if op == "edge":
        return {"op": op, "dh0": rng.randint(1, 4), "dh1": rng.randint(1, 4), "ch0": logint(5, 32),
                "ch1": logint(5, 32), **split}
    if op == "x2a_u1":
        c128 = rng.random() < 0.25
        fp64 = not c128 and rng.random() < 0.4
        D = rng.randint(3, 6) if fp64 else rng.randint(4, 9 if c128 else 12)
        case = {"op": "x2a", "sym": "u1", "D": D, "chi": rng.randint(max(9, 4 * D), 8 * D), "layout": layout,
                **({"prec": "fp64"} if fp64 else split)}
        if c128:
            case["dtype"] = "c128"
        return case
    if op == "x2a_u1u1":
        return {"op": "x2a", "sym": "u1u1", "D": rng.randint(9, 17), "layout": layout, **split}
    if op == "corner":
        return {"op": op, "D": rng.randint(9, 13), "layout": layout, **split}
    if op in ("moves", "scalars"):
        return {"op": op, "sym": "u1u1", "D": rng.randint(10, 17), "layout": layout}
    return {"op": op, "requests": rng.randint(6, 24), "layout": layout, **split}


# ---------------------------------------------------------------------- structures

class Leg:
    """A leg: signature, charges [n][nsym] (ascending) and their dimensions."""

    def __init__(self, s, t, D):
        order = sorted(range(len(t)), key=lambda i: tuple(t[i]))
        self.s = s
        self.t = np.array([tuple(t[i]) for i in order], np.int64)
        self.D = np.array([int(D[i]) for i in order], np.int64)

    def sig(self, s):
        return Leg(s, [tuple(q) for q in self.t], list(self.D))


def _reduce(x, mods):
    m = np.array(mods, np.int64)
    return np.where(m > 0, np.mod(x, np.where(m > 0, m, 1)), x)


def _record(mods, legs, n=None, dtype="f64"):
    """The tensor record of every allowed block on ``legs``, in canonical order."""
    nsym = len(mods)
    n = np.zeros(nsym, np.int64) if n is None else np.array(n, np.int64)
    grids = np.meshgrid(*[np.arange(len(l.D)) for l in legs[:-1]], indexing="ij")
    idx = [g.ravel() for g in grids]
    tot = sum(l.s * l.t[i] for l, i in zip(legs[:-1], idx))
    last = legs[-1]
    need = _reduce(last.s * (n[None, :] - tot), mods)
    where = {tuple(q): i for i, q in enumerate(last.t.tolist())}
    li = np.array([where.get(tuple(q), -1) for q in need.tolist()], np.int64)
    keep = li >= 0
    idx = [i[keep] for i in idx] + [li[keep]]
    t = np.stack([l.t[i] for l, i in zip(legs, idx)], axis=1)
    D = np.stack([l.D[i] for l, i in zip(legs, idx)], axis=1)
    order = np.lexsort(t.reshape(len(t), -1).T[::-1])
    rec = {"mods": tuple(mods), "sig": tuple(l.s for l in legs), "n": tuple(int(x) for x in n),
           "t": t[order].astype(np.int32), "D": D[order]}
    if dtype == "c128":
        rec["dtype"] = "c128"
    return rec


def _size(rec):
    return int(np.prod(rec["D"], axis=1).sum())


def _offsets(rec):
    sizes = np.prod(rec["D"], axis=1)
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _composition(total, parts, rng):
    cuts = sorted(rng.choice(np.arange(1, total), size=parts - 1, replace=False).tolist())
    bounds = [0] + cuts + [total]
    return [bounds[i + 1] - bounds[i] for i in range(parts)]


def _double_leg(v, mods):
    """The D^2 leg of a double layer: charges ket minus bra."""
    acc = {}
    for q1, d1 in zip(v.t, v.D):
        for q2, d2 in zip(v.t, v.D):
            q = tuple(int(x) for x in _reduce(q1 - q2, mods))
            acc[q] = acc.get(q, 0) + int(d1 * d2)
    return Leg(1, list(acc), list(acc.values()))


def _gaussian_leg(D, layout):
    """A U(1)xU(1) virtual leg of dimension D, sector sizes a discrete Gaussian: nine
    candidate charges below D = 14, 25 from there on."""
    r, width = (1, 1.0) if D < 14 else (2, 1.5)
    cand = [(a, b) for a in range(-r, r + 1) for b in range(-r, r + 1)]
    w = np.array([math.exp(-(a * a + b * b) / (2 * width * width)) for a, b in cand])
    least = 1 if r == 1 else 0
    extra = np.random.default_rng(layout).multinomial(D - least * len(cand), w / w.sum())
    got = [(q, least + int(e)) for q, e in zip(cand, extra) if least + e > 0]
    return Leg(1, [q for q, _ in got], [d for _, d in got])


def _x2_legs(sym, D, chi, layout):
    """(mods, chi leg, double-layer leg)."""
    if sym == "u1u1":
        dl = _double_leg(_gaussian_leg(D, layout), (0, 0))
        return (0, 0), dl, dl
    rng = np.random.default_rng(layout)
    nv = 3 if D < 6 else 5
    v = Leg(1, [(q,) for q in range(-(nv // 2), nv // 2 + 1)], _composition(D, nv, rng))
    c = Leg(1, [(q,) for q in range(-4, 5)], _composition(chi, 9, rng))
    return (0,), c, _double_leg(v, (0,))


def _x2_a(sym, D, chi, layout, dtype="f64"):
    mods, c, dl = _x2_legs(sym, D, chi, layout)
    X2 = _record(mods, [c, dl.sig(1), dl.sig(-1), c.sig(-1)], dtype=dtype)
    a = _record(mods, [dl.sig(-1), dl.sig(1), dl.sig(1), dl.sig(-1)], dtype=dtype)
    return X2, a


def _z2_leg(d0, d1, s=1):
    return Leg(s, [(0,), (1,)], [d0, d1])


def _serving_runs(layout, count):
    """(X2, a) records of the requests: D of each run uniform in {4, 6, 8, 10, 12}, chi
    in [4 D, 8 D]."""
    rng = np.random.default_rng(layout)
    runs = []
    for _ in range(max(1, count // 2)):
        D = int(rng.choice([4, 6, 8, 10, 12]))
        runs.append((D, int(rng.integers(4 * D, 8 * D + 1)), int(rng.integers(1 << 20))))
    return [_x2_a("u1", *runs[int(rng.integers(len(runs)))]) for _ in range(count)]


def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k != "name"))


def _inputs(case):
    """The case's input records and its contraction, structure only."""
    return _inputs_cached(_key(case))


@functools.lru_cache(maxsize=24)
def _inputs_cached(key):
    c = dict(key)
    op, dtype = c["op"], c.get("dtype", "f64")
    if op == "mps":
        v = Leg(1, [(-2,), (-1,), (0,), (1,), (2,)], [int(x) for x in c["sizes"].split(",")])
        p = Leg(1, [(-1,), (1,)], [1, 1])
        A = _record((0,), [v, p, v.sig(-1)])
        return {"recs": [A, A], "axa": (2,), "axb": (0,)}
    if op == "double_layer":
        v, p = _z2_leg(c["dh0"], c["dh1"]), _z2_leg(1, 1)
        return {"recs": [_record((2,), [v.sig(-1), v, v, v.sig(-1), p])]}
    if op == "edge":
        dl = _double_leg(_z2_leg(c["dh0"], c["dh1"]), (2,))
        chi = _z2_leg(c["ch0"], c["ch1"])
        T = _record((2,), [chi, dl.sig(1), chi.sig(-1)])
        a = _record((2,), [dl.sig(-1), dl.sig(1), dl.sig(1), dl.sig(-1)])
        return {"recs": [T, a], "axa": (1,), "axb": (0,)}
    if op == "x2a":
        X2, a = _x2_a(c["sym"], c["D"], c.get("chi"), c["layout"], dtype)
        return {"recs": [X2, a], "axa": (1, 2), "axb": (0, 1)}
    if op == "corner":
        mods, chi, dl = _x2_legs("u1u1", c["D"], None, c["layout"])
        C = _record(mods, [chi, chi.sig(-1)])
        T = _record(mods, [chi, dl.sig(1), chi.sig(-1)])
        a = _record(mods, [dl.sig(-1), dl.sig(1), dl.sig(1), dl.sig(-1)])
        return {"recs": [C, T, T, a], "labels": [[1, 2], [2, 3, -1], [-2, 4, 1], [3, -3, -4, 4]]}
    if op in ("moves", "scalars"):
        X2, _ = _x2_a(c["sym"], c["D"], None, c["layout"])
        return {"recs": [X2] if op == "moves" else [X2, X2]}
    reqs = _serving_runs(c["layout"], c["requests"])
    return {"recs": [r for pair in reqs for r in pair], "axa": (1, 2), "axb": (0, 1)}


# ------------------------------------------------------------------- state and run

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = ytn.ytn_ctx_create(0)
    return _ctx


def _data(case, seed):
    """One N(0, 1) buffer per input tensor, from the seed alone."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    cw = 2 if case.get("dtype") == "c128" else 1
    return [torch.randn(_size(r) * cw, dtype=torch.float64, device=DEV, generator=gen)
            for r in _inputs(case)["recs"]]


def _empty(rec):
    cw = 2 if rec.get("dtype") == "c128" else 1
    return torch.empty(max(int(rec["size"]) * cw, 1), dtype=torch.float64, device=DEV)


def _workspace(nbytes):
    return torch.empty(max(int(nbytes), 256), dtype=torch.uint8, device=DEV)


def _precision(case):
    if case.get("prec") == "split":
        return {"prec": ytn.YTN_SPLIT_BF16, "rtol": case["rtol"]}
    return {"prec": ytn.YTN_FP64, "rtol": 0.0}


DOUBLE_LAYER_GROUPS = [(0, 4), (1, 5), (2, 6), (3, 7)]
MATRIX_GROUPS = [(0, 1), (2, 3)]


def prepare(case, seed):
    ctx, op, pr = _context(), case["op"], _precision(case)
    inp, data = _inputs(case), _data(case, seed)
    recs = inp["recs"]
    st = {"op": op, "data": data, **pr}
    if op in ("mps", "edge", "x2a"):
        plan = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, recs[0], recs[1], inp["axa"], inp["axb"])
        st.update(plan=plan, out=_empty(plan.out), ws=_workspace(ytn.ytn_workspace_size(plan, pr["prec"], pr["rtol"])))
    elif op == "double_layer":
        conj = ytn.ytn_plan(ctx, ytn.YTN_OP_CONJ, recs[0])
        dot = ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, recs[0], conj.out, (4,), (4,))
        fuse = ytn.ytn_plan(ctx, ytn.YTN_OP_FUSE, dot.out, groups=DOUBLE_LAYER_GROUPS)
        st.update(conj=conj, dot=dot, fuse=fuse, outs=[_empty(p.out) for p in (conj, dot, fuse)],
                  ws=_workspace(ytn.ytn_workspace_size(dot, pr["prec"], pr["rtol"])))
    elif op == "corner":
        net = ytn.ytn_ncon_plan(ctx, recs, inp["labels"])
        st.update(net=net, out=_empty(net.out), ws=_workspace(ytn.ytn_ncon_workspace_size(net, pr["prec"], pr["rtol"])))
    elif op == "moves":
        swap = ytn.ytn_plan(ctx, ytn.YTN_OP_SWAP_GATE, recs[0], groups=MATRIX_GROUPS)
        fuse = ytn.ytn_plan(ctx, ytn.YTN_OP_FUSE, swap.out, groups=MATRIX_GROUPS)
        unfuse = ytn.ytn_plan(ctx, ytn.YTN_OP_UNFUSE, fuse.out, axa=(0, 1))
        st.update(swap=swap, fuse=fuse, unfuse=unfuse, outs=[_empty(p.out) for p in (swap, fuse, unfuse)])
    elif op == "scalars":
        dot = ytn.ytn_plan(ctx, ytn.YTN_OP_VDOT, recs[0], recs[1])
        trace = ytn.ytn_plan(ctx, ytn.YTN_OP_TRACE, recs[0], axa=(0,), axb=(3,))
        st.update(dot=dot, trace=trace, outs=[torch.empty(1, dtype=torch.float64, device=DEV), _empty(trace.out)],
                  ws=_workspace(ytn.ytn_workspace_size(dot)))
    elif op == "serving":
        plans = [ytn.ytn_plan(ctx, ytn.YTN_OP_TENSORDOT, recs[i], recs[i + 1], inp["axa"], inp["axb"])
                 for i in range(0, len(recs), 2)]
        need = max(ytn.ytn_workspace_size(p, pr["prec"], pr["rtol"]) for p in plans)
        arena = _workspace(4 * need)
        torch.cuda.synchronize()   # the inputs are read on the server's own streams
        st.update(plans=plans, outs=[_empty(p.out) for p in plans], server=ytn.ytn_server_create(ctx, 8, arena))
    return st


def run(st):
    op, d, stream = st["op"], st["data"], torch.cuda.current_stream()
    if op in ("mps", "edge", "x2a"):
        ytn.ytn_tensordot(st["plan"], d[0], d[1], st["out"], prec=st["prec"], rtol=st["rtol"], workspace=st["ws"],
                          stream=stream)
        return st["out"]
    if op == "double_layer":
        bra, double, fused = st["outs"]
        ytn.ytn_conj(st["conj"], d[0], bra, stream=stream)
        ytn.ytn_tensordot(st["dot"], d[0], bra, double, prec=st["prec"], rtol=st["rtol"], workspace=st["ws"],
                          stream=stream)
        ytn.ytn_fuse(st["fuse"], double, fused, stream=stream)
        return fused
    if op == "corner":
        ytn.ytn_ncon(st["net"], d, st["out"], prec=st["prec"], rtol=st["rtol"], workspace=st["ws"], stream=stream)
        return st["out"]
    if op == "moves":
        gated, matrix, back = st["outs"]
        ytn.ytn_swap_gate(st["swap"], d[0], gated, stream=stream)
        ytn.ytn_fuse(st["fuse"], gated, matrix, stream=stream)
        ytn.ytn_unfuse(st["unfuse"], matrix, back, stream=stream)
        return [gated, matrix, back]
    if op == "scalars":
        overlap, traced = st["outs"]
        ytn.ytn_vdot(st["dot"], d[0], d[1], overlap, workspace=st["ws"], stream=stream)
        ytn.ytn_trace(st["trace"], d[0], traced, stream=stream)
        return [overlap, traced]
    server = st["server"]
    for i, plan in enumerate(st["plans"]):
        server.submit(i, plan, d[2 * i], d[2 * i + 1], st["outs"][i], prec=st["prec"], rtol=st["rtol"])
    server.drain()
    server.poll()
    return st["outs"]


# ----------------------------------------------------------- work and exact values

def _free(rank, axes):
    return [i for i in range(rank) if i not in axes]


def _sectors(A, B, axa, axb):
    """Per charge carried through the contracted legs: A's rows, B's columns and the
    contracted tuples of both with their dimensions, and the blocks of both."""
    out = {}
    for which, (R, con, sign) in enumerate(((A, list(axa), 1), (B, list(axb), -1))):
        t, D = R["t"].astype(np.int64), R["D"]
        free = _free(t.shape[1], con)
        q = _reduce(sum(sign * R["sig"][i] * t[:, i, :] for i in con), R["mods"])
        f, k = t[:, free, :].reshape(len(t), -1), t[:, con, :].reshape(len(t), -1)
        fd, kd = np.prod(D[:, free], axis=1), np.prod(D[:, con], axis=1)
        for b, (qq, ff, kk, m, c) in enumerate(zip(map(tuple, q.tolist()), map(tuple, f.tolist()),
                                                   map(tuple, k.tolist()), fd.tolist(), kd.tolist())):
            s = out.setdefault(qq, ({}, {}, ({}, {}), ([], [])))
            s[which][ff] = m
            s[2][which][kk] = c
            s[3][which].append((b, ff, kk))
    return {q: s for q, s in out.items() if s[3][0] and s[3][1]}


def _running(dims, order):
    off, at = {}, 0
    for x in order:
        off[x] = at
        at += dims[x]
    return off, at


def _dot(A, B, axa, axb, a=None, b=None):
    """(record, buffer, flops) of the contraction; with data, sector by sector as dense
    64-bit products, else the structure alone."""
    axa, axb = list(axa), list(axb)
    fa, fb = _free(A["t"].shape[1], axa), _free(B["t"].shape[1], axb)
    oa, ob, DA, DB = _offsets(A), _offsets(B), A["D"].tolist(), B["D"].tolist()
    blocks, flops = {}, 0.0
    for rows, cols, (xa, xb), (ba, bb) in _sectors(A, B, axa, axb).values():
        common = sorted(set(xa) & set(xb))
        if not common:
            continue
        ro, M = _running(rows, sorted(rows))
        co, N = _running(cols, sorted(cols))
        ko, K = _running(xa, common)
        flops += 2.0 * M * N * K
        P = Q = None
        if a is not None:
            P = torch.zeros(M, K, dtype=a.dtype, device=a.device)
            Q = torch.zeros(K, N, dtype=b.dtype, device=b.device)
        hasa, hasb, shape_r, shape_c = {}, {}, {}, {}
        for i, r, x in ba:
            if x in ko:
                hasa.setdefault(r, set()).add(x)
                shape_r[r] = [DA[i][f] for f in fa]
                if P is not None:
                    P[ro[r]:ro[r] + rows[r], ko[x]:ko[x] + xa[x]] = \
                        a[oa[i]:oa[i + 1]].view(DA[i]).permute(fa + axa).reshape(rows[r], xa[x])
        for i, c, x in bb:
            if x in ko:
                hasb.setdefault(c, set()).add(x)
                shape_c[c] = [DB[i][f] for f in fb]
                if Q is not None:
                    Q[ko[x]:ko[x] + xa[x], co[c]:co[c] + cols[c]] = \
                        b[ob[i]:ob[i + 1]].view(DB[i]).permute(axb + fb).reshape(xa[x], cols[c])
        C = P @ Q if P is not None else None
        full = all(len(x) == len(common) for x in (*hasa.values(), *hasb.values()))
        for r in hasa:
            for c in hasb:
                if full or hasa[r] & hasb[c]:
                    v = None if C is None else C[ro[r]:ro[r] + rows[r], co[c]:co[c] + cols[c]]
                    blocks[r + c] = (v, shape_r[r] + shape_c[c])
    order = sorted(blocks)
    nsym, rank = len(A["mods"]), len(fa) + len(fb)
    rec = {"mods": A["mods"], "sig": tuple(A["sig"][i] for i in fa) + tuple(B["sig"][i] for i in fb),
           "t": np.array(order, np.int32).reshape(len(order), rank, nsym),
           "D": np.array([blocks[k][1] for k in order], np.int64).reshape(len(order), rank)}
    if a is None:
        return rec, None, flops
    off = _offsets(rec)
    out = torch.empty(int(off[-1]), dtype=a.dtype, device=a.device)
    for k, at in zip(order, off.tolist()):
        v = blocks[k][0]
        out[at:at + v.numel()].view(v.shape).copy_(v)
    return rec, out, flops


def _permute(R, axes, r=None):
    t = R["t"][:, axes, :]
    order = np.lexsort(t.reshape(len(t), -1).T[::-1])
    rec = {"mods": R["mods"], "sig": tuple(R["sig"][i] for i in axes), "t": t[order], "D": R["D"][:, axes][order]}
    if r is None:
        return rec, None
    off, D = _offsets(R).tolist(), R["D"].tolist()
    return rec, torch.cat([r[off[i]:off[i + 1]].view(D[i]).permute(axes).reshape(-1) for i in order.tolist()])


def _corner(recs, data=None):
    """The corner network's pairwise contractions: (record, buffer, flops)."""
    C, T, _, a = recs
    dC, dT1, dT2, da = data if data is not None else [None] * 4
    X, x, f0 = _dot(C, T, (0,), (2,), dC, dT2)            # legs 2, -2, 4
    X, x, f1 = _dot(X, T, (0,), (0,), x, dT1)             # legs -2, 4, 3, -1
    X, x, f2 = _dot(X, a, (2, 1), (0, 3), x, da)          # legs -2, -1, -3, -4
    X, x = _permute(X, [1, 0, 2, 3], x)
    return X, x, f0 + f1 + f2


def _fuse(R, groups, r):
    """The buffer of the fused tensor: per fused leg the charge s_g sum_i s_i rho_i with
    the signature s_g of the group's first leg, sub-blocks in the order of their charges."""
    t, D, mods = R["t"].astype(np.int64), R["D"], R["mods"]
    rows, cons, dims, place = [], [], [], []
    for g in groups:
        g = list(g)
        q = _reduce(R["sig"][g[0]] * sum(R["sig"][i] * t[:, i, :] for i in g), mods)
        rows.append(list(map(tuple, q.tolist())))
        cons.append(list(map(tuple, t[:, g, :].reshape(len(t), -1).tolist())))
        dims.append(np.prod(D[:, g], axis=1).tolist())
        at, start = {}, {}
        for qq, ss, dd in sorted(set(zip(rows[-1], cons[-1], dims[-1]))):
            start[(qq, ss)] = at.get(qq, 0)
            at[qq] = at.get(qq, 0) + dd
        place.append((start, at))
    names = sorted(set(zip(*rows)))
    shape = {nm: [place[g][1][nm[g]] for g in range(len(groups))] for nm in names}
    off, total = _running({nm: math.prod(shape[nm]) for nm in names}, names)
    out = torch.zeros(total, dtype=r.dtype, device=r.device)
    view = {nm: out[off[nm]:off[nm] + math.prod(shape[nm])].view(shape[nm]) for nm in names}
    src, axes, DL = _offsets(R).tolist(), [i for g in groups for i in g], D.tolist()
    for b, (nm, cc, dd) in enumerate(zip(zip(*rows), zip(*cons), zip(*dims))):
        at = [place[g][0][(nm[g], cc[g])] for g in range(len(groups))]
        v = r[src[b]:src[b + 1]].view(DL[b]).permute(axes).reshape(dd)
        view[nm][tuple(slice(o, o + n) for o, n in zip(at, dd))] = v
    return out


def _swap(R, groups, r):
    """Blocks where both groups of legs carry an odd parity change sign."""
    odd = [R["t"][:, list(g), :].astype(np.int64).sum(axis=(1, 2)) % 2 for g in groups]
    sign = torch.from_numpy(np.where(odd[0] * odd[1] > 0, -1.0, 1.0)).to(r.device)
    return r * torch.repeat_interleave(sign, torch.from_numpy(np.prod(R["D"], axis=1)).to(r.device))


def _trace(R, r):
    """The sum over equal indices of the first and the last of four legs."""
    off, D, t = _offsets(R).tolist(), R["D"].tolist(), R["t"]
    out = {}
    for i in np.nonzero(np.all(t[:, 0, :] == t[:, 3, :], axis=1))[0].tolist():
        k = tuple(t[i, 1:3, :].reshape(-1).tolist())
        v = torch.einsum("iabi->ab", r[off[i]:off[i + 1]].view(D[i])).reshape(-1)
        out[k] = out[k] + v if k in out else v
    return torch.cat([out[k] for k in sorted(out)])


def _conj(R):
    return {**R, "sig": tuple(-s for s in R["sig"]), "n": tuple(-x for x in R["n"])}


def work(case):
    b, f = _work_cached(_key(case))
    return {"bytes": b, "flops": f}


@functools.lru_cache(maxsize=64)
def _work_cached(key):
    case = dict(key)
    op, inp = case["op"], _inputs(case)
    recs, cw = inp["recs"], 2 if case.get("dtype") == "c128" else 1
    read = 8.0 * cw * sum(_size(r) for r in recs)
    if op in ("mps", "edge", "x2a", "serving"):
        done, written, flops = {}, 0, 0.0
        for A, B in zip(recs[::2], recs[1::2]):
            k = (A["D"].tobytes(), B["D"].tobytes())
            if k not in done:
                C, _, fl = _dot(A, B, inp["axa"], inp["axb"])
                done[k] = (_size(C), fl)
            written += done[k][0]
            flops += done[k][1] * (4 if cw == 2 else 1)
        return read + 8.0 * cw * written, flops
    if op == "double_layer":
        C, _, flops = _dot(recs[0], _conj(recs[0]), (4,), (4,))
        return read + 8.0 * _size(C), flops
    if op == "corner":
        C, _, flops = _corner(recs)
        return read + 8.0 * _size(C), flops
    if op == "moves":   # three calls, each reads and writes the tensor
        return 6.0 * read, 0.0
    # the overlap reads both tensors; the trace reads the diagonals of one
    t, D = recs[0]["t"], recs[0]["D"]
    diag = np.all(t[:, 0, :] == t[:, 3, :], axis=1)
    return read + 8.0 * float(np.prod(D[diag][:, :3], axis=1).sum()), 2.0 * _size(recs[0])


def exact(case, seed):
    op, inp = case["op"], _inputs(case)
    recs, data = inp["recs"], _data(case, seed)
    if op in ("mps", "edge", "x2a"):
        if case.get("dtype") == "c128":
            data = [torch.view_as_complex(d.view(-1, 2)) for d in data]
        out = _dot(recs[0], recs[1], inp["axa"], inp["axb"], data[0], data[1])[1]
        return torch.view_as_real(out).reshape(-1) if out.is_complex() else out
    if op == "double_layer":
        C, c, _ = _dot(recs[0], _conj(recs[0]), (4,), (4,), data[0], data[0])
        return _fuse(C, DOUBLE_LAYER_GROUPS, c)
    if op == "corner":
        return _corner(recs, data)[1]
    if op == "moves":
        gated = _swap(recs[0], MATRIX_GROUPS, data[0])
        return [gated, _fuse(recs[0], MATRIX_GROUPS, gated), gated]
    if op == "scalars":
        return [torch.dot(data[0], data[1]).reshape(1), _trace(recs[0], data[0])]
    return [_dot(recs[i], recs[i + 1], inp["axa"], inp["axb"], data[i], data[i + 1])[1]
            for i in range(0, len(recs), 2)]
