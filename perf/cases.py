"""Workloads of the repair library, timed and compared through its public entry points.

A case is a plain dict.  ``kind`` names the call a program makes:

  index       one sketch with one hole over a box: a wrong index, stride or tile bound in a loop nest
  conv        one sketch with three holes over a box: an im2col lowering with two indices and a loop bound missing
  table       one sketch over an explicit list of points with the source's values as a table, typed quasi-affine grammar
  batch       many small table sketches in one load and one search: what one pass over many snippets leaves
  pair        source and erroneous expression in, repaired expression out
  joint       two holes inside one constraint
  behaviours  bottom-up enumeration with observational-equivalence pruning

``call`` says what of it is timed: ``whole`` creates the grammar, loads the sketch, searches it and reads the
answer (what a snippet costs that is searched once); ``search`` searches a sketch that stays loaded, ``static``
does so without allocating, ``window`` searches one rank's share of it.

Everything is drawn from the seed with integer arithmetic on non-negative operands and positive divisors; the
results are whole numbers and have to be the same.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2505_02146_b200 as xp
from xp_instances import (Hole, JointHole, Sketch, Variable, constant_set, free_grammar, parse_expr,
                          quasi_affine_grammar)

NAMES = ["i", "j", "k", "l", "m"]
ARITH = ["+", "-", "*", "/", "%"]


def listed():
    return [
        # A serving loop: the sketch of a two-variable 16x16 nest stays loaded and a one-operator repair of it is
        # searched without allocating.  The smallest call there is: launches and latency.
        {"name": "serve_static", "kind": "index", "call": "static", "extents": "16x16", "cmin": -8, "cmax": 8, "pow2": 0, "size": 3, "ops": "arith", "ctx": False},
        # The ordinary small repair, end to end: two-variable nest, expressions of up to five nodes.
        {"name": "index_16x16", "kind": "index", "call": "whole", "extents": "16x16", "cmin": -8, "cmax": 8, "pow2": 0, "size": 5, "ops": "arith", "ctx": False},
        # A remainder-tile bound (min / max in the grammar) inside a fixed context, ragged extents.
        {"name": "tile_bound", "kind": "index", "call": "whole", "extents": "17x33x7", "cmin": -6, "cmax": 33, "pow2": 3, "size": 5, "ops": "minmax", "ctx": True},
        # The thread-binding repair of a 256x256 matmul tile nest: 136 leaves, up to seven nodes, 2.1e11 candidates.
        {"name": "thread_binding", "kind": "index", "call": "whole", "extents": "64x256x8", "cmin": -64, "cmax": 64, "pow2": 11, "size": 7, "ops": "arith", "ctx": False},
        # The conv2d im2col lowering: three holes, about 1.8 million iteration points.
        {"name": "conv_three_holes", "kind": "conv", "call": "whole", "channels": 64, "side": 56, "kernel": 3, "size": 6},
        # An index map known by its values only: device tensors of a ragged number of points, up to seven nodes.
        {"name": "table_ragged", "kind": "table", "call": "whole", "vars": 3, "points": 37123, "consts": 128, "size": 7, "device": True},
        # The large search on a sketch that stays loaded: four variables, 2^20 points, up to nine nodes, 3.2e11 candidates.
        {"name": "table_large", "kind": "table", "call": "search", "vars": 4, "points": 1 << 20, "consts": 128, "size": 9, "device": False},
        # A pass over one program: some dozens of small snippets.
        {"name": "batch_40", "kind": "batch", "call": "whole", "n": 40, "points": 1000, "consts": 16, "size": 5},
        # A pass over a suite of programs: a thousand snippets of 4096 points, a tenth of them without a solution.
        {"name": "batch_1024", "kind": "batch", "call": "whole", "n": 1024, "points": 4096, "consts": 16, "size": 6},
        # A source / erroneous expression pair after a loop split: one sketch per node of the erroneous expression.
        {"name": "pair_split_loop", "kind": "pair", "call": "whole", "split": 8, "outer": 12, "inner": 5, "consts": 20, "size": 5},
        # Stride and offset wrong at once: a product search over pairs of expressions.
        {"name": "joint_stride_offset", "kind": "joint", "call": "whole", "rows": 24, "cols": 20, "consts": 30, "size": 3},
        # Pruning by behaviour to reach one size further than the exhaustive bound of the small nest.
        {"name": "behaviours_size7", "kind": "behaviours", "call": "search", "rows": 16, "cols": 16, "consts": 8, "sig": 12, "size": 7},
    ]


# ------------------------------------------------------------------------------------------
# more cases of the same ranges
# ------------------------------------------------------------------------------------------

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extents(rng, n, most):
    while True:
        e = [_log(rng, 3, 256) for _ in range(n)]
        if 256 <= math.prod(e) <= most:
            return "x".join(map(str, e))


def draw(rng):
    kind = rng.choice(["index", "index", "index", "conv", "table", "table", "batch", "pair", "joint", "behaviours"])
    if kind == "index":
        size = rng.choice([3, 5, 7])
        nv = rng.randint(2, 4)
        leaves = {3: _log(rng, 6, 300), 5: _log(rng, 8, 140), 7: _log(rng, 8, 130)}[size]       # (size 7: up to 1.8e11 candidates)
        ncon = max(3, leaves - nv)
        cmin = -rng.randint(0, ncon // 2)
        call = rng.choice(["whole", "whole", "search", "static", "window"])
        if call == "static" and (size > 5 or leaves > 40):       # (its survivor queue is made for small searches)
            call = "search"
        return {"kind": "index", "call": call, "extents": _extents(rng, nv, 2_000_000), "cmin": cmin, "cmax": cmin + ncon - 1,
                "pow2": 0, "size": size, "ops": rng.choice(["arith", "arith", "minmax"]) if size < 7 else "arith", "ctx": rng.random() < 0.3}
    if kind == "conv":
        kernel = rng.choice([3, 3, 3, 5])
        return {"kind": "conv", "call": rng.choice(["whole", "search"]), "channels": _log(rng, 8, 64 if kernel == 3 else 22),
                "side": _log(rng, 14, 56), "kernel": kernel, "size": rng.choice([5, 6])}
    if kind == "table":
        size = rng.choice([5, 7, 9])
        nv = rng.randint(2, 4)
        consts = _log(rng, 8, 128)
        if size == 9 and nv == 4:
            consts = min(consts, 120)
        return {"kind": "table", "call": rng.choice(["whole", "search"]), "vars": nv, "points": _log(rng, 500, 1 << 20) | 1,
                "consts": consts, "size": size, "device": rng.random() < 0.5}
    if kind == "batch":
        n = _log(rng, 4, 900)
        return {"kind": "batch", "call": rng.choice(["whole", "search"]), "n": n, "points": _log(rng, 100, 4096), "consts": rng.randint(4, 16),
                "size": rng.choice([5, 6])}
    if kind == "pair":
        return {"kind": "pair", "call": "whole", "split": rng.randint(3, 32), "outer": rng.randint(2, 40), "inner": rng.randint(2, 9),
                "consts": _log(rng, 6, 60), "size": rng.choice([3, 5])}
    if kind == "joint":
        return {"kind": "joint", "call": "whole", "rows": rng.randint(5, 60), "cols": rng.randint(5, 60), "consts": _log(rng, 6, 60), "size": 3}
    return {"kind": "behaviours", "call": "search", "rows": rng.randint(6, 40), "cols": rng.randint(6, 40), "consts": rng.randint(2, 8),
            "sig": rng.randint(6, 16), "size": rng.choice([5, 7])}


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------

def _rng(case, seed):
    return np.random.Generator(np.random.PCG64(np.random.SeedSequence([0x7065, int(seed)])))


def _pick(r, seq):
    return seq[int(r.integers(len(seq)))]


def _index_constants(case):
    return constant_set(case["cmin"], case["cmax"], [2 ** e for e in range(case["pow2"])])


def _index_ops(case):
    return ARITH + (["min", "max"] if case["ops"] == "minmax" else [])


def _index_grammar(case):
    ext = [int(x) for x in case["extents"].split("x")]
    vs = [Variable(NAMES[d], 0, e) for d, e in enumerate(ext)]
    return free_grammar(vs, _index_constants(case), ops=_index_ops(case))


def _index_target(r, case):
    """A planted index expression of at most ``size`` nodes over the grammar's leaves."""
    ext = [int(x) for x in case["extents"].split("x")]
    order = [int(x) for x in r.permutation(len(ext))]
    a, b = NAMES[order[0]], NAMES[order[1]]
    c = NAMES[order[2]] if len(order) > 2 else a
    big = [v for v in _index_constants(case) if v >= 2] or [1]
    C, D = int(_pick(r, big)), int(_pick(r, big))
    if case["size"] == 3:
        return _pick(r, [f"{a}*{C}", f"{a}+{C}", f"{a}%{C}", f"{a}/{C}", f"{C}-{a}", f"{C}*{b}"])
    if case["size"] == 5:
        forms = [f"({a}*{C})+{b}", f"{b}+({a}*{C})", f"({a}*{C})-{b}", f"({a}+{b})%{C}", f"({a}/{C})+{b}", f"({C}*{a})+{D}"]
        if case["ops"] == "minmax":
            forms = [f"min({C},{a}*{D})", f"max({a},{C}-{b})", f"min({C},{a}+{b})", f"max({C}-{a},{b})"] + forms[:2]
        return _pick(r, forms)
    return _pick(r, [f"({a}*{C})+({b}*{D})", f"(({a}*{C})+{b})+{c}", f"(({a}*{C})+{b})/{D}", f"({a}*{C})+({b}%{D})",
                     f"(({b}/{D})*{C})+{c}", f"({b}*{D})+({a}*{C})"])


def _index_sketch(case, seed):
    r = _rng(case, seed)
    g = _index_grammar(case)
    vs = g.variables
    target = _index_target(r, case)
    if case["ctx"]:                     # the hole sits inside a row-major address
        pitch = int(r.integers(3, 200))
        last = vs[-1].name
        return Sketch(g, [Hole(0, case["size"], ctx=parse_expr(f"(HOLE*{pitch})+{last}", vs),
                               spec_expr=parse_expr(f"(({target})*{pitch})+{last}", vs))])
    return Sketch(g, [Hole(0, case["size"], spec_expr=parse_expr(target, vs))])


def _conv_sketch(case, seed):
    r = _rng(case, seed)
    C, k = case["channels"], case["kernel"]
    H, W = case["side"] - int(r.integers(0, 5)), case["side"] - int(r.integers(0, 5))
    pitch, pad = W + int(r.integers(0, 9)), int(r.integers(0, 2))
    plane = pitch * H
    vs = [Variable("c", 0, C), Variable("oh", 0, H), Variable("ow", 0, W), Variable("kh", 0, k), Variable("kw", 0, k)]
    g = free_grammar(vs, constant_set(-64, 64, [128, 256, 512, 1024, plane]))
    row, col = f"((oh+kh)-{pad})", f"((ow+kw)-{pad})"
    cols = bool(r.integers(2))
    ctx1 = f"((c*{plane})+({row}*{pitch}))+HOLE" if cols else f"((c*{plane})+(HOLE*{pitch}))+{col}"
    spec1 = f"((c*{plane})+({row}*{pitch}))+{col}"
    ctx2 = f"((((c*{k * k})+HOLE)*{H * W})+(oh*{W}))+ow"
    spec2 = f"((((c*{k * k})+((kh*{k})+kw))*{H * W})+(oh*{W}))+ow"
    o, kk, n = ("ow", "kw", W) if cols else ("oh", "kh", H)
    K = case["size"]
    return Sketch(g, [Hole(0, K, ctx=parse_expr(ctx1, vs), spec_expr=parse_expr(spec1, vs)),
                      Hole(0, K, ctx=parse_expr(ctx2, vs), spec_expr=parse_expr(spec2, vs)),
                      Hole(0, K, ctx=parse_expr(f"{kk}<HOLE", vs), spec_expr=parse_expr(f"(({o}+{kk})-{pad})<{n}", vs))])


def _points(r, ext, n):
    """n distinct points of the box [0, ext): its corners, then a random sample, as int32 rows."""
    total = math.prod(ext)
    n = min(n, total)
    corners = [0]
    for e in ext:
        corners = [c * e + x for c in corners for x in ((0, e - 1) if e > 1 else (0,))]
    first = np.array(corners, dtype=np.int64)[:n]
    pool = np.unique(r.integers(0, total, size=n + n // 4 + 64)) if total > 4 * n else np.arange(total, dtype=np.int64)
    pool = r.permutation(np.setdiff1d(pool, first, assume_unique=True))
    while len(first) + len(pool) < n:
        pool = np.setdiff1d(np.union1d(pool, r.integers(0, total, size=n)), first)
        pool = r.permutation(pool)
    rem = np.concatenate([first, pool[:n - len(first)]])
    out = np.empty((n, len(ext)), dtype=np.int32)
    for d in range(len(ext) - 1, -1, -1):
        out[:, d] = rem % ext[d]
        rem //= ext[d]
    return out


def _table_grammar(case, ext):
    vs = [Variable(NAMES[d], 0, e) for d, e in enumerate(ext)]
    return quasi_affine_grammar(vs, constant_set(-case["consts"], case["consts"]), list(range(1, case["consts"] + 1)))


def _table_sketch(case, seed):
    r = _rng(case, seed)
    nv = case["vars"]
    most = {2: 4096, 3: 512, 4: 256}[nv]
    while True:
        ext = [int(x) for x in r.integers(4, most + 1, size=nv)]
        if math.prod(ext) >= 2 * case["points"]:
            break
    coords = _points(r, ext, case["points"])
    a, b = (int(x) for x in r.choice([d for d in range(nv) if ext[d] >= 4], size=2, replace=False))
    P1, P2 = (int(r.integers(2, min(case["consts"], ext[d]) + 1)) for d in (a, b))
    K1 = int(r.integers(2, case["consts"] + 1)) * (1 if r.integers(2) else -1)
    va, vb = coords[:, a].astype(np.int64), coords[:, b].astype(np.int64)
    spec = {5: lambda: va * K1 + vb, 7: lambda: (va // P1) * K1 + vb, 9: lambda: (va // P1) * K1 + vb % P2}[case["size"]]()
    return Sketch(_table_grammar(case, ext), [Hole(0, case["size"], spec_table=spec)], coords)


def _batch_sketches(case, seed):
    r = _rng(case, seed)
    out = []
    for _ in range(case["n"]):
        nv = int(r.integers(2, 4))
        while True:
            ext = [int(x) for x in r.integers(2, 65, size=nv)]
            if math.prod(ext) >= case["points"] // 2:
                break
        coords = _points(r, ext, case["points"])
        vs = [Variable(NAMES[d], 0, e) for d, e in enumerate(ext)]
        ia, ib = (int(x) for x in r.choice(nv, size=2, replace=False))
        xa, xb = coords[:, ia].astype(np.int64), coords[:, ib].astype(np.int64)
        C, D = (int(x) for x in r.integers(2, case["consts"] + 1, size=2))
        if r.random() < 0.1:            # beyond the size bound: no solution
            spec = _pick(r, [xa * C + xb * D, (xa // C) * D + xb, xa % C + xb * D])
        else:
            spec = _pick(r, [xa * C + xb, xa // C + xb, (xa + xb) % C, xa * C - xb, xa + xb * D, xa % C, xa * C])
        g = free_grammar(vs, constant_set(-case["consts"], case["consts"]))
        out.append(Sketch(g, [Hole(0, case["size"], spec_table=spec)], coords))
    return out


def _pair_inputs(case, seed):
    """i = io*split + ii, an address that uses a wrong stride, operator or variable after the split."""
    r = _rng(case, seed)
    S, n = case["split"], case["inner"]
    tv = [Variable("io", 0, case["outer"]), Variable("ii", 0, S), Variable("k", 0, n)]
    sv = [Variable("i", 0, case["outer"] * S), Variable("k", 0, n)]
    consts = sorted(set(range(-1, case["consts"] - 1)) | {S, n, S * n})
    g = free_grammar(tv, consts)
    m = int(r.integers(2, 40))
    source = parse_expr(f"((i*{n})+k)+{m}", sv)
    wrong = _pick(r, [f"(((io*{S})+(ii*{n}))+k)+{m}", f"((((io*{S})+ii)*{n + 1})+k)+{m}", f"((((io*{S})+ii)*{n})+ii)+{m}",
                      f"((((io-{S})+ii)*{n})+k)+{m}", f"((((io*{S})+ii)*{n})+k)+{m + 1}"])
    return g, source, parse_expr(wrong, tv), [parse_expr(f"(io*{S})+ii", tv), parse_expr("k", tv)]


def _joint_inputs(case, seed):
    r = _rng(case, seed)
    R, Cn = case["rows"], case["cols"]
    vs = [Variable("i", 0, R), Variable("j", 0, Cn)]
    g = free_grammar(vs, constant_set(-2, case["consts"] - 3))
    pitch = int(r.integers(2, 64))
    c0, c1 = (int(x) for x in r.integers(1, case["consts"] - 2, size=2))
    e0 = _pick(r, [f"i+{c0}", f"i*{c0}", "i+j", f"i/{c0 + 1 if c0 + 1 < case['consts'] - 2 else c0}"])
    e1 = _pick(r, [f"j+{c1}", f"j*{c1}", f"j%{c1}", f"i-{c1}"])
    sk = Sketch(g, [Hole(0, 1, spec_expr=parse_expr("i", vs))])
    K = case["size"]
    return sk, JointHole((0, 0), (K, K), parse_expr(f"(HOLE0*{pitch})+HOLE1", vs), spec_expr=parse_expr(f"(({e0})*{pitch})+({e1})", vs))


def _behaviour_inputs(case, seed):
    r = _rng(case, seed)
    R, Cn = case["rows"], case["cols"]
    vs = [Variable("i", 0, R), Variable("j", 0, Cn)]
    g = free_grammar(vs, constant_set(-case["consts"], case["consts"]))
    c, d = (int(x) for x in r.integers(2, case["consts"] + 1, size=2))
    target = _pick(r, [f"((i*{c})+j)%{d}", f"((i/{c})*{d})+j", f"(i*{c})+(j*{d})", f"(i%{c})+(j*{d})"]) if case["size"] == 7 else \
        _pick(r, [f"(i*{c})+j", f"(i+j)%{c}", f"(i/{c})+j", f"(j*{c})-i"])
    n = R * Cn
    sig = [0, n - 1] + [int(x) for x in r.choice(np.arange(1, n - 1), size=case["sig"] - 2, replace=False)]
    return Sketch(g, [Hole(0, case["size"], spec_expr=parse_expr(target, vs))]), sig


class State:
    """What the program holds before the call."""


def _load(st, sk, **kw):
    st.loaded = [xp.xp_sketch_load(xp.xp_grammar_create(sk.grammar), sk, **kw)]
    st.workspace = torch.empty(xp.xp_workspace_bytes(st.loaded), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    st = State()
    st.case, st.windows = case, None
    kind, call = case["kind"], case["call"]
    if kind in ("index", "conv"):
        st.sketch = _index_sketch(case, seed) if kind == "index" else _conv_sketch(case, seed)
        if call != "whole":
            _load(st, st.sketch)
        if call == "window":            # the share of rank 3 of 8
            counts = xp.xp_grammar_count(st.loaded[0].grammar, 0, case["size"])
            st.windows = [(0, k, 3 * counts[k] // 8, 4 * counts[k] // 8) for k in range(1, case["size"] + 1) if counts[k]]
    elif kind == "table":
        st.sketch = _table_sketch(case, seed)
        if case["device"]:              # the points and values come from another computation on the GPU
            st.coords = torch.from_numpy(st.sketch.coords).cuda()
            st.specs = {0: torch.from_numpy(st.sketch.holes[0].spec_table).cuda()}
        else:
            st.coords = st.specs = None
        if call == "search":
            _load(st, st.sketch, coords=st.coords, spec_tables=st.specs)
    elif kind == "batch":
        st.sketches = _batch_sketches(case, seed)
        if call == "search":
            grs = [xp.xp_grammar_create(sk.grammar) for sk in st.sketches]
            st.loaded = xp.xp_sketch_load_batch(grs, st.sketches)
            st.workspace = torch.empty(xp.xp_workspace_bytes(st.loaded), dtype=torch.uint8, device="cuda")
    elif kind == "pair":
        g, st.source, st.erroneous, st.var_map = _pair_inputs(case, seed)
        st.grammar = g
    elif kind == "joint":
        st.sketch, st.joint = _joint_inputs(case, seed)
    else:
        sk, st.sig = _behaviour_inputs(case, seed)
        _load(st, sk)
    return st


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------

def _text(*parts):
    """Texts as bytes, in 512 places whatever their length."""
    b = b"\n".join(p if isinstance(p, bytes) else p.encode() for p in parts)
    return np.frombuffer(b[:512].ljust(512, b"\0"), dtype=np.uint8)


def _code(code, most):
    """Postfix code as rows of (kind, arg, value), in ``most`` places whatever its length."""
    out = np.full((most, 3), -1, dtype=np.int64)
    if code:
        out[:len(code)] = code
    return out


def _holes(results):
    """The answers of hole results as arrays: counts per size, least solution (size, rank, postfix code)."""
    return {"cand": np.array([r.cand_count for r in results], dtype=np.int64),
            "match": np.array([r.match_count for r in results], dtype=np.int64),
            "least": np.array([(int(r.solved), r.least_size, r.least_rank) for r in results], dtype=np.int64),
            "code": np.stack([_code(r.least_code, 15) for r in results])}


def _summaries(packed):
    a = xp.summaries_as_numpy(packed)
    return {"cand": a["cand_count"].astype(np.int64), "match": a["match_count"].astype(np.int64),
            "least": np.stack([a["solved"].astype(np.int64), a["least_size"].astype(np.int64), a["least_rank"].astype(np.int64)]),
            "text": np.frombuffer(a["least_text"].tobytes(), dtype=np.uint8)}


def run(st):
    case = st.case
    kind, call = case["kind"], case["call"]
    if kind in ("index", "conv", "table"):
        if call == "static":
            out = xp.xp_repair_static(st.loaded[0])
            return {"cand": np.array([list(r.cand_count) for r in out], dtype=np.int64),
                    "match": np.array([list(r.match_count) for r in out], dtype=np.int64),
                    "least": np.array([(r.solved, r.least_size, r.least_rank) for r in out], dtype=np.int64),
                    "text": _text(*(r.least_text for r in out))}
        if call == "whole":
            gr = xp.xp_grammar_create(st.sketch.grammar)
            if kind == "table":
                loaded = xp.xp_sketch_load(gr, st.sketch, coords=st.coords, spec_tables=st.specs)
            else:
                loaded = xp.xp_sketch_load(gr, st.sketch)
            return _holes(xp.xp_repair(loaded))
        return _holes(xp.xp_repair(st.loaded[0], workspace=st.workspace, rank_ranges=st.windows))
    if kind == "batch":
        if call == "search":
            packed, _ = xp.xp_repair_batch(st.loaded, packed=True, workspace=st.workspace)
            return _summaries(packed)
        grs = [xp.xp_grammar_create(sk.grammar) for sk in st.sketches]
        loaded = xp.xp_sketch_load_batch(grs, st.sketches)
        if case["n"] < 200:             # a program that handles its snippets one by one reads one result per hole
            return _holes([h for res in xp.xp_repair_batch(loaded) for h in res])
        packed, _ = xp.xp_repair_batch(loaded, packed=True)
        return _summaries(packed)
    if kind == "pair":
        r = xp.xp_repair_pair(xp.xp_grammar_create(st.grammar), st.source, st.erroneous, 0, case["size"], var_map=st.var_map)
        return {"head": np.array([int(r.solved), r.n_sketches, r.node_first, r.node_last, r.least_size, r.least_rank, r.candidates], dtype=np.int64),
                "code": _code(r.stitched_code, 64), "text": _text(r.stitched_text)}
    if kind == "joint":
        loaded = xp.xp_sketch_load(xp.xp_grammar_create(st.sketch.grammar), st.sketch)
        r = xp.xp_repair_joint(loaded, st.joint)
        return {"cand": np.array(r.cand_count, dtype=np.int64), "match": np.array(r.match_count, dtype=np.int64),
                "least": np.array([int(r.solved), r.least_total, r.least_size0, r.least_rank0, r.least_rank1], dtype=np.int64),
                "text": _text(r.least_text0, r.least_text1)}
    r = xp.xp_behaviours(st.loaded[0], st.sig)
    return {"enumerated": np.array(list(r.enumerated), dtype=np.int64), "distinct": np.array(list(r.distinct), dtype=np.int64),
            "head": np.array([r.sig_matches, r.hit, r.hit_size, r.hit_index, r.hit_verified, r.solved, r.solution_size,
                              r.solution_index, r.representatives], dtype=np.int64),
            "text": _text(r.hit_text, r.solution_text)}


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------

def _counts(n_leaves, n_ops, size):
    c = [0] * (size + 1)
    c[1] = n_leaves
    for s in range(3, size + 1):
        c[s] = n_ops * sum(c[a] * c[s - 1 - a] for a in range(1, s - 1))
    return c


def _typed_counts(nv, consts, size):
    nk, npos = 2 * consts + 1, consts
    c = [0] * (size + 1)
    c[1] = nv
    for s in range(3, size + 1):
        c[s] = 2 * sum(c[a] * c[s - 1 - a] for a in range(1, s - 1)) + c[s - 2] * (nk + 2 * npos)
    return c


def work(case):
    """Bytes: points, source values, grammar and answers once.  Operations: one for every expression that can
    stand beside the last operator (each of them has to be known at one point at least), one for every point
    that the reported solution has to be held against."""
    kind = case["kind"]
    size = case["size"]
    below = size - 2 if size > 2 else 1
    n = 1
    if kind == "index":
        leaves = len(case["extents"].split("x")) + len(_index_constants(case))
        c = _counts(leaves, len(_index_ops(case)), size)
        points, values = math.prod(int(x) for x in case["extents"].split("x")), 0
    elif kind == "conv":
        leaves, n = 5 + 129 + 5, 3
        c = _counts(leaves, 5, size)
        points, values = case["channels"] * case["side"] ** 2 * case["kernel"] ** 2, 0
    elif kind == "table":
        leaves = case["vars"] + 3 * case["consts"] + 1
        c = _typed_counts(case["vars"], case["consts"], size)
        points, values = case["points"], case["points"] * (8 + 4 * case["vars"])
    elif kind == "batch":
        leaves, n = 3 + 2 * case["consts"] + 1, case["n"]
        c = _counts(leaves, 5, size)
        points, values = case["points"], case["points"] * (8 + 4 * 2.5)
    elif kind == "pair":
        leaves, n = 3 + case["consts"], 11
        c = _counts(leaves, 5, size)
        points, values = case["outer"] * case["split"] * case["inner"], 0
    elif kind == "joint":
        leaves, n = 2 + case["consts"], 2
        c = _counts(leaves, 5, size)
        below = size
        points, values = case["rows"] * case["cols"], 0
    else:
        leaves = 2 + 2 * case["consts"] + 1
        c = _counts(leaves, 5, size)
        points, values = case["rows"] * case["cols"], 0
    operands = sum(c[1:below + 1]) * (case["sig"] if kind == "behaviours" else 1)
    return {"bytes": n * (values + 16.0 * leaves + 300), "flops": n * (operands + points * size)}


def tolerance(case):
    return "exact"
