"""Searches over operand classes (operands that no probe tells apart are met once, and taken apart where a candidate
passes): against the oracle, and cut into rank windows small enough to be searched operand by operand."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from tests.util import assert_same, check_sketch
from xp_instances import Hole, Sketch, Variable, constant_set, free_grammar, parse_expr, quasi_affine_grammar

pytestmark = pytest.mark.gpu

VS = [Variable("i", 0, 9), Variable("j", 0, 7)]


@pytest.mark.parametrize("ops,consts", [
    (["+", "-", "*", "/", "%"], constant_set(-13, 13)),                       # 4 205 operands of three nodes: just enough for classes
    (["+", "-", "*", "min", "max", "%"], constant_set(-9, 14) + [1 << 20, 5]),
    (["+", "*", "<<", ">>", "/"], constant_set(-4, 24)),                      # undefined shifts and divisions
])
@pytest.mark.parametrize("ctx,spec", [("i<HOLE", "i<((j*2)+1)"), ("HOLE<=j", "(i/3)<=j"), ("(j-HOLE)<(i-2)", "(i%4)<5")])
def test_comparing_contexts(xp, ops, consts, ctx, spec):
    g = free_grammar(VS, sorted(set(consts)), ops=ops)
    r = check_sketch(xp, Sketch(g, [Hole(0, 5, ctx=parse_expr(ctx, VS), spec_expr=parse_expr(spec, VS))], name=f"{ctx}: {spec}"))[0]
    assert r.cand_count[3] >= 4096
    if max(consts) < 100 and "<<" not in ops:            # (shifts and wide operands go the exact way: a test per leaf)
        assert r.filter_tests < 0.7 * r.cand_count[3] * 10 * 3


def _large(spec, ops=("+", "-", "*", "/", "%"), consts=None, ctx=None):
    """45 leaves, operators five at the root: the operands of five nodes of a search up to seven are above the tables."""
    g = free_grammar(VS, consts or constant_set(-17, 25), ops=list(ops))
    return Sketch(g, [Hole(0, 7, ctx=parse_expr(ctx, VS) if ctx else [], spec_expr=parse_expr(spec, VS))], name=spec)


@pytest.mark.parametrize("sk", [
    _large("((i*7)+j)*3"),
    _large("(i/2)+(j%3)"),                                                    # small targets: most divisors are open
    _large("min(i*3,j+4)", ops=("+", "-", "*", "min", "max")),
    _large("(i*9)+j", consts=constant_set(-10, 30) + [1 << 20, 1 << 30]),     # operands beyond 31 bits
    _large("(((i*3)+j)*8)+1", ctx="(HOLE*8)+1"),
], ids=lambda s: s.name)
def test_a_window_against_the_oracle(xp, sk):
    """Windows wide enough to be searched by class, over both sides of a block's border, cut inside a class."""
    gr = xp.xp_grammar_create(sk.grammar)
    ls = xp.xp_sketch_load(gr, sk)
    n = xp.xp_grammar_count(gr, 0, 7)[7]
    width = min(n // 6, 60_000_000)
    for begin in (n // 9, 3 * n // 5 + 12_345):
        w = {7: (begin, begin + width)}
        got = xp.xp_repair(ls, size_min=7, size_max=7, rank_ranges=[(0, 7, *w[7])])[0]
        want = oracle.repair_hole(sk, 0, rank_ranges={**{k: (0, 0) for k in range(1, 7)}, **w})
        assert got.match_count[7] == want.match_count[7], (sk.name, begin)
        if want.match_count[7]:
            assert (got.least_rank, got.least_text) == (want.least_rank, want.least_text)


def _cut(xp, ls, size, n, parts):
    """Matches and least rank at `size`, searched in rank windows."""
    match, least = 0, None
    for p in range(parts):
        r = xp.xp_repair(ls, size_min=size, size_max=size, rank_ranges=[(0, size, n * p // parts, n * (p + 1) // parts)])[0]
        match += r.match_count[size]
        if r.match_count[size] and least is None:
            least = r.least_rank
    return match, least


@pytest.mark.parametrize("spec", ["((i*7)+j)*3", "(i/2)+(j%3)", "((i+j)%5)*2"])
def test_free_grammar_equals_its_windows(xp, spec):
    sk = _large(spec)
    gr = xp.xp_grammar_create(sk.grammar)
    ls = xp.xp_sketch_load(gr, sk)
    n = xp.xp_grammar_count(gr, 0, 7)[7]
    r = xp.xp_repair(ls, size_min=7, size_max=7)[0]
    match, least = _cut(xp, ls, 7, n, 61)
    assert match > 0 and r.match_count[7] == match and r.least_rank == least
    xp.xp_sketch_refine(ls)                              # other probes, other classes, the same answer
    again = xp.xp_repair(ls)[0]
    assert again.match_count[7] == match


@pytest.mark.parametrize("table", [False, True])
def test_quasi_affine_grammar_equals_its_windows(xp, table):
    """Classes of five nodes under operands of seven (typed grammar, three nonterminals), over a box and a table of points."""
    vs = [Variable("i", 0, 40), Variable("j", 0, 30)]
    g = quasi_affine_grammar(vs, constant_set(-40, 40), list(range(1, 51)))
    spec = "((i/3)*5)+(j%4)"
    if table:
        r = np.random.default_rng(3)
        coords = np.stack([r.integers(0, 40, 333), r.integers(0, 30, 333)], axis=1).astype(np.int32)
        want = (coords[:, 0].astype(np.int64) // 3) * 5 + coords[:, 1] % 4
        sk = Sketch(g, [Hole(0, 9, spec_table=want)], coords)
    else:
        sk = Sketch(g, [Hole(0, 9, spec_expr=parse_expr(spec, vs))])
    gr = xp.xp_grammar_create(g)
    ls = xp.xp_sketch_load(gr, sk)
    n = xp.xp_grammar_count(gr, 0, 9)[9]
    r = xp.xp_repair(ls, size_min=9, size_max=9)[0]
    match, least = _cut(xp, ls, 9, n, 64)
    assert match > 0 and r.match_count[9] == match and r.least_rank == least


def test_matches_in_large_classes(xp):
    """A target with a term that is 0 (j / 28): millions of matches, most of them in a few classes, which are listed and shared by all
    warps; with a queue and a list that run over, and in bounded launches."""
    import torch
    sk = _large("((j/28)*13)+i")
    gr = xp.xp_grammar_create(sk.grammar)
    ls = xp.xp_sketch_load(gr, sk)
    n = xp.xp_grammar_count(gr, 0, 7)[7]
    only7 = dict(size_min=7, size_max=7)
    r = xp.xp_repair(ls, **only7)[0]
    match, least = _cut(xp, ls, 7, n, 61)
    assert match > 2**20 and r.match_count[7] == match and r.least_rank == least
    need = xp.xp_workspace_bytes([ls], **only7)
    ws = torch.empty(need - 40 * (2**20 - 2**16), dtype=torch.uint8, device="cuda")
    small = xp.xp_repair(ls, workspace=ws, **only7)[0]
    assert small.match_count[7] == match and small.least_rank == least
    bounded = xp.xp_repair(ls, timeout_ms=60_000, **only7)[0]
    assert bounded.match_count[7] == match and bounded.least_rank == least
    few = _large("((i*7)+j)*3")                          # (a launch takes 8192 pieces of 64 members; here there are none)
    few = xp.xp_repair(xp.xp_sketch_load(gr, few), timeout_ms=60_000, **only7)[0]
    assert bounded.n_launches >= few.n_launches + 3


def test_guards_that_nearly_always_hold(xp):
    """Where most candidates match, operands do not go by class: 1.7e7 matches, each operand met for itself."""
    g = free_grammar(VS, constant_set(1, 68))
    sk = Sketch(g, [Hole(0, 5, ctx=parse_expr("(0-HOLE)<1000000", VS), spec_expr=parse_expr("0<1", VS))])
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), sk)
    r = xp.xp_repair(ls)[0]
    n = r.cand_count
    assert n[3] > 4096 and sum(n) > 2**24                # (enough for classes, and for 2^24 matches)
    undefined = 0                                        # quotients and remainders with a divisor that is 0 somewhere
    few = 200_000
    for begin in (0, n[5] // 2, n[5] - few):
        w = {1: (0, 0), 3: (0, 0), 5: (begin, begin + few)}
        want = oracle.repair_hole(sk, 0, rank_ranges=w)
        got = xp.xp_repair(ls, size_min=5, size_max=5, rank_ranges=[(0, 5, *w[5])])[0]
        assert got.match_count[5] == want.match_count[5]
        undefined += few - want.match_count[5]
    match, least = _cut(xp, ls, 5, n[5], 7)
    assert r.match_count[5] == match and match > 0.9 * n[5]
    assert r.filter_tests > 0.8 * n[3] * 10 * 3          # every operand, five operators on either side, the constants and two variables


def test_classes_of_many_holes_in_one_load(xp):
    """Sketches with one, two and no holes with classes, of several grammars, in one load: as if loaded one by one, and as the oracle has it."""
    sks = []
    for q in range(12):
        consts = constant_set(-13, 13 + 2 * (q % 4)) if q % 3 else constant_set(-4, 4)
        g = free_grammar(VS, consts, ops=["+", "-", "*", "/", "%"][:5 - q % 2 * (q % 3 == 0)])
        holes = [Hole(0, 5, ctx=parse_expr("i<HOLE", VS), spec_expr=parse_expr(f"i<((j*2)+{q - 3})", VS))]
        if q % 2:
            holes.append(Hole(0, 5, ctx=parse_expr("(j-HOLE)<2", VS), spec_expr=parse_expr(f"(j-(i/{q}))<2", VS)))
            holes.append(Hole(0, 3, spec_expr=parse_expr("i*2", VS)))
        sks.append(Sketch(g, holes, name=f"sketch {q}"))
    vs = [Variable("i", 0, 40), Variable("j", 0, 30)]
    typed = quasi_affine_grammar(vs, constant_set(-20, 20), list(range(1, 31)))
    sks.append(Sketch(typed, [Hole(0, 7, ctx=parse_expr("j<HOLE", vs), spec_expr=parse_expr("j<((i/2)+1)", vs))], name="typed"))
    grs = [xp.xp_grammar_create(s.grammar) for s in sks]
    many = xp.xp_sketch_load_batch(grs, sks)
    together = xp.xp_repair_batch(many)
    for q, sk in enumerate(sks):
        alone = xp.xp_repair(xp.xp_sketch_load(grs[q], sk))
        got = xp.xp_repair(many[q])
        for h in range(len(sk.holes)):
            if sk.name != "typed":
                assert_same(alone[h], oracle.repair_hole(sk, h), f"{sk.name} hole {h}")
            assert_same(got[h], alone[h], f"{sk.name} hole {h}")
            assert_same(together[q][h], alone[h], f"{sk.name} hole {h} in the batch")
            assert got[h].filter_tests == alone[h].filter_tests                  # (tests count classes where there are some)
            if sk.name != "typed" and q % 3 and len(sk.holes[h].ctx):
                assert got[h].filter_tests < 0.7 * got[h].cand_count[3] * 10 * 3


def test_a_thousand_holes_share_a_load(xp):
    """1100 guards whose classes are made in several groups of launches (their scratch has a bound)."""
    g = [free_grammar(VS, constant_set(-k, 60 - k)) for k in range(4)]
    sks = [Sketch(g[q % 4], [Hole(0, 5, ctx=parse_expr("i<HOLE", VS), spec_expr=parse_expr(f"i<((j*{q % 5})-{q % 7})", VS))]) for q in range(1100)]
    grs = [xp.xp_grammar_create(m) for m in g]
    ls = xp.xp_sketch_load_batch([grs[q % 4] for q in range(1100)], sks)
    for q in (0, 1, 333, 700, 1098, 1099):
        one = xp.xp_repair(xp.xp_sketch_load(grs[q % 4], sks[q]), size_max=3)
        got = xp.xp_repair(ls[q], size_max=3)
        assert_same(got[0], one[0])
        w = [(0, 5, 3_000_000, 4_000_000)]
        a, b = (xp.xp_repair(s, size_min=5, rank_ranges=w)[0] for s in (ls[q], xp.xp_sketch_load(grs[q % 4], sks[q])))
        assert_same(a, b)
        assert a.filter_tests == b.filter_tests


def test_a_static_call_of_many_comparing_holes(xp):
    """64 holes whose contexts compare, at three sizes with nine productions: the fixed scratch holds the plan that keeps an
    operand set's operators together."""
    g = free_grammar(VS, constant_set(1, 3), ops=["+", "-", "*", "/", "%", "min", "max", "+", "-"])
    holes = [Hole(0, 7, ctx=parse_expr("i<HOLE", VS), spec_expr=parse_expr(f"i<(({1 + h % 5}+(j*{h % 4}))-{h % 3})", VS)) for h in range(64)]
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), Sketch(g, holes))
    flag = dict(flags=xp.XP_FLAG_ALWAYS_FILTER)          # (size 3 too)
    want = xp.xp_repair(ls, **flag)
    got = xp.xp_repair_static(ls, **flag)
    for h in range(64):
        assert list(got[h].match_count)[:8] == want[h].match_count, h
        assert got[h].solved == want[h].solved and (not want[h].solved or got[h].least_rank == want[h].least_rank)
    assert any(w.solved for w in want)


def test_a_window_counts_its_own_candidates(xp):
    """Candidates visited (tested or decided without a test) of a window that is searched by class: those of the window."""
    sk = _large("((i*7)+j)*3")
    gr = xp.xp_grammar_create(sk.grammar)
    ls = xp.xp_sketch_load(gr, sk)
    n = xp.xp_grammar_count(gr, 0, 7)
    begin = n[1] * n[5] + n[3] * n[3]                     # the first production's sums of five nodes and a leaf
    for width in (n[1] * 1_500_000, n[1] * 4_000_000):
        r = xp.xp_repair(ls, size_min=7, size_max=7, rank_ranges=[(0, 7, begin, begin + width)])[0]
        assert r.filter_tests < width // n[1] * 3        # (by class, or this test does not test what it says)
        assert r.filter_tests + r.candidates_skipped == width


def test_calls_that_leave_classes_out(xp):
    """Comparing contexts go by operand where the scratch is small for their candidates, and where few sketches of a large batch have one."""
    g = free_grammar(VS, constant_set(-4, 6), ops=["+", "-", "*", "/", "%", "min", "max"])
    sk = Sketch(g, [Hole(0, 7, ctx=parse_expr("i<HOLE", VS), spec_expr=parse_expr(f"i<((i/{h + 2})+(j%{h + 3}))", VS)) for h in range(3)])
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), sk)
    for got, want in zip(xp.xp_repair_static(ls), xp.xp_repair(ls)):
        assert list(got.match_count)[:8] == want.match_count and got.least_rank == want.least_rank
        assert got.evals_executed > want.evals_executed  # (every operand is met for itself)
    g5 = free_grammar(VS, constant_set(-13, 17))
    sks = [Sketch(g5, [Hole(0, 5, ctx=parse_expr("i<HOLE", VS), spec_expr=parse_expr("i<((j*2)+1)", VS))])] + \
          [Sketch(g5, [Hole(0, 3, spec_expr=parse_expr(f"(i*{q % 5})+j", VS))]) for q in range(69)]
    gr = xp.xp_grammar_create(g5)
    batch = xp.xp_sketch_load_batch([gr] * len(sks), sks)
    together, alone = xp.xp_repair_batch(batch)[0][0], xp.xp_repair(batch[0])[0]
    assert_same(together, alone)
    assert together.filter_tests > 1.5 * alone.filter_tests


def test_a_target_that_collapses_to_a_variable(xp):
    """A variable is the target (k / 28 is 0): more matches than the list of classes is for, so a window wide enough for classes goes by operand."""
    vs = [Variable("i", 0, 4), Variable("j", 0, 7), Variable("k", 0, 8)]
    g = free_grammar(vs, constant_set(-64, 64, [2**e for e in range(11)]))
    gr = xp.xp_grammar_create(g)
    ls, other = (xp.xp_sketch_load(gr, Sketch(g, [Hole(0, 7, spec_expr=parse_expr(spec, vs))])) for spec in ("((k/28)*13)+j", "((i*13)+j)*5"))
    n = xp.xp_grammar_count(gr, 0, 7)
    begin, width = n[1] * n[5] + n[3] * n[3], n[1] * 8_000_000            # sums of five nodes and a leaf

    def window(s, lo, hi):
        return xp.xp_repair(s, size_min=7, size_max=7, rank_ranges=[(0, 7, begin + lo, begin + hi)])[0]
    r = window(ls, 0, width)
    parts = [window(ls, width * p // 16, width * (p + 1) // 16) for p in range(16)]
    assert r.match_count[7] == sum(x.match_count[7] for x in parts) > 0
    assert r.least_rank == next(x.least_rank for x in parts if x.match_count[7])
    assert window(other, 0, width).n_launches == r.n_launches + 1           # (members_kernel: by class)


def _odd_guard():
    """j < HOLE holds everywhere but at one interior point, which no sample has: candidates survive the probes and fail there."""
    vs = [Variable("i", 0, 40), Variable("j", 0, 40)]
    ids = np.arange(1600, dtype=np.int64)
    coords = np.stack([ids // 40, ids % 40], axis=1).astype(np.int32)
    spec = np.ones(1600, dtype=np.int64)
    spec[23 * 40 + 31] = 0
    return Sketch(free_grammar(vs, constant_set(17, 47)), [Hole(0, 5, ctx=parse_expr("j<HOLE", vs), spec_table=spec)], coords, name="odd guard")


def test_classes_after_a_refinement(xp):
    """Promoted points are other probes and make other classes; a workspace made before still serves."""
    import torch
    sk = _odd_guard()
    gr = xp.xp_grammar_create(sk.grammar)
    ls = xp.xp_sketch_load(gr, sk)
    ws = torch.empty(xp.xp_workspace_bytes([ls]), dtype=torch.uint8, device="cuda")
    before = xp.xp_repair(ls, workspace=ws)[0]
    assert before.cand_count[3] > 4096 and before.probe_survivors > sum(before.match_count)
    assert xp.xp_sketch_refine(ls) >= 1
    after = xp.xp_repair(ls, workspace=ws)[0]
    assert_same(after, before)
    assert after.probe_survivors < before.probe_survivors
    w = {1: (0, 0), 3: (0, 0), 5: (300_000, 340_000)}
    got = xp.xp_repair(ls, size_min=5, rank_ranges=[(0, 5, *w[5])])[0]
    assert got.match_count[5] == oracle.repair_hole(sk, 0, rank_ranges=w).match_count[5]


def test_a_load_without_memory_for_classes(xp, monkeypatch):
    """The checked build can be told to refuse memory: a load (its own memory, or a batch's scratch) and a refinement without it."""
    if os.environ.get("XP_CHECKED_BUILD") != "1":
        pytest.skip("run through test_classes_under_the_checked_build")
    sk = _odd_guard()
    gr = xp.xp_grammar_create(sk.grammar)
    plain = xp.xp_sketch_load(gr, sk)
    want = xp.xp_repair(plain)[0]
    size = xp.xp_sketch_info_get(plain).device_bytes

    def by_operand(ls):
        r = xp.xp_repair(ls)[0]
        assert_same(r, want)
        return r.filter_tests > 1.5 * want.filter_tests
    monkeypatch.setenv("XP_POOL_MOST", str(size - 1))
    assert by_operand(xp.xp_sketch_load(gr, sk))                                 # no room beside its tables
    with pytest.raises(xp.XpError) as e:
        monkeypatch.setenv("XP_POOL_MOST", "65536")
        xp.xp_sketch_load(gr, sk)
    assert e.value.status == 5
    monkeypatch.setenv("XP_POOL_MOST", str(size + 4096))
    many = xp.xp_sketch_load_batch([gr] * 8, [sk] * 8)                           # no room for the scratch of all
    assert all(by_operand(ls) for ls in many[::3])
    monkeypatch.delenv("XP_POOL_MOST")
    assert xp.xp_sketch_refine(many[0]) >= 1 and not by_operand(many[0])         # (a refinement makes them)
    monkeypatch.setenv("XP_POOL_MOST", "65536")
    assert xp.xp_sketch_refine(many[0]) >= 0
    assert_same(xp.xp_repair(many[0])[0], want)


def test_classes_under_the_checked_build():
    """Slots, places, members and entries of the list, with index checks compiled in (a failed one makes every search an error)."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    cases = "comparing_contexts or many_holes or large_classes or static_call or window_counts or refinement or without_memory or typed or quasi"
    r = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu", "-p", "no:cacheprovider", "tests/test_classes_gpu.py", "-k",
                        f"({cases}) and not checked_build"], cwd=root, env=dict(os.environ, XP_CHECKED_BUILD="1"), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-1000:]
    assert " passed" in r.stdout and "skipped" not in r.stdout
