"""The search's kernels at the sizes where each can go wrong, against the CPU oracle, bit for bit (whole numbers
throughout: the tolerance is zero)."""
import ctypes as C
import os
import subprocess
import threading
import time

import numpy as np
import pytest

import oracle
from tests.conftest import ROOT
from tests.util import assert_same, check_sketch
from xp_instances import Hole, JointHole, Sketch, Variable, constant_set, free_grammar, parse_expr
from tests.test_behaviours_gpu import _check as check_behaviours
from tests.test_joint_gpu import _check as check_joint

IJ = [Variable("i", 0, 9), Variable("j", -3, 6)]
W = 1 << 33


@pytest.mark.gpu
@pytest.mark.parametrize("consts,ops,ctx,spec", [
    (constant_set(-30, 30), "+-*/%", "", "(i*7)+j"),                   # more constants than a lane's registers hold
    (constant_set(-30, 30), "+-*/%", "", "(i/3)*-5"),
    (constant_set(-30, 30), "+-*/%", "", "(i+j)%11"),
    ([2], "+-*/%", "", "(i*2)-j"),                                     # one constant
    ([], "+-*/%", "", "(i*j)+j"),                                      # none
    ([0, 1, -1], "+-*/%", "", "0"),                                    # zero target: every product with a zero operand
    ([W, -W, 3, 2**31 - 1, -2**31], "+-*/%", "", f"(i*{W})+j"),        # operands and targets outside int32
    ([W, 5, 2**62, -2**63], "+-*/%", "", f"(j*{W})/5"),
    ([1, 2, 7], ["+", "min", "max", "<<", ">>"], "", "min(i<<2,7)"),
    ([1, 2, 70], ["-", "<<", ">>"], "", "(i<<1)>>2"),                  # shifts that are undefined
    (constant_set(-9, 9), "+-*/%", "(HOLE*3)+(i*16)", "((i+j)*3)+(i*16)"),
    (constant_set(-9, 9), "+-*/%", "HOLE/4", "(i*9)/4"),               # a context that loses values
    (constant_set(-9, 9), "+-*/%", "HOLE*HOLE", "(i-j)*(i-j)"),
    (constant_set(-9, 9), "+-*/%", "(HOLE%5)+(j/(i-4))", "((i*j)%5)+(j/(i-4))"),
    (constant_set(-40, 40), "+-*/%", "HOLE<=i", "(j*2)<=i"),           # comparisons: runs of constants
    (constant_set(-40, 40), "+-*/%", "(i-3)<(HOLE*-2)", "(i-3)<(j/2)"),
    ([W, 3, -W], "+-*/%", f"HOLE<(i*{W})", f"(j*{W})<(i*{W})"),
    (constant_set(-9, 9), "+-*/%", "", "i/0"),                         # never defined
])
def test_a_leaf_at_the_root(xp, consts, ops, ctx, spec):
    g = free_grammar(IJ, consts, ops=list(ops))
    sk = Sketch(g, [Hole(0, 5, ctx=parse_expr(ctx, IJ) if ctx else [], spec_expr=parse_expr(spec, IJ))], name=f"{ctx} = {spec}")
    n = check_sketch(xp, sk)[0].cand_count
    b, e = n[3] // 3 + 1, n[5] - n[5] // 3 - 1                          # windows whose ends lie inside blocks
    check_sketch(xp, sk, windows={1: (0, 1), 3: (1, b), 5: (n[5] // 7 + 1, e)})


@pytest.mark.gpu
@pytest.mark.parametrize("top", [12, 11])                               # 1125^2 pairs of size 3: an index; 980^2: a test per pair
@pytest.mark.parametrize("spec", ["(i*3)+(j*2)", "(i+2)*(j-1)", "(i*5)/(j+4)", "(i+j)%(j+5)", "j-j", "(i*1048576)*(j*65536)"])
def test_two_operands_of_three_nodes(xp, top, spec):
    g = free_grammar(IJ, list(range(0, top)) + [65536])
    sk = Sketch(g, [Hole(0, 7, spec_expr=parse_expr(spec, IJ))], name=spec)
    g7 = oracle.counts(g, 0, 7)[7]
    check_sketch(xp, sk, windows={7: (0, 1_500_000)})                   # the first blocks: a leaf left, then pairs
    check_sketch(xp, sk, windows={7: (g7 // 2 - 700_000, g7 // 2 + 700_001)})
    check_sketch(xp, sk, windows={5: (3, 40_000), 7: (g7 - 1_500_000, g7 - 1)})


DEEP = "((i+1)*2)-(((j+1)*3)-(((i-j)+1)-(((i*j)+2)-HOLE)))"


@pytest.mark.gpu
@pytest.mark.parametrize("points", [1, 31, 255, 256, 257, 4096, 4097, 9000])
@pytest.mark.parametrize("ctx", ["", "((i*2)+(j*3))*((HOLE+1)+(i*j))", DEEP, f"(HOLE*{W})+i", "(17-HOLE)/-3", "((HOLE%7)+(i/(j+1)))-(5%(i+1))",
                                 "max(HOLE,i)<(min(j,3)+4)"])
def test_whole_domain_check_of_many_matches(xp, points, ctx):
    """Programs with pushed values, too deep ones, values outside int32, constant and variable divisors; tables that end
    inside a step, a piece and a chunk; and boxes of at most one chunk."""
    g = free_grammar(IJ, [0, 1, 2])
    context = parse_expr(ctx, IJ) if ctx else []
    S = parse_expr(ctx.replace("HOLE", "(i+j)") if ctx else "i+j", IJ)
    rng = np.random.default_rng(points)
    coords = np.stack([rng.integers(0, 200, size=points), rng.integers(0, 30, size=points)], axis=1).astype(np.int32)
    check_sketch(xp, Sketch(g, [Hole(0, 5, ctx=context, spec_expr=S)], coords, name=f"table {points}: {ctx}"))
    vs = [Variable("i", 0, points if points < 300 else 64), Variable("j", 0, 1 if points < 300 else points // 64)]
    check_sketch(xp, Sketch(free_grammar(vs, [0, 1, 2]), [Hole(0, 5, ctx=context, spec_expr=S)], name=f"box {points}: {ctx}"))


@pytest.mark.gpu
@pytest.mark.parametrize("ctx,spec", [
    ("((c*3136)+(HOLE*56))+w", "((c*3136)+((r+1)*56))+w"),              # the shared terms cancel
    ("((c*3136)+(HOLE*56))+w", "((c*3136)+(r*56))+(w*2)"),              # one does not
    ("(HOLE*(w+1))+(c/2)", "((r*2)*(w+1))+(c/2)"),                      # a variable in the factor; a common quotient
    ("(HOLE*4)+(w/(c-3))", "(r*4)+(w/(c-3))"),                          # undefined where c is 3
    ("((HOLE+c)*(HOLE+1))-(c*HOLE)", "((r+c)*(r+1))-(c*r)"),            # not affine
    ("(HOLE*4611686018427387904)+(c*r)", "(r*4611686018427387904)+(r*c)"),
])
def test_variables_that_cancel_on_a_large_box(xp, ctx, spec):
    vs = [Variable("c", 0, 11), Variable("r", 0, 56), Variable("w", 0, 57)]
    g = free_grammar(vs, [0, 1, 2], ops=["+", "*", "/"])
    check_sketch(xp, Sketch(g, [Hole(0, 3, ctx=parse_expr(ctx, vs), spec_expr=parse_expr(spec, vs))], name=ctx))


@pytest.mark.gpu
@pytest.mark.parametrize("ctx,spec,K", [
    ("(HOLE0*16)+HOLE1", "((i+2)*16)+(j*3)", (3, 5)),
    ("(HOLE0*3)-(HOLE1*i)", "((i/2)*3)-(j*i)", (3, 3)),                 # the factor of a part is zero at some points
    ("(HOLE0*(12/(i-3)))+HOLE1", "j", (3, 3)),                          # the context is undefined at some points
    (f"(HOLE0*{W})+HOLE1", f"((i*j)*{W})+i", (3, 3)),
    ("(HOLE0*0)+(HOLE1*0)", "0", (5, 3)),                               # more pairs pass than the list holds
])
def test_joint_search_from_one_side(xp, ctx, spec, K):
    g = free_grammar(IJ, [1, 2, 3, 16])
    sk = Sketch(g, [Hole(0, 1, spec_expr=parse_expr("i", IJ))], name=ctx)
    check_joint(xp, sk, JointHole((0, 0), K, parse_expr(ctx, IJ), spec_expr=parse_expr(spec, IJ)))


@pytest.mark.gpu
@pytest.mark.parametrize("n_sig", [1, 2, 9, 16])
def test_behaviour_tables_grow(xp, n_sig):
    """Two hundred thousand behaviours (nine and more signature points): the tables are enlarged between passes."""
    g = free_grammar(IJ, [1, 2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31])
    sk = Sketch(g, [Hole(0, 7, spec_expr=parse_expr("((i*5)+j)%7", IJ))], name="grow")
    check_behaviours(xp, sk, [(k * 7) % 81 for k in range(n_sig)])


@pytest.mark.gpu
@pytest.mark.parametrize("n", [3, 130])
def test_batch_load_in_pieces(xp, n):
    """Tables of some 10^4 points each: the staged copy spans several pieces; from 128 sketches on threads fill them.  Two
    grammars are shared, so one load sends a grammar's tables for all sketches of it."""
    vs = [Variable("i", 0, 256), Variable("j", 0, 64)]
    models = [free_grammar(vs, [1, 2, 3]), free_grammar(vs, [2, 5])]
    rng = np.random.default_rng(n)
    sks = []
    for k in range(n):
        points = int(rng.integers(1, 16000)) if k else 32768            # (the first: exactly the largest that is staged)
        coords = np.stack([rng.integers(0, 256, size=points), rng.integers(0, 64, size=points)], axis=1).astype(np.int32)
        a, b = coords[:, 0].astype(np.int64), coords[:, 1].astype(np.int64)
        sks.append(Sketch(models[k % 2], [Hole(0, 3, spec_table=[a + b, a * 2, a // 5, b - a][k % 4])], coords))
    grs = [xp.xp_grammar_create(m) for m in models]
    got = xp.xp_repair_batch(xp.xp_sketch_load_batch([grs[k % 2] for k in range(n)], sks))
    for k in range(n):
        assert_same(got[k][0], oracle.repair_hole(sks[k]), f"sketch {k}")


def test_integers_of_descriptors():
    """What the C structures take as an integer: no float, no text, unsigned 64-bit constants by their bits; and the first error is the one reported."""
    import array
    from paper_2505_02146_b200 import binding as B
    from xp_instances.model import Grammar, Production
    B.load()
    vs = [Variable("i", 0, 9)]
    big = free_grammar(vs, [2**63, 2**64 - 1, -2**63])
    d = B.marshal_grammar(big).desc
    assert [d.productions[k].value for k in (1, 2, 3)] == [-2**63, -1, -2**63]
    ok = [Production(0, 0, var=0), Production(0, 1, value=3)]
    for variables, prods in (([Variable("i", 0.0, 9)], ok), ([Variable("i", 0, "9")], ok), ([Variable("i", 0, 2.5)], ok), (vs, [Production(0, 1, value=1.5)]),
                             (vs, [Production(0, 1, value="7")]), (vs, [Production(0.0, 0)]), (vs, [Production(0, 0, var="0")]), (vs, [Production(0, 2, op=None)])):
        with pytest.raises(TypeError):
            B.marshal_grammar(Grammar(variables, 1, prods))
    with pytest.raises(OverflowError):
        B.marshal_grammar(free_grammar(vs, [2**64]))
    with pytest.raises(AttributeError, match="lo"):                     # (not a later one)
        B.marshal_grammar(Grammar([type("V", (), {"name": "i"})()], 1, [object()]))
    g = free_grammar(vs, [1])
    rows = np.zeros((3, 1), dtype=np.int32)
    for hole, coords in ((Hole(0, 3, ctx=None, spec_expr=parse_expr("i", vs)), None), (Hole(0, 3), None), (Hole(0, 3.0, spec_expr=parse_expr("i", vs)), None),
                         (Hole(0, 3, spec_table=array.array("q", [1, 2, 3])), rows), (Hole(0, 3, spec_expr=[(1, 0, 1.0)]), None)):
        with pytest.raises((TypeError, AttributeError)):
            B.marshal_sketches([Sketch(g, [hole], coords)])


@pytest.mark.parametrize("bad", ["kind", "pair", "value", "attr"])
def test_descriptors_from_models(bad):
    """Integers of any kind, arrays of other types and strides, and what is refused."""
    from paper_2505_02146_b200 import binding as B
    B.load()
    g = free_grammar([Variable("i", np.int64(0), np.int32(9))], [np.int64(-5), 1])
    made = B.marshal_grammar(g)
    d = made.desc
    assert (d.n_vars, d.vars[0].name, d.vars[0].hi, d.n_productions) == (1, b"i", 9, 8)
    assert [d.productions[k].value for k in range(3) if d.productions[k].kind == 1] == [-5, 1]
    wide = np.arange(40, dtype=np.int64).reshape(10, 4)[::2, :1]
    spec = np.arange(10, dtype=np.int16)[::2]
    descs, nhs, keep = B.marshal_sketches([Sketch(g, [Hole(0, 3, ctx=parse_expr("HOLE+i", g.variables), spec_table=spec)], wide)])
    assert nhs == [1] and descs[0].n_points == 5 and descs[0].holes[0].ctx_len == 3
    assert list((C.c_int32 * 5).from_address(descs[0].coords)) == [0, 8, 16, 24, 32]
    assert list((C.c_int64 * 5).from_address(descs[0].holes[0].spec_table)) == [0, 2, 4, 6, 8]
    hole = Hole(0, 3, spec_expr={"kind": [("x", 0, 0)], "pair": [(0, 0)], "value": [(0, 0, 2**70)], "attr": [7]}[bad])
    with pytest.raises((TypeError, ValueError, OverflowError)):
        B.marshal_sketches([Sketch(g, [hole])])


@pytest.mark.gpu
@pytest.mark.parametrize("holes,points", [(40, 32768), (1200, 0)])
def test_a_first_share_larger_than_a_piece(xp, holes, points):
    """One sketch whose share of the staged copy (host tables of 256 KB each, or a thousand hole records) is larger than a
    piece: the lists in front of it travel with it."""
    g = free_grammar(IJ, [1, 2])
    specs = ["i+j", "i*2", "j-1", "2-i", "i/2", "j%2", "i"]
    if points:
        rng = np.random.default_rng(points)
        coords = np.stack([rng.integers(0, 200, size=points), rng.integers(-30, 30, size=points)], axis=1).astype(np.int32)
        i, j = coords[:, 0].astype(np.int64), coords[:, 1].astype(np.int64)
        tables = [i + j, i * 2, j - 1, 2 - i, i // 2, np.fmod(j, 2), i]
        sk = Sketch(g, [Hole(0, 3, spec_table=tables[h % 7]) for h in range(holes)], coords)
    else:
        sk = Sketch(g, [Hole(0, 3, spec_expr=parse_expr(specs[h % 7], IJ)) for h in range(holes)])
    want = [oracle.repair_hole(sk, h) for h in range(7)]
    got = xp.xp_repair(xp.xp_sketch_load(xp.xp_grammar_create(g), sk))
    for h in range(holes):
        assert_same(got[h], want[h % 7], f"hole {h}")


@pytest.mark.gpu
def test_one_sketch_under_both_plans_from_several_threads(xp):
    """xp_repair may take blocks to the pair join, xp_repair_static and a batch of more than eight sketches may not: two plans of
    one sketch, used in turn and at the same time."""
    g = free_grammar(IJ, list(range(0, 12)) + [65536])
    load = lambda spec: xp.xp_sketch_load(xp.xp_grammar_create(g), Sketch(g, [Hole(0, 7, spec_expr=parse_expr(spec, IJ))]))
    ls, others = load("(i*3)+(j*2)"), [load("i+j") for _ in range(8)]
    ref = xp.xp_repair(ls)[0]
    key = lambda r, K=7: ([int(c) for c in r.match_count][:K + 1], r.least_size, int(r.least_rank))
    calls = [lambda: key(xp.xp_repair(ls)[0]), lambda: key(xp.xp_repair_static(ls)[0]), lambda: key(xp.xp_repair_batch([ls] + others)[0][0])]
    for _ in range(3):
        for call in calls:
            assert call() == key(ref)
    bad = []

    def work(call):
        for _ in range(40):
            r = call()
            if r != key(ref):
                bad.append(r)
    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def run_on_host(tmp_path, name, body):
    """Compiles and runs a C++ program over the structures and rules that host and kernels share."""
    src, exe = tmp_path / f"{name}.cpp", tmp_path / name
    src.write_text('#include <cstdio>\n#include "xp_dev.h"\nusing namespace xp;\n' + body)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "paper_2505_02146_b200", "csrc"), "-I" + os.path.join(ROOT, "include"),
                           "-I/usr/local/cuda/include", str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert (r.returncode, r.stdout) == (0, "")


def test_least_number_with_two_residues(tmp_path):
    run_on_host(tmp_path, "residues", r"""
static u64 plain(u64 u0, u64 u1, u64 t0, u64 t1) { for (u64 k = 0; k < u1; ++k) if ((t0 + u0 * k) % u1 == t1) return t0 + u0 * k; return ~0ull; }
static bool same(u32 u0, u32 u1, u32 t0, u32 t1) {
    if (residue_least(u0, u1, t0, t1) == plain(u0, u1, t0, t1)) return true;
    printf("%u %u %u %u\n", u0, u1, t0, t1);
    return false;
}
int main() {
    for (u32 u0 = 1; u0 < 26; ++u0) for (u32 u1 = 1; u1 < 26; ++u1)
        for (u32 t0 = 0; t0 < u0; ++t0) for (u32 t1 = 0; t1 < u1; ++t1) if (!same(u0, u1, t0, t1)) return 1;
    const u32 big = 0x7fffffffu;
    u64 x = 1;
    auto next = [&]() { x = x * 6364136223846793005ull + 1442695040888963407ull; return (u32)(x >> 33); };
    for (int n = 0; n < 2000; ++n) {
        const u32 u1 = 1 + next() % 3000, f = 1 + next() % 40, u0 = n % 3 ? 1 + next() % (big - 1) : u1 * f;
        if (!same(u0, u1, next() % u0, next() % u1)) return 1;
        const u32 v0 = 1 + next() % (big - 1), v1 = 1 + next() % (big - 1), m = next();      // m itself is one: the least is no larger, and has its residues
        const u64 l = residue_least(v0, v1, m % v0, m % v1);
        if (l > m || l % v0 != m % v0 || l % v1 != m % v1) { printf("%u %u of %u\n", v0, v1, m); return 1; }
    }
    return 0;
}
""")


def test_the_list_of_long_walks_holds_every_piece(tmp_path):
    """Division kernel of the pair join: all walks together never list more pieces than the list has room for (nor than 32
    bits count), and the pieces of a walk cover it."""
    run_on_host(tmp_path, "walks", r"""
int main() {
    const u32 sizes[] = {1, 31, 32, 33, 63, 64, 65, 129, 1125, 9245, 92480, 3150592, 1u << 22};
    for (u32 nl : sizes) for (u32 nr : sizes) {
        const u32 pieces = pair_pieces(nl, nr);
        const u64 room = pair_list_entries(nl, nr);
        const u32 spans[] = {1, 2, 31, 32, 33, 63, 64, 65, 96, 97, nr / 3 + 1, nr / 2 + 1, nr - nr / 7, nr - 1, nr};
        u64 most = 0;
        for (u32 span : spans) {
            if (span < 1 || span > nr) continue;
            const u32 piece = pair_piece(span, pieces), more = span > piece ? (span - 1) / piece : 0;
            if (piece < kPairWalk || piece % 32 || (u64)more * piece >= span || (u64)(more + 1) * piece < span) { printf("%u %u span %u piece %u\n", nl, nr, span, piece); return 1; }
            if (more > most) most = more;
        }
        if (!pair_fits(0, kPairShort) || !pair_fits(kPairShort, 0) || pair_fits(kPairShort, 1) || pair_fits(5, kPairShort - 4) || pair_fits(~0u, 7)) return 2;
        if (kPairShort + 2ull * ((nl + 31) / 32) * most > room || room >> 31) { printf("%u %u: %llu in %llu\n", nl, nr, 2ull * ((nl + 31) / 32) * most, room); return 1; }
    }
    return 0;
}
""")


@pytest.mark.gpu
@pytest.mark.parametrize("spec", ["((k*13)+i)/60", "(i+(k*9))%37", "(i/50)+(k/7)"])
def test_walks_of_small_targets(xp, spec):
    """A small target at the first probe leaves most divisors open: walks of 92 480 divisors.  Against the operand tiles,
    which a batch of more than eight sketches keeps to, and the oracle in windows."""
    vs = [Variable("i", 0, 64), Variable("j", 0, 256), Variable("k", 0, 8)]
    g = free_grammar(vs, constant_set(-64, 64, [128, 256, 512, 1024]))
    sk = Sketch(g, [Hole(0, 7, spec_expr=parse_expr(spec, vs))], name=spec)
    n = oracle.counts(g, 0, 7)
    load = lambda s: xp.xp_sketch_load(xp.xp_grammar_create(s.grammar), s)
    ls = load(sk)
    small = free_grammar(IJ, [1])
    others = [load(Sketch(small, [Hole(0, 3, spec_expr=parse_expr("i+j", IJ))])) for _ in range(8)]
    at = 3 * n[7] // 5 + n[1] * n[5]                                     # the first quotient of two operands of three nodes
    kw = dict(rank_ranges=[(0, 7, at, at + 300_000_000)], size_min=7)
    a, b = xp.xp_repair(ls)[0], xp.xp_repair_batch([ls] + others)[0][0]
    assert (a.match_count, a.least_size, a.least_rank) == (b.match_count, b.least_size, b.least_rank)
    a, b = xp.xp_repair(ls, **kw)[0], xp.xp_repair_batch([ls] + others, **kw)[0][0]
    assert (a.match_count, a.solved, a.least_rank) == (b.match_count, b.solved, b.least_rank)
    check_sketch(xp, sk, windows={7: (at + 12_345_678, at + 13_345_678)})


@pytest.mark.gpu
def test_cancel_word_and_time_limit_between_two_operands_of_three_nodes(xp):
    """450 000 operands of three nodes a side: blocks that the pair join takes whole, unless a call wants to be stopped."""
    vs = [Variable("i", 0, 64), Variable("j", 0, 256), Variable("k", 0, 8)]
    g = free_grammar(vs, constant_set(-148, 148))
    n = oracle.counts(g, 0, 7)
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), Sketch(g, [Hole(0, 7, spec_expr=parse_expr("((i*13)+j)+(k*5)", vs))]))
    blocks = dict(rank_ranges=[(0, 7, n[7] // 5 + n[1] * n[5], n[7] // 5 + n[1] * n[5] + n[3] * n[3])], size_min=7)
    with pytest.raises(xp.XpError) as e:
        xp.xp_repair(ls, timeout_ms=3, **blocks)
    assert e.value.status == 7
    word = C.c_int32(0)
    threading.Timer(0.005, lambda: setattr(word, "value", 1)).start()
    t0 = time.perf_counter()
    with pytest.raises(xp.XpError) as e:
        xp.xp_repair(ls, cancel=word, **dict(blocks, rank_ranges=None))
    assert e.value.status == 8 and "between launches" in str(e.value) and time.perf_counter() - t0 < 2.0
    a, b = xp.xp_repair(ls, cancel=C.c_int32(0), timeout_ms=60_000, **blocks)[0], xp.xp_repair(ls, **blocks)[0]
    assert (a.match_count, a.least_rank) == (b.match_count, b.least_rank) and a.n_launches > b.n_launches


@pytest.mark.gpu
def test_a_workspace_made_before_a_refinement(xp):
    """Products of two operands of three nodes go to the pair join where no target is zero.  Here every sampled point but the
    first wants 0; the points that end the survivors want 5 and become probes, and the search needs more scratch than before."""
    import torch
    vs = [Variable("a", 0, 9), Variable("b", 0, 9)]
    g = free_grammar(vs, constant_set(1, 40), ops=["*"])
    coords = np.zeros((6000, 2), dtype=np.int32)
    coords[:, 1] = np.arange(6000) % 7
    coords[0] = (2, 3)
    spec = np.zeros(6000, dtype=np.int64)
    spec[0] = 6
    spec[100:106] = 5
    sk = Sketch(g, [Hole(0, 7, spec_table=spec)], coords)
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), sk)
    flag = dict(flags=xp.XP_FLAG_ALWAYS_PAIR)                          # (a block this small goes to the tiles)
    need = xp.xp_workspace_bytes([ls], **flag)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    before = xp.xp_repair(ls, workspace=ws, **flag)[0]
    assert before.probe_survivors > 0 and xp.xp_sketch_refine(ls) >= 1
    assert xp.xp_workspace_bytes([ls], **flag) > need                           # (or this test does not test what it says)
    assert_same(xp.xp_repair(ls, workspace=ws, **flag)[0], before)
    assert_same(xp.xp_repair(ls, **flag)[0], before)
    assert_same(xp.xp_repair(ls, workspace=ws[:need - 40 * (2**20 - 65536)], **flag)[0], before)      # (with the shortest survivor queue)
    with pytest.raises(xp.XpError) as e:                                # too small for any plan: refused as ever
        xp.xp_repair(ls, workspace=ws[:1 << 20], **flag)
    assert e.value.status == 5


@pytest.mark.gpu
def test_more_operands_than_32_bits_count(xp):
    """The plan of a search does not grow with the number of its operands (4e14 of size 9 here), and a warp that passes 2^32
    operands of a segment loses none: 1.1e10 operands against the same in five windows."""
    vs = [Variable("i", 0, 64), Variable("j", 0, 256), Variable("k", 0, 8)]
    g = free_grammar(vs, constant_set(-64, 64, [128, 256, 512, 1024]))
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), Sketch(g, [Hole(0, 11, spec_expr=parse_expr("(i*13)+j", vs))]))
    assert xp.xp_workspace_bytes([ls], size_min=11) < (40 * 2**20) + (1 << 20)      # (40 bytes for each of 2^20 survivors; 190 000 segments took 20 MB)
    with pytest.raises(xp.XpError) as e:
        xp.xp_repair(ls, timeout_ms=20, size_min=11)
    assert e.value.status == 7
    g = free_grammar(vs, constant_set(-31, 30))
    n = oracle.counts(g, 0, 9)
    sk = Sketch(g, [Hole(0, 9, spec_expr=parse_expr("i+((j*7)%(i+3))", vs))])
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), sk)
    run = lambda b, e: xp.xp_repair(ls, rank_ranges=[(0, 9, b, e)], size_min=9)[0]
    cuts = [n[7] * k // 5 for k in range(6)]                            # i + (every operand of size 7)
    parts = [run(b, e) for b, e in zip(cuts, cuts[1:])]
    whole = run(0, n[7])
    assert n[7] > 2 * 2**32 and whole.match_count[9] == sum(p.match_count[9] for p in parts) > 0
    assert whole.least_rank == min(p.least_rank for p in parts if p.solved) > 2**32


@pytest.mark.gpu
@pytest.mark.parametrize("factor", ["3000000000", "-3000000001", "2147483648", "3221225472", "4294967296", "8589934593", "5497558138880",
                                    "4611686018427387904", "-9223372036854775808", "9223372036854775807", "i", "(i-4)", "(j*1048576)"])
def test_factors_of_the_context(xp, factor):
    """Odd and even factors beyond 31 bits (even ones leave more than one hole value open modulo 2^64), and factors that are zero
    at some of the points: leaf join, pair join and tiles against the oracle."""
    c = [0, 1, 2, 3, 5, 7, -1, -4, 65536]
    for g, size, spec in ((free_grammar(IJ, constant_set(-20, 20) + [65536, 2**31 - 1]), 5, "(i*7)+j"), (free_grammar(IJ, c), 5, "(i/3)-(j%5)"),
                          (free_grammar(IJ, list(range(0, 12)) + [65536]), 7, "(i*3)+(j*2)")):
        sk = Sketch(g, [Hole(0, size, ctx=parse_expr(f"(HOLE*{factor})+(j*3)", IJ), spec_expr=parse_expr(f"(({spec})*{factor})+(j*3)", IJ))], name=f"{factor} {spec}")
        n = oracle.counts(g, 0, size)[size]
        if size == 5:
            check_sketch(xp, sk)
        else:
            check_sketch(xp, sk, windows={7: (n // 2 - 300_000, n // 2 + 300_001), 5: (3, 400_000)})


@pytest.mark.gpu
@pytest.mark.parametrize("consts,ops,ctx,spec", [
    (list(range(0, 18)), ["+", "*", "<<", ">>"], "", "((i<<3)+j)*2"),
    (list(range(0, 17)) + [63, 64, -1], ["-", "%", "<<", ">>"], "", "(i<<2)-(j>>1)"),
    (list(range(1, 18)) + [W], "+-*/%", "", f"((i*{W})+j)-3"),
    (list(range(1, 18)) + [W, 2**31 - 1, -2**31], "+-*/%", "(HOLE*3)+i", f"(j*{W})/5"),
    (list(range(1, 18)) + [2**31 - 1], "+-*/%", "", "(i*2147483647)+(j*3)"),      # narrow leaves, wide operands
    (list(range(1, 18)) + [2**31 - 1, 1000003], "%+*-/", "", "1000003%((i*37)+(j+90))"),     # residues of large constants
    (list(range(1, 18)) + [2**30], ["+", "-", "*", "min", "max", "/"], "", "(i*1073741824)/(j+7)"),
    (list(range(0, 18)) + [W], ["+", "-", "<<"], "j<HOLE", "i-2"),
])
def test_many_operands_in_the_exact_form(xp, consts, ops, ctx, spec):
    """Some 4e5 operands of size 5: shifts, leaves and operands of 2^31 or more, 32 at a time; windows at the first block of each
    production, across the end of its blocks with a leaf on the left, and at its end."""
    g = free_grammar(IJ, consts, ops=list(ops))
    text = ctx.replace("HOLE", f"({spec})") if ctx else spec
    sk = Sketch(g, [Hole(0, 7, ctx=parse_expr(ctx, IJ) if ctx else [], spec_expr=parse_expr(text, IJ))], name=text)
    n = oracle.counts(g, 0, 7)
    per = n[7] // len(ops)
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), sk)
    for p in range(len(ops)):
        for at in (p * per, p * per + n[1] * n[5] - 100_000, (p + 1) * per - 200_000):
            w = (max(at, 0), min(at + 200_000, n[7]))
            got = xp.xp_repair(ls, rank_ranges=[(0, 7, *w)], size_min=7)[0]
            want = oracle.repair_hole(sk, rank_ranges={1: (0, 0), 3: (0, 0), 5: (0, 0), 7: w})
            assert (got.match_count[7], got.solved) == (want.match_count[7], want.solved), w
            assert not want.solved or (got.least_rank, got.least_text) == (want.least_rank, want.least_text)


@pytest.mark.gpu
def test_more_survivors_than_the_queue_of_a_small_workspace_holds(xp):
    """A workspace made for 65 536 survivors, as callers have had, is taken with what it holds: the warps check the others themselves."""
    import torch
    vs = [Variable("i", 0, 16), Variable("j", 0, 16)]
    g = free_grammar(vs, constant_set(-12, 12))
    sk = Sketch(g, [Hole(0, 5, spec_expr=parse_expr("0", vs))])
    ls = xp.xp_sketch_load(xp.xp_grammar_create(g), sk)
    want = oracle.repair_hole(sk)
    assert want.match_count[5] > 65536
    need = xp.xp_workspace_bytes([ls])
    small = need - 40 * (2**20 - 65536)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    for size in (need, small + 1_000_000, small):
        assert_same(xp.xp_repair(ls, workspace=ws[:size])[0], want, f"{size} bytes")
    assert_same(xp.xp_repair(ls)[0], want)
    with pytest.raises(xp.XpError) as e:
        xp.xp_repair(ls, workspace=ws[:small - 256])
    assert e.value.status == 5


@pytest.mark.gpu
@pytest.mark.parametrize("spec", ["(i*3)+(j*2)", "(i+2)*(j-1)", "(i*5)/(j+4)", "(i+j)%(j+5)", "j-j", "(i*1048576)*(j*65536)"])
def test_indexed_operands_in_rank_windows(xp, spec):
    """The pair join of blocks that a window cuts to some of their left operands, small ones too."""
    g = free_grammar(IJ, list(range(0, 12)) + [65536])
    sk = Sketch(g, [Hole(0, 7, spec_expr=parse_expr(spec, IJ))], name=spec)
    n = oracle.counts(g, 0, 7)
    flag = dict(flags=xp.XP_FLAG_ALWAYS_PAIR)
    per, mid = n[7] // 5, n[1] * n[5]                                   # a production's first pair of two operands of three nodes
    for p in range(5):
        at = p * per + mid
        check_sketch(xp, sk, windows={7: (at + 5 * n[3] + 17, at + 9 * n[3] + 3), 5: (3, 40_000)}, **flag)
    check_sketch(xp, sk, windows={7: (per + mid + 1000 * n[3] + 5, 2 * per + mid + 100 * n[3])}, **flag)      # ends of one block, starts of the next
    check_sketch(xp, sk, windows={7: (0, 100_000)}, **flag)


@pytest.mark.gpu
@pytest.mark.parametrize("ctx,spec", [("j<HOLE", "i*2"), ("HOLE<=(i-j)", "(i%7)-3"), ("(j-HOLE)<4", "i/3")])
def test_many_operands_under_a_comparison(xp, ctx, spec):
    """Operand tiles with a leaf on either side, for a hole whose context compares."""
    g = free_grammar(IJ, list(range(-6, 11)))
    sk = Sketch(g, [Hole(0, 7, ctx=parse_expr(ctx, IJ), spec_expr=parse_expr(ctx.replace("HOLE", f"({spec})"), IJ))], name=ctx)
    n = oracle.counts(g, 0, 7)
    assert n[5] > 2**18
    whole = xp.xp_repair(xp.xp_sketch_load(xp.xp_grammar_create(g), sk), size_min=7, size_max=7)[0]
    assert whole.n_launches == 2                                        # tiles and the whole-domain check, no leaf join
    for p in range(5):
        at = p * (n[7] // 5)
        check_sketch(xp, sk, windows={1: (0, 0), 3: (0, 0), 5: (0, 0), 7: (at + 7, at + 100_000)})
    check_sketch(xp, sk, windows={1: (0, 0), 3: (0, 0), 5: (0, 0), 7: (n[7] - 100_000, n[7])})


@pytest.mark.gpu
def test_threads_that_load_the_same_new_grammars(xp):
    """Two grammars that nobody has loaded yet, in batches that name them in either order, from six threads at once: each load finds the
    tables in place, and none waits for another for good."""
    vs = [Variable("i", 0, 50), Variable("j", 0, 40)]
    models = [free_grammar(vs, [1, 2, 3]), free_grammar(vs, [2, 5])]
    rng = np.random.default_rng(1)
    coords = np.stack([rng.integers(0, 50, size=9000), rng.integers(0, 40, size=9000)], axis=1).astype(np.int32)
    table = coords[:, 0].astype(np.int64) * 2 + coords[:, 1]
    sks = [Sketch(m, [Hole(0, 5, spec_table=table)], coords) for m in models]
    want = [oracle.repair_hole(s) for s in sks]
    for _ in range(8):
        grs = [xp.xp_grammar_create(m) for m in models]
        got, failed = [], []

        def work(k):
            try:
                order = [k % 2, 1 - k % 2, k % 2]
                for which, r in zip(order, xp.xp_repair_batch(xp.xp_sketch_load_batch([grs[o] for o in order], [sks[o] for o in order]))):
                    got.append((which, r[0]))
            except Exception as e:      # noqa: BLE001
                failed.append(e)
        threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
        for t in threads:
            t.start()
        for t in threads:
            t.join(60)
        assert not failed and len(got) == 18
        for which, r in got:
            assert_same(r, want[which])
