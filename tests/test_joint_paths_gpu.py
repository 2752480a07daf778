"""The joint search where it changes form: a part above 65 536 candidates (a lane per candidate instead of sixteen), and more
listed pairs than a CTA each is worth (a warp per pair)."""
import pytest

import oracle
from xp_instances import Hole, JointHole, Sketch, Variable, constant_set, free_grammar, parse_expr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extents,consts,K,ctx,spec", [
    ((9, 7), constant_set(-20, 95), (3, 1), "(HOLE0*5)+HOLE1", "((i*3)*5)+j"),       # 118 leaves: 69 738 candidates of part 0
    ((9, 7), constant_set(-20, 95), (1, 3), "(HOLE0*5)+HOLE1", "(i*5)+(j%4)"),       # ... of part 1
    ((33, 31), constant_set(-8, 10), (3, 3), "(HOLE0*0)+HOLE1", "j+2"),              # every candidate of part 0 with every match of part 1
    ((33, 31), constant_set(-8, 10), (3, 3), "HOLE0-HOLE1", "i-j"),
])
def test_forms_of_the_joint_search(xp, extents, consts, K, ctx, spec):
    vs = [Variable("i", 0, extents[0]), Variable("j", 0, extents[1])]
    g = free_grammar(vs, consts)
    sk = Sketch(g, [Hole(0, 1, spec_expr=parse_expr("i", vs))])
    J = JointHole((0, 0), K, parse_expr(ctx, vs), spec_expr=parse_expr(spec, vs))
    want = oracle.repair_joint(sk, J)
    got = xp.xp_repair_joint(xp.xp_sketch_load(xp.xp_grammar_create(g), sk), J)
    assert got.cand_count == want.cand_count and got.match_count == want.match_count
    assert want.solved and got.solved
    assert (got.least_total, got.least_size0, got.least_rank0, got.least_rank1) == (want.least_total, want.least_size0, want.least_rank0, want.least_rank1)
