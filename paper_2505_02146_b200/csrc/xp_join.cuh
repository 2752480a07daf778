// The leaf join: candidates  E op leaf  and  leaf op E, decided from the operand's side.
//
// Nearly all candidates of a search have a leaf as one operand of their root (a free grammar of 136 leaves at size 7:
// four in five; the typed grammar with 257 multipliers and 128 divisors at size 9: 97 %).  Testing them one by one costs
// operands x leaves x operators.  Here a thread computes an operand's values (a0, a1) at two probes and asks per operator
// for which leaves the result can be the target (t0, t1) at both:
//   constants c have ONE value at both probes, so
//     a + c = t   needs  a0 - a1 = t0 - t1, and c = t0 - a0 in the constants' range       (a - c and c - a likewise);
//     a * c = t   needs  a0 * t1 = a1 * t0;
//     a / c = t   needs  an integer |c| in (|a|/(|t|+1), |a|/|t|] at both probes          (single precision, widened);
//     c / a = t   needs  |c| in [|t||a|, (|t|+1)|a|) at both;
//     a % c = t   needs  |c| to divide |a| - |t| at both and to exceed the target at EVERY probe (a greatest common divisor);
//     c % a = t   needs  |c| = |t| mod |a| at both (stepping through the few such |c|);
//     min, max    need   c = t0 or c = t1, or a itself to be the target at both;
//   variables (and constants when a nonterminal has four or fewer) are entries tested one by one, at both probes.
// These are necessary conditions in 32-bit arithmetic for operands below JoinSet::lim in magnitude.  An operand that passes
// one (a suspect) waits in the warp's first queue until 32 have gathered; then every lane takes one, finds the leaves its
// conditions leave open (binary search among the sorted constants) and holds each against both probes.  What is left
// goes to a second queue, and 32 at a time (a lane each, none idle) are checked exactly, in 64 bits, at the other probes.
// A context that compares asks for an interval of values at every probe.  Every operator but % is monotone in a constant
// (on either side of zero, for a / c): its constants are one or two runs, the intersection of the probes' intervals
// (range_runs); remainders are tested constant by constant at the first probe with reciprocals.
// Operands of JoinSet::lim or more, leaf sets with a wider leaf and shifts take the exact form, in 64 bits: 32 operands at a time, a
// lane each (they too wait in a queue), or, where a segment has few operands, one at a time, lanes over the leaves.
// Warps work on their own; nothing here waits for another warp.
//
// This file is compiled twice.  XP_JOIN_BATCH: the form for batches without classes or tickets in parts.  Such a call has warps enough at
// work to hide a check's chain, and waits for instructions instead: everything that only shortens the chain (probes side by side, several a step,
// operators side by side) or serves classes is left out of it (search of 40 sketches 0.23 ms with it, 0.20 without; of 1024 3.97, 3.76).
namespace xp {
#undef XP_CLASSES
#if XP_JOIN_BATCH
#define XP_CLASSES(seg) 0
namespace join_batch {
#else
#define XP_CLASSES(seg) (seg).classes
namespace join_full {
#endif

constexpr int kJoinThreads = 256;
constexpr int kJoinWarps = kJoinThreads / 32;
constexpr int kJoinP = 4;                                 // operands per lane and step
constexpr u32 kJoinQueue = 32 + 32 * kJoinP;              // suspects: fewer than 32 wait when a step adds up to 32 per operand of a lane

// What the conditions need of one group (leaf set) of the segment at hand.
struct GroupCtx {
    u32 cf, cs, ef, es;                                   // operators whose condition can hold: constants, entries; forward, swapped
    i32 cmin, cmax;
    u32 cabs, mm;
    float fc;
    i32 n_entries;
    const JoinSet* set;
};

// What the conditions need of the hole.
struct JoinCtx {
    u32 t0, t1, ut0, ut1;                                 // targets (low words) and their magnitudes (0 where 31 bits do not hold them)
    float rt0, rt1, rl0, rl1, h0, h1, ft0, ft1;           // 1/|t|, 1/(|t|+1), huge where t = 0, |t|
    u32 tmod;
    bool tz, small;                                       // both targets are zero; both are below 2^31
};

// The entries of all groups as the hot loop tests them (an operand that passes a test of any group is a suspect): sums,
// differences and products share one comparison each of a mixed pair, three comparisons per variable instead of ten.
constexpr int kJoinLin = 3 * kJoinEntries * 2;            // most wanted pairs kept (more: the exact form)
constexpr u32 kPairMix = 0x9E3779B1u;                     // a pair (x, y) is compared as x + kPairMix * y
struct __align__(16) JoinHot {
    u32 lin[kJoinLin + 4];                                // a + v, a - v, v - a: the pair that a has to be, mixed
    u32 mul0[kJoinEntries], mul1[kJoinEntries];           // a * v: a0 * mul0 + a1 * mul1 has to be mul_t
    u32 mul_t;
    i32 n_lin, n_mul, n_other, n_set;
    const JoinEntry* other[kJoinEntries];                 // entries under / % min max, with their operators
    u32 other_f[kJoinEntries], other_s[kJoinEntries];
    i32 set[kJoinGroups];                                 // groups whose constants have a condition
    u32 lim;                                              // operand limit of the segment (0: some leaf set goes the exact way)
    u32 tests;                                            // what an operand counts for in filter_tests
    u64 pairs;                                            // candidates per operand
};

struct JoinWarp {
    JoinHot hot;
    JoinCtx x;
    i32 seg;                                              // segment that grp, x and hot are filled for (-1: none)
    u64 base;                                             // operand that the queues' numbers count from
    u32 q_off[kJoinQueue];                                // suspects: operand number relative to `base`,
    i32 q_a0[kJoinQueue], q_a1[kJoinQueue];               //   its values at the two probes
    u32 c_off[64], c_pos[64], c_code[64];                 // candidates: operand, leaf position, group << 8 | slot << 1 | swapped
    u32 w_off[kJoinQueue];                                // wide operands
    u32 nq, nc, nw;                                       // suspects, candidates and wide operands waiting (of segment `seg`)
    GroupCtx grp[kJoinGroups];
    CandShared cand;                                      // candidate of a whole-domain check that the warp does itself
};

// What a warp has counted for the accumulator it works on (the sums over lanes are taken when it moves on).
struct JoinCount { u64 evals; u64 tests, cands; u32 suspects, passes; };

// v = x op y in 64-bit semantics; false when undefined.  The lanes of a check have different operators, and a branch per operator had them take
// turns, each with a 64-bit division of its own: where both values are below 2^31 in magnitude every operator but the shifts is computed
// and one selected (two-variable nest 163 -> 159 us a call, expression pair 322 -> 317).
__device__ __forceinline__ bool op_value(int op, i64 x, i64 y, i64& v) {
#if XP_JOIN_BATCH
    return apply_op(op, x, y, v);
#else
    constexpr i64 kEdge = 1ll << 31;
    if (x > -kEdge && x < kEdge && y > -kEdge && y < kEdge && (op <= XP_OP_MOD || op == XP_OP_MIN || op == XP_OP_MAX)) {
        const i32 a = (i32)x, b = (i32)y, d = b ? b : 1, q = a / d, r = a - q * d;      // (no overflow: a is not -2^31)
        const i64 sum = x + (op == XP_OP_SUB ? -y : y);
        const i32 least = a < b ? a : b, most = a < b ? b : a;
        v = op <= XP_OP_SUB ? sum : op == XP_OP_MUL ? x * y : (i64)(op == XP_OP_DIV ? q : op == XP_OP_MOD ? r : op == XP_OP_MIN ? least : most);
        return b != 0 || (op != XP_OP_DIV && op != XP_OP_MOD);
    }
    return apply_op(op, x, y, v);
#endif
}

// An operand subtree by reference: a table entry, an operation on two table entries, or (mode 2) its rank.
struct OperandRef { i32 mode, op; u64 a, b; };

__device__ __forceinline__ OperandRef operand_ref(const GrammarDev* g, const HoleDev* hole, int nt, int size, u64 rank) {
    OperandRef r;
    r.op = 0; r.b = 0;
    const int tmax = hole->tab_max_size;
    if (size <= tmax) { r.mode = 0; r.a = hole->tab_off[nt][size] + rank; return r; }
    if (tmax >= 1 && size >= 3) {
        int lnt, rnt, a;
        u64 l, q;
        unrank_root(g, nt, size, rank, r.op, lnt, rnt, a, l, q);
        if (a <= tmax && size - 1 - a <= tmax) {
            r.mode = 1; r.a = hole->tab_off[lnt][a] + l; r.b = hole->tab_off[rnt][size - 1 - a] + q;
            return r;
        }
    }
    r.mode = 2; r.a = rank;
    return r;
}

__device__ __noinline__ bool ref_value_full(const GrammarDev* g, const HoleDev* hole, int nt, int size, u64 rank, int j, i64& v) {
    u32 code[kMaxSize];
    const int n = unrank(g, nt, size, rank, code);
    return eval_cand(code, n, g->leaves, hole->probe_pt[j], v);
}

__device__ __forceinline__ bool ref_value(const GrammarDev* g, const HoleDev* hole, const OperandRef& r, int nt, int size, int j, i64& v) {
    if (r.mode == 2) return ref_value_full(g, hole, nt, size, r.a, j, v);
    const u64 base = (u64)j * hole->tab_total;
    if (!XP_CHECKED(j < hole->tab_probes && r.a < hole->tab_total && r.b < hole->tab_total, kChkTable)) return false;
    if (!hole->tab_ok[base + r.a]) return false;
    v = hole->tab_val[base + r.a];
    if (r.mode == 0) return true;
    if (!hole->tab_ok[base + r.b]) return false;
    return op_value(r.op, v, hole->tab_val[base + r.b], v);
}

__device__ __forceinline__ u32 ref_vars(const HoleDev* hole, const OperandRef& r) {
    if (r.mode == 2) return 0xffu;                        // (always a safe answer)
    return (u32)hole->tab_vars[r.a] | (r.mode == 1 ? (u32)hole->tab_vars[r.b] : 0u);
}

// Does hole value v satisfy the constraint at probe j (one of the first n_exact)?
__device__ __forceinline__ bool probe_accepts(const HoleDev* hole, int j, i64 v) {
    if ((hole->aff_okmask >> j) & 1u) return (u64)v * hole->aff_Aj[j] + hole->aff_Bj[j] == (u64)hole->probe_spec[j];
    if (v > -(1ll << 62) && v < (1ll << 62)) return v >= hole->rng_lo[j] && v <= hole->rng_hi[j];
    return true;                                          // (a value of 2^62 or more is left to the whole-domain check)
}

__device__ __forceinline__ int op_of_slot(int slot) { return slot <= 4 ? slot : slot <= 6 ? slot - 5 + XP_OP_MIN : slot - 7 + XP_OP_SHL; }

// Candidates checked one by one look at the probes four at a time: their table entries lie in four places that nothing has
// touched before, and one probe after the other a candidate that passes 16 probes waits 16 times for memory (the direct
// tickets of a small search: 20.7 -> 18.6 us).  Candidates of the join mostly end at the next probe and keep the plain order.
constexpr int kProbeStep = 4;

// An operand's values at the probes j0 .. j0 + 3 (those below n); returns the mask of those it is defined at.
__device__ __forceinline__ u32 ref_value4(const GrammarDev* g, const HoleDev* hole, const OperandRef& r, int nt, int size, int j0, int n, i64 (&v)[kProbeStep]) {
    u32 ok = 0;
    if (r.mode == 2) {
#pragma unroll 1
        for (int k = 0; k < kProbeStep; ++k) {
            i64 x = 0;
            if (j0 + k < n && ref_value_full(g, hole, nt, size, r.a, j0 + k, x)) ok |= 1u << k;
#pragma unroll
            for (int q = 0; q < kProbeStep; ++q) if (q == k) v[q] = x;
        }
        return ok;
    }
    const u64 total = hole->tab_total;
    const bool in = XP_CHECKED(n <= hole->tab_probes && r.a < total && r.b < total, kChkTable);
    i64 y[kProbeStep];
#pragma unroll
    for (int k = 0; k < kProbeStep; ++k) {
        v[k] = 0; y[k] = 0;
        if (j0 + k < n && in) {
            const u64 at = (u64)(j0 + k) * total;
            ok |= (u32)(hole->tab_ok[at + r.a] != 0) << k;
            v[k] = hole->tab_val[at + r.a];
            if (r.mode == 1) { if (!hole->tab_ok[at + r.b]) ok &= ~(1u << k); y[k] = hole->tab_val[at + r.b]; }
        }
    }
    if (r.mode == 1) {
#pragma unroll 1
        for (int k = 0; k < kProbeStep; ++k) {
            i64 x = v[0], z = y[0];
#pragma unroll
            for (int q = 1; q < kProbeStep; ++q) if (q == k) { x = v[q]; z = y[q]; }
            if (((ok >> k) & 1u) && !op_value(r.op, x, z, x)) ok &= ~(1u << k);
#pragma unroll
            for (int q = 0; q < kProbeStep; ++q) if (q == k) v[q] = x;
        }
    }
    return ok;
}

// Do the values v at the probes j0 .. j0 + 3 (those below n) satisfy the constraint?
__device__ __forceinline__ bool probes_accept(const HoleDev* hole, int j0, int n, const i64 (&v)[kProbeStep]) {
    const u32 aff = hole->aff_okmask >> j0;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < kProbeStep; ++k) {
        if (j0 + k >= n) continue;
        const int j = j0 + k;
        if ((aff >> k) & 1u) ok = ok && (u64)v[k] * hole->aff_Aj[j] + hole->aff_Bj[j] == (u64)hole->probe_spec[j];
        else if (v[k] > -(1ll << 62) && v[k] < (1ll << 62)) ok = ok && v[k] >= hole->rng_lo[j] && v[k] <= hole->rng_hi[j];
    }
    return ok;
}

// The candidate (operand, leaf) at the probes that have tables, in order; the first failure ends it.
#if XP_JOIN_BATCH
__device__ __forceinline__
#else
__device__ __noinline__
#endif
bool exact_pair(const GrammarDev* g, const HoleDev* hole, const OperandRef& ref, int nt, int esize, i32 var, i64 cval,
                                           bool swap, int op, int from, int n_exact, u64& evals) {
    for (int j = from; j < n_exact; ++j) {
        ++evals;
        i64 a, v;
        if (!ref_value(g, hole, ref, nt, esize, j, a)) return false;
        const i64 c = var >= 0 ? hole->probe_pt[j][var] : cval;
        if (!op_value(op, swap ? c : a, swap ? a : c, v) || !probe_accepts(hole, j, v)) return false;
    }
    return true;
}

// The same four probes at a time, for holes whose context compares: their candidates have passed the first four already, mostly pass all the
// others, and one probe after the other waited 16 times for memory.
__device__ __noinline__ bool exact_pair4(const GrammarDev* g, const HoleDev* hole, const OperandRef& ref, int nt, int esize, i32 var, i64 cval,
                                         bool swap, int op, int from, int n_exact, u64& evals) {
    for (int j0 = from; j0 < n_exact; j0 += kProbeStep) {
        const int here = n_exact - j0 < kProbeStep ? n_exact - j0 : kProbeStep;
        evals += (u64)here;
        i64 v[kProbeStep];
        if (ref_value4(g, hole, ref, nt, esize, j0, n_exact, v) != (1u << here) - 1u) return false;
        bool ok = true;
#pragma unroll 1
        for (int k = 0; k < here; ++k) {
            i64 a = v[0], r = 0;
#pragma unroll
            for (int q = 1; q < kProbeStep; ++q) if (q == k) a = v[q];
            const i64 c = var >= 0 ? hole->probe_pt[j0 + k][var] : cval;
            ok = op_value(op, swap ? c : a, swap ? a : c, r) && ok;
#pragma unroll
            for (int q = 0; q < kProbeStep; ++q) if (q == k) v[q] = r;
        }
        if (!ok || !probes_accept(hole, j0, n_exact, v)) return false;
    }
    return true;
}

// The warp checks one candidate on the whole domain itself (the survivor queue is full).
__device__ __noinline__ void join_verify(CandShared& cand, const PlanDev& plan, const SketchDev* sk, const HoleDev* hole, int size, int acc, u64 rank,
                                         u32 vars, u64& evals) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane == 0) { stage_candidate(cand, sk, hole, size, rank); (void)proj_points(sk, hole, vars, &cand); }
    __syncwarp();
    i64 fail_pid = 0;
    const bool ok = check_points(cand, sk, hole, 0, proj_points(sk, hole, vars, nullptr), evals, &fail_pid);
    if (ok && lane == 0) {
        atomicAdd(&plan.acc[acc].match_count[size], 1ull);
        atomicMin(&plan.acc[acc].min_rank[size], rank);
    }
    __syncwarp();
}

// Candidates that passed the probes (one per lane at most) go to the survivor queue, or are checked
// by the warp.  Called by all 32 lanes together.
__device__ __forceinline__ void join_survive(CandShared& cand, const PlanDev& plan, const SketchDev* sk, const HoleDev* hole, const JoinSeg& seg,
                                             bool pass, u64 rank, u32 vars, JoinCount& n) {
    u32 m = __ballot_sync(0xffffffffu, pass);
    if (!m) return;
    n.passes += (u32)__popc(m);
#if XP_JOIN_BATCH
    const bool pending = pass && !push_survivor(plan, sk, hole, seg.sketch, seg.hole, seg.size, seg.acc, rank, vars);
    m = __ballot_sync(0xffffffffu, pending);
#else
    m = __ballot_sync(0xffffffffu, push_survivors(plan, sk, hole, seg.sketch, seg.hole, seg.size, seg.acc, pass, rank, vars));
#endif
    while (m) {
        const int src = __ffs((int)m) - 1;
        m &= m - 1;
        join_verify(cand, plan, sk, hole, seg.size, seg.acc, __shfl_sync(0xffffffffu, rank, src), __shfl_sync(0xffffffffu, vars, src), n.evals);
    }
}

// The candidates of the lanes with `pass` at the probes without tables (from n_exact on), rebuilt in full: a few one after the other with the
// probes over the lanes, many with a lane each.  (A lane by itself evaluated eight probes one after the other, and those without need
// once more: 50 us at the end of a search over 800 000 operands of five nodes: whole call 384 -> 349 us.)  Called by all lanes.
__device__ __noinline__ bool join_full_check(const GrammarDev* g, const HoleDev* hole, int size, bool pass, u64 rank, u64& evals) {
    const int lane = threadIdx.x & 31, n_exact = hole->n_exact, n_probe = hole->n_probe;
#if XP_JOIN_BATCH
    (void)lane; (void)n_exact; (void)n_probe;
    if (!pass) return false;
    u32 code[kMaxSize];
    const int n = unrank(g, hole->start_nt, size, rank, code);
    return probe_check(g, hole, code, n, evals, n_exact);
#else
    u32 m = __ballot_sync(0xffffffffu, pass);
    if (!m || n_exact >= n_probe) return pass;
    u32 code[kMaxSize];
    if (__popc(m) > 4) {
        if (!pass) return false;
        const int n = unrank(g, hole->start_nt, size, rank, code);
        return probe_check(g, hole, code, n, evals, n_exact);
    }
    u32 good = 0;
    for (; m; m &= m - 1) {
        const int src = __ffs((int)m) - 1, j = n_exact + lane;
        const int n = unrank(g, hole->start_nt, size, __shfl_sync(0xffffffffu, rank, src), code);
        bool ok = true;
        if (j < n_probe) {
            i64 h = 0;
            ++evals;
            ok = ((hole->probe_spec_ok >> j) & 1u) && eval_cand(code, n, g->leaves, hole->probe_pt[j], h) &&
                 ctx_matches(hole, hole->probe_pt[j], h, hole->probe_spec[j]);
        }
        if (__all_sync(0xffffffffu, ok)) good |= 1u << src;
    }
    return (good >> lane) & 1u;
#endif
}

// A member per lane (in: this lane has one): operand `member` of (nt, esize) under the leaf and operator of pos and code.  Called by all lanes.
__device__ __forceinline__ void join_member(CandShared& cand, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, bool in, u64 member, u32 pos,
                                         u32 code, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int swap = (int)(code & 1u), slot = (int)((code >> 1) & 15u);
    const JoinGroup& grp = plan.jgroups[seg.first_group + (int)(code >> 8)];
    bool ok = false;
    u64 rank = 0;
    u32 vars = 0;
    if (in) {
        const u64 nl = g->cnt[grp.leaf_nt][1], ne = g->cnt[seg.nt][seg.esize];
        rank = grp.base[swap][slot] + (swap ? (u64)pos * ne + member : member * nl + (u64)pos);
        ok = rank >= seg.rank_begin && rank < seg.rank_end &&
             XP_CHECKED(member < ne && (u64)pos < nl && rank < g->cnt[hole->start_nt][seg.size], kChkQueue);
    }
    if (hole->n_exact < hole->n_probe) ok = join_full_check(g, hole, seg.size, ok, rank, n.evals);
    if (ok) {
        const LeafDev lf = g->leaves[g->leaf_begin[grp.leaf_nt] + (int)pos];
        vars = ref_vars(hole, operand_ref(g, hole, seg.nt, seg.esize, member)) | (lf.var >= 0 ? 1u << lf.var : 0u);
    }
    join_survive(cand, plan, sk, hole, seg, ok, rank, vars, n);
}

// Candidates of a segment that counts by class, one per lane (pass: this lane has one, and it satisfies the probes with tables):
// every member of the class is a candidate of its own, 32 at a time over all lanes' members, or left to members_kernel.  Called by all lanes.
__device__ __noinline__ void join_members(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, bool pass, u64 e, u32 pos,
                                          u32 code, JoinCount& n) {
    if (!__any_sync(0xffffffffu, pass)) return;
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    u64 mine = pass ? class_operand(g, hole, seg.nt, seg.esize, e).members() : 0ull, incl, total;
    for (int listed = 0;; ++listed) {
        incl = mine;
        for (int o = 1; o < 32; o <<= 1) { const u64 v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
        total = __shfl_sync(0xffffffffu, incl, 31);
        if (listed || total <= member_own(plan)) break;
        if (list_members(plan, mine > 0u, mine, e, pos, code, (i32)(&seg - plan.jsegs))) mine = 0;
    }
    for (u64 k0 = 0; k0 < total; k0 += 32u) {
        const u64 k = k0 + (u64)lane < total ? k0 + (u64)lane : total - 1u;
        int src = 0;                                      // the lane whose member this is: the first with incl > k
        for (int step = 16; step > 0; step >>= 1) { const u64 v = __shfl_sync(0xffffffffu, incl, src + step - 1); if (v <= k) src += step; }
        const u64 before = __shfl_sync(0xffffffffu, incl, src ? src - 1 : 0), e2 = __shfl_sync(0xffffffffu, e, src);
        const u32 pos2 = __shfl_sync(0xffffffffu, pos, src), code2 = __shfl_sync(0xffffffffu, code, src);
        const bool in = k0 + (u64)lane < total;
        join_member(w.cand, plan, seg, sk, hole, in, in ? class_operand(g, hole, seg.nt, seg.esize, e2).rank(src ? k - before : k) : 0ull, pos2, code2, n);
    }
}

// The candidates in the warp's second queue: the probes from `from` on, exactly.  Up to four, what a warp leaves a segment or a small call with,
// have their probes side by side in 16 lanes each; more take a lane each and, in a call of one wave, which waits for this chain, and for
// contexts that compare, four probes a step (exact_pair4).  A member's values are its class's: one check serves for all of them.  Called by all lanes.
__device__ __noinline__ void join_check(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, int from, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const u32 nc = w.nc;
    const int n_exact = hole->n_exact;
    const bool classes = XP_CLASSES(seg) != 0, four = !XP_JOIN_BATCH && (!hole->aff_ok || plan.n_join <= (u64)gridDim.x * kJoinWarps);
    for (u32 at = 0; at < nc; at += 32) {
        const bool spread = !XP_JOIN_BATCH && nc - at <= 4u;
        u32 good = 0;                                     // spread: bit i: candidate i passes
        bool pass = false;
        u64 rank = 0, e = 0;
        u32 vars = 0, code = 0, pos = 0;
#pragma unroll 1
        for (u32 i0 = 0; i0 < (spread ? nc - at : 1u); i0 += 2u) {
            const u32 i = spread ? i0 + (u32)(lane >> 4) : (u32)lane;
            bool ok = at + i < nc;
            if (ok) {
                code = w.c_code[at + i]; pos = w.c_pos[at + i]; e = w.base + w.c_off[at + i];
                const int swap = (int)(code & 1u), slot = (int)((code >> 1) & 15u), op = op_of_slot(slot);
                const JoinGroup& grp = plan.jgroups[seg.first_group + (int)(code >> 8)];
                const u64 nl = g->cnt[grp.leaf_nt][1], ne = g->cnt[seg.nt][seg.esize];
                const u64 first = classes ? class_operand(g, hole, seg.nt, seg.esize, e).rank(0) : e;
                rank = grp.base[swap][slot] + (swap ? (u64)pos * ne + first : first * nl + (u64)pos);
                ok = (classes || (rank >= seg.rank_begin && rank < seg.rank_end)) &&
                     XP_CHECKED(first < ne && (u64)pos < nl && rank < g->cnt[hole->start_nt][seg.size], kChkQueue);
                if (ok) {
                    const OperandRef ref = operand_ref(g, hole, seg.nt, seg.esize, first);
                    const LeafDev lf = g->leaves[g->leaf_begin[grp.leaf_nt] + (int)pos];
                    if (spread) {
                        const int j = from + (lane & 15);
                        if (j < n_exact) {
                            i64 a = 0, v = 0;
                            ++n.evals;
                            ok = ref_value(g, hole, ref, seg.nt, seg.esize, j, a);
                            const i64 c = lf.var >= 0 ? hole->probe_pt[j][lf.var] : lf.value;
                            ok = ok && op_value(op, swap ? c : a, swap ? a : c, v) && probe_accepts(hole, j, v);
                        }
                    } else ok = four ? exact_pair4(g, hole, ref, seg.nt, seg.esize, lf.var, lf.value, swap != 0, op, from, n_exact, n.evals)
                                     : exact_pair(g, hole, ref, seg.nt, seg.esize, lf.var, lf.value, swap != 0, op, from, n_exact, n.evals);
                    if (ok && !spread) vars = ref_vars(hole, ref) | (lf.var >= 0 ? 1u << lf.var : 0u);
                }
            }
            if (spread) {
                const u32 b = __ballot_sync(0xffffffffu, ok);
                good |= (u32)((b & 0xffffu) == 0xffffu) << i0 | (u32)(b >> 16 == 0xffffu) << (i0 + 1u);
            } else pass = ok;
        }
        if (spread) {                                     // candidate i to lane i
            pass = lane < 4 && ((good >> lane) & 1u);
            if (at + (u32)lane < nc && lane < 4) {
                code = w.c_code[at + lane]; pos = w.c_pos[at + lane]; e = w.base + w.c_off[at + lane];
                if (pass && !classes) {
                    const int swap = (int)(code & 1u), slot = (int)((code >> 1) & 15u);
                    const JoinGroup& grp = plan.jgroups[seg.first_group + (int)(code >> 8)];
                    rank = grp.base[swap][slot] + (swap ? (u64)pos * g->cnt[seg.nt][seg.esize] + e : e * g->cnt[grp.leaf_nt][1] + (u64)pos);
                    const LeafDev lf = g->leaves[g->leaf_begin[grp.leaf_nt] + (int)pos];
                    vars = ref_vars(hole, operand_ref(g, hole, seg.nt, seg.esize, e)) | (lf.var >= 0 ? 1u << lf.var : 0u);
                }
            }
        }
        if (classes) { join_members(w, plan, seg, sk, hole, pass, e, pos, code, n); continue; }
        if (n_exact < hole->n_probe) pass = join_full_check(g, hole, seg.size, pass, rank, n.evals);
        join_survive(w.cand, plan, sk, hole, seg, pass, rank, vars, n);
    }
    __syncwarp();
    if (lane == 0) w.nc = 0;
    __syncwarp();
}

// Lanes with a candidate put it into the second queue (checked when a warp's worth has gathered).  Called by all lanes.
__device__ __forceinline__ void join_push(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, bool have,
                                          u32 off, u32 pos, int group, int slot, int swap, int from, JoinCount& n) {
    const u32 b = __ballot_sync(0xffffffffu, have);
    if (!b) return;
    const int lane = threadIdx.x & 31;
    const u32 nc = w.nc;
    if (have) {
        const u32 at = nc + (u32)__popc(b & ((1u << lane) - 1u));      // (nc < 32)
        w.c_off[at] = off; w.c_pos[at] = pos; w.c_code[at] = ((u32)group << 8) | ((u32)slot << 1) | (u32)swap;
    }
    __syncwarp();
    if (lane == 0) w.nc = nc + (u32)__popc(b);
    __syncwarp();
    if (nc + (u32)__popc(b) >= 32u) join_check(w, plan, seg, sk, hole, from, n);
}

// ---- the conditions ----

__device__ __forceinline__ bool in_range(u32 c, const GroupCtx& s) { return c - (u32)s.cmin <= (u32)s.cmax - (u32)s.cmin; }

// a * c = t at both probes for some c, given that a0 * t1 = a1 * t0: the operand divides the target.
__device__ __noinline__ bool factor_exists(i32 a0, i32 a1, const JoinCtx& x, u32 cabs) {
    if (!x.small) return true;                            // (decided when the suspect is taken up)
    const u32 u = a0 != 0 ? abs_u32(a0) : abs_u32(a1), t = a0 != 0 ? x.ut0 : x.ut1;
    if (a0 == 0 && x.ut0 != 0u) return false;
    return u == 0u ? t == 0u : t % u == 0u && t / u <= cabs;
}

__device__ __noinline__ bool gcd_exceeds(u32 x, u32 y, u32 least) {      // gcd(x, y) > least (gcd(0, 0) counts as infinite)
    if (x == 0u && y == 0u) return true;
    while (y != 0u) {
        if (y <= least) return false;                     // the divisor sought divides y, and exceeds `least`
        const u32 r = x % y;
        x = y; y = r;
    }
    return x > least;
}

// Is there a magnitude m <= cabs with m mod u0 = ut0 and m mod u1 = ut1?  Stepping along the larger of the two where that is a few
// steps, otherwise by the least such m.  (With a constant of 2^31 - 1 the steps, up to 46 000 an operand, were the search: 69 leaves, size 7,
// 118 -> 10 ms.)
__device__ __noinline__ bool residue_exists(u32 u0, u32 u1, u32 ut0, u32 ut1, u32 cabs) {
    if (u0 <= ut0 || u1 <= ut1) return false;
    if (u0 < u1) { u32 s = u0; u0 = u1; u1 = s; s = ut0; ut0 = ut1; ut1 = s; }
    if (u1 > kResidueSteps && cabs / u0 > kResidueSteps) return residue_least(u0, u1, ut0, ut1) <= cabs;
    u32 steps = u1;                                       // (the residues repeat after u1 steps)
    for (u64 m = ut0; m <= cabs && steps > 0u; m += u0, --steps) if ((u32)m % u1 == ut1) return true;
    return false;
}

enum { kSlotAdd = 0, kSlotSub = 1, kSlotMul = 2, kSlotDiv = 3, kSlotMod = 4, kSlotMn = 5, kSlotMx = 6, kSlotShl = 7, kSlotShr = 8 };

__device__ __forceinline__ bool const_div_fwd(float f0, float f1, const JoinCtx& x, float fc) {       // some |c| in (|a|/(|t|+1), |a|/|t|] at both
    const float hi = fminf(f0 * x.rt0 + x.h0, f1 * x.rt1 + x.h1) * 1.000002f, lo = fmaxf(f0 * x.rl0, f1 * x.rl1) * 0.999998f;
    const float c = floorf(fminf(hi, fc));
    return c >= 1.f && c > lo;
}
__device__ __forceinline__ bool const_div_swap(float f0, float f1, const JoinCtx& x, float fc) {      // some |c| in [|t||a|, (|t|+1)|a|) at both
    const float lo = fmaxf(f0 * x.ft0, f1 * x.ft1) * 0.999998f;
    const float hi = fminf(f0 * (x.ft0 + 1.f), f1 * (x.ft1 + 1.f)) * 1.000002f;
    return lo < hi && lo <= fc;
}
__device__ __forceinline__ bool const_minmax(i32 a0, i32 a1, const JoinCtx& x, u32 mm, bool mx) {
    const i32 t0 = (i32)x.t0, t1 = (i32)x.t1;
    auto f = [&](i32 a, i32 b) { return mx ? (a > b ? a : b) : (a < b ? a : b); };
    bool h = a0 == t0 && a1 == t1;
    if (mm & 1u) h |= f(a0, t0) == t0 && f(a1, t0) == t1;
    if (mm & 2u) h |= f(a0, t1) == t0 && f(a1, t1) == t1;
    return h;
}

// One condition on one operand (used again when a suspect is taken up): constants, operator slot, side.
__device__ __forceinline__ bool const_condition(int slot, int swap, i32 a0, i32 a1, const JoinCtx& x, const GroupCtx& s) {
    const u32 u0 = abs_u32(a0), u1 = abs_u32(a1);
    switch (slot) {
        case kSlotAdd: return (u32)a0 - (u32)a1 == x.t0 - x.t1 && in_range(x.t0 - (u32)a0, s);
        case kSlotSub: return swap ? (u32)a0 - (u32)a1 == x.t1 - x.t0 && in_range(x.t0 + (u32)a0, s)
                                   : (u32)a0 - (u32)a1 == x.t0 - x.t1 && in_range((u32)a0 - x.t0, s);
        case kSlotMul: return (u32)a0 * x.t1 == (u32)a1 * x.t0 && factor_exists(a0, a1, x, s.cabs);
        case kSlotDiv: return swap ? const_div_swap((float)u0, (float)u1, x, s.fc) : const_div_fwd((float)u0, (float)u1, x, s.fc);
        case kSlotMod: return swap ? residue_exists(u0, u1, x.ut0, x.ut1, s.cabs)
                                   : u0 >= x.ut0 && u1 >= x.ut1 && gcd_exceeds(u0 - x.ut0, u1 - x.ut1, x.tmod);
        case kSlotMn: return const_minmax(a0, a1, x, s.mm, false);
        case kSlotMx: return const_minmax(a0, a1, x, s.mm, true);
    }
    return false;
}

// The entry's candidates at the two probes, for the operators in f (E op entry) and s (entry op E).
template <int P>
__device__ __forceinline__ void entry_conditions(const JoinEntry& e, u32 f, u32 s, const i32 (&a0)[P], const i32 (&a1)[P], const JoinCtx& x, bool (&any)[P]) {
    if ((f | s) & (1u << kSlotAdd)) {
        const u32 d0 = x.t0 - e.v0, d1 = x.t1 - e.v1;
#pragma unroll
        for (int p = 0; p < P; ++p) any[p] |= (u32)a0[p] == d0 && (u32)a1[p] == d1;
    }
    if (f & (1u << kSlotSub)) {
        const u32 d0 = x.t0 + e.v0, d1 = x.t1 + e.v1;
#pragma unroll
        for (int p = 0; p < P; ++p) any[p] |= (u32)a0[p] == d0 && (u32)a1[p] == d1;
    }
    if (s & (1u << kSlotSub)) {
        const u32 d0 = e.v0 - x.t0, d1 = e.v1 - x.t1;
#pragma unroll
        for (int p = 0; p < P; ++p) any[p] |= (u32)a0[p] == d0 && (u32)a1[p] == d1;
    }
    if ((f | s) & (1u << kSlotMul)) {
#pragma unroll
        for (int p = 0; p < P; ++p) any[p] |= (u32)a0[p] * e.v0 == x.t0 && (u32)a1[p] * e.v1 == x.t1;
    }
    if ((f & (1u << kSlotDiv)) && e.u0 != 0u && e.u1 != 0u) {              // floor(|a| / |v|) = |t|  <=>  |a| - |t||v| < |v|
#pragma unroll
        for (int p = 0; p < P; ++p) any[p] |= abs_u32(a0[p]) - e.low0 < e.u0 && abs_u32(a1[p]) - e.low1 < e.u1;
    }
    if (s & (1u << kSlotDiv)) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const u32 u0 = abs_u32(a0[p]), u1 = abs_u32(a1[p]);
            any[p] |= e.u0 - u0 * x.ut0 < u0 && e.u1 - u1 * x.ut1 < u1;    // (a product past 32 bits can only let more through)
        }
    }
    if ((f & (1u << kSlotMod)) && e.cm0 != 0u && e.cm1 != 0u) {            // |v| divides |a| - |t|
        const u32 k0 = e.k0k1 & 255u, k1 = e.k0k1 >> 8;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const u32 u0 = abs_u32(a0[p]), u1 = abs_u32(a1[p]);
            any[p] |= u0 >= x.ut0 && rotr32((u0 - x.ut0) * e.inv0, k0) <= e.cm0 && u1 >= x.ut1 && rotr32((u1 - x.ut1) * e.inv1, k1) <= e.cm1;
        }
    }
    if ((s & (1u << kSlotMod)) && e.u0 >= x.ut0 && e.u1 >= x.ut1) {        // |a| divides |v| - |t| and exceeds |t|
        const u32 y0 = e.u0 - x.ut0, y1 = e.u1 - x.ut1;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const u32 u0 = abs_u32(a0[p]), u1 = abs_u32(a1[p]);
            if (u0 > x.ut0 && u1 > x.ut1 && (u0 <= y0 || y0 == 0u) && (u1 <= y1 || y1 == 0u)) any[p] |= y0 % u0 == 0u && y1 % u1 == 0u;
        }
    }
    if ((f | s) & (1u << kSlotMn)) {
#pragma unroll
        for (int p = 0; p < P; ++p)
            any[p] |= (a0[p] < (i32)e.v0 ? a0[p] : (i32)e.v0) == (i32)x.t0 && (a1[p] < (i32)e.v1 ? a1[p] : (i32)e.v1) == (i32)x.t1;
    }
    if ((f | s) & (1u << kSlotMx)) {
#pragma unroll
        for (int p = 0; p < P; ++p)
            any[p] |= (a0[p] > (i32)e.v0 ? a0[p] : (i32)e.v0) == (i32)x.t0 && (a1[p] > (i32)e.v1 ? a1[p] : (i32)e.v1) == (i32)x.t1;
    }
}

// The constants of a group as a set.  CF, CS: the operators, known at compile time for the usual groups (-1: taken from s).
template <int P, int CF, int CS>
__device__ __forceinline__ void set_conditions(const GroupCtx& s, const i32 (&a0)[P], const i32 (&a1)[P], const JoinCtx& x, bool (&any)[P]) {
    const u32 cf = CF < 0 ? s.cf : (u32)CF, cs = CS < 0 ? s.cs : (u32)CS;
    if ((cf | cs) & ((1u << kSlotAdd) | (1u << kSlotSub))) {
        const u32 dt = x.t0 - x.t1, nt = 0u - dt;
        const bool rsub = (cs >> kSlotSub) & 1u;
        bool maybe = false;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const u32 d = (u32)a0[p] - (u32)a1[p];
            maybe |= d == dt || (rsub && d == nt);
        }
        if (maybe) {                                      // (rarely: an operand mostly differs otherwise than the target does)
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const u32 d = (u32)a0[p] - (u32)a1[p];
                bool h = false;
                if ((cf | cs) & (1u << kSlotAdd)) h |= d == dt && in_range(x.t0 - (u32)a0[p], s);
                if (cf & (1u << kSlotSub)) h |= d == dt && in_range((u32)a0[p] - x.t0, s);
                if (rsub) h |= d == nt && in_range(x.t0 + (u32)a0[p], s);
                any[p] |= h;
            }
        }
    }
    if ((cf | cs) & (1u << kSlotMul)) {
        bool maybe = false;
#pragma unroll
        for (int p = 0; p < P; ++p) maybe |= (u32)a0[p] * x.t1 == (u32)a1[p] * x.t0;
        if (maybe) {
            const u32 cabs = s.cabs;
#pragma unroll 1
            for (int p = 0; p < P; ++p) {
                i32 v0 = a0[0], v1 = a1[0];
#pragma unroll
                for (int k = 1; k < P; ++k) if (k == p) { v0 = a0[k]; v1 = a1[k]; }
                const bool h = (u32)v0 * x.t1 == (u32)v1 * x.t0 && ((v0 | v1) != 0 || x.tz) && factor_exists(v0, v1, x, cabs);
#pragma unroll
                for (int k = 0; k < P; ++k) any[k] |= h && k == p;
            }
        }
    }
    if ((cf | cs) & (1u << kSlotDiv)) {
        const float fc = s.fc;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const float f0 = fabsf((float)a0[p]), f1 = fabsf((float)a1[p]);
            if (cf & (1u << kSlotDiv)) any[p] |= const_div_fwd(f0, f1, x, fc);
            if (cs & (1u << kSlotDiv)) any[p] |= const_div_swap(f0, f1, x, fc);
        }
    }
    if ((cf | cs) & (1u << kSlotMod)) {
        const u32 cabs = s.cabs;
#pragma unroll 1
        for (int p = 0; p < P; ++p) {
            i32 v0 = a0[0], v1 = a1[0];
            bool h = any[0];
#pragma unroll
            for (int k = 1; k < P; ++k) if (k == p) { v0 = a0[k]; v1 = a1[k]; h = any[k]; }
            const u32 u0 = abs_u32(v0), u1 = abs_u32(v1);
            if (!h && (cf & (1u << kSlotMod)) && u0 >= x.ut0 && u1 >= x.ut1) h = gcd_exceeds(u0 - x.ut0, u1 - x.ut1, x.tmod);
            if (!h && (cs & (1u << kSlotMod))) h = residue_exists(u0, u1, x.ut0, x.ut1, cabs);
#pragma unroll
            for (int k = 0; k < P; ++k) any[k] |= h && k == p;
        }
    }
    if ((cf | cs) & (1u << kSlotMn)) {
#pragma unroll
        for (int p = 0; p < P; ++p) any[p] |= const_minmax(a0[p], a1[p], x, s.mm, false);
    }
    if ((cf | cs) & (1u << kSlotMx)) {
#pragma unroll
        for (int p = 0; p < P; ++p) any[p] |= const_minmax(a0[p], a1[p], x, s.mm, true);
    }
}

// ---- suspects ----

// First constant of [lo, hi) that is not below v.
__device__ __forceinline__ i32 const_lower(const ConstDev* c, i32 lo, i32 hi, i64 v) {
    while (lo < hi) {
        const i32 mid = (lo + hi) >> 1;
        if (c[mid].value < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The constants that operator slot `slot` leaves open for an operand: up to two runs of the ascending list.
__device__ __noinline__ void const_runs(const ConstDev* c, i32 lo, i32 hi, int slot, int swap, i64 a0, i64 a1, i64 t0, i64 t1, u64 tmod, i32 (&run)[4]) {
    run[0] = run[2] = lo; run[1] = run[3] = lo;
    auto one = [&](i64 v) { run[0] = const_lower(c, lo, hi, v); run[1] = const_lower(c, run[0], hi, v + 1); };
    auto magnitudes = [&](u64 from, u64 to) {             // from <= |c| <= to, c != 0
        if (from < 1) from = 1;
        const u64 most = 1ull << 31;
        if (to > most) to = most;
        if (from > to) return;
        run[0] = const_lower(c, lo, hi, -(i64)to); run[1] = const_lower(c, run[0], hi, -(i64)from + 1);
        run[2] = const_lower(c, lo, hi, (i64)from); run[3] = const_lower(c, run[2], hi, (i64)to + 1);
    };
    const u64 u0 = (u64)(a0 < 0 ? -a0 : a0), u1 = (u64)(a1 < 0 ? -a1 : a1), v0 = (u64)(t0 < 0 ? -t0 : t0), v1 = (u64)(t1 < 0 ? -t1 : t1);
    switch (slot) {
        case kSlotAdd: one(t0 - a0); return;
        case kSlotSub: one(swap ? t0 + a0 : a0 - t0); return;
        case kSlotMul: {
            const i64 a = a0 != 0 ? a0 : a1, t = a0 != 0 ? t0 : t1;
            if (a0 == 0 && t0 != 0) return;
            if (a == 0) { if (t == 0) { run[0] = lo; run[1] = hi; } return; }
            if (t % a == 0) one(t / a);
            return;
        }
        case kSlotDiv:
            if (!swap) {
                const u64 l0 = u0 / (v0 + 1) + 1, l1 = u1 / (v1 + 1) + 1;
                const u64 h0 = v0 ? u0 / v0 : ~0ull, h1 = v1 ? u1 / v1 : ~0ull;
                magnitudes(l0 > l1 ? l0 : l1, h0 < h1 ? h0 : h1);
            } else if (u0 != 0 && u1 != 0) {
                const u64 l0 = v0 * u0, l1 = v1 * u1, h0 = l0 + u0 - 1, h1 = l1 + u1 - 1;
                const u64 l = l0 > l1 ? l0 : l1, h = h0 < h1 ? h0 : h1;
                if (l == 0) { run[0] = const_lower(c, lo, hi, -(i64)h); run[1] = const_lower(c, run[0], hi, (i64)h + 1); }      // (0 among them)
                else magnitudes(l, h);
            }
            return;
        case kSlotMod:
            // a % c: |c| exceeds every target and divides |a| - |t| at both probes, so it is a divisor of their greatest common
            // one, and that one itself where its half is no longer above the targets.  c % a: |c| is |t| plus a multiple of
            // |a|, so |t| itself where one |a| more is beyond every constant.  (With every constant
            // above the target open: join of the large table 9.00 -> 8.91 ms, of the four-variable nest 1.96 -> 1.92.)
            if (!swap) {
                u64 g = u0 - v0, r = u1 - v1;
                if (u0 < v0 || u1 < v1) return;
                while (r) { const u64 q = (u32)g % (u32)r; g = r; r = q; }      // (both below 2^31)
                magnitudes(g && g / 2 <= tmod ? g : tmod + 1, g ? g : ~0ull);
                if (g && g <= tmod) { run[1] = run[0]; run[3] = run[2]; }
                return;
            }
            {
                const u64 big = u0 > u1 ? u0 : u1, at = u0 > u1 ? v0 : v1;
                const u64 m0 = (u64)(c[lo].value < 0 ? -c[lo].value : c[lo].value), m1 = (u64)(c[hi - 1].value < 0 ? -c[hi - 1].value : c[hi - 1].value);
                if (at + big > (m0 > m1 ? m0 : m1)) { if (at) magnitudes(at, at); else one(0); return; }
            }
            run[0] = lo; run[1] = hi; return;
        default: run[0] = lo; run[1] = hi; return;
    }
}

// v = x op y at one probe for narrow x, y; false when undefined.
__device__ __forceinline__ bool narrow_op(int slot, i32 x, i32 y, i64& v) {
    switch (slot) {
        case kSlotAdd: v = (i64)x + y; return true;
        case kSlotSub: v = (i64)x - y; return true;
        case kSlotMul: v = (i64)x * y; return true;
        case kSlotDiv: if (y == 0) return false; v = y == -1 ? -(i64)x : (i64)(x / y); return true;
        case kSlotMod: if (y == 0) return false; v = y == -1 ? 0 : (i64)(x % y); return true;
        case kSlotMn: v = x < y ? x : y; return true;
        default: v = x > y ? x : y; return true;
    }
}

// For which operators is the result of operand x and leaf c the target t (both narrow: above -2^31, below 2^31)?  Bit = slot
// for x op c, 16 + slot for c op x.  Straight through all operators, without a branch per operator: one division serves
// quotient and remainder.
__device__ __forceinline__ u32 narrow_bits(i32 x, i32 c, i64 t, bool divide) {
    const i64 X = x, C = c;
    u32 b = ((u32)(X + C == t) << kSlotAdd) * 0x10001u | ((u32)(X * C == t) << kSlotMul) * 0x10001u |
            (u32)(X - C == t) << kSlotSub | (u32)(C - X == t) << (16 + kSlotSub) |
            ((u32)((X < C ? X : C) == t) << kSlotMn) * 0x10001u | ((u32)((X > C ? X : C) == t) << kSlotMx) * 0x10001u;
    if (divide) {
        const i32 cd = c ? c : 1, xd = x ? x : 1, q = x / cd, p = c / xd;      // (no overflow: neither is -2^31)
        b |= (u32)(c != 0 && (i64)q == t) << kSlotDiv | (u32)(c != 0 && (i64)(x - q * cd) == t) << kSlotMod |
             (u32)(x != 0 && (i64)p == t) << (16 + kSlotDiv) | (u32)(x != 0 && (i64)(c - p * xd) == t) << (16 + kSlotMod);
    }
    return b;
}

// The suspects in the warp's first queue, one per lane.  Called by all 32 lanes together.  Small searches wait for a few of
// these passes and nothing else: an entry is held against all operators at once (narrow_bits) with its values from another
// lane's register (operator by operator, with a load each, a pass took some 6000 instructions: join of a tile bound 52 -> 45 us,
// of 1024 small sketches 2.50 -> 2.16 ms).
__device__ __noinline__ void join_drain(JoinWarp& w, u32 n_q, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const JoinCtx& x = w.x;
    n.suspects += n_q;
    const i64 t0 = hole->join_t0, t1 = hole->join_t1;
    const u64 tmod = hole->join_tmod;
    const int from = hole->join_p1 ? 2 : 1;               // probes that the second queue's check starts at
    for (u32 at = 0; at < n_q; at += 32) {
        const bool live = at + lane < n_q;
        const u32 off = live ? w.q_off[at + lane] : 0u;
        const i32 b0 = live ? w.q_a0[at + lane] : 0, b1 = live ? w.q_a1[at + lane] : 0;
        auto holds = [&](int slot, int swap, i32 x0, i32 x1, i32 c0, i32 c1) {       // exactly, at both probes
            i64 v = 0;
            return narrow_op(slot, swap ? c0 : x0, swap ? x0 : c0, v) && v == t0 && narrow_op(slot, swap ? c1 : x1, swap ? x1 : c1, v) && v == t1;
        };
        for (int gi = 0; gi < seg.n_groups; ++gi) {
            const GroupCtx& s = w.grp[gi];
            const JoinSet* S = s.set;
            if (s.ef | s.es) {
                const u32 want = s.ef | (s.es << 16);
                const bool divide = ((s.ef | s.es) & ((1u << kSlotDiv) | (1u << kSlotMod))) != 0u;
                const int n_e = s.n_entries;
                i32 e0 = 0, e1 = 0;
                u32 ep = 0;
                if (lane < n_e) { e0 = (i32)S->e[lane].v0; e1 = (i32)S->e[lane].v1; ep = S->e[lane].pos; }
                for (int i = 0; i < n_e; ++i) {
                    const i32 v0 = __shfl_sync(0xffffffffu, e0, i), v1 = __shfl_sync(0xffffffffu, e1, i);
                    u32 hits = live ? want : 0u;
#pragma unroll 1
                    for (int k = 0; k < 2; ++k) {         // (most suspects end at the first probe for most entries)
                        hits &= narrow_bits(k ? b1 : b0, k ? v1 : v0, k ? t1 : t0, divide);
                        if (!__any_sync(0xffffffffu, hits != 0u)) break;
                    }
                    const u32 pos = __shfl_sync(0xffffffffu, ep, i);
#pragma unroll 1
                    for (u32 m = __reduce_or_sync(0xffffffffu, hits); m; m &= m - 1) {
                        const int bit = __ffs((int)m) - 1;
                        join_push(w, plan, seg, sk, hole, (hits >> bit) & 1u, off, pos, gi, bit & 15, bit >> 4, from, n);
                    }
                }
            }
            if (!(s.cf | s.cs)) continue;
            const i32 clo = S->const_begin, chi = clo + S->n_const;
            for (int swap = 0; swap < 2; ++swap)
#pragma unroll 1
                for (u32 m = swap ? s.cs : s.cf; m; m &= m - 1) {
                    const int slot = __ffs((int)m) - 1;
                    const bool act = live && const_condition(slot, swap, b0, b1, x, s);
                    if (!__any_sync(0xffffffffu, act)) continue;
                    i32 run[4] = {clo, clo, clo, clo};
                    if (act) const_runs(g->consts, clo, chi, slot, swap, b0, b1, t0, t1, tmod, run);
                    const i32 len0 = run[1] - run[0], len = len0 + run[3] - run[2];
                    // A lane per suspect, or, where few suspects have long runs (a remainder leaves every constant above the
                    // target open), the suspects one after the other with the lanes over their constants.
                    const i32 longest = (i32)__reduce_max_sync(0xffffffffu, (u32)len);
                    const i32 steps = (i32)__reduce_add_sync(0xffffffffu, (u32)((len + 31) / 32));
                    if (longest <= steps) {
                        for (i32 i = 0; i < longest; ++i) {
                            bool on = i < len;
                            const ConstDev c = g->consts[on ? (i < len0 ? run[0] + i : run[2] + i - len0) : clo];
                            if (on) on = holds(slot, swap, b0, b1, (i32)c.value, (i32)c.value);
                            join_push(w, plan, seg, sk, hole, on, off, (u32)c.pos, gi, slot, swap, from, n);
                        }
                    } else
                        for (u32 q = __ballot_sync(0xffffffffu, len > 0); q; q &= q - 1) {
                            const int src = __ffs((int)q) - 1;
                            const i32 r0 = __shfl_sync(0xffffffffu, run[0], src), r2 = __shfl_sync(0xffffffffu, run[2], src);
                            const i32 n0 = __shfl_sync(0xffffffffu, len0, src), nn = __shfl_sync(0xffffffffu, len, src);
                            const i32 x0 = __shfl_sync(0xffffffffu, b0, src), x1 = __shfl_sync(0xffffffffu, b1, src);
                            const u32 o = __shfl_sync(0xffffffffu, off, src);
                            for (i32 i0 = 0; i0 < nn; i0 += 32) {
                                const i32 i = i0 + lane;
                                bool on = i < nn;
                                const ConstDev c = g->consts[on ? (i < n0 ? r0 + i : r2 + i - n0) : clo];
                                if (on) on = holds(slot, swap, x0, x1, (i32)c.value, (i32)c.value);
                                join_push(w, plan, seg, sk, hole, on, o, (u32)c.pos, gi, slot, swap, from, n);
                            }
                        }
                }
        }
    }
    __syncwarp();
}

// The exact form where a segment has few operands (kExactFew): one at a time (the same for all lanes), lanes over the leaves, every
// operator; the first two probes here, the others when a warp's worth of candidates has gathered.
__device__ __noinline__ void join_exact(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, u64 e, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    const OperandRef ref = operand_ref(g, hole, seg.nt, seg.esize, e);
    i64 a0, a1 = 0;
    if (!ref_value(g, hole, ref, seg.nt, seg.esize, 0, a0)) return;
    const bool two = hole->n_exact >= 2;
    if (two && !ref_value(g, hole, ref, seg.nt, seg.esize, 1, a1)) return;
    if (w.nc) join_check(w, plan, seg, sk, hole, hole->join_p1 && hole->join_on ? 2 : 1, n);      // (what waits was held against the pair)
    for (int gi = 0; gi < seg.n_groups; ++gi) {
        const JoinGroup& grp = plan.jgroups[seg.first_group + gi];
        const int nl = (int)g->cnt[grp.leaf_nt][1];
        n.tests += (u64)nl * (u64)(__popc(grp.fmask) + __popc(grp.smask));
        for (int l0 = 0; l0 < nl; l0 += 32) {
            const int pos = l0 + lane;
            const LeafDev lf = g->leaves[g->leaf_begin[grp.leaf_nt] + (pos < nl ? pos : 0)];
            const i64 c0 = lf.var >= 0 ? hole->probe_pt[0][lf.var] : lf.value, c1 = two && lf.var >= 0 ? hole->probe_pt[1][lf.var] : lf.value;
            for (int swap = 0; swap < 2; ++swap)
                for (u32 m = swap ? grp.smask : grp.fmask; m; m &= m - 1) {
                    const int slot = __ffs((int)m) - 1, op = op_of_slot(slot);
                    i64 v;
                    bool hit = pos < nl && apply_op(op, swap ? c0 : a0, swap ? a0 : c0, v) && probe_accepts(hole, 0, v);
                    if (two && hit) hit = apply_op(op, swap ? c1 : a1, swap ? a1 : c1, v) && probe_accepts(hole, 1, v);
                    n.suspects += (u32)__popc(__ballot_sync(0xffffffffu, hit));
                    join_push(w, plan, seg, sk, hole, hit, (u32)(e - w.base), (u32)pos, gi, slot, swap, two ? 2 : 1, n);
                }
        }
    }
    if (w.nc) join_check(w, plan, seg, sk, hole, two ? 2 : 1, n);
}

// What a probe demands of a candidate's value, in registers.
struct ProbeWant { bool affine; u64 A, D; i64 lo, hi; };
__device__ __forceinline__ ProbeWant probe_want(const HoleDev* hole, int j) {
    ProbeWant p;
    p.affine = (hole->aff_okmask >> j) & 1u;
    p.A = hole->aff_Aj[j]; p.D = (u64)hole->probe_spec[j] - hole->aff_Bj[j];
    p.lo = hole->rng_lo[j]; p.hi = hole->rng_hi[j];
    return p;
}
__device__ __forceinline__ bool wanted(const ProbeWant& p, i64 v) {      // (probe_accepts)
    if (p.affine) return (u64)v * p.A == p.D;
    return v <= -(1ll << 62) || v >= (1ll << 62) || (v >= p.lo && v <= p.hi);
}

// For which of the operators `ops` is the result of operand a and leaf c what the probe wants?  Bit = slot for a op c, 16 + slot for
// c op a.  In 64 bits, one division for quotient and remainder; `ops` is the same for all lanes.
__device__ __forceinline__ u32 exact_bits(i64 a, i64 c, u32 ops, const ProbeWant& p) {
    auto both = [](int slot) { return 0x10001u << slot; };
    u32 b = 0;
    i64 v;
    if (ops & both(kSlotAdd)) { (void)apply_op(XP_OP_ADD, a, c, v); if (wanted(p, v)) b |= both(kSlotAdd); }
    if (ops & (1u << kSlotSub)) { (void)apply_op(XP_OP_SUB, a, c, v); if (wanted(p, v)) b |= 1u << kSlotSub; }
    if (ops & (0x10000u << kSlotSub)) { (void)apply_op(XP_OP_SUB, c, a, v); if (wanted(p, v)) b |= 0x10000u << kSlotSub; }
    if (ops & both(kSlotMul)) { (void)apply_op(XP_OP_MUL, a, c, v); if (wanted(p, v)) b |= both(kSlotMul); }
    if (ops & both(kSlotMn)) { if (wanted(p, a < c ? a : c)) b |= both(kSlotMn); }
    if (ops & both(kSlotMx)) { if (wanted(p, a > c ? a : c)) b |= both(kSlotMx); }
#pragma unroll 1
    for (int swap = 0; swap < 2; ++swap) {
        const u32 o = swap ? ops >> 16 : ops & 0xffffu;
        const i64 x = swap ? c : a, y = swap ? a : c;
        u32 q = 0;
        if ((o & ((1u << kSlotDiv) | (1u << kSlotMod))) && apply_op(XP_OP_DIV, x, y, v)) {
            if (wanted(p, v)) q |= 1u << kSlotDiv;
            if (wanted(p, (i64)((u64)x - (u64)v * (u64)y))) q |= 1u << kSlotMod;
        }
        if ((o & (1u << kSlotShl)) && apply_op(XP_OP_SHL, x, y, v) && wanted(p, v)) q |= 1u << kSlotShl;
        if ((o & (1u << kSlotShr)) && apply_op(XP_OP_SHR, x, y, v) && wanted(p, v)) q |= 1u << kSlotShr;
        b |= swap ? q << 16 : q;
    }
    return b & ops;
}

// The exact form for 32 operands, one per lane (live: this lane has one): every leaf, every operator, at the first two probes; the
// others when a warp's worth of candidates has gathered (from probe `from` on).  Called by all 32 lanes together.  Bound by the
// 64-bit arithmetic.  (One operand at a time, each lookup and each vote was waited for: size 7, 63 leaves with shifts 72 -> 27 ms;
// 36 leaves with one of 2^33 16.3 -> 3.1 ms.)
__device__ __noinline__ void join_exact32(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, u64 e, bool live,
                                          int from, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const bool two = hole->n_exact >= 2;
    i64 a0 = 0, a1 = 0;
    if (live) {
        const OperandRef ref = operand_ref(g, hole, seg.nt, seg.esize, XP_CLASSES(seg) ? class_operand(g, hole, seg.nt, seg.esize, e).rank(0) : e);
        live = ref_value(g, hole, ref, seg.nt, seg.esize, 0, a0) && (!two || ref_value(g, hole, ref, seg.nt, seg.esize, 1, a1));
    }
    const u32 n_live = (u32)__popc(__ballot_sync(0xffffffffu, live));
    if (n_live == 0u) return;
    const ProbeWant p0 = probe_want(hole, 0), p1 = probe_want(hole, two ? 1 : 0);
    const u32 off = (u32)(e - w.base);
    for (int gi = 0; gi < seg.n_groups; ++gi) {
        const JoinGroup& grp = plan.jgroups[seg.first_group + gi];
        const int nl = (int)g->cnt[grp.leaf_nt][1], lb = g->leaf_begin[grp.leaf_nt];
        const u32 ops = grp.fmask | (grp.smask << 16);
        n.tests += (u64)nl * (u64)__popc(ops) * n_live;
        for (int l = 0; l < nl; ++l) {
            const LeafDev lf = g->leaves[lb + l];
            u32 hits = live ? exact_bits(a0, lf.var >= 0 ? hole->probe_pt[0][lf.var] : lf.value, ops, p0) : 0u;
            if (!__any_sync(0xffffffffu, hits != 0u)) continue;
            if (two && hits) hits &= exact_bits(a1, lf.var >= 0 ? hole->probe_pt[1][lf.var] : lf.value, ops, p1);
#pragma unroll 1
            for (u32 m = __reduce_or_sync(0xffffffffu, hits); m; m &= m - 1) {
                const int bit = __ffs((int)m) - 1;
                const u32 b = __ballot_sync(0xffffffffu, (hits >> bit) & 1u);
                n.suspects += (u32)__popc(b);
                join_push(w, plan, seg, sk, hole, (hits >> bit) & 1u, off, (u32)l, gi, bit & 15, bit >> 4, from, n);
            }
        }
    }
}

// The first n_w wide operands of the warp's queue, 32 at a time.
__device__ __noinline__ void join_wide(JoinWarp& w, u32 n_w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, JoinCount& n) {
    const u32 lane = threadIdx.x & 31u;
    __syncwarp();
    for (u32 at = 0; at < n_w; at += 32u) {
        const bool live = at + lane < n_w;
        join_exact32(w, plan, seg, sk, hole, w.base + (live ? w.w_off[at + lane] : 0u), live, hole->join_p1 ? 2 : 1, n);
    }
    __syncwarp();
}

// Wide operands (bit p of `wide`: number off + 32 p) into their queue; whole warps of them are taken up.  Called by all lanes.
__device__ __noinline__ void join_push_wide(JoinWarp& w, u32 wide, u32 off, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole,
                                            JoinCount& n) {
    const int lane = threadIdx.x & 31;
    u32 nw = w.nw;
    for (u32 any = __reduce_or_sync(0xffffffffu, wide); any; any &= any - 1) {
        const int p = __ffs((int)any) - 1;
        const bool h = (wide >> p) & 1u;
        const u32 b = __ballot_sync(0xffffffffu, h);
        if (h) w.w_off[nw + (u32)__popc(b & ((1u << lane) - 1u))] = off + 32u * (u32)p;
        nw += (u32)__popc(b);
    }
    if (nw >= 32u) {
        const u32 full = nw & ~31u;
        join_wide(w, full, plan, seg, sk, hole, n);
        nw -= full;
        const u32 o = lane < (int)nw ? w.w_off[full + lane] : 0u;
        __syncwarp();
        if (lane < (int)nw) w.w_off[lane] = o;
    }
    __syncwarp();
    if (lane == 0) w.nw = nw;
    __syncwarp();
}

// ---- operands in rank order ----

// A run of operands of (nt, size) in rank order that one production and pair of sizes builds: entries of the pair
// table, or (one size above the tables) products of two ranges of them.  The same for all lanes of a warp, so that a
// lane finds its operand with one division by an invariant.  Mode 2: neither (unranked in full, one by one).
struct JoinRun {
    i32 mode, op;
    const int2* L;
    const int2* R;
    u32 l0, r0, cr, inv;                                  // first operands; right operands per left one and 2^32 / that
    u64 left;                                             // operands to the end of the run
    u64 rank;                                             // (mode 2) rank of the first
};

// The run that operand number `rank` of (nt, size) is in; classes: the number counts by class (class_operand).
__device__ __noinline__ JoinRun join_run(const GrammarDev* g, const HoleDev* hole, int nt, int size, u64 rank, bool classes) {
    JoinRun c;
    const int2* pair = reinterpret_cast<const int2*>(hole->tab_pair);
    const int tmax = hole->tab_max_size;
    const u64 total = g->cnt[nt][size];
    c.mode = 2; c.op = 0; c.l0 = c.r0 = 0; c.cr = 1; c.inv = 0xffffffffu; c.L = c.R = pair; c.left = total - rank; c.rank = rank;
    if (size <= tmax) {
        const OperandSide s = operand_side(g, hole, nt, size, classes);
        c.mode = 0; c.R = s.pair + rank; c.left = s.n - rank;
        return c;
    }
    if (tmax < 1 || size < 3) return c;
    int p = g->bin_begin[nt], a = 1;
    const int pe = g->bin_begin[nt + 1];
    u64 rem = rank, cl = 0, cr = 0, base = 0;
    if (!classes) {
        while (p + 1 < pe && g->bins[p + 1].off[size] <= rank) ++p;
        base = g->bins[p].off[size]; rem = rank - base;
    }
    for (;; ++p) {                                        // (without classes the production is known)
        const int lnt = g->bins[p].lnt, rnt = g->bins[p].rnt;
        if (classes) base = g->bins[p].off[size];
        bool here = false;
        for (a = 1; a <= size - 2; ++a) {
            const u64 fl = g->cnt[lnt][a], fr = g->cnt[rnt][size - 1 - a];
            cl = fl; cr = fr;
            if (classes && a <= tmax && size - 1 - a <= tmax) {
                cl = operand_side(g, hole, lnt, a, true).n; cr = operand_side(g, hole, rnt, size - 1 - a, true).n;
            }
            here = rem < cl * cr || (!classes && a == size - 2);
            if (here) break;
            rem -= cl * cr; base += fl * fr;
        }
        if (here || p + 1 >= pe) break;
    }
    c.left = cl * cr - rem;
    c.rank = base + rem;
    if (a > tmax || size - 1 - a > tmax) return c;        // (an operand above the tables: the whole run goes one by one)
    u64 l, r;
    divmod_u64(rem, cr, l, r);
    c.mode = 1; c.op = g->bins[p].op;
    c.L = operand_side(g, hole, g->bins[p].lnt, a, classes).pair; c.R = operand_side(g, hole, g->bins[p].rnt, size - 1 - a, classes).pair;
    c.l0 = (u32)l; c.r0 = (u32)r; c.cr = (u32)cr;
    c.inv = cr > 1 ? (u32)((1ull << 32) / cr) : 0xffffffffu;
    return c;
}

__device__ __forceinline__ bool narrow31(i64 v) { return v > -(1ll << 31) && v < (1ll << 31); }

// An operand's values at the two probes: 0 undefined at one of them, 1 both below 2^31 in magnitude, 2 not.
__device__ __noinline__ int join_value_slow(const GrammarDev* g, const HoleDev* hole, int nt, int size, u64 rank, i32& a0, i32& a1) {
    i64 x, y;
    if (!operand_value(g, hole, 0, nt, size, rank, x)) return 0;
    y = x;
    if (hole->join_p1 && !operand_value(g, hole, hole->join_p1, nt, size, rank, y)) return 0;
    a0 = (i32)x; a1 = (i32)y;
    return narrow31(x) && narrow31(y) ? 1 : 2;
}

// Operator OP on the pairs of P operands.
template <int OP, int P>
__device__ __forceinline__ void pair_op(const int2 (&x)[P], const int2 (&y)[P], i32 (&a0)[P], i32 (&a1)[P], u32& alive, u32& wide) {
#pragma unroll
    for (int p = 0; p < P; ++p) {
        if (OP == XP_OP_DIV || OP == XP_OP_MOD) {         // (magnitudes below 2^31: no overflow)
            const i32 d0 = y[p].x == 0 ? 1 : y[p].x, d1 = y[p].y == 0 ? 1 : y[p].y;
            if (y[p].x == 0 || y[p].y == 0) alive &= ~(1u << p);
            const i32 q0 = x[p].x / d0, q1 = x[p].y / d1;
            a0[p] = OP == XP_OP_DIV ? q0 : x[p].x - q0 * d0;
            a1[p] = OP == XP_OP_DIV ? q1 : x[p].y - q1 * d1;
        } else if (OP == XP_OP_MIN) { a0[p] = min(x[p].x, y[p].x); a1[p] = min(x[p].y, y[p].y); }
        else if (OP == XP_OP_MAX) { a0[p] = max(x[p].x, y[p].x); a1[p] = max(x[p].y, y[p].y); }
        else if (OP == XP_OP_MUL) {
            const i64 r0 = (i64)x[p].x * y[p].x, r1 = (i64)x[p].y * y[p].y;
            a0[p] = (i32)r0; a1[p] = (i32)r1;
            if ((i32)(r0 >> 32) != (a0[p] >> 31) || (i32)(r1 >> 32) != (a1[p] >> 31)) wide |= 1u << p;
        } else {                                          // (-2^31 itself is left to the operand limit)
            const i32 b0 = OP == XP_OP_ADD ? y[p].x : -y[p].x, b1 = OP == XP_OP_ADD ? y[p].y : -y[p].y;
            a0[p] = (i32)((u32)x[p].x + (u32)b0); a1[p] = (i32)((u32)x[p].y + (u32)b1);
            if ((((x[p].x ^ a0[p]) & (b0 ^ a0[p])) | ((x[p].y ^ a1[p]) & (b1 ^ a1[p]))) < 0) wide |= 1u << p;
        }
    }
}

// Operands at + 32 p + lane of a run (those below n), their values at the two probes.
template <int P>
__device__ __forceinline__ void run_values(const JoinRun& c, const GrammarDev* g, const HoleDev* hole, int nt, int size, u32 at, u32 n,
                                           i32 (&a0)[P], i32 (&a1)[P], u32& alive, u32& wide) {
    const u32 lane = threadIdx.x & 31u;
    alive = wide = 0;
#pragma unroll
    for (int p = 0; p < P; ++p) { a0[p] = 0; a1[p] = 0; if (at + 32u * p + lane < n) alive |= 1u << p; }
    if (c.mode == 0) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int2 y = (alive >> p) & 1u ? c.R[at + 32u * p + lane] : make_int2(kPairNone, 0);
            a0[p] = y.x; a1[p] = y.y;
            if (y.x == kPairNone) { if ((alive >> p) & 1u) wide |= (u32)(y.y != 0) << p; alive &= ~(1u << p); }
        }
        return;
    }
    if (c.mode == 2) {
#pragma unroll 1
        for (int p = 0; p < P; ++p) {
            if (!((alive >> p) & 1u)) continue;
            i32 v0 = 0, v1 = 0;
            const int st = join_value_slow(g, hole, nt, size, c.rank + at + 32u * p + lane, v0, v1);
#pragma unroll
            for (int k = 0; k < P; ++k) if (k == p) { a0[k] = v0; a1[k] = v1; }
            if (st != 1) { alive &= ~(1u << p); wide |= (u32)(st == 2) << p; }
        }
        return;
    }
    int2 x[P], y[P];
    u32 none = 0;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const u32 rel = (alive >> p) & 1u ? c.r0 + at + 32u * p + lane : c.r0;
        u32 q = __umulhi(rel, c.inv), r = rel - q * c.cr; // the estimate is the quotient or one less
        if (r >= c.cr) { ++q; r -= c.cr; }
        x[p] = c.L[c.l0 + q]; y[p] = c.R[r];
    }
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const bool nx = x[p].x == kPairNone, ny = y[p].x == kPairNone;
        if (nx | ny) {
            none |= 1u << p;
            if (!((nx && x[p].y == 0) || (ny && y[p].y == 0)) && ((alive >> p) & 1u)) wide |= 1u << p;      // (defined, but not narrow)
            x[p] = y[p] = make_int2(1, 1);
        }
    }
    alive &= ~none;
    u32 w2 = 0;
    switch (c.op) {
        case XP_OP_ADD: pair_op<XP_OP_ADD, P>(x, y, a0, a1, alive, w2); break;
        case XP_OP_SUB: pair_op<XP_OP_SUB, P>(x, y, a0, a1, alive, w2); break;
        case XP_OP_MUL: pair_op<XP_OP_MUL, P>(x, y, a0, a1, alive, w2); break;
        case XP_OP_DIV: pair_op<XP_OP_DIV, P>(x, y, a0, a1, alive, w2); break;
        case XP_OP_MOD: pair_op<XP_OP_MOD, P>(x, y, a0, a1, alive, w2); break;
        case XP_OP_MIN: pair_op<XP_OP_MIN, P>(x, y, a0, a1, alive, w2); break;
        case XP_OP_MAX: pair_op<XP_OP_MAX, P>(x, y, a0, a1, alive, w2); break;
        default: w2 = (1u << P) - 1u; break;              // (shifts: exactly)
    }
    w2 &= alive;
    alive &= ~w2;
    wide |= w2;
}

// ---- the kernel ----

__device__ __forceinline__ void join_flush(const PlanDev& plan, int acc, JoinCount& n) {
    u64 e = n.evals;
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if ((threadIdx.x & 31) == 0 && acc >= 0) {
        AccDev* a = &plan.acc[acc];
        if (e) atomicAdd(&a->evals, e);
        if (n.tests) { atomicAdd(&a->filter_tests, n.tests); atomicAdd(&a->join_tests, n.tests); }
        if (n.cands) atomicAdd(&a->tile_cands, n.cands);
        if (n.suspects) atomicAdd(&a->filter_survivors, (u64)n.suspects);
        if (n.passes) atomicAdd(&a->probe_survivors, (u64)n.passes);
    }
    n = JoinCount{0, 0, 0, 0, 0};
}

// Fills what the warp's loops need of a segment: targets, groups and the merged tests.
__device__ __noinline__ void join_fill(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const GrammarDev* g, const HoleDev* hole) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    JoinCtx x;
    {
        const i64 t0 = hole->join_t0, t1 = hole->join_t1;
        const u64 v0 = (u64)(t0 < 0 ? -t0 : t0), v1 = (u64)(t1 < 0 ? -t1 : t1), tm = hole->join_tmod;
        x.t0 = (u32)(u64)t0; x.t1 = (u32)(u64)t1;
        x.small = (v0 | v1) >> 31 == 0;
        x.ut0 = x.small ? (u32)v0 : 0u; x.ut1 = x.small ? (u32)v1 : 0u;
        x.rt0 = hole->join_rt0; x.rt1 = hole->join_rt1; x.rl0 = hole->join_rl0; x.rl1 = hole->join_rl1; x.h0 = hole->join_h0; x.h1 = hole->join_h1;
        x.ft0 = (float)x.ut0; x.ft1 = (float)x.ut1;
        x.tmod = tm < 0xffffffffull ? (u32)tm : 0xffffffffu;
        x.tz = (t0 | t1) == 0;
    }
    u32 lim = 0x7fffffffu, tests = 0;
    u64 pairs = 0;
    i32 n_lin = 0, n_mul = 0, n_other = 0, n_set = 0;
    constexpr u32 kNarrow = (1u << kSlotDiv) | (1u << kSlotMod) | (1u << kSlotMn) | (1u << kSlotMx);
    for (int gi = 0; gi < seg.n_groups; ++gi) {
        const JoinGroup& grp = plan.jgroups[seg.first_group + gi];
        const JoinSet* S = &hole->join_sets[grp.leaf_nt];
        const u32 cabs = S->cabs;
        const int n_entries = S->n_entries, n_const = S->n_const;
        const int n_ops = __popc(grp.fmask) + __popc(grp.smask);
        tests += (u32)((n_entries + (n_const > 0 ? 1 : 0)) * n_ops);
        pairs += g->cnt[grp.leaf_nt][1] * (u64)n_ops;
        u32 cf = grp.fmask, cs = grp.smask, ef = cf, es = cs;
        // operators that cannot reach the target: quotients, remainders, minima and maxima of narrow operands are narrow;
        // a remainder is below its divisor; c / a and c % a are at most |c|
        if (!x.small) { cf &= ~kNarrow; cs &= ~kNarrow; ef &= ~kNarrow; es &= ~kNarrow; }
        if (x.tmod >= cabs) cf &= ~(1u << kSlotMod);
        if (x.tmod > cabs) cs &= ~((1u << kSlotDiv) | (1u << kSlotMod));
        if (n_const == 0) cf = cs = 0;
        if (n_entries == 0) ef = es = 0;
        if (hole->join_none) cf = cs = ef = es = 0;
        const u32 slim = S->ok ? S->lim : 0u;
        lim = slim < lim ? slim : lim;
        if (lane == 0) {
            GroupCtx c;
            c.set = S;
            c.cmin = S->cmin; c.cmax = S->cmax; c.cabs = cabs; c.mm = S->mm; c.fc = (float)cabs; c.n_entries = n_entries;
            c.cf = cf; c.cs = cs; c.ef = ef; c.es = es;
            w.grp[gi] = c;
            if (cf | cs) w.hot.set[n_set] = gi;
        }
        n_set += (cf | cs) != 0u;
        const bool on = lane < n_entries && (ef | es) != 0u;
        JoinEntry e;
        if (on) e = S->e[lane];
        const u32 below = (1u << lane) - 1u;
        const int others = __popc(__ballot_sync(0xffffffffu, on && ((ef | es) & kNarrow)));
        for (int k = 0; k < 3; ++k) {                     // a + v, a - v, v - a
            const bool want = on && (k == 0 ? ((ef | es) >> kSlotAdd) & 1u : k == 1 ? (ef >> kSlotSub) & 1u : (es >> kSlotSub) & 1u);
            const u32 b = __ballot_sync(0xffffffffu, want);
            const int at = n_lin + __popc(b & below);
            if (want && at < kJoinLin) {
                const u32 d0 = k == 0 ? x.t0 - e.v0 : k == 1 ? x.t0 + e.v0 : e.v0 - x.t0, d1 = k == 0 ? x.t1 - e.v1 : k == 1 ? x.t1 + e.v1 : e.v1 - x.t1;
                w.hot.lin[at] = d0 + kPairMix * d1;
            }
            n_lin += __popc(b);
        }
        {
            const bool want = on && (((ef | es) >> kSlotMul) & 1u);
            const u32 b = __ballot_sync(0xffffffffu, want);
            const int at = n_mul + __popc(b & below);
            if (want && at < kJoinEntries) { w.hot.mul0[at] = e.v0; w.hot.mul1[at] = kPairMix * e.v1; }
            n_mul += __popc(b);
        }
        if (others) {
            const int at = n_other + lane;
            if (on && at < kJoinEntries) { w.hot.other[at] = &S->e[lane]; w.hot.other_f[at] = ef & kNarrow; w.hot.other_s[at] = es & kNarrow; }
            n_other += others;
        }
    }
    __syncwarp();
    // (more entries than the lists hold: the exact way)
    if (n_lin > kJoinLin || n_mul > kJoinEntries || n_other > kJoinEntries) lim = 0u;
    else if (lane < 4 && n_lin > 0) w.hot.lin[n_lin + lane] = w.hot.lin[0];
    if (lane == 0) {
        w.x = x;
        w.hot.mul_t = x.t0 + kPairMix * x.t1;
        w.hot.n_lin = n_lin; w.hot.n_mul = n_mul; w.hot.n_other = n_other; w.hot.n_set = n_set;
        w.hot.lim = lim; w.hot.tests = tests; w.hot.pairs = pairs;
    }
    __syncwarp();
}

// What `count` operands from number `first` on stand for in the count of candidates: themselves, or, where the segment counts by class, the
// first ticket's for all that the window covers.
__device__ __forceinline__ u64 seg_operands(const JoinSeg& seg, u64 first, u64 count) {
    return !XP_CLASSES(seg) ? count : first == 0ull ? seg.e_begin : 0ull;
}

// Operands [first, first + count) of a segment against the leaves (count <= the segment's chunk).
template <int P>
__device__ __noinline__ void join_ticket(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole,
                                         u64 first, u64 count, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    n.cands += seg_operands(seg, first, count) * w.hot.pairs;
    const u32 lim = w.hot.lim;
    if (seg.exact == kExactFew) {
        for (u64 i = 0; i < count; ++i) join_exact(w, plan, seg, sk, hole, first + i, n);
        return;
    }
    if (seg.exact || !hole->join_on || lim == 0u) {
        for (u64 i = 0; i < count; i += 32u) join_exact32(w, plan, seg, sk, hole, first + i + lane, i + lane < count, hole->join_p1 ? 2 : 1, n);
        return;
    }
    const JoinCtx x = w.x;
    const int n_lin = w.hot.n_lin, n_mul = w.hot.n_mul, n_other = w.hot.n_other, n_set = w.hot.n_set;
    const u32 mul_t = w.hot.mul_t;
    const u32 tests_each = w.hot.tests;
    u32 nq = w.nq;
    u32 n_alive = 0;
    for (u64 done = 0; done < count;) {
        const JoinRun c = join_run(g, hole, seg.nt, seg.esize, first + done, XP_CLASSES(seg) != 0);
        const u32 n_run = (u32)(c.left < count - done ? c.left : count - done);
        const u32 off0 = (u32)(first + done - w.base) + lane;
        for (u32 at = 0; at < n_run; at += 32u * P) {
            i32 a0[P], a1[P];
            u32 alive, wide;
            run_values<P>(c, g, hole, seg.nt, seg.esize, at, n_run, a0, a1, alive, wide);
            bool any[P];
#pragma unroll
            for (int p = 0; p < P; ++p) {
                any[p] = false;
                if (((alive >> p) & 1u) && (abs_u32(a0[p]) >= lim || abs_u32(a1[p]) >= lim)) { alive &= ~(1u << p); wide |= 1u << p; }
            }
            n_alive += (u32)__popc(alive);
            if (n_lin > 0) {
                u32 h[P];
#pragma unroll
                for (int p = 0; p < P; ++p) h[p] = (u32)a0[p] + kPairMix * (u32)a1[p];
                for (int i = 0; i < n_lin; i += 4) {
                    const uint4 d = *reinterpret_cast<const uint4*>(&w.hot.lin[i]);
#pragma unroll
                    for (int p = 0; p < P; ++p) any[p] |= h[p] == d.x || h[p] == d.y || h[p] == d.z || h[p] == d.w;
                }
            }
            for (int i = 0; i < n_mul; ++i) {
                const u32 v0 = w.hot.mul0[i], v1 = w.hot.mul1[i];
#pragma unroll
                for (int p = 0; p < P; ++p) any[p] |= (u32)a0[p] * v0 + (u32)a1[p] * v1 == mul_t;
            }
            for (int i = 0; i < n_other; ++i) {
                const JoinEntry en = *w.hot.other[i];
                const u32 f = w.hot.other_f[i], s = w.hot.other_s[i];
                constexpr u32 kDivMod = (1u << kSlotDiv) | (1u << kSlotMod);
                if (f == kDivMod && s == kDivMod) entry_conditions<P>(en, kDivMod, kDivMod, a0, a1, x, any);      // (compile-time operators)
                else entry_conditions<P>(en, f, s, a0, a1, x, any);
            }
            for (int i = 0; i < n_set; ++i) {
                const GroupCtx& s = w.grp[w.hot.set[i]];
                const u32 cf = s.cf, cs = s.cs;
                constexpr u32 kRing = (1u << kSlotAdd) | (1u << kSlotSub) | (1u << kSlotMul), kDiv = 1u << kSlotDiv, kMul = 1u << kSlotMul;
                if (cf == kMul && cs == 0u) set_conditions<P, (int)kMul, 0>(s, a0, a1, x, any);
                else if (cf == kDiv && cs == 0u) set_conditions<P, (int)kDiv, 0>(s, a0, a1, x, any);
                else if (cf == (kRing | kDiv) && cs == kRing) set_conditions<P, (int)(kRing | kDiv), (int)kRing>(s, a0, a1, x, any);
                else set_conditions<P, -1, -1>(s, a0, a1, x, any);
            }
            u32 hits = 0;
#pragma unroll
            for (int p = 0; p < P; ++p) hits |= (u32)any[p] << p;
            hits &= alive;
            if (__any_sync(0xffffffffu, hits != 0u)) {
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const bool h = (hits >> p) & 1u;
                    const u32 b = __ballot_sync(0xffffffffu, h);
                    if (h) {
                        const u32 q = nq + (u32)__popc(b & ((1u << lane) - 1u));
                        w.q_off[q] = off0 + at + 32u * p; w.q_a0[q] = a0[p]; w.q_a1[q] = a1[p];
                    }
                    nq += (u32)__popc(b);
                }
                if (nq >= 32u) {                          // whole warps of suspects; the rest waits
                    const u32 full = nq & ~31u;
                    join_drain(w, full, plan, seg, sk, hole, n);
                    nq -= full;
                    u32 o = 0;
                    i32 v0 = 0, v1 = 0;
                    if (lane < (int)nq) { o = w.q_off[full + lane]; v0 = w.q_a0[full + lane]; v1 = w.q_a1[full + lane]; }
                    __syncwarp();
                    if (lane < (int)nq) { w.q_off[lane] = o; w.q_a0[lane] = v0; w.q_a1[lane] = v1; }
                    __syncwarp();
                }
            }
            if (__any_sync(0xffffffffu, wide != 0u)) join_push_wide(w, wide, off0 + at, plan, seg, sk, hole, n);
        }
        done += n_run;
    }
    n.tests += (u64)tests_each * (u64)__reduce_add_sync(0xffffffffu, n_alive);
    if (lane == 0) w.nq = nq;                             // (fewer than 32: they wait for the warp's next ticket of this segment)
    __syncwarp();
}

// Operands [first, first + count), at most 32, against part `part` of the segment's leaves, for small calls: every operator at both probes, without
// conditions and suspects in between (two-variable nest of 1 805 operands and 19 leaves, five operators: join 42 -> 28 us).
__device__ __noinline__ void join_few(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole, u64 first, u64 count,
                                      int part, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    i64 t0 = hole->join_t0, t1 = hole->join_t1;
    const int p1 = hole->join_p1, from = p1 ? 2 : 1;
    u32 lim = hole->join_on ? 0x7fffffffu : 0u, pairs = 0;
    for (int gi = 0; gi < seg.n_groups; ++gi) {
        const JoinGroup& grp = plan.jgroups[seg.first_group + gi];
        const JoinSet* S = &hole->join_sets[grp.leaf_nt];
        const u32 l = S->ok ? S->lim : 0u;
        lim = l < lim ? l : lim;
        pairs += (u32)g->cnt[grp.leaf_nt][1] * (u32)(__popc(grp.fmask) + __popc(grp.smask));
    }
    if (part == 0) n.cands += count * (u64)pairs;
    for (u64 done = 0; done < count;) {
        const JoinRun c = join_run(g, hole, seg.nt, seg.esize, first + done, false);
        const u32 n_run = (u32)(c.left < count - done ? c.left : count - done);
        i32 a0[1], a1[1];
        u32 alive, wide;
        run_values<1>(c, g, hole, seg.nt, seg.esize, 0u, n_run, a0, a1, alive, wide);
        if (alive && (abs_u32(a0[0]) >= lim || abs_u32(a1[0]) >= lim)) { alive = 0u; wide = 1u; }
        const u64 e = first + done + lane;
        // (wide operands meet all leaves at once, in the first part)
        if (part == 0 && __any_sync(0xffffffffu, wide != 0u)) join_exact32(w, plan, seg, sk, hole, e, wide != 0u, from, n);
        const u32 off = (u32)(e - w.base), n_alive = (u32)__popc(__ballot_sync(0xffffffffu, alive != 0u));
        if (n_alive != 0u && !hole->join_none)
            for (int gi = 0; gi < seg.n_groups; ++gi) {
                const JoinGroup& grp = plan.jgroups[seg.first_group + gi];
                const u32 want = grp.fmask | (grp.smask << 16);
                const bool divide = (want & (0x10001u << kSlotDiv | 0x10001u << kSlotMod)) != 0u;
                const int nl = (int)g->cnt[grp.leaf_nt][1], lb = g->leaf_begin[grp.leaf_nt];
                const int l0 = (int)((i64)nl * part / seg.parts), l1 = (int)((i64)nl * (part + 1) / seg.parts);
                n.tests += (u64)((l1 - l0) * __popc(want)) * n_alive;
                for (int at = l0; at < l1; at += 32) {
                    i32 c0 = 0, c1 = 0;
                    if (at + lane < l1) {
                        const LeafDev lf = g->leaves[lb + at + lane];
                        c0 = (i32)(lf.var >= 0 ? hole->probe_pt[0][lf.var] : lf.value);
                        c1 = (i32)(lf.var >= 0 ? hole->probe_pt[p1][lf.var] : lf.value);
                    }
                    const int m = l1 - at < 32 ? l1 - at : 32;
#pragma unroll 1
                    for (int i = 0; i < m; ++i) {
                        u32 hits = alive ? want : 0u;
#pragma unroll 1
                        for (int k = 0; k < 2; ++k) {
                            hits &= narrow_bits(k ? a1[0] : a0[0], __shfl_sync(0xffffffffu, k ? c1 : c0, i), k ? t1 : t0, divide);
                            if (!__any_sync(0xffffffffu, hits != 0u)) break;
                        }
                        n.suspects += (u32)__reduce_add_sync(0xffffffffu, (u32)__popc(hits));
#pragma unroll 1
                        for (u32 b = __reduce_or_sync(0xffffffffu, hits); b; b &= b - 1) {
                            const int bit = __ffs((int)b) - 1;
                            join_push(w, plan, seg, sk, hole, (hits >> bit) & 1u, off, (u32)(at + i), gi, bit & 15, bit >> 4, from, n);
                        }
                    }
                }
            }
        done += n_run;
    }
}

// What waits in the warp's queues when it leaves segment `index`.
__device__ __noinline__ void join_leave(JoinWarp& w, const PlanDev& plan, int index, JoinCount& n) {
    const JoinSeg& seg = plan.jsegs[index];
    const SketchDev* sk = plan.sketches[seg.sketch];
    const HoleDev* hole = &sk->holes[seg.hole];
    if (w.nq) join_drain(w, w.nq, plan, seg, sk, hole, n);
    if (w.nw) join_wide(w, w.nw, plan, seg, sk, hole, n);
    if (w.nc) join_check(w, plan, seg, sk, hole, hole->join_p1 ? 2 : 1, n);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) { w.nq = w.nw = 0; w.seg = -1; }
    __syncwarp();
}

// ---- contexts that compare ----

// Operand values at the first kRangeProbes probes sit in registers; leaves are held against those with an early exit.
constexpr int kRangeProbes = 4;

// The constants c of the ascending list [cb, vb) for which  a op c  (swap: c op a) can lie in the hole's interval at all np
// probes (a: the operand's values there), as up to two runs.  For * / min and max; a necessary condition: bounds are taken
// in double precision and widened by more than its rounding.  (With four probes instead of all the runs were so much
// longer that testing them was most of the ticket.)
__device__ __noinline__ void range_runs(const HoleDev* hole, int np, const ConstDev* c, i32 cb, i32 vb, int slot, int swap, const i32 (&a)[kMaxProbe],
                                        i32 (&run)[4]) {
    constexpr i64 kMost = 1ll << 62;
    run[0] = run[1] = run[2] = run[3] = cb;
    constexpr i64 kEnd = (1ll << 31) + 1;
    constexpr double kEps = 1e-15;
    auto clip = [](double x) { return (i64)(x < -2147483650.0 ? -2147483650.0 : x > 2147483650.0 ? 2147483650.0 : x); };
    if (slot == kSlotDiv && !swap) {                      // floor(|a| / |c|) in an interval that depends on the signs
        i64 f[2] = {1, 1}, t[2] = {kEnd, kEnd};           // |c| for c > 0 and c < 0
        for (int j = 0; j < np && (f[0] <= t[0] || f[1] <= t[1]); ++j) {
            const double u = fabs((double)a[j]);
            const i64 l = hole->rng_lo[j] < -kMost ? -kMost : hole->rng_lo[j], h = hole->rng_hi[j] > kMost ? kMost : hole->rng_hi[j];
            for (int k = 0; k < 2; ++k) {
                const bool same = (a[j] >= 0) == (k == 0);
                const i64 L = same ? l : -h, H = same ? h : -l;
                if (H < 0) { t[k] = 0; continue; }
                const i64 from = clip(floor(u / ((double)H + 1.0) * (1.0 - kEps))) + 1;
                f[k] = from > f[k] ? from : f[k];
                if (L > 0) { const i64 to = clip(floor(u / (double)L * (1.0 + kEps))); t[k] = to < t[k] ? to : t[k]; }
            }
        }
        if (f[0] <= t[0]) { run[0] = const_lower(c, cb, vb, f[0]); run[1] = const_lower(c, run[0], vb, t[0] + 1); }
        if (f[1] <= t[1]) { run[2] = const_lower(c, cb, vb, -t[1]); run[3] = const_lower(c, run[2], vb, -f[1] + 1); }
        return;
    }
    i64 f = -kEnd, t = kEnd;
    for (int j = 0; j < np && f <= t; ++j) {
        const i64 l = hole->rng_lo[j] < -kMost ? -kMost : hole->rng_lo[j], h = hole->rng_hi[j] > kMost ? kMost : hole->rng_hi[j], v = a[j];
        i64 from = -kEnd, to = kEnd;
        if (slot == kSlotMul) {
            if (v == 0) { if (l > 0 || h < 0) return; }
            else {
                const double q0 = (double)(v > 0 ? l : h) / (double)v, q1 = (double)(v > 0 ? h : l) / (double)v;
                from = clip(ceil(q0 - fabs(q0) * kEps)); to = clip(floor(q1 + fabs(q1) * kEps));
            }
        } else if (slot == kSlotDiv) {                    // c / a
            if (v == 0) return;
            const i64 m = v < 0 ? -v : v;
            i64 L = v > 0 ? l : -h, H = v > 0 ? h : -l;   // c / |a| in [L, H]
            L = L < -kEnd ? -kEnd : L > kEnd ? kEnd : L; H = H < -kEnd ? -kEnd : H > kEnd ? kEnd : H;
            from = L > 0 ? L * m : (L - 1) * m + 1; to = H < 0 ? H * m : (H + 1) * m - 1;
        } else if (slot == kSlotMn) {
            if (v < l) return;
            from = l; if (v > h) to = h;
        } else {
            if (v > h) return;
            to = h; if (v < l) from = l;
        }
        f = from > f ? from : f; t = to < t ? to : t;
    }
    if (f <= t) { run[0] = const_lower(c, cb, vb, f); run[1] = const_lower(c, run[0], vb, t + 1); }
}

// Is  x op y  in range at all of the kRangeProbes probes?  The operator is chosen once, the probes are straight-line code.
template <int SLOT>
__device__ __forceinline__ bool range_holds(const i32 (&x)[kRangeProbes], const i32 (&y)[kRangeProbes], const i64 (&lo)[kRangeProbes], const i64 (&hi)[kRangeProbes]) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < kRangeProbes; ++j) {
        i64 v = 0;
        ok = narrow_op(SLOT, x[j], y[j], v) && ok && v >= lo[j] && v <= hi[j];
    }
    return ok;
}
__device__ __forceinline__ bool range_accepts(int slot, const i32 (&x)[kRangeProbes], const i32 (&y)[kRangeProbes], const i64 (&lo)[kRangeProbes],
                                              const i64 (&hi)[kRangeProbes]) {
    switch (slot) {
        case kSlotAdd: return range_holds<kSlotAdd>(x, y, lo, hi);
        case kSlotSub: return range_holds<kSlotSub>(x, y, lo, hi);
        case kSlotMul: return range_holds<kSlotMul>(x, y, lo, hi);
        case kSlotDiv: return range_holds<kSlotDiv>(x, y, lo, hi);
        case kSlotMod: return range_holds<kSlotMod>(x, y, lo, hi);
        case kSlotMn: return range_holds<kSlotMn>(x, y, lo, hi);
        default: return range_holds<kSlotMx>(x, y, lo, hi);
    }
}

// Operands [first, first + count) of a segment against the leaves, for a hole whose context compares: the value has to
// lie in [rng_lo, rng_hi] at every probe.
// Against part `part` of the constants where a segment has several (the variables and wide operands are in the first).
__device__ __noinline__ void range_ticket(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole,
                                          u64 first, u64 count, int part, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    const int np = hole->n_exact, nr = np < kRangeProbes ? np : kRangeProbes;
    static_assert(kRangeProbes == kProbeStep, "the first step's values are the range probes'");
    constexpr i64 kMost = 1ll << 62;
    i64 lo[kRangeProbes], hi[kRangeProbes];
#pragma unroll
    for (int j = 0; j < kRangeProbes; ++j) {              // (probes beyond the last repeat the first)
        const int k = j < nr ? j : 0;
        lo[j] = hole->rng_lo[k] < -kMost ? -kMost : hole->rng_lo[k];
        hi[j] = hole->rng_hi[k] > kMost ? kMost : hole->rng_hi[k];
    }
    bool sets_ok = (hole->aff_okmask & ((1u << np) - 1u)) == 0u;      // (every probe compares: it does not depend on the point)
    u64 pairs = 0;
    for (int gi = 0; gi < seg.n_groups; ++gi) {
        const JoinGroup& grp = plan.jgroups[seg.first_group + gi];
        pairs += g->cnt[grp.leaf_nt][1] * (u64)(__popc(grp.fmask) + __popc(grp.smask));
        sets_ok = sets_ok && hole->join_sets[grp.leaf_nt].ok != 0;
    }
    const int parts = seg.parts > 1 ? seg.parts : 1;
    if (part == 0) n.cands += seg_operands(seg, first, count) * pairs;
    for (u64 at = 0; at < count; at += 32) {
        const u64 e = first + at + lane;
        const bool have = at + lane < count;
        OperandRef ref;
        ref.mode = 2; ref.op = 0; ref.a = ref.b = 0;
        i32 a[kRangeProbes] = {0}, every[kMaxProbe];      // its values at the first probes, and at all of them
        // interval of constants c with a + c in range at every probe, and (swapped difference) with c - a in range
        i64 pl = -kMost, ph = kMost, ml = -kMost, mh = kMost;
        bool live = false, wide = false;
        if (have) {
            ref = operand_ref(g, hole, seg.nt, seg.esize, XP_CLASSES(seg) ? class_operand(g, hole, seg.nt, seg.esize, e).rank(0) : e);
            live = true;
            for (int j0 = 0; j0 < np && live && !wide; j0 += kProbeStep) {
                i64 val[kProbeStep];
                const int here = np - j0 < kProbeStep ? np - j0 : kProbeStep;
                live = ref_value4(g, hole, ref, seg.nt, seg.esize, j0, np, val) == (1u << here) - 1u;
#pragma unroll
                for (int q = 0; q < kProbeStep; ++q) {
                    if (q >= here) continue;
                    const int j = j0 + q;
                    const i64 v = val[q];
                    wide = wide || !narrow31(v);
                    every[j] = (i32)v;
                    const i64 l = hole->rng_lo[j] < -kMost ? -kMost : hole->rng_lo[j], h = hole->rng_hi[j] > kMost ? kMost : hole->rng_hi[j];
                    pl = pl > l - v ? pl : l - v; ph = ph < h - v ? ph : h - v;
                    ml = ml > l + v ? ml : l + v; mh = mh < h + v ? mh : h + v;
                    if (j0 == 0) {
#pragma unroll
                        for (int k = 0; k < kRangeProbes; ++k) if (k == q || (k >= nr && q == 0)) a[k] = (i32)v;
                    }
                }
            }
        }
        if (!sets_ok) wide = live;
        if (part == 0 && __any_sync(0xffffffffu, live && wide)) join_exact32(w, plan, seg, sk, hole, e, live && wide, 0, n);
        live = live && !wide;
        const u32 off = (u32)(e - w.base);
        const u32 n_live = (u32)__popc(__ballot_sync(0xffffffffu, live));
        if (n_live == 0u) continue;
        auto accepted = [&](int slot, int swap, const i32 (&cv)[kRangeProbes]) {      // at the first nr probes
            i32 x[kRangeProbes], y[kRangeProbes];
#pragma unroll
            for (int j = 0; j < kRangeProbes; ++j) { x[j] = swap ? cv[j] : a[j]; y[j] = swap ? a[j] : cv[j]; }
            return range_accepts(slot, x, y, lo, hi);
        };
        auto give = [&](bool on, u32 pos, int gi, int slot, int swap) {
            const u32 b = __ballot_sync(0xffffffffu, on);
            if (!b) return;
            n.suspects += (u32)__popc(b);
            join_push(w, plan, seg, sk, hole, on, off, pos, gi, slot, swap, 0, n);
        };
        // Remainders: magnitude in [mag, mag + span] for a value >= 0 (0) or <= 0 (1); kNever where no such value is in range.
        constexpr u32 kNever = 0x80000000u;
        auto bound = [](i64 l, i64 h, u32& from, u32& span) {
            if (h < 0 || l > 0x7fffffffll) { from = kNever; span = 0; return; }
            from = l < 0 ? 0u : (u32)l;
            span = (u32)(h > 0x7fffffffll ? 0x7fffffffll : h) - from;
            if (h < (i64)from) { from = kNever; span = 0; }
        };
        u32 ua[kRangeProbes], ra[kRangeProbes], pm[kRangeProbes], ps[kRangeProbes], nm[kRangeProbes], ns[kRangeProbes];
        bool none0 = false;                               // some a is zero (no remainder by it)
#pragma unroll
        for (int j = 0; j < kRangeProbes; ++j) {
            ua[j] = abs_u32(a[j]);
            ra[j] = ua[j] <= 1u ? 0xffffffffu : 0xffffffffu / ua[j];
            none0 = none0 || ua[j] == 0u;
            bound(lo[j], hi[j], pm[j], ps[j]);
            bound(-hi[j], -lo[j], nm[j], ns[j]);
        }
        for (int gi = 0; gi < seg.n_groups; ++gi) {
            const JoinGroup& grp = plan.jgroups[seg.first_group + gi];
            const i32 c_first = g->const_begin[grp.leaf_nt], vb_all = g->var_begin[grp.leaf_nt];
            const i32 cb = c_first + (vb_all - c_first) * part / parts, vb = c_first + (vb_all - c_first) * (part + 1) / parts;      // this part's constants
            const i32 v_first = part == 0 ? vb_all : g->const_begin[grp.leaf_nt + 1], ve = g->const_begin[grp.leaf_nt + 1];
            for (int swap = 0; swap < 2; ++swap) {
                const u32 mask = swap ? grp.smask : grp.fmask;
                n.tests += (u64)n_live * (u64)(__popc(mask) * ((part == 0 ? 1 : 0) + ve - v_first));
                for (u32 m = cb < vb ? mask & ~(1u << kSlotMod) : 0u; m; m &= m - 1) {
                    const int slot = __ffs((int)m) - 1;
                    i32 run[4] = {cb, cb, cb, cb};
                    if (slot <= kSlotSub) {               // by the intersection over all probes
                        const i64 from = slot == kSlotAdd ? pl : swap ? ml : -ph, to = slot == kSlotAdd ? ph : swap ? mh : -pl;
                        if (live && from <= to) { run[0] = const_lower(g->consts, cb, vb, from); run[1] = const_lower(g->consts, run[0], vb, to + 1); }
                    } else if (live) range_runs(hole, np, g->consts, cb, vb, slot, swap, every, run);
                    const i32 len0 = run[1] - run[0], len = len0 + run[3] - run[2];
                    for (i32 i = 0; __any_sync(0xffffffffu, i < len); ++i) {
                        bool on = i < len;
                        const ConstDev c = g->consts[on ? (i < len0 ? run[0] + i : run[2] + i - len0) : cb];
                        if (on && slot > kSlotSub) {
                            const i32 cv[kRangeProbes] = {(i32)c.value, (i32)c.value, (i32)c.value, (i32)c.value};
                            on = accepted(slot, swap, cv);
                        }
                        give(on, (u32)c.pos, gi, slot, swap);
                    }
                }
                if (((mask >> kSlotMod) & 1u) && cb < vb) {
                    if (!swap) {                          // a % c: the sign of a
                        u32 m[kRangeProbes], sp[kRangeProbes];
                        bool can = live;
#pragma unroll
                        for (int j = 0; j < kRangeProbes; ++j) {
                            m[j] = a[j] >= 0 ? pm[j] : nm[j]; sp[j] = a[j] >= 0 ? ps[j] : ns[j];
                            can = can && m[j] != kNever;
                        }
                        if (__any_sync(0xffffffffu, can))
                            for (i32 c0 = cb; c0 < vb; c0 += 32) {      // 32 constants without a branch, then those with a hit
                                const int nc = vb - c0 < 32 ? vb - c0 : 32;
                                u32 hits = 0;
#pragma unroll 4
                                for (int k = 0; k < nc; ++k) {
                                    const ConstDev c = g->consts[c0 + k];
                                    const u32 uc = abs_u32((i32)c.value);
                                    u32 on = uc != 0u;
#pragma unroll
                                    for (int j = 0; j < kRangeProbes; ++j) {
                                        u32 r = ua[j] - __umulhi(ua[j], c.recip) * uc;
                                        r = r >= uc ? r - uc : r;
                                        on &= (u32)(r - m[j] <= sp[j]);
                                    }
                                    hits |= on << k;
                                }
                                if (!can) hits = 0;
                                for (u32 q = __reduce_or_sync(0xffffffffu, hits); q; q &= q - 1) {
                                    const int k = __ffs((int)q) - 1;
                                    give((hits >> k) & 1u, (u32)g->consts[c0 + k].pos, gi, kSlotMod, 0);
                                }
                            }
                    } else if (__any_sync(0xffffffffu, live && !none0))
                        for (i32 c0 = cb; c0 < vb; c0 += 32) {          // c % a: the sign of c
                            const int nc = vb - c0 < 32 ? vb - c0 : 32;
                            u32 hits = 0;
#pragma unroll 4
                            for (int k = 0; k < nc; ++k) {
                                const ConstDev c = g->consts[c0 + k];
                                const u32 uc = abs_u32((i32)c.value);
                                const bool pos = c.value >= 0;
                                u32 on = 1u;
#pragma unroll
                                for (int j = 0; j < kRangeProbes; ++j) {
                                    u32 r = uc - __umulhi(uc, ra[j]) * ua[j];
                                    r = r >= ua[j] ? r - ua[j] : r;
                                    on &= (u32)(r - (pos ? pm[j] : nm[j]) <= (pos ? ps[j] : ns[j]));
                                }
                                hits |= on << k;
                            }
                            if (!live || none0) hits = 0;
                            for (u32 q = __reduce_or_sync(0xffffffffu, hits); q; q &= q - 1) {
                                const int k = __ffs((int)q) - 1;
                                give((hits >> k) & 1u, (u32)g->consts[c0 + k].pos, gi, kSlotMod, 1);
                            }
                        }
                }
                for (i32 ci = v_first; ci < ve; ++ci) {   // variables one by one
                    const ConstDev c = g->consts[ci];
                    i32 cv[kRangeProbes];
#pragma unroll
                    for (int j = 0; j < kRangeProbes; ++j) cv[j] = (i32)hole->probe_pt[j < nr ? j : 0][c.value];
                    for (u32 m = mask; m; m &= m - 1) {
                        const int slot = __ffs((int)m) - 1;
                        give(live && accepted(slot, swap, cv), (u32)c.pos, gi, slot, swap);
                    }
                }
            }
        }
    }
    if (w.nc) join_check(w, plan, seg, sk, hole, 0, n);
}

// Candidates [first, first + count) of (start nonterminal, size) themselves, checked on the probes one by one.
__device__ __noinline__ void direct_ticket(JoinWarp& w, const PlanDev& plan, const JoinSeg& seg, const SketchDev* sk, const HoleDev* hole,
                                           u64 first, u64 count, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    const int n_exact = hole->n_exact;
    for (u64 at = first; at < first + count; at += 32) {
        const u64 rank = at + lane;
        bool pass = false;
        u32 vars = 0;
        if (rank < first + count) {
            const OperandRef ref = operand_ref(g, hole, seg.nt, seg.esize, rank);
            pass = true;
            for (int j0 = 0; j0 < n_exact && pass; j0 += kProbeStep) {
                const int here = n_exact - j0 < kProbeStep ? n_exact - j0 : kProbeStep;
                n.evals += (u64)here;
                i64 v[kProbeStep];
                pass = ref_value4(g, hole, ref, seg.nt, seg.esize, j0, n_exact, v) == (1u << here) - 1u && probes_accept(hole, j0, n_exact, v);
            }
            vars = ref_vars(hole, ref);
        }
        if (n_exact < hole->n_probe) pass = join_full_check(g, hole, seg.size, pass, rank, n.evals);
        const u32 b = __ballot_sync(0xffffffffu, pass);
        n.suspects += (u32)__popc(b);
        join_survive(w.cand, plan, sk, hole, seg, pass, rank, vars, n);
    }
}

template <int P>
__global__ void __launch_bounds__(kJoinThreads, 2) join_kernel(const __grid_constant__ PlanDev plan) {
    chain_wait();
    __shared__ JoinWarp sh[kJoinWarps];
    JoinWarp& w = sh[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    if (lane == 0) { w.nq = w.nc = w.nw = 0; w.seg = -1; }
    __syncwarp();
    JoinCount n{0, 0, 0, 0, 0};
    int acc = -1;
    const u64 warps = (u64)gridDim.x * kJoinWarps;
    // the first ticket is the warp's number (warp-in-CTA major, so that a small search spreads over the SMs), the others
    // come from the counter
    u64 t = plan.join_base + (u64)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    while (t < plan.n_join) {
        int lo = 0, k = plan.n_jsegs;
        while (k > 1) {                                   // last segment with first_ticket <= t: one probe per lane and round
            const int step = (k + 31) / 32;
            const int pos = lo + lane * step;
            const bool le = pos < lo + k && plan.jsegs[pos].first_ticket <= t;
            const u32 mask = __ballot_sync(0xffffffffu, le);
            const int j = 31 - __clz((int)(mask | 1u));
            const int nlo = lo + j * step;
            k = (lo + k - nlo) < step ? (lo + k - nlo) : step;
            lo = nlo;
        }
        const JoinSeg& seg = plan.jsegs[lo];
        const u64 chunk = seg.chunk;
        u32 part = 0;
        u64 block = t - seg.first_ticket;
        if (seg.parts > 1) { part = (u32)block % (u32)seg.parts; block = (u32)block / (u32)seg.parts; }      // (few tickets: see number_joins)
        const u64 from = block * chunk, first = (XP_CLASSES(seg) ? 0ull : seg.e_begin) + from;
        // (what waits in the queues is numbered in 32 bits, and a warp's tickets ascend)
        if (w.seg >= 0 && (w.seg != lo || (first + chunk - w.base) >> 32)) join_leave(w, plan, w.seg, n);
        if (seg.acc != acc) { join_flush(plan, acc, n); acc = seg.acc; }
        const SketchDev* sk = plan.sketches[seg.sketch];
        const HoleDev* hole = &sk->holes[seg.hole];
        if (seg.kind == kJoinLeaf && w.seg != lo) {
            const bool fill = hole->aff_ok || seg.exact;
            if (fill && seg.parts == 0) join_fill(w, plan, seg, sk->g, hole);
            if (lane == 0) { w.base = first; if (fill) w.seg = lo; }
            __syncwarp();
        }
        const u32 all = hole->n_probe >= 32 ? 0xffffffffu : (1u << hole->n_probe) - 1u;
        if ((hole->probe_spec_ok & all) == all && from < seg.e_count) {      // (a spec undefined at a probe: nothing can match)
            const u64 count = seg.e_count - from < chunk ? seg.e_count - from : chunk;
            if (seg.kind == kJoinDirect) direct_ticket(w, plan, seg, sk, hole, first, count, n);
            else if (!hole->aff_ok && !seg.exact) range_ticket(w, plan, seg, sk, hole, first, count, (int)part, n);
#if !XP_JOIN_BATCH
            else if (seg.parts > 0) join_few(w, plan, seg, sk, hole, first, count, (int)part, n);
#endif
            else join_ticket<P>(w, plan, seg, sk, hole, first, count, n);
        }
        u64 next = 0;
        if (lane == 0) next = atomicAdd(plan.join_ticket, 1ull);
        t = plan.join_base + warps + __shfl_sync(0xffffffffu, next, 0);
    }
    if (w.seg >= 0) join_leave(w, plan, w.seg, n);
    join_flush(plan, acc, n);
}

}
}  // namespace xp
