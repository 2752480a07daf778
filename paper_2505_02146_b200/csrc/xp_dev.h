// Structures shared by the host encoder and the device kernels of libxpiler_repair.
// Everything here is plain data laid out by the host and read by the kernels.
#pragma once

#include <stdint.h>
#include <vector_types.h>

#include "xp.h"

namespace xp {

typedef unsigned long long u64;
typedef long long i64;
typedef unsigned int u32;
typedef int i32;

constexpr int kMaxSize = XP_MAX_SIZE;
constexpr int kMaxVars = XP_MAX_VARS;
constexpr int kMaxNt = XP_MAX_NONTERMINALS;
constexpr int kMaxCode = XP_MAX_CODE;
constexpr int kMaxStack = 16;        // deepest operand stack of a context / spec expression
constexpr int kCandStack = 8;        // deepest operand stack of a candidate (size <= 15 => <= 8 leaves)
constexpr int kMaxProbe = 16;        // probe points per sketch
constexpr int kProbeSamples = 64;    // sample points the probes are chosen from
constexpr int kThreads = 256;        // threads per CTA of the evaluation kernel
constexpr int kLinearChunk = kThreads * 4;   // ranks per linear ticket
constexpr int kNA = 8;                // tile tickets: register-side operands per thread
constexpr int kRegTile = kThreads * kNA;     // register-side operands per tile
constexpr int kBcTile = 512;          // broadcast-side operands per tile
constexpr int kBcTileSlow = 8;        // ... of a hole whose context compares (interval test in 64 bits per candidate)
constexpr u64 kStageMaxPoints = 1ull << 26;  // largest box whose points and spec values are staged in HBM at load
constexpr int kProgMax = 64;          // candidate substituted into its context: longest staged program
constexpr u64 kTabBudgetBytes = 64ull << 20;   // subtree-value tables of one hole, all probes together
constexpr u64 kTabMaxEntries = 1ull << 22;   // largest (nonterminal, size) subtree-value table per hole
constexpr u32 kOpBit = 0x80000000u;  // candidate code word: operator (low bits = XP_OP_*) or leaf index
constexpr int kMaxFamily = 8;         // tile segments that may share one fill of the register-side operands (a hit's
                                      // queue entry names its member in 3 bits)

// A leaf production: a variable (var >= 0) or a constant.
struct LeafDev { i32 var; i32 pad; i64 value; };

// A binary production and, per candidate size s, the number of trees of its nonterminal that
// precede its first tree (off[s]), i.e. the rank offset of the production at that size.
struct BinDev { i32 op, lnt, rnt, pad; u64 off[kMaxSize + 2]; };

struct ConstDev;
struct GrammarDev {
    i32 n_vars, n_nt, n_leaves, n_bins;
    i32 leaf_begin[kMaxNt + 1];      // leaves of nonterminal nt: leaves[leaf_begin[nt] .. leaf_begin[nt+1])
    i32 bin_begin[kMaxNt + 1];       // binary productions of nt: bins[bin_begin[nt] .. bin_begin[nt+1])
    u64 cnt[kMaxNt][kMaxSize + 1];   // trees of nt with exactly s nodes
    i32 const_begin[kMaxNt + 1];     // constants of nt, ascending: consts[const_begin[nt] .. var_begin[nt]); then its
    i32 var_begin[kMaxNt];           // variables: consts[var_begin[nt] .. const_begin[nt+1]), value = variable
    const LeafDev* leaves;           // device
    const BinDev* bins;              // device
    const ConstDev* consts;          // device
};

// ---- the leaf join (csrc/xp_join.cuh) ----
//
// Candidates  E op leaf  and  leaf op E  are not tested one by one: a thread holds the operand E's values at two
// probes (a0, a1) and asks, per operator, for which leaves the result can be the target at both.  Constants have the
// same value at both probes, so one condition on (a0, a1) decides all of them at once; the variables, and constants
// when there are only a few, are entries that are tested one by one.
//
// Least m with m mod u0 = t0 and m mod u1 = t1, ~0 when there is none (u0 > t0, u1 > t1, both below 2^31): m = t0 + u0 k with
// u0 k = t1 - t0 modulo u1, solved by the extended Euclidean algorithm.
#ifdef __CUDACC__
#define XP_HD __host__ __device__
#else
#define XP_HD
#endif
constexpr u32 kResidueSteps = 24;     // as many steps cost about what that algorithm does
XP_HD inline u64 residue_least(u32 u0, u32 u1, u32 t0, u32 t1) {
    u32 g = u1, r = u0 % u1;
    i32 x = 0, y = 1;                 // y u0 = r, x u0 = g (modulo u1)
    while (r != 0u) {
        const u32 q = g / r, s = g - q * r;
        const i32 z = x - (i32)q * y;
        g = r; r = s;
        x = y; y = z;
    }
    const i64 d = (i64)t1 - (i64)t0;
    if (d % (i64)g != 0) return ~0ull;
    const u32 n = u1 / g;             // k is known modulo n
    const i64 inv = x < 0 ? (i64)x + (i64)n : (i64)x, e = (d / (i64)g) % (i64)n;
    const u64 k = (u64)(inv % (i64)n) * (u64)(e < 0 ? e + (i64)n : e) % (u64)n;
    return (u64)t0 + (u64)u0 * k;
}
constexpr int kOpSlots = 9;           // + - * / % min max << >> (in this order; the last two only in the exact form)
constexpr int kJoinEntries = 12;      // most leaves of a nonterminal that are tested one by one
constexpr int kJoinFewConsts = 4;     // constants up to this many are entries too
struct __align__(16) JoinEntry {
    u32 v0, v1, u0, u1;               // value at the two probes, and its magnitude
    u32 low0, low1, cm0, cm1;         // as divisor: |target| * |v| (0x80000000: never); floor((2^32-1) / |v|), 0 when the remainder is impossible
    u32 inv0, inv1, k0k1, pos;        // inverse of |v|'s odd part, trailing zero bits (k0 | k1 << 8); position among the nonterminal's leaves
};
struct JoinSet {                      // the leaves of one nonterminal, for one hole
    i32 ok;                           // every value is below 2^31 in magnitude and the entries fit
    i32 n_entries, n_const;           // n_const: constants decided as a set (0 when they are entries)
    i32 cmin, cmax;                   // ... their range
    u32 cabs;                         // ... and largest magnitude
    u32 lim;                          // operands of this magnitude or more are left to the exact form
    u32 mm;                           // bit 0 / 1: the target at probe 0 / 1 is one of the constants (min and max)
    i32 const_begin;                  // into GrammarDev::consts (ascending)
    i32 pad[3];
    JoinEntry e[kJoinEntries];
};

// A constant leaf of a nonterminal (position among its leaves); recip: floor(2^32 / |value|), 2^32 - 1 for 1, 0 for 0 and
// values of 2^31 or more.
struct ConstDev { i64 value; i32 pos; u32 recip; };

struct HoleDev {
    i32 start_nt, max_size, ctx_len, spec_len;   // spec_len == 0: the spec is a table
    const i64* spec_table;                        // device, n_points values: the caller's table, or the spec
                                                  // expression evaluated once per point at load (null: evaluate)
    xp_instr ctx[kMaxCode];
    xp_instr spec[kMaxCode];
    // Probe points of this hole, most discriminating first (written by the prepare kernel).
    i32 n_probe;
    u32 probe_spec_ok;                            // bit j: the spec is defined at probe j
    i64 probe_id[kMaxProbe];
    i64 probe_pt[kMaxProbe][kMaxVars];
    i64 probe_spec[kMaxProbe];                    // spec at the probe points
    // Context at probe 0 as an affine map of the hole value, ctx(h) = aff_A * h + aff_B in
    // wrap-around arithmetic (possible when the hole only passes through + - * with
    // hole-free operands); aff_ok == 0: not of that form, the probe filter is not used.
    i32 aff_ok;
    u32 aff_okmask;                               // bit j: the context is affine in the hole at probe j too,
    u64 aff_A, aff_B;                             //        ctx(h) = aff_Aj[j] * h + aff_Bj[j]
    u64 aff_Aj[kMaxProbe], aff_Bj[kMaxProbe];
    // Contexts that compare: when the context is  X < c,  X <= c,  c < X  or  c <= X  with X = +-h + B
    // (h the hole value, B and c hole-free), the hole values that satisfy the constraint at probe j
    // form the interval [rng_lo[j], rng_hi[j]] (LLONG_MIN / LLONG_MAX for an open end; lo > hi: none).
    // Such a hole (a loop bound stated through its guard predicate) is filtered on that interval
    // where an affine context is filtered on equality.  Bit j of rng_okmask: probe j has the form.
    u32 rng_okmask, pad3;
    i64 rng_lo[kMaxProbe], rng_hi[kMaxProbe];
    // Values at probe 0 of every subtree of the small sizes 1..tab_max_size, by (nonterminal,
    // size, rank): tab_val[tab_off[nt][size] + rank], with tab_ok telling whether the subtree
    // is defined there (no zero divisor).  Built bottom-up once per sketch; operands of the
    // filter stage are looked up here instead of being unranked again in every tile.
    // The tables exist for the probes 0 .. tab_probes-1, one copy after the other (stride tab_total).
    // Hits of the filter are checked exactly there (two lookups and one operation per probe); only
    // probes without tables need the candidate unranked in full.
    // second: filter hits are also checked exactly at probe 1 before they are queued (needs tables, a
    // defined spec and an affine context at probe 1); sample_pass0: how many of the sample_n small
    // candidates sampled at load satisfied probe 0 (a high rate makes the second look worth its cost).
    i32 second, sample_pass0, sample_n, sample_pass;      // sample_pass: how many of them satisfied every probe that has tables
    i32 second_ok;                                // the second look is possible (tables, spec and context at probe 1): a
                                                  // CTA that sees many filter hits for this hole turns it on for itself
    // Set by the host before the load's kernels run: the largest subtree size and the number of
    // probes that the tables may cover (their memory is laid out for that many), and whether the
    // search is small (then the second look is always taken).  prepare_kernel derives
    // tab_max_size, tab_probes, second and filter_ok from them and from the probes it chose.
    i32 tab_size_cap, tab_probes_cap, small_search;
    i32 filter_ok;                                // the probe filter applies: probe 0 exists, its context is affine or compares
    i32 tab_max_size, tab_probes;
    u64 tab_total;
    u64 tab_off[kMaxNt][kMaxSize + 1];
    i64* tab_val;                                 // device
    unsigned char* tab_ok;                        // device
    unsigned char* tab_vars;                      // device, one copy: bit v set if variable v occurs in the subtree
    // Variables that can decide whether a hole value satisfies the constraint (all of them when the spec is the
    // caller's table; see constraint_vars).  On a box domain a candidate is checked on the sub-box of these and its
    // own variables only: no other variable can change either side of the constraint.
    u32 fixed_vars, spec_bad;                     // spec_bad: set by the load when the spec is undefined at some point
    // The leaf join: values (a0, a1) at its two probes of every tabulated subtree, 8 bytes each (same index as
    // tab_val; a0 = kPairNone: undefined at one of them (a1 = 0) or not below 2^31 in magnitude (a1 = 1)); the leaf sets
    // of the nonterminals; the targets.  join_on: the context is affine at both probes with a factor that has
    // at most 31 zero bits at its end.
    i32 join_on, join_p1;                         // second probe (0 when there is only one that serves)
    i32 join_none, n_exact;                       // no value below the operand limit can be the target; probes checked from the tables
    i32 join_shift, pad5;                         // zero bits at the end of the context's factor (the larger of the two probes')
    i64 join_t0, join_t1;                         // hole values that satisfy the constraint at the two probes
    u64 join_tmod;                                // largest |target| over the probes: a remainder's divisor must exceed it
    float join_rt0, join_rt1, join_rl0, join_rl1; // 1 / |target| (0 for 0), 1 / (|target| + 1)
    float join_h0, join_h1;                       // a huge number where the target is 0, else 0
    JoinSet* join_sets;                           // device, one per nonterminal
    i32* tab_pair;                                // device
    // Operand classes (csrc/xp_classes.cuh): the subtrees of cls_size nodes, the largest size with any in the tables, by their
    // values at the first n_exact probes.  Class c of nonterminal nt: the pair of values that its members share
    // (cls_pair), and their ranks cls_mem[cls_start[c] .. cls_start[c + 1]).  Subtrees undefined at one of those probes are in
    // none.  A nonterminal's share of the arrays starts at tab_off[nt][cls_size] - tab_off[0][cls_size] (of cls_start, nt further on).
    i32 cls_top, cls_want;                        // host: that size, and for which contexts classes are made (kClassAffine, kClassCompare)
    i32 cls_size, pad6;                           // 0: there are none
    u32 cls_n[kMaxNt];
    u64 cls_count[kMaxNt];                        // members << 32 | classes while they are numbered, zero before
    int2* cls_pair;                               // device
    u32* cls_start;                               // device
    u32* cls_mem;                                 // device
    // Points that ended a survivor's whole-domain check (a candidate that passed every probe and then
    // failed somewhere): a small open-addressed table of point ids (-1: free) with the number of
    // survivors each has ended.  Written by verify_kernel, read and cleared by xp_sketch_refine, which
    // promotes the most frequent ones to probes.  (Counters only: nothing in a search reads them.)
    i64* kill_pid;                                // device, kKillSlots entries
    u32* kill_cnt;                                // device, kKillSlots entries
};
constexpr int kKillSlots = 64;
enum { kClassAffine = 1, kClassCompare = 2 };

struct SketchDev {
    const GrammarDev* g;                          // device
    i32 n_vars, n_holes, domain_kind, n_samples;
    i32 pad, project;                             // project: box domain with staged points (see HoleDev::fixed_vars)
    i64 n_points;
    const i32* coords;                            // device: the points of a table domain, or the staged
                                                  // points of a box (null: derive them from the point id)
    i64 lo[kMaxVars], ext[kMaxVars];              // box: range start and extent per variable
    i64 vmin[kMaxVars], vmax[kMaxVars];           // smallest and largest coordinate of each variable over the domain
                                                  // (box: from the ranges; table: reduced over the rows at load)
    HoleDev* holes;                               // device
    i64 sample_id[kProbeSamples];                 // point ids the probes are chosen from (host-chosen)
};

// One hole of one sketch, for the kernels that run at load over a whole batch of sketches.
struct LoadJob { SketchDev* s; i32 hole, pad; };

// A piece of a load's staged copy (`src` bytes from its start) and where it belongs.
struct LoadCopy { char* dst; u64 src, bytes; };

// What the load's kernels settled for a hole, as the host reads it back.
struct LoadOut { i32 filter_ok, tab_probes, aff_ok, join_on, second, n_probe, tab_max, target_zero, sample_pass, sample_n; u32 spec_bad; i32 cls_size; u32 cls_n[kMaxNt]; };

// One hole whose operands are put into classes (csrc/xp_classes.cuh).
struct ClassJob {
    SketchDev* s;
    i32 hole;
    u32 first_block;                 // blocks of the jobs before it
    u64* table;                      // mask + 1 words, zero at launch: members << 32 | first subtree + 1, then members << 32 | first place
    uint2* at;                       // per subtree: slot and number among the members (kClassNone: in no class)
    LoadOut* out;                    // null: a refinement, the host reads the hole's record
    u32 mask, pad;
};

// Per (sketch, hole) accumulators, zeroed (min_rank to all-ones) by the host before the launch.
struct AccDev {
    u64 match_count[kMaxSize + 1];
    u64 min_rank[kMaxSize + 1];
    u64 evals;                       // exact candidate-point evaluations that ran: stage 2 (probes) and stage 3 (domain points)
    u64 filter_survivors, probe_survivors, pad;
    u64 ops_skipped;                 // cost-model operations that the filter did not have to carry out (remainders
                                     // of a tile none of whose divisors exceeds the target's magnitude)
    u64 filter_tests;                // filter-stage tests that ran.  Tiles: (register operand defined at probe 0) x (broadcast
                                     // operand defined there) x (operators whose loop was entered); leaf join: operands
                                     // defined at the probes x (entries tested one by one + one for a set of constants) x operators
    u64 tile_cands;                  // candidates of the tiles and joins visited, tested or not
    u64 join_tests;                  // ... filter_tests that the leaf join ran
};
constexpr i32 kPairNone = (i32)0x80000000u;

// A piece of the leaf join's work: operands e_begin .. e_begin + e_count of (nt, esize), each against the leaves of
// n_groups nonterminals.  kJoinDirect: candidates of (nt, esize) themselves, e_begin .. , checked on the probes one by one.
enum { kJoinLeaf = 0, kJoinDirect = 1 };
enum { kExactFew = 1, kExactMany = 2 };      // a warp per operand; a lane per operand
constexpr int kJoinGroups = 8;        // most groups of a segment
struct JoinGroup {
    i32 leaf_nt, pad;
    u32 fmask, smask;                // operator slots of  E op leaf  and  leaf op E
    u64 base[2][kOpSlots];           // rank of (E 0, leaf 0) per operator: forward, swapped
};
struct JoinSeg {
    u64 first_ticket;
    u64 rank_begin, rank_end;        // window of ranks searched at this size
    i32 sketch, hole, size;
    int16_t kind, parts;             // parts > 0: a ticket is 32 operands against one of so many parts of the leaves (join_few, range_ticket)
    i32 acc, nt, esize, n_groups;
    i32 first_group;
    i32 exact;                       // kExactFew, kExactMany: there is no condition (shifts, a leaf of 2^31 or more), every candidate is evaluated on its own
    u32 chunk;                       // operands per ticket (until the tickets are numbered: leaves of its groups)
    int16_t heavy;                   // an operand costs many times the usual (exact form, contexts that compare): these go first
    int16_t classes;                 // operands are counted by class: e_count combinations of classes (class_operands), from the first on;
                                     // e_begin: operands of the rank window that they stand for
    u64 e_begin, e_count;
};
static_assert(sizeof(JoinSeg) == 88, "sketches of many holes just fit the fixed scratch of a call that may not allocate");

// One (left operands, right operands) block of the pair join (csrc/xp_pairs.cuh): every  L op R  of its operators.
//
// The division kernel's walks: a block of 32 dividends may have any number of divisors to meet.  A walk is cut into pieces of
// kPairWalk divisors; the first is walked at once, the others are listed for a second launch.  They go to a list of kPairShort
// entries while it has room, and otherwise, in longer pieces, at most `pieces` a walk, to a second list of
// 2 * blocks * pieces entries, which is the most that all walks together can list: neither list is written past its end
// and neither counter passes it, whatever the operands are.  (Short pieces as long as they fit: where most of a walk
// agrees at both probes, every 32 divisors are 32 exact checks, and with pieces of 512 one such search took 60 ms longer.)
constexpr u32 kPairWalk = 64;        // divisors that a warp of the division kernel meets in one go, at least
constexpr u32 kPairShort = 1u << 18; // entries of the list of short pieces (2 MB)
constexpr u32 kPairLong = 1u << 20;  // entries of the list of long ones that `pieces` aims at (8 MB)
XP_HD inline bool pair_fits(u32 taken, u32 more) { return taken <= kPairShort && more <= kPairShort - taken; }
XP_HD inline u32 pair_blocks(u32 nl) { return (nl + 31u) / 32u; }
XP_HD inline u32 pair_pieces(u32 nl, u32 nr) {
    const u32 share = nl ? kPairLong / (2u * pair_blocks(nl)) : 0u, most = share > 8u ? share : 8u, all = nr ? (nr - 1u) / kPairWalk : 0u;
    return all < most ? all : most;
}
XP_HD inline u64 pair_list_entries(u32 nl, u32 nr) { return kPairShort + 2ull * pair_blocks(nl) * pair_pieces(nl, nr); }      // both lists
XP_HD inline u32 pair_piece(u32 span, u32 pieces) {      // divisors per long piece of a walk over `span` of them, a multiple of 32
    const u32 even = ((span + pieces) / (pieces + 1u) + 31u) & ~31u;
    return even > kPairWalk ? even : kPairWalk;
}
struct PairSeg {
    u64 rank_begin, rank_end;        // window of ranks searched at this size
    i32 sketch, hole, size, acc;
    i32 lnt, la, rnt, ra;            // nonterminal and size of either operand
    u32 l_begin, nl, nr;             // first of the left operands (a rank window may leave some out), and how many there are
    i32 lcls, rcls;                  // the left / right operands are classes (nl, nr of them; l_begin = 0)
    u64 right_count, pairs;          // right operands by rank; pairs of operands that the block stands for
    u32 ops;                         // operator slots (+ - * / %)
    i32 index_right;                 // the chains index the right operands (else the left ones)
    u64 base[5];                     // rank of (l_begin, 0) per operator
    u32 head_mask, far_pieces;       // far_pieces: long pieces that a walk lists at most (pair_pieces)
    // device scratch of the call
    u32* head;                       // head_mask + 1, all ones at launch
    u32* next;
    u32* counters;                   // [2] wide operands left, right, [2] entries of the two lists; zero at launch
    u64* ticket;                     // [2] of the division kernel's two launches, zero at launch
    uint2* far;                      // (block of dividends | long piece << 30 | remainder << 31, first divisor): what the second launch takes; the list of
                                     // short pieces, then that of long ones
    u32 *wide_l, *wide_r;
    u32* hist[2];                    // 1024 each, zero at launch
    u32* start[2];                   // 1025 each
    u32* id[2];                      // operands by magnitude
    int2* val[2];
};

// A candidate over operand classes that stands for many, left to members_kernel (csrc/xp_members.cuh) in pieces.
struct MemberRec {
    u64 e;                           // leaf join: number of the operand; pair join: left | right << 32
    u64 first;                       // pieces of the entries before it
    u32 pos, code;                   // leaf join: position of the leaf, group << 8 | slot << 1 | swapped; pair join: -, slot
    i32 seg;                         // of the leaf join, or ~ of the pair join
    u32 pieces;
};
constexpr u32 kMemberPiece = 64;     // members of a piece

// One contiguous piece of work.  kind 0 (linear): ranks [rank_begin, rank_end) of `size`,
// every candidate unranked on its own.  kind 1 (tile): the product of left subtrees
// [a_begin, a_begin+a_count) x right subtrees of one (production group, left size).
enum { kSegLinear = 0, kSegTile = 1 };
struct SegDev {
    u64 first_ticket;                // tickets before this segment
    u64 rank_begin, rank_end;        // window of ranks searched at this size
    i32 sketch, hole, size, kind;
    i32 acc;                         // accumulator slot
    // tile segments
    i32 reg_nt, reg_size;            // register-side operand: nonterminal, size
    i32 bc_nt, bc_size;              // broadcast-side operand
    i32 swap;                        // 1: the register side is the RIGHT operand
    i32 n_ops;                       // productions sharing (left nt, right nt) at this split
    i32 op[5];
    u64 op_base[5];                  // rank of (left 0, right 0) for each of them
    u64 reg_begin, reg_count;        // register-side subtree ranks covered by the window
    u64 bc_begin, bc_count;          // broadcast-side subtree ranks covered
    u64 right_count;                 // trees of the right operand (rank = base + l * right_count + r)
    u32 reg_tiles, bc_tiles;         // tickets = reg_tiles * bc_tiles
    i32 has_div;                     // some production of the group is / or %
    i32 generic;                     // some production of the group has no 32-bit filter loop (the shifts): the group's
                                     // candidates are evaluated exactly, in 64 bits, at the probe
    i32 bc_base, bc_keep;            // slots [bc_base, bc_base + bc_count) of the CTA's broadcast tile belong to this
                                     // segment; bc_keep (first of a family): all members' broadcast operands fit the
                                     // tile side by side and do not depend on the ticket, so a CTA fills them once
    i32 bc_tile;                     // broadcast operands per ticket (<= kBcTile; smaller where a candidate costs
                                     // more than a comparison, so that the search still spreads over all SMs)
    i32 family;                      // tile segments that share the register-side operands sit next to each
                                     // other: the first holds the tickets and the count of them (>= 1), the
                                     // others (family == 0) are visited by its tickets, one fill for all
};

// A candidate that passed every probe point and waits for the whole-domain check.  The check
// is cut into chunks of kVerifyChunk points (or pieces of one) that any CTA may take; state counts the pieces
// that passed, its top bit says that some point failed.
constexpr int kVerifyChunk = 4096;
constexpr u32 kSurvFailed = 0x80000000u;
struct SurvDev { u64 rank; i32 sketch, hole, size, acc; u32 state, vars; };   // vars: variables the candidate mentions

struct PlanDev {
    u64 ticket_base;                 // tickets [ticket_base, n_tickets) belong to this launch (a search that polls a
                                     // cancel word is cut into several launches); the counter starts at zero each time
    u64 n_tickets;
    i32 n_segs, n_sketches;
    const SegDev* segs;              // device
    const JoinSeg* jsegs;            // device
    const JoinGroup* jgroups;        // device
    const PairSeg* psegs;            // device
    i32 n_jsegs, n_psegs;
    u64 join_base, n_join;           // tickets of the leaf join that belong to this launch
    u64* join_ticket;                // device counter, zero at launch
    const SketchDev* const* sketches;  // device table of device pointers
    AccDev* acc;                     // device
    u64* ticket;                     // device counter, zero at launch
    SurvDev* surv;                   // device queue of survivors
    u32* surv_n;                     // device counter of pushes (may run past surv_cap), zero at launch
    u64* verify_ticket;              // device counter, zero at launch
    u32 surv_cap;
    u32 max_chunks;                  // chunks of the largest domain among the sketches
    i32 first_points;                // points of the first chunk: the largest domain's, at most kVerifyChunk
    u32* err;                        // device word for the checked build's index checks (0: none failed)
    // Survivors in hole order (null when the call has one hole): queued survivors per accumulator slot
    // (counted by eval_kernel), the slots' offsets (a scan of the counts) and, per slot side by side, the
    // queue indices of its survivors (a scatter).  The verification kernel walks surv_sorted.
    i32 n_acc;
    u32* surv_hist;                  // device, n_acc, zero at launch
    u32* surv_off;                   // device, n_acc + 1
    u32* surv_sorted;                // device, surv_cap
    // Survivors whose check spans more than one chunk of points (queue indices, in no particular order),
    // listed after the search so that the later chunks are walked for them alone.
    u32* surv_long;                  // device, surv_cap
    u32* surv_long_n;                // device counter, zero at launch
    // The list of members_kernel (null: no operand of the call is a class): entries << 44 | their pieces (entries may run past
    // member_cap), zero at launch; the counter of pieces taken; the pieces [member_base, member_end) belong to this launch.
    MemberRec* members;
    u64 *members_n, *member_ticket;
    u64 member_base, member_end;
    u32 member_cap, pad1;
    u32* verify_done;                // device counter of finished CTAs of the verification kernel, zero at launch
    AccDev* told;                    // page-locked: where the CTA that finishes last puts the accumulators (null: the host copies them)
};

}  // namespace xp
