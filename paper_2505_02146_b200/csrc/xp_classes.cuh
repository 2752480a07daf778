// Operand classes: the subtrees of the largest tabulated size that no probe tells apart.
//
// Two operands with the same values at the first n_exact probes meet every condition of a search, up to the whole-domain check,
// alike.  Most subtrees of three nodes and more have many such twins (constants combined with constants, operands
// exchanged, quotients of small values: 92 480 subtrees of three nodes over 136 leaves are some 5 000 classes; 1.1 million
// of five nodes of a quasi-affine grammar with 513 constants some 300 000), and the operands one size further up are their combinations
// with a leaf.  So the joins run over classes, and a class is taken apart where a candidate has passed the probes.
//   class_insert_kernel  -- thread = subtree: hash of its values, and its class's slot (open addressing; a word is the subtree that came
//                           first, whose values are compared, and the members counted so far);
//   class_number_kernel  -- the member counted first numbers its class and takes the members' places, in the order of the subtrees
//                           (a scan per block, one atomic per block);
//   class_member_kernel  -- every member to its place.
// One launch of each for all holes of a load (a block finds its job by its number: hole by hole, 1000 guards of 29 leaves took 35 ms of a load, now 2.8).
// Bound by the latency of the table and of the values in L2: 45 us for either example, of a load.  The leaf join of the first search (2.1e11
// candidates) went from 1.93 to 0.14 ms, whole calls of six inputs from 2.95 to 1.05 ms on average; the second (3.2e11) from 6.3 to 2.0 ms,
// and from 14.4 to 6.8 on inputs with millions of suspects.  (Classes by the two join probes alone would be half as many in the second
// grammar, but then each member has to be held against the other probes by itself.)
#pragma once

namespace xp {

constexpr u32 kClassNone = 0xffffffffu;

__device__ __forceinline__ bool class_wanted(const HoleDev* hole) {
    if (hole->cls_top < 3 || hole->tab_max_size < hole->cls_top || hole->n_exact < 1) return false;
    // (a single probe tells next to nothing apart: a quasi-affine grammar, 4.1 million subtrees, size 9: 0.51 s operand by operand, 9.9 by class)
    if (hole->n_exact < 2 && hole->n_probe > hole->n_exact) return false;
    return hole->aff_ok ? (hole->cls_want & kClassAffine) && hole->join_on : (hole->cls_want & kClassCompare) != 0;
}

// The job of this block, and of its nonterminals the one whose subtrees [first, first + kClassThreads) the block has.
struct ClassPart { ClassJob job; u32 first; i32 nt; };
__device__ __forceinline__ ClassPart class_part(const ClassJob* jobs, int n_jobs, const ClassJob& only) {
    int lo = 0;
    for (int hi = n_jobs; hi - lo > 1;) { const int mid = (lo + hi) >> 1; if (jobs[mid].first_block <= blockIdx.x) lo = mid; else hi = mid; }
    ClassPart p;
    p.job = n_jobs == 1 ? only : jobs[lo];             // (one hole: it comes with the launch)
    const GrammarDev* g = p.job.s->g;
    const int top = p.job.s->holes[p.job.hole].cls_top;
    u32 block = blockIdx.x - p.job.first_block;
    for (p.nt = 0; p.nt + 1 < g->n_nt; ++p.nt) {
        const u32 here = ((u32)g->cnt[p.nt][top] + kClassThreads - 1) / kClassThreads;
        if (block < here) break;
        block -= here;
    }
    p.first = block * kClassThreads;
    return p;
}

__global__ void __launch_bounds__(kClassThreads) class_insert_kernel(const ClassJob* jobs, int n_jobs, const __grid_constant__ ClassJob only) {
    chain_wait();
    const ClassPart part = class_part(jobs, n_jobs, only);
    const ClassJob& job = part.job;
    const HoleDev* hole = &job.s->holes[job.hole];
    if (!class_wanted(hole)) return;
    const int nt = part.nt, top = hole->cls_top, np = hole->n_exact;
    const u64 first = hole->tab_off[0][top], base = hole->tab_off[nt][top], total = hole->tab_total;
    const u32 count = (u32)job.s->g->cnt[nt][top], i = part.first + threadIdx.x;
    if (part.first >= count) return;
    const i64* val = hole->tab_val + base;
    const unsigned char* def = hole->tab_ok + base;
    bool on = i < count;
    u64 h = 0x243F6A8885A308D3ull + (u64)nt;
    for (int j = 0; j < np && on; ++j) {
        on = def[(u64)j * total + i] != 0;
        h = (h ^ (u64)val[(u64)j * total + i]) * 0x9E3779B97F4A7C15ull;
        h ^= h >> 29;
    }
    u32 slot = kClassNone;
    if (on) {
        const u32 me = (u32)(base - first) + i + 1u;      // (of all nonterminals' subtrees, so that their classes stay apart)
        u32 s = (u32)(h >> 20) & job.mask;
        for (u32 step = 0; step <= job.mask; ++step, s = (s + 1u) & job.mask) {
            u64 w = job.table[s];
            if ((u32)w == 0u) w = atomicCAS((unsigned long long*)&job.table[s], 0ull, (u64)me);
            if ((u32)w == 0u) { slot = s; break; }
            const u32 other = (u32)w - 1u - (u32)(base - first);
            bool same = other < count;
            for (int j = 0; j < np && same; ++j) same = val[(u64)j * total + other] == val[(u64)j * total + i];
            if (same) { slot = s; break; }
        }
    }
    (void)XP_CHECKED(!on || slot != kClassNone, kChkSlot);      // (the table has twice as many words as subtrees)
    // one atomic per class and warp (large classes are runs of neighbours)
    const int lane = threadIdx.x & 31;
    const u32 same = __match_any_sync(0xffffffffu, slot);
    const int leader = __ffs((int)same) - 1;
    u64 old = 0;
    if (slot != kClassNone && lane == leader) old = atomicAdd((unsigned long long*)&job.table[slot], (u64)__popc(same) << 32);
    old = __shfl_sync(0xffffffffu, old, leader);
    if (i < count) job.at[(u32)(base - first) + i] = make_uint2(slot, (u32)(old >> 32) + (u32)__popc(same & ((1u << lane) - 1u)));
}

__global__ void __launch_bounds__(kClassThreads) class_number_kernel(const ClassJob* jobs, int n_jobs, const __grid_constant__ ClassJob only) {
    chain_wait();
    __shared__ u32 s_classes[kClassThreads / 32], s_members[kClassThreads / 32];
    __shared__ u64 s_base;
    const ClassPart part = class_part(jobs, n_jobs, only);
    const ClassJob& job = part.job;
    HoleDev* hole = &job.s->holes[job.hole];
    if (!class_wanted(hole)) return;
    const int nt = part.nt, top = hole->cls_top, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u64 base = hole->tab_off[nt][top];
    const u32 off = (u32)(base - hole->tab_off[0][top]);
    const u32 count = (u32)job.s->g->cnt[nt][top], i = part.first + threadIdx.x;
    if (part.first >= count) return;
    const uint2 at = i < count ? job.at[off + i] : make_uint2(kClassNone, 0u);
    const bool first = at.x != kClassNone && at.y == 0u;
    const u32 n = first ? (u32)(job.table[at.x] >> 32) : 0u, mine = __ballot_sync(0xffffffffu, first);
    u32 incl = n;
    for (int o = 1; o < 32; o <<= 1) { const u32 v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
    if (lane == 31) { s_members[warp] = incl; s_classes[warp] = (u32)__popc(mine); }
    __syncthreads();
    if (threadIdx.x == 0) {
        u32 c = 0, m = 0;
        for (int w = 0; w < kClassThreads / 32; ++w) { const u32 a = s_classes[w], b = s_members[w]; s_classes[w] = c; s_members[w] = m; c += a; m += b; }
        s_base = c ? atomicAdd((unsigned long long*)&hole->cls_count[nt], ((u64)m << 32) | c) : 0ull;
    }
    __syncthreads();
    if (!first) return;
    const u32 id = (u32)s_base + s_classes[warp] + (u32)__popc(mine & ((1u << lane) - 1u));
    const u32 place = (u32)(s_base >> 32) + s_members[warp] + incl - n;
    if (!XP_CHECKED(id < count && place + n <= count, kChkSlot)) return;
    hole->cls_pair[off + id] = reinterpret_cast<const int2*>(hole->tab_pair)[base + i];
    hole->cls_start[off + (u32)nt + id] = place;
    job.table[at.x] = ((u64)n << 32) | place;
}

__global__ void __launch_bounds__(kClassThreads) class_member_kernel(const ClassJob* jobs, int n_jobs, const __grid_constant__ ClassJob only) {
    chain_wait();
    const ClassPart part = class_part(jobs, n_jobs, only);
    const ClassJob& job = part.job;
    HoleDev* hole = &job.s->holes[job.hole];
    const bool wanted = class_wanted(hole);
    const int top = hole->cls_top;
    const GrammarDev* g = job.s->g;
    if (blockIdx.x == job.first_block && (int)threadIdx.x < g->n_nt) {
        const int nt = (int)threadIdx.x;
        const u32 n = wanted ? (u32)hole->cls_count[nt] : 0u;
        hole->cls_n[nt] = n;
        if (wanted) hole->cls_start[(u32)(hole->tab_off[nt][top] - hole->tab_off[0][top]) + (u32)nt + n] = (u32)(hole->cls_count[nt] >> 32);
        if (nt == 0) hole->cls_size = wanted ? top : 0;
        if (job.out) { job.out->cls_n[nt] = n; if (nt == 0) job.out->cls_size = wanted ? top : 0; }
    }
    if (!wanted) return;
    const u32 off = (u32)(hole->tab_off[part.nt][top] - hole->tab_off[0][top]);
    const u32 count = (u32)g->cnt[part.nt][top], i = part.first + threadIdx.x;
    if (i >= count) return;
    const uint2 at = job.at[off + i];
    if (at.x != kClassNone && XP_CHECKED(at.x <= job.mask && (u32)job.table[at.x] + at.y < count, kChkSlot)) hole->cls_mem[off + (u32)job.table[at.x] + at.y] = i;
}

// ---- what the joins read ----

// Operands of (nt, size) as one side of a run: their pairs of values and, where they are classes, the members' ranks.
struct OperandSide { const int2* pair; const u32* start; const u32* mem; u64 n; };
__device__ __forceinline__ OperandSide operand_side(const GrammarDev* g, const HoleDev* hole, int nt, int size, bool classes) {
    OperandSide s;
    if (classes && size == hole->cls_size) {
        const u64 off = hole->tab_off[nt][size] - hole->tab_off[0][size];
        s.pair = hole->cls_pair + off; s.start = hole->cls_start + off + nt; s.mem = hole->cls_mem + off; s.n = hole->cls_n[nt];
    } else {
        s.pair = reinterpret_cast<const int2*>(hole->tab_pair) + hole->tab_off[nt][size]; s.start = s.mem = nullptr; s.n = g->cnt[nt][size];
    }
    return s;
}

// An operand of a segment that counts by class, taken apart: member (l, r) is the subtree of rank
// base + left(l) * cr + right(r) of its nonterminal and size.
struct ClassOperand {
    u64 base, cr;
    const u32 *lmem, *rmem;          // ranks of the left and right operand's members (null: the one rank l0, r0)
    u32 ln, rn, l0, r0;
    __device__ __forceinline__ u64 members() const { return (u64)ln * rn; }
    __device__ __forceinline__ u64 rank(u64 k) const {
        u64 a = 0, b = k;
        if (ln > 1u) divmod_u64(k, (u64)rn, a, b);
        return base + (u64)(lmem ? lmem[a] : l0) * cr + (rmem ? rmem[b] : r0);
    }
};

// Operand number e of (nt, size): the combinations of one production and pair of sizes after the other.  Both operands of a
// run come from the tables, those of cls_size nodes by class; a run with an operand above the tables is counted in full.
__device__ __noinline__ ClassOperand class_operand(const GrammarDev* g, const HoleDev* hole, int nt, int size, u64 e) {
    ClassOperand c;
    c.base = 0; c.cr = 1; c.lmem = c.rmem = nullptr; c.ln = c.rn = 1; c.l0 = c.r0 = 0;
    auto members = [](const OperandSide& s, u64 i, const u32*& mem, u32& n, u32& only) {
        if (s.start) { const u32 at = s.start[i]; mem = s.mem + at; n = s.start[i + 1] - at; }
        else only = (u32)i;
    };
    const int tmax = hole->tab_max_size;
    if (size <= tmax) { members(operand_side(g, hole, nt, size, true), e, c.rmem, c.rn, c.r0); return c; }
    u64 rem = e;
    for (int p = g->bin_begin[nt]; p < g->bin_begin[nt + 1]; ++p) {
        const int lnt = g->bins[p].lnt, rnt = g->bins[p].rnt;
        u64 base = g->bins[p].off[size];
        for (int a = 1; a <= size - 2; ++a) {
            const u64 cl = g->cnt[lnt][a], cr = g->cnt[rnt][size - 1 - a];
            if (a > tmax || size - 1 - a > tmax) {
                if (rem < cl * cr) { c.base = base + rem; return c; }
                rem -= cl * cr;
            } else if (cl * cr != 0) {
                const OperandSide L = operand_side(g, hole, lnt, a, true), R = operand_side(g, hole, rnt, size - 1 - a, true);
                const u64 block = L.n * R.n;
                if (rem < block) {
                    u64 l, r;
                    divmod_u64(rem, R.n, l, r);
                    c.base = base; c.cr = cr;
                    members(L, l, c.lmem, c.ln, c.l0); members(R, r, c.rmem, c.rn, c.r0);
                    return c;
                }
                rem -= block;
            }
            base += cl * cr;
        }
    }
    (void)XP_CHECKED(false, kChkRank);
    return c;                                             // (not reached: e is below the count that the host made the same way)
}

// ---- candidates that stand for many ----

// A warp that has met candidates over classes takes them apart by itself while that is a few steps (member_own: fewer as the survivor queue fills;
// once it is full each member that is left costs a whole-domain check).  Larger ones go to a list, whose
// pieces all warps of the device share afterwards: subtrees that are 0 everywhere are one class of thousands, and where the target is one of
// a few values (a term that collapses, a domain of few points, a guard that always holds) most matches belong to a few such classes, hence to a few
// warps.  (16x12x8 points, 45 and 53 leaves, size 7, 6 and 10 million matches: operand by operand 1.19 and 1.45 s, by class
// and the warps that met them 3.2 and 6.6.)
constexpr u64 kMemberLeast = 16;             // members from which an entry pays; four times as many for each quarter of the list that is taken, so that the
                                             // largest classes find a place (68 leaves, 2.2e7 matches: 7.8 s without, 2.1 with it)
constexpr u64 kMemberMost = 1ull << 32;      // members of an entry; a larger one stays with its warp (entries, 2^17 and a warp's 32 more each, and
                                             // pieces, 2^43 and 2^31 a warp, then stay in their parts of the counter)
__device__ __forceinline__ u64 member_own(const PlanDev& plan) {
    const u32 taken = __shfl_sync(0xffffffffu, *(volatile const u32*)plan.surv_n, 0);
    return taken >= plan.surv_cap ? 32u : taken >= plan.surv_cap / 4u ? 256u : 1024u;
}
// The candidates of the lanes with `want` (count members each) to the list; returns whether this lane's is in it.  Called by all lanes.
__device__ __noinline__ bool list_members(const PlanDev& plan, bool want, u64 count, u64 e, u32 pos, u32 code, i32 seg) {
    const int lane = threadIdx.x & 31;
    if (!plan.members) return false;
    u64 now = 0;
    if (lane == 31) now = *(volatile const u64*)plan.members_n;
    now = __shfl_sync(0xffffffffu, now, 31);
    if ((now >> 44) >= plan.member_cap || ((now >> 43) & 1u)) return false;
    want = want && count >= kMemberLeast << (2u * ((u32)(now >> 44) * 4u / plan.member_cap)) && count <= kMemberMost;
    const u32 m = __ballot_sync(0xffffffffu, want);
    if (!m) return false;
    const u64 pieces = want ? (count + kMemberPiece - 1) / kMemberPiece : 0ull;
    u64 incl = pieces;
    for (int o = 1; o < 32; o <<= 1) { const u64 v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
    u64 old = 0;
    if (lane == 31) old = atomicAdd((unsigned long long*)plan.members_n, ((u64)__popc(m) << 44) | incl);
    old = __shfl_sync(0xffffffffu, old, 31);
    const u64 at = (old >> 44) + (u64)__popc(m & ((1u << lane) - 1u));
    const bool in = want && at < plan.member_cap;
    if (in) plan.members[at] = MemberRec{e, (old & ((1ull << 44) - 1)) + incl - pieces, pos, code, seg, (u32)pieces};
    return in;
}

}  // namespace xp
