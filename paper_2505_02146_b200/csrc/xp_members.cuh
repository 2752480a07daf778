// The members of candidates over operand classes that the joins have listed (xp_classes.cuh), shared by all warps of the device.
//
// A ticket is a piece of kMemberPiece members of one entry; the first ticket is the warp's number, the others come from a counter, and no warp waits for
// another.  Bound by the whole-domain checks once the survivor queue is full, before that by the latency of taking an entry apart (operand,
// members, remaining probes).  64 members: two steps of a warp, against one search among the entries and one walk of class_operand.  (6 and 10 million
// matches of the example in xp_classes.cuh: 0.27 and 0.58 s; three conv holes, which list none, 0.68 ms a call with it and without.)
#pragma once

namespace xp {

constexpr int kMemberThreads = 256;
constexpr int kMemberWarps = kMemberThreads / 32;
__global__ void __launch_bounds__(kMemberThreads, 2) members_kernel(const __grid_constant__ PlanDev plan) {
    chain_wait();
    __shared__ CandShared sh[kMemberWarps];
    CandShared& cand = sh[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const u64 listed = *plan.members_n >> 44;
    const i32 entries = (i32)(listed < plan.member_cap ? listed : plan.member_cap);
    if (entries == 0) return;
    u64 end = plan.members[entries - 1].first + plan.members[entries - 1].pieces;
    end = end < plan.member_end ? end : plan.member_end;
    JoinCount n{0, 0, 0, 0, 0};
    int acc = -1;
    i32 at = 0;                                           // the entry at hand
    const u64 warps = (u64)gridDim.x * kMemberWarps;
    u64 t = plan.member_base + (u64)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    while (t < end) {
        if (t - plan.members[at].first >= plan.members[at].pieces) {      // (unsigned: a piece before it as well)
            i32 k = entries;
            at = 0;
            while (k > 1) {                               // last entry with first <= t: one probe per lane and round
                const i32 step = (k + 31) / 32, pos = at + lane * step;
                const u32 mask = __ballot_sync(0xffffffffu, pos < at + k && plan.members[pos].first <= t);
                const i32 to = at + (31 - __clz((int)(mask | 1u))) * step;
                k = (at + k - to) < step ? (at + k - to) : step;
                at = to;
            }
        }
        const MemberRec rec = plan.members[at];
        if (!XP_CHECKED(t - rec.first < rec.pieces && (rec.seg >= 0 ? rec.seg < plan.n_jsegs : ~rec.seg < plan.n_psegs), kChkSegment)) break;
        const u64 k_first = (t - rec.first) * kMemberPiece;
        const bool join = rec.seg >= 0;
        const int sketch = join ? plan.jsegs[rec.seg].sketch : plan.psegs[~rec.seg].sketch, hole_index = join ? plan.jsegs[rec.seg].hole : plan.psegs[~rec.seg].hole;
        const int to_acc = join ? plan.jsegs[rec.seg].acc : plan.psegs[~rec.seg].acc;
        if (to_acc != acc) { join_flush(plan, acc, n); acc = to_acc; }
        const SketchDev* sk = plan.sketches[sketch];
        const HoleDev* hole = &sk->holes[hole_index];
        if (join) {
            const JoinSeg& seg = plan.jsegs[rec.seg];
            const ClassOperand c = class_operand(sk->g, hole, seg.nt, seg.esize, rec.e);
            const u64 m = c.members();
            for (u64 k0 = k_first; k0 < k_first + kMemberPiece && k0 < m; k0 += 32u) {
                const bool in = k0 + (u64)lane < m;
                join_member(cand, plan, seg, sk, hole, in, in ? c.rank(k0 + (u64)lane) : 0ull, rec.pos, rec.code, n);
            }
        } else {
            const PairSeg& seg = plan.psegs[~rec.seg];
            const PairSide L = pair_side(sk->g, hole, seg, false), R = pair_side(sk->g, hole, seg, true);
            const u32 l = (u32)rec.e, r = (u32)(rec.e >> 32), rn = R.members(r);
            const u64 m = (u64)L.members(l) * rn;
            for (u64 k0 = k_first; k0 < k_first + kMemberPiece && k0 < m; k0 += 32u) {
                const bool in = k0 + (u64)lane < m;
                u64 kl = 0, kr = 0;
                if (in) divmod_u64(k0 + (u64)lane, (u64)rn, kl, kr);
                pair_member(cand, plan, seg, sk, hole, L, R, in, in ? L.member(l, (u32)kl) : 0u, in ? R.member(r, (u32)kr) : 0u, (int)rec.code, n);
            }
        }
        u64 next = 0;
        if (lane == 0) next = atomicAdd((unsigned long long*)plan.member_ticket, 1ull);
        t = plan.member_base + warps + __shfl_sync(0xffffffffu, next, 0);
    }
    join_flush(plan, acc, n);
}

}  // namespace xp
