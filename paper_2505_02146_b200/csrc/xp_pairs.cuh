// The pair join: candidates  L op R  whose operands both have three nodes or more.
//
// The tile kernel tests every pair of two operand sets (config 2's size 7 = 3 + 1 + 3: 92 480^2 pairs and five operators,
// 4 ms).  Here the pairs that can reach the target (t0, t1) at the join's two probes are found from an index of one set:
//   pair_build_kernel  -- hash chains over one set, by its values (v0, v1) at the two probes;
//   pair_hash_kernel   -- + - *: an operand x of the other set asks for its partner's values directly (t - x, x - t, t + x, t / x);
//   pair_sort_*        -- both sets by magnitude at the first probe (992 buckets of a float's exponent and five mantissa
//                         bits; order inside a bucket does not matter);
//   pair_div_kernel    -- / %: a warp takes 32 dividends next to each other in that order and walks only the divisors that
//                         can reach the target: |r| in (|l|/(|t|+1), |l|/|t|] for a quotient, (|t|, |l| - |t|] for a remainder
//                         (any above |t| when l is the target itself);
//   pair_wide_kernel   -- operands that are not narrow (31 bits, or fewer where the context's factor ends in zero bits), exactly.
// Candidates that agree at both probes wait in a warp's queue and are checked 32 at a time at the other probes.
// Operands of the classes' size are met by class (xp_classes.cuh): 5 000 x 5 000 instead of 92 480 x 92 480, no chains of equal values, and
// walks a twentieth as long (thread binding, whole calls of six inputs: 1.05 -> 0.52 ms; pair join of one of them 0.3 -> 0.07).
#pragma once

namespace xp {

constexpr int kPairThreads = 256;
constexpr int kPairWarps = kPairThreads / 32;

struct PairWarp {
    u32 c_l[64], c_r[64], c_op[64];
    u32 nc;
    CandShared cand;
};

// One side of a block: the pairs of values of its operands, and where operand i is in the tables (a class: its first member).
struct PairSide {
    const int2* pair;
    const u32 *start, *mem;                               // (null: operands by rank)
    u64 off;                                              // table entry of the first
    __device__ __forceinline__ u64 entry(u32 i) const { return off + (start ? mem[start[i]] : i); }
    __device__ __forceinline__ u32 members(u32 i) const { return start ? start[i + 1] - start[i] : 1u; }
    __device__ __forceinline__ u32 member(u32 i, u32 k) const { return start ? mem[start[i] + k] : i; }
};
__device__ __forceinline__ PairSide pair_side(const GrammarDev* g, const HoleDev* hole, const PairSeg& seg, bool right) {
    const int nt = right ? seg.rnt : seg.lnt, size = right ? seg.ra : seg.la;
    const OperandSide s = operand_side(g, hole, nt, size, (right ? seg.rcls : seg.lcls) != 0);
    const u32 skip = right ? 0u : seg.l_begin;
    return PairSide{s.pair + skip, s.start, s.mem, hole->tab_off[nt][size] + skip};
}

// A member per lane (in: this lane has one): left and right operand by rank.  Called by all lanes.
__device__ __noinline__ void pair_member(CandShared& cand, const PlanDev& plan, const PairSeg& seg, const SketchDev* sk, const HoleDev* hole, const PairSide& L, const PairSide& R,
                                         bool in, u32 lr, u32 rr, int slot, JoinCount& n) {
    const GrammarDev* g = sk->g;
    bool ok = false;
    u64 rank = 0;
    u32 vars = 0;
    if (in) {
        rank = seg.base[slot] + (u64)lr * seg.right_count + rr;
        ok = rank >= seg.rank_begin && rank < seg.rank_end && XP_CHECKED(rr < seg.right_count && rank < g->cnt[hole->start_nt][seg.size], kChkQueue);
        if (ok) vars = (u32)hole->tab_vars[L.off + lr] | (u32)hole->tab_vars[R.off + rr];
    }
    if (hole->n_exact < hole->n_probe) ok = join_full_check(g, hole, seg.size, ok, rank, n.evals);
    u32 m = __ballot_sync(0xffffffffu, ok);
    if (!m) return;
    n.passes += (u32)__popc(m);
    m = __ballot_sync(0xffffffffu, push_survivors(plan, sk, hole, seg.sketch, seg.hole, seg.size, seg.acc, ok, rank, vars));
    while (m) {
        const int at = __ffs((int)m) - 1;
        m &= m - 1;
        join_verify(cand, plan, sk, hole, seg.size, seg.acc, __shfl_sync(0xffffffffu, rank, at), __shfl_sync(0xffffffffu, vars, at), n.evals);
    }
}

// Pairs that satisfy the probes, one per lane (pass: this lane has one): to the survivor queue, the members of classes one by one, 32 at a
// time over all lanes' pairs, or left to members_kernel.  Called by all lanes.
__device__ __noinline__ void pair_members(PairWarp& w, const PlanDev& plan, const PairSeg& seg, const SketchDev* sk, const HoleDev* hole, bool pass, u32 l, u32 r,
                                          int slot, JoinCount& n) {
    if (!__any_sync(0xffffffffu, pass)) return;
    const int lane = threadIdx.x & 31;
    const PairSide L = pair_side(sk->g, hole, seg, false), R = pair_side(sk->g, hole, seg, true);
    const u32 rn = pass ? R.members(r) : 1u;
    u64 mine = pass ? (u64)L.members(l) * rn : 0ull, incl, total;
    for (int listed = 0;; ++listed) {
        incl = mine;
        for (int o = 1; o < 32; o <<= 1) { const u64 v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
        total = __shfl_sync(0xffffffffu, incl, 31);
        if (listed || total <= member_own(plan)) break;
        if (list_members(plan, mine > 0u, mine, (u64)l | (u64)r << 32, 0u, (u32)slot, ~(i32)(&seg - plan.psegs))) mine = 0;
    }
    for (u64 k0 = 0; k0 < total; k0 += 32u) {
        const u64 k = k0 + (u64)lane < total ? k0 + (u64)lane : total - 1u;
        int src = 0;                                      // the lane whose member this is: the first with incl > k
        for (int step = 16; step > 0; step >>= 1) { const u64 v = __shfl_sync(0xffffffffu, incl, src + step - 1); if (v <= k) src += step; }
        const u64 before = __shfl_sync(0xffffffffu, incl, src ? src - 1 : 0);
        const u32 l2 = __shfl_sync(0xffffffffu, l, src), r2 = __shfl_sync(0xffffffffu, r, src), rn2 = __shfl_sync(0xffffffffu, rn, src);
        const int slot2 = __shfl_sync(0xffffffffu, slot, src);
        const bool in = k0 + (u64)lane < total;
        u64 kl = 0, kr = 0;
        if (in) divmod_u64(src ? k - before : k, (u64)rn2, kl, kr);
        pair_member(w.cand, plan, seg, sk, hole, L, R, in, in ? L.member(l2, (u32)kl) : 0u, in ? R.member(r2, (u32)kr) : 0u, slot2, n);
    }
}

// The lane's candidate against the queue's remaining probes.  Called by all lanes.
__device__ __noinline__ void pair_check(PairWarp& w, const PlanDev& plan, const PairSeg& seg, const SketchDev* sk, const HoleDev* hole, int from, JoinCount& n) {
    const GrammarDev* g = sk->g;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const u32 nc = w.nc;
    const PairSide L = pair_side(g, hole, seg, false), R = pair_side(g, hole, seg, true);
    for (u32 at = 0; at < nc; at += 32) {
        bool pass = false;
        u32 l = 0, r = 0;
        int slot = 0;
        if (at + lane < nc) {
            l = w.c_l[at + lane]; r = w.c_r[at + lane];
            slot = (int)w.c_op[at + lane];
            if (XP_CHECKED(l < seg.nl && r < seg.nr, kChkQueue)) {
                const u64 le = L.entry(l), re = R.entry(r);
                pass = true;
                for (int j = from; j < hole->n_exact && pass; ++j) {
                    ++n.evals;
                    const u64 b = (u64)j * hole->tab_total;
                    i64 v;
                    pass = hole->tab_ok[b + le] && hole->tab_ok[b + re] &&
                           op_value(op_of_slot(slot), hole->tab_val[b + le], hole->tab_val[b + re], v) && probe_accepts(hole, j, v);
                }
            }
        }
        pair_members(w, plan, seg, sk, hole, pass, l, r, slot, n);
    }
    __syncwarp();
    if (lane == 0) w.nc = 0;
    __syncwarp();
}

__device__ __forceinline__ void pair_push(PairWarp& w, const PlanDev& plan, const PairSeg& seg, const SketchDev* sk, const HoleDev* hole, bool have, u32 l, u32 r,
                                          int slot, int from, JoinCount& n) {
    const u32 b = __ballot_sync(0xffffffffu, have);
    if (!b) return;
    const int lane = threadIdx.x & 31;
    const u32 nc = w.nc;
    n.suspects += (u32)__popc(b);
    if (have) {
        const u32 at = nc + (u32)__popc(b & ((1u << lane) - 1u));
        w.c_l[at] = l; w.c_r[at] = r; w.c_op[at] = (u32)slot;
    }
    __syncwarp();
    if (lane == 0) w.nc = nc + (u32)__popc(b);
    __syncwarp();
    if (nc + (u32)__popc(b) >= 32u) pair_check(w, plan, seg, sk, hole, from, n);
}

// Operand i of a side: its values at the two probes; 0 undefined, 1 narrow, 2 wide.
__device__ __forceinline__ int pair_entry(const PairSide& side, u32 i, u32 lim, int2& v) {
    v = side.pair[i];
    if (v.x == kPairNone) return v.y ? 2 : 0;
    return abs_u32(v.x) < lim && abs_u32(v.y) < lim ? 1 : 2;
}

__device__ __forceinline__ u32 pair_slot(int2 v, u32 mask) {
    u32 h = (u32)v.x * 0x9E3779B1u ^ ((u32)v.y + 0x7F4A7C15u) * 0x85EBCA77u;
    h ^= h >> 15; h *= 0xC2B2AE3Du; h ^= h >> 13;
    return h & mask;
}

// Narrow values stay below this: products of two must not reach 2^(62 - join_shift) (see join_targets).
__device__ __forceinline__ u32 pair_limit(const HoleDev* hole) {
    const int z = hole->join_shift;
    u32 l = 0x7fffffffu;
    while ((u64)l * l >= 1ull << (62 - z)) l >>= 1;       // (a power of two less one: at most a bit below the root)
    return l;
}

// Chains of the indexed set (narrow entries), and the lists of wide entries of both sets.
__global__ void __launch_bounds__(kPairThreads) pair_build_kernel(const __grid_constant__ PlanDev plan, int index) {
    chain_wait();
    const PairSeg& seg = plan.psegs[index];
    const SketchDev* sk = plan.sketches[seg.sketch];
    const HoleDev* hole = &sk->holes[seg.hole];
    const u32 lim = pair_limit(hole);
    const u32 i = blockIdx.x * blockDim.x + threadIdx.x;
    for (int side = 0; side < 2; ++side) {                // 0: left, 1: right
        const u32 n = side ? seg.nr : seg.nl;
        if (i >= n) continue;
        int2 v;
        const int st = pair_entry(pair_side(sk->g, hole, seg, side != 0), i, lim, v);
        if (st == 2) (side ? seg.wide_r : seg.wide_l)[atomicAdd(&seg.counters[side], 1u)] = i;
        if (side == seg.index_right && st == 1) seg.next[i] = atomicExch(&seg.head[pair_slot(v, seg.head_mask)], i);
    }
}

// + - *: one thread per operand x of the set that is not indexed.
__global__ void __launch_bounds__(kPairThreads, 3) pair_hash_kernel(const __grid_constant__ PlanDev plan, int index) {
    chain_wait();
    __shared__ PairWarp sh[kPairWarps];
    PairWarp& w = sh[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    if (lane == 0) w.nc = 0;
    __syncwarp();
    const PairSeg& seg = plan.psegs[index];
    const SketchDev* sk = plan.sketches[seg.sketch];
    const HoleDev* hole = &sk->holes[seg.hole];
    JoinCount n{0, 0, 0, 0, 0};
    const bool ir = seg.index_right != 0;
    const u32 nx = ir ? seg.nl : seg.nr;
    const PairSide X = pair_side(sk->g, hole, seg, !ir);
    const int2* Y = pair_side(sk->g, hole, seg, ir).pair;
    const u32 lim = pair_limit(hole);
    const i64 t0 = hole->join_t0, t1 = hole->join_t1;
    const int from = hole->join_p1 ? 2 : 1;
    const u32 ops = hole->join_none ? 0u : seg.ops & ((1u << kSlotAdd) | (1u << kSlotSub) | (1u << kSlotMul));
    for (u32 x0 = (blockIdx.x * kPairWarps + (threadIdx.x >> 5)) * 32u; x0 < nx; x0 += gridDim.x * kPairThreads) {
        const u32 x = x0 + lane;
        int2 v = make_int2(0, 0);
        const bool live = x < nx && pair_entry(X, x, lim, v) == 1;
        for (u32 m = ops; m; m &= m - 1) {
            const int slot = __ffs((int)m) - 1;
            i64 w0 = 0, w1 = 0;
            bool ok = live;
            if (slot == kSlotAdd) { w0 = t0 - v.x; w1 = t1 - v.y; }
            else if (slot == kSlotSub) {                  // L - R = t
                if (ir) { w0 = (i64)v.x - t0; w1 = (i64)v.y - t1; } else { w0 = t0 + v.x; w1 = t1 + v.y; }
            } else {                                      // (the plan leaves products to the tiles where a target is zero)
                ok = ok && v.x != 0 && v.y != 0 && t0 % (v.x ? v.x : 1) == 0 && t1 % (v.y ? v.y : 1) == 0;
                if (ok) { w0 = t0 / v.x; w1 = t1 / v.y; }
            }
            ok = ok && w0 > -(i64)lim && w0 < (i64)lim && w1 > -(i64)lim && w1 < (i64)lim;
            n.tests += (u64)__popc(__ballot_sync(0xffffffffu, live));
            const int2 want = make_int2((i32)w0, (i32)w1);
            u32 y = ok ? seg.head[pair_slot(want, seg.head_mask)] : 0xffffffffu;
            while (__any_sync(0xffffffffu, y != 0xffffffffu)) {
                bool hit = false;
                u32 at = 0;
                if (y != 0xffffffffu) {
                    const int2 q = Y[y];
                    hit = q.x == want.x && q.y == want.y;
                    at = y;
                    y = seg.next[y];
                }
                pair_push(w, plan, seg, sk, hole, hit, ir ? x : at, ir ? at : x, slot, from, n);
            }
        }
    }
    if (w.nc) pair_check(w, plan, seg, sk, hole, from, n);
    if (blockIdx.x == 0 && threadIdx.x == 0) n.cands += seg.pairs * (u64)__popc(seg.ops);
    join_flush(plan, seg.acc, n);
}

// ---- / and % ----

// Bucket of a magnitude below 2^31: exponent and five bits below the leading one (0 for 0).
__device__ __forceinline__ u32 pair_bucket(u32 u) {
    if (u == 0u) return 0u;
    const int e = 31 - __clz((int)u);
    const u32 frac = e >= 5 ? (u >> (e - 5)) & 31u : (u << (5 - e)) & 31u;
    return 1u + (u32)e * 32u + frac;
}
constexpr int kPairBuckets = 1024;

__global__ void __launch_bounds__(kPairThreads) pair_sort_count_kernel(const __grid_constant__ PlanDev plan, int index) {
    chain_wait();
    __shared__ u32 hist[kPairBuckets];
    const PairSeg& seg = plan.psegs[index];
    const int side = blockIdx.y;
    const HoleDev* hole = &plan.sketches[seg.sketch]->holes[seg.hole];
    const u32 n = side ? seg.nr : seg.nl, lim = pair_limit(hole);
    const PairSide set = pair_side(plan.sketches[seg.sketch]->g, hole, seg, side != 0);
    for (int b = threadIdx.x; b < kPairBuckets; b += kPairThreads) hist[b] = 0;
    __syncthreads();
    for (u32 i = blockIdx.x * kPairThreads + threadIdx.x; i < n; i += gridDim.x * kPairThreads) {
        int2 v;
        if (pair_entry(set, i, lim, v) == 1) atomicAdd(&hist[pair_bucket(abs_u32(v.x))], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kPairBuckets; b += kPairThreads) if (hist[b]) atomicAdd(&seg.hist[side][b], hist[b]);
}

// One CTA per side: bucket starts (start[kPairBuckets] = entries), and the cursors of the scatter.
__global__ void __launch_bounds__(kPairBuckets) pair_sort_scan_kernel(const __grid_constant__ PlanDev plan, int index) {
    chain_wait();
    __shared__ u32 part[kPairBuckets];
    const PairSeg& seg = plan.psegs[index];
    const int side = blockIdx.x, t = threadIdx.x;
    const u32 mine = seg.hist[side][t];
    part[t] = mine;
    __syncthreads();
    for (int d = 1; d < kPairBuckets; d <<= 1) {
        const u32 v = t >= d ? part[t - d] : 0u;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    seg.start[side][t] = part[t] - mine;
    seg.hist[side][t] = part[t] - mine;
    if (t == kPairBuckets - 1) seg.start[side][kPairBuckets] = part[t];
}

__global__ void __launch_bounds__(kPairThreads) pair_sort_scatter_kernel(const __grid_constant__ PlanDev plan, int index) {
    chain_wait();
    const PairSeg& seg = plan.psegs[index];
    const int side = blockIdx.y, lane = threadIdx.x & 31;
    const HoleDev* hole = &plan.sketches[seg.sketch]->holes[seg.hole];
    const u32 n = side ? seg.nr : seg.nl, lim = pair_limit(hole);
    const PairSide set = pair_side(plan.sketches[seg.sketch]->g, hole, seg, side != 0);
    for (u32 i0 = (blockIdx.x * kPairThreads + threadIdx.x) & ~31u; i0 < n; i0 += gridDim.x * kPairThreads) {
        const u32 i = i0 + lane;
        int2 v = make_int2(0, 0);
        const bool on = i < n && pair_entry(set, i, lim, v) == 1;
        const u32 b = on ? pair_bucket(abs_u32(v.x)) : 0xffffffffu;
        const u32 same = __match_any_sync(0xffffffffu, b);          // one atomic per bucket and warp
        const int leader = __ffs((int)same) - 1;
        u32 at = 0;
        if (on && lane == leader) at = atomicAdd(&seg.hist[side][b], (u32)__popc(same));
        at = __shfl_sync(0xffffffffu, at, leader) + (u32)__popc(same & ((1u << lane) - 1u));
        if (!on) continue;
        seg.id[side][at] = i;
        seg.val[side][at] = v;
    }
}

// First sorted position whose bucket is at least that of magnitude u, and one past the last whose bucket is at most that.
__device__ __forceinline__ u32 pair_from(const PairSeg& seg, u64 u) { return seg.start[1][u >> 31 ? kPairBuckets : pair_bucket((u32)u)]; }
__device__ __forceinline__ u32 pair_to(const PairSeg& seg, u64 u) { return seg.start[1][u >> 31 ? kPairBuckets : pair_bucket((u32)u) + 1u]; }

// The sorted divisors [lo, hi) that the dividends with magnitudes amin .. amax (self: one of them is the target's) may meet.
__device__ __forceinline__ void pair_span(const PairSeg& seg, int which, u64 m0, u32 amin, u32 amax, bool self, u32 nr, u32& lo, u32& hi) {
    if (which == 0) {                                     // quotient
        lo = pair_from(seg, (u64)amin / (m0 + 1) + 1);
        hi = m0 ? pair_to(seg, (u64)amax / m0) : nr;
    } else {                                              // remainder (at most its dividend)
        lo = pair_from(seg, m0 + 1);
        hi = amax < m0 ? lo : self ? nr : pair_to(seg, (u64)amax - m0);
    }
}

// 32 dividends next to each other in magnitude order, and the divisors that they may meet.  Blocks differ by three
// orders of magnitude in how many those are (a dividend that is the target itself leaves the remainder of every larger
// divisor open), and one such walk by one warp was the kernel's whole time: a warp meets one piece of the walk and lists the
// others (see pair_pieces), which the second launch (phase 1) takes one by one (92 480 x 92 480 pairs: 780 -> 105 us; with
// walks of 512 divisors 730: where most of a walk agrees at both probes, every 32 divisors are 32 exact checks).
__global__ void __launch_bounds__(kPairThreads, 3) pair_div_kernel(const __grid_constant__ PlanDev plan, int index, int phase) {
    chain_wait();
    __shared__ PairWarp sh[kPairWarps];
    PairWarp& w = sh[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    if (lane == 0) w.nc = 0;
    __syncwarp();
    const PairSeg& seg = plan.psegs[index];
    const SketchDev* sk = plan.sketches[seg.sketch];
    const HoleDev* hole = &sk->holes[seg.hole];
    JoinCount n{0, 0, 0, 0, 0};
    const i64 t0 = hole->join_t0, t1 = hole->join_t1;
    const u64 m0 = (u64)(t0 < 0 ? -t0 : t0), m1 = (u64)(t1 < 0 ? -t1 : t1);
    const int from = hole->join_p1 ? 2 : 1;
    const bool small = ((m0 | m1) >> 31) == 0 && !hole->join_none;      // (otherwise no narrow quotient or remainder is the target)
    const u32 u0t = (u32)m0, u1t = (u32)m1;
    const u32 nl = seg.start[0][kPairBuckets], nr = seg.start[1][kPairBuckets];
    const u32 blocks = (nl + 31u) / 32u, n_short = phase ? seg.counters[2] : 0u, n_far = phase ? n_short + seg.counters[3] : 0u;
    const u64 tickets = !small ? 0ull : phase ? (u64)n_far : (u64)blocks;
    for (;;) {
        u64 t = 0;
        if (lane == 0) t = atomicAdd((unsigned long long*)&seg.ticket[phase], 1ull);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= tickets) break;
        uint2 far = make_uint2(blocks - 1u - (u32)t, 0u);     // (the largest dividends meet the most divisors: first)
        if (phase) far = seg.far[t < n_short ? t : kPairShort + (t - n_short)];
        const u32 li = (far.x & 0x3fffffffu) * 32u + lane;
        const bool live = li < nl;
        const int2 lv = live ? seg.val[0][li] : make_int2(0, 0);
        const u32 lid = live ? seg.id[0][li] : 0u;
        const u32 a0 = abs_u32(lv.x), a1 = abs_u32(lv.y);
        const u32 amin = __reduce_min_sync(0xffffffffu, live ? a0 : 0xffffffffu), amax = __reduce_max_sync(0xffffffffu, a0);
        const bool self = __any_sync(0xffffffffu, live && a0 == u0t);
        const u32 n_live = (u32)__popc(__ballot_sync(0xffffffffu, live));
        for (int which = phase ? (int)(far.x >> 31) : 0; which < (phase ? (int)(far.x >> 31) + 1 : 2); ++which) {
            if (!((seg.ops >> (which ? kSlotMod : kSlotDiv)) & 1u)) continue;
            u32 lo, hi;
            pair_span(seg, which, m0, amin, amax, self, nr, lo, hi);
            if (lo >= hi) continue;
            u32 piece = kPairWalk, p0 = lo;
            if (phase) {
                p0 = far.y;
                if ((far.x >> 30) & 1u) piece = pair_piece(hi - lo, seg.far_pieces);
            } else if (hi - lo > piece) {                 // the first piece here, the others listed
                u32 more = (hi - lo - 1u) / piece, at = 0, is_long = 0;
                if (lane == 0) {
                    at = *(volatile u32*)&seg.counters[2];
                    for (;;) {                            // (a failed exchange means that another warp has listed its walk)
                        is_long = pair_fits(at, more) ? 0u : 1u;
                        const u32 seen = is_long ? at : atomicCAS(&seg.counters[2], at, at + more);
                        if (seen == at) break;
                        at = seen;
                    }
                }
                is_long = __shfl_sync(0xffffffffu, is_long, 0);
                if (is_long) {
                    piece = pair_piece(hi - lo, seg.far_pieces);
                    more = (hi - lo - 1u) / piece;
                    if (lane == 0) at = kPairShort + atomicAdd(&seg.counters[3], more);
                }
                at = __shfl_sync(0xffffffffu, at, 0);
                if (XP_CHECKED((u64)at + more <= pair_list_entries(seg.nl, seg.nr), kChkQueue))
                    for (u32 k = lane; k < more; k += 32u) seg.far[at + k] = make_uint2(far.x | (is_long << 30) | ((u32)which << 31), lo + (k + 1u) * piece);
            }
            const u32 p1 = hi - p0 < piece ? hi : p0 + piece;
            n.tests += (u64)(p1 - p0) * (u64)n_live;
            const u32 x0 = a0 >= u0t ? a0 - u0t : 1u;
            const bool can = live && (which == 0 || (a0 >= u0t && a1 >= u1t));
            for (u32 r0 = p0; r0 < p1; r0 += 32u) {
                // lanes fetch 32 divisors (and prepare them); all lanes then meet each of them
                const u32 k = r0 + lane < p1 ? r0 + lane : p1 - 1u;
                const int2 rv = seg.val[1][k];
                const u32 b0 = abs_u32(rv.x), b1 = abs_u32(rv.y);
                u32 q0 = 0, q1 = 0, q2 = 0;
                if (which == 0) { q0 = u0t * b0; q1 = ((u64)u0t * b0) >> 31 ? 0u : 1u; }
                else if (b0 > u0t && b1 > u1t) {
                    const u32 kk = (u32)__ffs((int)b0) - 1u;
                    q0 = inv_odd(b0 >> kk); q1 = 0xffffffffu / b0; q2 = kk;
                }
                const int m = p1 - r0 < 32u ? (int)(p1 - r0) : 32;
                u32 hits = 0;                             // bit s: this lane's dividend meets divisor s at the first probe
                if (which == 0) {
                    for (int s = 0; s < m; ++s) {
                        const u32 bb = __shfl_sync(0xffffffffu, b0, s), lw = __shfl_sync(0xffffffffu, q0, s), fit = __shfl_sync(0xffffffffu, q1, s);
                        hits |= (u32)(a0 - lw < bb && fit != 0u) << s;
                    }
                } else {
                    for (int s = 0; s < m; ++s) {
                        const u32 iv = __shfl_sync(0xffffffffu, q0, s), cm = __shfl_sync(0xffffffffu, q1, s), kk = __shfl_sync(0xffffffffu, q2, s);
                        hits |= (u32)(rotr32(x0 * iv, kk) <= cm && cm != 0u) << s;
                    }
                }
                if (!can) hits = 0;
                while (__any_sync(0xffffffffu, hits != 0u)) {
                    const int s = hits ? __ffs((int)hits) - 1 : 0;
                    const i32 d0 = __shfl_sync(0xffffffffu, rv.x, s), d1 = __shfl_sync(0xffffffffu, rv.y, s);
                    bool on = hits != 0u && d0 != 0 && d1 != 0;
                    hits &= hits - 1;
                    if (on) {                             // exactly, at both probes
                        i64 v0, v1;
                        on = narrow_op(which ? kSlotMod : kSlotDiv, lv.x, d0, v0) && v0 == t0 && narrow_op(which ? kSlotMod : kSlotDiv, lv.y, d1, v1) && v1 == t1;
                    }
                    pair_push(w, plan, seg, sk, hole, on, lid, on ? seg.id[1][r0 + (u32)s] : 0u, which ? kSlotMod : kSlotDiv, from, n);
                }
            }
        }
    }
    if (w.nc) pair_check(w, plan, seg, sk, hole, from, n);
    join_flush(plan, seg.acc, n);
}

// Wide operands: each against the whole other set, lanes over it, from the first probe on, exactly.
__global__ void __launch_bounds__(kPairThreads) pair_wide_kernel(const __grid_constant__ PlanDev plan, int index) {
    chain_wait();
    __shared__ PairWarp sh[kPairWarps];
    PairWarp& w = sh[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    if (lane == 0) w.nc = 0;
    __syncwarp();
    const PairSeg& seg = plan.psegs[index];
    const u32 wl = seg.counters[0], wr = seg.counters[1];
    if (wl + wr == 0u) return;
    const SketchDev* sk = plan.sketches[seg.sketch];
    const HoleDev* hole = &sk->holes[seg.hole];
    const u32 lim = pair_limit(hole);
    const PairSide L = pair_side(sk->g, hole, seg, false), R = pair_side(sk->g, hole, seg, true);
    JoinCount n{0, 0, 0, 0, 0};
    const u64 nl = wl, total = nl + wr;
    for (u64 i = blockIdx.x * kPairWarps + (threadIdx.x >> 5); i < total; i += (u64)gridDim.x * kPairWarps) {
        const bool left = i < nl;
        const u32 x = left ? seg.wide_l[i] : seg.wide_r[i - nl];
        const u64 xe = left ? L.entry(x) : R.entry(x);
        if (!hole->tab_ok[xe]) continue;
        const i64 xv = hole->tab_val[xe];
        const u32 m = left ? seg.nr : seg.nl;
        for (u32 y0 = 0; y0 < m; y0 += 32u) {
            const u32 y = y0 + lane;
            const u64 ye = y >= m ? 0ull : left ? R.entry(y) : L.entry(y);
            bool on = y < m && hole->tab_ok[ye] != 0;
            if (on && !left) { int2 v; on = pair_entry(L, y, lim, v) == 1; }      // (two wide operands: the left one's turn)
            const i64 yv = on ? hole->tab_val[ye] : 0;
            for (u32 o = seg.ops; o; o &= o - 1) {
                const int slot = __ffs((int)o) - 1;
                i64 v;
                n.tests += (u64)__popc(__ballot_sync(0xffffffffu, on));
                const bool hit = on && apply_op(op_of_slot(slot), left ? xv : yv, left ? yv : xv, v) && probe_accepts(hole, 0, v);
                pair_push(w, plan, seg, sk, hole, hit, left ? x : y, left ? y : x, slot, 1, n);
            }
        }
    }
    if (w.nc) pair_check(w, plan, seg, sk, hole, 1, n);
    join_flush(plan, seg.acc, n);
}

}  // namespace xp
