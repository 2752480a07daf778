// The behaviour mode of include/xp.h (xp_behaviours): bottom-up enumeration with
// observational-equivalence pruning on signature points.
//
// Representatives of every (nonterminal, size) live side by side in device memory: their
// signatures (n_sig int64 values each) and a 16-byte record (operator or leaf, the two operand
// representatives).  One pass per (size, nonterminal), in chunks of kBehChunk candidates:
//   beh_insert_kernel  -- thread = candidate of the pruned space: finds its (production, left size) block, computes its
//                         signature in registers from the operands' (which stay in cache: a few thousand rows serve
//                         millions of candidates) and puts it into the nonterminal's hash table (open addressing, one
//                         64-bit word per class: 24 bits of the signature's hash, a kind bit, an id).  A word with the same
//                         24 bits is confirmed by comparing the signatures themselves (another candidate's is computed
//                         again).  A class that a representative already owns drops the candidate;
//                         among the chunk's candidates the smallest index takes the word (an atomic minimum:
//                         no thread waits for another);
//   beh_flag_kernel    -- a candidate is new iff its class's word carries its own index; counts per block, and their exclusive
//                         scan by the block that finishes last;
//   beh_append_kernel  -- the new ones, in candidate order, become representatives: signature and
//                         record are appended, and the class's word now names the representative.
// A table starts small and grows with the passes (beh_rehash_kernel puts the representatives into the larger one), so that a
// call clears what it uses and not what its bound would allow.
// Then the representatives of the hole's nonterminal are held against the constraint at the
// signature points (beh_match_kernel) and the few that satisfy it are checked on the whole domain,
// in order (beh_verify_kernel: thread = point, the representative's tree walked with a small stack).
// Candidates' signatures used to be written to memory, read back twice and compared from there: 290 us of a million
// candidates with 12 points.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cstddef>
#include <cstring>
#include <functional>
#include <string>
#include <vector>

#include "xp_device.cuh"
#include "xp_launch.h"

namespace xp {

constexpr int kBehBlocks = 64;                            // (production, left size) blocks of one pass
constexpr u64 kBehChunk = 1ull << 22;                     // candidates per chunk
constexpr int kBehThreads = 256;
constexpr u64 kEmpty = ~0ull;
constexpr u64 kKindCand = 1ull << 39;
constexpr u64 kIdMask = (1ull << 39) - 1;
constexpr int kMatchCap = 256;                            // representatives that satisfy the signature, kept for the whole-domain check
constexpr u32 kLeafBit = 0x80000000u;

struct RepDesc { u32 op_or_leaf, left, right, size; };    // leaf: kLeafBit | index into the grammar's leaves; else operator and operand ids

struct BehDev {
    const SketchDev* sk;
    const HoleDev* hole;
    i32 n_sig, n_nt;
    u32 spec_ok, pad0;
    i64 sig_id[XP_MAX_SIG];
    i64 sig_pt[XP_MAX_SIG][kMaxVars];
    i64 sig_spec[XP_MAX_SIG];
    i64* rep_sig;                                         // [max_reps][n_sig]
    RepDesc* rep_desc;
    u64* table;                                           // [n_nt][table_size]
    u64 table_size;                                       // a power of two: the most a nonterminal's table may have
    u64* buf_slot;                                        // per candidate of the chunk: slot of its class (kNoSlot: dropped)
    u32* block_count;                                     // per block of the chunk: new candidates, then their exclusive scan
    u64* told;                                            // page-locked: chunk_new and err as the host reads them (null: by copy)
    u32 blocks_done, pad1;                                // blocks of the flag kernel that have counted, zero between passes
    // results, read back from here on
    u64 chunk_new;                                        // new representatives of the chunk at hand
    u32 err, pad;                                         // err: a probe sequence ran its limit (table too full)
    u64 match_count;
    u32 match_n, pad2;
    u32 match_id[kMatchCap];
    u32 verify_fail, n_nodes;                             // whole-domain check of one representative, and its tree in preorder
    RepDesc node[kMaxSize];
};
constexpr u64 kNoSlot = ~0ull;
constexpr u64 kBehTable = 1ull << 17;                     // slots a table starts with (1 MB: cleared in 2 us)

// mirror: the operator commutes and both operands are of one nonterminal, so that exchanging them gives a candidate of
// the same behaviour -- 1: always an earlier one (the smaller operand on the left), 2: an earlier one where the left
// operand's number is the larger, 0: none such.
struct BehBlock { u64 first, cr, lbase, rbase; i32 op, mirror; };
struct BehPass {
    i32 nt, size, n_blocks, leaf_first;                   // size 1: candidates are the leaves leaf_first ...
    u64 n_cand, mask;                                     // mask: the table's size at this pass, less one
    BehBlock blocks[kBehBlocks];
};

__device__ __forceinline__ u64 sig_hash(const i64* s, int n) {
    u64 h = 0x243F6A8885A308D3ull;
    for (int j = 0; j < n; ++j) { h = (h ^ (u64)s[j]) * 0x9E3779B97F4A7C15ull; h ^= h >> 29; }
    return h;
}

__global__ void beh_points_kernel(BehDev* B) {
    chain_wait();
    const int t = threadIdx.x;
    const SketchDev* sk = B->sk;
    bool ok = false;
    if (t < B->n_sig) {
        i64 pt[kMaxVars];
        point_coords(sk, B->sig_id[t], pt);
        for (int d = 0; d < sk->n_vars; ++d) B->sig_pt[t][d] = pt[d];
        i64 v = 0;
        ok = true;
        // (a spec expression is evaluated here even when the load staged its values: the staged table does
        // not say where the expression is undefined)
        if (B->hole->spec_len > 0) ok = eval_code(B->hole->spec, B->hole->spec_len, pt, 0, v);
        else v = B->hole->spec_table[B->sig_id[t]];
        B->sig_spec[t] = v;
    }
    const u32 m = __ballot_sync(0xffffffffu, ok);
    if (t == 0) B->spec_ok = m;
}

// Candidate idx of the pass: its operator and its operands (size 1: its leaf).
struct BehOperands { i32 op, mirror; LeafDev leaf; u64 l, r; };
__device__ __forceinline__ BehOperands beh_operands(const BehDev* B, const BehPass& P, u64 idx) {
    BehOperands o;
    o.op = -1; o.mirror = 0; o.l = o.r = 0;
    o.leaf = LeafDev{-1, 0, 0};
    if (P.size == 1) { o.leaf = B->sk->g->leaves[P.leaf_first + (i32)idx]; return o; }
    int b = 0;
    while (b + 1 < P.n_blocks && P.blocks[b + 1].first <= idx) ++b;
    const BehBlock& k = P.blocks[b];
    u64 l, r;
    divmod_u64(idx - k.first, k.cr, l, r);
    o.op = k.op; o.mirror = k.mirror; o.l = k.lbase + l; o.r = k.rbase + r;
    return o;
}

// Operator OP on two signatures, point by point, given to f(j, value); returns whether all are defined.  The operator is
// chosen once per candidate (beh_signature): with the choice inside the unrolled loop the kernel was ten times the size and
// waited for its instructions.
template <int OP, int NS, typename F>
__device__ __forceinline__ bool beh_apply(const i64* __restrict__ ls, const i64* __restrict__ rs, int ns, F f) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < NS; ++j)
        if (j < ns) {
            i64 v = 0;
            ok = apply_op(OP, ls[j], rs[j], v) && ok;
            f(j, v);
        }
    return ok;
}
template <int NS, typename F>
__device__ __forceinline__ bool beh_signature(const BehDev* B, const BehOperands& o, int ns, F f) {
    const i64* ls = B->rep_sig + o.l * ns;
    const i64* rs = B->rep_sig + o.r * ns;
    switch (o.op) {
        case -1:
#pragma unroll
            for (int j = 0; j < NS; ++j) if (j < ns) f(j, o.leaf.var >= 0 ? B->sig_pt[j][o.leaf.var] : o.leaf.value);
            return true;
        case XP_OP_ADD: return beh_apply<XP_OP_ADD, NS>(ls, rs, ns, f);
        case XP_OP_SUB: return beh_apply<XP_OP_SUB, NS>(ls, rs, ns, f);
        case XP_OP_MUL: return beh_apply<XP_OP_MUL, NS>(ls, rs, ns, f);
        case XP_OP_DIV: return beh_apply<XP_OP_DIV, NS>(ls, rs, ns, f);
        case XP_OP_MOD: return beh_apply<XP_OP_MOD, NS>(ls, rs, ns, f);
        case XP_OP_MIN: return beh_apply<XP_OP_MIN, NS>(ls, rs, ns, f);
        case XP_OP_MAX: return beh_apply<XP_OP_MAX, NS>(ls, rs, ns, f);
        case XP_OP_SHL: return beh_apply<XP_OP_SHL, NS>(ls, rs, ns, f);
        default: return beh_apply<XP_OP_SHR, NS>(ls, rs, ns, f);
    }
}

// Is the signature behind a table word (a representative's, or another candidate's of the pass) equal to `mine`?
template <int NS>
__device__ __forceinline__ bool beh_same(const BehDev* B, const BehPass& P, u64 word, const i64 (&mine)[NS], int ns) {
    const u64 id = word & kIdMask;
    bool eq = true;
    if (!(word & kKindCand)) {
        const i64* s = B->rep_sig + id * ns;
#pragma unroll
        for (int j = 0; j < NS; ++j) if (j < ns) eq = eq && s[j] == mine[j];
        return eq;
    }
    (void)beh_signature<NS>(B, beh_operands(B, P, id), ns, [&](int j, i64 v) { eq = eq && v == mine[j]; });
    return eq;
}

// (n_sig <= NS: the signature stays in registers.)  Bound by the latency of the table and of the operands' signatures in L2: four
// CTAs per SM cost 50 bytes of spills and are faster than three (1.07 million candidates of 12 points: 196 -> 183 us).  A
// candidate whose mirror image comes earlier cannot be the first of its class and is not evaluated (183 -> 171 us), and a class is
// compared once per slot however often its word is lowered meanwhile (171 -> 137 us).
template <int NS>
__global__ void __launch_bounds__(kBehThreads, 4) beh_insert_kernel(BehDev* B, const __grid_constant__ BehPass P, u64 chunk_first, u32 chunk_n) {
    chain_wait();
    const u32 c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= chunk_n) return;
    const int ns = B->n_sig;
    const BehOperands o = beh_operands(B, P, chunk_first + c);
    if (o.mirror == 1 || (o.mirror == 2 && o.l > o.r)) { B->buf_slot[c] = kNoSlot; return; }
    i64 mine[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) mine[j] = 0;
    const bool defined = beh_signature<NS>(B, o, ns, [&](int j, i64 v) { mine[j] = v; });
    u64 h = 0x243F6A8885A308D3ull;                        // (sig_hash)
#pragma unroll
    for (int j = 0; j < NS; ++j) if (j < ns) { h = (h ^ (u64)mine[j]) * 0x9E3779B97F4A7C15ull; h ^= h >> 29; }
    u64 place = kNoSlot;
    if (defined) {
        const u64 me = ((h & 0xffffffull) << 40) | kKindCand | (chunk_first + c);
        u64* tab = B->table + (u64)P.nt * B->table_size;
        u64 slot = (h >> 24) & P.mask;
        bool done = false;
        for (u64 step = 0; step <= P.mask && !done; ++step, slot = (slot + 1) & P.mask) {
            u64 w = tab[slot];
            if (w == kEmpty) {
                const u64 old = atomicCAS((unsigned long long*)&tab[slot], kEmpty, me);
                if (old == kEmpty) { place = slot; done = true; break; }
                w = old;
            }
            if ((w >> 40) != (me >> 40) || !beh_same<NS>(B, P, w, mine, ns)) continue;
            // A slot's class never changes, so what the word has become meanwhile needs no second look: a representative's word
            // and an earlier candidate's are smaller than this one and stay.
            done = true;
            if ((w & kKindCand) && w > me && atomicMin((unsigned long long*)&tab[slot], me) > me) place = slot;
        }
        if (!done) atomicOr(&B->err, 1u);
    }
    B->buf_slot[c] = place;
}

// Which candidates of the chunk own their class, counted per block; the block that finishes last scans the counts and
// tells the host how many there are (a launch and a copy fewer per pass: with the append queued before the host looks,
// 410 -> 388 us at four passes).
__global__ void __launch_bounds__(kBehThreads) beh_flag_kernel(BehDev* B, int nt, u64 chunk_first, u32 chunk_n) {
    chain_wait();
    const u32 c = blockIdx.x * blockDim.x + threadIdx.x;
    bool is_new = false;
    if (c < chunk_n) {
        const u64 slot = B->buf_slot[c];
        if (slot != kNoSlot) {                            // it has held its class's word: does it still?
            is_new = (B->table[(u64)nt * B->table_size + slot] & ((1ull << 40) - 1)) == (kKindCand | (chunk_first + c));
            if (!is_new) B->buf_slot[c] = kNoSlot;
        }
    }
    const int n = __syncthreads_count(is_new);
    __shared__ u32 part[kBehThreads];
    __shared__ bool s_last;
    const int t = threadIdx.x;
    if (t == 0) {
        B->block_count[blockIdx.x] = (u32)n;
        __threadfence();
        s_last = atomicAdd(&B->blocks_done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int n_blocks = (int)gridDim.x, per = (n_blocks + kBehThreads - 1) / kBehThreads;
    const int lo = t * per < n_blocks ? t * per : n_blocks, hi = lo + per < n_blocks ? lo + per : n_blocks;
    u32 sum = 0;
    for (int i = lo; i < hi; ++i) sum += __ldcg(&B->block_count[i]);
    part[t] = sum;
    __syncthreads();
    for (int d = 1; d < kBehThreads; d <<= 1) {
        const u32 v = t >= d ? part[t - d] : 0u;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    u32 run = part[t] - sum;
    for (int i = lo; i < hi; ++i) { const u32 h = __ldcg(&B->block_count[i]); B->block_count[i] = run; run += h; }
    if (t == 0) {
        const u32 total = part[kBehThreads - 1];
        B->chunk_new = total;
        B->blocks_done = 0u;
        if (B->told) { B->told[0] = total; B->told[1] = B->err; }
    }
}

// A nonterminal's representatives, by size.
struct BehRanges { i32 n; i32 pad; u64 first[kMaxSize], count[kMaxSize], total; };
__device__ __forceinline__ u64 range_id(const BehRanges& R, u64 i) {
    int k = 0;
    while (k + 1 < R.n && i >= R.count[k]) { i -= R.count[k]; ++k; }
    return R.first[k] + i;
}

// Representatives of a nonterminal into its (cleared) table.
__global__ void __launch_bounds__(kBehThreads) beh_rehash_kernel(BehDev* B, int nt, u64 mask, const __grid_constant__ BehRanges R) {
    chain_wait();
    const u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= R.total) return;
    const u64 id = range_id(R, i);
    const u64 h = sig_hash(B->rep_sig + id * B->n_sig, B->n_sig);
    const u64 word = ((h & 0xffffffull) << 40) | id;
    u64* tab = B->table + (u64)nt * B->table_size;
    u64 slot = (h >> 24) & mask;
    for (u64 step = 0; step <= mask; ++step, slot = (slot + 1) & mask)       // (their signatures differ: the first free slot)
        if (atomicCAS((unsigned long long*)&tab[slot], kEmpty, word) == kEmpty) return;
    atomicOr(&B->err, 1u);
}

__global__ void __launch_bounds__(kBehThreads) beh_append_kernel(BehDev* B, const __grid_constant__ BehPass P, u64 chunk_first, u32 chunk_n, u64 rep_base, u64 max_reps) {
    chain_wait();
    if (B->err || rep_base + B->chunk_new > max_reps) return;      // (the host has not looked yet: it will give up)
    __shared__ u32 warp_sum[kBehThreads / 32];
    const u32 c = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool is_new = c < chunk_n && B->buf_slot[c] != kNoSlot;
    const u32 bal = __ballot_sync(0xffffffffu, is_new);
    if (lane == 0) warp_sum[warp] = (u32)__popc(bal);
    __syncthreads();
    if (!is_new) return;
    u32 pos = B->block_count[blockIdx.x] + (u32)__popc(bal & ((1u << lane) - 1u));
    for (int w = 0; w < warp; ++w) pos += warp_sum[w];
    const u64 gid = rep_base + pos;
    const int ns = B->n_sig;
    const u64 idx = chunk_first + c;
    const BehOperands o = beh_operands(B, P, idx);
    i64* dst = B->rep_sig + gid * ns;
    (void)beh_signature<XP_MAX_SIG>(B, o, ns, [&](int j, i64 v) { dst[j] = v; });
    RepDesc d;
    d.size = (u32)P.size;
    if (P.size == 1) { d.op_or_leaf = kLeafBit | (u32)(P.leaf_first + (i32)idx); d.left = d.right = 0; }
    else { d.op_or_leaf = (u32)o.op; d.left = (u32)o.l; d.right = (u32)o.r; }
    B->rep_desc[gid] = d;
    u64* tab = B->table + (u64)P.nt * B->table_size;
    const u64 slot = B->buf_slot[c];
    tab[slot] = (tab[slot] & ~((1ull << 40) - 1)) | gid;  // the class's word now names the representative
}

// All of them against the constraint at the signature points.
__global__ void __launch_bounds__(kBehThreads) beh_match_kernel(BehDev* B, const __grid_constant__ BehRanges R) {
    chain_wait();
    const u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= R.total) return;
    const u64 id = range_id(R, i);
    const int ns = B->n_sig;
    const u32 all = ns >= 32 ? 0xffffffffu : (1u << ns) - 1u;
    if ((B->spec_ok & all) != all) return;                // the spec is undefined at a signature point: nothing satisfies it
    const i64* s = B->rep_sig + id * ns;
    bool ok = true;
    for (int j = 0; j < ns && ok; ++j) ok = ctx_matches(B->hole, B->sig_pt[j], s[j], B->sig_spec[j]);
    if (!ok) return;
    atomicAdd((unsigned long long*)&B->match_count, 1ull);
    const u32 at = atomicAdd(&B->match_n, 1u);
    if (at < (u32)kMatchCap) B->match_id[at] = (u32)id;
}

// Value of representative `gid` at one point: its tree is walked with an explicit stack.
__device__ bool rep_value(const BehDev* B, u32 gid, const i64* pt, i64& out) {
    u32 todo[2 * kMaxSize + 2];                           // node ids; kLeafBit set: "apply this node's operator now"
    i64 val[kCandStack + 1];
    int nt = 0, nv = 0;
    todo[nt++] = gid;
    const LeafDev* leaves = B->sk->g->leaves;
    while (nt > 0) {
        const u32 x = todo[--nt];
        if (x & kLeafBit) {                               // operator of node x & ~kLeafBit: operands are on the value stack
            const RepDesc d = B->rep_desc[x & ~kLeafBit];
            const i64 b = val[--nv], a = val[nv - 1];
            i64 r;
            if (!apply_op((int)d.op_or_leaf, a, b, r)) return false;
            val[nv - 1] = r;
            continue;
        }
        const RepDesc d = B->rep_desc[x];
        if (d.op_or_leaf & kLeafBit) {
            const LeafDev lf = leaves[d.op_or_leaf & ~kLeafBit];
            if (!XP_CHECKED(nv <= kCandStack, kChkStack)) return false;
            val[nv++] = lf.var >= 0 ? pt[lf.var] : lf.value;
        } else {
            if (!XP_CHECKED(nt + 3 <= 2 * kMaxSize + 2, kChkStack)) return false;
            todo[nt++] = x | kLeafBit;
            todo[nt++] = d.right;
            todo[nt++] = d.left;
        }
    }
    out = val[0];
    return true;
}

// gid = kFirstMatch: the smallest of the representatives that beh_match_kernel has listed (none: nothing to do), so that the usual case, in which
// that one is the answer, needs no look by the host in between (a pass to size 7: 353 -> 326 us).
constexpr u32 kFirstMatch = 0xffffffffu;
__global__ void __launch_bounds__(kBehThreads) beh_verify_kernel(BehDev* B, u32 gid) {
    chain_wait();
    if (gid == kFirstMatch) {
        const u32 n = B->match_n;
        if (n == 0u || n > (u32)kMatchCap) return;
        __shared__ u32 s_least;
        if (threadIdx.x == 0) s_least = 0xffffffffu;
        __syncthreads();
        for (u32 i = threadIdx.x; i < n; i += blockDim.x) atomicMin(&s_least, B->match_id[i]);
        __syncthreads();
        gid = s_least;
    }
    const SketchDev* sk = B->sk;
    const HoleDev* hole = B->hole;
    if (blockIdx.x == 0 && threadIdx.x == 0) {            // its tree, for the text: nodes in preorder
        u32 todo[kMaxSize + 1];
        int n = 0, k = 0;
        todo[n++] = gid;
        while (n > 0 && k < kMaxSize) {
            const RepDesc d = B->rep_desc[todo[--n]];
            B->node[k++] = d;
            if (!(d.op_or_leaf & kLeafBit) && n + 2 <= kMaxSize + 1) { todo[n++] = d.right; todo[n++] = d.left; }
        }
        B->n_nodes = (u32)k;
    }
    for (i64 pid = (i64)blockIdx.x * blockDim.x + threadIdx.x; pid < sk->n_points; pid += (i64)gridDim.x * blockDim.x) {
        if (*(volatile u32*)&B->verify_fail) return;
        i64 pt[kMaxVars];
        point_coords(sk, pid, pt);
        i64 want = 0, h;
        bool ok = true;
        if (hole->spec_len > 0) ok = eval_code(hole->spec, hole->spec_len, pt, 0, want);
        else want = hole->spec_table[pid];
        ok = ok && rep_value(B, gid, pt, h) && ctx_matches(hole, pt, h, want);
        if (!ok) { atomicOr(&B->verify_fail, 1u); return; }
    }
}

}  // namespace xp

using namespace xp;

namespace {
struct Cuda { cudaError_t e = cudaSuccess; void operator()(cudaError_t x) { if (e == cudaSuccess) e = x; } bool ok() const { return e == cudaSuccess; } };
}

extern "C" xp_status xp_behaviours(const xp_sketch* sketch, const xp_behaviour_desc* d, const xp_repair_opts* opts,
                                   xp_behaviour_summary* out) {
    if (!sketch || !d || !out) return set_error(XP_ERR_INVALID_ARG, "xp_behaviours: null argument");
    memset(out, 0, sizeof(*out));
    const auto t0 = std::chrono::steady_clock::now();
    const SketchInternals si = sketch_internals(sketch);
    const HoleSpec hs = sketch_hole(sketch, d->hole);
    if (hs.start_nt < 0) return set_error(XP_ERR_INVALID_ARG, "xp_behaviours: hole out of range");
    if (d->n_sig < 1 || d->n_sig > XP_MAX_SIG || !d->sig_points) return set_error(XP_ERR_INVALID_ARG, "xp_behaviours: n_sig must be 1..16");
    for (int j = 0; j < d->n_sig; ++j)
        if (d->sig_points[j] < 0 || d->sig_points[j] >= si.n_points) return set_error(XP_ERR_INVALID_ARG, "xp_behaviours: a signature point lies outside the domain");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return set_error(XP_ERR_CUDA, "no CUDA device is usable");
    if (dev != si.device) return set_error(XP_ERR_INVALID_ARG, "xp_behaviours: the sketch was loaded on another device than the current one");
    const GrammarHost gh = grammar_host(si.g);
    const int ns = d->n_sig, K = hs.max_size, n_nt = gh.n_nt;
    const u64 max_reps = d->max_representatives ? d->max_representatives : (1ull << 22);
    if (max_reps >= (1ull << 31)) return set_error(XP_ERR_TOO_LARGE, "xp_behaviours: max_representatives must stay below 2^31");
    u64 tsize = 1024;
    while (tsize < 2 * max_reps + 2 * kBehChunk) tsize <<= 1;      // (at least kBehTable)
    // one device block
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    size_t off = al(sizeof(BehDev));
    const size_t o_sig = off;   off += al(sizeof(i64) * max_reps * ns);
    const size_t o_desc = off;  off += al(sizeof(RepDesc) * max_reps);
    const size_t o_tab = off;   off += al(sizeof(u64) * tsize * n_nt);
    const size_t o_bslot = off; off += al(sizeof(u64) * kBehChunk);
    const size_t o_bcnt = off;  off += al(sizeof(u32) * (kBehChunk / kBehThreads + 1));
    char* block = nullptr;
    size_t granted = 0;
    int bdev = 0;
    if (device_alloc((void**)&block, off, &bdev, &granted) != cudaSuccess) {
        (void)cudaGetLastError();
        return set_error(XP_ERR_NOMEM, ("xp_behaviours: device memory (" + std::to_string(off) + " bytes)").c_str());
    }
    StageMemory stage(2 * sizeof(BehDev));                // what goes out, and what comes back behind it
    StageEvents ev, counted;
    if (!stage.p) { device_release(block, granted, bdev); return set_error(XP_ERR_NOMEM, "out of host memory"); }
    BehDev& h = *(BehDev*)stage.p;
    BehDev& back = *(BehDev*)(stage.p + sizeof(BehDev));
    memset(&h, 0, sizeof(h));
    h.sk = si.d_s; h.hole = sketch_hole_dev(sketch, d->hole); h.n_sig = ns; h.n_nt = n_nt;
    for (int j = 0; j < ns; ++j) h.sig_id[j] = d->sig_points[j];
    h.rep_sig = (i64*)(block + o_sig); h.rep_desc = (RepDesc*)(block + o_desc);
    h.table = (u64*)(block + o_tab); h.table_size = tsize;
    h.buf_slot = (u64*)(block + o_bslot); h.block_count = (u32*)(block + o_bcnt);
    BehDev* dB = (BehDev*)block;
    cudaStream_t stream = opts ? (cudaStream_t)opts->stream : nullptr;
    constexpr size_t kBackAt = offsetof(BehDev, chunk_new);
    Cuda cu;
    h.told = stage.locked ? &back.chunk_new : nullptr;
    cu(ev.open());
    cu(counted.open());
    cu(cudaMemcpyAsync(dB, &h, sizeof(h), cudaMemcpyHostToDevice, stream));
    if (cu.ok()) cu(cudaEventRecord(ev.e0, stream));
    int launches = 0;
    if (cu.ok()) { chain(beh_points_kernel, 1, 32, 0, stream, dB); ++launches; cu(cudaGetLastError()); }
    std::vector<std::vector<u64>> count(n_nt, std::vector<u64>(K + 1, 0)), base(n_nt, std::vector<u64>(K + 1, 0));
    std::vector<u64> table(n_nt, 0), held(n_nt, 0);       // per nonterminal: size of its table so far, representatives in it
    auto ranges_of = [&](int nt) {
        BehRanges R;
        memset(&R, 0, sizeof(R));
        for (int s = 1; s <= K; ++s)
            if (count[nt][s] > 0) { R.first[R.n] = base[nt][s]; R.count[R.n++] = count[nt][s]; R.total += count[nt][s]; }
        return R;
    };
    u64 n_reps = 0, bytes = 0;
    xp_status st = XP_OK;
    std::string why;
    for (int s = 1; s <= K && cu.ok() && st == XP_OK; ++s)
        for (int nt = 0; nt < n_nt && cu.ok() && st == XP_OK; ++nt) {
            BehPass P;
            memset(&P, 0, sizeof(P));
            P.nt = nt; P.size = s;
            if (s == 1) { P.leaf_first = gh.leaf_begin[nt]; P.n_cand = (u64)(gh.leaf_begin[nt + 1] - gh.leaf_begin[nt]); }
            else
                for (int b = gh.bin_begin[nt]; b < gh.bin_begin[nt + 1] && st == XP_OK; ++b)
                    for (int a = 1; a <= s - 2; ++a) {
                        const u64 cl = count[gh.bins[b].lnt][a], cr = count[gh.bins[b].rnt][s - 1 - a];
                        if (cl == 0 || cr == 0) continue;
                        if (P.n_blocks == kBehBlocks) { st = XP_ERR_TOO_LARGE; why = "xp_behaviours: more than 64 (production, left size) blocks in one pass"; break; }
                        BehBlock& k = P.blocks[P.n_blocks++];
                        k.first = P.n_cand; k.cr = cr; k.lbase = base[gh.bins[b].lnt][a]; k.rbase = base[gh.bins[b].rnt][s - 1 - a]; k.op = gh.bins[b].op;
                        const bool commutes = k.op == XP_OP_ADD || k.op == XP_OP_MUL || k.op == XP_OP_MIN || k.op == XP_OP_MAX;
                        k.mirror = !commutes || gh.bins[b].lnt != gh.bins[b].rnt || 2 * a < s - 1 ? 0 : 2 * a == s - 1 ? 2 : 1;
                        P.n_cand += cl * cr;
                        if (P.n_cand >= kKindCand) { st = XP_ERR_TOO_LARGE; why = "xp_behaviours: 2^39 candidates or more in one pass"; break; }
                    }
            base[nt][s] = n_reps;
            if (st != XP_OK) break;
            if (nt == hs.start_nt) out->enumerated[s] = P.n_cand;
            bytes += P.n_cand * (u64)(2 * 8 * ns + 16);
            for (u64 first = 0; first < P.n_cand && cu.ok() && st == XP_OK; first += kBehChunk) {
                const u32 n = (u32)(P.n_cand - first < kBehChunk ? P.n_cand - first : kBehChunk);
                const int nb = (int)((n + kBehThreads - 1) / kBehThreads);
                // room for every candidate of the chunk at half the slots
                u64 want = table[nt] ? table[nt] : kBehTable;
                while (want < 2 * (held[nt] + n)) want <<= 1;
                if (want > tsize) want = tsize;
                if (want != table[nt]) {
                    cu(cudaMemsetAsync((u64*)(block + o_tab) + tsize * nt, 0xff, sizeof(u64) * want, stream));
                    const BehRanges R = ranges_of(nt);
                    if (R.total > 0 && cu.ok()) {
                        chain(beh_rehash_kernel, (unsigned)((R.total + kBehThreads - 1) / kBehThreads), kBehThreads, 0, stream, dB, nt, want - 1, R);
                        ++launches;
                    }
                    table[nt] = want;
                }
                P.mask = table[nt] - 1;
                if (ns <= 8) chain(beh_insert_kernel<8>, nb, kBehThreads, 0, stream, dB, P, first, n);
                else chain(beh_insert_kernel<XP_MAX_SIG>, nb, kBehThreads, 0, stream, dB, P, first, n);
                chain(beh_flag_kernel, nb, kBehThreads, 0, stream, dB, nt, first, n);
                if (!stage.locked) cu(cudaMemcpyAsync(&back.chunk_new, (char*)dB + kBackAt, 2 * sizeof(u64), cudaMemcpyDeviceToHost, stream));
                cu(cudaEventRecord(counted.e0, stream));
                chain(beh_append_kernel, nb, kBehThreads, 0, stream, dB, P, first, n, n_reps, max_reps);
                launches += 3;
                cu(cudaGetLastError());
                cu(cudaEventSynchronize(counted.e0));     // (the append runs on while the host prepares the next pass)
                if (!cu.ok()) break;
                if (back.err) { st = XP_ERR_TOO_LARGE; why = "xp_behaviours: the hash table is too full (raise max_representatives)"; break; }
                if (n_reps + back.chunk_new > max_reps) {
                    st = XP_ERR_TOO_LARGE;
                    why = "xp_behaviours: more than " + std::to_string(max_reps) + " representatives (size " + std::to_string(s) + ")";
                    break;
                }
                n_reps += back.chunk_new;
                held[nt] += back.chunk_new;
                count[nt][s] += back.chunk_new;
                bytes += back.chunk_new * (u64)(2 * 8 * ns + 24);
            }
            if (nt == hs.start_nt) out->distinct[s] = count[nt][s];
        }
    // the hole's representatives against the constraint, then the whole-domain checks in order (the first of them queued with it)
    int sms = 148;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const i64 point_ctas = (si.n_points + kBehThreads - 1) / kBehThreads, verify_ctas = point_ctas < 1 ? 1 : point_ctas < sms * 8 ? point_ctas : sms * 8;
    std::vector<u32> ids;
    if (cu.ok() && st == XP_OK) {
        const BehRanges R = ranges_of(hs.start_nt);
        if (R.total > 0) {
            chain(beh_match_kernel, (unsigned)((R.total + kBehThreads - 1) / kBehThreads), kBehThreads, 0, stream, dB, R);
            chain(beh_verify_kernel, (unsigned)verify_ctas, kBehThreads, 0, stream, dB, kFirstMatch);
            launches += 2;
        }
        cu(cudaGetLastError());
        cu(cudaEventRecord(ev.e1, stream));
        cu(cudaMemcpyAsync(&back.chunk_new, (char*)dB + kBackAt, sizeof(BehDev) - kBackAt, cudaMemcpyDeviceToHost, stream));
        cu(cudaStreamSynchronize(stream));
        if (cu.ok()) {
            out->sig_matches = back.match_count;
            const u32 n = back.match_n < (u32)kMatchCap ? back.match_n : (u32)kMatchCap;
            ids.assign(back.match_id, back.match_id + n);
            std::sort(ids.begin(), ids.end());            // ids grow with (size, order found) within a nonterminal
            if (back.match_n > (u32)kMatchCap) { st = XP_ERR_TOO_LARGE; why = "xp_behaviours: more than 256 representatives satisfy the signature points"; }
        }
    }
    auto locate = [&](u32 gid, int* size, u64* index) {
        for (int s = 1; s <= K; ++s)
            if (gid >= base[hs.start_nt][s] && gid < base[hs.start_nt][s] + count[hs.start_nt][s]) { *size = s; *index = gid - base[hs.start_nt][s]; }
    };
    // text of the tree that the last whole-domain check left in `back` (nodes in preorder)
    std::function<void(u32&, std::string&)> text_of = [&](u32& at, std::string& t) {
        if (at >= back.n_nodes) return;
        const RepDesc r = back.node[at++];
        if (r.op_or_leaf & kLeafBit) {
            const LeafDev& lf = gh.leaves[r.op_or_leaf & ~kLeafBit];
            t += lf.var >= 0 ? std::string(gh.var_names[lf.var]) : std::to_string((long long)lf.value);
            return;
        }
        static const char* const kText[] = {"+", "-", "*", "/", "%", "<", "<=", "==", "!=", "min", "max", "&&", "||", "<<", ">>"};
        const bool call = r.op_or_leaf == XP_OP_MIN || r.op_or_leaf == XP_OP_MAX;
        t += call ? std::string(kText[r.op_or_leaf]) + "(" : std::string("(");
        text_of(at, t);
        t += call ? "," : kText[r.op_or_leaf];
        text_of(at, t);
        t += ")";
    };
    constexpr size_t kCheckAt = offsetof(BehDev, verify_fail);
    for (size_t k = 0; k < ids.size() && cu.ok() && st == XP_OK && !out->solved; ++k) {
        if (k > 0) {
            cu(cudaMemsetAsync((char*)dB + kCheckAt, 0, sizeof(u32), stream));
            chain(beh_verify_kernel, (unsigned)verify_ctas, kBehThreads, 0, stream, dB, ids[k]);
            ++launches;
            cu(cudaGetLastError());
            cu(cudaEventRecord(ev.e1, stream));
            cu(cudaMemcpyAsync(&back.verify_fail, (char*)dB + kCheckAt, sizeof(BehDev) - kCheckAt, cudaMemcpyDeviceToHost, stream));
            cu(cudaStreamSynchronize(stream));
            if (!cu.ok()) break;
        }
        const u32 fail = back.verify_fail;
        std::string t;
        int size = 0;
        u64 index = 0;
        locate(ids[k], &size, &index);
        u32 node = 0;
        text_of(node, t);
        if (k == 0) {
            out->hit = 1; out->hit_size = size; out->hit_index = index; out->hit_verified = fail ? 0 : 1;
            snprintf(out->hit_text, sizeof(out->hit_text), "%s", t.c_str());
        }
        if (!fail) {
            out->solved = 1; out->solution_size = size; out->solution_index = index;
            snprintf(out->solution_text, sizeof(out->solution_text), "%s", t.c_str());
        }
    }
    float ms = 0.f;
    if (cu.ok() && st == XP_OK) cu(cudaEventElapsedTime(&ms, ev.e0, ev.e1));      // (recorded before the last copy, which has been waited for)
    else cudaStreamSynchronize(stream);
    device_release(block, granted, bdev);
    if (!cu.ok()) return set_error(XP_ERR_CUDA, (std::string("xp_behaviours: ") + cudaGetErrorString(cu.e)).c_str());
    if (st != XP_OK) return set_error(st, why.c_str());
    out->max_size = K;
    out->representatives = n_reps;
    out->bytes_moved = bytes;
    out->kernel_ms = ms;
    out->n_launches = launches;
    out->total_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return XP_OK;
}
