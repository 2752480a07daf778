// Two holes inside one constraint: the product search of xp_repair_joint (include/xp.h).
//
//   joint_probe_kernel   -- coordinates and spec values of the probe points (the first sample points
//                           of the sketch: box corners first, then ids spread by a fixed hash).
// A context that is affine in both parts, A0 h0 + A1 h1 + B (the usual one: a stride and an offset), is searched from
// one side: the pair satisfies the probes iff A1 h1 = spec - B - A0 h0 at all of them.
//   joint_key_kernel     -- thread = candidate of one part: its side of that equation at every probe, hashed to 64 bits.
//                           Part 1 goes into hash chains; part 0 then walks the chain of its own key and lists
//                           the partners.  N0 + N1 candidates are evaluated instead of N0 * N1 pairs.
//   joint_check_kernel   -- a warp per listed pair: the whole domain, lane = point, vote exit.
// Any other context (and a list that ran over):
//   joint_values_kernel  -- value at every probe of every candidate of either part (every size up
//                           to its bound): thread = (table entry, probe).
//   joint_pairs_kernel   -- one (size of part 0, size of part 1) block of the pair space: thread =
//                           pair, rank of part 1 fastest; the constraint is evaluated at the probes
//                           from the tables, first failure ends the pair; the pairs of a warp that
//                           pass every probe are checked on the whole domain by the warp together.
// Matches go into per-total-size counts (sum) and least keys (min) by atomics.
// No CTA or warp waits for another.
#include <cuda_runtime.h>

#include <chrono>
#include <cstddef>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "xp_device.cuh"
#include "xp_launch.h"

namespace xp {

constexpr int kJointProbes = 16;
constexpr int kJointTotal = 2 * kMaxSize;                 // largest total size of a pair
constexpr u64 kJointMaxEntries = 1ull << 22;              // candidates of one part and size
constexpr u64 kJointMaxPairs = 1ull << 40;

struct JointDev {
    const SketchDev* sk;
    i32 n_probe, ctx_len, spec_len, pad;
    u32 spec_ok, pad2;                                    // bit j: the spec is defined at probe j
    i32 start_nt[2], max_size[2];
    i64 probe_id[kJointProbes];
    i64 probe_pt[kJointProbes][kMaxVars];
    i64 probe_spec[kJointProbes];
    xp_instr ctx[kMaxCode], spec[kMaxCode];
    const i64* spec_table;                                // device, or null: evaluate `spec`
    u64 tab_off[2][kMaxSize + 1];                         // first entry of each size in a part's table
    u64 tab_total[2];
    i64* tab_val[2];                                      // device, [probe][entry]
    unsigned char* tab_ok[2];
    // the search from one side: context coefficients per probe, part 1's chains, the listed pairs
    u64 A0[kJointProbes], A1[kJointProbes], B[kJointProbes];
    u32 undefined, head_mask;                             // undefined: bit j: a hole-free part of the context is undefined at probe j
    u32* head;                                            // device, all ones at launch: (head_mask + 1) x lanes per candidate
    uint4* node;                                          // per candidate of part 1: key (low, high word), next in its chain
    uint2* list;                                          // device, kJointList entries (candidate of part 0, of part 1)
    // results, read back together
    u64 match_count[kJointTotal + 1];
    u64 min_key[kJointTotal + 1];                         // size of part 0 << 48 | rank 0 << 24 | rank 1 (all-ones: none)
    u64 evals, survivors, listed;
};
constexpr u64 kJointList = 1ull << 20;                    // pairs that pass the probes, at most (more: the other form)

// The context at one point as A0 h0 + A1 h1 + B in wrap-around arithmetic (its form was checked on the host); false when
// a hole-free operand is undefined there.
__device__ bool joint_affine_at(const xp_instr* code, int n, const i64* pt, u64& A0, u64& A1, u64& B) {
    u64 a[kMaxStack], b[kMaxStack], c[kMaxStack];
    u32 has = 0;
    int sp = 0;
    for (int i = 0; i < n; ++i) {
        const xp_instr q = code[i];
        if (q.kind != XP_I_OP) {
            a[sp] = q.kind == XP_I_HOLE && q.arg == 0 ? 1ull : 0ull;
            b[sp] = q.kind == XP_I_HOLE && q.arg == 1 ? 1ull : 0ull;
            c[sp] = q.kind == XP_I_VAR ? (u64)pt[q.arg] : q.kind == XP_I_CONST ? (u64)q.value : 0ull;
            has = (has & ~(1u << sp)) | ((u32)(q.kind == XP_I_HOLE) << sp);
            ++sp;
            continue;
        }
        --sp;
        const bool hy = (has >> sp) & 1u, hx = (has >> (sp - 1)) & 1u;
        if (!hx && !hy) {
            i64 r;
            if (!apply_op(q.arg, (i64)c[sp - 1], (i64)c[sp], r)) return false;
            c[sp - 1] = (u64)r;
            continue;
        }
        if (q.arg == XP_OP_ADD) { a[sp - 1] += a[sp]; b[sp - 1] += b[sp]; c[sp - 1] += c[sp]; }
        else if (q.arg == XP_OP_SUB) { a[sp - 1] -= a[sp]; b[sp - 1] -= b[sp]; c[sp - 1] -= c[sp]; }
        else {                                            // a product with one hole-free side
            const u64 f = hx ? c[sp] : c[sp - 1];
            const int k = hx ? sp - 1 : sp;
            a[sp - 1] = a[k] * f; b[sp - 1] = b[k] * f; c[sp - 1] = c[k] * f;
        }
        has |= 1u << (sp - 1);
    }
    A0 = a[0]; A1 = b[0]; B = c[0];
    return true;
}

// Value of the joint context at one point from the values of its two parts.
__device__ __forceinline__ bool eval_joint(const xp_instr* code, int n, const i64* pt, i64 h0, i64 h1, i64& out) {
    i64 st[kMaxStack];
    int sp = 0;
    for (int i = 0; i < n; ++i) {
        const xp_instr c = code[i];
        if (c.kind == XP_I_OP) {
            const i64 b = st[--sp];
            const i64 a = st[sp - 1];
            i64 r;
            if (!apply_op(c.arg, a, b, r)) return false;
            st[sp - 1] = r;
        } else {
            if (!XP_CHECKED(sp < kMaxStack, kChkStack)) return false;
            st[sp++] = c.kind == XP_I_VAR ? pt[c.arg] : (c.kind == XP_I_CONST ? c.value : (c.arg == 0 ? h0 : h1));
        }
    }
    out = st[0];
    return true;
}

__global__ void joint_probe_kernel(JointDev* J, int affine) {
    chain_wait();
    const int t = threadIdx.x;
    const SketchDev* sk = J->sk;
    bool ok = false;
    if (t < J->n_probe) {
        i64 pt[kMaxVars];
        const i64 pid = sk->sample_id[t];
        point_coords(sk, pid, pt);
        for (int d = 0; d < sk->n_vars; ++d) J->probe_pt[t][d] = pt[d];
        J->probe_id[t] = pid;
        i64 v = 0;
        ok = true;
        if (J->spec_table != nullptr) v = J->spec_table[pid];
        else ok = eval_code(J->spec, J->spec_len, pt, 0, v);
        J->probe_spec[t] = v;
    }
    const u32 m = __ballot_sync(0xffffffffu, ok);
    if (t == 0) J->spec_ok = m;
    if (!affine) return;
    bool undef = false;
    if (t < J->n_probe) undef = !joint_affine_at(J->ctx, J->ctx_len, J->probe_pt[t], J->A0[t], J->A1[t], J->B[t]);
    const u32 u = __ballot_sync(0xffffffffu, undef);
    if (t == 0) J->undefined = u;
}

// Size and rank of candidate number e of a part.
__device__ __forceinline__ int joint_locate(const JointDev* J, int part, u64 e, u64& rank) {
    int s = 1;
    while (s < J->max_size[part] && J->tab_off[part][s + 1] <= e) ++s;
    rank = e - J->tab_off[part][s];
    return s;
}

// LANES threads per candidate, each with every LANES-th probe: sixteen evaluations one after the other were the kernel's whole time where
// there are few candidates (5 000: 18 us for part 1, now 7), and unranking the candidate once per lane is what the others
// pay for it where there are many.
// The lanes of a candidate of part 0 also share the partners: a key has a chain for every LANES-th candidate of part 1, and each lane walks
// one (five thousand candidates, a few hundred with the same key: 150 us in one chain, now 20).
constexpr u64 kJointSpread = 1ull << 16;                  // candidates of either part up to which 16 lanes share one
template <int LANES>
__global__ void __launch_bounds__(128) joint_key_kernel(JointDev* J, int part) {
    chain_wait();
    const SketchDev* sk = J->sk;
    const GrammarDev* g = sk->g;
    const u64 e = ((u64)blockIdx.x * blockDim.x + threadIdx.x) / LANES;
    const int np = J->n_probe, sub = (int)(threadIdx.x % LANES);
    const u32 all = np >= 32 ? 0xffffffffu : (1u << np) - 1u;
    if ((J->spec_ok & all) != all || (J->undefined & all) != 0u) return;      // nothing can match
    u32 ran = 0;
    u64 key = 0;
    bool ok = e < J->tab_total[part];
    if (ok) {
        u64 rank;
        const int s = joint_locate(J, part, e, rank);
        u32 code[kMaxSize];
        const int n = unrank(g, J->start_nt[part], s, rank, code);
#pragma unroll 1
        for (int j = sub; j < np && ok; j += LANES) {
            i64 h;
            ++ran;
            ok = eval_cand(code, n, g->leaves, J->probe_pt[j], h);
            u64 v = part ? J->A1[j] * (u64)h : (u64)J->probe_spec[j] - J->B[j] - J->A0[j] * (u64)h;
            v = (v + (u64)(j + 1) * 0x9E3779B97F4A7C15ull) * 0xD1342543DE82EF95ull;      // (a sum over the probes, in any order)
            v = (v ^ (v >> 32)) * 0xDA942042E4DD58B5ull;
            key += v ^ (v >> 29);
        }
    }
    if (LANES > 1) {
#pragma unroll
        for (int o = LANES / 2; o > 0; o >>= 1) key += __shfl_xor_sync(0xffffffffu, key, o);
        const u32 mine = ((1u << (LANES & 31)) - 1u) << ((threadIdx.x & 31) & ~(LANES - 1));
        ok = (__ballot_sync(0xffffffffu, ok) & mine) == mine && (part == 0 || sub == 0);
    }
    if (ok) {
        u32* head = &J->head[(((u32)(key >> 32) & J->head_mask) * LANES + (part ? (u32)(e % LANES) : (u32)sub))];
        if (part) J->node[e] = make_uint4((u32)key, (u32)(key >> 32), atomicExch(head, (u32)e), 0u);
        else
            for (u32 y = *head; y != 0xffffffffu;) {
                const uint4 q = J->node[y];
                if (q.x == (u32)key && q.y == (u32)(key >> 32)) {      // (an equal key that is no match fails on the domain, probes among it)
                    const u64 at = atomicAdd((unsigned long long*)&J->listed, 1ull);
                    if (at >= kJointList) break;          // (the host takes the other form)
                    J->list[at] = make_uint2((u32)e, y);
                }
                y = q.z;
            }
    }
    for (int o = 16; o > 0; o >>= 1) ran += __shfl_down_sync(0xffffffffu, ran, o);
    if ((threadIdx.x & 31) == 0 && ran) atomicAdd((unsigned long long*)&J->evals, (u64)ran);
}

__global__ void __launch_bounds__(256) joint_values_kernel(JointDev* J, int part, int size) {
    chain_wait();
    const SketchDev* sk = J->sk;
    const GrammarDev* g = sk->g;
    const int nt = J->start_nt[part];
    const u64 rank = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    const int pr = blockIdx.y;
    if (rank >= g->cnt[nt][size] || pr >= J->n_probe) return;
    u32 code[kMaxSize];
    const int n = unrank(g, nt, size, rank, code);
    i64 v = 0;
    const bool ok = eval_cand(code, n, g->leaves, J->probe_pt[pr], v);
    const u64 at = (u64)pr * J->tab_total[part] + J->tab_off[part][size] + rank;
    J->tab_val[part][at] = v;
    J->tab_ok[part][at] = ok ? 1 : 0;
}

// The pair (tree r0 of size s0, tree r1 of size s1) on every domain point; called by all 32
// lanes of a warp together, or by all threads of a CTA.  Adds the points tried to evals.
template <bool CTA>
__device__ __noinline__ bool joint_check_domain(const JointDev* J, int s0, u64 r0, int s1, u64 r1, u64& evals) {
    const SketchDev* sk = J->sk;
    const GrammarDev* g = sk->g;
    const int width = CTA ? (int)blockDim.x : 32;
    u32 c0[kMaxSize], c1[kMaxSize];
    const int n0 = unrank(g, J->start_nt[0], s0, r0, c0);
    const int n1 = unrank(g, J->start_nt[1], s1, r1, c1);
#pragma unroll 1
    for (i64 base = 0; base < sk->n_points; base += width) {
        bool bad = false;
        const i64 pid = base + (CTA ? (int)threadIdx.x : (int)(threadIdx.x & 31));
        if (pid < sk->n_points) {
            ++evals;
            i64 pt[kMaxVars];
            point_coords(sk, pid, pt);
            i64 want = 0, h0, h1, v;
            bool ok = true;
            if (J->spec_table != nullptr) want = J->spec_table[pid];
            else ok = eval_code(J->spec, J->spec_len, pt, 0, want);
            ok = ok && eval_cand(c0, n0, g->leaves, pt, h0) && eval_cand(c1, n1, g->leaves, pt, h1) &&
                 eval_joint(J->ctx, J->ctx_len, pt, h0, h1, v) && v == want;
            bad = !ok;
        }
        if (CTA ? __syncthreads_or(bad) != 0 : __any_sync(0xffffffffu, bad)) return false;
    }
    return true;
}

__global__ void __launch_bounds__(256) joint_pairs_kernel(JointDev* J, int s0, int s1, u64 n0, u64 n1) {
    chain_wait();
    const int lane = threadIdx.x & 31;
    const u64 pairs = n0 * n1;
    const u64 stride = (u64)gridDim.x * blockDim.x;
    const int np = J->n_probe;
    const u32 spec_ok = J->spec_ok;
    const u64 all_ok = np >= 32 ? 0xffffffffu : (1u << np) - 1u;
    u64 evals = 0, survivors = 0;
    // (whole warps walk the loop together: the bound is rounded up to a multiple of the warp's 32 pairs)
    for (u64 q0 = ((u64)blockIdx.x * blockDim.x + threadIdx.x) & ~31ull; q0 < pairs; q0 += stride) {
        const u64 q = q0 + lane;
        bool pass = q < pairs && (spec_ok & all_ok) == all_ok;          // a spec undefined at a probe: nothing matches
        u64 r0 = 0, r1 = 0;
        if (pass) {
            r0 = q / n1; r1 = q - r0 * n1;
            const u64 e0 = J->tab_off[0][s0] + r0, e1 = J->tab_off[1][s1] + r1;
            for (int j = 0; j < np && pass; ++j) {
                ++evals;
                const u64 a0 = (u64)j * J->tab_total[0] + e0, a1 = (u64)j * J->tab_total[1] + e1;
                i64 v;
                pass = J->tab_ok[0][a0] && J->tab_ok[1][a1] &&
                       eval_joint(J->ctx, J->ctx_len, J->probe_pt[j], J->tab_val[0][a0], J->tab_val[1][a1], v) && v == J->probe_spec[j];
            }
        }
        u32 m = __ballot_sync(0xffffffffu, pass);
        survivors += (u64)__popc(m) * (lane == 0);
        while (m) {                                       // the warp checks its survivors on the whole domain, one by one
            const int src = __ffs((int)m) - 1;
            m &= m - 1;
            const u64 x0 = __shfl_sync(0xffffffffu, r0, src), x1 = __shfl_sync(0xffffffffu, r1, src);
            if (joint_check_domain<false>(J, s0, x0, s1, x1, evals) && lane == 0) {
                atomicAdd(&J->match_count[s0 + s1], 1ull);
                atomicMin(&J->min_key[s0 + s1], ((u64)s0 << 48) | (x0 << 24) | x1);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) evals += __shfl_down_sync(0xffffffffu, evals, o);
    if (lane == 0) {
        if (evals) atomicAdd(&J->evals, evals);
        if (survivors) atomicAdd(&J->survivors, survivors);
    }
}

// A CTA per listed pair while every CTA has few of them, a warp per pair where there are many: a pair's domain is a chain of steps that each
// wait for the interpreter (480 points in 15 steps of a warp: 51 us, in 2 of a CTA: 14).
__global__ void __launch_bounds__(256) joint_check_kernel(JointDev* J) {
    chain_wait();
    const u64 n = J->listed;
    if (n > kJointList) return;                           // (the list ran over: the host takes the other form)
    const bool wide = n <= 4ull * gridDim.x;
    u64 evals = 0;
    for (u64 i = wide ? (u64)blockIdx.x : (u64)blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += wide ? (u64)gridDim.x : (u64)gridDim.x * 8) {
        u64 r0, r1;
        const int s0 = joint_locate(J, 0, J->list[i].x, r0), s1 = joint_locate(J, 1, J->list[i].y, r1);
        const bool ok = wide ? joint_check_domain<true>(J, s0, r0, s1, r1, evals) : joint_check_domain<false>(J, s0, r0, s1, r1, evals);
        if (ok && (threadIdx.x & (wide ? 255 : 31)) == 0) {
            atomicAdd(&J->match_count[s0 + s1], 1ull);
            atomicMin(&J->min_key[s0 + s1], ((u64)s0 << 48) | (r0 << 24) | r1);
        }
    }
    for (int o = 16; o > 0; o >>= 1) evals += __shfl_down_sync(0xffffffffu, evals, o);
    if ((threadIdx.x & 31) == 0 && evals) atomicAdd(&J->evals, evals);
}

}  // namespace xp

using namespace xp;

// Is the context affine in both parts whatever the point: no hole under an operator but + - *, none times another?
static bool joint_is_affine(const xp_instr* code, int n) {
    bool has[kMaxStack + 1];
    int sp = 0;
    for (int i = 0; i < n; ++i) {
        if (code[i].kind != XP_I_OP) { has[sp++] = code[i].kind == XP_I_HOLE; continue; }
        --sp;
        const bool x = has[sp - 1], y = has[sp];
        if (x || y) {
            if (code[i].arg > XP_OP_MUL || (code[i].arg == XP_OP_MUL && x && y)) return false;
            has[sp - 1] = true;
        }
    }
    return true;
}

struct xp_joint_result {
    int solved = 0, max_total = 0, least_total = 0, least_size[2] = {0, 0};
    u64 cand[kJointTotal + 1] = {0}, match[kJointTotal + 1] = {0};
    u64 least_rank[2] = {0, 0};
    std::string text[2];
    u64 evals = 0, survivors = 0;
    double kernel_ms = 0, total_ms = 0;
    int n_launches = 0;
};

extern "C" xp_status xp_joint_result_get(const xp_joint_result* r, xp_joint_view* v) {
    if (!r || !v) return set_error(XP_ERR_INVALID_ARG, "xp_joint_result_get: null argument");
    v->solved = r->solved; v->max_total = r->max_total;
    v->cand_count = (const uint64_t*)r->cand; v->match_count = (const uint64_t*)r->match;
    v->least_total = r->least_total;
    for (int k = 0; k < 2; ++k) { v->least_size[k] = r->least_size[k]; v->least_rank[k] = r->least_rank[k]; v->least_text[k] = r->text[k].c_str(); }
    v->evals_executed = r->evals; v->probe_survivors = r->survivors;
    v->kernel_ms = r->kernel_ms; v->total_ms = r->total_ms; v->n_launches = r->n_launches;
    return XP_OK;
}

extern "C" void xp_joint_result_free(xp_joint_result* r) { delete r; }

static bool joint_code_ok(const xp_instr* code, int n, int n_vars, bool holes, int* parts_seen) {
    if (n < 1 || n > kMaxCode || !code) return false;
    int sp = 0;
    for (int i = 0; i < n; ++i) {
        const xp_instr& c = code[i];
        if (c.kind == XP_I_OP) { if (c.arg < XP_OP_ADD || c.arg > XP_OP_SHR || sp < 2) return false; --sp; continue; }
        if (c.kind == XP_I_VAR) { if (c.arg < 0 || c.arg >= n_vars) return false; }
        else if (c.kind == XP_I_HOLE) { if (!holes || c.arg < 0 || c.arg > 1) return false; *parts_seen |= 1 << c.arg; }
        else if (c.kind != XP_I_CONST) return false;
        if (++sp > kMaxStack) return false;
    }
    return sp == 1;
}

extern "C" xp_status xp_repair_joint(const xp_sketch* sketch, const xp_joint_desc* d, const xp_repair_opts* opts, xp_joint_result** out) {
    if (!sketch || !d || !out) return set_error(XP_ERR_INVALID_ARG, "xp_repair_joint: null argument");
    *out = nullptr;
    const auto t0 = std::chrono::steady_clock::now();
    const SketchInternals si = sketch_internals(sketch);
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return set_error(XP_ERR_CUDA, "no CUDA device is usable");
    if (dev != si.device) return set_error(XP_ERR_INVALID_ARG, "xp_repair_joint: the sketch was loaded on another device than the current one");
    int parts = 0, none = 0;
    if (!joint_code_ok(d->ctx, d->ctx_len, si.n_vars, true, &parts) || parts != 3)
        return set_error(XP_ERR_SKETCH, "xp_repair_joint: malformed context, or one that does not mention both parts");
    if (d->spec_kind == XP_SPEC_EXPR) {
        if (!joint_code_ok(d->spec_expr, d->spec_len, si.n_vars, false, &none)) return set_error(XP_ERR_SKETCH, "xp_repair_joint: malformed spec expression");
    } else if (d->spec_kind != XP_SPEC_TABLE || (si.n_points > 0 && !d->spec_table)) return set_error(XP_ERR_SKETCH, "xp_repair_joint: bad spec");
    xp_joint_result* r = new (std::nothrow) xp_joint_result;
    if (!r) return set_error(XP_ERR_NOMEM, "out of host memory");
    JointDev h;
    memset(&h, 0, sizeof(h));
    u64 entries[2] = {0, 0};
    for (int k = 0; k < 2; ++k) {
        const int nt = d->start_nt[k], K = d->max_size[k];
        if (nt < 0 || nt >= grammar_nonterminals(si.g) || K < 1 || K > kMaxSize) { delete r; return set_error(XP_ERR_SKETCH, "xp_repair_joint: start_nt or max_size out of range"); }
        if (K > grammar_ok_size(si.g)) { delete r; return set_error(XP_ERR_TOO_LARGE, "a candidate count reaches 2^63 within the size bound"); }
        h.start_nt[k] = nt; h.max_size[k] = K;
        for (int s = 1; s <= K; ++s) {
            const u64 c = grammar_cnt(si.g, nt, s);
            if (c >= kJointMaxEntries) { delete r; return set_error(XP_ERR_TOO_LARGE, "xp_repair_joint: a part has 2^22 candidates or more of one size"); }
            h.tab_off[k][s] = entries[k];
            entries[k] += c;
        }
        h.tab_total[k] = entries[k];
    }
    r->max_total = d->max_size[0] + d->max_size[1];
    u64 all_pairs = 0;
    for (int s0 = 1; s0 <= d->max_size[0]; ++s0)
        for (int s1 = 1; s1 <= d->max_size[1]; ++s1) {
            const u64 p = grammar_cnt(si.g, d->start_nt[0], s0) * grammar_cnt(si.g, d->start_nt[1], s1);      // (< 2^44)
            r->cand[s0 + s1] += p;
            all_pairs += p;
        }
    if (all_pairs > kJointMaxPairs) { delete r; return set_error(XP_ERR_TOO_LARGE, "xp_repair_joint: more than 2^40 pairs"); }
    if (si.n_points == 0) {                                 // no constraint at all: every pair satisfies it
        for (int t = 2; t <= r->max_total; ++t) r->match[t] = r->cand[t];
        for (int t = 2; t <= r->max_total && !r->solved; ++t)
            for (int s0 = 1; s0 < t && !r->solved; ++s0)
                if (s0 <= d->max_size[0] && t - s0 <= d->max_size[1] && grammar_cnt(si.g, d->start_nt[0], s0) * grammar_cnt(si.g, d->start_nt[1], t - s0) > 0) {
                    r->solved = 1; r->least_total = t; r->least_size[0] = s0; r->least_size[1] = t - s0;
                    for (int k = 0; k < 2; ++k) {
                        char buf[1024];
                        if (xp_grammar_unrank(si.g, d->start_nt[k], r->least_size[k], 0, nullptr, 0, buf, sizeof(buf)) == XP_OK) r->text[k] = buf;
                    }
                }
        r->total_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
        *out = r;
        return XP_OK;
    }
    const int n_probe = (int)(si.n_points < kJointProbes ? si.n_points : kJointProbes);
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const bool copy_spec = d->spec_kind == XP_SPEC_TABLE && si.n_points > 0 && !d->spec_table_on_device;
    const bool affine = joint_is_affine(d->ctx, d->ctx_len);
    const size_t result_at = offsetof(JointDev, match_count), result_bytes = sizeof(JointDev) - result_at;
    StageMemory stage(sizeof(JointDev));
    StageEvents ev;
    cudaStream_t stream = opts ? (cudaStream_t)opts->stream : nullptr;
    float ms = 0.f;
    int launches = 0, sms = 148;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (!stage.p) { delete r; return set_error(XP_ERR_NOMEM, "out of host memory"); }
    JointDev& back = *(JointDev*)stage.p;
    // The search from one side first where the context allows it; the pair by pair form otherwise, or when more pairs
    // pass the probes than the list holds.
    for (int form = affine ? 0 : 1; form < 2; ++form) {
        // one device block: the record, the spec table (if it is the host's), then the form's tables
        size_t off = al(sizeof(JointDev));
        const size_t off_spec = off;
        if (copy_spec) off += al(sizeof(i64) * (size_t)si.n_points);
        size_t off_val[2] = {0, 0}, off_ok[2] = {0, 0}, off_head = 0, off_node = 0, off_list = 0;
        const bool spread = entries[0] <= kJointSpread && entries[1] <= kJointSpread;
        const u32 lanes = spread ? 16u : 1u;
        u32 heads = 1024;
        while ((u64)heads * lanes < 2 * entries[1]) heads <<= 1;
        if (form == 0) {
            off_head = off; off += al(sizeof(u32) * heads * lanes);
            off_node = off; off += al(sizeof(uint4) * entries[1]);
            off_list = off; off += al(sizeof(uint2) * kJointList);
        } else
            for (int k = 0; k < 2; ++k) {
                off_val[k] = off; off += al(sizeof(i64) * entries[k] * (size_t)n_probe);
                off_ok[k] = off; off += al(entries[k] * (size_t)n_probe);
            }
        char* block = nullptr;
        size_t granted = 0;
        int bdev = 0;
        if (device_alloc((void**)&block, off, &bdev, &granted) != cudaSuccess) {
            (void)cudaGetLastError();
            delete r;
            return set_error(XP_ERR_NOMEM, "xp_repair_joint: device memory for the tables");
        }
        h.sk = si.d_s; h.n_probe = n_probe; h.ctx_len = d->ctx_len;
        memcpy(h.ctx, d->ctx, sizeof(xp_instr) * d->ctx_len);
        if (d->spec_kind == XP_SPEC_EXPR) { h.spec_len = d->spec_len; memcpy(h.spec, d->spec_expr, sizeof(xp_instr) * d->spec_len); }
        else if (si.n_points > 0) h.spec_table = copy_spec ? (const i64*)(block + off_spec) : (const i64*)d->spec_table;
        for (int k = 0; k < 2; ++k) { h.tab_val[k] = (i64*)(block + off_val[k]); h.tab_ok[k] = (unsigned char*)(block + off_ok[k]); }
        h.head = (u32*)(block + off_head); h.node = (uint4*)(block + off_node); h.list = (uint2*)(block + off_list);
        h.head_mask = heads - 1;
        for (int t = 0; t <= kJointTotal; ++t) h.min_key[t] = ~0ull;
        JointDev* dJ = (JointDev*)block;
        memcpy(stage.p, &h, sizeof(h));
        cudaError_t e = ev.e0 ? cudaSuccess : ev.open();
        if (e == cudaSuccess) e = cudaMemcpyAsync(dJ, stage.p, sizeof(h), cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess && copy_spec) e = cudaMemcpyAsync(block + off_spec, d->spec_table, sizeof(i64) * (size_t)si.n_points, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess && form == 0) e = cudaMemsetAsync(block + off_head, 0xff, sizeof(u32) * heads * lanes, stream);
        if (e == cudaSuccess) e = cudaEventRecord(ev.e0, stream);
        if (e == cudaSuccess) {
            chain(joint_probe_kernel, 1, 32, 0, stream, dJ, form == 0 ? 1 : 0);
            ++launches;
            e = cudaGetLastError();
        }
        if (form == 0) {
            for (int part = 1; part >= 0 && e == cudaSuccess; --part) {
                if (entries[part] == 0) continue;
                if (spread) chain(joint_key_kernel<16>, (unsigned)((entries[part] + 7) / 8), 128, 0, stream, dJ, part);
                else chain(joint_key_kernel<1>, (unsigned)((entries[part] + 127) / 128), 128, 0, stream, dJ, part);
                ++launches;
                e = cudaGetLastError();
            }
            if (e == cudaSuccess) {
                chain(joint_check_kernel, (unsigned)sms * 4, 256, 0, stream, dJ);
                ++launches;
                e = cudaGetLastError();
            }
        } else {
            for (int k = 0; k < 2 && e == cudaSuccess; ++k)
                for (int s = 1; s <= d->max_size[k] && e == cudaSuccess; ++s) {
                    const u64 c = grammar_cnt(si.g, d->start_nt[k], s);
                    if (c == 0) continue;
                    chain(joint_values_kernel, dim3((unsigned)((c + 255) / 256), (unsigned)n_probe), 256, 0, stream, dJ, k, s);
                    ++launches;
                    e = cudaGetLastError();
                }
            for (int t = 2; t <= r->max_total && e == cudaSuccess; ++t)      // total size ascending (any order gives the same sums and minima)
                for (int s0 = 1; s0 < t && e == cudaSuccess; ++s0) {
                    const int s1 = t - s0;
                    if (s0 > d->max_size[0] || s1 > d->max_size[1]) continue;
                    const u64 n0 = grammar_cnt(si.g, d->start_nt[0], s0), n1 = grammar_cnt(si.g, d->start_nt[1], s1);
                    if (n0 == 0 || n1 == 0) continue;
                    const u64 want = (n0 * n1 + 255) / 256, most = (u64)sms * 8;
                    chain(joint_pairs_kernel, (unsigned)(want < most ? want : most), 256, 0, stream, dJ, s0, s1, n0, n1);
                    ++launches;
                    e = cudaGetLastError();
                }
        }
        float part_ms = 0.f;
        if (e == cudaSuccess) e = cudaEventRecord(ev.e1, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(stage.p + result_at, (char*)dJ + result_at, result_bytes, cudaMemcpyDeviceToHost, stream);
        const cudaError_t e2 = cudaStreamSynchronize(stream);
        if (e == cudaSuccess) e = e2;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&part_ms, ev.e0, ev.e1);
        device_release(block, granted, bdev);
        if (e != cudaSuccess) { delete r; return set_error(XP_ERR_CUDA, (std::string("xp_repair_joint: ") + cudaGetErrorString(e)).c_str()); }
        ms += part_ms;
        if (form == 0 && back.listed <= kJointList) { back.survivors = back.listed; break; }
    }
    for (int t = 2; t <= r->max_total; ++t) {
        r->match[t] = back.match_count[t];
        if (!r->solved && back.match_count[t] > 0) {
            r->solved = 1; r->least_total = t;
            const u64 key = back.min_key[t];
            r->least_size[0] = (int)(key >> 48); r->least_size[1] = t - r->least_size[0];
            r->least_rank[0] = (key >> 24) & 0xffffffull; r->least_rank[1] = key & 0xffffffull;
            for (int k = 0; k < 2; ++k) {
                char buf[1024];
                if (xp_grammar_unrank(si.g, d->start_nt[k], r->least_size[k], r->least_rank[k], nullptr, 0, buf, sizeof(buf)) == XP_OK) r->text[k] = buf;
            }
        }
    }
    r->evals = back.evals; r->survivors = back.survivors;
    r->kernel_ms = ms; r->n_launches = launches;
    r->total_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    *out = r;
    return XP_OK;
}
