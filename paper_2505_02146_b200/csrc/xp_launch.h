// Host-callable launchers of the kernels in xp_kernels.cu.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "xp_dev.h"

namespace xp {

// Kernels of one stream that follow one another: the next kernel's blocks are brought onto the SMs while the last blocks of the
// one before it still run, and wait there (chain_wait, the first statement of every kernel launched this way) until
// that one has finished and its writes are visible.  What a launch costs between two kernels (set-up, distribution of the blocks)
// is then spent while the first one runs (load and search of a two-variable nest, 7 launches: 211 -> 190 us with the merged
// staging and table launches; joint search 258 -> 242, behaviours 431 -> 413 us).
template <typename... P, typename... A>
inline cudaError_t chain(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args) {
    cudaLaunchAttribute early;
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid; c.blockDim = block; c.dynamicSmemBytes = smem; c.stream = stream;
    c.attrs = &early; c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();            // (the next kernel's blocks may come; they wait for this kernel's end)
}
#endif

size_t prepare_scratch_bytes(int n_jobs);
cudaError_t launch_prepare(const LoadJob* jobs, int n_jobs, const void* scratch, LoadOut* out, cudaStream_t stream);
cudaError_t launch_stage_sample(SketchDev* const* list, int n_sketches, i64 most_points, const LoadJob* jobs, int n_jobs, void* scratch, cudaStream_t stream);
cudaError_t launch_scatter(const LoadCopy* copies, int n_copies, const char* src, cudaStream_t stream);
constexpr size_t kPutMost = 31744;                   // (a launch takes 32 764 bytes of parameters)
struct PutPlaces { char* dst[3]; u32 end[3]; };      // 16-byte words [end[k - 1], end[k]) go to dst[k]
cudaError_t launch_put(const PutPlaces& to, const char* src, cudaStream_t stream);
cudaError_t launch_reprobe(const LoadJob* jobs, int n_jobs, cudaStream_t stream);
cudaError_t launch_coord_bounds(SketchDev* const* list, int n_sketches, i64 most_points, cudaStream_t stream);
cudaError_t launch_subvalues(const LoadJob* jobs, int n_jobs, int size, int last, int most_probes, u64 most_entries, cudaStream_t stream);
// Operand classes (csrc/xp_classes.cuh) of `n_jobs` holes at once (first: the first of them), `blocks` blocks in all; tables: what lies at the start of `scratch` and is zeroed.
inline u32 class_slots(u64 entries) { u32 n = 1024; while (n < 2 * entries) n <<= 1; return n; }
inline size_t class_table_bytes(u64 entries) { return sizeof(u64) * (size_t)class_slots(entries); }
inline size_t class_place_bytes(u64 entries) { return sizeof(uint2) * (size_t)entries; }
constexpr int kClassThreads = 256;
cudaError_t launch_classes(const ClassJob* jobs, int n_jobs, const ClassJob& first, u32 blocks, char* scratch, size_t tables, cudaStream_t stream);
// Layout of one call's device scratch (byte offsets from its 256-byte aligned base):
//   0: eval ticket (u64), 8: verify ticket (u64), 16: survivor pushes (u32), 20: failed-check word (u32; checked
//      build only), 24: long survivors (u32), 32: join ticket (u64), 40: finished verification CTAs (u32), 48: listed members
//      (u64: MemberRec entries and pieces), 56: ticket of those pieces (u64)   -- zero at launch
//   segs, jsegs, jgroups, psegs, sketches, acc: staged from the host;  [0, head) is what the host copies in
//   hist: survivors per accumulator slot, zero at launch (staged);
//   surv: the survivor queue (surv_cap entries); sort_off, sorted: its hole order (before that the list of members_kernel) -- written by the kernels only
struct SearchLayout {
    size_t segs, jsegs, jgroups, psegs, sketches, acc, hist, head, surv, sort_off, sorted, longs, total;
    size_t pair_ones, pair_zeros, pair_rest;      // scratch of the pair join: [pair_ones, pair_zeros) all ones, [pair_zeros, pair_rest) zero at launch
    i32 first_points;                // points of the largest domain, at most kVerifyChunk
    u32 member_cap;                  // entries of the list of members_kernel (0: no operand of the call is a class)
    u32 surv_cap, max_chunks;        // max_chunks: chunks of the whole-domain check that the largest domain needs
    int n_segs, n_jsegs, n_psegs, n_sketches, n_acc;
    int dense;                       // some hole of the plan takes the second look: launch the search kernel's dense form
    int join_wide;                   // tickets of the leaf join are long enough for several operands per lane
    int join_batch;                  // a batch without classes or tickets in parts: the leaf join's form for those
    int empty_domain;                // some sketch has no points at all
};

// The whole search on a staged scratch, or the same in pieces: one range of tickets at a time, then the rest.
cudaError_t launch_search_part(char* base, const SearchLayout& L, bool join, u64 t_begin, u64 t_end, bool restart, cudaStream_t stream,
                               int* n_launches);
cudaError_t launch_pairs(char* base, const SearchLayout& L, const PairSeg* host_segs, cudaStream_t stream, int* n_launches);
cudaError_t launch_members(char* base, const SearchLayout& L, u64 begin, u64 end, bool restart, cudaStream_t stream, int* n_launches);
cudaError_t launch_search_end(char* base, const SearchLayout& L, bool any_tickets, AccDev* acc_out, bool* told, cudaStream_t stream, int* n_launches);
int search_warps();                                  // warps of the leaf join that run at a time
constexpr size_t kStaticScratchBytes = 1u << 20;     // fixed scratch of the allocation-free entry point
cudaError_t launch_search_static(const void* stage, const SearchLayout& L, u64 n_tickets, u64 n_join, AccDev* acc_out, bool locked, cudaStream_t stream);
cudaError_t launch_int32_peak(int which, u32* out, int blocks, int iters, cudaStream_t stream);

// What the library's other source files may know of a grammar and a loaded sketch (defined in xp_api.cu).
struct SketchInternals { const SketchDev* d_s; const xp_grammar* g; i64 n_points; int device, n_vars; };
SketchInternals sketch_internals(const xp_sketch* s);
u64 grammar_cnt(const xp_grammar* g, int nt, int size);      // trees of nt with exactly `size` nodes
int grammar_nonterminals(const xp_grammar* g);
int grammar_ok_size(const xp_grammar* g);                    // counts are exact (< 2^63) up to this size
// The grammar as the kernels see it (host copy of the tables): leaves and binary productions grouped by nonterminal.
struct GrammarHost { int n_nt, n_vars; const int* leaf_begin; const int* bin_begin; const LeafDev* leaves; const BinDev* bins;
                     const char* const* var_names; };
GrammarHost grammar_host(const xp_grammar* g);
struct HoleSpec { int start_nt, max_size; };
HoleSpec sketch_hole(const xp_sketch* s, int hole);           // hole < 0 or >= n_holes: start_nt = -1
const HoleDev* sketch_hole_dev(const xp_sketch* s, int hole); // device pointer
cudaError_t device_alloc(void** out, size_t bytes, int* device, size_t* granted);     // the library's device pool
void device_release(void* ptr, size_t granted, int device);
xp_status set_error(xp_status st, const char* msg);
// Page-locked host memory and a pair of timing events from the library's pools (given back when the holder goes).
struct StageMemory {
    StageMemory(size_t bytes);
    ~StageMemory();
    char* p;                         // null: out of host memory
    bool locked;                     // page-locked: kernels may write to it
    void* block;
    StageMemory(const StageMemory&) = delete;
    StageMemory& operator=(const StageMemory&) = delete;
};
struct StageEvents {
    StageEvents();
    ~StageEvents();
    cudaError_t open();
    cudaEvent_t e0, e1;
    void* pair;
    StageEvents(const StageEvents&) = delete;
    StageEvents& operator=(const StageEvents&) = delete;
};

}  // namespace xp
