// Host side of libxpiler_repair: grammar tables, sketch encoding, launch planning, result
// decoding and the C ABI declared in include/xp.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <system_error>
#include <thread>
#include <vector>

#include "xp_dev.h"
#include "xp_launch.h"

using namespace xp;

// ------------------------------------------------------------------------------------------
// errors
// ------------------------------------------------------------------------------------------

static thread_local std::string g_last_error;

static xp_status fail(xp_status st, const std::string& msg) {
    g_last_error = msg;
    return st;
}

namespace xp {
xp_status set_error(xp_status st, const char* msg) { return fail(st, msg); }      // for the library's other source files
}

#define XP_CUDA(call)                                                                          \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess)                                                                 \
            return fail(e_ == cudaErrorMemoryAllocation ? XP_ERR_NOMEM : XP_ERR_CUDA,          \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                   \
    } while (0)

// ------------------------------------------------------------------------------------------
// device memory of grammars and sketches
// ------------------------------------------------------------------------------------------
//
// Blocks up to kPoolBigBytes are carved from 64 MiB slabs and, when released, kept in a
// free list by size for the next load (a loop that loads and destroys the same sketch never
// reaches cudaMalloc or cudaFree, whose cost and device-wide synchronisation would otherwise
// dominate small searches).  Larger blocks come from cudaMalloc; released ones are kept too,
// up to kPoolBigKeep bytes in all, and handed out again to a request of the same size.  Slabs
// and kept blocks are returned to the driver when the process ends.  One pool per device.
namespace {
constexpr size_t kPoolSlabBytes = 64ull << 20, kPoolBigBytes = 16ull << 20, kPoolBigKeep = 24ull << 30;
struct DevPool {
    std::multimap<size_t, char*> free_blocks;
    std::multimap<size_t, char*> big_blocks;
    size_t big_kept = 0;
    char* slab = nullptr;
    size_t slab_left = 0;
};
std::mutex g_pool_mu;
std::map<int, DevPool> g_pools;

// *granted receives the size of the block handed out (>= bytes): it is what pool_release must be given.
cudaError_t pool_alloc(void** out, size_t bytes, int* device_out, size_t* granted) {
    const size_t need = ((bytes ? bytes : 1) + 255) & ~(size_t)255;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    *device_out = dev;
    *granted = need;
#ifdef XP_CHECKS
    if (const char* most = getenv("XP_POOL_MOST")) if (need > strtoull(most, nullptr, 10)) return cudaErrorMemoryAllocation;      // (a test's full device)
#endif
    std::lock_guard<std::mutex> lock(g_pool_mu);
    DevPool& p = g_pools[dev];
    // a kept block fits a request when it wastes at most an eighth of itself (sketches of varying
    // sizes then reuse each other's blocks instead of growing the pool without bound)
    auto fits = [&](std::multimap<size_t, char*>& m) {
        auto it = m.lower_bound(need);
        return (it != m.end() && it->first - need <= it->first / 8) ? it : m.end();
    };
    if (need > kPoolBigBytes) {
        auto big = fits(p.big_blocks);
        if (big == p.big_blocks.end()) return cudaMalloc(out, need);
        *out = big->second;
        *granted = big->first;
        p.big_kept -= big->first;
        p.big_blocks.erase(big);
        return cudaSuccess;
    }
    auto it = fits(p.free_blocks);
    if (it != p.free_blocks.end()) { *out = it->second; *granted = it->first; p.free_blocks.erase(it); return cudaSuccess; }
    if (p.slab_left < need) {
        if (p.slab_left >= 256) p.free_blocks.insert({p.slab_left, p.slab});      // the old slab's tail stays usable
        char* slab = nullptr;
        e = cudaMalloc((void**)&slab, kPoolSlabBytes);
        if (e != cudaSuccess) { p.slab = nullptr; p.slab_left = 0; return e; }
        p.slab = slab;
        p.slab_left = kPoolSlabBytes;
    }
    *out = p.slab;
    p.slab += need;
    p.slab_left -= need;
    return cudaSuccess;
}

void pool_release(void* ptr, size_t bytes, int device) {
    if (!ptr) return;
    const size_t need = ((bytes ? bytes : 1) + 255) & ~(size_t)255;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    DevPool& p = g_pools[device];
    if (need > kPoolBigBytes) {
        if (p.big_kept + need > kPoolBigKeep) { cudaFree(ptr); return; }
        p.big_blocks.insert({need, (char*)ptr});
        p.big_kept += need;
        return;
    }
    p.free_blocks.insert({need, (char*)ptr});
}
}  // namespace

struct xp_sketch;
static xp_status check_device(const xp_sketch* const* sk, size_t n);

namespace {
// Page-locked blocks for what a search sends and reads back, and pairs of events that time it: kept from call to
// call in lists that any thread may use (a copy from ordinary memory goes through the driver's staging buffer and
// makes the host wait; creating a pair of events takes longer than recording it).  A block that would take the list past
// kStageKeep bytes is freed when it comes back.
constexpr size_t kStageKeep = 512ull << 20, kStageLeast = 16ull << 10;
struct StagePool {
    std::mutex mu;
    std::multimap<size_t, char*> blocks;
    size_t kept = 0;
};
StagePool g_stage;
struct StageBlock {                   // returned to the pool when it goes out of scope; nothing may be copying then
    char* p = nullptr;
    size_t bytes = 0;
    bool locked = false;
    StageBlock(size_t want) {
        size_t need = kStageLeast;
        while (need < want) need <<= 1;
        {
            std::lock_guard<std::mutex> lock(g_stage.mu);
            auto it = g_stage.blocks.lower_bound(need);
            if (it != g_stage.blocks.end() && it->first <= 4 * need) {
                p = it->second; bytes = it->first; locked = true;
                g_stage.kept -= bytes;
                g_stage.blocks.erase(it);
                return;
            }
        }
        bytes = need;
        void* q = nullptr;
        if (cudaHostAlloc(&q, need, cudaHostAllocPortable) == cudaSuccess) { p = (char*)q; locked = true; return; }
        (void)cudaGetLastError();
        p = (char*)malloc(need);      // (ordinary memory serves too, more slowly)
    }
    ~StageBlock() {
        if (!p) return;
        if (!locked) { free(p); return; }
        std::lock_guard<std::mutex> lock(g_stage.mu);
        if (g_stage.kept + bytes > kStageKeep) { cudaFreeHost(p); return; }
        g_stage.blocks.insert({bytes, p});
        g_stage.kept += bytes;
    }
    StageBlock(const StageBlock&) = delete;
    StageBlock& operator=(const StageBlock&) = delete;
};

struct EventPool { std::mutex mu; std::map<int, std::vector<std::pair<cudaEvent_t, cudaEvent_t>>> free_pairs; };
EventPool g_events;
struct EventPair {                    // events belong to the device that was current when they were made
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int dev = -1;
    cudaError_t open() {
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        {
            std::lock_guard<std::mutex> lock(g_events.mu);
            auto& v = g_events.free_pairs[dev];
            if (!v.empty()) { e0 = v.back().first; e1 = v.back().second; v.pop_back(); return cudaSuccess; }
        }
        if ((e = cudaEventCreate(&e0)) != cudaSuccess) return e;
        return cudaEventCreate(&e1);
    }
    ~EventPair() {
        if (!e0 || !e1) { if (e0) cudaEventDestroy(e0); return; }
        std::lock_guard<std::mutex> lock(g_events.mu);
        auto& v = g_events.free_pairs[dev];
        if (v.size() >= 64) { cudaEventDestroy(e0); cudaEventDestroy(e1); return; }
        v.push_back({e0, e1});
    }
};
}  // namespace

static const char* const kOpText[] = {"+", "-", "*", "/", "%", "<", "<=", "==", "!=", "min", "max", "&&", "||", "<<", ">>"};

// ------------------------------------------------------------------------------------------
// grammar
// ------------------------------------------------------------------------------------------

struct xp_grammar {
    int n_vars = 0, n_nt = 0;
    std::vector<std::string> names;
    std::vector<i64> lo, hi;
    std::vector<LeafDev> leaves;
    std::vector<BinDev> bins;
    std::vector<ConstDev> consts;    // per nonterminal: its constants ascending, then its variables (see GrammarDev::consts)
    int const_begin[kMaxNt + 1] = {0}, var_begin[kMaxNt] = {0};
    int leaf_begin[kMaxNt + 1] = {0};
    int bin_begin[kMaxNt + 1] = {0};
    u64 cnt[kMaxNt][kMaxSize + 1] = {{0}};
    u32 wide_leaf = 0;               // nonterminals with a leaf that may be 2^31 or more in magnitude
    int ok_size = kMaxSize;          // counts are exact (< 2^63) up to this size
    // device copy, made on first use
    GrammarDev* d_g = nullptr;       // one block: header, leaves, binary productions
    size_t d_bytes = 0;
    int d_device = 0;
    bool d_pending = false;          // some load has taken the block and not yet queued the tables (under g_load_mu)
};

// cnt[nt][s] by the recurrence over productions and left sizes; off[s] of a binary production
// is the number of size-s trees of its nonterminal that come before it.  Sizes from the first
// one at which a count reaches 2^63 are marked unusable (ok_size).
static void build_counts(xp_grammar* g) {
    for (int s = 1; s <= kMaxSize; s += 2) {              // (every node has no or two children: no trees of even size)
        bool overflow = g->ok_size < s;
        for (int nt = 0; nt < g->n_nt && !overflow; ++nt) {
            unsigned __int128 total = 0;
            if (s == 1) total = (unsigned)(g->leaf_begin[nt + 1] - g->leaf_begin[nt]);
            unsigned __int128 block = 0;                  // trees of the previous production's operands (most productions share them)
            for (int b = g->bin_begin[nt]; b < g->bin_begin[nt + 1] && !overflow; ++b) {
                BinDev& bd = g->bins[b];
                bd.off[s] = (u64)total;
                if (b == g->bin_begin[nt] || bd.lnt != (&bd)[-1].lnt || bd.rnt != (&bd)[-1].rnt) {
                    block = 0;
                    const u64 *l = g->cnt[bd.lnt], *r = g->cnt[bd.rnt];
                    for (int a = 1; a <= s - 2 && !overflow; a += 2) {
                        block += (unsigned __int128)l[a] * r[s - 1 - a];
                        overflow = (block >> 63) != 0;
                    }
                }
                total += block;
                overflow = overflow || (total >> 63) != 0;
            }
            g->cnt[nt][s] = (u64)total;
        }
        if (overflow) {
            if (g->ok_size >= s) g->ok_size = s - 1;
            for (int nt = 0; nt < g->n_nt; ++nt) g->cnt[nt][s] = 0;
        }
    }
}

static u32 reciprocal(i64 v) {       // (ConstDev::recip)
    const u64 m = v < 0 ? 0ull - (u64)v : (u64)v;
    if (m == 0 || m >> 31) return 0u;
    if (m == 1) return 0xffffffffu;
    const u32 d = (u32)m, q = 0xffffffffu / d;            // (2^32 - 1: one less where d divides 2^32)
    return q + ((d & (d - 1)) == 0 ? 1u : 0u);
}

extern "C" xp_status xp_grammar_create(const xp_grammar_desc* d, xp_grammar** out) {
    if (!d || !out) return fail(XP_ERR_INVALID_ARG, "xp_grammar_create: null argument");
    *out = nullptr;
    if (d->n_vars < 0 || d->n_vars > kMaxVars) return fail(XP_ERR_GRAMMAR, "n_vars out of range");
    if (d->n_nonterminals < 1 || d->n_nonterminals > kMaxNt) return fail(XP_ERR_GRAMMAR, "n_nonterminals out of range");
    if (d->n_productions < 1 || !d->productions) return fail(XP_ERR_GRAMMAR, "no productions");
    if (d->n_vars > 0 && !d->vars) return fail(XP_ERR_GRAMMAR, "vars is null");
    xp_grammar* g = new (std::nothrow) xp_grammar;
    if (!g) return fail(XP_ERR_NOMEM, "out of host memory");
    g->n_vars = d->n_vars;
    g->n_nt = d->n_nonterminals;
    g->names.reserve(d->n_vars); g->lo.reserve(d->n_vars); g->hi.reserve(d->n_vars);
    for (int i = 0; i < d->n_vars; ++i) {
        if (d->vars[i].hi < d->vars[i].lo) { delete g; return fail(XP_ERR_GRAMMAR, "variable range with hi < lo"); }
        if (d->vars[i].name) g->names.emplace_back(d->vars[i].name);
        else g->names.push_back("v" + std::to_string(i));
        g->lo.push_back(d->vars[i].lo);
        g->hi.push_back(d->vars[i].hi);
    }
    size_t n_leaves = 0, n_bins = 0;
    for (int i = 0; i < d->n_productions; ++i) {
        const xp_production& p = d->productions[i];
        bool ok = p.lhs >= 0 && p.lhs < g->n_nt;
        if (p.kind == XP_PROD_VAR) ok = ok && p.var >= 0 && p.var < g->n_vars;
        else if (p.kind == XP_PROD_BIN) ok = ok && ((p.op >= XP_OP_ADD && p.op <= XP_OP_MOD) || p.op == XP_OP_MIN || p.op == XP_OP_MAX || p.op == XP_OP_SHL || p.op == XP_OP_SHR) && p.left >= 0 && p.left < g->n_nt && p.right >= 0 && p.right < g->n_nt;
        else if (p.kind != XP_PROD_CONST) ok = false;
        if (!ok) { delete g; return fail(XP_ERR_GRAMMAR, "production " + std::to_string(i) + " is malformed"); }
        ++(p.kind == XP_PROD_BIN ? n_bins : n_leaves);
    }
    g->leaves.reserve(n_leaves);
    g->consts.reserve(n_leaves);
    g->bins.reserve(n_bins);
    for (int nt = 0; nt < g->n_nt; ++nt) {          // leaves and binaries grouped per nonterminal, order kept
        g->leaf_begin[nt] = (int)g->leaves.size();
        g->bin_begin[nt] = (int)g->bins.size();
        for (int i = 0; i < d->n_productions; ++i) {
            const xp_production& p = d->productions[i];
            if (p.lhs != nt) continue;
            if (p.kind == XP_PROD_BIN) {
                BinDev b;
                memset(&b, 0, sizeof(b));
                b.op = p.op; b.lnt = p.left; b.rnt = p.right;
                g->bins.push_back(b);
            } else {
                LeafDev l;
                l.var = p.kind == XP_PROD_VAR ? p.var : -1;
                l.pad = 0;
                l.value = p.kind == XP_PROD_CONST ? p.value : 0;
                g->leaves.push_back(l);
            }
        }
    }
    g->leaf_begin[g->n_nt] = (int)g->leaves.size();
    g->bin_begin[g->n_nt] = (int)g->bins.size();
    for (int nt = 0; nt < g->n_nt; ++nt) {
        const int lb = g->leaf_begin[nt], le = g->leaf_begin[nt + 1];
        g->const_begin[nt] = (int)g->consts.size();
        for (int i = lb; i < le; ++i) if (g->leaves[i].var < 0) g->consts.push_back(ConstDev{g->leaves[i].value, i - lb, reciprocal(g->leaves[i].value)});
        auto before = [](const ConstDev& a, const ConstDev& b) { return a.value != b.value ? a.value < b.value : a.pos < b.pos; };
        const auto first = g->consts.begin() + g->const_begin[nt];
        if (!std::is_sorted(first, g->consts.end(), before)) std::sort(first, g->consts.end(), before);
        g->var_begin[nt] = (int)g->consts.size();
        for (int i = lb; i < le; ++i) if (g->leaves[i].var >= 0) g->consts.push_back(ConstDev{g->leaves[i].var, i - lb, 0u});
    }
    g->const_begin[g->n_nt] = (int)g->consts.size();
    for (int nt = 0; nt < g->n_nt; ++nt)
        for (int i = g->leaf_begin[nt]; i < g->leaf_begin[nt + 1]; ++i) {
            const LeafDev& l = g->leaves[i];
            const i64 lo = l.var >= 0 ? g->lo[l.var] : l.value, hi = l.var >= 0 ? g->hi[l.var] : l.value + (l.value < 0);
            if (lo <= INT32_MIN || hi > (l.var >= 0 ? 1ll << 31 : (1ll << 31) - 1)) g->wide_leaf |= 1u << nt;
        }
    build_counts(g);
    *out = g;
    return XP_OK;
}

extern "C" void xp_grammar_destroy(xp_grammar* g) {
    if (!g) return;
    pool_release(g->d_g, g->d_bytes, g->d_device);
    delete g;
}

extern "C" xp_status xp_grammar_count(const xp_grammar* g, int32_t nt, int32_t max_size, uint64_t* out) {
    if (!g || !out || nt < 0 || nt >= g->n_nt || max_size < 0 || max_size > kMaxSize)
        return fail(XP_ERR_INVALID_ARG, "xp_grammar_count: bad argument");
    if (max_size > g->ok_size) return fail(XP_ERR_TOO_LARGE, "a candidate count reaches 2^63");
    out[0] = 0;
    for (int s = 1; s <= max_size; ++s) out[s] = g->cnt[nt][s];
    return XP_OK;
}

// rank -> tree, appended to `code` in postfix and to `text` in infix.
static bool host_unrank(const xp_grammar* g, int nt, int size, u64 rank, std::vector<xp_instr>* code, std::string* text) {
    if (size < 1 || size > g->ok_size || rank >= g->cnt[nt][size]) return false;
    if (size == 1) {
        const LeafDev& l = g->leaves[g->leaf_begin[nt] + (int)rank];
        xp_instr in;
        in.kind = l.var >= 0 ? XP_I_VAR : XP_I_CONST;
        in.arg = l.var >= 0 ? l.var : 0;
        in.value = l.value;
        code->push_back(in);
        *text += l.var >= 0 ? g->names[l.var] : std::to_string((long long)l.value);
        return true;
    }
    int p = g->bin_begin[nt];
    const int pe = g->bin_begin[nt + 1];
    while (p + 1 < pe && g->bins[p + 1].off[size] <= rank) ++p;
    const BinDev& b = g->bins[p];
    u64 rem = rank - b.off[size];
    for (int a = 1; a <= size - 2; ++a) {
        const u64 cr = g->cnt[b.rnt][size - 1 - a];
        const u64 block = g->cnt[b.lnt][a] * cr;
        if (rem >= block) { rem -= block; continue; }
        const bool call = b.op == XP_OP_MIN || b.op == XP_OP_MAX;      // printed min(l,r) / max(l,r)
        *text += call ? std::string(kOpText[b.op]) + "(" : std::string("(");
        if (!host_unrank(g, b.lnt, a, rem / cr, code, text)) return false;
        *text += call ? "," : kOpText[b.op];
        if (!host_unrank(g, b.rnt, size - 1 - a, rem % cr, code, text)) return false;
        *text += ")";
        xp_instr in;
        in.kind = XP_I_OP; in.arg = b.op; in.value = 0;
        code->push_back(in);
        return true;
    }
    return false;
}

extern "C" xp_status xp_grammar_unrank(const xp_grammar* g, int32_t nt, int32_t size, uint64_t rank,
                                       xp_instr* code, int32_t code_cap, char* text, size_t text_cap) {
    if (!g || nt < 0 || nt >= g->n_nt || size < 1 || size > kMaxSize)
        return fail(XP_ERR_INVALID_ARG, "xp_grammar_unrank: bad argument");
    std::vector<xp_instr> c;
    std::string t;
    if (!host_unrank(g, nt, size, rank, &c, &t)) return fail(XP_ERR_INVALID_ARG, "xp_grammar_unrank: rank out of range");
    if (code) {
        if (code_cap < (int)c.size()) return fail(XP_ERR_INVALID_ARG, "xp_grammar_unrank: code buffer too small");
        memcpy(code, c.data(), c.size() * sizeof(xp_instr));
    }
    if (text) {
        if (text_cap < t.size() + 1) return fail(XP_ERR_INVALID_ARG, "xp_grammar_unrank: text buffer too small");
        memcpy(text, t.c_str(), t.size() + 1);
    }
    return XP_OK;
}

// Layout of a grammar's tables in one device block: header | leaves | binary productions | constants.
struct GrammarLayout { size_t leaves, bins, consts, total; };
static GrammarLayout grammar_layout(const xp_grammar* g) {
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    GrammarLayout l;
    l.leaves = al(sizeof(GrammarDev));
    l.bins = l.leaves + al(sizeof(LeafDev) * g->leaves.size());
    l.consts = l.bins + al(sizeof(BinDev) * g->bins.size());
    l.total = l.consts + al(sizeof(ConstDev) * g->consts.size());
    return l;
}

// The tables as they go to the device block at g->d_g.
static void grammar_image(const xp_grammar* g, char* out) {
    const GrammarLayout l = grammar_layout(g);
    GrammarDev& h = *(GrammarDev*)out;
    memset(&h, 0, sizeof(h));
    h.n_vars = g->n_vars; h.n_nt = g->n_nt;
    h.n_leaves = (int)g->leaves.size(); h.n_bins = (int)g->bins.size();
    memcpy(h.leaf_begin, g->leaf_begin, sizeof(h.leaf_begin));
    memcpy(h.bin_begin, g->bin_begin, sizeof(h.bin_begin));
    memcpy(h.cnt, g->cnt, sizeof(h.cnt));
    memcpy(h.const_begin, g->const_begin, sizeof(h.const_begin));
    memcpy(h.var_begin, g->var_begin, sizeof(h.var_begin));
    const char* block = (const char*)g->d_g;
    h.leaves = (const LeafDev*)(block + l.leaves);
    h.bins = (const BinDev*)(block + l.bins);
    h.consts = (const ConstDev*)(block + l.consts);
    if (!g->leaves.empty()) memcpy(out + l.leaves, g->leaves.data(), sizeof(LeafDev) * g->leaves.size());
    if (!g->bins.empty()) memcpy(out + l.bins, g->bins.data(), sizeof(BinDev) * g->bins.size());
    if (!g->consts.empty()) memcpy(out + l.consts, g->consts.data(), sizeof(ConstDev) * g->consts.size());
}

// Device memory for a grammar's tables, on first use; *fresh: the caller has to send the image.
// (Under g_load_mu; a grammar whose block another load has taken and not yet filled is waited for before.)
static xp_status grammar_block(xp_grammar* g, bool* fresh) {
    *fresh = false;
    if (g->d_g) {
        // the device copy was made on the device that was current at the first load and serves that device only
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess || dev != g->d_device)
            return fail(XP_ERR_INVALID_ARG, "the grammar's tables live on device " + std::to_string(g->d_device) +
                        ", the current device is " + std::to_string(dev) + ": use one grammar handle per device");
        return XP_OK;
    }
    char* block = nullptr;
    XP_CUDA(pool_alloc((void**)&block, grammar_layout(g).total, &g->d_device, &g->d_bytes));
    g->d_g = (GrammarDev*)block;
    *fresh = true;
    return XP_OK;
}

// ------------------------------------------------------------------------------------------
// sketch
// ------------------------------------------------------------------------------------------

struct HoleHost {
    int start_nt = 0, max_size = 0;
    bool filter_ok = false;          // the probe filter applies (probe 0 exists, context affine or a comparison there, subtree tables)
    bool never = false;              // the spec is undefined at some point: no candidate can match
    bool exact = false;              // the leaf join's conditions do not apply (a context factor of 0, or with more than 31 zero bits at its end)
    bool join_on = false;            // the context is affine, and they do
    bool target_zero = false;        // the hole value wanted is zero at one of the join's two probes
    int tab_max = 0;                 // subtrees up to this size are tabulated
    bool compares = false;           // the filter works on an interval of hole values (the context compares)
    bool second = false;             // filter hits are looked at once more at probe 1 from the start (hits are frequent)
    int cls_size = 0;                // operands of this size are in classes, cls_n of each nonterminal (0: none)
    u32 cls_n[kMaxNt] = {0};
    double pass_rate = 0;            // share of the load's sampled candidates that satisfied every probe with tables
    // What the load makes classes of: the size, and for which contexts (0: none); a grammar's subtrees of that size.
    int cls_top = 0, cls_want = 0;
    u64 cls_entries = 0;
    u32 cls_blocks = 0;              // blocks of the kernels that make them
};

struct Plan {
    std::vector<SegDev> segs;
    std::vector<JoinSeg> jsegs;
    std::vector<JoinGroup> jgroups;
    std::vector<PairSeg> psegs;
    std::vector<AccDev> acc;
    std::vector<u64> nominal_ops;    // per accumulator: cost-model operations of the filter stage
    u64 n_tickets = 0, n_join = 0;
    bool join_wide = false;
    bool whole = false;              // comparing contexts: every operator in one segment, whatever their number (the fewest bytes)          // several operands per lane and step
};

struct xp_sketch {
    xp_grammar* g = nullptr;
    int n_holes = 0;
    i64 n_points = 0;
    std::vector<HoleHost> holes;
    SketchDev* d_s = nullptr;
    HoleDev* d_holes = nullptr;
    // Device memory of the sketch: one block laid out at load for everything (sketch and hole
    // records, copies of host tables, staged points and specs, subtree-value tables).
    char* arena = nullptr;
    size_t arena_bytes = 0, arena_used = 0;
    int arena_device = 0;
    size_t load_h2d = 0, load_d2h = 0;               // bytes the load moved
    std::vector<int> n_probes;                       // per hole, as the load (or the last refinement) left them
    int n_refined = 0;                               // points promoted to probes by xp_sketch_refine
    std::vector<size_t> off_kill;                    // per hole: offset of its table of whole-domain failures in the arena
    size_t off_holes = 0;
    int tab_size_cap = 0, tab_probes_cap = 0;        // most sizes / probes that the subtree tables of a hole cover
    u64 entries_at[kMaxSize + 1] = {0};              // subtree-table entries per size (all nonterminals)
    // The sketch's part of a launch plan under default options (every size, no rank window, no flag), as
    // if it were the only sketch of the call: built on the first such call and copied, with ticket, sketch
    // and accumulator numbers shifted, into the plan of every later one (a batch of thousands of small
    // sketches would otherwise spend longer planning than some of its searches take).
    // One per form (PlanForm): each is built once, under the lock, and only read from then on
    // (calls on several threads copy them at the same time); a refinement, during which no search may run, drops them.
    mutable std::mutex plan_mu;
    mutable std::unique_ptr<const Plan> plan_kept[35];     // per form and for which holes classes are left out (ClassUse)
};

// What the load's kernels settled for a hole.
static void hole_decided(HoleHost* h, const LoadOut& o) {
    // the filter applies where the context at probe 0 is affine in the hole, or a comparison
    h->filter_ok = o.filter_ok != 0 && o.tab_probes > 0;
    h->compares = o.filter_ok != 0 && o.aff_ok == 0;
    h->exact = o.aff_ok != 0 && o.join_on == 0;
    h->join_on = o.aff_ok != 0 && o.join_on != 0;
    h->target_zero = o.target_zero != 0;
    h->tab_max = o.tab_max;
    h->second = o.second != 0;
    h->cls_size = o.cls_size;
    memcpy(h->cls_n, o.cls_n, sizeof(h->cls_n));
    h->pass_rate = o.sample_n > 0 ? (double)o.sample_pass / (double)o.sample_n : 0.0;
    if (o.spec_bad) h->never = true;                      // the spec is undefined at some point
}

// Checks a postfix expression; returns false when malformed or too deep.
static bool check_code(const xp_instr* code, int n, int n_vars, bool hole_allowed) {
    if (n < 0 || n > kMaxCode || (n > 0 && !code)) return false;
    int sp = 0;
    for (int i = 0; i < n; ++i) {
        const xp_instr& c = code[i];
        if (c.kind == XP_I_OP) {
            if (c.arg < XP_OP_ADD || c.arg > XP_OP_SHR || sp < 2) return false;
            --sp;
        } else {
            if (c.kind == XP_I_VAR) { if (c.arg < 0 || c.arg >= n_vars) return false; }
            else if (c.kind == XP_I_HOLE) { if (!hole_allowed) return false; }
            else if (c.kind != XP_I_CONST) return false;
            if (++sp > kMaxStack) return false;
        }
    }
    return n == 0 || sp == 1;
}

static u64 mix64(u64 x) {            // SplitMix64 finaliser: spreads sample ids over the domain
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

extern "C" void xp_sketch_destroy(xp_sketch* s) {
    if (!s) return;
    pool_release(s->arena, s->arena_bytes, s->arena_device);
    delete s;
}

// Entries of the subtree-value tables of a hole with size bound max_size: sizes 1, 2, ... while
// every nonterminal has at most kTabMaxEntries trees of that size; apart from the leaves never the sizes
// that only occur as whole candidates (operands have at most max_size - 2 nodes).
static u64 table_entries(const xp_grammar* g, int max_size, u64 (*off)[kMaxSize + 1], int* tmax_out) {
    u64 total = 0;
    int tmax = 0;
    for (int k = 1; k == 1 || k <= max_size - 2; ++k) {
        bool fits = true;
        for (int nt = 0; nt < g->n_nt; ++nt) fits = fits && g->cnt[nt][k] <= kTabMaxEntries;
        if (!fits) break;
        for (int nt = 0; nt < g->n_nt; ++nt) { if (off) off[nt][k] = total; total += g->cnt[nt][k]; }
        tmax = k;
    }
    if (tmax_out) *tmax_out = tmax;
    return total;
}

// Is a hole's search made of enough combinations of its largest tabulated subtrees that they are put into classes first?  Where an
// operand of the search is itself above the tables, each of them is met at least a hundred times; where the context compares, an
// operand costs some ten thousand instructions against some hundred here.  Otherwise every operand is met once, and would be here too.
constexpr u64 kClassLeast = 4096;            // subtrees from which it pays
constexpr u64 kRangeMost = 1ull << 18;       // operands of a hole whose context compares from which the tiles take a leaf at the root too
static void class_plan(const xp_grammar* g, const xp_hole_desc& hd, HoleHost* h) {
    int tmax = 0, top = 0, need = 0;
    (void)table_entries(g, hd.max_size, nullptr, &tmax);
    for (int nt = 0; nt < g->n_nt; ++nt)
        for (int k = 1; k <= hd.max_size - 2; ++k)
            if (g->cnt[nt][k] > 0) { need = k > need ? k : need; if (k <= tmax) top = k > top ? k : top; }
    if (top < 3) return;
    u64 all = 0, blocks = 0;
    for (int nt = 0; nt < g->n_nt; ++nt) { all += g->cnt[nt][top]; blocks += (g->cnt[nt][top] + kClassThreads - 1) / kClassThreads; }
    if (all < kClassLeast) return;
    bool compares = false;
    for (int i = 0; i < hd.ctx_len; ++i) compares = compares || (hd.ctx[i].kind == XP_I_OP && (hd.ctx[i].arg == XP_OP_LT || hd.ctx[i].arg == XP_OP_LE));
    compares = compares && g->cnt[hd.start_nt][top] <= kRangeMost;       // (with more, such a context's operands go as tiles)
    h->cls_want = (need > top ? kClassAffine : 0) | (compares ? kClassCompare : 0);
    if (h->cls_want) { h->cls_top = top; h->cls_entries = all; h->cls_blocks = (u32)blocks; }
}

// One sketch on its way through a load: everything between its description and the moment the
// load's kernels have run.
struct LoadState {
    xp_sketch* s = nullptr;
    const xp_sketch_desc* d = nullptr;
    struct Hole {                            // what begin settles per hole; the record itself is made in its place in the staged copy
        size_t off_spec = 0;                 // its spec values in the device block (0: none there)
        size_t off_tabv = 0, off_tabk = 0, off_tabm = 0, off_pair = 0, off_sets = 0, off_cls = 0;
        u64 entries = 0;
        int probes = 0;
    };
    std::vector<Hole> hole;
    size_t off_coords = 0, head = 0;         // [0, head) of the block is staged on the host
    bool copy_coords = false, stage = false, stage_box = false;
    bool grammar_fresh = false;              // this sketch's load sends its grammar's tables
    i64 n_points = 0;
    size_t grammar_bytes = 0;
    size_t stage_at = 0;                     // where its part of the staged copy starts (head, then the grammar's tables)
    size_t piece = 0;
};
constexpr size_t kPackMax = 256u << 10;      // host tables up to this size travel in the staged copy
static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

// Which variables can decide whether a hole value satisfies the constraint?  Where the context is an affine map of the
// hole, A h + B = spec, it is those of A and of D = spec - B, taken as polynomials over the variables (coefficients modulo
// 2^64, so + - * are exact) with every other subexpression as an atom of its own: terms that both sides share cancel
// (c * 3136 + HOLE * 56 + col against c * 3136 + row * 56 + col leaves the variables of row).  On a box the whole-domain
// check then runs over those and the candidate's own variables only.  Subexpressions that may be undefined keep theirs.
namespace {
struct Poly { std::map<std::vector<int>, u64> t; };       // monomial (sorted atoms) -> coefficient, none zero
struct PolyAtoms { std::map<std::string, int> ids; std::vector<u32> vars; u32 may_fail = 0; };
constexpr size_t kPolyTerms = 64;

void poly_add(Poly& a, const Poly& b, u64 f) {
    for (const auto& m : b.t) {
        const u64 c = (a.t[m.first] += f * m.second);
        if (c == 0) a.t.erase(m.first);
    }
}
bool poly_mul(const Poly& a, const Poly& b, Poly& out) {
    out.t.clear();
    for (const auto& x : a.t)
        for (const auto& y : b.t) {
            std::vector<int> m(x.first);
            m.insert(m.end(), y.first.begin(), y.first.end());
            if (m.size() > 8) return false;
            std::sort(m.begin(), m.end());
            const u64 c = (out.t[m] += x.second * y.second);
            if (c == 0) out.t.erase(m);
            if (out.t.size() > kPolyTerms) return false;
        }
    return true;
}
std::string poly_key(const Poly& p) {
    std::string s;
    for (const auto& m : p.t) {
        s += std::to_string(m.second) + ":";
        for (int a : m.first) s += std::to_string(a) + ",";
        s += ";";
    }
    return s;
}
u32 poly_vars(const Poly& p, const PolyAtoms& atoms) {
    u32 v = 0;
    for (const auto& m : p.t) for (int a : m.first) v |= atoms.vars[a];
    return v;
}
// code = A h + B; false when it is not of that form (or too large to follow).
bool poly_affine(const xp_instr* code, int n, PolyAtoms& atoms, Poly& A, Poly& B) {
    struct E { Poly a, b; };
    std::vector<E> st;
    for (int i = 0; i < n; ++i) {
        const xp_instr& c = code[i];
        if (c.kind != XP_I_OP) {
            E e;
            if (c.kind == XP_I_HOLE) e.a.t[{}] = 1;
            else if (c.kind == XP_I_VAR) e.b.t[{c.arg}] = 1;
            else if (c.value != 0) e.b.t[{}] = (u64)c.value;
            st.push_back(std::move(e));
            continue;
        }
        E y = std::move(st.back()); st.pop_back();
        E x = std::move(st.back()); st.pop_back();
        E r;
        if (c.arg == XP_OP_ADD || c.arg == XP_OP_SUB) {
            const u64 f = c.arg == XP_OP_ADD ? 1ull : ~0ull;
            r = std::move(x);
            poly_add(r.a, y.a, f); poly_add(r.b, y.b, f);
            if (r.a.t.size() > kPolyTerms || r.b.t.size() > kPolyTerms) return false;
        } else if (c.arg == XP_OP_MUL) {
            if (!x.a.t.empty() && !y.a.t.empty()) return false;
            const Poly& h = x.a.t.empty() ? y.a : x.a;
            const Poly& k = x.a.t.empty() ? x.b : y.b;
            if (!poly_mul(h, k, r.a) || !poly_mul(x.b, y.b, r.b)) return false;
        } else {
            if (!x.a.t.empty() || !y.a.t.empty()) return false;      // (the hole under another operator)
            const u32 v = poly_vars(x.b, atoms) | poly_vars(y.b, atoms);
            const std::string key = std::to_string(c.arg) + "(" + poly_key(x.b) + "|" + poly_key(y.b) + ")";
            auto it = atoms.ids.find(key);
            if (it == atoms.ids.end()) { it = atoms.ids.insert({key, (int)atoms.vars.size()}).first; atoms.vars.push_back(v); }
            const bool divides = c.arg == XP_OP_DIV || c.arg == XP_OP_MOD, shifts = c.arg == XP_OP_SHL || c.arg == XP_OP_SHR;
            const bool constant = y.b.t.empty() || (y.b.t.size() == 1 && y.b.t.begin()->first.empty());
            const u64 value = y.b.t.empty() || !constant ? 0ull : y.b.t.begin()->second;
            if ((divides && (!constant || value == 0)) || (shifts && (!constant || value > 63))) atoms.may_fail |= v;
            r.b.t[{it->second}] = 1;
        }
        st.push_back(std::move(r));
    }
    A = std::move(st.back().a); B = std::move(st.back().b);
    return true;
}
}  // namespace

// Variables that the constraint of a hole with a spec expression depends on beside the hole's value (bits).  Below
// kPolyPoints points the check is short whatever the variables, and the algebra would cost the load more than it saves.
constexpr i64 kPolyPoints = 1 << 15;
static u32 constraint_vars(const xp_hole_desc& hd, int n_vars, i64 n_points) {
    u32 fv = 0;
    for (int i = 0; i < hd.ctx_len; ++i) if (hd.ctx[i].kind == XP_I_VAR) fv |= 1u << hd.ctx[i].arg;
    for (int i = 0; i < hd.spec_len; ++i) if (hd.spec_expr[i].kind == XP_I_VAR) fv |= 1u << hd.spec_expr[i].arg;
    if (hd.ctx_len == 0 || n_points < kPolyPoints) return fv;
    PolyAtoms atoms;
    for (int v = 0; v < n_vars; ++v) atoms.vars.push_back(1u << v);
    Poly A, B, none, D;
    if (!poly_affine(hd.ctx, hd.ctx_len, atoms, A, B) || A.t.empty()) return fv;
    if (!poly_affine(hd.spec_expr, hd.spec_len, atoms, none, D)) return fv;
    poly_add(D, B, ~0ull);
    return fv & (poly_vars(A, atoms) | poly_vars(D, atoms) | atoms.may_fail);
}

// First part of a load: checks the description.
static xp_status load_check(const xp_grammar* g, const xp_sketch_desc* d, LoadState* L) {
    if (!g || !d) return fail(XP_ERR_INVALID_ARG, "xp_sketch_load: null argument");
    if (d->n_holes < 1 || !d->holes) return fail(XP_ERR_SKETCH, "a sketch needs at least one hole");
    if (d->domain_kind != XP_DOMAIN_BOX && d->domain_kind != XP_DOMAIN_TABLE) return fail(XP_ERR_SKETCH, "bad domain_kind");
    const int nv = g->n_vars;
    i64 n_points = 0;
    if (d->domain_kind == XP_DOMAIN_BOX) {
        unsigned __int128 n = 1;
        for (int v = 0; v < nv; ++v) {
            n *= (unsigned __int128)(u64)(g->hi[v] - g->lo[v]);
            if (n >> 62) return fail(XP_ERR_TOO_LARGE, "box domain has 2^62 points or more");
        }
        n_points = (i64)n;
    } else {
        if (d->n_points < 0 || (d->n_points > 0 && !d->coords)) return fail(XP_ERR_SKETCH, "table domain without coords");
        n_points = d->n_points;
    }
    for (int h = 0; h < d->n_holes; ++h) {
        const xp_hole_desc& hd = d->holes[h];
        if (hd.start_nt < 0 || hd.start_nt >= g->n_nt) return fail(XP_ERR_SKETCH, "hole start_nt out of range");
        if (hd.max_size < 1 || hd.max_size > kMaxSize) return fail(XP_ERR_SKETCH, "hole max_size out of range");
        if (hd.max_size > g->ok_size) return fail(XP_ERR_TOO_LARGE, "a candidate count reaches 2^63 within the size bound");
        if (!check_code(hd.ctx, hd.ctx_len, nv, true)) return fail(XP_ERR_SKETCH, "malformed context expression");
        if (hd.spec_kind == XP_SPEC_EXPR) {
            if (hd.spec_len < 1 || !check_code(hd.spec_expr, hd.spec_len, nv, false)) return fail(XP_ERR_SKETCH, "malformed spec expression");
        } else if (hd.spec_kind == XP_SPEC_TABLE) {
            if (n_points > 0 && !hd.spec_table) return fail(XP_ERR_SKETCH, "spec table is null");
        } else return fail(XP_ERR_SKETCH, "bad spec_kind");
    }
    L->n_points = n_points;
    return XP_OK;
}

// Second part: lays out and allocates the sketch's device block.
static xp_status load_begin(const xp_grammar* gc, const xp_sketch_desc* d, LoadState* L) {
    xp_grammar* g = const_cast<xp_grammar*>(gc);
    const int nv = g->n_vars;
    const i64 n_points = L->n_points;
    xp_sketch* s = new (std::nothrow) xp_sketch;
    if (!s) return fail(XP_ERR_NOMEM, "out of host memory");
    s->g = g; s->n_holes = d->n_holes; s->n_points = n_points;
    // One device block for the whole sketch, laid out here before anything runs: first what the
    // host provides (sketch, holes, small tables: part of the load's staged copy), then what the load's
    // kernels produce (staged points and specs, subtree tables).
    const int nh = d->n_holes;
    const size_t np = (size_t)n_points, row = (size_t)(nv ? nv : 1);
    bool i32_ok = true;
    for (int v = 0; v < nv; ++v) i32_ok = i32_ok && g->lo[v] >= INT32_MIN && g->hi[v] <= (i64)INT32_MAX + 1;
    L->stage = n_points > 0 && (u64)n_points <= kStageMaxPoints;
    L->stage_box = d->domain_kind == XP_DOMAIN_BOX && L->stage && i32_ok && nv > 0;
    L->copy_coords = d->domain_kind == XP_DOMAIN_TABLE && np > 0 && !d->coords_on_device;
    const size_t coords_bytes = sizeof(i32) * np * row, spec_bytes = sizeof(i64) * np;
    size_t off = 0;
    const size_t off_sketch = off;  off += al256(sizeof(SketchDev));
    const size_t off_holes = off;   off += al256(sizeof(HoleDev) * nh);
    L->hole.resize(nh);
    s->holes.resize(nh);
    if (L->copy_coords && coords_bytes <= kPackMax) { L->off_coords = off; off += al256(coords_bytes); }
    for (int h = 0; h < nh; ++h)
        if (d->holes[h].spec_kind == XP_SPEC_TABLE && np > 0 && !d->holes[h].spec_table_on_device && spec_bytes <= kPackMax) {
            L->hole[h].off_spec = off; off += al256(spec_bytes);
        }
    s->off_kill.assign(nh, 0);
    for (int h = 0; h < nh; ++h) { s->off_kill[h] = off; off += al256((sizeof(i64) + sizeof(u32)) * kKillSlots); }
    L->head = off;                                        // [0, head): staged on the host
    if ((L->copy_coords && coords_bytes > kPackMax) || L->stage_box) { L->off_coords = off; off += al256(coords_bytes); }
    for (int h = 0; h < nh; ++h) {
        const xp_hole_desc& hd = d->holes[h];
        LoadState::Hole& o = L->hole[h];
        if (np > 0 && o.off_spec == 0 &&
            ((hd.spec_kind == XP_SPEC_TABLE && !hd.spec_table_on_device) || (hd.spec_kind == XP_SPEC_EXPR && L->stage))) {
            o.off_spec = off; off += al256(spec_bytes);
        }
        int size_cap = 0;
        const u64 entries = table_entries(g, hd.max_size, nullptr, &size_cap);
        u64 probes = kMaxProbe;
        while (probes > 1 && entries * 9 * probes > kTabBudgetBytes) --probes;
        o.entries = entries;
        o.probes = entries > 0 ? (int)probes : 0;
        if (entries > 0) {
            o.off_tabv = off; off += al256(sizeof(i64) * entries * probes);
            o.off_tabk = off; off += al256(entries * probes);
            o.off_tabm = off; off += al256(entries);
            o.off_pair = off; off += al256(2 * sizeof(i32) * entries);
        }
        class_plan(g, hd, &s->holes[h]);
        o.off_sets = off; off += al256(sizeof(JoinSet) * (size_t)g->n_nt);
        if (size_cap > s->tab_size_cap) s->tab_size_cap = size_cap;
        if (o.probes > s->tab_probes_cap) s->tab_probes_cap = o.probes;
    }
    const size_t plain = off;                             // the classes come last: where memory is short the sketch does without
    for (int h = 0; h < nh; ++h)
        if (const size_t c = s->holes[h].cls_entries) { L->hole[h].off_cls = off; off += al256(8 * c) + al256(4 * (c + kMaxNt + 1)) + al256(4 * c); }
    size_t arena_granted = 0;
    cudaError_t got = pool_alloc((void**)&s->arena, off, &s->arena_device, &arena_granted);
    if (got != cudaSuccess && off > plain) {
        (void)cudaGetLastError();
        off = plain;
        for (int h = 0; h < nh; ++h) { L->hole[h].off_cls = 0; s->holes[h].cls_entries = 0; }
        got = pool_alloc((void**)&s->arena, off, &s->arena_device, &arena_granted);
    }
    if (got != cudaSuccess) {
        (void)cudaGetLastError();
        delete s;
        return fail(XP_ERR_NOMEM, "device memory for the sketch (" + std::to_string(off) + " bytes)");
    }
    s->arena_bytes = arena_granted;
    s->arena_used = off;
    char* base = s->arena;
    s->d_s = (SketchDev*)(base + off_sketch);
    s->d_holes = (HoleDev*)(base + off_holes);
    s->off_holes = off_holes;
    for (int h = 0; h < nh; ++h) { s->holes[h].start_nt = d->holes[h].start_nt; s->holes[h].max_size = d->holes[h].max_size; }
    for (int k = 1; k <= s->tab_size_cap; ++k)
        for (int nt = 0; nt < g->n_nt; ++nt) s->entries_at[k] += g->cnt[nt][k];
    L->s = s;
    L->d = d;
    return XP_OK;
}

// A hole's record.
static void hole_image(const LoadState* L, int h, HoleDev* out) {
    const xp_sketch* s = L->s;
    const xp_grammar* g = s->g;
    const xp_hole_desc& hd = L->d->holes[h];
    const LoadState::Hole& at = L->hole[h];
    char* base = s->arena;
    HoleDev& o = *out;
    memset(&o, 0, sizeof(o));
    table_entries(g, hd.max_size, o.tab_off, &o.tab_size_cap);
    o.tab_total = at.entries;
    o.tab_probes_cap = at.probes;
    u64 c = 0;
    for (int k = 1; k <= hd.max_size; ++k) c += g->cnt[hd.start_nt][k];
    o.small_search = c <= 100000000ull ? 1 : 0;
    o.start_nt = hd.start_nt; o.max_size = hd.max_size; o.ctx_len = hd.ctx_len;
    if (hd.ctx_len) memcpy(o.ctx, hd.ctx, sizeof(xp_instr) * hd.ctx_len);
    if (hd.spec_kind == XP_SPEC_EXPR) {
        o.spec_len = hd.spec_len;
        memcpy(o.spec, hd.spec_expr, sizeof(xp_instr) * hd.spec_len);
        if (at.off_spec) o.spec_table = (const i64*)(base + at.off_spec);       // staged by the load, before anything reads it
    } else if (s->n_points > 0) {
        o.spec_table = hd.spec_table_on_device ? (const i64*)hd.spec_table : (const i64*)(base + at.off_spec);
    }
    if (at.entries > 0) {
        o.tab_val = (i64*)(base + at.off_tabv);
        o.tab_ok = (unsigned char*)(base + at.off_tabk);
        o.tab_vars = (unsigned char*)(base + at.off_tabm);
        o.tab_pair = (i32*)(base + at.off_pair);
    }
    if (at.off_cls) {
        const HoleHost& hh = s->holes[h];
        const size_t c = hh.cls_entries;
        o.cls_top = hh.cls_top; o.cls_want = hh.cls_want;
        o.cls_pair = (int2*)(base + at.off_cls);
        o.cls_start = (u32*)(base + at.off_cls + al256(8 * c));
        o.cls_mem = (u32*)(base + at.off_cls + al256(8 * c) + al256(4 * (c + kMaxNt + 1)));
    }
    o.join_sets = (JoinSet*)(base + at.off_sets);
    // variables that decide beside the candidate's own (a caller's spec table may depend on all)
    o.fixed_vars = hd.spec_kind != XP_SPEC_EXPR ? 0xffffffffu : constraint_vars(hd, g->n_vars, s->n_points);
    o.kill_pid = (i64*)(base + s->off_kill[h]);
    o.kill_cnt = (u32*)(base + s->off_kill[h] + sizeof(i64) * kKillSlots);
}

// The sketch's record.
static void sketch_image(const LoadState* L, SketchDev* out) {
    const xp_sketch* s = L->s;
    const xp_grammar* g = s->g;
    const xp_sketch_desc* d = L->d;
    const int nv = g->n_vars;
    const i64 n_points = s->n_points;
    char* base = s->arena;
    SketchDev& hs = *out;
    memset(&hs, 0, sizeof(hs));
    hs.g = g->d_g; hs.n_vars = nv; hs.n_holes = s->n_holes; hs.domain_kind = d->domain_kind; hs.n_points = n_points;
    hs.holes = s->d_holes;
    for (int v = 0; v < nv; ++v) {
        hs.lo[v] = g->lo[v]; hs.ext[v] = g->hi[v] - g->lo[v];
        const bool table = d->domain_kind == XP_DOMAIN_TABLE;      // a table's bounds are reduced over its rows by the load
        hs.vmin[v] = table ? LLONG_MAX : g->lo[v];
        hs.vmax[v] = table ? LLONG_MIN : g->hi[v] - 1;
    }
    if (d->domain_kind == XP_DOMAIN_TABLE && n_points > 0) hs.coords = d->coords_on_device ? d->coords : (const i32*)(base + L->off_coords);
    if (L->stage_box) { hs.coords = (const i32*)(base + L->off_coords); hs.project = 1; }
    // Sample points the probes are chosen from: box corners first (they expose bound and
    // padding mistakes), then ids spread over the domain by a fixed hash.
    int ns = 0;
    unsigned char slot[4 * kProbeSamples] = {0};          // which ids are there: open addressing, number of the sample plus one
    auto add = [&](i64 id) {
        unsigned at = (unsigned)(mix64((u64)id) >> 32) % (4 * kProbeSamples);
        for (; slot[at]; at = (at + 1) % (4 * kProbeSamples)) if (hs.sample_id[slot[at] - 1] == id) return;
        hs.sample_id[ns++] = id;
        slot[at] = (unsigned char)ns;
    };
    static_assert(kProbeSamples < 256, "a sample's number fits a byte");
    if (n_points > 0) {
        if (d->domain_kind == XP_DOMAIN_BOX) {
            const int ncorner = 1 << (nv < 5 ? nv : 5);
            for (int m = 0; m < ncorner && ns < kProbeSamples / 2; ++m) {
                i64 id = 0;
                for (int v = 0; v < nv; ++v) {
                    const i64 ext = hs.ext[v];
                    const i64 c = (v < 5 && ((m >> v) & 1)) ? ext - 1 : 0;
                    id = id * ext + c;
                }
                add(id);
            }
        } else {
            for (i64 id = 0; id < n_points && ns < 4; ++id) add(id);
        }
        for (u64 k = 0; ns < kProbeSamples && k < 4 * kProbeSamples; ++k) {
            add((i64)(mix64(k) % (u64)n_points));
        }
    }
    hs.n_samples = ns;
}

// Third part: the sketch's share of the staged copy (its head, then its grammar's tables when they are new).
static void load_fill(const LoadState* L, char* stg) {
    const xp_sketch* s = L->s;
    const xp_sketch_desc* d = L->d;
    const int nh = s->n_holes;
    const size_t np = (size_t)s->n_points, row = (size_t)(s->g->n_vars ? s->g->n_vars : 1);
    const size_t coords_bytes = sizeof(i32) * np * row, spec_bytes = sizeof(i64) * np;
    sketch_image(L, (SketchDev*)stg);
    for (int h = 0; h < nh; ++h) hole_image(L, h, (HoleDev*)(stg + s->off_holes) + h);
    if (L->copy_coords && coords_bytes <= kPackMax) memcpy(stg + L->off_coords, d->coords, coords_bytes);
    for (int h = 0; h < nh; ++h) {
        const xp_hole_desc& hd = d->holes[h];
        if (hd.spec_kind == XP_SPEC_TABLE && np > 0 && !hd.spec_table_on_device && spec_bytes <= kPackMax)
            memcpy(stg + L->hole[h].off_spec, hd.spec_table, spec_bytes);
        memset(stg + s->off_kill[h], 0xff, sizeof(i64) * kKillSlots);           // no point noted yet (ids -1, counts 0)
        memset(stg + s->off_kill[h] + sizeof(i64) * kKillSlots, 0, sizeof(u32) * kKillSlots);
    }
    if (L->grammar_fresh) grammar_image(s->g, stg + L->head);
}

// The launches that make subtree tables: sizes 1 and 3 together, then one after the other (even sizes have no trees).
static cudaError_t make_tables(const LoadJob* jobs, int n_jobs, int size_cap, int probes_cap, const u64* entries_at) {
    if (size_cap < 1) return cudaSuccess;
    cudaError_t e = launch_subvalues(jobs, n_jobs, 1, 3, probes_cap, entries_at[1] + (size_cap >= 3 ? entries_at[3] : 0), nullptr);
    for (int k = 5; k <= size_cap && e == cudaSuccess; k += 2) e = launch_subvalues(jobs, n_jobs, k, k, probes_cap, entries_at[k], nullptr);
    return e;
}

// The classes of all holes of a load (or a refinement) that are to have them: groups of holes that share the scratch, a launch of each kernel for
// a group.  A group's scratch: the tables of its holes, then where their subtrees belong.
struct ClassGroup { size_t first, n, tables, bytes; u32 blocks; };
constexpr size_t kClassScratch = 256ull << 20;            // scratch up to which holes share a group (1000 guards of 29 leaves: 165 MB)
struct ClassPlan {
    std::vector<ClassJob> jobs;                           // tables and places as offsets from the start of the scratch
    std::vector<ClassGroup> groups;
    size_t scratch = 0;                                   // of the largest group
    void add(const xp_sketch* s, int hole, LoadOut* out) {
        const HoleHost& h = s->holes[hole];
        if (h.cls_entries == 0) return;
        const size_t table = class_table_bytes(h.cls_entries), place = class_place_bytes(h.cls_entries);
        if (groups.empty() || groups.back().bytes + table + place > kClassScratch || (u64)groups.back().blocks + h.cls_blocks >= 1ull << 30)
            groups.push_back(ClassGroup{jobs.size(), 0, 0, 0, 0u});
        ClassGroup& g = groups.back();
        ClassJob j;
        j.s = s->d_s; j.hole = hole; j.first_block = g.blocks; j.out = out; j.pad = 0;
        j.table = (u64*)g.tables; j.at = (uint2*)(g.bytes - g.tables);
        j.mask = class_slots(h.cls_entries) - 1u;
        jobs.push_back(j);
        ++g.n; g.tables += table; g.bytes += table + place; g.blocks += h.cls_blocks;
        scratch = g.bytes > scratch ? g.bytes : scratch;
    }
    // The jobs as the kernels read them, and their launches (jobs_dev: where the host's copy of them goes).
    void place(char* base) {
        for (const ClassGroup& g : groups)
            for (size_t i = g.first; i < g.first + g.n; ++i) {
                jobs[i].table = (u64*)(base + (size_t)jobs[i].table);
                jobs[i].at = (uint2*)(base + g.tables + (size_t)jobs[i].at);
            }
    }
    cudaError_t launch(const ClassJob* jobs_dev, char* base) const {
        cudaError_t e = cudaSuccess;
        for (size_t i = 0; i < groups.size() && e == cudaSuccess; ++i)
            e = launch_classes(jobs_dev + groups[i].first, (int)groups[i].n, jobs[groups[i].first], groups[i].blocks, base, groups[i].tables, nullptr);
        return e;
    }
};

// Loads of several threads run side by side (their kernels follow one another on the default stream).  A grammar's tables are sent by
// the first load that needs them, and others may queue kernels that read them once that copy has been queued: a load takes the
// blocks of all its new grammars at one time, when no grammar of its list is on its way in another load, and waits for that
// holding none.
static std::mutex g_load_mu;
static std::condition_variable g_load_cv;
static std::mutex g_batch_mu;                // batch loads: one at a time spreads over the cores (four at once, 200 sketches each, took 2.0 ms a load, one after the other 1.3)
constexpr size_t kBatchLoad = 8;             // sketches from which a load is one

extern "C" xp_status xp_sketch_load_batch(const xp_grammar* const* grammars, const xp_sketch_desc* descs, size_t n,
                                          xp_sketch** outs) {
    if (!grammars || !descs || !outs || n == 0) return fail(XP_ERR_INVALID_ARG, "xp_sketch_load_batch: null argument");
    for (size_t i = 0; i < n; ++i) outs[i] = nullptr;
    std::unique_lock<std::mutex> batch(g_batch_mu, std::defer_lock);
    if (n >= kBatchLoad) batch.lock();                    // (before any grammar is taken)
    std::vector<LoadState> st(n);
    char* dev_block = nullptr;
    size_t dev_bytes = 0;
    int dev_device = 0;
    bool sent = false;
    bool claimed = false;                                 // grammars of this load are on their way
    auto settle = [&]() {                                 // they have been sent, or never will be
        if (!claimed) return;
        claimed = false;
        std::lock_guard<std::mutex> lock(g_load_mu);
        for (size_t i = 0; i < n; ++i) {
            if (!st[i].grammar_fresh) continue;
            xp_grammar* g = const_cast<xp_grammar*>(grammars[i]);
            if (!sent) { pool_release(g->d_g, g->d_bytes, g->d_device); g->d_g = nullptr; }
            g->d_pending = false;
        }
        g_load_cv.notify_all();
    };
    struct Settle { decltype(settle)& f; ~Settle() { f(); } } at_the_end{settle};      // (whatever way the call ends)
    auto undo = [&]() {
        cudaStreamSynchronize(nullptr);                   // nothing may still be writing into the blocks
        settle();
        for (size_t i = 0; i < n; ++i) if (st[i].s) xp_sketch_destroy(st[i].s);
        pool_release(dev_block, dev_bytes, dev_device);
    };
#define XP_CUDA_B(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) { undo(); \
        return fail(e_ == cudaErrorMemoryAllocation ? XP_ERR_NOMEM : XP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); } } while (0)
    int ndev = 0;
    // (a description that is wrong is reported as such also where no device can be used)
    const bool no_device = cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1;
    auto refuse = [&](xp_status e, size_t i) {
        const std::string why = no_device && e == XP_ERR_CUDA ? std::string("no CUDA device is usable") : g_last_error;
        undo();
        return fail(e, "sketch " + std::to_string(i) + ": " + why);
    };
    for (size_t i = 0; i < n; ++i) {
        const xp_status e = load_check(grammars[i], &descs[i], &st[i]);
        if (e != XP_OK) return refuse(e, i);
    }
    {
        xp_status e = XP_OK;
        size_t i = 0;
        {
            std::unique_lock<std::mutex> lock(g_load_mu);
            g_load_cv.wait(lock, [&]() {
                for (size_t k = 0; k < n; ++k) if (grammars[k]->d_pending) return false;
                return true;
            });
            claimed = true;
            for (; i < n && e == XP_OK; ++i) {
                xp_grammar* g = const_cast<xp_grammar*>(grammars[i]);
                e = grammar_block(g, &st[i].grammar_fresh);
                if (st[i].grammar_fresh) { g->d_pending = true; st[i].grammar_bytes = grammar_layout(g).total; }
            }
        }
        if (e != XP_OK) return refuse(e, i - 1);
    }
    for (size_t i = 0; i < n; ++i) {
        const xp_status e = load_begin(grammars[i], &descs[i], &st[i]);
        if (e != XP_OK) return refuse(e, i);
    }
    // The staged copy: the job lists, then the sketches' shares, in pieces of about kPieceBytes that page-locked memory
    // holds one by one.  The pieces go to one block of device memory, and a kernel puts the shares in their places:
    // a few large copies instead of two per sketch (a batch of 1024 sketches: 2048 copies, 10 ms of the copy engine's time).
    constexpr size_t kPieceBytes = 8ull << 20, kJobs = 32768;
    size_t n_jobs = 0;
    for (size_t i = 0; i < n; ++i) n_jobs += (size_t)st[i].s->n_holes;
    std::vector<LoadCopy> copies;
    copies.reserve(2 * n);
    for (size_t i = 0; i < n; ++i) copies.push_back(LoadCopy{st[i].s->arena, 0, st[i].head});
    for (size_t i = 0; i < n; ++i) if (st[i].grammar_fresh) copies.push_back(LoadCopy{(char*)st[i].s->g->d_g, 0, st[i].grammar_bytes});
    const size_t at_list = 0, at_jobs = at_list + al256(sizeof(SketchDev*) * n), at_copies = at_jobs + al256(sizeof(LoadJob) * n_jobs);
    ClassPlan cls;
    for (size_t i = 0; i < n; ++i) for (int h = 0; h < st[i].s->n_holes; ++h) cls.add(st[i].s, h, nullptr);
    const size_t at_cls = at_copies + al256(sizeof(LoadCopy) * copies.size()), at_shares = at_cls + al256(sizeof(ClassJob) * cls.jobs.size());
    std::vector<size_t> piece_at;                         // start of each piece; the lists are in the first
    size_t at = at_shares;
    piece_at.push_back(0);
    for (size_t i = 0, c = n; i < n; ++i) {
        const size_t share = st[i].head + st[i].grammar_bytes;
        // (a piece is closed only when it holds a sketch: whoever fills the last one sends it; the lists, and a share of any
        // size, may make a piece larger than that)
        if (i > 0 && at + share - piece_at.back() > kPieceBytes) piece_at.push_back(at);
        st[i].stage_at = at; st[i].piece = piece_at.size() - 1;
        copies[i].src = at;
        if (st[i].grammar_fresh) copies[c++].src = at + st[i].head;
        at += share;
    }
    const size_t staged = at;
    const bool put = n == 1 && staged <= kPutMost;        // (a small sketch alone: straight to its places, without copy and scatter)
    const size_t at_out = al256(staged), at_scratch = at_out + al256(sizeof(LoadOut) * n_jobs);
    const size_t at_classes = at_scratch + al256(prepare_scratch_bytes((int)(n_jobs < kJobs ? n_jobs : kJobs)));
    size_t class_bytes = cls.scratch, total = at_classes + class_bytes;
    cudaError_t got = pool_alloc((void**)&dev_block, total, &dev_device, &dev_bytes);
    if (got != cudaSuccess && class_bytes > 0) {          // (memory is short: without classes)
        (void)cudaGetLastError();
        class_bytes = 0;
        total = at_classes;
        got = pool_alloc((void**)&dev_block, total, &dev_device, &dev_bytes);
    }
    XP_CUDA_B(got);
    StageBlock back(sizeof(LoadOut) * n_jobs);
    if (!back.p) { undo(); return fail(XP_ERR_NOMEM, "out of host memory"); }
    {
        std::vector<StageBlock*> hold;
        std::vector<std::atomic<size_t>> left(piece_at.size());
        std::vector<size_t> first(piece_at.size() + 1, n);       // sketches of a piece: [first[p], first[p + 1])
        for (size_t i = n; i-- > 0;) first[st[i].piece] = i;
        auto piece_end = [&](size_t p) { return p + 1 < piece_at.size() ? piece_at[p + 1] : staged; };
        bool ok = true;
        for (size_t p = 0; p < piece_at.size() && ok; ++p) {
            hold.push_back(new (std::nothrow) StageBlock(piece_end(p) - piece_at[p]));
            ok = hold.back() != nullptr && hold.back()->p != nullptr;
        }
        cudaError_t err = cudaSuccess;
        if (ok) {
            char* lists = hold[0]->p;
            size_t j = 0;
            for (size_t i = 0; i < n; ++i) {
                ((SketchDev**)(lists + at_list))[i] = st[i].s->d_s;
                for (int h = 0; h < st[i].s->n_holes; ++h, ++j) ((LoadJob*)(lists + at_jobs))[j] = LoadJob{st[i].s->d_s, h, 0};
            }
            memcpy(lists + at_copies, copies.data(), sizeof(LoadCopy) * copies.size());
            // (what the classes come to goes straight to page-locked memory like the rest of LoadOut)
            LoadOut* out = (LoadOut*)(back.locked ? back.p : dev_block + at_out);
            cls.place(dev_block + at_classes);
            for (size_t i = 0, c = 0; i < n; out += st[i].s->n_holes, ++i)
                for (int h = 0; h < st[i].s->n_holes; ++h) if (st[i].s->holes[h].cls_entries > 0) cls.jobs[c++].out = out + h;
            memcpy(lists + at_cls, cls.jobs.data(), sizeof(ClassJob) * cls.jobs.size());
            // large batches fill their pieces with a few threads; whoever finishes a piece's last share sends the piece
            size_t n_threads = staged / (1u << 20) < n / 8 ? staged / (1u << 20) : n / 8;      // (starting a thread takes as long as filling some 300 KB)
            const unsigned hw = std::thread::hardware_concurrency();
            if (n_threads > 8) n_threads = 8;
            if (hw > 0 && n_threads > hw) n_threads = hw;
            for (size_t p = 0; p < piece_at.size(); ++p) left[p].store(first[p + 1] - first[p]);
            std::atomic<size_t> next(0);
            std::atomic<int> bad(0);
            auto send = [&](size_t p) {
                if (put) return;
                const cudaError_t e = cudaMemcpyAsync(dev_block + piece_at[p], hold[p]->p, piece_end(p) - piece_at[p], cudaMemcpyHostToDevice, nullptr);
                if (e != cudaSuccess) bad.store((int)e);
            };
            auto work = [&](bool own) {
                if (own) cudaSetDevice(dev_device);
                for (;;) {
                    const size_t i = next.fetch_add(1);
                    if (i >= n) break;
                    const size_t p = st[i].piece;
                    load_fill(&st[i], hold[p]->p + (st[i].stage_at - piece_at[p]));
                    if (left[p].fetch_sub(1) == 1) send(p);
                }
            };
            if (n_threads < 2) work(false);
            else {
                std::vector<std::thread> pool;
                pool.reserve(n_threads);
                try {
                    for (size_t t = 0; t + 1 < n_threads; ++t) pool.emplace_back(work, true);
                } catch (const std::system_error&) {      // (no more threads to be had: those there are do the work)
                }
                work(false);
                for (std::thread& th : pool) th.join();
            }
            err = (cudaError_t)bad.load();
            if (put) {
                const u32 a = (u32)(at_shares / 16), b = a + (u32)(st[0].head / 16), c = b + (u32)(st[0].grammar_bytes / 16);
                const PutPlaces to = {{dev_block, st[0].s->arena, (char*)st[0].s->g->d_g}, {a, b, c}};
                err = launch_put(to, hold[0]->p, nullptr);
            } else if (err == cudaSuccess) err = launch_scatter((const LoadCopy*)(dev_block + at_copies), (int)copies.size(), dev_block, nullptr);
            if (err == cudaSuccess) { sent = true; settle(); }
        }
        // (the staging blocks may go back once the copies have been made: they are waited for below, with everything else)
        struct Hold { std::vector<StageBlock*>& v; ~Hold() { for (StageBlock* b : v) delete b; } } release{hold};
        if (!ok || err != cudaSuccess) {
            cudaStreamSynchronize(nullptr);
            undo();
            return ok ? fail(XP_ERR_CUDA, std::string("xp_sketch_load: ") + cudaGetErrorString(err)) : fail(XP_ERR_NOMEM, "out of host memory");
        }
        // host tables too large for the staged copy
        i64 most_points = 0, most_staged = 0;
        int size_cap = 0, probes_cap = 0;
        u64 most_entries[kMaxSize + 1] = {0};
        for (size_t i = 0; i < n; ++i) {
            const LoadState& L = st[i];
            xp_sketch* s = L.s;
            const size_t np = (size_t)s->n_points, row = (size_t)(s->g->n_vars ? s->g->n_vars : 1);
            const size_t coords_bytes = sizeof(i32) * np * row, spec_bytes = sizeof(i64) * np;
            s->load_h2d = L.head + L.grammar_bytes + sizeof(SketchDev*) + sizeof(LoadJob) * (size_t)s->n_holes + sizeof(LoadCopy) * (L.grammar_fresh ? 2 : 1);
            for (const HoleHost& hh : s->holes) if (hh.cls_entries > 0) s->load_h2d += sizeof(ClassJob);
            s->load_d2h = sizeof(LoadOut) * (size_t)s->n_holes;
            if (L.copy_coords && coords_bytes > kPackMax) {
                XP_CUDA_B(cudaMemcpyAsync(s->arena + L.off_coords, L.d->coords, coords_bytes, cudaMemcpyHostToDevice, nullptr));
                s->load_h2d += coords_bytes;
            }
            for (int h = 0; h < s->n_holes; ++h) {
                const xp_hole_desc& hd = L.d->holes[h];
                if (hd.spec_kind == XP_SPEC_TABLE && np > 0 && !hd.spec_table_on_device && spec_bytes > kPackMax) {
                    XP_CUDA_B(cudaMemcpyAsync(s->arena + L.hole[h].off_spec, hd.spec_table, spec_bytes, cudaMemcpyHostToDevice, nullptr));
                    s->load_h2d += spec_bytes;
                }
                if (hd.spec_kind == XP_SPEC_EXPR && L.stage && s->n_points > most_staged) most_staged = s->n_points;
            }
            if (L.d->domain_kind == XP_DOMAIN_TABLE && s->n_points > most_points) most_points = s->n_points;
            if (L.stage_box && s->n_points > most_staged) most_staged = s->n_points;
            if (s->tab_size_cap > size_cap) size_cap = s->tab_size_cap;
            if (s->tab_probes_cap > probes_cap) probes_cap = s->tab_probes_cap;
            for (int k = 1; k <= s->tab_size_cap; ++k) most_entries[k] = s->entries_at[k] > most_entries[k] ? s->entries_at[k] : most_entries[k];
        }
        // The load's kernels, in stream order, one launch of each for the whole batch: points of the boxes and values of
        // spec expressions (so that the whole-domain check, and the probe choice, read tables for every kind of domain);
        // bounds of the tables' coordinates; the probe choice; the subtree tables, bottom-up, for as many sizes and probes
        // as there can be (blocks beyond what the probe choice settled on for their hole return at once); the operand classes.
        // Grids are cut into pieces of at most kJobs jobs (a grid dimension holds 65 535).
        SketchDev* const* d_list = (SketchDev* const*)(dev_block + at_list);
        const LoadJob* d_jobs = (const LoadJob*)(dev_block + at_jobs);
        for (size_t q = 0; q < n; q += kJobs) {
            const int m = (int)(n - q < kJobs ? n - q : kJobs);
            XP_CUDA_B(launch_coord_bounds(d_list + q, m, most_points, nullptr));
        }
        for (size_t q = 0; q < n_jobs; q += kJobs) {
            const int m = (int)(n_jobs - q < kJobs ? n_jobs - q : kJobs);
            // (what it decides per hole goes straight to page-locked memory: a few bytes, and no copy to queue behind the tables)
            LoadOut* out = (LoadOut*)(back.locked ? back.p : dev_block + at_out);
            XP_CUDA_B(launch_stage_sample(d_list, q == 0 ? (int)n : 0, most_staged, d_jobs + q, m, dev_block + at_scratch, nullptr));
            XP_CUDA_B(launch_prepare(d_jobs + q, m, dev_block + at_scratch, out + q, nullptr));
        }
        for (size_t q = 0; q < n_jobs; q += kJobs)
            XP_CUDA_B(make_tables(d_jobs + q, (int)(n_jobs - q < kJobs ? n_jobs - q : kJobs), size_cap, probes_cap, most_entries));
        if (class_bytes > 0) XP_CUDA_B(cls.launch((const ClassJob*)(dev_block + at_cls), dev_block + at_classes));
        if (!back.locked) XP_CUDA_B(cudaMemcpyAsync(back.p, dev_block + at_out, sizeof(LoadOut) * n_jobs, cudaMemcpyDeviceToHost, nullptr));
        XP_CUDA_B(cudaStreamSynchronize(nullptr));
    }
#undef XP_CUDA_B
    pool_release(dev_block, dev_bytes, dev_device);
    const LoadOut* o = (const LoadOut*)back.p;
    for (size_t i = 0; i < n; ++i) {
        xp_sketch* s = st[i].s;
        for (int h = 0; h < s->n_holes; ++h, ++o) { hole_decided(&s->holes[h], *o); s->n_probes.push_back(o->n_probe); }
        outs[i] = s;
    }
    return XP_OK;
}

extern "C" xp_status xp_sketch_load(const xp_grammar* g, const xp_sketch_desc* d, xp_sketch** out) {
    if (!g || !d || !out) return fail(XP_ERR_INVALID_ARG, "xp_sketch_load: null argument");
    return xp_sketch_load_batch(&g, d, 1, out);
}

namespace xp {
SketchInternals sketch_internals(const xp_sketch* s) { return SketchInternals{s->d_s, s->g, s->n_points, s->arena_device, s->g->n_vars}; }
u64 grammar_cnt(const xp_grammar* g, int nt, int size) { return g->cnt[nt][size]; }
int grammar_nonterminals(const xp_grammar* g) { return g->n_nt; }
int grammar_ok_size(const xp_grammar* g) { return g->ok_size; }
GrammarHost grammar_host(const xp_grammar* g) {
    static thread_local std::vector<const char*> names;
    names.clear();
    for (const std::string& n : g->names) names.push_back(n.c_str());
    return GrammarHost{g->n_nt, g->n_vars, g->leaf_begin, g->bin_begin, g->leaves.data(), g->bins.data(), names.data()};
}
HoleSpec sketch_hole(const xp_sketch* s, int hole) {
    if (hole < 0 || hole >= s->n_holes) return HoleSpec{-1, 0};
    return HoleSpec{s->holes[hole].start_nt, s->holes[hole].max_size};
}
const HoleDev* sketch_hole_dev(const xp_sketch* s, int hole) { return s->d_holes + hole; }
StageMemory::StageMemory(size_t bytes) : p(nullptr), locked(false), block(new (std::nothrow) StageBlock(bytes)) {
    if (block) { p = ((StageBlock*)block)->p; locked = ((StageBlock*)block)->locked; }
}
StageMemory::~StageMemory() { delete (StageBlock*)block; }
StageEvents::StageEvents() : e0(nullptr), e1(nullptr), pair(new (std::nothrow) EventPair) {}
StageEvents::~StageEvents() { delete (EventPair*)pair; }
cudaError_t StageEvents::open() {
    if (!pair) return cudaErrorMemoryAllocation;
    const cudaError_t e = ((EventPair*)pair)->open();
    e0 = ((EventPair*)pair)->e0; e1 = ((EventPair*)pair)->e1;
    return e;
}
cudaError_t device_alloc(void** out, size_t bytes, int* device, size_t* granted) { return pool_alloc(out, bytes, device, granted); }
void device_release(void* ptr, size_t granted, int device) { pool_release(ptr, granted, device); }
}  // namespace xp

extern "C" xp_status xp_sketch_info_get(const xp_sketch* s, xp_sketch_info* out) {
    if (!s || !out) return fail(XP_ERR_INVALID_ARG, "xp_sketch_info_get: null argument");
    memset(out, 0, sizeof(*out));
    out->n_holes = s->n_holes; out->device = s->arena_device; out->n_points = s->n_points;
    out->device_bytes = s->arena_bytes; out->load_h2d_bytes = s->load_h2d; out->load_d2h_bytes = s->load_d2h;
    for (int h = 0; h < s->n_holes && h < 8; ++h) out->n_probes[h] = s->n_probes[h];
    out->n_refined = s->n_refined;
    return XP_OK;
}

// Promotes the points that ended whole-domain checks to probes (see include/xp.h).  The hole
// records and the tables of noted points are read back; per hole the new probe list is
// [probe 0, promoted points by how many survivors each ended, the other old probes]; the records
// go back with the new ids, one small kernel derives coordinates, spec values and context forms
// of the probes again, and the subtree tables are rebuilt for them.
extern "C" xp_status xp_sketch_refine(xp_sketch* s, int32_t max_promote, int32_t* n_promoted) {
    if (n_promoted) *n_promoted = 0;
    if (!s || max_promote < 0) return fail(XP_ERR_INVALID_ARG, "xp_sketch_refine: bad argument");
    const xp_sketch* cs = s;
    xp_status st = check_device(&cs, 1);
    if (st != XP_OK) return st;
    const int nh = s->n_holes;
    const int most = max_promote == 0 ? 4 : max_promote;
    const size_t kill_bytes = (sizeof(i64) + sizeof(u32)) * kKillSlots;
    std::vector<HoleDev> hh(nh);
    std::vector<char> kills(kill_bytes * nh);
    XP_CUDA(cudaStreamSynchronize(nullptr));
    XP_CUDA(cudaMemcpy(hh.data(), s->arena + s->off_holes, sizeof(HoleDev) * nh, cudaMemcpyDeviceToHost));
    for (int h = 0; h < nh; ++h)
        XP_CUDA(cudaMemcpy(&kills[kill_bytes * h], s->arena + s->off_kill[h], kill_bytes, cudaMemcpyDeviceToHost));
    int promoted = 0;
    std::vector<LoadJob> jobs;
    for (int h = 0; h < nh; ++h) {
        HoleDev& o = hh[h];
        const i64* pid = (const i64*)&kills[kill_bytes * h];
        const u32* cnt = (const u32*)(&kills[kill_bytes * h] + sizeof(i64) * kKillSlots);
        std::vector<std::pair<u32, i64>> found;          // (survivors ended, point), most frequent first
        for (int k = 0; k < kKillSlots; ++k)
            if (pid[k] >= 0 && pid[k] < s->n_points && cnt[k] > 0) found.push_back({cnt[k], pid[k]});
        std::sort(found.begin(), found.end(), [](const std::pair<u32, i64>& a, const std::pair<u32, i64>& b) {
            return a.first != b.first ? a.first > b.first : a.second < b.second; });
        if (found.empty() || o.n_probe < 1) continue;
        std::vector<i64> ids;
        ids.push_back(o.probe_id[0]);
        int taken = 0;
        for (size_t k = 0; k < found.size() && taken < most && (int)ids.size() < kMaxProbe; ++k) {
            bool dup = false;
            for (int j = 0; j < o.n_probe; ++j) dup = dup || o.probe_id[j] == found[k].second;
            if (!dup) { ids.push_back(found[k].second); ++taken; }
        }
        if (taken == 0) continue;
        for (int j = 1; j < o.n_probe && (int)ids.size() < kMaxProbe; ++j) ids.push_back(o.probe_id[j]);
        o.n_probe = (i32)ids.size();
        for (int j = 0; j < o.n_probe; ++j) o.probe_id[j] = ids[j];
        promoted += taken;
        LoadJob job;
        job.s = s->d_s; job.hole = h; job.pad = 0;
        jobs.push_back(job);
    }
    // the notes start afresh whether or not anything was promoted
    std::vector<char> fresh(kill_bytes, 0);
    memset(fresh.data(), 0xff, sizeof(i64) * kKillSlots);
    for (int h = 0; h < nh; ++h) XP_CUDA(cudaMemcpyAsync(s->arena + s->off_kill[h], fresh.data(), kill_bytes, cudaMemcpyHostToDevice, nullptr));
    if (!jobs.empty()) {
        char* jobs_dev = nullptr;
        size_t jobs_bytes = 0;
        int jobs_device = 0;
        ClassPlan cls;
        for (int h = 0; h < nh; ++h) cls.add(s, h, nullptr);
        const size_t at_cls = al256(sizeof(LoadJob) * jobs.size()), at_classes = at_cls + al256(sizeof(ClassJob) * cls.jobs.size());
        size_t class_bytes = cls.scratch;
        cudaError_t got = pool_alloc((void**)&jobs_dev, at_classes + class_bytes, &jobs_device, &jobs_bytes);
        if (got != cudaSuccess && class_bytes > 0) {      // (memory is short: without classes from here on)
            (void)cudaGetLastError();
            class_bytes = 0;
            got = pool_alloc((void**)&jobs_dev, at_classes, &jobs_device, &jobs_bytes);
        }
        XP_CUDA(got);
        for (HoleDev& o : hh) { memset(o.cls_count, 0, sizeof(o.cls_count)); o.cls_size = 0; }      // (holes without a promoted point are numbered again too)
        cudaError_t e = cudaMemcpyAsync(s->arena + s->off_holes, hh.data(), sizeof(HoleDev) * nh, cudaMemcpyHostToDevice, nullptr);
        if (e == cudaSuccess) e = cudaMemcpyAsync(jobs_dev, jobs.data(), sizeof(LoadJob) * jobs.size(), cudaMemcpyHostToDevice, nullptr);
        cls.place(jobs_dev + at_classes);
        if (e == cudaSuccess && class_bytes > 0) e = cudaMemcpyAsync(jobs_dev + at_cls, cls.jobs.data(), sizeof(ClassJob) * cls.jobs.size(), cudaMemcpyHostToDevice, nullptr);
        if (e == cudaSuccess) e = launch_reprobe((const LoadJob*)jobs_dev, (int)jobs.size(), nullptr);
        if (e == cudaSuccess) e = make_tables((const LoadJob*)jobs_dev, (int)jobs.size(), s->tab_size_cap, s->tab_probes_cap, s->entries_at);
        if (e == cudaSuccess && class_bytes > 0) e = cls.launch((const ClassJob*)(jobs_dev + at_cls), jobs_dev + at_classes);
        if (e == cudaSuccess) e = cudaMemcpyAsync(hh.data(), s->arena + s->off_holes, sizeof(HoleDev) * nh, cudaMemcpyDeviceToHost, nullptr);
        const cudaError_t e2 = cudaStreamSynchronize(nullptr);
        pool_release(jobs_dev, jobs_bytes, jobs_device);
        if (e != cudaSuccess || e2 != cudaSuccess)
            return fail(XP_ERR_CUDA, std::string("xp_sketch_refine: ") + cudaGetErrorString(e != cudaSuccess ? e : e2));
        for (int h = 0; h < nh; ++h) {
            LoadOut o{hh[h].filter_ok, hh[h].tab_probes, hh[h].aff_ok, hh[h].join_on, hh[h].second, hh[h].n_probe, hh[h].tab_max_size,
                      hh[h].join_t0 == 0 || hh[h].join_t1 == 0, hh[h].sample_pass, hh[h].sample_n, 0u, hh[h].cls_size, {0}};
            memcpy(o.cls_n, hh[h].cls_n, sizeof(o.cls_n));
            hole_decided(&s->holes[h], o);
            s->n_probes[h] = hh[h].n_probe;
        }
        std::lock_guard<std::mutex> lock(s->plan_mu);
        for (auto& kept : s->plan_kept) kept.reset();     // (the plan depends on which holes the filter serves)
    } else {
        XP_CUDA(cudaStreamSynchronize(nullptr));
    }
    s->n_refined += promoted;
    if (n_promoted) *n_promoted = promoted;
    return XP_OK;
}

// ------------------------------------------------------------------------------------------
// repair
// ------------------------------------------------------------------------------------------

struct HoleResult {
    int max_size = 0, solved = 0, least_size = 0;
    u64 cand_count[kMaxSize + 1] = {0};
    u64 match_count[kMaxSize + 1] = {0};
    u64 least_rank = 0;
    std::vector<xp_instr> code;
    std::string text;
    u64 evals = 0, filter_survivors = 0, probe_survivors = 0, nominal_ops = 0;
    u64 filter_tests = 0, skipped = 0;
};

struct xp_result {
    std::vector<HoleResult> holes;
    double kernel_ms = 0, total_ms = 0;
    int n_launches = 0;
    u64 h2d_bytes = 0, d2h_bytes = 0;
};

// Scratch of calls that bring no workspace: one block per process, reused while no other call
// is using it (a concurrent call allocates its own).
static std::mutex g_ws_mu;
static char* g_ws = nullptr;
static size_t g_ws_bytes = 0;
static int g_ws_device = -1;

static const xp_repair_opts kDefaultOpts = {0, 0, 0, nullptr, nullptr, nullptr, 0, 0u, nullptr, 0};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

static void add_linear(Plan* plan, int sketch, int hole, int acc, int k, u64 lo, u64 hi) {
    SegDev sg;
    memset(&sg, 0, sizeof(sg));
    sg.first_ticket = plan->n_tickets;
    sg.rank_begin = lo; sg.rank_end = hi;
    sg.sketch = sketch; sg.hole = hole; sg.size = k; sg.kind = kSegLinear; sg.acc = acc;
    plan->segs.push_back(sg);
    plan->n_tickets += (hi - lo + (u64)kLinearChunk - 1) / (u64)kLinearChunk;
}

constexpr size_t kPairMaxSketches = 8;       // (each block has scratch of its own: 12 MB for 92 480 operands a side)
constexpr u64 kPairMost = 1ull << 22;        // operands of either side (the size of the subtree tables)
// Pairs from which the pair join is taken.  It costs a block some ten launches one after the other, where the tiles of all blocks and
// sketches are one launch (size 7, tiles / pair join: one sketch 0.15 / 0.16 ms at 2.6e7 pairs a block, 0.39 / 0.25 at 1.3e8;
// four 0.75 / 0.81 at 1.3e8, 1.67 / 1.36 at 4.2e8).
constexpr u64 kPairLeast = 1ull << 26, kPairLeastBatch = 1ull << 28;
constexpr u64 kPairLeastRing = 1ull << 20;   // ... of a nonterminal without / and % there: half the launches (a ragged table, 2.4e6 pairs: 0.36 / 0.34 ms)
constexpr size_t kPairFew = 2;               // sketches up to which kPairLeast holds
// A rank window cuts a block to some of its left operands, but the other side is indexed whole: a block with fewer rows than this,
// or thereabouts, is done as tiles before the index is made (450 000 operands a side, remainders: 2 222 rows 0.26 ms, the index 1.9).
constexpr u64 kPairEach = 1ull << 12;
constexpr int kRangeParts = 4;               // parts of the constants there: a warp checks its suspects by itself, some hundred of them from 32 operands and all
                                             // constants (three conv holes: join 440 us in one part, 350 with 8 operands a ticket, 330 so)
constexpr u64 kRangeSplit = 1ull << 15;      // ... up to which an operator is a segment of its own (with more there are warps enough at work)

// Does the pair join know the block (production, left size a) of size k?  Both operands tabulated, an operator it has
// (products only where neither target is zero: a zero operand would leave its partner open).
static bool pair_joins(const xp_grammar* g, const HoleHost& ho, const BinDev& bd, int a, int k) {
    const int b = k - 1 - a;
    if (!ho.join_on || bd.op > XP_OP_MOD || (bd.op == XP_OP_MUL && ho.target_zero)) return false;
    if (a > ho.tab_max || b > ho.tab_max) return false;
    return g->cnt[bd.lnt][a] <= kPairMost && g->cnt[bd.rnt][b] <= kPairMost;
}

// Pair-join blocks of (start nonterminal, size k) that ranks [lo, hi) touch: one per (left, right) operand sets.  taken: per
// production of the nonterminal a bit for every left size whose block is here and not for the tiles.
static void add_pairs(Plan* plan, const xp_grammar* g, const HoleHost& ho, int sketch, int hole, int acc, int k, u64 lo, u64 hi, u64 least, std::vector<u32>* taken) {
    const size_t first_seg = plan->psegs.size();
    const int nt = ho.start_nt;
    taken->assign((size_t)(g->bin_begin[nt + 1] - g->bin_begin[nt]), 0u);
    bool divides = false;
    for (int b = g->bin_begin[nt]; b < g->bin_begin[nt + 1]; ++b) {
        const BinDev& bd = g->bins[b];
        if (bd.op != XP_OP_DIV && bd.op != XP_OP_MOD) continue;
        for (int a = 2; a < k - 2; ++a) divides = divides || (g->cnt[bd.lnt][a] > 0 && g->cnt[bd.rnt][k - 1 - a] > 0);
    }
    if (!divides && least > kPairLeastRing) least = kPairLeastRing;
    for (int b = g->bin_begin[nt]; b < g->bin_begin[nt + 1]; ++b) {
        const BinDev& bd = g->bins[b];
        u64 base = bd.off[k];
        for (int a = 1; a <= k - 2; ++a) {
            const u64 cl = g->cnt[bd.lnt][a], cr = g->cnt[bd.rnt][k - 1 - a], block = cl * cr;
            const u64 this_base = base;
            base += block;
            if (a == 1 || a == k - 2 || block == 0 || !pair_joins(g, ho, bd, a, k)) continue;
            if (this_base + block <= lo || this_base >= hi) continue;
            const u64 wlo = lo > this_base ? lo - this_base : 0, whi = hi - this_base < block ? hi - this_base : block;
            const u64 l0 = wlo / cr, nl = (whi + cr - 1) / cr - l0;      // left operands that the window covers
            if (nl * cr < least || (least > 1 && nl < cl && nl * cr < kPairEach * (nl + cr))) continue;
            taken->at(b - g->bin_begin[nt]) |= 1u << a;
            // (a side of classes; the left one where the window covers more operands than there are)
            auto classes = [&](int n, int size, u64 all) { return size == ho.cls_size && ho.cls_n[n] > 0 && ho.cls_n[n] < all; };
            const bool lcls = classes(bd.lnt, a, nl), rcls = classes(bd.rnt, k - 1 - a, cr);
            const u64 first = lcls ? 0 : l0, left = lcls ? ho.cls_n[bd.lnt] : nl, right = rcls ? ho.cls_n[bd.rnt] : cr;
            PairSeg* sg = nullptr;
            for (size_t i = first_seg; i < plan->psegs.size() && !sg; ++i) {
                PairSeg& c = plan->psegs[i];
                if (c.lnt == bd.lnt && c.rnt == bd.rnt && c.la == a && c.l_begin == first && c.nl == left && c.pairs == nl * cr && !((c.ops >> bd.op) & 1u)) sg = &c;
            }
            if (!sg) {
                PairSeg c;
                memset(&c, 0, sizeof(c));
                c.rank_begin = lo; c.rank_end = hi;
                c.sketch = sketch; c.hole = hole; c.size = k; c.acc = acc;
                c.lnt = bd.lnt; c.la = a; c.rnt = bd.rnt; c.ra = k - 1 - a;
                c.l_begin = (u32)first; c.nl = (u32)left; c.nr = (u32)right;
                c.lcls = lcls ? 1 : 0; c.rcls = rcls ? 1 : 0;
                c.right_count = cr; c.pairs = nl * cr;
                c.index_right = right <= left ? 1 : 0;       // the smaller side is indexed (its chains stay in L2)
                u32 heads = 1024;
                while (heads < (c.index_right ? c.nr : c.nl)) heads <<= 1;
                c.head_mask = heads - 1;
                c.far_pieces = pair_pieces(c.nl, c.nr);
                plan->psegs.push_back(c);
                sg = &plan->psegs.back();
            }
            sg->ops |= 1u << bd.op;
            sg->base[bd.op] = this_base + first * cr;
        }
    }
}

constexpr u64 kFamilyMaxWork = 512;          // candidates per register operand below which segments share a fill
constexpr u64 kTileTickets = 148;            // tickets that a segment of a small call is cut into, if it has the operands

// Tile segments of (start nonterminal, size k) restricted to ranks [lo, hi): one per
// (left size, group of productions with the same operand nonterminals and the same rows).
// taken: blocks that the pair join has (null: none); few: the call has so few sketches that a ticket for every SM is wanted;
// leaves: blocks with a leaf as an operand too.
static void add_tiles(Plan* plan, const xp_grammar* g, const std::vector<u32>* taken, int nt, int sketch, int hole, int acc, int k, u64 lo, u64 hi, int bc_tile, bool few, bool leaves) {
    const size_t first_seg = plan->segs.size();
    for (int b = g->bin_begin[nt]; b < g->bin_begin[nt + 1]; ++b) {
        const BinDev& bd = g->bins[b];
        u64 base = bd.off[k];
        for (int a = 1; a <= k - 2; ++a) {
            const u64 cl = g->cnt[bd.lnt][a], cr = g->cnt[bd.rnt][k - 1 - a];
            const u64 block = cl * cr;
            if (block == 0) continue;
            const u64 this_base = base;
            base += block;
            if ((a == 1 || a == k - 2) && !leaves) continue; // (a leaf at the root: add_joins)
            if (taken && ((taken->at(b - g->bin_begin[nt]) >> a) & 1u)) continue;      // (add_pairs)
            if (this_base + block <= lo || this_base >= hi) continue;
            const u64 wlo = lo > this_base ? lo - this_base : 0;
            const u64 whi = hi - this_base < block ? hi - this_base : block;
            const u64 l0 = wlo / cr, l1 = (whi + cr - 1) / cr;
            const bool reg_left = (l1 - l0) >= cr;
            SegDev* sg = nullptr;
            for (size_t i = first_seg; i < plan->segs.size() && !sg; ++i) {       // an open group this production fits in
                SegDev& c = plan->segs[i];
                const int c_lnt = c.swap ? c.bc_nt : c.reg_nt, c_rnt = c.swap ? c.reg_nt : c.bc_nt;
                const int c_a = c.swap ? c.bc_size : c.reg_size;
                const u64 c_l0 = c.swap ? c.bc_begin : c.reg_begin, c_l1 = c_l0 + (c.swap ? c.bc_count : c.reg_count);
                bool has_op = false;
                for (int o = 0; o < c.n_ops; ++o) has_op = has_op || c.op[o] == bd.op;
                if (c_lnt == bd.lnt && c_rnt == bd.rnt && c_a == a && c_l0 == l0 && c_l1 == l1 && !has_op && c.n_ops < 5) sg = &c;
            }
            if (!sg) {
                SegDev n;
                memset(&n, 0, sizeof(n));
                n.rank_begin = lo; n.rank_end = hi;
                n.sketch = sketch; n.hole = hole; n.size = k; n.kind = kSegTile; n.acc = acc;
                n.swap = reg_left ? 0 : 1;
                n.reg_nt = reg_left ? bd.lnt : bd.rnt;  n.reg_size = reg_left ? a : k - 1 - a;
                n.bc_nt = reg_left ? bd.rnt : bd.lnt;   n.bc_size = reg_left ? k - 1 - a : a;
                n.reg_begin = reg_left ? l0 : 0;        n.reg_count = reg_left ? l1 - l0 : cr;
                n.bc_begin = reg_left ? 0 : l0;         n.bc_count = reg_left ? cr : l1 - l0;
                n.right_count = cr;
                n.reg_tiles = (u32)((n.reg_count + kRegTile - 1) / kRegTile);
                n.bc_tile = bc_tile;
                n.bc_tiles = (u32)((n.bc_count + bc_tile - 1) / bc_tile);
                plan->segs.push_back(n);
                sg = &plan->segs.back();
            }
            sg->op[sg->n_ops] = bd.op;
            sg->op_base[sg->n_ops] = this_base;
            sg->n_ops += 1;
            if (bd.op == XP_OP_DIV || bd.op == XP_OP_MOD) sg->has_div = 1;
            if (bd.op == XP_OP_SHL || bd.op == XP_OP_SHR) sg->generic = 1;
        }
    }
    // A small segment of a small call: narrower broadcast tiles, until there are as many tickets as SMs.  (Its few tickets ran on as many
    // SMs: four sketches of 12 leaves, size 7, 0.28 -> 0.12 ms; one of 5 leaves, size 9, where most of a tile hits, 1.86 -> 0.65.)
    if (few)
        for (size_t i = first_seg; i < plan->segs.size(); ++i) {
            SegDev& c = plan->segs[i];
            if ((u64)c.reg_tiles * c.bc_tiles >= kTileTickets || c.bc_count * (u64)c.n_ops < kFamilyMaxWork) continue;
            const u64 share = (c.bc_count * c.reg_tiles + kTileTickets - 1) / kTileTickets, tile = (share + 15) & ~15ull;
            if (tile >= (u64)c.bc_tile) continue;
            c.bc_tile = (i32)tile;
            c.bc_tiles = (u32)((c.bc_count + tile - 1) / tile);
        }
    // Families: segments with the same register-side operands and a single broadcast tile are
    // put next to each other; the first takes the tickets (one per register tile) and visits
    // the others, so the register operands are fetched once for all of them.
    std::vector<SegDev> ordered;
    std::vector<char> placed(plan->segs.size() - first_seg, 0);
    for (size_t i = first_seg; i < plan->segs.size(); ++i) {
        if (placed[i - first_seg]) continue;
        const SegDev head = plan->segs[i];
        placed[i - first_seg] = 1;
        const size_t at = ordered.size();
        ordered.push_back(head);
        int members = 1;
        // (worth it only for segments with little work per register operand: the fill is then a large share)
        if (head.bc_tiles == 1 && head.bc_count * (u64)head.n_ops < kFamilyMaxWork)
            for (size_t j = i + 1; j < plan->segs.size(); ++j) {
                const SegDev& c = plan->segs[j];
                if (members == kMaxFamily) break;               // the rest head families of their own
                if (placed[j - first_seg] || c.bc_tiles != 1 || c.bc_count * (u64)c.n_ops >= kFamilyMaxWork || c.reg_nt != head.reg_nt || c.reg_size != head.reg_size ||
                    c.reg_begin != head.reg_begin || c.reg_count != head.reg_count) continue;
                placed[j - first_seg] = 1;
                ordered.push_back(c);
                ordered.back().family = 0;
                ++members;
            }
        ordered[at].family = members;
        // broadcast slots side by side when the whole family fits the tile and has one tile each
        u64 slots = 0;
        bool one_tile = true;
        for (int m = 0; m < members; ++m) { slots += ordered[at + m].bc_count; one_tile = one_tile && ordered[at + m].bc_tiles == 1; }
        if (one_tile && slots <= (u64)kBcTile) {
            u64 base = 0;
            for (int m = 0; m < members; ++m) { ordered[at + m].bc_base = (i32)base; base += ordered[at + m].bc_count; }
            ordered[at].bc_keep = 1;
        }
    }
    for (size_t i = 0; i < ordered.size(); ++i) plan->segs[first_seg + i] = ordered[i];
    for (size_t i = first_seg; i < plan->segs.size(); ++i) {
        SegDev& c = plan->segs[i];
        c.first_ticket = plan->n_tickets;                          // members: where the next head starts
        if (c.family >= 1) plan->n_tickets += (u64)c.reg_tiles * c.bc_tiles;
        // cost model: operation + comparison per evaluation; / and % share one reciprocal division
        u64 per_pair = 0;
        bool div = false, mod = false;
        for (int o = 0; o < c.n_ops; ++o) {
            if (c.op[o] == XP_OP_DIV) div = true;
            else if (c.op[o] == XP_OP_MOD) mod = true;
            else per_pair += 2;
        }
        if (div || mod) per_pair += 7 + (div ? 1 : 0) + (mod ? 2 : 0);
        plan->nominal_ops[acc] += c.reg_count * c.bc_count * per_pair;
    }
}

static int slot_of_op(int op) { return op <= XP_OP_MOD ? op : op <= XP_OP_MAX ? op - XP_OP_MIN + 5 : op - XP_OP_SHL + 7; }

static JoinSeg new_join_seg(int sketch, int hole, int acc, int k, u64 lo, u64 hi) {
    JoinSeg sg;
    memset(&sg, 0, sizeof(sg));
    sg.rank_begin = lo; sg.rank_end = hi;
    sg.sketch = sketch; sg.hole = hole; sg.size = k; sg.acc = acc;
    return sg;
}

// Operands of (nt, size) counted by class (class_operand walks them in the same order); without classes, all of them.
static u64 class_operands(const xp_grammar* g, const HoleHost& ho, int nt, int size) {
    if (ho.cls_size == 0 || size < ho.cls_size) return g->cnt[nt][size];
    auto side = [&](int n, int k) { return k == ho.cls_size ? (u64)ho.cls_n[n] : g->cnt[n][k]; };
    if (size <= ho.tab_max) return side(nt, size);
    u64 sum = 0;
    for (int b = g->bin_begin[nt]; b < g->bin_begin[nt + 1]; ++b)
        for (int a = 1; a <= size - 2; ++a) {
            const int l = g->bins[b].lnt, r = g->bins[b].rnt, z = size - 1 - a;
            sum += a > ho.tab_max || z > ho.tab_max ? g->cnt[l][a] * g->cnt[r][z] : side(l, a) * side(r, z);
        }
    return sum;
}

enum RangeSplit { kSplitNone, kSplitClasses, kSplitAll };     // which comparing contexts have a segment per operator and side

// Leaf-join segments of (start nonterminal, size k >= 3) restricted to ranks [lo, hi): one per operand nonterminal, with
// a group per leaf nonterminal, for every operator with a leaf of it on either side of such an operand.  Copies of one
// production open segments of their own; so do shifts, which only the exact form knows.
static void add_joins(Plan* plan, const xp_grammar* g, const HoleHost& ho, int sketch, int hole, int acc, int k, u64 lo, u64 hi, RangeSplit split) {
    const int nt = ho.start_nt;
    const bool exact = ho.exact, compares = ho.compares;
    struct Open { JoinSeg seg; bool shifts; std::vector<JoinGroup> groups; };
    std::vector<Open> open;
    for (int b = g->bin_begin[nt]; b < g->bin_begin[nt + 1]; ++b) {
        const BinDev& bd = g->bins[b];
        u64 base = bd.off[k];
        for (int a = 1; a <= k - 2; ++a) {
            const u64 cl = g->cnt[bd.lnt][a], cr = g->cnt[bd.rnt][k - 1 - a];
            const u64 block = cl * cr;
            const u64 this_base = base;
            base += block;
            if (block == 0 || (a != 1 && a != k - 2)) continue;
            if (this_base + block <= lo || this_base >= hi) continue;
            const u64 wlo = lo > this_base ? lo - this_base : 0, whi = hi - this_base < block ? hi - this_base : block;
            const int swap = a == k - 2 ? 0 : 1;             // (k == 3: both operands are leaves; the left one is the operand)
            const int ent = swap ? bd.rnt : bd.lnt, lnt = swap ? bd.lnt : bd.rnt;
            u64 e0 = 0, e1 = swap ? cr : cl;                 // operands that the window covers
            if (!swap) { e0 = wlo / cr; e1 = (whi + cr - 1) / cr; }
            else if (wlo / cr == (whi - 1) / cr) { e0 = wlo % cr; e1 = (whi - 1) % cr + 1; }
            const int slot = slot_of_op(bd.op);
            const bool shifts = slot >= 7, ex = exact || shifts;      // (`exact` is the hole's; comparing contexts and classes make further segments below, for few sketches)
            Open* at = nullptr;
            JoinGroup* grp = nullptr;
            for (size_t i = 0; i < open.size() && !at; ++i) {
                Open& c = open[i];
                if (c.seg.nt != ent || c.shifts != shifts) continue;
                grp = nullptr;
                for (JoinGroup& q : c.groups) if (q.leaf_nt == lnt) grp = &q;
                if (grp ? !(((swap ? grp->smask : grp->fmask) >> slot) & 1u) : c.groups.size() < (size_t)kJoinGroups) at = &c;
            }
            if (!at) {
                Open c;
                c.shifts = shifts;
                c.seg = new_join_seg(sketch, hole, acc, k, lo, hi);
                c.seg.kind = kJoinLeaf; c.seg.nt = ent; c.seg.esize = k - 2; c.seg.exact = ex ? kExactMany : 0; c.seg.heavy = ex || compares ? 1 : 0;
                c.seg.e_begin = e0; c.seg.e_count = e1 - e0;
                open.push_back(c);
                at = &open.back();
                grp = nullptr;
            }
            if (!grp) {
                JoinGroup q;
                memset(&q, 0, sizeof(q));
                q.leaf_nt = lnt;
                at->groups.push_back(q);
                grp = &at->groups.back();
            }
            JoinSeg& sg = at->seg;
            const u64 end = sg.e_begin + sg.e_count;
            if (e0 < sg.e_begin) sg.e_begin = e0;
            sg.e_count = (e1 > end ? e1 : end) - sg.e_begin;
            (swap ? grp->smask : grp->fmask) |= 1u << slot;
            grp->base[swap][slot] = this_base;
        }
    }
    for (Open& c : open) {
        c.seg.first_group = (i32)plan->jgroups.size();
        c.seg.n_groups = (i32)c.groups.size();
        for (const JoinGroup& q : c.groups) if ((g->wide_leaf >> q.leaf_nt) & 1u) { c.seg.exact = kExactMany; c.seg.heavy = 1; }
        for (const JoinGroup& q : c.groups) c.seg.chunk += (u32)g->cnt[q.leaf_nt][1];
        // (a rank window may cover fewer operands than there are combinations of classes)
        if (!c.seg.exact && ho.cls_size > 0 && c.seg.esize >= ho.cls_size) {
            const u64 m = class_operands(g, ho, c.seg.nt, c.seg.esize);
            if (m > 0 && m < c.seg.e_count) { c.seg.classes = 1; c.seg.e_begin = c.seg.e_count; c.seg.e_count = m; }
        }
        // An operand of a context that compares takes some hundred microseconds of a lane, and classes leave a few thousand of them: a
        // segment per operator and side, so that as many warps share them (three conv holes: join 540 -> 430 us).
        if ((split == kSplitAll || (split == kSplitClasses && c.seg.classes)) && compares && !c.seg.exact && c.seg.e_count <= kRangeSplit) {
            c.seg.parts = kRangeParts;
            for (const JoinGroup& q : c.groups)
                for (int b = 0; b < 2 * kOpSlots; ++b) {
                    const int swap = b / kOpSlots, slot = b % kOpSlots;
                    if (!(((swap ? q.smask : q.fmask) >> slot) & 1u)) continue;
                    JoinGroup one = q;
                    one.fmask = swap ? 0u : 1u << slot; one.smask = swap ? 1u << slot : 0u;
                    c.seg.first_group = (i32)plan->jgroups.size();
                    c.seg.n_groups = 1;
                    plan->jgroups.push_back(one);
                    plan->jsegs.push_back(c.seg);
                }
            continue;
        }
        plan->jgroups.insert(plan->jgroups.end(), c.groups.begin(), c.groups.end());
        plan->jsegs.push_back(c.seg);
    }
}

// Every candidate of the window on its own, from the subtree tables.
static void add_direct(Plan* plan, int nt, int sketch, int hole, int acc, int k, u64 lo, u64 hi) {
    JoinSeg sg = new_join_seg(sketch, hole, acc, k, lo, hi);
    sg.kind = kJoinDirect; sg.nt = nt; sg.esize = k;
    sg.e_begin = lo; sg.e_count = hi - lo;
    plan->jsegs.push_back(sg);
}

// Small calls are bound by the chain of a ticket: conditions, suspects taken apart, probes one after the other.  Where all the
// operands of a segment times its leaves are few, every one is tested at both probes instead (join_few), a ticket being 32 operands and a part
// of the leaves, so that the call has a ticket for every warp.  (Two-variable nest, load and search:
// 179 -> 168 us; tile bound 267 -> 213, expression pair 373 -> 313, means of five inputs, with the probes of a check four at a time.)
constexpr u64 kFewPairs = 1ull << 20;        // (operand, leaf) pairs of a segment
constexpr u64 kFewCall = 1ull << 23;         // ... and of all such segments of a call

// Tickets of the leaf join.  A step is 32 operands (one per lane).  A ticket takes so
// many steps that every warp of the device gets about four: fewer and the last wave is uneven, more and the
// warps spend their time taking tickets.  64 steps at most.  In the exact form a ticket is one step, which costs as much as some
// hundred others; with fewer steps than two for every warp it is one operand, so that the warps share those.
static void number_joins(Plan* plan, size_t n_sketches) {
    if (plan->jsegs.empty()) return;
    // the heavy tickets of a few large sketches first, so that none of them is a call's last (batches are long enough to even out)
    if (plan->jsegs.size() <= 64 || n_sketches <= kPairMaxSketches)
        std::stable_partition(plan->jsegs.begin(), plan->jsegs.end(), [](const JoinSeg& c) { return c.heavy != 0; });
    u64 steps = 0, exact_steps = 0;
    for (const JoinSeg& c : plan->jsegs) (c.exact ? exact_steps : steps) += (c.e_count + 31) / 32;
    const u64 warps = (u64)search_warps();
    u64 few_pairs = 0, few_steps = 0;
    auto few = [](const JoinSeg& c) { return c.kind == kJoinLeaf && !c.exact && !c.heavy && !c.classes && c.chunk > 0 && c.e_count * (u64)c.chunk <= kFewPairs; };
    for (const JoinSeg& c : plan->jsegs) if (few(c)) { few_pairs += c.e_count * (u64)c.chunk; few_steps += (c.e_count + 31) / 32; }
    const u64 share = few_pairs <= kFewCall && few_steps > 0 ? (warps > few_steps ? warps / few_steps : 1) : 0;      // parts, if the leaves are enough
    const i32 form = exact_steps < 2 * warps ? kExactFew : kExactMany;
    u64 per = steps / (warps * 4);
    if (per < 1) per = 1;
    if (per > 64) per = 64;
    if (per >= 4) per &= ~3ull;
    plan->join_wide = per >= 4;
    for (JoinSeg& c : plan->jsegs) {
        if (c.exact) c.exact = form;
        c.first_ticket = plan->n_join;
        if (share && few(c)) {
            const u64 most = ((u64)c.chunk + 3) / 4, parts = share < most ? share : most;
            c.chunk = 32;
            c.parts = (int16_t)(parts < 32767u ? parts : 32767u);
        } else c.chunk = (u32)(c.exact ? (form == kExactFew ? 1 : 32) : c.parts > 0 ? 32 : per * 32);
        plan->n_join += (c.e_count + c.chunk - 1) / c.chunk * (u64)(c.parts > 0 ? c.parts : 1);
    }
}

constexpr u64 kTileMinRanks = 4096;          // smaller windows are searched rank by rank

// Matches (candidates that satisfy the probes with tables, by the load's sample) that a call's comparing contexts may have for their operands to go by
// class.  With more the list of members_kernel runs over, and where most candidates of an operand match, sharing the operands among the
// warps shares the work best.  (100 guards of 29, 40 and 60 leaves, 1000 of 29, a quarter of them nearly always true: 1.7e6, 6e6, 2.6e7, 1.2e7 by the sample;
// 95, 361, 1131, 715 ms operand by operand, 18, 870, 4500, 1190 by class.  An affine context has few matches per operand: the examples in
// xp_classes.cuh are 2e7 by the sample.)
constexpr double kClassMatches = 4.0;                     // ... for each entry of the survivor queue
// Candidates of such contexts, likewise: the sample does not see what is rarer than one in 256.  (On the fixed scratch, with its 8192 entries: guards of 29 and 60
// leaves, 1.2e6 and 1.1e7 candidates, 0.18, 0.36 ms operand by operand, 0.10, 0.15 by class; 20 of 12 leaves, size 7, 3.5e7 each, 28.7 against 41 to 60.)
constexpr double kClassCandidates = 2048.0;
// Matches of affine contexts: 136 leaves, size 7, 131 072 points, a target that is a variable (8.3e8 by the sample, 9.4e7 in fact): 48 s operand by operand, 101 by class.
constexpr double kClassMatchesAffine = 256.0;

// What a plan may use: kFormMany, a batch: no pair join; the others, at most kPairMaxSketches sketches: narrow tiles where a block is small, and
// without the pair join, with it from kPairLeastBatch pairs on, or from kPairLeast on.  kFormDozens: a batch of up to kRangeSketches, in which comparing
// contexts over classes are still cut into segments by operator: a tenth of the operands leaves too few tickets otherwise (10 guards of 29, 40 and 60
// leaves: search 0.49, 0.74, 1.04 ms operand by operand, 0.56, 0.75, 1.01 by class in one segment, 0.37, 0.53, 0.80 so).
constexpr size_t kRangeSketches = 64;
// A larger batch goes by operand where fewer than one sketch in so many has a comparing hole with classes: these would take the whole call to the longer
// form of the leaf join (500 sketches, 5 of them guards: search 2.19 ms, 2.39 so).
constexpr size_t kClassShare = 16;
enum PlanForm { kFormMany = 0, kFormTiles = 1, kFormPairsSome = 2, kFormPairs = 3, kFormDozens = 4, kForms = 5 };
// Classes of comparing holes: all, not where the sample has matches, none; kUseSparseAffine (beside these): of the others not where it has some.
enum ClassUse { kUseAll = 0, kUseSparse = 1, kUseFew = 2, kUseSparseAffine = 4 };
static void plan_sketch(const xp_sketch* s, size_t i, const xp_repair_opts* o, PlanForm form, ClassUse use, Plan* plan);

// A sketch's tables, and the library's scratch, live on the device that was current when the sketch was
// loaded: a call made with another device current would hand the kernels pointers of the wrong GPU.
static xp_status check_device(const xp_sketch* const* sk, size_t n) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return fail(XP_ERR_CUDA, "no CUDA device is usable");
    for (size_t i = 0; i < n; ++i)
        if (sk[i] && sk[i]->arena_device != dev)
            return fail(XP_ERR_INVALID_ARG, "sketch " + std::to_string(i) + " was loaded on device " + std::to_string(sk[i]->arena_device) +
                        ", the current device is " + std::to_string(dev));
    return XP_OK;
}

// (may_pair: the call's scratch has room for the pair join's index; queue: entries of its survivor queue)
static xp_status build_plan(const xp_sketch* const* sk, size_t n, const xp_repair_opts* o, bool may_pair, u32 queue, Plan* plan) {
    // the pair join takes its blocks one after the other, several launches each: a batch keeps to the tiles, which
    // search all holes in one launch.  So does a call with a cancel word or a time limit: its launches are bounded, and the
    // host looks at both between them; a pair join's launch covers a whole block.
    const bool pairs = may_pair && !o->cancel && o->timeout_ms <= 0;
    const PlanForm form = n > kRangeSketches ? kFormMany : n > kPairMaxSketches ? kFormDozens : !pairs ? kFormTiles : n > kPairFew ? kFormPairsSome : kFormPairs;
    const bool plain = o->size_min <= 0 && o->size_max <= 0 && o->n_rank_ranges == 0 && o->flags == 0;
    double candidates = 0, matches = 0, affine = 0;       // of comparing holes with classes; matches by the sample, and those of the other holes with some
    size_t with = 0;                                      // sketches that have some
    for (size_t i = 0; i < n; ++i)
        if (sk[i]) {
            bool some = false;
            for (const HoleHost& h : sk[i]->holes) {
                if (h.cls_size == 0) continue;
                if (!h.compares) {
                    for (int k = 1; k <= h.max_size; ++k) affine += h.pass_rate * (double)sk[i]->g->cnt[h.start_nt][k];
                    continue;
                }
                some = true;
                for (int k = 1; k <= h.max_size; ++k) {
                    const double c = (double)sk[i]->g->cnt[h.start_nt][k];
                    candidates += c; matches += h.pass_rate * c;
                }
            }
            with += some ? 1u : 0u;
        }
    const int left_out = (form == kFormMany && with * kClassShare < n) || candidates > kClassCandidates * queue ? kUseFew : matches > kClassMatches * queue ? kUseSparse : kUseAll;
    const ClassUse use = (ClassUse)(left_out | (affine > kClassMatchesAffine * queue ? kUseSparseAffine : 0));
    if (n > 16) { plan->segs.reserve(n * 8); plan->acc.reserve(n * 2); plan->nominal_ops.reserve(n * 2); }
    for (size_t i = 0; i < n; ++i) {
        const xp_sketch* s = sk[i];
        if (!s) return fail(XP_ERR_INVALID_ARG, "null sketch in batch");
        if (!plain || plan->whole) { plan_sketch(s, i, o, form, use, plan); continue; }
        const Plan* own;
        {
            std::lock_guard<std::mutex> lock(s->plan_mu);
            std::unique_ptr<const Plan>& kept = s->plan_kept[form + kForms * use];
            if (!kept) {
                std::unique_ptr<Plan> made(new Plan);
                plan_sketch(s, 0, o, form, use, made.get());
                made->acc.clear();                        // (made per call, below)
                kept = std::move(made);
            }
            own = kept.get();
        }
        const int acc_base = (int)plan->acc.size();
        AccDev a;
        memset(&a, 0, sizeof(a));
        for (int k = 0; k <= kMaxSize; ++k) a.min_rank[k] = ~0ull;
        for (int h = 0; h < s->n_holes; ++h) { plan->acc.push_back(a); plan->nominal_ops.push_back(own->nominal_ops[h]); }
        const size_t at = plan->segs.size();
        plan->segs.insert(plan->segs.end(), own->segs.begin(), own->segs.end());
        for (size_t j = at; j < plan->segs.size(); ++j) {
            SegDev& c = plan->segs[j];
            c.first_ticket += plan->n_tickets;
            c.sketch = (i32)i;
            c.acc += acc_base;
        }
        plan->n_tickets += own->n_tickets;
        const size_t jat = plan->jsegs.size();
        plan->jsegs.insert(plan->jsegs.end(), own->jsegs.begin(), own->jsegs.end());
        for (const PairSeg& ps : own->psegs) { plan->psegs.push_back(ps); plan->psegs.back().sketch = (i32)i; plan->psegs.back().acc += acc_base; }
        const i32 group_base = (i32)plan->jgroups.size();
        plan->jgroups.insert(plan->jgroups.end(), own->jgroups.begin(), own->jgroups.end());
        for (size_t j = jat; j < plan->jsegs.size(); ++j) {
            plan->jsegs[j].sketch = (i32)i; plan->jsegs[j].acc += acc_base; plan->jsegs[j].first_group += group_base;
        }
    }
    number_joins(plan, n);
    return XP_OK;
}

// One sketch's segments, accumulators and tickets, appended to the plan as sketch number i.
static void plan_sketch(const xp_sketch* s, size_t i, const xp_repair_opts* o, PlanForm form, ClassUse use, Plan* plan) {
    std::vector<u32> taken;
    {
        for (int h = 0; h < s->n_holes; ++h) {
            HoleHost ho = s->holes[h];
            const int left_out = use & 3;
            if (ho.compares ? left_out == kUseFew || (left_out == kUseSparse && ho.pass_rate > 0) : (use & kUseSparseAffine) && ho.pass_rate > 0) ho.cls_size = 0;
            AccDev a;
            memset(&a, 0, sizeof(a));
            for (int k = 0; k <= kMaxSize; ++k) a.min_rank[k] = ~0ull;
            const int acc = (int)plan->acc.size();
            plan->acc.push_back(a);
            plan->nominal_ops.push_back(0);
            int kmin = 1, kmax = ho.max_size;
            if (o->size_min > 0) kmin = o->size_min;
            if (o->size_max > 0 && o->size_max < kmax) kmax = o->size_max;
            for (int k = kmin; k <= kmax && !ho.never; ++k) {
                u64 lo = 0, hi = s->g->cnt[ho.start_nt][k];
                for (int r = 0; r < o->n_rank_ranges; ++r) {
                    const xp_rank_range& rr = o->rank_ranges[r];
                    if ((rr.hole == -1 || rr.hole == h) && rr.size == k) {
                        if (rr.begin > lo) lo = rr.begin;
                        if (rr.end < hi) hi = rr.end;
                    }
                }
                if (lo >= hi) continue;
                const bool forced = (o->flags & XP_FLAG_ALWAYS_FILTER) != 0;
                if (!ho.filter_ok || (o->flags & XP_FLAG_NO_FILTER)) { add_linear(plan, (int)i, h, acc, k, lo, hi); continue; }
                if (k < 3 || (!forced && hi - lo < kTileMinRanks)) { add_direct(plan, ho.start_nt, (int)i, h, acc, k, lo, hi); continue; }
                // (A range of hole values: the join's interval arithmetic per operand against a test per candidate.  27 leaves, size 7, 984 000
                // operands, four specs: 13.4, 26.5, 10.2, 14.4 ms by the join, 14.9, 19.8, 10.7, 8.2 as tiles; 40 leaves, size 5: 0.4 against 1.4.
                // What decides is the operands, not their classes: with so many the tables hold few probes, and a class is taken apart for each
                // candidate that passes those.  40 leaves, size 7, 3.2 million operands, three specs: 210, 1290, 212 ms as tiles, 2270, 4220,
                // 2400 by the join over classes; with a shift 144, 128 against 1500, 159, with a leaf of 2^33 119, 965 against 64, 807.)
                const bool leaves = ho.compares && s->g->cnt[ho.start_nt][k - 2] > kRangeMost;
                if (!leaves) add_joins(plan, s->g, ho, (int)i, h, acc, k, lo, hi, plan->whole || form == kFormMany || (use & 3) == kUseFew ? kSplitNone : form == kFormDozens ? kSplitClasses : kSplitAll);
                const bool pairs = form == kFormPairsSome || form == kFormPairs;
                if (pairs) add_pairs(plan, s->g, ho, (int)i, h, acc, k, lo, hi, o->flags & XP_FLAG_ALWAYS_PAIR ? 1 : form == kFormPairs ? kPairLeast : kPairLeastBatch, &taken);
                add_tiles(plan, s->g, pairs ? &taken : nullptr, ho.start_nt, (int)i, h, acc, k, lo, hi, ho.compares ? kBcTileSlow : kBcTile, form != kFormMany && form != kFormDozens, leaves);
            }
        }
    }
}

// Survivor queue entries of a call with its own workspace.  A survivor that finds the queue full is checked by the warp that has it, alone
// and at once, at some ten times the cost (a loop bound in a guard, 133 503 survivors on 65 536 points: 254 ms with 65 536
// entries, 13 with 2^20).  A caller's workspace made for fewer entries is taken with as many as it holds, from surv_least on.
constexpr u32 kSurvMost = 1u << 20;          // (42 MB)
static u32 surv_least(size_t n_sketches) {
    const size_t want = n_sketches * 256;
    return (u32)(want < 65536 ? 65536 : (want > kSurvMost ? kSurvMost : want));
}
constexpr u32 kSurvCapStatic = 8192;         // ... of a call on the library's fixed scratch

// Scratch of a pair-join block beside its chain heads: counters and histograms (zero at launch), and what kernels fill.
constexpr size_t kPairZeros = 256 + 2 * 4096;
static size_t pair_rest_bytes(const PairSeg& c) {
    const size_t nl = c.nl, nr = c.nr;
    return align256(sizeof(u32) * (c.index_right ? nr : nl)) + align256(sizeof(u32) * nl) + align256(sizeof(u32) * nr) +
           ((c.ops & 24u) ? align256(sizeof(uint2) * (size_t)pair_list_entries(c.nl, c.nr)) + 2 * align256(sizeof(u32) * 1025) + align256(12 * nl) + align256(12 * nr) + 512 : 0);
}
static void pair_place(PairSeg& c, char* ones, char* zeros, char* rest) {
    const size_t nl = c.nl, nr = c.nr;
    c.head = (u32*)ones;
    c.counters = (u32*)zeros;
    c.ticket = (u64*)(zeros + 64);
    c.hist[0] = (u32*)(zeros + 256); c.hist[1] = (u32*)(zeros + 256 + 4096);
    auto take = [&](size_t bytes) { char* p = rest; rest += align256(bytes); return p; };
    c.next = (u32*)take(sizeof(u32) * (c.index_right ? nr : nl));
    c.wide_l = (u32*)take(sizeof(u32) * nl);
    c.wide_r = (u32*)take(sizeof(u32) * nr);
    if (c.ops & 24u) {
        c.far = (uint2*)take(sizeof(uint2) * (size_t)pair_list_entries(c.nl, c.nr));
        for (int k = 0; k < 2; ++k) {
            const size_t n = k ? nr : nl;
            c.start[k] = (u32*)take(sizeof(u32) * 1025);
            char* p = take(12 * n);
            c.val[k] = (int2*)p;
            c.id[k] = (u32*)(p + 8 * n);
        }
    }
}

static SearchLayout ws_layout(const Plan& plan, const xp_sketch* const* sk, size_t n_sketches, u32 surv_cap) {
    SearchLayout w;
    const size_t n_acc = plan.acc.size();
    w.segs = 256;
    w.jsegs = w.segs + align256(sizeof(SegDev) * plan.segs.size());
    w.jgroups = w.jsegs + align256(sizeof(JoinSeg) * plan.jsegs.size());
    w.psegs = w.jgroups + align256(sizeof(JoinGroup) * plan.jgroups.size());
    w.sketches = w.psegs + align256(sizeof(PairSeg) * plan.psegs.size());
    w.acc = w.sketches + align256(sizeof(SketchDev*) * (n_sketches + 1));
    w.hist = w.acc + align256(sizeof(AccDev) * (n_acc + 1));
    w.head = w.hist + align256(sizeof(u32) * (n_acc + 1));
    w.surv = w.head;
    w.sort_off = w.surv + align256(sizeof(SurvDev) * (size_t)surv_cap);
    w.sorted = w.sort_off + align256(sizeof(u32) * (n_acc + 2));
    w.longs = w.sorted + align256(sizeof(u32) * (size_t)surv_cap);
    w.total = w.longs + align256(sizeof(u32) * (size_t)surv_cap);
    // (the list of what candidates over classes stand for is where the hole order will be: that is made once the list has been worked off)
    bool classes = false;
    for (const JoinSeg& c : plan.jsegs) classes = classes || c.classes;
    for (const PairSeg& c : plan.psegs) classes = classes || c.lcls || c.rcls;
    w.member_cap = classes ? (u32)(sizeof(u32) * (size_t)surv_cap / sizeof(MemberRec)) : 0;
    w.n_psegs = (int)plan.psegs.size();
    w.pair_ones = w.total;
    for (const PairSeg& c : plan.psegs) w.total += align256(sizeof(u32) * ((size_t)c.head_mask + 1));
    w.pair_zeros = w.total;
    for (size_t i = 0; i < plan.psegs.size(); ++i) w.total += kPairZeros;
    w.pair_rest = w.total;
    for (const PairSeg& c : plan.psegs) w.total += pair_rest_bytes(c);
    w.n_acc = (int)n_acc; w.n_segs = (int)plan.segs.size(); w.n_jsegs = (int)plan.jsegs.size(); w.n_sketches = (int)n_sketches;
    w.surv_cap = surv_cap;
    w.join_wide = plan.join_wide ? 1 : 0;
    // (the longer form is for classes, tickets in parts, and few sketches whose tickets are one wave: with more the warps hide the chain
    // of a check, and it is the shorter code that counts.  A quasi-affine
    // grammar with 4.1 million operands, size 9, two targets: 511, 193 ms, in the longer form 577, 224.)
    const bool wave = n_sketches <= kPairMaxSketches && plan.n_join <= (u64)search_warps();
    w.join_batch = 1;
    for (const JoinSeg& c : plan.jsegs)
        if (c.classes || c.parts > 0 || (c.kind != kJoinDirect && wave)) { w.join_batch = 0; break; }
    i64 most = 0;
    w.dense = w.empty_domain = 0;
    for (size_t i = 0; i < n_sketches; ++i) {
        most = sk[i]->n_points > most ? sk[i]->n_points : most;
        if (sk[i]->n_points == 0) w.empty_domain = 1;
        for (const HoleHost& h : sk[i]->holes) if (h.second) w.dense = 1;      // (frequent filter hits)
    }
    w.max_chunks = (u32)((most + kVerifyChunk - 1) / kVerifyChunk);
    w.first_points = (i32)(most < kVerifyChunk ? most : kVerifyChunk);
    return w;
}

// The smallest size with a match (0: none).
static int least_size(const AccDev& a, int max_size) {
    for (int k = 1; k <= max_size; ++k) if (a.match_count[k] > 0) return k;
    return 0;
}

// What a call sends to the device in one copy: counters at zero, segments, sketches, accumulators in their start state.
static void stage_plan(char* stage, char* ws, const SearchLayout& w, Plan& plan, const xp_sketch* const* sketches) {
    memset(stage, 0, 256);
    if (!plan.segs.empty()) memcpy(stage + w.segs, plan.segs.data(), sizeof(SegDev) * plan.segs.size());
    if (!plan.jsegs.empty()) memcpy(stage + w.jsegs, plan.jsegs.data(), sizeof(JoinSeg) * plan.jsegs.size());
    {
        char *ones = ws + w.pair_ones, *zeros = ws + w.pair_zeros, *rest = ws + w.pair_rest;
        for (PairSeg& c : plan.psegs) {
            pair_place(c, ones, zeros, rest);
            ones += align256(sizeof(u32) * ((size_t)c.head_mask + 1)); zeros += kPairZeros; rest += pair_rest_bytes(c);
        }
        if (!plan.psegs.empty()) memcpy(stage + w.psegs, plan.psegs.data(), sizeof(PairSeg) * plan.psegs.size());
    }
    if (!plan.jgroups.empty()) memcpy(stage + w.jgroups, plan.jgroups.data(), sizeof(JoinGroup) * plan.jgroups.size());
    for (int i = 0; i < w.n_sketches; ++i) ((const SketchDev**)(stage + w.sketches))[i] = sketches[i]->d_s;
    memcpy(stage + w.acc, plan.acc.data(), sizeof(AccDev) * plan.acc.size());
    memset(stage + w.hist, 0, w.head - w.hist);
}

extern "C" size_t xp_workspace_bytes(const xp_sketch* const* sketches, size_t n, const xp_repair_opts* opts) {
    if (!sketches || n == 0) return 0;
    Plan plan;
    if (build_plan(sketches, n, opts ? opts : &kDefaultOpts, true, kSurvMost, &plan) != XP_OK) return 0;
    return ws_layout(plan, sketches, n, kSurvMost).total;
}

extern "C" xp_status xp_repair_batch(const xp_sketch* const* sketches, size_t n, const xp_repair_opts* opts,
                                     xp_result** outs) {
    if (!sketches || !outs || n == 0) return fail(XP_ERR_INVALID_ARG, "xp_repair_batch: null argument");
    for (size_t i = 0; i < n; ++i) outs[i] = nullptr;
    const xp_repair_opts* o = opts ? opts : &kDefaultOpts;
    if (o->n_rank_ranges < 0 || (o->n_rank_ranges > 0 && !o->rank_ranges)) return fail(XP_ERR_INVALID_ARG, "bad rank_ranges");
    if (o->cancel && *o->cancel) return fail(XP_ERR_CANCELLED, "cancelled before launch");
    const auto t0 = std::chrono::steady_clock::now();
    Plan plan;
    xp_status st = build_plan(sketches, n, o, true, kSurvMost, &plan);
    if (st == XP_OK) st = check_device(sketches, n);
    if (st != XP_OK) return st;
    cudaStream_t stream = (cudaStream_t)o->stream;

    SearchLayout w = ws_layout(plan, sketches, n, kSurvMost);
    char* ws = (char*)o->workspace;
    auto shrink = [&]() {                                 // to the caller's workspace, if the queue can be made small enough
        for (u32 cap = kSurvMost; w.total > o->workspace_bytes && cap > surv_least(n);) {
            cap = cap / 2 > surv_least(n) ? cap / 2 : surv_least(n);
            w = ws_layout(plan, sketches, n, cap);
        }
    };
    if (ws) shrink();
    if (ws && o->workspace_bytes < w.total && !plan.psegs.empty()) {
        // A refinement can change which blocks the pair join may take (a target that is no longer zero), and so what a call
        // needs: a caller's workspace made before it holds the plan without the pair join.
        plan = Plan();
        st = build_plan(sketches, n, o, false, kSurvMost, &plan);
        if (st != XP_OK) return st;
        w = ws_layout(plan, sketches, n, kSurvMost);
        shrink();
    }
    bool own_ws = false, cached_ws = false;
    if (ws) {
        if (o->workspace_bytes < w.total || ((uintptr_t)ws & 255)) return fail(XP_ERR_NOMEM, "workspace too small or misaligned");
    } else if (g_ws_mu.try_lock()) {
        // the library's own scratch, kept from call to call (grown when a call needs more)
        cached_ws = true;
        int dev = -1;
        cudaGetDevice(&dev);
        if (g_ws_bytes < w.total || g_ws_device != dev) {
            if (g_ws) cudaFree(g_ws);                // (a block of another device is freed from here as well)
            g_ws_device = dev;
            g_ws = nullptr; g_ws_bytes = 0;
            cudaError_t e = cudaMalloc((void**)&g_ws, w.total);
            if (e != cudaSuccess) { g_ws_mu.unlock(); return fail(XP_ERR_NOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e)); }
            g_ws_bytes = w.total;
        }
        ws = g_ws;
    } else {                                       // another call holds the kept scratch
        XP_CUDA(cudaMalloc((void**)&ws, w.total));
        own_ws = true;
    }
    float ms = 0.f;
    int launches = 0;
    const size_t n_acc = plan.acc.size(), acc_bytes = sizeof(AccDev) * n_acc;
    StageBlock stage(w.head + acc_bytes + 256);
    EventPair ev;
    auto give_back = [&]() { if (own_ws) cudaFree(ws); if (cached_ws) g_ws_mu.unlock(); };
#define XP_CUDA_R(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) { cudaStreamSynchronize(stream); give_back(); \
        return fail(e_ == cudaErrorMemoryAllocation ? XP_ERR_NOMEM : XP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); } } while (0)
    if (!stage.p) { give_back(); return fail(XP_ERR_NOMEM, "out of host memory"); }
    stage_plan(stage.p, ws, w, plan, sketches);
    const AccDev* acc = (const AccDev*)(stage.p + w.head);
    u32* check_word = (u32*)(stage.p + w.head + acc_bytes);
    *check_word = 0;
    XP_CUDA_R(ev.open());
    XP_CUDA_R(cudaMemcpyAsync(ws, stage.p, w.head, cudaMemcpyHostToDevice, stream));
    XP_CUDA_R(cudaEventRecord(ev.e0, stream));
    xp_status stopped = XP_OK;
    auto give_up = [&](bool more) {                       // after a bounded launch
        if (o->cancel && *o->cancel) return XP_ERR_CANCELLED;
        const double spent = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
        return o->timeout_ms > 0 && more && spent >= (double)o->timeout_ms ? XP_ERR_TIMEOUT : XP_OK;
    };
    if (!o->cancel && o->timeout_ms <= 0) {
        XP_CUDA_R(launch_search_part(ws, w, true, 0, plan.n_join, false, stream, &launches));
        XP_CUDA_R(launch_search_part(ws, w, false, 0, plan.n_tickets, false, stream, &launches));
    } else {
        // Bounded launches: the host waits for each and then looks at the cancel word and the clock.
        // Nothing on the device waits for either, and when the call gives up no kernel is in flight.
        for (int kind = 0; kind < 2 && stopped == XP_OK; ++kind) {
            const u64 n_items = kind == 0 ? plan.n_join : plan.n_tickets;
            for (u64 t = 0; t < n_items && stopped == XP_OK; t += (u64)XP_CANCEL_TICKETS) {
                const u64 t_end = t + (u64)XP_CANCEL_TICKETS < n_items ? t + (u64)XP_CANCEL_TICKETS : n_items;
                XP_CUDA_R(launch_search_part(ws, w, kind == 0, t, t_end, t > 0, stream, &launches));
                XP_CUDA_R(cudaStreamSynchronize(stream));
                stopped = give_up(t_end < n_items || (kind == 0 && plan.n_tickets > 0));
            }
        }
    }
    if (stopped == XP_OK) {
        XP_CUDA_R(launch_pairs(ws, w, plan.psegs.data(), stream, &launches));
        if (!o->cancel && o->timeout_ms <= 0) XP_CUDA_R(launch_members(ws, w, 0, ~0ull, false, stream, &launches));
    }
    if (stopped == XP_OK && (o->cancel || o->timeout_ms > 0) && w.member_cap > 0) {
        // (in bounded launches too; how many pieces there are is known by now)
        u64* listed = (u64*)(check_word + 2);
        XP_CUDA_R(cudaMemcpyAsync(listed, ws + 48, sizeof(*listed), cudaMemcpyDeviceToHost, stream));
        XP_CUDA_R(cudaStreamSynchronize(stream));
        const u64 pieces = *listed & ((1ull << 44) - 1);
        for (u64 t = 0; (t == 0 || t < pieces) && stopped == XP_OK; t += (u64)XP_CANCEL_TICKETS) {
            const u64 end = t + (u64)XP_CANCEL_TICKETS < pieces ? t + (u64)XP_CANCEL_TICKETS : pieces;
            XP_CUDA_R(launch_members(ws, w, t, end, t > 0, stream, &launches));
            XP_CUDA_R(cudaStreamSynchronize(stream));
            stopped = give_up(end < pieces);
        }
    }
    if (stopped == XP_OK) {
        bool told = false;
        XP_CUDA_R(launch_search_end(ws, w, plan.n_tickets + plan.n_join + plan.psegs.size() > 0, stage.locked ? (AccDev*)(stage.p + w.head) : nullptr, &told, stream, &launches));
        XP_CUDA_R(cudaEventRecord(ev.e1, stream));
        if (!told) XP_CUDA_R(cudaMemcpyAsync(stage.p + w.head, ws + w.acc, acc_bytes, cudaMemcpyDeviceToHost, stream));
#ifdef XP_CHECKS
        XP_CUDA_R(cudaMemcpyAsync(check_word, ws + 20, sizeof(*check_word), cudaMemcpyDeviceToHost, stream));
#endif
        XP_CUDA_R(cudaStreamSynchronize(stream));
        XP_CUDA_R(cudaEventElapsedTime(&ms, ev.e0, ev.e1));
    }
#undef XP_CUDA_R
    give_back();
    if (stopped == XP_ERR_CANCELLED) return fail(stopped, "cancelled between launches (" + std::to_string(launches) + " done)");
    if (stopped == XP_ERR_TIMEOUT) return fail(stopped, "time limit of " + std::to_string((long long)o->timeout_ms) + " ms reached between launches (" + std::to_string(launches) + " done)");
    if (*check_word != 0) return fail(XP_ERR_CUDA, "an index check of the checked build failed (code " + std::to_string(*check_word) + ")");

    size_t ai = 0;
    for (size_t i = 0; i < n; ++i) {
        const xp_sketch* s = sketches[i];
        xp_result* r = new (std::nothrow) xp_result;
        if (!r) {
            for (size_t j = 0; j < i; ++j) { delete outs[j]; outs[j] = nullptr; }
            return fail(XP_ERR_NOMEM, "out of host memory");
        }
        r->holes.resize(s->n_holes);
        for (int h = 0; h < s->n_holes; ++h, ++ai) {
            HoleResult& hr = r->holes[h];
            const AccDev& a = acc[ai];
            hr.max_size = s->holes[h].max_size;
            for (int k = 1; k <= hr.max_size; ++k) {
                hr.cand_count[k] = s->g->cnt[s->holes[h].start_nt][k];
                hr.match_count[k] = a.match_count[k];
            }
            hr.evals = a.evals + a.filter_tests; hr.filter_survivors = a.filter_survivors; hr.probe_survivors = a.probe_survivors;
            hr.filter_tests = a.filter_tests;
            hr.skipped = a.tile_cands > a.filter_tests ? a.tile_cands - a.filter_tests : 0;
            hr.nominal_ops = plan.nominal_ops[ai] - (a.ops_skipped < plan.nominal_ops[ai] ? a.ops_skipped : plan.nominal_ops[ai]) + 2 * a.join_tests;
            const int ls = least_size(a, hr.max_size);
            if (ls >= 1) {
                hr.solved = 1; hr.least_size = ls; hr.least_rank = a.min_rank[ls];
                host_unrank(s->g, s->holes[h].start_nt, ls, hr.least_rank, &hr.code, &hr.text);
            }
        }
        r->kernel_ms = ms;
        r->n_launches = launches;
        r->h2d_bytes = w.head;
        r->d2h_bytes = acc_bytes;
        outs[i] = r;
    }
    const double total = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    for (size_t i = 0; i < n; ++i) outs[i]->total_ms = total;
    return XP_OK;
}

extern "C" xp_status xp_repair(const xp_sketch* sketch, const xp_repair_opts* opts, xp_result** out) {
    if (!sketch || !out) return fail(XP_ERR_INVALID_ARG, "xp_repair: null argument");
    return xp_repair_batch(&sketch, 1, opts, out);
}

// The search of one sketch with every byte of device scratch taken from a fixed array inside
// the library: no device memory is allocated or freed, no event or stream is created.
extern "C" xp_status xp_repair_static(const xp_sketch* sketch, const xp_repair_opts* opts, xp_hole_summary* out,
                                      int32_t out_cap) {
    if (!sketch || !out) return fail(XP_ERR_INVALID_ARG, "xp_repair_static: null argument");
    if (out_cap < sketch->n_holes) return fail(XP_ERR_INVALID_ARG, "xp_repair_static: out has fewer entries than the sketch has holes");
    const xp_repair_opts* o = opts ? opts : &kDefaultOpts;
    if (o->n_rank_ranges < 0 || (o->n_rank_ranges > 0 && !o->rank_ranges)) return fail(XP_ERR_INVALID_ARG, "bad rank_ranges");
    if (o->cancel && *o->cancel) return fail(XP_ERR_CANCELLED, "cancelled before launch");
    Plan plan;
    xp_status st = build_plan(&sketch, 1, o, false, kSurvCapStatic, &plan);
    if (st == XP_OK) st = check_device(&sketch, 1);
    if (st != XP_OK) return st;
    SearchLayout w = ws_layout(plan, &sketch, 1, kSurvCapStatic);
    if (w.total > kStaticScratchBytes) {                  // (many holes: the plan with the fewest segments)
        plan = Plan();
        plan.whole = true;
        st = build_plan(&sketch, 1, o, false, kSurvCapStatic, &plan);
        if (st != XP_OK) return st;
        w = ws_layout(plan, &sketch, 1, kSurvCapStatic);
    }
    if (plan.acc.size() > 64)
        return fail(XP_ERR_TOO_LARGE, "xp_repair_static: the sketch has more than 64 holes; use xp_repair with a workspace");
    if (w.total > kStaticScratchBytes)
        return fail(XP_ERR_TOO_LARGE, "xp_repair_static: the call needs " + std::to_string(w.total) +
                    " bytes of scratch, the fixed array holds " + std::to_string(kStaticScratchBytes) +
                    "; use xp_repair with a workspace");
    StageBlock stage(w.head + sizeof(AccDev) * plan.acc.size());       // (page-locked host memory that the library keeps)
    if (!stage.p) return fail(XP_ERR_NOMEM, "out of host memory");
    stage_plan(stage.p, nullptr, w, plan, &sketch);
    const AccDev* acc = (const AccDev*)(stage.p + w.head);
    cudaStream_t stream = (cudaStream_t)o->stream;
    cudaError_t e = launch_search_static(stage.p, w, plan.n_tickets, plan.n_join, (AccDev*)(stage.p + w.head), stage.locked, stream);
    const cudaError_t e2 = cudaStreamSynchronize(stream);         // (before the staging block goes back, whatever happened)
    if (e == cudaSuccess) e = e2;
    if (e != cudaSuccess) return fail(XP_ERR_CUDA, std::string("xp_repair_static: ") + cudaGetErrorString(e));
    for (int h = 0; h < sketch->n_holes; ++h) {
        xp_hole_summary& r = out[h];
        memset(&r, 0, sizeof(r));
        const AccDev& a = acc[h];
        r.max_size = sketch->holes[h].max_size;
        for (int k = 1; k <= r.max_size; ++k) {
            r.cand_count[k] = sketch->g->cnt[sketch->holes[h].start_nt][k];
            r.match_count[k] = a.match_count[k];
        }
        r.evals_executed = a.evals + a.filter_tests;
        const int ls = least_size(a, r.max_size);
        if (ls >= 1) {
            r.solved = 1; r.least_size = ls; r.least_rank = a.min_rank[ls];
            std::vector<xp_instr> code;
            std::string text;
            host_unrank(sketch->g, sketch->holes[h].start_nt, ls, r.least_rank, &code, &text);
            snprintf(r.least_text, sizeof(r.least_text), "%s", text.c_str());
        }
    }
    return XP_OK;
}

extern "C" xp_status xp_result_get(const xp_result* r, int32_t hole, xp_result_view* v) {
    if (!r || !v || hole < 0 || hole >= (int)r->holes.size()) return fail(XP_ERR_INVALID_ARG, "xp_result_get: bad argument");
    const HoleResult& h = r->holes[hole];
    v->solved = h.solved;
    v->max_size = h.max_size;
    v->cand_count = (const uint64_t*)h.cand_count;
    v->match_count = (const uint64_t*)h.match_count;
    v->least_size = h.least_size;
    v->least_rank = h.least_rank;
    v->least_code = h.code.data();
    v->least_len = (int)h.code.size();
    v->least_text = h.text.c_str();
    v->evals_executed = h.evals;
    v->filter_survivors = h.filter_survivors;
    v->probe_survivors = h.probe_survivors;
    v->nominal_ops = h.nominal_ops;
    v->kernel_ms = r->kernel_ms;
    v->total_ms = r->total_ms;
    v->n_launches = r->n_launches;
    v->filter_tests = h.filter_tests;
    v->candidates_skipped = h.skipped;
    v->h2d_bytes = r->h2d_bytes;
    v->d2h_bytes = r->d2h_bytes;
    return XP_OK;
}

extern "C" xp_status xp_result_pack(const xp_result* const* results, size_t n, xp_hole_summary* out, size_t out_cap, size_t* n_out) {
    if (n_out) *n_out = 0;
    if (!results || !out) return fail(XP_ERR_INVALID_ARG, "xp_result_pack: null argument");
    size_t at = 0;
    for (size_t i = 0; i < n; ++i) {
        if (!results[i]) return fail(XP_ERR_INVALID_ARG, "xp_result_pack: result " + std::to_string(i) + " is null");
        for (const HoleResult& h : results[i]->holes) {
            if (at >= out_cap) return fail(XP_ERR_INVALID_ARG, "xp_result_pack: out holds fewer entries than the results have holes");
            xp_hole_summary& r = out[at++];
            memset(&r, 0, sizeof(r));
            r.solved = h.solved; r.max_size = h.max_size; r.least_size = h.least_size; r.least_rank = h.least_rank;
            memcpy(r.cand_count, h.cand_count, sizeof(r.cand_count));
            memcpy(r.match_count, h.match_count, sizeof(r.match_count));
            r.evals_executed = h.evals;
            snprintf(r.least_text, sizeof(r.least_text), "%s", h.text.c_str());
        }
    }
    if (n_out) *n_out = at;
    return XP_OK;
}

extern "C" void xp_result_free(xp_result* r) { delete r; }

extern "C" const char* xp_last_error(void) { return g_last_error.c_str(); }

// ------------------------------------------------------------------------------------------
// integer peak
// ------------------------------------------------------------------------------------------

// Divisions per second of the two division forms (see the kernels): 64 per chain, 4 chains per thread.
extern "C" xp_status xp_int_div_rate(double* out_divs) {
    if (!out_divs) return fail(XP_ERR_INVALID_ARG, "xp_int_div_rate: null argument");
    int dev = 0, sms = 1;
    XP_CUDA(cudaGetDevice(&dev));
    XP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    u32* d = nullptr;
    XP_CUDA(cudaMalloc(&d, 256));
    cudaEvent_t e0, e1;
    XP_CUDA(cudaEventCreate(&e0));
    XP_CUDA(cudaEventCreate(&e1));
    const int blocks = sms * 8;
    for (int which = 2; which < 4; ++which) {
        const int iters = which == 2 ? 64 : 2048;
        float best = 1e30f;
        for (int rep = 0; rep < 4; ++rep) {
            XP_CUDA(cudaEventRecord(e0, nullptr));
            XP_CUDA(launch_int32_peak(which, d, blocks, iters, nullptr));
            XP_CUDA(cudaEventRecord(e1, nullptr));
            XP_CUDA(cudaEventSynchronize(e1));
            float ms = 0.f;
            XP_CUDA(cudaEventElapsedTime(&ms, e0, e1));
            if (rep > 0 && ms < best) best = ms;
        }
        out_divs[which - 2] = (double)blocks * 256.0 * (double)iters * 64.0 / (best * 1e-3);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(d);
    return XP_OK;
}

extern "C" xp_status xp_int32_peak(double* out_ops, double* out_ms) {
    if (!out_ops) return fail(XP_ERR_INVALID_ARG, "xp_int32_peak: null argument");
    int dev = 0, sms = 1;
    XP_CUDA(cudaGetDevice(&dev));
    XP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    u32* d = nullptr;
    XP_CUDA(cudaMalloc(&d, 256));
    cudaEvent_t e0, e1;
    XP_CUDA(cudaEventCreate(&e0));
    XP_CUDA(cudaEventCreate(&e1));
    const int blocks = sms * 8, iters = 4096;
    for (int which = 0; which < 2; ++which) {
        float best = 1e30f;
        for (int rep = 0; rep < 4; ++rep) {
            XP_CUDA(cudaEventRecord(e0, nullptr));
            XP_CUDA(launch_int32_peak(which, d, blocks, iters, nullptr));
            XP_CUDA(cudaEventRecord(e1, nullptr));
            XP_CUDA(cudaEventSynchronize(e1));
            float ms = 0.f;
            XP_CUDA(cudaEventElapsedTime(&ms, e0, e1));
            if (rep > 0 && ms < best) best = ms;
        }
        const double ops = (double)blocks * 256.0 * (double)iters * 128.0;
        out_ops[which] = ops / (best * 1e-3);
        if (out_ms) out_ms[which] = best;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(d);
    return XP_OK;
}
