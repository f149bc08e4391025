// C ABI of the library (include/lcg.h): contexts, the BuildGram round driver
// (rounds enqueued without host synchronisation, and their CUDA graph),
// MergeGrams, expansion, export / import and post-processing.  Host code only
// orchestrates: every step of the method runs in the kernels of parse.cu,
// grammar.cu and post.cu.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "lcg.h"
#include "lcg_internal.h"

using namespace lcg;

// --------------------------------------------------------------------------
// objects
// --------------------------------------------------------------------------

namespace {

struct Level {
    u64 g = 0, G = 0;          // rules and right-hand-side symbols
    u64 cap_g = 0, cap_G = 0;  // allocated capacity
    u64* rhs_off = nullptr;    // cap_g + 1 entries
    u32* rhs = nullptr;
    u32* F = nullptr;
    void* rtab = nullptr;      // table over the rules (for parses against this grammar and merges)
    u64 rcap = 0;
    bool rvalid = false;
    bool shared_rules = false, shared_rhs = false;  // rhs_off and F, rhs: parts of one of the grammar's slabs
};

// A captured graph, kept by its context and by the grammar that its last launch wrote.
// That grammar's memory is the graph's allocations, and it is freed before the graph is
// destroyed: after a graph that was destroyed first, two later graphs were seen to be
// given the same physical memory, and one's grammar overwrote the other's.
struct GraphHold {
    int device = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    GraphHold() = default;
    GraphHold(const GraphHold&) = delete;
    GraphHold& operator=(const GraphHold&) = delete;
    ~GraphHold() {  // (nothing of it runs, or is allocated, any more)
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        // the graph's memory goes back to the device now, not when another graph would
        // reuse it
        if (graph) cudaDeviceGraphMemTrim(device);
    }
};

}  // namespace

struct lcg_grammar {
    int device = 0;
    std::shared_ptr<GraphHold> hold;  // the graph whose launch wrote it
    lcg_ctx* owner = nullptr;  // the context that created it, while that context lives
    u64 tag = 0;
    u32* F0 = nullptr;  // 256 fingerprints of bytes (device)
    std::vector<Level> lv;
    u32 k = 0, cap_k = 0;
    u32* c_level = nullptr;
    u32* c_rank = nullptr;
    std::vector<void*> slabs;  // allocations that hold the arrays of several levels
};

namespace {
struct GraphBuild;
}

struct lcg_ctx {
    int device = 0;
    int sms = 1;                         // SMs of the device
    bool use_graph = false;              // builds may run as a captured CUDA graph
    GraphBuild* graph = nullptr;         // the graph of the last shape
    cudaStream_t st = nullptr;
    std::vector<lcg_grammar*> live;  // grammars created here and not yet freed
    double plan_slack = 1.0;         // multiplier of the planned buffer sizes (adaptive)
    // table load, k_parse blocks per SM, miss flush, slots cap, stripes, parse tile
    lcg_tuning tuning{0.35, 0, 64, 0, 1, 4096, 16};
    bool own_stream = false;
    u32 blocks_max = 0;  // of cooperative launches (lcg_selftest_blocks), 0: one per SM
    u64 fail_alloc = 0;  // the allocation from now that fails (lcg_selftest_alloc_failure), 0: none
    std::vector<u64> a, b, c;
    u32 levels = 0, m_bits = 32;
    u64 mmask = 0xffffffffull;
    u64 tag = 0;
    std::string err;
    // persistent device scratch
    DevStatus* ds = nullptr;
    u64* ctr = nullptr;     // tile counter of single-pass kernels (never reset)
    u64 ctr_val = 0;        // its value after all launched tiles ran
    u64 epoch = 0;          // look-back epoch, one per launch
    u64* scratch = nullptr; // small device scalars: [0] phrases, [1..2] totals
    void* lb1 = nullptr;
    u64 lb1_tiles = 0;
    void* heads = nullptr;  // k_breaks' look-ahead words (its own: epoch-tagged, nothing else writes them)
    u64 heads_steps = 0;
    void* lb2 = nullptr;
    u64 lb2_tiles = 0;
    double ratio_hint[64] = {0};  // new rules per phrase, per level (decaying maximum over builds)
    double p_hint[64] = {0};      // phrases per symbol, per level (decaying maximum)
    double glen_hint[64] = {0};   // symbols per new rule, per level (decaying maximum)
    u32 hint_rounds = 0;          // rounds of the last build (0: none yet)
    // per-round device status, counts and totals (rounds enqueued without syncs)
    DevStatus* ds_arr = nullptr;
    RoundCounts* rc_arr = nullptr;
    u64* tot_arr = nullptr;
    lcg_build_stats stats{};
    u64 launches = 0;
    // per-kernel CUDA-event timing (optional)
    int ktime = 0;  // 0 off, 1 every launch, 2 parse launches only
    bool capturing = false;              // the stream is being captured into a graph
    unsigned char* mail = nullptr;       // page-locked: what the host reads of a step (see fetch)
    std::vector<std::shared_ptr<const void>> uploads;  // host arrays that copies may still read (see upload)
    unsigned char* upload = nullptr;     // host input of graph builds, at a fixed address
    u64 upload_cap = 0;
    struct KRec {
        const char* name;
        cudaEvent_t a, b;
        double bytes;
        u32 round;  // BuildGram round of a parse launch, else 0
        bool graph;  // the events belong to a captured graph
        bool part = false;  // a further round of the launch before: no events, no time of its own
    };
    std::vector<KRec> krecs;
    std::vector<cudaEvent_t> evpool;
    std::vector<lcg_kernel_time> ktimes;
    std::vector<lcg_kernel_launch> klaunches;
};

namespace {

constexpr u64 kMaxRank = 0x7fffffffull;  // ranks are tagged with one bit in the phrase slots
constexpr u32 kMaxRounds = 63;

struct Fail {
    int code;
};

void fail_if(lcg_ctx* ctx, bool cond, int code, const std::string& msg) {
    if (cond) {
        ctx->err = msg;
        throw Fail{code};
    }
}

void ck(lcg_ctx* ctx, cudaError_t e, const char* what) {
    if (e != cudaSuccess) {
        ctx->err = std::string(what) + ": " + cudaGetErrorString(e);
        throw Fail{e == cudaErrorMemoryAllocation ? LCG_ENOMEM : LCG_EDEVICE};
    }
}

cudaError_t alloc_async(lcg_ctx* ctx, void** p, u64 bytes) {
    if (ctx->fail_alloc && --ctx->fail_alloc == 0) return cudaErrorMemoryAllocation;  // lcg_selftest_alloc_failure
    return cudaMallocAsync(p, bytes, ctx->st);
}

template <typename T>
T* dalloc(lcg_ctx* ctx, u64 count) {
    void* p = nullptr;
    if (count == 0) count = 1;
    ck(ctx, alloc_async(ctx, &p, count * sizeof(T)), "cudaMallocAsync");
    return (T*)p;
}

void dfree(lcg_ctx* ctx, void* p) {
    if (p) cudaFreeAsync(p, ctx->st);
}

// Blocks of a cooperative launch: one per SM.
u32 coop_blocks(const lcg_ctx* ctx) {
    return ctx->blocks_max ? std::min(ctx->blocks_max, (u32)ctx->sms) : (u32)ctx->sms;
}

// A call's device scratch: freed when the call is done with it (drop), and at its end,
// also when it fails.
struct Temps {
    explicit Temps(lcg_ctx* c) : ctx(c) {}
    Temps(const Temps&) = delete;
    Temps& operator=(const Temps&) = delete;
    ~Temps() {
        for (void* p : ptrs) dfree(ctx, p);
    }
    template <typename T>
    T* get(u64 n) {
        ptrs.reserve(ptrs.size() + 1);
        T* p = dalloc<T>(ctx, n);
        ptrs.push_back(p);
        return p;
    }
    void drop(void* p) {
        const auto at = std::find(ptrs.begin(), ptrs.end(), p);
        if (at == ptrs.end()) return;
        ptrs.erase(at);
        dfree(ctx, p);
    }
    lcg_ctx* const ctx;
    std::vector<void*> ptrs;
};

void sync(lcg_ctx* ctx) {
    ck(ctx, cudaStreamSynchronize(ctx->st), "stream synchronize");
    ctx->uploads.clear();
}

// Copies a host array to the device.  The context keeps it until it has waited for the
// stream: where the device reads pageable memory directly, nothing says that the copy
// is over when the call returns.
template <typename T>
void upload(lcg_ctx* ctx, T* dst, std::vector<T>&& src, const char* what) {
    auto kept = std::make_shared<const std::vector<T>>(std::move(src));
    ctx->uploads.push_back(kept);
    ck(ctx, cudaMemcpyAsync(dst, kept->data(), kept->size() * sizeof(T), cudaMemcpyHostToDevice, ctx->st), what);
}

// ---- per-kernel timing: events around each launch when enabled -----------

cudaEvent_t kt_event(lcg_ctx* ctx) {
    if (!ctx->evpool.empty()) {
        cudaEvent_t e = ctx->evpool.back();
        ctx->evpool.pop_back();
        return e;
    }
    cudaEvent_t e;
    ck(ctx, cudaEventCreate(&e), "cudaEventCreate");
    return e;
}

// Under stream capture a plain record only marks a dependency; an external
// record becomes an event node that the graph records at every launch.
cudaError_t record_event(lcg_ctx* ctx, cudaEvent_t e) {
    return ctx->capturing ? cudaEventRecordWithFlags(e, ctx->st, cudaEventRecordExternal) : cudaEventRecord(e, ctx->st);
}

void kt_reset(lcg_ctx* ctx) {
    for (auto& r : ctx->krecs) {
        if (r.graph || r.part) continue;  // recorded by a graph's event nodes: the graph owns them
        ctx->evpool.push_back(r.a);
        ctx->evpool.push_back(r.b);
    }
    ctx->krecs.clear();
    ctx->ktimes.clear();
    ctx->klaunches.clear();
}

// Record the start of a launch of kernel `name` that moves `bytes` algorithmic
// bytes; returns a handle for kt_end (or -1 when timing is off).
int kt_begin(lcg_ctx* ctx, const char* name, double bytes, u32 round = 0) {
    // mode 2: the parse launches only (k_parse, and k_parse_small of short rounds)
    if (ctx->ktime == 0 || (ctx->ktime == 2 && std::strncmp(name, "k_parse", 7) != 0)) return -1;
    lcg_ctx::KRec r{name, kt_event(ctx), kt_event(ctx), bytes, round, false};
    ck(ctx, record_event(ctx, r.a), "cudaEventRecord");
    ctx->krecs.push_back(r);
    return (int)ctx->krecs.size() - 1;
}

void kt_end(lcg_ctx* ctx, int h) {
    if (h >= 0) ck(ctx, record_event(ctx, ctx->krecs[h].b), "cudaEventRecord");
}

// The launch of record h runs `more` further rounds: a record without a time
// for each of them.
void kt_parts(lcg_ctx* ctx, int h, u32 more) {
    if (h < 0) return;
    for (u32 x = 1; x <= more; x++) {
        const lcg_ctx::KRec& r = ctx->krecs[h];
        ctx->krecs.push_back(lcg_ctx::KRec{r.name, nullptr, nullptr, 0.0, r.round + x, false, true});
    }
}

// After the call's last synchronisation: sum the times per kernel kind.
void kt_collect(lcg_ctx* ctx) {
    ctx->ktimes.clear();
    ctx->klaunches.clear();
    for (auto& r : ctx->krecs) {
        float ms = 0.f;
        if (r.part) {
            if (r.round > ctx->stats.rounds) continue;  // the build was done before it
        } else {
            ck(ctx, cudaEventElapsedTime(&ms, r.a, r.b), "cudaEventElapsedTime");
        }
        lcg_kernel_launch kl{};
        std::strncpy(kl.name, r.name, sizeof(kl.name) - 1);
        kl.round = r.round;
        kl.shared = r.part ? 1 : 0;
        kl.ms = ms;
        kl.bytes = r.bytes;
        ctx->klaunches.push_back(kl);
        lcg_kernel_time* t = nullptr;
        for (auto& x : ctx->ktimes)
            if (std::strncmp(x.name, r.name, sizeof(x.name)) == 0) t = &x;
        if (!t) {
            lcg_kernel_time z{};
            std::strncpy(z.name, r.name, sizeof(z.name) - 1);
            ctx->ktimes.push_back(z);
            t = &ctx->ktimes.back();
        }
        t->launches++;
        t->ms += ms;
        t->bytes += r.bytes;
        if (r.round >= 1 && r.round <= 64) {
            lcg_round_stats& rs = ctx->stats.round[r.round - 1];
            rs.round_ms += ms;
            if (std::strcmp(r.name, "k_parse") == 0) rs.parse_ms += ms;
        }
    }
}

void check_device_status(lcg_ctx* ctx, const DevStatus& h) {
    switch (h.error) {
        case kErrNone: return;
        case kErrTimeout: fail_if(ctx, true, LCG_ETIMEOUT, "a bounded device wait gave up"); break;
        case kErrTableFull: fail_if(ctx, true, LCG_ETABLE, "phrase table full"); break;
        case kErrPhraseLong: fail_if(ctx, true, LCG_EOVERFLOW, "phrase of 2^32 symbols or more"); break;
        case kErrMismatch: fail_if(ctx, true, LCG_EMISMATCH, "equal rules with different fingerprints"); break;
        case kErrFormat: fail_if(ctx, true, LCG_EINVAL, "malformed VByte stream"); break;
        default: fail_if(ctx, true, LCG_EDEVICE, "device error " + std::to_string(h.error));
    }
}

// A call starts with a clear status: an error of an earlier call does not
// carry over.
void reset_status(lcg_ctx* ctx) {
    ck(ctx, cudaMemsetAsync(ctx->ds, 0, sizeof(DevStatus), ctx->st), "reset status");
}

// Waits for the stream and reads small values from the device, all of them through the
// context's page-locked buffer: a copy to pageable memory is a wait of its own, and a
// step mostly reads two or three (some 10 us each on the host, the device idle).
constexpr u64 kMailBytes = 16384;
struct Read {
    void* dst;
    const void* src;
    u64 bytes;
};
void fetch(lcg_ctx* ctx, std::initializer_list<Read> reads) {
    u64 total = 0;
    for (const Read& r : reads) total += (r.bytes + 15) & ~15ull;
    const bool mail = total <= kMailBytes;
    u64 at = 0;
    for (const Read& r : reads) {
        if (r.bytes)
            ck(ctx, cudaMemcpyAsync(mail ? (void*)(ctx->mail + at) : r.dst, r.src, r.bytes, cudaMemcpyDeviceToHost,
                                    ctx->st),
               "read");
        at += (r.bytes + 15) & ~15ull;
    }
    sync(ctx);
    at = 0;
    for (const Read& r : reads) {
        if (mail && r.bytes) std::memcpy(r.dst, ctx->mail + at, r.bytes);
        at += (r.bytes + 15) & ~15ull;
    }
}

DevStatus read_status(lcg_ctx* ctx) {
    DevStatus h;
    fetch(ctx, {{&h, ctx->ds, sizeof(h)}});
    return h;
}

// The status, and another value of the same step.
DevStatus read_status(lcg_ctx* ctx, void* dst, const void* src, u64 bytes) {
    DevStatus h;
    fetch(ctx, {{&h, ctx->ds, sizeof(h)}, {dst, src, bytes}});
    return h;
}

LevelHash level_hash(const lcg_ctx* ctx, u32 i) {
    LevelHash h;
    h.a = ctx->a[i];
    h.b = ctx->b[i];
    h.c = ctx->c[i];
    h.mmask = ctx->mmask;
    return h;
}

// The planned rounds did not fit (or a graph capture had to be abandoned):
// the build is redone round by round.
struct Retry {
    bool levels = false;  // only the short rounds' levels did not: no reason for larger plans
};

void destroy_graph(lcg_ctx* ctx);

// NVTX range for profilers (a no-op when no tool is attached): calls, rounds.
struct Range {
    explicit Range(const char* name) { nvtxRangePushA(name); }
    Range(const char* what, u32 i) {
        char b[48];
        std::snprintf(b, sizeof(b), "%s %u", what, i);
        nvtxRangePushA(b);
    }
    ~Range() { nvtxRangePop(); }
    Range(const Range&) = delete;
    Range& operator=(const Range&) = delete;
};

void ensure_lb(lcg_ctx* ctx, void** lb, u64* have, u64 tiles, size_t bytes) {
    if (tiles <= *have) return;
    u64 want = std::max<u64>(tiles, *have * 2);
    size_t nb = bytes / (tiles ? tiles : 1) * want;
    // a graph being captured has its buffers sized beforehand; should one
    // not fit, the capture is abandoned and the build runs round by round
    if (ctx->capturing) throw Retry{};
    // a captured graph uses the current look-back buffers: it goes with them
    if (*lb && ctx->graph) destroy_graph(ctx);
    if (*lb) dfree(ctx, *lb);
    void* p = nullptr;
    *have = 0;
    *lb = nullptr;
    ck(ctx, alloc_async(ctx, &p, nb), "cudaMallocAsync lb");
    ck(ctx, cudaMemsetAsync(p, 0, nb, ctx->st), "memset lb");
    *lb = p;
    *have = want;
}

// grow a level's arrays to hold `need_g` rules and `need_G` symbols
void grow_level(lcg_ctx* ctx, Level& L, u64 need_g, u64 need_G) {
    if (need_g > L.cap_g || L.rhs_off == nullptr) {
        u64 cap = std::max<u64>(need_g, std::max<u64>(L.cap_g * 2, 256));
        Temps fresh(ctx);  // (the level has all of its new arrays or none)
        u64* ro = fresh.get<u64>(cap + 1);
        u32* F = fresh.get<u32>(cap);
        if (L.rhs_off) {
            ck(ctx, cudaMemcpyAsync(ro, L.rhs_off, (L.g + 1) * sizeof(u64), cudaMemcpyDeviceToDevice, ctx->st), "copy");
            ck(ctx, cudaMemcpyAsync(F, L.F, L.g * sizeof(u32), cudaMemcpyDeviceToDevice, ctx->st), "copy");
            if (!L.shared_rules) {
                dfree(ctx, L.rhs_off);
                dfree(ctx, L.F);
            }
        } else {
            ck(ctx, cudaMemsetAsync(ro, 0, sizeof(u64), ctx->st), "memset");
        }
        fresh.ptrs.clear();
        L.rhs_off = ro;
        L.F = F;
        L.cap_g = cap;
        L.shared_rules = false;
    }
    if (need_G > L.cap_G || L.rhs == nullptr) {
        u64 cap = std::max<u64>(need_G, std::max<u64>(L.cap_G * 2, 1024));
        u32* r = dalloc<u32>(ctx, cap);
        if (L.rhs) {
            ck(ctx, cudaMemcpyAsync(r, L.rhs, L.G * sizeof(u32), cudaMemcpyDeviceToDevice, ctx->st), "copy");
            if (!L.shared_rhs) dfree(ctx, L.rhs);
        }
        L.rhs = r;
        L.cap_G = cap;
        L.shared_rhs = false;
    }
}

// Drop the grammar's highest level.
void pop_level(lcg_ctx* ctx, lcg_grammar* G) {
    Level& L = G->lv.back();
    if (!L.shared_rules) {
        dfree(ctx, L.rhs_off);
        dfree(ctx, L.F);
    }
    if (!L.shared_rhs) dfree(ctx, L.rhs);
    dfree(ctx, L.rtab);
    G->lv.pop_back();
}

const u32* fprev_of(const lcg_grammar* G, u32 i) { return i == 1 ? G->F0 : G->lv[i - 2].F; }

// (Re)build the table over the rules of level i so that it can take
// `need_g` rules at load <= 1/2.
void ensure_resident(lcg_ctx* ctx, lcg_grammar* G, u32 i, u64 need_g) {
    Level& L = G->lv[i - 1];
    if (L.rvalid && L.rcap >= 2 * need_g) return;
    const u64 cap = std::max<u64>(1024, 3 * need_g);
    dfree(ctx, L.rtab);
    L.rtab = nullptr;
    L.rvalid = false;
    L.rtab = dalloc<unsigned char>(ctx, cap * slot_bytes());
    L.rcap = cap;
    ck(ctx, cudaMemsetAsync(L.rtab, 0xFF, cap * slot_bytes(), ctx->st), "memset table");
    ck(ctx, launch_resident_build(L.rhs, L.rhs_off, 0, L.g, i == 1, fprev_of(G, i), level_hash(ctx, i), L.rtab,
                                  cap, ctx->ds, ctx->st),
       "resident build");
    ctx->launches++;
    L.rvalid = true;
}

// The rules of an imported grammar against their fingerprints (the host reads the
// status afterwards); `temps` gets what is to be freed then.
void check_fingerprints(lcg_ctx* ctx, const lcg_grammar* G, std::vector<void*>& temps) {
    std::vector<FpLevel> lv;
    u64 blocks = 0;
    for (u32 i = 1; i <= G->lv.size(); i++) {
        const Level& L = G->lv[i - 1];
        if (L.g == 0) continue;
        lv.push_back(FpLevel{L.rhs, L.rhs_off, fprev_of(G, i), L.F, L.g, blocks, level_hash(ctx, i)});
        blocks += (L.g + 255) / 256;
    }
    if (lv.empty()) return;
    FpLevel* d = dalloc<FpLevel>(ctx, lv.size());
    temps.push_back(d);
    const u32 n = (u32)lv.size();
    upload(ctx, d, std::move(lv), "levels");
    ck(ctx, launch_check_fp(d, n, blocks, ctx->ds, ctx->st), "k_check_fp");
    ctx->launches++;
}

void grow_c(lcg_ctx* ctx, lcg_grammar* G, u32 need) {
    if (need <= G->cap_k && G->c_level) return;
    u32 cap = std::max<u32>(need, std::max<u32>(G->cap_k * 2, 16));
    Temps fresh(ctx);
    u32* cl = fresh.get<u32>(cap);
    u32* cr = fresh.get<u32>(cap);
    if (G->c_level) {
        ck(ctx, cudaMemcpyAsync(cl, G->c_level, G->k * sizeof(u32), cudaMemcpyDeviceToDevice, ctx->st), "copy");
        ck(ctx, cudaMemcpyAsync(cr, G->c_rank, G->k * sizeof(u32), cudaMemcpyDeviceToDevice, ctx->st), "copy");
        dfree(ctx, G->c_level);
        dfree(ctx, G->c_rank);
    }
    fresh.ptrs.clear();
    G->c_level = cl;
    G->c_rank = cr;
    G->cap_k = cap;
}

// A grammar with no strings yet: F^0 on the device.  `registered`: the
// context tracks it (every grammar handed to a caller).
lcg_grammar* new_grammar(lcg_ctx* ctx, bool registered = true) {
    lcg_grammar* G = new lcg_grammar();
    G->device = ctx->device;
    G->tag = ctx->tag;
    if (registered) {
        G->owner = ctx;
        ctx->live.push_back(G);
    }
    G->F0 = dalloc<u32>(ctx, 256);
    ck(ctx, launch_h0(level_hash(ctx, 0), G->F0, ctx->st), "h0");
    ctx->launches++;
    return G;
}

void graph_grammar_freed(lcg_ctx* ctx, const lcg_grammar* G);

// Release a grammar.  While its context lives, the memory goes back to the
// pool in the order of that context's stream (later calls reuse it without a
// device synchronisation); otherwise it is freed at once.
void free_grammar_now(lcg_grammar* G) {
    if (!G) return;
    cudaSetDevice(G->device);
    cudaStream_t st = nullptr;
    if (G->owner) {
        auto& v = G->owner->live;
        v.erase(std::remove(v.begin(), v.end(), G), v.end());
        st = G->owner->st;
        graph_grammar_freed(G->owner, G);
    }
    auto release = [&](void* p) {
        if (!p) return;
        if (st) cudaFreeAsync(p, st); else cudaFree(p);
    };
    release(G->F0);
    for (Level& L : G->lv) {
        if (!L.shared_rules) {
            release(L.rhs_off);
            release(L.F);
        }
        if (!L.shared_rhs) release(L.rhs);
        release(L.rtab);
    }
    for (void* p : G->slabs) release(p);
    release(G->c_level);
    release(G->c_rank);
    if (G->hold.use_count() == 1) cudaStreamSynchronize(st);  // the graph goes with it, once all is freed
    delete G;
}

// --------------------------------------------------------------------------
// BuildGram round driver
// --------------------------------------------------------------------------

// Per-round ratios that size the next build's buffers: the largest seen,
// decaying by 2 % per build, so that a context that sees collections of
// changing make-up (a serving loop) keeps plans that fit.
void record_hints(lcg_ctx* ctx, u32 i, u64 n, u64 P, u64 g, u64 G) {
    if (i >= 64) return;
    // the largest ratio seen, fading by 2 % per build: a context fed collections
    // of changing make-up (a serving lane) keeps plans that fit its larger ones
    auto keep = [](double old, double x) { return std::max(x, 0.98 * old); };
    ctx->ratio_hint[i] = keep(ctx->ratio_hint[i], P ? (double)g / (double)P : 0.0);
    ctx->p_hint[i] = keep(ctx->p_hint[i], n ? (double)P / (double)n : 0.0);
    ctx->glen_hint[i] = keep(ctx->glen_hint[i], g ? (double)G / (double)g : 2.0);
}

// The sequence a round reads: T^i, its fingerprints (rounds >= 2) and the
// offsets and ids of its active strings.
struct RoundInput {
    const void* S;
    void* S_owned;
    const u32* Sf;
    int symb;
    u64 n;          // |T^i| (host value when known)
    u64 n_cap;      // symbols that the buffers S and Sf hold
    u32 kk;         // active strings (host value when known)
    u64* soff;
    u32* sid;
    const u64* d_n;  // device values, for rounds enqueued without a sync
    const u64* d_k;
    bool own_offsets = true;  // soff / sid are this build's to free
    // rounds >= 2: what names the symbols (ids) of the sequence: ids below
    // prev_base are ranks of the level below, the others claims of the round
    // before (at most prev_cap), whose ranks are in rank_prev
    u32* rank_prev = nullptr;
    u32 prev_base = 0;
    u64 prev_cap = 0;
};


void free_round_input(lcg_ctx* ctx, RoundInput& in) {
    if (in.own_offsets) {
        dfree(ctx, in.soff);
        dfree(ctx, in.sid);
    }
    if (in.S_owned) dfree(ctx, in.S_owned);
    if (in.Sf) dfree(ctx, (void*)in.Sf);
    dfree(ctx, in.rank_prev);
    in.rank_prev = nullptr;
    in.soff = nullptr;
    in.sid = nullptr;
    in.S_owned = nullptr;
    in.Sf = nullptr;
}

// Buffers of one round.
struct RoundBufs {
    u64 tiles = 0, Pmax = 0, Tcap = 0, cap = 0, first_words = 0;
    u32 tp = 512;  // positions per parse unit
    u64* string_first = nullptr;
    u64* soff_next = nullptr;
    u32* sid_next = nullptr;
    u64* R_phr = nullptr;
    u32* R_sid = nullptr;
    u32* tile_cnt = nullptr;
    u64* tile_pfx = nullptr;
    u32* Tnext = nullptr;
    u32* Fnext = nullptr;
    u32* step_str = nullptr;
    u32* brk = nullptr;
    u32* sbm = nullptr;
    u64 sbm_words = 0;
    unsigned char* tab = nullptr;  // phrase table: cap slots
    u64 id_cap = 0;                // claim numbers
    u32 id_chunk = 1;
    unsigned char* crec = nullptr; // the claims' records
    u64* minpos = nullptr;         // and first occurrences
    u32* rank_of = nullptr;        // their ranks, once named (kept until the next round is named)
    uint2* first = nullptr;        // first-occurrence bitmap and prefix
    u64 r_cap = 0;
    unsigned char* rrec = nullptr; // the claims' records in rank order
};

// The next sequence (Tnext, Fnext) gets `t_cap` entries; 0 leaves it to
// alloc_next.
void alloc_next(lcg_ctx* ctx, RoundBufs& b, u64 t_cap) {
    b.Tcap = std::min<u64>(t_cap, b.Pmax);
    b.Tnext = dalloc<u32>(ctx, b.Tcap);
    b.Fnext = dalloc<u32>(ctx, b.Tcap);
}

// Positions per parse tile of a round of at most n symbols: the tuning's
// tile, halved (down to 1024) while the round would have fewer than
// parse_tile_min tiles per SM, so that short rounds (late rounds, small
// batches) still give every resident k_parse block several tiles.
u32 round_tile(const lcg_ctx* ctx, u64 n) {
    u32 tp = ctx->tuning.parse_tile;
    const u64 want = (u64)ctx->tuning.parse_tile_min * (u64)ctx->sms;
    while (tp > 1024 && (n + tp - 1) / tp < want) tp >>= 1;
    return tp;
}

void alloc_round(lcg_ctx* ctx, RoundBufs& b, u64 n_bound, u32 kk, u64 t_cap) {
    b.tp = parse_unit(round_tile(ctx, n_bound));
    b.tiles = (n_bound + b.tp - 1) / b.tp;
    // every phrase but a string's first has length >= 2
    b.Pmax = n_bound / 2 + 2ull * kk + 1;
    b.string_first = dalloc<u64>(ctx, kk);
    b.soff_next = dalloc<u64>(ctx, kk + 1);
    b.sid_next = dalloc<u32>(ctx, kk);
    b.R_phr = dalloc<u64>(ctx, kk);
    b.R_sid = dalloc<u32>(ctx, kk);
    b.tile_cnt = dalloc<u32>(ctx, b.tiles);
    b.tile_pfx = dalloc<u64>(ctx, b.tiles);
    if (t_cap) alloc_next(ctx, b, t_cap);
    b.step_str = dalloc<u32>(ctx, breaks_steps(b.tiles, b.tp));
    b.brk = dalloc<u32>(ctx, b.tiles * b.tp / 32);
    b.sbm_words = b.tiles * b.tp / 32 + 2;  // positions 0 .. n inclusive
    b.sbm = dalloc<u32>(ctx, b.sbm_words);
    ck(ctx, cudaMemsetAsync(b.sbm, 0, b.sbm_words * sizeof(u32), ctx->st), "memset starts");
}

// A phrase table of `cap` slots, and numbers for `claims` claims (at most 0.8
// of the slots: past it the table is too full).  The blocks of the parse take
// the numbers in ranges (a quarter of the claims that a block makes on
// average, at least a warp's worth), of which each may leave all but one
// unused.  All that may stay unused is a tenth of the slots at most (one number at a
// time in the smallest tables), so a pass that fills between 0.8 and 0.9 of the slots,
// as the claims fall on the blocks, runs out of numbers.  (One that ends before it does
// is as good as any, and not rerun for its load.)  `most`: ids that follow the resident ones and are below 2^31.
void alloc_table(lcg_ctx* ctx, RoundBufs& b, int sym_bytes, u64 cap, u64 claims, u64 most) {
    b.cap = cap;
    claims = std::min(claims, cap - cap / 5);
    const u64 blocks = parse_blocks_most(sym_bytes, b.tiles, (u64)ctx->sms);
    const u64 chunk = std::min<u64>(2048, std::max<u64>(32, claims / (4 * blocks)));
    b.id_chunk = (u32)std::min<u64>(chunk, 1 + cap / 10 / blocks);
    b.id_cap = claims + blocks * (b.id_chunk - 1);
    if (b.id_cap > most) {  // a level near its last rule: no number stays unused
        b.id_chunk = 1;
        b.id_cap = std::min(claims, most);
    }
    b.tab = dalloc<unsigned char>(ctx, cap * slot_bytes());
    b.crec = dalloc<unsigned char>(ctx, b.id_cap * claim_rec_bytes());
    b.minpos = dalloc<u64>(ctx, b.id_cap);
    b.rank_of = dalloc<u32>(ctx, b.id_cap);
    ck(ctx, cudaMemsetAsync(b.tab, 0xFF, cap * slot_bytes(), ctx->st), "memset table");
    ck(ctx, cudaMemsetAsync(b.minpos, 0xFF, b.id_cap * sizeof(u64), ctx->st), "memset positions");
}

void free_table(lcg_ctx* ctx, RoundBufs& b) {
    for (void* p : {(void*)b.tab, (void*)b.crec, (void*)b.minpos, (void*)b.rank_of}) dfree(ctx, p);
    b.tab = nullptr;
    b.crec = nullptr;
    b.minpos = nullptr;
    b.rank_of = nullptr;
}

// Naming arrays for up to r_cap new rules and `phrases` phrases.
void alloc_naming(lcg_ctx* ctx, RoundBufs& b, u64 r_cap, u64 phrases) {
    b.r_cap = r_cap;
    b.first_words = phrases / 32 + 1;
    b.first = dalloc<uint2>(ctx, b.first_words);
    b.rrec = dalloc<unsigned char>(ctx, r_cap * claim_rec_bytes());
    ck(ctx, cudaMemsetAsync(b.first, 0, b.first_words * sizeof(uint2), ctx->st), "memset bits");
}

// Free a round's buffers except those that become the next round's input.
void free_round(lcg_ctx* ctx, RoundBufs& b) {
    for (void* p : {(void*)b.string_first, (void*)b.R_phr, (void*)b.R_sid, (void*)b.tile_cnt, (void*)b.tile_pfx,
                    (void*)b.step_str, (void*)b.brk, (void*)b.sbm, (void*)b.first, (void*)b.rrec, (void*)b.tab,
                    (void*)b.crec, (void*)b.minpos})
        dfree(ctx, p);
}

// Free all of a round's buffers, when the round fails: to be called by the caller of a
// function that throws between its first allocation and next_input.
void drop_round(lcg_ctx* ctx, RoundBufs& b) {
    free_round(ctx, b);
    for (void* p : {(void*)b.soff_next, (void*)b.sid_next, (void*)b.Tnext, (void*)b.Fnext, (void*)b.rank_of})
        dfree(ctx, p);
}

// Bits that hold every rank below `count` (at least 1).
int rank_width(u64 count) {
    int w = 1;
    while (w < 31 && (1ull << w) < count) w++;
    return w;
}

RoundArgs round_args(lcg_ctx* ctx, lcg_grammar* R, const RoundInput& in, RoundBufs& b, u32 i) {
    RoundArgs a{};
    a.sym_bytes = in.symb;
    a.sym_w = in.symb == 1 ? 8 : 31;
    a.S = in.S;
    a.Sf = in.Sf;
    a.n = in.n;
    a.d_n = in.d_n;
    a.n_cap = in.n_cap;
    a.soff = in.soff;
    a.sid = in.sid;
    a.k = in.kk;
    a.d_k = in.d_k;
    a.Fprev = fprev_of(R, i);
    a.lh = level_hash(ctx, i);
    a.level = i;
    a.parse_blocks = ctx->tuning.parse_blocks_per_sm;
    a.stripes = ctx->tuning.tile_stripes;
    a.prev_base = in.prev_base;
    a.rank_prev = in.rank_prev;
    a.tiles_bound = b.tiles;
    a.tp = b.tp;
    a.string_first = b.string_first;
    a.step_str = b.step_str;
    a.brk = b.brk;
    a.sbm = b.sbm;
    a.sbm_words = b.sbm_words;
    a.tile_cnt = b.tile_cnt;
    a.tile_pfx = b.tile_pfx;
    a.ctr = ctx->ctr;
    a.ds = ctx->ds_arr + (i - 1);
    a.rc = ctx->rc_arr + (i - 1);
    a.total = ctx->tot_arr + 3 * (i - 1);  // [0] phrases; [1], [2] scratch of the scans
    a.d_tiles = &a.rc->tiles;
    a.d_gnew = &a.ds->claims;
    a.d_ids = &a.ds->aux[1];
    a.d_Gnew = &a.ds->claim_len;
    a.soff_next = b.soff_next;
    a.sid_next = b.sid_next;
    a.R_phr = b.R_phr;
    a.R_sid = b.R_sid;
    a.T_cap = b.Tcap;
    a.Tnext = b.Tnext;
    a.Fnext = b.Fnext;
    a.c_level = R->c_level;
    a.c_rank = R->c_rank;
    return a;
}

void set_table(RoundArgs& a, RoundBufs& b) {
    a.tab = b.tab;
    a.tab_cap = b.cap;
    a.id_cap = b.id_cap;
    a.id_chunk = b.id_chunk;
    a.crec = b.crec;
    a.minpos = b.minpos;
    a.rank_of = b.rank_of;
}

// The round's phrases: tile strings, breaks, tile scan, strings.
void enqueue_phrases(lcg_ctx* ctx, RoundArgs& a, u64 n_for_bytes) {
    // k_breaks' look-ahead words: a buffer of their own, so that no other
    // kernel's data can read as a head of this launch's epoch
    const u64 steps = breaks_steps(a.tiles_bound, a.tp);
    ensure_lb(ctx, &ctx->heads, &ctx->heads_steps, steps, steps * sizeof(u64));
    a.heads = reinterpret_cast<u64*>(ctx->heads);
    a.brk_epoch = ++ctx->epoch;
    const Range range("phrases, round", a.level);
    const int ht = kt_begin(ctx, "k_tile_strings", 4.0 * (double)a.tiles_bound, a.level);
    ck(ctx, launch_tile_strings(a, ctx->st), "k_tile_strings");
    kt_end(ctx, ht);
    int h = kt_begin(ctx, "k_breaks", (a.sym_bytes == 1 ? 1.0 : 4.0) * n_for_bytes + (double)n_for_bytes / 8.0, a.level);
    ck(ctx, launch_breaks(a, ctx->st), "k_breaks");
    kt_end(ctx, h);
    const u64 stiles = std::max<u64>(1, scan2_tiles_for(a.tiles_bound));
    ensure_lb(ctx, &ctx->lb2, &ctx->lb2_tiles, stiles, scan2_lb_bytes(stiles));
    u64 grid = 0;
    h = kt_begin(ctx, "k_scan2", 12.0 * (double)a.tiles_bound, a.level);
    ck(ctx, launch_scan2(a.tile_cnt, nullptr, a.tiles_bound, a.tile_pfx, nullptr, a.total, ctx->lb2, ++ctx->epoch,
                         ctx->ctr, ctx->ctr_val, a.ds, ctx->st, &grid, a.d_tiles),
       "scan");
    kt_end(ctx, h);
    ctx->ctr_val += grid;
    h = kt_begin(ctx, "k_strings", 40.0 * a.k, a.level);
    ck(ctx, launch_strings(a, ctx->st), "k_strings");
    kt_end(ctx, h);
    ctx->launches += 4;
}

// Parse: the phrases' lookups, and the next sequence.
void enqueue_parse(lcg_ctx* ctx, RoundArgs& a, u64 n_for_bytes) {
    const Range range("parse, round", a.level);
    const double tab_bytes = a.tab_cap * (double)slot_bytes();
    const double tbytes = tab_bytes > kL2Bytes ? 32.0 * (double)n_for_bytes / 3.0 : 0.0;
    const int h = kt_begin(ctx, "k_parse",
                           (a.sym_bytes == 1 ? 1.0 : 8.0) * n_for_bytes + (double)n_for_bytes / 8.0 +
                               8.0 * (double)n_for_bytes / 3.0 + tbytes, a.level);
    ck(ctx, launch_parse(a, ctx->st), "k_parse");
    kt_end(ctx, h);
    ctx->launches += 1;
}

// Naming: mark, popcount scan, rank, rule offsets, rules.
void enqueue_naming(lcg_ctx* ctx, RoundArgs& a, RoundBufs& b, double g_bytes, double G_bytes) {
    const Range range("naming, round", a.level);
    a.first = b.first;
    a.first_words = b.first_words;
    a.rrec = b.rrec;
    a.r_cap = b.r_cap;
    const u64 g_grid = std::max<u64>(1, b.r_cap);
    int h = kt_begin(ctx, "k_mark", 8.0 * g_bytes, a.level);
    ck(ctx, launch_mark(a, g_grid, ctx->st), "k_mark");
    kt_end(ctx, h);
    const u64 ptiles = std::max<u64>(1, popscan_tiles_for(b.first_words));
    const u64 rtiles = rule_offs_tiles(g_grid);
    const u64 lbt = std::max(ptiles, rtiles);
    ensure_lb(ctx, &ctx->lb1, &ctx->lb1_tiles, lbt, lb1_bytes(lbt));
    a.lb1 = ctx->lb1;
    a.epoch = ++ctx->epoch;
    a.ctr_base = ctx->ctr_val;
    ctx->ctr_val += ptiles;
    h = kt_begin(ctx, "k_popscan", 12.0 * (double)b.first_words, a.level);
    ck(ctx, launch_popscan(a, ctx->st), "k_popscan");
    kt_end(ctx, h);
    h = kt_begin(ctx, "k_rank", 76.0 * g_bytes, a.level);
    ck(ctx, launch_rank(a, g_grid, ctx->st), "k_rank");
    kt_end(ctx, h);
    a.epoch = ++ctx->epoch;
    a.ctr_base = ctx->ctr_val;
    ctx->ctr_val += rtiles;
    h = kt_begin(ctx, "k_rule_offs", 16.0 * g_bytes, a.level);
    ck(ctx, launch_rule_offs(a, g_grid, ctx->st), "k_rule_offs");
    kt_end(ctx, h);
    h = kt_begin(ctx, "k_rules", 4.0 * G_bytes + 44.0 * g_bytes, a.level);
    ck(ctx, launch_rules(a, g_grid, ctx->st), "k_rules");
    kt_end(ctx, h);
    ctx->launches += 5;
}

void next_input(lcg_ctx* ctx, RoundInput& in, RoundBufs& b) {
    if (in.own_offsets) {
        dfree(ctx, in.soff);
        dfree(ctx, in.sid);
    }
    in.own_offsets = true;
    if (in.S_owned) dfree(ctx, in.S_owned);
    if (in.Sf) dfree(ctx, (void*)in.Sf);
    dfree(ctx, in.rank_prev);
    in.rank_prev = b.rank_of;
    in.prev_cap = b.id_cap;
    in.S = b.Tnext;
    in.S_owned = b.Tnext;
    in.Sf = b.Fnext;
    in.n_cap = b.Tcap;
    in.symb = 4;
    in.soff = b.soff_next;
    in.sid = b.sid_next;
}

// ---- the short rounds ------------------------------------------------------
//
// A round whose tile is the smallest (see round_tile) and that has at most
// kTailSymbols symbols, and every round after it, run in two launches.  All
// their buffers are parts of one allocation, sized by what a round can have at
// most (n symbols in k strings: (n + k) / 2 phrases), so nothing is
// regrown or waited for.  The levels of a fresh build share one allocation too, which
// the grammar keeps: from kTailPlanned symbols on a plan makes it about as large as they
// need (tail_levels), and where there is none it is replaced afterwards if they need
// less (compact_levels).

// (Where the slots of a table are limited the rounds that could need more run one by
// one: theirs start within the limit.  Where larger tiles are asked for they are kept
// until one block takes the round, which has no tiles: a build of 2 MB with
// parse_tile_min 0 1.27 ms with ordinary rounds to its end, 1.14 so.)
bool is_tail(const lcg_ctx* ctx, u64 n, const lcg_grammar* resident = nullptr) {
    // (nor where a level is so full that the numbers a short round takes might not fit)
    if (resident)
        for (const Level& L : resident->lv)
            if (L.g > kMaxRank - 2 * kTailSymbols) return false;
    const u64 most = ctx->tuning.table_slots_max;
    return n <= kTailSymbols && (n <= kSoloSymbols || round_tile(ctx, n) == 1024) && (most == 0 || 3 * n <= most);
}

// Rules and symbols of a level.
struct LevelSize {
    u64 g, G;
};
// Below, the levels' arrays take what they can need at most (20 bytes a symbol over all
// of them, 1 MB): a server's short requests, each of another make-up, are never redone.
constexpr u64 kTailPlanned = 50000;

// Offsets of the parts of one allocation.
struct Parts {
    u64 size = 0;
    u64 take(u64 bytes) {
        const u64 at = size;
        size += (bytes + 255) & ~255ull;
        return at;
    }
};

// Enqueue round i and those after it (at most n_bound symbols in kk strings
// enter it); returns how many there may be.  `in` becomes what follows the
// last (nothing); cap[r]: the table slots of round r.
// `planned`: what the arrays of a fresh build's levels are made for (those that it does
// not name: for what they can have); a level that has more flags a capacity error.
u32 tail_enqueue(lcg_ctx* ctx, lcg_grammar* R, RoundInput& in, u32 i, u64 n_bound, u32 kk, bool against_resident,
                 const DevStatus* ds_prev, u64* cap, const std::vector<LevelSize>& planned) {
    fail_if(ctx, i >= ctx->levels || i > kMaxRounds,
            LCG_ELEVELS, "hash family too short: needs more than " + std::to_string(ctx->levels) + " functions");
    const u32 most = std::min<u32>({kTailRounds, ctx->levels - i, kMaxRounds - i + 1});
    const u32 tp = parse_unit(1024);
    struct Size {
        u64 n, k, P, units, cap, ids, words;
        u64 sbm, first, tab, minpos;                                          // cleared parts
        u64 string_first, soff, sid, R_phr, R_sid, cnt, pfx, brk, T, F, crec, rank_of, rrec;
        LevelSize lv;                                                         // the level's arrays
        u64 off, rhs, lvF;                                                    // in the levels' slab
    };
    std::vector<Size> z;
    Parts zero, ones, plain, slab;
    const u64 bar = zero.take(4 * sizeof(u64));
    u64 chunks = 0;
    u32 chunk_ids = 32;
    for (u64 n = n_bound, k = std::min<u64>(kk, n_bound / 2 + 1); z.size() < most && n > 0; ) {
        Size x{};
        x.n = n;
        x.k = k;
        x.P = (n + k) / 2 + 1;
        x.units = (n + tp - 1) / tp;
        x.cap = 3 * x.P + 64;
        // the parse's blocks take numbers for a warp's claims at a time, at least
        x.ids = x.P + (u64)chunk_ids * std::min<u64>((u64)ctx->sms, (x.units + kParseWarps - 1) / kParseWarps);
        x.words = x.P / 32 + 1;
        x.sbm = zero.take((n / 32 + 2) * 4);
        x.first = zero.take(x.words * sizeof(uint2));
        x.tab = ones.take(x.cap * slot_bytes());
        x.minpos = ones.take(x.ids * 8);
        x.string_first = plain.take(k * 8);
        x.soff = plain.take((k + 1) * 8);
        x.sid = plain.take(k * 4);
        x.R_phr = plain.take(k * 8);
        x.R_sid = plain.take(k * 4);
        x.cnt = plain.take(x.units * 4);
        x.pfx = plain.take(x.units * 8);
        x.brk = plain.take((x.units * tp / 32) * 4);
        x.T = plain.take(x.P * 4);
        x.F = plain.take(x.P * 4);
        x.crec = plain.take(x.ids * claim_rec_bytes());
        x.rank_of = plain.take(x.ids * 4);
        x.rrec = plain.take(x.P * claim_rec_bytes());
        x.lv = LevelSize{x.P, n};
        if (z.size() < planned.size())
            x.lv = LevelSize{std::min(x.P, planned[z.size()].g), std::min(n, planned[z.size()].G)};
        x.off = slab.take((x.lv.g + 1) * 8);
        x.rhs = slab.take(x.lv.G * 4);
        x.lvF = slab.take(x.lv.g * 4);
        chunks += rule_chunks(x.P);
        z.push_back(x);
        // the strings left have two symbols or more each
        const u64 n1 = (n + k) / 2;
        k = std::min<u64>(k, n1 / 2);
        n = k ? n1 : 0;
    }
    const u32 rounds = (u32)z.size();
    const u64 chunk_len = plain.take(chunks * 8);
    const u64 retired = plain.take((u64)ctx->sms * 8);
    Temps fresh(ctx);  // (freed if a step below fails)
    unsigned char* base = fresh.get<unsigned char>(zero.size + ones.size + plain.size);
    unsigned char *b0 = base, *b1 = base + zero.size, *b2 = b1 + ones.size;
    ck(ctx, cudaMemsetAsync(b0, 0, zero.size, ctx->st), "memset");
    ck(ctx, cudaMemsetAsync(b1, 0xFF, ones.size, ctx->st), "memset tables");
    unsigned char* lv = nullptr;
    if (!against_resident) {
        lv = dalloc<unsigned char>(ctx, slab.size);
        R->slabs.push_back(lv);
    }
    const u64 steps = breaks_steps(z[0].units, tp);
    ensure_lb(ctx, &ctx->heads, &ctx->heads_steps, steps, steps * sizeof(u64));
    TailArgs t{};
    t.rounds = rounds;
    t.bar = (u64*)(b0 + bar);
    t.chunk_len = (u64*)(b2 + chunk_len);
    t.retired = (u64*)(b2 + retired);
    for (u32 r = 0; r < rounds; r++) {
        const Size& x = z[r];
        const u32 lev = i + r;
        if (R->lv.size() < lev) R->lv.emplace_back();
        Level& L = R->lv[lev - 1];
        if (against_resident) {
            if (L.g > 0) ensure_resident(ctx, R, lev, L.g + x.P);
            grow_level(ctx, L, L.g + x.P, L.G + x.n);
            if (L.g == 0) ensure_resident(ctx, R, lev, x.P);
        } else {
            L.rhs_off = (u64*)(lv + x.off);
            L.rhs = (u32*)(lv + x.rhs);
            L.F = (u32*)(lv + x.lvF);
            L.cap_g = x.lv.g;
            L.cap_G = x.lv.G;
            L.shared_rules = L.shared_rhs = true;
            L.rvalid = false;
        }
        RoundArgs& a = t.r[r];
        a.sym_bytes = r == 0 ? in.symb : 4;
        a.S = r == 0 ? in.S : b2 + z[r - 1].T;
        a.Sf = r == 0 ? in.Sf : (u32*)(b2 + z[r - 1].F);
        a.n = r == 0 ? in.n : 0;
        a.d_n = r == 0 ? in.d_n : &ctx->rc_arr[lev - 2].n_next;
        a.n_cap = r == 0 ? in.n_cap : z[r - 1].P;
        a.soff = r == 0 ? in.soff : (u64*)(b2 + z[r - 1].soff);
        a.sid = r == 0 ? in.sid : (u32*)(b2 + z[r - 1].sid);
        a.k = r == 0 ? in.kk : 0;
        a.d_k = r == 0 ? in.d_k : &ctx->rc_arr[lev - 2].k_next;
        a.Fprev = fprev_of(R, lev);
        a.lh = level_hash(ctx, lev);
        a.level = lev;
        a.stripes = 1;
        a.tp = tp;
        a.prev_base = r == 0 ? in.prev_base : t.r[r - 1].id_base;
        a.id_base = against_resident ? (u32)L.g : 0;
        a.rank_prev = r == 0 ? in.rank_prev : t.r[r - 1].rank_of;
        a.tiles_bound = x.units;
        a.brk = (u32*)(b2 + x.brk);
        a.sbm = (u32*)(b0 + x.sbm);
        a.sbm_words = x.n / 32 + 2;
        a.tile_cnt = (u32*)(b2 + x.cnt);
        a.tile_pfx = (u64*)(b2 + x.pfx);
        a.string_first = (u64*)(b2 + x.string_first);
        a.heads = (u64*)ctx->heads;
        a.brk_epoch = ++ctx->epoch;
        a.ds = ctx->ds_arr + (lev - 1);
        a.ds_prev = r == 0 ? ds_prev : ctx->ds_arr + (lev - 2);
        a.rc = ctx->rc_arr + (lev - 1);
        a.d_tiles = &a.rc->tiles;
        a.total = ctx->tot_arr + 3 * (lev - 1);
        a.soff_next = (u64*)(b2 + x.soff);
        a.sid_next = (u32*)(b2 + x.sid);
        if (r + 1 < rounds) {
            a.sbm_next = (u32*)(b0 + z[r + 1].sbm);
            a.sbm_next_words = z[r + 1].n / 32 + 2;
        }
        a.R_phr = (u64*)(b2 + x.R_phr);
        a.R_sid = (u32*)(b2 + x.R_sid);
        a.tab = b1 + x.tab;
        a.tab_cap = x.cap;
        a.id_cap = x.ids;
        a.id_chunk = chunk_ids;
        a.crec = b2 + x.crec;
        a.minpos = (u64*)(b1 + x.minpos);
        a.rank_of = (u32*)(b2 + x.rank_of);
        a.T_cap = x.P;
        a.Tnext = (u32*)(b2 + x.T);
        a.Fnext = (u32*)(b2 + x.F);
        a.c_level = R->c_level;
        a.c_rank = R->c_rank;
        a.d_gnew = &a.ds->claims;
        a.d_ids = &a.ds->aux[1];
        a.d_Gnew = &a.ds->claim_len;
        a.cap_g = L.cap_g;
        a.cap_G = L.cap_G;
        a.first_words = x.words;
        a.first = (uint2*)(b0 + x.first);
        a.r_cap = x.P;
        a.rrec = b2 + x.rrec;
        a.g_base = L.g;
        a.G_base = L.G;
        a.rhs = L.rhs;
        a.rhs_off = L.rhs_off;
        a.F = L.F;
        // keys as narrow as the symbols' ids allow (tables of resident grammars
        // keep the full width)
        a.sym_w = a.sym_bytes == 1 ? 8 : against_resident ? 31
                  : rank_width(r == 0 ? in.prev_base + in.prev_cap : z[r - 1].ids);
        if (against_resident) {
            if (L.g > 0) {
                a.rtab = L.rtab;
                a.rtab_cap = L.rcap;
                a.rrhs = L.rhs;
                a.rrhs_off = L.rhs_off;
            }
            a.rtab_w = L.rtab;
            a.rtab_w_cap = L.rcap;
        }
        cap[lev] = x.cap;
    }
    const Range range("short rounds from", i);
    int h = kt_begin(ctx, "k_parse_small", 5.0 * (double)n_bound, i);
    ck(ctx, launch_parse_small(t, ctx->blocks_max, ctx->st), "k_parse_small");
    kt_end(ctx, h);
    kt_parts(ctx, h, rounds - 1);
    h = kt_begin(ctx, "k_naming_small", 12.0 * (double)n_bound, i);
    ck(ctx, launch_naming_small(t, ctx->blocks_max, ctx->st), "k_naming_small");
    kt_end(ctx, h);
    ctx->launches += 2;
    free_round_input(ctx, in);
    fresh.drop(base);
    const u64 n = in.n;
    in = RoundInput{};
    in.n = n;
    return rounds;
}

// Copies of 32-bit columns, all of them in one launch.
struct Copies {
    std::vector<CopyCol> cols;
    u64 blocks = 0;
    // pad: a zero follows when n is odd
    void add(void* dst, const void* src, u64 n, bool pad = false) {
        if (n == 0) return;
        cols.push_back(CopyCol{(u32*)dst, (const u32*)src, n, blocks, pad && (n & 1)});
        blocks += copy_blocks(n);
    }
    void run(lcg_ctx* ctx, std::vector<void*>& temps) {
        if (cols.empty()) return;
        CopyCol* d = dalloc<CopyCol>(ctx, cols.size());
        temps.push_back(d);
        const u32 n = (u32)cols.size();
        upload(ctx, d, std::move(cols), "columns");
        ck(ctx, launch_copy_cols(d, n, blocks, ctx->st), "copy columns");
        ctx->launches++;
    }
};

// The levels from i on, all in the grammar's last slab: into one that holds what they
// have, when that is less than half of it and a megabyte less (a string of 20 kB is built
// in 390 us the first time, 410 with the copy).  Where there is no memory for it they
// stay.
void compact_levels(lcg_ctx* ctx, lcg_grammar* R, u32 i) {
    if (R->slabs.empty()) return;
    Parts have, need;
    for (size_t l = i - 1; l < R->lv.size(); l++) {
        const Level& L = R->lv[l];
        if (!L.shared_rules || !L.shared_rhs) return;
        have.take((L.cap_g + 1) * 8 + L.cap_G * 4 + L.cap_g * 4);
        need.take((L.g + 1) * 8);
        need.take(L.G * 4);
        need.take(L.g * 4);
    }
    if (have.size < 2 * need.size + 20 * kTailPlanned) return;
    void* p = nullptr;
    if (alloc_async(ctx, &p, need.size) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    std::vector<void*> temps;
    std::vector<Level> lv(R->lv.begin() + (i - 1), R->lv.end());
    try {
        Parts at;
        Copies copies;
        for (Level& L : lv) {
            unsigned char* const off = (unsigned char*)p + at.take((L.g + 1) * 8);
            unsigned char* const rhs = (unsigned char*)p + at.take(L.G * 4);
            unsigned char* const F = (unsigned char*)p + at.take(L.g * 4);
            copies.add(off, L.rhs_off, 2 * (L.g + 1));
            copies.add(rhs, L.rhs, L.G);
            copies.add(F, L.F, L.g);
            L.rhs_off = (u64*)off;
            L.rhs = (u32*)rhs;
            L.F = (u32*)F;
            L.cap_g = L.g;
            L.cap_G = L.G;
        }
        copies.run(ctx, temps);
    } catch (const Fail&) {
        for (void* x : temps) dfree(ctx, x);
        dfree(ctx, p);
        return;
    }
    for (void* x : temps) dfree(ctx, x);
    std::copy(lv.begin(), lv.end(), R->lv.begin() + (i - 1));
    dfree(ctx, R->slabs.back());
    R->slabs.back() = p;
}

// The short rounds of a build that is run round by round: one host
// synchronisation after all of them.
void tail_sync(lcg_ctx* ctx, lcg_grammar* R, RoundInput& in, u32& i, bool against_resident) {
    u64 cap[kMaxRounds + kTailRounds + 2] = {0};
    u64 n = in.n;
    u32 k = in.kk;
    const u32 rounds = tail_enqueue(ctx, R, in, i, in.n, in.kk, against_resident, nullptr, cap, {});
    std::vector<DevStatus> st(rounds);
    std::vector<RoundCounts> rc(rounds);
    fetch(ctx, {{st.data(), ctx->ds_arr + (i - 1), rounds * sizeof(DevStatus)},
                {rc.data(), ctx->rc_arr + (i - 1), rounds * sizeof(RoundCounts)}});
    for (const DevStatus& x : st) {
        check_device_status(ctx, x);
        fail_if(ctx, x.overflow != 0, LCG_ETABLE, "phrase table full");  // not reached: it has room for every phrase
    }
    u32 r = 0;
    for (; r < rounds && k > 0; r++) {
        Level& L = R->lv[i + r - 1];
        fail_if(ctx, L.g + st[r].claims > kMaxRank, LCG_EOVERFLOW, "level with 2^31 rules or more");
        L.g += st[r].claims;
        L.G += st[r].claim_len;
        lcg_round_stats& rs = ctx->stats.round[std::min<u32>(i + r - 1, 63)];
        rs.n = n;
        rs.strings = k;
        rs.phrases = rc[r].phrases;
        rs.g = st[r].claims;
        rs.G = st[r].claim_len;
        rs.table_cap = cap[i + r];
        record_hints(ctx, i + r, n, rc[r].phrases, st[r].claims, st[r].claim_len);
        n = rc[r].n_next;
        k = (u32)rc[r].k_next;
        ctx->stats.rounds = i + r;
    }
    // levels that no round reached
    while (R->lv.size() > (size_t)(i + r - 1) && R->lv.back().g == 0) pop_level(ctx, R);
    if (!against_resident) compact_levels(ctx, R, i);
    i += r;
    in.kk = k;
    in.n = n;
    fail_if(ctx, k > 0, LCG_ELEVELS,
            "hash family too short: needs more than " + std::to_string(ctx->levels) + " functions");
}

// One round (b: its buffers, for the caller to free on failure) with a host
// synchronisation after the parse: the table is
// regrown and the parse rerun until it fits, and all later sizes are exact.
// A round of up to kExactNext phrases gets room for as many as it can have (8 bytes
// each) instead of waiting for their number: six builds of 12 MB into a growing
// grammar 7.60 ms with 2^22, 7.51 with 2^24 (0.7 to 1.7 % in each of four pairs of runs).
constexpr u64 kExactNext = 1ull << 24;  // phrases

void round_sync(lcg_ctx* ctx, lcg_grammar* R, RoundInput& in, u32 i, bool against_resident, double& prev_ratio,
                double& p_ratio, RoundBufs& b) {
    fail_if(ctx, i >= ctx->levels || i > kMaxRounds,
            LCG_ELEVELS, "hash family too short: needs more than " + std::to_string(ctx->levels) + " functions");
    if (R->lv.size() < i) R->lv.emplace_back();
    lcg_round_stats& rs = ctx->stats.round[std::min<u32>(i - 1, 63)];
    const u64 n = in.n;
    rs.n = n;
    rs.strings = in.kk;
    alloc_round(ctx, b, n, in.kk, 0);
    Level& L = R->lv[i - 1];
    RoundArgs a = round_args(ctx, R, in, b, i);
    a.d_n = nullptr;
    a.d_k = nullptr;
    // inline keys as narrow as the symbols' ids allow; tables of resident
    // grammars keep the full width
    if (i > 1 && !against_resident) a.sym_w = rank_width(in.prev_base + in.prev_cap);
    const u64 id_base = L.g;  // ids below it are ranks of resident rules
    a.id_base = (u32)id_base;
    if (against_resident && L.g > 0) {
        ensure_resident(ctx, R, i, L.g);
        a.rtab = L.rtab;
        a.rtab_cap = L.rcap;
        a.rrhs = L.rhs;
        a.rrhs_off = L.rhs_off;
    }
    // Phrase table: sized from the distinct/phrase ratio of this level in the
    // context's previous build when there is one (at the tuning's load, 0.35 by
    // default: short probe sequences), else from a generous guess; an
    // overflowing table is regrown and the parse rerun.
    const double hint = ctx->ratio_hint[std::min<u32>(i, 63)];
    u64 cap;
    if (hint > 0) {
        const u64 P_est = std::min<u64>(b.Pmax, (u64)(ctx->p_hint[std::min<u32>(i, 63)] * (double)n) + 64);
        cap = std::max<u64>(8192, (u64)(hint * (double)P_est / ctx->tuning.table_load) + 1024);
    } else {
        const u64 P_est = std::min<u64>(b.Pmax, (u64)(p_ratio * 1.2 * (double)n) + 64);
        const double ratio = (i == 1) ? 0.02 : std::min(1.0, std::max(prev_ratio * 2.0, 0.05));
        cap = 2 * std::max<u64>(4096, std::min<u64>(P_est, (u64)(ratio * 1.3 * (double)P_est) + 1));
    }
    if (ctx->tuning.table_slots_max) cap = std::min<u64>(cap, ctx->tuning.table_slots_max);
    // the claims' ids follow the resident ranks and are below 2^31; the claims
    // that the table is expected to see, with slack
    const u64 max_ids = kMaxRank + 1 - id_base;
    const double g_hint = hint * ctx->p_hint[std::min<u32>(i, 63)] * (double)n * 1.5 + 1024;
    u32 retries = 0;
    bool all = false;  // numbers for all the claims that the table may hold
    DevStatus st;
    RoundCounts rc;
    ck(ctx, cudaMemsetAsync(a.ds, 0, sizeof(DevStatus), ctx->st), "reset counters");
    enqueue_phrases(ctx, a, n);
    // The next sequence: at most Pmax symbols; a large one gets exactly the
    // round's phrases, which the host then waits for.
    u64 t_cap = b.Pmax;
    if (t_cap > kExactNext) {
        fetch(ctx, {{&rc, a.rc, sizeof(rc)}, {&st, a.ds, sizeof(st)}});
        check_device_status(ctx, st);
        t_cap = rc.phrases + 1;
    }
    alloc_next(ctx, b, t_cap);
    a.Tnext = b.Tnext;
    a.Fnext = b.Fnext;
    a.T_cap = b.Tcap;
    while (true) {
        fail_if(ctx, cap > kMaxRank + 1, LCG_ETABLE, "phrase table would exceed 2^31 slots");
        // (a table of more than 2^28 slots, 8 GB, gets numbers for half of them without a
        // hint: they take more memory than the slots.  With half from 2^26 slots on round 3
        // of a first build of 4 x 3.1 Gbp, which fills 139 M slots to 0.795, was rerun with
        // 555 M: in as much time, with twice the memory)
        const u64 most = all || cap <= (1ull << 28) ? cap : std::max<u64>(cap / 2, (u64)g_hint);
        alloc_table(ctx, b, in.symb, cap, most, max_ids);
        set_table(a, b);
        enqueue_parse(ctx, a, n);
        fetch(ctx, {{&rc, a.rc, sizeof(rc)}, {&st, a.ds, sizeof(st)}});
        check_device_status(ctx, st);
        if (!st.overflow) break;
        free_table(ctx, b);
        const bool ran_out = st.aux[1] >= b.id_cap;  // of numbers
        fail_if(ctx, ran_out && b.id_cap >= max_ids, LCG_EOVERFLOW, "level with 2^31 rules or more");
        // where the next larger table would be one too large (2^31 slots) and this one has
        // more room than numbers, it is tried with all of them
        all = ran_out && b.id_cap < cap - cap / 5 && !all && cap * 4 > kMaxRank + 1;
        if (!all) cap *= 4;
        retries++;
        ck(ctx, cudaMemsetAsync(a.ds, 0, sizeof(DevStatus), ctx->st), "reset counters");
    }
    const u64 P = rc.phrases;
    rs.phrases = P;
    fail_if(ctx, P > b.Pmax, LCG_EDEVICE, "round produced more phrases than its bound");
    p_ratio = n ? (double)P / (double)n : 0.35;
    rs.table_cap = cap;
    rs.retries = retries;
    const u64 g_new = st.claims, G_new = st.claim_len;
    fail_if(ctx, L.g + g_new > kMaxRank, LCG_EOVERFLOW, "level with 2^31 rules or more");
    rs.g = g_new;
    rs.G = G_new;
    prev_ratio = P ? (double)g_new / (double)P : 0.0;
    record_hints(ctx, i, n, P, g_new, G_new);
    grow_level(ctx, L, L.g + g_new, L.G + G_new);
    if (against_resident) {
        ensure_resident(ctx, R, i, L.g + g_new);
        a.rtab_w = L.rtab;
        a.rtab_w_cap = L.rcap;
    } else {
        L.rvalid = false;
    }
    alloc_naming(ctx, b, g_new, P);
    a.g_base = L.g;
    a.G_base = L.G;
    a.cap_g = L.cap_g;
    a.cap_G = L.cap_G;
    a.rhs = L.rhs;
    a.rhs_off = L.rhs_off;
    a.F = L.F;
    enqueue_naming(ctx, a, b, (double)g_new, (double)G_new);
    in.prev_base = (u32)id_base;
    L.g += g_new;
    L.G += G_new;
    free_round(ctx, b);
    next_input(ctx, in, b);
    b = RoundBufs{};
    in.prev_cap = std::min(in.prev_cap, st.aux[1]);  // (the numbers that were taken: keys as narrow as can be)
    in.n = rc.n_next;
    in.kk = (u32)rc.k_next;
    ctx->stats.rounds = i;
}

// Sizes of the rounds of a build enqueued without host synchronisation,
// planned from the context's hints (new rules per phrase, phrases per symbol,
// symbols per rule of each level) and its plan slack.
struct RoundPlan {
    u64 n_bound = 0, n_est = 0, n_alloc = 0, cap = 0, g_alloc = 0, G_alloc = 0, t_cap = 0;
    double P_est = 0, g_est = 0, G_est = 0;
    bool tail = false;  // this round and all after it run as the short rounds (n_alloc symbols at most)
    std::vector<LevelSize> levels;  // of those rounds
};

// x rounded up to a step of 2^(1/4) (about 19 %): plans from slightly
// different hints get the same buffers, so a captured graph can be reused.
u64 bucket(u64 x) {
    if (x <= 16) return x;
    const int e = 63 - __builtin_clzll(x);
    const u64 b = 1ull << e;
    for (const double f : {1.0, 1.189207115, 1.414213562, 1.681792831, 2.0}) {
        const u64 v = (u64)std::ceil((double)b * f);
        if (v >= x) return v;
    }
    return 2 * b;
}

// What the arrays of the short rounds' levels from round r on are made for, as far as the
// context has seen such levels: twice the estimates (times the plan slack) and room for
// a few rules.  (What the rounds could have at most is far more, and a grammar keeps it:
// 100 strings of 5 kB, all alike, held 10.0 MB so, now 0.26.)
std::vector<LevelSize> tail_levels(const lcg_ctx* ctx, u32 r, double n_est) {
    std::vector<LevelSize> v;
    for (; r <= kMaxRounds && ctx->p_hint[r] > 0; r++) {
        const double P = ctx->p_hint[r] * n_est, g = ctx->ratio_hint[r] * P, sl = 2.0 * ctx->plan_slack;
        v.push_back(LevelSize{bucket((u64)(g * sl) + 512), bucket((u64)(ctx->glen_hint[r] * g * sl) + 2048)});
        n_est = P + 64;
    }
    return v;
}

std::vector<RoundPlan> plan_rounds(lcg_ctx* ctx, u64 n1, u32 kk, u32 planned) {
    std::vector<RoundPlan> v(planned + 1);
    u64 n_bound = n1, n_est = n1;
    for (u32 r = 1; r <= planned; r++) {
        RoundPlan& p = v[r];
        p.n_bound = n_bound;
        p.n_est = n_est;
        // the round's sequence is at most the planned next sequence of the
        // round before (which flags a capacity error past it)
        p.n_alloc = (r == 1) ? n_bound : std::min<u64>(n_bound, v[r - 1].t_cap);
        p.tail = is_tail(ctx, p.n_alloc);
        if (p.tail) {
            if (p.n_alloc >= kTailPlanned) p.levels = tail_levels(ctx, r, n_est);
            v.resize(r + 1);
            break;
        }
        p.P_est = ctx->p_hint[r] * (double)n_est;
        p.g_est = ctx->ratio_hint[r] * p.P_est;
        p.G_est = ctx->glen_hint[r] * p.g_est;
        // slack over the estimates: 10-25 % times the context's plan slack,
        // which grows after a plan that did not fit and shrinks while plans fit
        const double sl = ctx->plan_slack;
        p.cap = std::min<u64>(bucket(std::max<u64>(8192, (u64)(p.g_est * 1.1 * sl / ctx->tuning.table_load) + 1024)),
                              kMaxRank + 1);
        if (ctx->tuning.table_slots_max) p.cap = std::min<u64>(p.cap, ctx->tuning.table_slots_max);
        // (never more than a round can have: a context that has seen runs, then many short
        // rules, estimates their product)
        p.g_alloc = std::min<u64>(bucket((u64)(p.g_est * 1.25 * sl) + 1024), p.n_alloc / 2 + 2ull * kk + 1);
        p.G_alloc = (u64)std::min((double)p.n_alloc, p.G_est * 1.25 * sl + 4096.0);
        p.G_alloc = std::min<u64>(bucket(p.G_alloc), p.n_alloc);
        // the next sequence: the estimated phrases with the same slack (a
        // round past it flags a capacity error and the build is redone)
        p.t_cap = std::min<u64>(bucket((u64)(p.P_est * 1.1 * sl) + 4096), n_bound / 2 + 2ull * kk + 1);
        n_bound = n_bound / 2 + 2ull * kk + 1;  // every phrase but a string's first has length >= 2
        n_est = (u64)p.P_est + 64;
    }
    return v;
}

// Rounds enqueued without host synchronisation, between their enqueueing and
// the reading of their statuses.
struct AsyncRounds {
    u32 planned = 0, kk = 0;  // rounds (with those of the tail), strings
    std::vector<RoundPlan> plan;
    std::vector<u64> g_base, G_base, cap;
    u32 tail = 0;  // the first of the short rounds (0: none)
};

// Enqueue the planned rounds of a fresh build: every size comes from the plan;
// kernels read the actual sizes from the device and flag a round that
// outgrows its buffers.  b: the round at hand, for the caller to free on failure.
void rounds_async_enqueue(lcg_ctx* ctx, lcg_grammar* R, RoundInput& in, AsyncRounds& ar, RoundBufs& b) {
    const u32 kk = ar.kk;
    ar.planned = (u32)ar.plan.size() - 1;
    ar.g_base.assign(kMaxRounds + 1, 0);
    ar.G_base.assign(kMaxRounds + 1, 0);
    ar.cap.assign(kMaxRounds + 1, 0);
    for (u32 r = 1; r < ar.plan.size(); r++) {
        const RoundPlan& p = ar.plan[r];
        if (p.tail) {
            const DevStatus* before = r > 1 ? ctx->ds_arr + (r - 2) : nullptr;
            const u32 rounds = tail_enqueue(ctx, R, in, r, p.n_alloc, kk, false, before, ar.cap.data(), p.levels);
            ar.tail = r;
            ar.planned = r - 1 + rounds;
            return;
        }
        ar.cap[r] = p.cap;
        if (R->lv.size() < r) R->lv.emplace_back();
        Level& L = R->lv[r - 1];
        alloc_round(ctx, b, p.n_alloc, kk, p.t_cap);
        RoundArgs a = round_args(ctx, R, in, b, r);
        // a round stops early when the one before it failed
        if (r > 1) a.ds_prev = ctx->ds_arr + (r - 2);
        // every id is under the claims that the round before may make
        if (r > 1) a.sym_w = rank_width(in.prev_cap);
        // (the phrases first: the pool may take a while over the table, the largest
        // allocation, 0.4 ms for 0.5 GB in blocks that it has to piece together; 32 x 2 MB
        // of text 3.42 ms with the table first, 3.40 so in each of four pairs of runs)
        enqueue_phrases(ctx, a, p.n_est);
        alloc_table(ctx, b, in.symb, p.cap, p.g_alloc, kMaxRank + 1);
        set_table(a, b);
        enqueue_parse(ctx, a, p.n_est);
        grow_level(ctx, L, L.g + p.g_alloc, L.G + p.G_alloc);
        L.rvalid = false;
        // the phrases: the planned next sequence and the strings that retire
        alloc_naming(ctx, b, p.g_alloc, b.Tcap + kk);
        ar.g_base[r] = L.g;
        ar.G_base[r] = L.G;
        a.g_base = L.g;
        a.G_base = L.G;
        a.cap_g = L.cap_g;
        a.cap_G = L.cap_G;
        a.rhs = L.rhs;
        a.rhs_off = L.rhs_off;
        a.F = L.F;
        enqueue_naming(ctx, a, b, p.g_est, p.G_est);
        free_round(ctx, b);
        next_input(ctx, in, b);
        in.d_n = &a.rc->n_next;
        in.d_k = &a.rc->k_next;
        b = RoundBufs{};  // (freed, or the next round's input)
    }
}

void rounds_async_enqueue(lcg_ctx* ctx, lcg_grammar* R, RoundInput& in, AsyncRounds& ar) {
    RoundBufs b;
    try {
        rounds_async_enqueue(ctx, R, in, ar, b);
    } catch (...) {
        drop_round(ctx, b);
        throw;
    }
}

// After the enqueued rounds: read their statuses and counts (one host
// synchronisation), set the levels' sizes and the build statistics.  Returns
// 0, or -1 when a round did not fit (the build must then be redone round by
// round; -2 when it was only the arrays of a short round's level); `i` becomes the first round not yet run, and `in` its input.
int rounds_async_finish(lcg_ctx* ctx, lcg_grammar* R, RoundInput& in, const AsyncRounds& ar, u32& i) {
    const u32 planned = ar.planned;
    const u32 kk = ar.kk;
    std::vector<DevStatus> st(planned);
    std::vector<RoundCounts> rc(planned);
    fetch(ctx, {{st.data(), ctx->ds_arr, planned * sizeof(DevStatus)},
                {rc.data(), ctx->rc_arr, planned * sizeof(RoundCounts)}});
    for (u32 r = 0; r < planned; r++) {
        if (st[r].overflow || st[r].error == kErrHalted) return -1;
        if (st[r].error == kErrCapacity) {
            const Level& L = R->lv[r];
            return ar.tail && r + 1 >= ar.tail && (st[r].claims > L.cap_g || st[r].claim_len > L.cap_G) ? -2 : -1;
        }
        check_device_status(ctx, st[r]);
    }
    // rounds past the last active string (the data needed fewer rounds than
    // the previous build) leave empty levels: drop them
    u32 used = planned;
    for (u32 r = 1; r <= planned; r++) {
        const u64 k_in = (r == 1) ? kk : rc[r - 2].k_next;
        if (k_in == 0) { used = r - 1; break; }
    }
    while (R->lv.size() > used && R->lv.back().g == 0 && ar.g_base.size() > R->lv.size()) {
        if (st[R->lv.size() - 1].claims != 0) break;
        pop_level(ctx, R);
    }
    u64 n = in.n;
    for (u32 r = 1; r <= used; r++) {
        Level& L = R->lv[r - 1];
        const DevStatus& s = st[r - 1];
        const RoundCounts& c = rc[r - 1];
        fail_if(ctx, L.g + s.claims > kMaxRank, LCG_EOVERFLOW, "level with 2^31 rules or more");
        L.g = ar.g_base[r] + s.claims;
        L.G = ar.G_base[r] + s.claim_len;
        lcg_round_stats& rs = ctx->stats.round[r - 1];
        rs.n = n;
        rs.strings = (r == 1) ? kk : rc[r - 2].k_next;
        rs.phrases = c.phrases;
        rs.table_cap = ar.cap[r];
        rs.g = s.claims;
        rs.G = s.claim_len;
        record_hints(ctx, r, n, c.phrases, s.claims, s.claim_len);
        n = c.n_next;
        ctx->stats.rounds = r;
    }
    ctx->stats.async_rounds = used;
    in.n = rc[planned - 1].n_next;
    in.kk = (u32)rc[planned - 1].k_next;
    in.d_n = nullptr;
    in.d_k = nullptr;
    i = planned + 1;
    return 0;
}

u32 planned_rounds(const lcg_ctx* ctx) {
    return std::min<u32>(ctx->hint_rounds, std::min<u32>(ctx->levels - 1, kMaxRounds));
}

// The rounds of a fresh build, enqueued without host synchronisation and
// planned from the context's previous builds.
int rounds_async(lcg_ctx* ctx, lcg_grammar* R, RoundInput& in, u32& i) {
    AsyncRounds ar;
    ar.planned = planned_rounds(ctx);
    ar.kk = in.kk;
    ar.plan = plan_rounds(ctx, in.n, in.kk, ar.planned);
    rounds_async_enqueue(ctx, R, in, ar);
    return rounds_async_finish(ctx, R, in, ar, i);
}

// ---- the rounds of a build as one CUDA graph ------------------------------
//
// A context's builds of one shape (the same device input buffer, string
// lengths and plan) can run as one captured graph: the first such build
// captures every round's allocations, memsets and launches (the planned
// rounds, as enqueued without host synchronisation), later builds launch it.
// The graph writes the grammar into its own allocations, which keep their
// addresses at every launch: a launch therefore waits until the grammar of
// the previous launch has been freed (a serving loop's build -> use -> free),
// and otherwise the build runs as launches.  The graph resets the single-pass
// tile counter and the look-back flags it uses; the string offsets of round 1
// are uploaded to buffers outside the graph before each launch.

struct GraphBuild {
    // what the launches depend on
    const unsigned char* d_in = nullptr;
    u64 n1 = 0;
    u32 k = 0;
    std::vector<u64> lens;
    std::vector<double> params;  // planned rounds and launch parameters (graph_params)
    // round-1 offsets and ids, outside the graph
    u64* soff = nullptr;
    u32* sid = nullptr;
    std::shared_ptr<GraphHold> hold;
    lcg_grammar shape;  // host description of the grammar a launch writes
    AsyncRounds ar;
    u64 ctr_end = 0;    // tile counter after a launch
    u64 launches = 0;   // kernels per launch
    std::vector<lcg_ctx::KRec> krecs;  // timing events recorded by the graph
    lcg_grammar* live = nullptr;       // grammar of the last launch, until freed
};

// What a graph's launches depend on besides the input and the planned buffer
// sizes: the number of planned rounds and the launch parameters.
std::vector<double> graph_params(lcg_ctx* ctx, u32 planned) {
    return {(double)planned,    (double)ctx->tuning.parse_blocks_per_sm, (double)ctx->ktime,
            (double)ctx->tuning.tile_stripes, (double)ctx->tuning.parse_tile, (double)ctx->tuning.parse_tile_min};
}

// A captured graph serves a new plan when each of its rounds' buffers holds
// the new plan's (the kernels read the actual sizes from the device, so a
// larger buffer changes nothing but memory), and its phrase tables are not
// more than 4x the new plan's (a table far larger than needed costs its
// clearing and L2 room).  Hints that decay and a plan slack that shrinks
// after every build that fits therefore keep the graph; a plan that grows
// past it, or shrinks far below it, captures a new one.
bool plan_covers(const std::vector<RoundPlan>& have, const std::vector<RoundPlan>& need) {
    if (have.size() != need.size()) return false;
    for (size_t r = 1; r < have.size(); r++) {
        const RoundPlan& h = have[r];
        const RoundPlan& n = need[r];
        if (h.tail || n.tail) {
            if (!h.tail || !n.tail || h.n_alloc < n.n_alloc || h.levels.size() > n.levels.size()) return false;
            // (a plan is for twice the estimates; levels that the plan at hand does not name
            // have room for all they can have)
            for (size_t l = 0; l < h.levels.size(); l++)
                if (2 * h.levels[l].g < n.levels[l].g || 2 * h.levels[l].G < n.levels[l].G) return false;
            return true;
        }
        if (h.n_bound != n.n_bound || h.n_alloc < n.n_alloc || h.cap < n.cap || h.cap > 4 * n.cap ||
            h.g_alloc < n.g_alloc || h.G_alloc < n.G_alloc || h.t_cap < n.t_cap)
            return false;
    }
    return true;
}

void destroy_graph(lcg_ctx* ctx) {
    GraphBuild* gb = ctx->graph;
    if (!gb) return;
    cudaStreamSynchronize(ctx->st);
    // the records of the last launch name the graph's events: they go with them
    ctx->krecs.erase(std::remove_if(ctx->krecs.begin(), ctx->krecs.end(),
                                    [](const lcg_ctx::KRec& r) { return r.graph; }),
                     ctx->krecs.end());
    for (auto& r : gb->krecs) {
        if (r.part) continue;
        cudaEventDestroy(r.a);
        cudaEventDestroy(r.b);
    }
    if (gb->soff) cudaFreeAsync(gb->soff, ctx->st);
    if (gb->sid) cudaFreeAsync(gb->sid, ctx->st);
    ctx->graph = nullptr;
    cudaStreamSynchronize(ctx->st);
    const bool kept = gb->hold.use_count() > 1;
    delete gb;  // (and the graph, or with its live grammar)
    // what the graph does not hold for that grammar goes back to the device now
    if (kept) cudaDeviceGraphMemTrim(ctx->device);
}

void graph_grammar_freed(lcg_ctx* ctx, const lcg_grammar* G) {
    if (ctx->graph && ctx->graph->live == G) ctx->graph->live = nullptr;
}

// Capture the planned rounds of a build of this shape (nothing runs yet).
void capture_graph(lcg_ctx* ctx, const unsigned char* d_in, const std::vector<u64>& lens, u32 planned,
                   std::vector<double> params) {
    destroy_graph(ctx);
    const u32 k = (u32)lens.size();
    u64 n1 = 0;
    for (u64 x : lens) n1 += x;
    std::vector<RoundPlan> plan = plan_rounds(ctx, n1, k, planned);
    // look-back buffers and timing events for every launch, made before the
    // capture (the graph must not reallocate them)
    u64 t1 = 1, t2 = 1, hs = 1;
    for (u32 r = 1; r < plan.size(); r++) {
        const RoundPlan& p = plan[r];
        if (p.tail) {
            hs = std::max(hs, breaks_steps((kTailSymbols + parse_unit(1024) - 1) / parse_unit(1024), parse_unit(1024)));
            break;
        }
        const u32 tp = parse_unit(round_tile(ctx, p.n_alloc));
        const u64 tiles = (p.n_alloc + tp - 1) / tp;
        t1 = std::max({t1, popscan_tiles_for((p.t_cap + k) / 32 + 1), rule_offs_tiles(std::max<u64>(1, p.g_alloc))});
        t2 = std::max(t2, scan2_tiles_for(tiles));
        hs = std::max(hs, breaks_steps(tiles, tp));
    }
    ensure_lb(ctx, &ctx->lb1, &ctx->lb1_tiles, t1, lb1_bytes(t1));
    ensure_lb(ctx, &ctx->lb2, &ctx->lb2_tiles, t2, scan2_lb_bytes(t2));
    ensure_lb(ctx, &ctx->heads, &ctx->heads_steps, hs, hs * sizeof(u64));
    auto* gb = new GraphBuild;
    ctx->graph = gb;
    gb->d_in = d_in;
    gb->k = k;
    gb->lens = lens;
    gb->params = std::move(params);
    gb->hold = std::make_shared<GraphHold>();
    gb->hold->device = ctx->device;
    gb->n1 = n1;
    gb->soff = dalloc<u64>(ctx, k + 1);
    gb->sid = dalloc<u32>(ctx, k);
    gb->ar.planned = planned;
    gb->ar.kk = k;
    gb->ar.plan = std::move(plan);
    if (ctx->ktime)
        while (ctx->evpool.size() < 24ull * planned + 8) {
            cudaEvent_t e;
            ck(ctx, cudaEventCreate(&e), "cudaEventCreate");
            ctx->evpool.push_back(e);
        }
    sync(ctx);
    const size_t krec0 = ctx->krecs.size();
    const u64 launches0 = ctx->launches;
    const u64 ctr_before = ctx->ctr_val;  // the device counter until the graph runs
    ck(ctx, cudaStreamBeginCapture(ctx->st, cudaStreamCaptureModeThreadLocal), "begin capture");
    ctx->capturing = true;
    lcg_grammar* T = nullptr;
    try {
        ck(ctx, cudaMemsetAsync(ctx->ctr, 0, sizeof(u64), ctx->st), "reset tile counter");
        ctx->ctr_val = 0;
        ck(ctx, cudaMemsetAsync(ctx->lb1, 0, lb1_bytes(ctx->lb1_tiles), ctx->st), "reset look-back");
        // the graph's launches reuse its epochs: heads of the last launch must not read as published
        ck(ctx, cudaMemsetAsync(ctx->heads, 0, ctx->heads_steps * sizeof(u64), ctx->st), "reset heads");
        ck(ctx, cudaMemsetAsync(ctx->lb2, 0, scan2_lb_bytes(ctx->lb2_tiles), ctx->st), "reset look-back");
        T = new_grammar(ctx, false);
        grow_c(ctx, T, k);
        T->k = k;
        ck(ctx, cudaMemsetAsync(ctx->ds_arr, 0, kMaxRounds * sizeof(DevStatus), ctx->st), "reset status");
        ck(ctx, cudaMemsetAsync(ctx->rc_arr, 0, kMaxRounds * sizeof(RoundCounts), ctx->st), "reset counts");
        RoundInput in{};
        in.S = d_in;
        in.symb = 1;
        in.n = in.n_cap = gb->n1;
        in.kk = k;
        in.soff = gb->soff;
        in.sid = gb->sid;
        in.own_offsets = false;
        rounds_async_enqueue(ctx, T, in, gb->ar);
        free_round_input(ctx, in);  // the last round's outputs: the graph's own allocations
    } catch (...) {
        ctx->capturing = false;
        cudaGraph_t g = nullptr;
        cudaStreamEndCapture(ctx->st, &g);
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();  // (frees of a capture that was abandoned)
        delete T;
        ctx->ctr_val = ctr_before;
        destroy_graph(ctx);
        throw;
    }
    ctx->capturing = false;
    const cudaError_t e = cudaStreamEndCapture(ctx->st, &gb->hold->graph);
    gb->ctr_end = ctx->ctr_val;
    ctx->ctr_val = ctr_before;
    if (e != cudaSuccess) {
        delete T;
        destroy_graph(ctx);
        ck(ctx, e, "end capture");
    }
    gb->shape = *T;
    delete T;  // host object only: its device arrays are the graph's allocations
    gb->launches = ctx->launches - launches0;
    for (size_t x = krec0; x < ctx->krecs.size(); x++) {
        gb->krecs.push_back(ctx->krecs[x]);
        gb->krecs.back().graph = true;
    }
    ctx->krecs.resize(krec0);
    const cudaError_t ei = cudaGraphInstantiate(&gb->hold->exec, gb->hold->graph, 0);
    if (ei != cudaSuccess) {
        destroy_graph(ctx);
        ck(ctx, ei, "instantiate graph");
    }
}

// A build as a launch of the context's graph (captured first when the shape
// is new).  Returns the grammar, or nullptr when the build must run as
// launches (the graph's last grammar is still in use); throws Retry when the
// planned rounds did not fit.
lcg_grammar* build_with_graph(lcg_ctx* ctx, const unsigned char* d_in, const std::vector<u64>& lens) {
    const u32 k = (u32)lens.size();
    const u32 planned = planned_rounds(ctx);
    u64 n1 = 0;
    for (u64 x : lens) n1 += x;
    std::vector<double> params = graph_params(ctx, planned);
    GraphBuild* gb = ctx->graph;
    const bool same = gb && gb->d_in == d_in && gb->lens == lens && gb->params == params &&
                      plan_covers(gb->ar.plan, plan_rounds(ctx, n1, k, planned));
    if (same && gb->live) return nullptr;
    const u32 mode = same ? 2 : 1;
    if (!same) {
        capture_graph(ctx, d_in, lens, planned, std::move(params));
        gb = ctx->graph;
    }
    std::vector<u64> soff_h(k + 1, 0);
    std::vector<u32> sid_h(k);
    for (u32 j = 0; j < k; j++) {
        soff_h[j + 1] = soff_h[j] + lens[j];
        sid_h[j] = j;
    }
    ctx->stats = lcg_build_stats{};
    ctx->stats.input_bytes = gb->n1;
    ck(ctx, cudaMemcpyAsync(gb->soff, soff_h.data(), (k + 1) * sizeof(u64), cudaMemcpyHostToDevice, ctx->st),
       "upload offsets");
    ck(ctx, cudaMemcpyAsync(gb->sid, sid_h.data(), k * sizeof(u32), cudaMemcpyHostToDevice, ctx->st), "upload ids");
    cudaError_t el = cudaGraphLaunch(gb->hold->exec, ctx->st);
    if (el == cudaErrorMemoryAllocation) {
        // the graph has memory of its own beside the pool's: what earlier builds left in
        // the pool goes back to the device
        cudaGetLastError();
        sync(ctx);
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, ctx->device) == cudaSuccess) cudaMemPoolTrimTo(pool, 0);
        el = cudaGraphLaunch(gb->hold->exec, ctx->st);
    }
    ck(ctx, el, "graph launch");
    ctx->ctr_val = gb->ctr_end;
    ctx->launches += gb->launches;
    for (const auto& r : gb->krecs) ctx->krecs.push_back(r);
    lcg_grammar* G = new lcg_grammar(gb->shape);
    G->owner = ctx;
    ctx->live.push_back(G);
    G->hold = gb->hold;
    gb->live = G;
    RoundInput in{};
    in.n = gb->n1;
    in.kk = k;
    u32 i = 0;
    int r;
    try {
        r = rounds_async_finish(ctx, G, in, gb->ar, i);
    } catch (...) {
        free_grammar_now(G);
        throw;
    }
    if (r < 0 || in.kk > 0) {  // did not fit, or more rounds are needed: run as launches
        free_grammar_now(G);
        throw Retry{r == -2};
    }
    ctx->hint_rounds = ctx->stats.rounds;
    ctx->stats.kernel_launches = gb->launches;
    ctx->stats.graph = mode;
    return G;
}

// All rounds of a build: planned ones if there is a plan, then round by round.
void build_rounds(lcg_ctx* ctx, lcg_grammar* R, RoundInput& in, RoundBufs& b, bool against_resident, bool allow_async) {
    u32 i = 1;
    if (allow_async && !against_resident && ctx->hint_rounds > 0) {
        const int r = rounds_async(ctx, R, in, i);
        // a round outgrew its estimate: the caller starts again with synchronised rounds
        if (r < 0) throw Retry{r == -2};
    }
    double prev_ratio = 0.0, p_ratio = 0.35;
    while (in.kk > 0) {
        if (is_tail(ctx, in.n, against_resident ? R : nullptr)) tail_sync(ctx, R, in, i, against_resident);
        else round_sync(ctx, R, in, i++, against_resident, prev_ratio, p_ratio, b);
    }
}

void build_into(lcg_ctx* ctx, lcg_grammar* R, const uint8_t* data, const uint64_t* off, uint32_t k, int on_dev,
                bool against_resident, bool allow_async) {
    fail_if(ctx, k == 0 || off == nullptr || data == nullptr, LCG_EINVAL, "empty collection");
    fail_if(ctx, (u64)R->k + k > 0xffffffffull, LCG_EOVERFLOW, "too many strings");
    std::vector<u64> act_src, act_len, lvl0_pos;
    std::vector<u32> act_id, lvl0_id;
    for (u32 j = 0; j < k; j++) {
        fail_if(ctx, off[j + 1] <= off[j], LCG_EINVAL, "string " + std::to_string(j) + " is empty");
        const u64 len = off[j + 1] - off[j];
        if (len == 1) {
            lvl0_pos.push_back(off[j] - off[0]);
            lvl0_id.push_back(R->k + j);
        } else {
            act_src.push_back(off[j] - off[0]);
            act_len.push_back(len);
            act_id.push_back(R->k + j);
        }
    }
    ctx->stats = lcg_build_stats{};
    ctx->stats.input_bytes = off[k] - off[0];
    const u64 launches0 = ctx->launches;
    Temps owned(ctx);

    const u64 nbytes = off[k] - off[0];
    const unsigned char* d_in;
    if (on_dev) {
        d_in = data + off[0];
    } else {
        unsigned char* p = owned.get<unsigned char>(nbytes);
        ck(ctx, cudaMemcpyAsync(p, data + off[0], nbytes, cudaMemcpyHostToDevice, ctx->st), "copy input");
        d_in = p;
    }
    const u32 kbase = R->k;
    grow_c(ctx, R, R->k + k);
    R->k += k;

    if (!lvl0_id.empty()) {
        u64* dpos = owned.get<u64>(lvl0_pos.size());
        u32* dids = owned.get<u32>(lvl0_id.size());
        ck(ctx, cudaMemcpyAsync(dpos, lvl0_pos.data(), lvl0_pos.size() * 8, cudaMemcpyHostToDevice, ctx->st), "copy");
        ck(ctx, cudaMemcpyAsync(dids, lvl0_id.data(), lvl0_id.size() * 4, cudaMemcpyHostToDevice, ctx->st), "copy");
        ck(ctx, launch_level0(d_in, dpos, dids, (u32)lvl0_id.size(), R->c_level, R->c_rank, ctx->st), "level0");
        ctx->launches++;
    }
    (void)kbase;
    u32 kk = (u32)act_id.size();
    if (kk == 0) {
        sync(ctx);
        ctx->stats.kernel_launches = ctx->launches - launches0;
        return;
    }
    // round-1 sequence: the active strings back to back
    std::vector<u64> soff_h(kk + 1, 0);
    for (u32 x = 0; x < kk; x++) soff_h[x + 1] = soff_h[x] + act_len[x];
    const u64 n1 = soff_h[kk];
    Temps first(ctx);  // the first round's input, until it is the rounds' to free
    u64* d_soff = first.get<u64>(kk + 1);
    u32* d_sid = first.get<u32>(kk);
    ck(ctx, cudaMemcpyAsync(d_soff, soff_h.data(), (kk + 1) * 8, cudaMemcpyHostToDevice, ctx->st), "copy soff");
    ck(ctx, cudaMemcpyAsync(d_sid, act_id.data(), kk * 4, cudaMemcpyHostToDevice, ctx->st), "copy sid");
    const void* S = d_in;
    void* S_owned = nullptr;
    if (!lvl0_id.empty()) {
        unsigned char* g = first.get<unsigned char>(n1);
        u64* dsrc = owned.get<u64>(kk);
        ck(ctx, cudaMemcpyAsync(dsrc, act_src.data(), kk * 8, cudaMemcpyHostToDevice, ctx->st), "copy");
        ck(ctx, launch_gather_strings(d_in, dsrc, d_soff, kk, g, ctx->st), "gather");
        ctx->launches++;
        S = g;
        S_owned = g;
    }
    RoundInput in{};
    in.S = S;
    in.S_owned = S_owned;
    in.Sf = nullptr;
    in.symb = 1;
    in.n = in.n_cap = n1;
    in.kk = kk;
    in.soff = d_soff;
    in.sid = d_sid;
    ck(ctx, cudaMemsetAsync(ctx->ds_arr, 0, kMaxRounds * sizeof(DevStatus), ctx->st), "reset status");
    ck(ctx, cudaMemsetAsync(ctx->rc_arr, 0, kMaxRounds * sizeof(RoundCounts), ctx->st), "reset counts");
    first.ptrs.clear();
    RoundBufs b;  // of the round at hand
    try {
        build_rounds(ctx, R, in, b, against_resident, allow_async);
        check_device_status(ctx, read_status(ctx));
    } catch (...) {
        drop_round(ctx, b);
        free_round_input(ctx, in);
        throw;
    }
    ctx->hint_rounds = ctx->stats.rounds;
    free_round_input(ctx, in);
    ctx->stats.kernel_launches = ctx->launches - launches0;
}

// --------------------------------------------------------------------------
// MergeGrams
// --------------------------------------------------------------------------

// A level grows to what it may need at most, without waiting for what it does
// need, up to this many rules and symbols (16 + 8 MB; a doubling of the arrays adds
// as much).
constexpr u64 kMergeAheadRules = 1ull << 20, kMergeAheadSymbols = 1ull << 21;

// The levels i0 + 1 .. of G_b, all of them small, in one launch.  `temps` gets what is
// to be freed afterwards.
void merge_small(lcg_ctx* ctx, lcg_grammar* A, const lcg_grammar* B, u32 i0, const u32* Mprev, u64* bar, u64* d_tot,
                 u32* cb_rank, std::vector<void*>& temps) {
    const u32 nb = (u32)B->lv.size();
    const u32 blocks = coop_blocks(ctx);
    MergeSmall a{};
    a.bar = bar;
    Parts tmp, grown;
    struct At {
        u64 M, off, F, rhs, cap_g, cap_G;
        bool rules, syms, table;
    };
    std::vector<At> at;
    const u64 counts = tmp.take(2 * (u64)blocks * sizeof(u64));
    // all that can fail but the launch itself comes before G_a changes
    std::vector<Level> lv = A->lv;  // G_a's levels as they will be
    if (lv.size() < nb) lv.resize(nb);
    for (u32 i = i0 + 1; i <= nb; i++) {
        const Level &LA = lv[i - 1], &LB = B->lv[i - 1];
        At x{};
        x.M = tmp.take(LB.g * sizeof(u32));
        x.rules = LA.rhs_off == nullptr || LA.g + LB.g > LA.cap_g;
        x.syms = LA.rhs == nullptr || LA.G + LB.G > LA.cap_G;
        x.table = !(LA.rvalid && LA.rcap >= 2 * (LA.g + LB.g));
        if (x.rules) {
            x.cap_g = std::max<u64>({LA.g + LB.g, 2 * LA.cap_g, 256});
            x.off = grown.take((x.cap_g + 1) * sizeof(u64));
            x.F = grown.take(x.cap_g * sizeof(u32));
        }
        if (x.syms) {
            x.cap_G = std::max<u64>({LA.G + LB.G, 2 * LA.cap_G, 1024});
            x.rhs = grown.take(x.cap_G * sizeof(u32));
        }
        at.push_back(x);
    }
    Temps fresh(ctx);  // what the levels get
    unsigned char* t = fresh.get<unsigned char>(tmp.size);
    a.counts = (u64*)(t + counts);
    unsigned char* g = grown.size ? fresh.get<unsigned char>(grown.size) : nullptr;
    std::vector<void*> old;  // and what they had
    const u32* F_below = i0 == 0 ? A->F0 : lv[i0 - 1].F;
    for (u32 i = i0 + 1; i <= nb; i++) {
        Level& LA = lv[i - 1];
        const Level& LB = B->lv[i - 1];
        const At& x = at[i - i0 - 1];
        MergeLevel& m = a.lv[a.levels];
        MergeOld& o = a.old[a.levels];
        if (x.rules) {
            o.off = LA.rhs_off;
            o.F = LA.F;
            o.first = LA.rhs_off == nullptr;
            if (LA.rhs_off && !LA.shared_rules) {
                old.push_back(LA.rhs_off);
                old.push_back(LA.F);
            }
            LA.rhs_off = (u64*)(g + x.off);
            LA.F = (u32*)(g + x.F);
            LA.cap_g = x.cap_g;
            LA.shared_rules = true;
        }
        if (x.syms) {
            o.rhs = LA.rhs;
            if (LA.rhs && !LA.shared_rhs) old.push_back(LA.rhs);
            LA.rhs = (u32*)(g + x.rhs);
            LA.cap_G = x.cap_G;
            LA.shared_rhs = true;
        }
        if (x.table) {
            if (LA.rtab) old.push_back(LA.rtab);
            LA.rcap = std::max<u64>(1024, 3 * (LA.g + LB.g));
            LA.rtab = fresh.get<unsigned char>(LA.rcap * slot_bytes());
            o.fresh = true;
        }
        LA.rvalid = false;
        m.brhs = LB.rhs;
        m.boff = LB.rhs_off;
        m.bF = LB.F;
        m.gb = LB.g;
        m.M = (u32*)(t + x.M);
        m.Mprev = Mprev;
        m.aFprev = F_below;
        m.lh = level_hash(ctx, i);
        m.slots = LA.rtab;
        m.cap = LA.rcap;
        m.arhs = LA.rhs;
        m.aoff = LA.rhs_off;
        m.aF = LA.F;
        m.ga = LA.g;
        m.Ga = LA.G;
        m.c_level = B->c_level;
        m.c_rank = B->c_rank;
        m.c_out = cb_rank;
        m.kb = B->k;
        m.level = i;
        m.ds = ctx->ds;
        a.totals[a.levels++] = d_tot + 2 * (size_t)(i - 1);
        Mprev = m.M;
        F_below = LA.F;
    }
    temps.reserve(temps.size() + old.size() + 1);
    A->slabs.reserve(A->slabs.size() + 1);
    ck(ctx, launch_merge_small(a, blocks, ctx->st), "merge levels");
    ctx->launches++;
    fresh.ptrs.clear();
    A->lv.swap(lv);
    if (g) A->slabs.push_back(g);
    temps.push_back(t);
    temps.insert(temps.end(), old.begin(), old.end());
}

// All levels are enqueued before the host waits once, but for a level that is large
// and does not fit its arrays whatever G_b adds: there the host reads what it adds.
// G_a's sizes are set at the end, so that a failure leaves G_a as it was.
void merge(lcg_ctx* ctx, lcg_grammar* A, const lcg_grammar* B) {
    fail_if(ctx, A == B, LCG_EINVAL, "cannot merge a grammar into itself");
    fail_if(ctx, A->tag != B->tag || A->tag != ctx->tag, LCG_EMISMATCH, "grammars of different hash families");
    fail_if(ctx, (u64)A->k + B->k > 0xffffffffull, LCG_EOVERFLOW, "too many strings");
    const u32 kb = B->k;
    const u32 nb = (u32)B->lv.size();
    const size_t na = A->lv.size();
    std::vector<u64> tot(2 * (size_t)nb, 0);
    std::vector<void*> temps;
    auto temp = [&](auto* p) {
        temps.push_back(p);
        return p;
    };
    try {
        u32* cb_rank = temp(dalloc<u32>(ctx, kb));
        u64* d_tot = temp(dalloc<u64>(ctx, 2 * (size_t)nb + 2));  // and the small levels' barrier
        ck(ctx, cudaMemsetAsync(d_tot, 0, (tot.size() + 2) * 8, ctx->st), "memset totals");
        if (kb) ck(ctx, cudaMemcpyAsync(cb_rank, B->c_rank, kb * 4, cudaMemcpyDeviceToDevice, ctx->st), "copy");
        const u32* Mprev = nullptr;
        u32 large = nb;  // levels before the small ones
        while (large > 0 && nb - large < kMergeSmallLevels) {
            const Level& LB = B->lv[large - 1];
            const u64 g = LB.g + (large <= A->lv.size() ? A->lv[large - 1].g : 0);
            const u64 G = LB.G + (large <= A->lv.size() ? A->lv[large - 1].G : 0);
            if (LB.g == 0 || g > kMergeSmallRules || G > kMergeSmallSymbols) break;
            large--;
        }
        for (u32 i = 1; i <= large; i++) {
            if (A->lv.size() < i) A->lv.emplace_back();
            Level& LA = A->lv[i - 1];
            const Level& LB = B->lv[i - 1];
            const u64 gb = LB.g;
            if (LA.rhs_off == nullptr) grow_level(ctx, LA, 0, 0);
            if (gb == 0) {
                Mprev = nullptr;
                continue;
            }
            ensure_resident(ctx, A, i, LA.g + gb);
            LA.rvalid = false;  // until the rules it will hold are the level's
            MergeLevel m{};
            m.brhs = LB.rhs;
            m.boff = LB.rhs_off;
            m.bF = LB.F;
            m.gb = gb;
            m.Mprev = Mprev;
            m.aFprev = fprev_of(A, i);
            m.lh = level_hash(ctx, i);
            m.slots = LA.rtab;
            m.cap = LA.rcap;
            m.ga = LA.g;
            m.Ga = LA.G;
            // one allocation per level for the ranks (kept for the next level) and one
            // for what this level alone needs
            m.M = temp(dalloc<u32>(ctx, gb));
            u64* x = dalloc<u64>(ctx, 3 * gb);
            temps.push_back(x);
            m.xrank = x;
            m.xlen = x + gb;
            m.miss = (u32*)(x + 2 * gb);
            m.mlen = m.miss + gb;
            m.totals = d_tot + 2 * (size_t)(i - 1);
            m.c_level = B->c_level;
            m.c_rank = B->c_rank;
            m.c_out = cb_rank;
            m.kb = kb;
            m.level = i;
            m.ds = ctx->ds;
            const u64 stiles = std::max<u64>(1, scan2_tiles_for(gb));
            ensure_lb(ctx, &ctx->lb2, &ctx->lb2_tiles, stiles, scan2_lb_bytes(stiles));
            // (the lookup reads G_a's arrays as they are before they grow)
            m.arhs = LA.rhs;
            m.aoff = LA.rhs_off;
            m.aF = LA.F;
            ck(ctx, launch_merge_lookup(m, i == 1, ctx->st), "merge lookup");
            u64 grid = 0;
            ck(ctx, launch_scan2(m.miss, m.mlen, gb, x, x + gb, d_tot + 2 * (size_t)(i - 1), ctx->lb2, ++ctx->epoch,
                                 ctx->ctr, ctx->ctr_val, ctx->ds, ctx->st, &grid),
               "scan");
            ctx->ctr_val += grid;
            ctx->launches += 2;
            u64 more[2] = {gb, LB.G};
            const bool fits = m.ga + gb <= LA.cap_g && m.Ga + LB.G <= LA.cap_G;
            if (m.ga + gb > kMaxRank || (!fits && (m.ga + gb > kMergeAheadRules || m.Ga + LB.G > kMergeAheadSymbols))) {
                check_device_status(ctx, read_status(ctx, more, m.totals, 16));
                fail_if(ctx, m.ga + more[0] > kMaxRank, LCG_EOVERFLOW, "level with 2^31 rules or more");
            }
            grow_level(ctx, LA, m.ga + more[0], m.Ga + more[1]);
            m.arhs = LA.rhs;
            m.aoff = LA.rhs_off;
            m.aF = LA.F;
            ck(ctx, launch_merge_append(m, i == 1, ctx->st), "merge append");
            ctx->launches++;
            dfree(ctx, temps.back());
            temps.pop_back();
            Mprev = m.M;
        }
        if (large < nb) merge_small(ctx, A, B, large, Mprev, d_tot + tot.size(), d_tot, cb_rank, temps);
        grow_c(ctx, A, A->k + kb);
        if (kb) {
            ck(ctx, cudaMemcpyAsync(A->c_level + A->k, B->c_level, kb * 4, cudaMemcpyDeviceToDevice, ctx->st), "copy");
            ck(ctx, cudaMemcpyAsync(A->c_rank + A->k, cb_rank, kb * 4, cudaMemcpyDeviceToDevice, ctx->st), "copy");
        }
        check_device_status(ctx, read_status(ctx, tot.data(), d_tot, tot.size() * 8));
    } catch (...) {
        for (void* p : temps) dfree(ctx, p);
        while (A->lv.size() > na) pop_level(ctx, A);  // the levels that only G_b has
        throw;
    }
    for (void* p : temps) dfree(ctx, p);
    for (u32 i = 0; i < nb; i++) {
        Level& L = A->lv[i];
        if (B->lv[i].g == 0) continue;
        L.g += tot[2 * (size_t)i];
        L.G += tot[2 * (size_t)i + 1];
        L.rvalid = true;
    }
    A->k += kb;
}

// --------------------------------------------------------------------------
// exp(C[j])
// --------------------------------------------------------------------------

void decompress(lcg_ctx* ctx, const lcg_grammar* G, u32 j, uint8_t* out, u64 cap, uint64_t* out_len, int on_dev) {
    fail_if(ctx, j >= G->k, LCG_EINVAL, "string index out of range");
    // the upper levels, and the whole of a short string, in one launch
    ExpandState st{1, 0, 0};
    Temps temps(ctx);
    bool waited = false;  // for all that was enqueued
    u32 *cur = nullptr, *own = nullptr;  // the sequence, and the allocation that holds it
    u8* tmp = nullptr;  // bytes for a host buffer
    if (G->lv.size() <= 64) {
        ExpandLevels lv{};
        for (size_t l = 0; l < G->lv.size(); l++) {
            lv.off[l] = G->lv[l].rhs_off;
            lv.rhs[l] = G->lv[l].rhs;
        }
        cur = temps.get<u32>(kExpandSmall);
        if (!on_dev) tmp = temps.get<u8>(kExpandSmallBytes);
        ExpandState* d = (ExpandState*)(ctx->scratch + 4);
        ck(ctx, launch_expand_small(lv, G->c_level, G->c_rank, j, on_dev ? out : tmp,
                                    on_dev ? cap : std::min<u64>(cap, kExpandSmallBytes), cur, d, ctx->st),
           "k_expand_small");
        ctx->launches++;
        fetch(ctx, {{&st, d, sizeof(st)}});
        waited = st.level == 0 && on_dev;  // the whole string, in its place
        own = cur;
        // (the launches after it are judged by the status; what an earlier call left there
        // is not theirs)
        if (st.level >= 1) reset_status(ctx);
        if (st.level >= 2) {
            const u32 blocks = coop_blocks(ctx);
            u64* words = temps.get<u64>(2 + blocks);
            u32* mid = temps.get<u32>(2 * kExpandMid);
            ck(ctx, cudaMemsetAsync(words, 0, 2 * sizeof(u64), ctx->st), "memset barrier");
            ck(ctx, launch_expand_mid(lv, cur, mid, words + 2, words, d, ctx->ds, blocks, ctx->st), "k_expand_mid");
            ctx->launches++;
            temps.drop(words);
            check_device_status(ctx, read_status(ctx, &st, d, sizeof(st)));
            if (st.which < 2) {
                temps.drop(own);
                own = mid;
                cur = mid + st.which * kExpandMid;
            } else {
                temps.drop(mid);
            }
        }
    } else {
        u32 r = 0;
        ck(ctx, cudaMemcpyAsync(&st.level, G->c_level + j, 4, cudaMemcpyDeviceToHost, ctx->st), "read C");
        ck(ctx, cudaMemcpyAsync(&r, G->c_rank + j, 4, cudaMemcpyDeviceToHost, ctx->st), "read C");
        reset_status(ctx);
        own = cur = temps.get<u32>(1);
        ck(ctx, cudaMemcpyAsync(cur, G->c_rank + j, 4, cudaMemcpyDeviceToDevice, ctx->st), "copy");
        sync(ctx);
        if (st.level == 0 && cap >= 1) {
            const u8 b = (u8)r;
            if (!on_dev) tmp = temps.get<u8>(1);
            ck(ctx, cudaMemcpyAsync(on_dev ? out : tmp, &b, 1, cudaMemcpyHostToDevice, ctx->st), "copy");
        }
    }
    u64 cnt = st.count;
    auto too_small = [&] {
        *out_len = cnt;
        fail_if(ctx, true, LCG_EINVAL, "output buffer too small");
    };
    if (st.level == 0 && cap < cnt) too_small();
    for (u32 l = st.level; l >= 1; l--) {
        const Level& L = G->lv[l - 1];
        const u64 tiles = expand_tiles_for(cnt);
        u32* sums = temps.get<u32>(2 * tiles);
        u64* places = temps.get<u64>(2 * tiles);
        ck(ctx, launch_expand_count(cur, cnt, L.rhs_off, sums, sums + tiles, ctx->st), "k_expand_count");
        const u64 stiles = std::max<u64>(1, scan2_tiles_for(tiles));
        ensure_lb(ctx, &ctx->lb2, &ctx->lb2_tiles, stiles, scan2_lb_bytes(stiles));
        u64 grid = 0, tot[2] = {0, 0};
        ck(ctx, launch_scan2(sums, sums + tiles, tiles, places, places + tiles, ctx->scratch + 1, ctx->lb2,
                             ++ctx->epoch, ctx->ctr, ctx->ctr_val, ctx->ds, ctx->st, &grid),
           "scan");
        ctx->ctr_val += grid;
        check_device_status(ctx, read_status(ctx, tot, ctx->scratch + 1, 16));
        const u64 total = tot[0] + (tot[1] << 32);
        u32* next = nullptr;
        u8 *bytes = nullptr, *packed = nullptr;
        if (l == 1) {
            if (cap < total) {
                cnt = total;
                too_small();
            }
            if (!on_dev) {
                temps.drop(tmp);
                tmp = temps.get<u8>(total);
            }
            bytes = on_dev ? out : tmp;
            // the level's right-hand sides as bytes, when they are read several times
            if (total >= 4 * L.G) {
                packed = temps.get<u8>(L.G + 16);
                ck(ctx, launch_expand_pack(L.rhs, L.G, packed, ctx->st), "k_expand_pack");
                ctx->launches++;
            }
        } else {
            next = temps.get<u32>(total);
        }
        ck(ctx, launch_expand_tiles(cur, cnt, L.rhs_off, L.rhs, packed, places, places + tiles, next, bytes, ctx->st),
           "k_expand_tiles");
        ctx->launches += 3;
        for (void* p : {(void*)packed, (void*)sums, (void*)places, (void*)own}) temps.drop(p);
        own = cur = next;
        cnt = total;
    }
    *out_len = cnt;
    if (!on_dev) ck(ctx, cudaMemcpyAsync(out, tmp, cnt, cudaMemcpyDeviceToHost, ctx->st), "copy out");
    if (!waited) sync(ctx);
}

// --------------------------------------------------------------------------
// exp(C[j]) without allocation: scratch in a static device array
// --------------------------------------------------------------------------
//
// For callers that must not allocate device memory when they expand a string:
// code that runs inside an allocator's or a memory-pressure callback (it
// cannot call back into the allocator), and services that reserve their
// device memory up front and keep no room for transient buffers.  The scratch
// lives in this file-scope array, which every GPU that loads the library
// holds until the process exits.  Host code cannot use the array's name as a
// device address: its address is taken once per device, with that device
// current, by cudaGetSymbolAddress (under a lock, as contexts on several host
// threads may make their first call at once).  Every call shares the array:
// calls that overlap on the GPU race.

constexpr u64 kStaticMaxSymbols = 1ull << 20;  // longest string expanded: 1 MiB
constexpr u64 kStaticLbTiles = 1024;           // look-back slots for one scan of kStaticMaxSymbols

struct StaticScratch {
    u32 cur[kStaticMaxSymbols];
    u32 next[kStaticMaxSymbols];
    u32 lens[kStaticMaxSymbols];
    u64 offs[kStaticMaxSymbols];
    u64 totals[2];
    unsigned char lb[kStaticLbTiles * 48];
};

static __device__ __align__(256) unsigned char g_static_scratch[sizeof(StaticScratch)];

StaticScratch* static_scratch_of_device(lcg_ctx* ctx) {
    static std::mutex mu;
    static StaticScratch* addr[256] = {nullptr};
    fail_if(ctx, ctx->device < 0 || ctx->device >= 256, LCG_EDEVICE, "device index out of range");
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[ctx->device]) {
        void* p = nullptr;
        ck(ctx, cudaGetSymbolAddress(&p, g_static_scratch), "cudaGetSymbolAddress");
        addr[ctx->device] = (StaticScratch*)p;
    }
    return addr[ctx->device];
}

void decompress_static(lcg_ctx* ctx, const lcg_grammar* G, u32 j, uint8_t* out, u64 cap, uint64_t* out_len) {
    static_assert(scan2_lb_bytes_static(kStaticLbTiles) <= kStaticLbTiles * 48, "look-back slots");
    fail_if(ctx, j >= G->k, LCG_EINVAL, "string index out of range");
    StaticScratch* sc = static_scratch_of_device(ctx);
    reset_status(ctx);
    u32 lev = 0, r = 0;
    fetch(ctx, {{&lev, G->c_level + j, 4}, {&r, G->c_rank + j, 4}});
    u32* cur = sc->cur;
    u32* nxt = sc->next;
    ck(ctx, cudaMemcpyAsync(cur, &r, 4, cudaMemcpyHostToDevice, ctx->st), "copy");
    u64 cnt = 1;
    for (u32 l = lev; l >= 1; l--) {
        const Level& L = G->lv[l - 1];
        ck(ctx, launch_rule_lens(cur, cnt, L.rhs_off, sc->lens, ctx->st), "rule lens");
        // the look-back slots left by an earlier call (any context) must not
        // look published
        ck(ctx, cudaMemsetAsync(sc->lb, 0, sizeof(sc->lb), ctx->st), "clear look-back");
        u64 grid = 0;
        ck(ctx, launch_scan2(sc->lens, nullptr, cnt, sc->offs, nullptr, sc->totals, sc->lb, ++ctx->epoch, ctx->ctr,
                             ctx->ctr_val, ctx->ds, ctx->st, &grid),
           "scan");
        ctx->ctr_val += grid;
        u64 total = 0;
        check_device_status(ctx, read_status(ctx, &total, sc->totals, 8));
        if (total > kStaticMaxSymbols) {
            *out_len = total;  // a lower bound of the string's length
            fail_if(ctx, true, LCG_EOVERFLOW,
                    "string longer than the static scratch allows (1048576 symbols); use lcg_decompress");
        }
        ck(ctx, launch_expand(cur, cnt, sc->offs, L.rhs_off, L.rhs, nxt, ctx->st), "expand");
        ctx->launches += 3;
        u32* t = cur;
        cur = nxt;
        nxt = t;
        cnt = total;
    }
    *out_len = cnt;
    fail_if(ctx, cap < cnt, LCG_EINVAL, "output buffer too small");
    ck(ctx, launch_to_bytes(cur, cnt, out, ctx->st), "to bytes");
    ctx->launches++;
    sync(ctx);
}

}  // namespace

// --------------------------------------------------------------------------
// post-processing: RL, then Simp (kernels in post.cu)
// --------------------------------------------------------------------------

struct lcg_pp {
    int device = 0;
    u64 rules = 0, size = 0;
    u32 k = 0;
    u8* kind = nullptr;      // rules
    u64* rhs_off = nullptr;  // rules + 1
    u32* rhs = nullptr;      // size
    u32* c = nullptr;        // k
    lcg_pp_stats stats{};
};

namespace {

void free_pp(lcg_pp* pp) {
    if (!pp) return;
    cudaSetDevice(pp->device);
    cudaFree(pp->kind);
    cudaFree(pp->rhs_off);
    cudaFree(pp->rhs);
    cudaFree(pp->c);
    delete pp;
}

// Exclusive scan of up to two u32 columns (the library's single-pass scan);
// their totals go to totals[0] and [1] (on the device), the first also to *end0.
void pp_scan(lcg_ctx* ctx, const u32* in0, const u32* in1, u64 n, u64* out0, u64* out1, u64* totals,
             u64* end0 = nullptr) {
    u64 grid = 0;
    const u64 stiles = std::max<u64>(1, scan2_tiles_for(n));
    ensure_lb(ctx, &ctx->lb2, &ctx->lb2_tiles, stiles, scan2_lb_bytes(stiles));
    ck(ctx, launch_scan2(in0, in1, n, out0, out1, totals, ctx->lb2, ++ctx->epoch, ctx->ctr, ctx->ctr_val,
                         ctx->ds, ctx->st, &grid, nullptr, end0),
       "scan");
    ctx->ctr_val += grid;
    ctx->launches++;
}

// The totals of the scans since the last wait.
std::vector<u64> pp_totals(lcg_ctx* ctx, const u64* d, u64 n) {
    std::vector<u64> t(n, 0);
    check_device_status(ctx, read_status(ctx, t.data(), d, n * 8));
    return t;
}

// Each step runs over all levels before the host waits for what it needs of them:
// five waits in all.  (Level by level it was three to five waits a level.)
lcg_pp* postprocess(lcg_ctx* ctx, const lcg_grammar* G) {
    const u32 nl = (u32)G->lv.size();
    fail_if(ctx, nl > (u32)kPPMaxLevels, LCG_EINVAL, "grammar with too many levels");
    if (G->owner && G->owner != ctx) ck(ctx, cudaStreamSynchronize(G->owner->st), "grammar's stream");
    sync(ctx);
    reset_status(ctx);
    Temps tmp(ctx);
    PPLevels lv{};
    lv.n = nl;
    std::vector<u32*> uses(nl);
    u64 rl_total = 0, size_before = 0, size_rl = 0;
    // RL: the lengths of the rewritten rules and the runs of every level
    u64* d_tot = tmp.get<u64>(2 * (u64)nl + 2);
    std::vector<u64*> new_off(nl), rl_off(nl);
    for (u32 i = 0; i < nl; i++) {
        const Level& L = G->lv[i];
        size_before += L.G;
        u32* out_len = tmp.get<u32>(L.g);
        u32* rl_len = tmp.get<u32>(L.g);
        new_off[i] = tmp.get<u64>(L.g + 1);
        rl_off[i] = tmp.get<u64>(L.g);
        ck(ctx, launch_rl_count(L.rhs_off, L.rhs, L.g, out_len, rl_len, ctx->st), "k_rl_count");
        pp_scan(ctx, out_len, rl_len, L.g, new_off[i], rl_off[i], d_tot + 2 * i, new_off[i] + L.g);
        ctx->launches++;
    }
    std::vector<u64> tot = pp_totals(ctx, d_tot, 2 * (u64)nl);
    std::vector<u64> Gn(nl);
    // the rules without runs, and the distinct runs of the levels that have any
    struct Runs {
        u64 R = 0;
        u32 *y = nullptr, *len = nullptr;
        u64 *pos = nullptr, *first = nullptr, *rank_of = nullptr;
        u32* rhs = nullptr;
    };
    std::vector<Runs> runs(nl);
    bool any = false;
    for (u32 i = 0; i < nl; i++) {
        const Level& L = G->lv[i];
        const u64 R = tot[2 * i + 1];
        Gn[i] = tot[2 * i];
        Runs& x = runs[i];
        x.R = R;
        x.rhs = tmp.get<u32>(Gn[i]);
        size_rl += Gn[i];
        u64 cap = 64;
        while (cap < 2 * R + 16) cap <<= 1;
        u64 *keys = nullptr, *vals = nullptr;
        if (R) {
            x.y = tmp.get<u32>(R);
            x.len = tmp.get<u32>(R);
            x.pos = tmp.get<u64>(R);
            x.first = tmp.get<u64>(R);
            x.rank_of = tmp.get<u64>(R);
            keys = tmp.get<u64>(cap);
            vals = tmp.get<u64>(cap);
            ck(ctx, cudaMemsetAsync(keys, 0xFF, cap * 8, ctx->st), "memset");
            ck(ctx, cudaMemsetAsync(vals, 0xFF, cap * 8, ctx->st), "memset");
        }
        ck(ctx, launch_rl_write(L.rhs_off, L.rhs, L.g, new_off[i], rl_off[i], x.rhs, x.y, x.len, x.pos, keys, vals,
                                cap - 1, ctx->ds, ctx->st),
           "k_rl_write");
        ctx->launches++;
        if (R) {
            any = true;
            u32* first = tmp.get<u32>(R);
            ck(ctx, launch_rl_first(x.y, x.len, R, keys, vals, cap - 1, first, x.first, ctx->ds, ctx->st), "k_rl_first");
            pp_scan(ctx, first, nullptr, R, x.rank_of, nullptr, d_tot + 2 * i);
            ctx->launches++;
        }
    }
    if (any) tot = pp_totals(ctx, d_tot, 2 * (u64)nl);
    for (u32 i = 0; i < nl; i++) {
        const Runs& x = runs[i];
        const u64 Rd = x.R ? tot[2 * i] : 0;
        const u64 g = G->lv[i].g;
        u32* rl_y = tmp.get<u32>(Rd);
        u32* rl_l = tmp.get<u32>(Rd);
        ck(ctx, launch_rl_fix(x.y, x.len, x.pos, x.first, x.rank_of, x.R, x.rhs, rl_y, rl_l, ctx->ds, ctx->st),
           "k_rl_fix");
        ctx->launches++;
        lv.off[i] = new_off[i];
        lv.rhs[i] = x.rhs;
        lv.g[i] = g;
        lv.nrl[i] = Rd;
        lv.rl_y[i] = rl_y;
        lv.rl_l[i] = rl_l;
        rl_total += Rd;
        size_rl += 2 * Rd;
        uses[i] = tmp.get<u32>(g);
        lv.pinned[i] = tmp.get<u8>(g);
        ck(ctx, cudaMemsetAsync(uses[i], 0, g * 4, ctx->st), "memset");
        ck(ctx, cudaMemsetAsync(lv.pinned[i], 0, g, ctx->st), "memset");
    }
    // Simp: uses, kept rules, surviving rules and their ids
    for (u32 i = 1; i < nl; i++) {
        ck(ctx, launch_pp_uses(lv.rhs[i], Gn[i], uses[i - 1], ctx->st), "k_pp_uses");
        ck(ctx, launch_pp_pin_bases(lv.rl_y[i], lv.nrl[i], lv.pinned[i - 1], ctx->st), "k_pp_pin_bases");
        ctx->launches += 2;
    }
    ck(ctx, launch_pp_pin_roots(G->c_level, G->c_rank, G->k, lv, ctx->st), "k_pp_pin_roots");
    u64 next = 256, removed = 0;
    for (u32 i = 0; i < nl; i++) {
        u32* surv = tmp.get<u32>(lv.g[i]);
        u64* spre = tmp.get<u64>(lv.g[i]);
        ck(ctx, launch_pp_survive(uses[i], lv.pinned[i], lv.g[i], surv, ctx->st), "k_pp_survive");
        pp_scan(ctx, surv, nullptr, lv.g[i], spre, nullptr, d_tot + 2 * i);
        lv.surv[i] = surv;
        lv.spre[i] = spre;
        lv.explen[i] = tmp.get<u32>(lv.g[i]);
        lv.dst[i] = tmp.get<u64>(lv.g[i]);
        ck(ctx, cudaMemsetAsync(lv.dst[i], 0xFF, lv.g[i] * 8, ctx->st), "memset");
        ctx->launches += 1;
    }
    tot = pp_totals(ctx, d_tot, 2 * (u64)nl);
    for (u32 i = 0; i < nl; i++) {
        lv.S[i] = tot[2 * i];
        lv.base[i] = next;
        next += lv.S[i] + lv.nrl[i];
        removed += lv.g[i] - lv.S[i];
    }
    const u64 rules = next - 256;
    fail_if(ctx, next > 0xffffffffull, LCG_EOVERFLOW, "post-processed grammar with 2^32 symbols or more");
    u32* fin_len = tmp.get<u32>(rules);
    for (u32 i = 0; i < nl; i++) {
        ck(ctx, launch_pp_lengths(lv, i, fin_len, ctx->ds, ctx->st), "k_pp_explen");
        ctx->launches += 2;
    }
    auto* pp = new lcg_pp;
    pp->device = ctx->device;
    pp->rules = rules;
    pp->k = G->k;
    try {
        pp->rhs_off = dalloc<u64>(ctx, rules + 1);
        pp_scan(ctx, fin_len, nullptr, rules, pp->rhs_off, nullptr, d_tot, pp->rhs_off + rules);
        pp->size = pp_totals(ctx, d_tot, 1)[0];
        pp->rhs = dalloc<u32>(ctx, pp->size);
        pp->kind = dalloc<u8>(ctx, rules);
        pp->c = dalloc<u32>(ctx, G->k);
        for (u32 i = nl; i-- > 0;) {  // top level first: removed rules learn their place from above
            ck(ctx, launch_pp_write(lv, i, pp->rhs_off, pp->rhs, pp->kind, ctx->ds, ctx->st), "k_pp_place");
            ctx->launches += 2;
        }
        ck(ctx, launch_pp_roots(G->c_level, G->c_rank, G->k, lv, pp->c, ctx->st), "k_pp_roots");
        ctx->launches++;
        check_device_status(ctx, read_status(ctx));
    } catch (...) {
        sync(ctx);
        free_pp(pp);
        throw;
    }
    pp->stats.size_before = size_before;
    pp->stats.size_rl = size_rl;
    pp->stats.size = pp->size;
    pp->stats.rl_rules = rl_total;
    pp->stats.removed = removed;
    pp->stats.rules = rules;
    pp->stats.strings = G->k;
    return pp;
}

}  // namespace

// --------------------------------------------------------------------------
// C entry points
// --------------------------------------------------------------------------

#define LCG_GUARD_BEGIN try {
#define LCG_GUARD_END                                  \
    }                                                  \
    catch (const Fail& f) {                            \
        return f.code;                                 \
    }                                                  \
    catch (const std::bad_alloc&) {                    \
        ctx->err = "host allocation failed";           \
        return LCG_ENOMEM;                             \
    }

extern "C" {

int lcg_ctx_create(int device, const lcg_hash_family* H, void* stream, lcg_ctx** out) {
    if (!out) return LCG_EINVAL;
    *out = nullptr;
    if (!H || H->levels < 2 || H->levels > 4096 || H->m_bits < 1 || H->m_bits > 32 || !H->a || !H->b || !H->c)
        return LCG_EINVAL;
    for (u32 i = 0; i < H->levels; i++)
        if (H->a[i] == 0 || H->a[i] >= kP61 || H->b[i] >= kP61 || H->c[i] == 0 || H->c[i] >= kP61)
            return LCG_EINVAL;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return LCG_EDEVICE;
    lcg_ctx* ctx = new (std::nothrow) lcg_ctx();
    if (!ctx) return LCG_ENOMEM;
    ctx->device = device;
    ctx->a.assign(H->a, H->a + H->levels);
    ctx->b.assign(H->b, H->b + H->levels);
    ctx->c.assign(H->c, H->c + H->levels);
    ctx->levels = H->levels;
    ctx->m_bits = H->m_bits;
    ctx->mmask = (H->m_bits == 32) ? 0xffffffffull : ((1ull << H->m_bits) - 1);
    u64 tag = 1469598103934665603ull;
    for (u32 i = 0; i < H->levels; i++) {
        for (u64 w : {H->a[i], H->b[i], H->c[i]}) tag = (tag ^ w) * 1099511628211ull;
    }
    ctx->tag = (tag ^ ctx->mmask) * 1099511628211ull;
    try {
        ck(ctx, cudaSetDevice(device), "cudaSetDevice");
        ck(ctx, cudaDeviceGetAttribute(&ctx->sms, cudaDevAttrMultiProcessorCount, device), "device attribute");
        if (ctx->sms < 1) ctx->sms = 1;
        if (stream) {
            ctx->st = (cudaStream_t)stream;
        } else {
            ck(ctx, cudaStreamCreateWithFlags(&ctx->st, cudaStreamNonBlocking), "stream");
            ctx->own_stream = true;
        }
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, device) == cudaSuccess) {
            u64 thr = ~0ull;
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
        }
        ck(ctx, cudaHostAlloc((void**)&ctx->mail, kMailBytes, cudaHostAllocDefault), "cudaHostAlloc");
        ck(ctx, cudaMalloc(&ctx->ds, sizeof(DevStatus)), "cudaMalloc");
        ck(ctx, cudaMalloc(&ctx->ctr, sizeof(u64)), "cudaMalloc");
        ck(ctx, cudaMalloc(&ctx->scratch, 8 * sizeof(u64)), "cudaMalloc");
        ck(ctx, cudaMalloc(&ctx->ds_arr, kMaxRounds * sizeof(DevStatus)), "cudaMalloc");
        ck(ctx, cudaMalloc(&ctx->rc_arr, kMaxRounds * sizeof(RoundCounts)), "cudaMalloc");
        ck(ctx, cudaMalloc(&ctx->tot_arr, 3 * kMaxRounds * sizeof(u64)), "cudaMalloc");
        ck(ctx, cudaMemset(ctx->ds, 0, sizeof(DevStatus)), "memset");
        ck(ctx, cudaMemset(ctx->ctr, 0, sizeof(u64)), "memset");
        ck(ctx, cudaMemset(ctx->scratch, 0, 8 * sizeof(u64)), "memset");
        ck(ctx, cudaDeviceSynchronize(), "sync");
    } catch (const Fail& f) {
        lcg_ctx_destroy(ctx);
        return f.code;
    }
    *out = ctx;
    return LCG_OK;
}

void lcg_ctx_destroy(lcg_ctx* ctx) {
    if (!ctx) return;
    cudaSetDevice(ctx->device);
    if (ctx->st) cudaStreamSynchronize(ctx->st);
    for (lcg_grammar* G : ctx->live) G->owner = nullptr;  // they outlive the context
    ctx->live.clear();
    destroy_graph(ctx);
    if (ctx->upload) cudaFree(ctx->upload);
    if (ctx->mail) cudaFreeHost(ctx->mail);
    for (auto& r : ctx->krecs) {
        if (r.graph || r.part) continue;  // destroyed with the graph
        cudaEventDestroy(r.a);
        cudaEventDestroy(r.b);
    }
    for (auto e : ctx->evpool) cudaEventDestroy(e);
    if (ctx->lb1) cudaFree(ctx->lb1);
    if (ctx->heads) cudaFree(ctx->heads);
    if (ctx->lb2) cudaFree(ctx->lb2);
    cudaFree(ctx->ds);
    cudaFree(ctx->ctr);
    cudaFree(ctx->scratch);
    cudaFree(ctx->ds_arr);
    cudaFree(ctx->rc_arr);
    cudaFree(ctx->tot_arr);
    if (ctx->own_stream && ctx->st) cudaStreamDestroy(ctx->st);
    delete ctx;
}

const char* lcg_last_error(const lcg_ctx* ctx) { return ctx ? ctx->err.c_str() : "no context"; }

int lcg_last_build_stats(const lcg_ctx* ctx, lcg_build_stats* out) {
    if (!ctx || !out) return LCG_EINVAL;
    *out = ctx->stats;
    return LCG_OK;
}

int lcg_set_kernel_timing(lcg_ctx* ctx, int enable) {
    if (!ctx || enable < 0 || enable > 2) return LCG_EINVAL;
    ctx->ktime = enable;
    return LCG_OK;
}

int lcg_set_graph(lcg_ctx* ctx, int enable) {
    if (!ctx || enable < 0 || enable > 1) return LCG_EINVAL;
    ctx->use_graph = enable != 0;
    if (!ctx->use_graph) destroy_graph(ctx);
    return LCG_OK;
}

int lcg_set_tuning(lcg_ctx* ctx, const lcg_tuning* t) {
    if (!ctx || !t) return LCG_EINVAL;
    if (cudaSetDevice(ctx->device) != cudaSuccess) return LCG_EDEVICE;  // whose blocks per SM are asked for
    const int maxb = std::max(parse_max_blocks(1), parse_max_blocks(4));
    if (!(t->table_load >= 0.3 && t->table_load <= 0.78) || t->parse_blocks_per_sm > (uint32_t)maxb ||
        t->miss_flush < 32 || t->miss_flush > 256 || (t->table_slots_max != 0 && t->table_slots_max < 1024) ||
        t->tile_stripes < 1 || t->tile_stripes > 16 || !parse_tile_valid(t->parse_tile) ||
        t->parse_tile_min > 1024) {
        ctx->err = "tuning out of range: table_load in [0.3, 0.78], parse_blocks_per_sm <= " + std::to_string(maxb) +
                   ", miss_flush in [32, 256], table_slots_max 0 or >= 1024, tile_stripes in [1, 16], "
                   "parse_tile 1024, 2048 or 4096, parse_tile_min <= 1024";
        return LCG_EINVAL;
    }
    ctx->tuning = *t;
    return LCG_OK;
}

int lcg_get_tuning(const lcg_ctx* ctx, lcg_tuning* t) {
    if (!ctx || !t) return LCG_EINVAL;
    *t = ctx->tuning;
    return LCG_OK;
}

int lcg_last_kernel_times(const lcg_ctx* ctx, lcg_kernel_time* out, uint32_t cap, uint32_t* count) {
    if (!ctx || !count) return LCG_EINVAL;
    *count = (uint32_t)ctx->ktimes.size();
    for (uint32_t x = 0; x < cap && x < ctx->ktimes.size(); x++) out[x] = ctx->ktimes[x];
    return LCG_OK;
}

int lcg_last_kernel_launches(const lcg_ctx* ctx, lcg_kernel_launch* out, uint32_t cap, uint32_t* count) {
    if (!ctx || !count) return LCG_EINVAL;
    *count = (uint32_t)ctx->klaunches.size();
    for (uint32_t x = 0; x < cap && x < ctx->klaunches.size(); x++) out[x] = ctx->klaunches[x];
    return LCG_OK;
}

int lcg_build(lcg_ctx* ctx, const uint8_t* data, const uint64_t* offsets, uint32_t k, int data_on_device,
              lcg_grammar** out) {
    if (!ctx || !out) return LCG_EINVAL;
    const Range range("lcg_build");
    *out = nullptr;
    lcg_grammar* G = nullptr;
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    kt_reset(ctx);
    reset_status(ctx);
    std::vector<uint64_t> shifted;  // offsets into the context's upload buffer
    if (ctx->use_graph && k > 0 && offsets && data && ctx->hint_rounds > 0) {
        std::vector<u64> lens(k);
        bool ok = true;
        for (u32 j = 0; j < k && ok; j++) {
            lens[j] = offsets[j + 1] - offsets[j];
            ok = offsets[j + 1] > offsets[j] && lens[j] >= 2;  // strings of length one: not in graphs
        }
        if (ok && !data_on_device) {
            // host input: into the context's upload buffer, whose address a
            // captured graph can keep; the build then reads it there
            const u64 nbytes = offsets[k] - offsets[0];
            if (ctx->upload_cap < nbytes) {
                if (ctx->upload) {
                    if (ctx->graph) destroy_graph(ctx);
                    dfree(ctx, ctx->upload);
                    ctx->upload = nullptr;
                    ctx->upload_cap = 0;
                }
                const u64 cap = nbytes + nbytes / 8 + 4096;
                ctx->upload = dalloc<unsigned char>(ctx, cap);
                ctx->upload_cap = cap;
            }
            ck(ctx, cudaMemcpyAsync(ctx->upload, data + offsets[0], nbytes, cudaMemcpyHostToDevice, ctx->st),
               "copy input");
            shifted.resize(k + 1);
            for (u32 j = 0; j <= k; j++) shifted[j] = offsets[j] - offsets[0];
            data = ctx->upload;
            offsets = shifted.data();
            data_on_device = 1;
        }
        if (ok) {
            try {
                G = build_with_graph(ctx, data + offsets[0], lens);
            } catch (const Retry& r) {
                if (!r.levels) ctx->plan_slack = std::min(4.0, ctx->plan_slack * 1.6);
                G = nullptr;
                kt_reset(ctx);
                G = new_grammar(ctx);
                build_into(ctx, G, data, offsets, k, data_on_device, false, false);
                ctx->stats.redone = 1;
                ctx->stats.plan_slack = ctx->plan_slack;
                sync(ctx);
                kt_collect(ctx);
                *out = G;
                return LCG_OK;
            }
            if (G) {
                ctx->plan_slack = std::max(1.0, ctx->plan_slack * 0.97);
                ctx->stats.plan_slack = ctx->plan_slack;
                kt_collect(ctx);
                *out = G;
                return LCG_OK;
            }
        }
    }
    G = new_grammar(ctx);
    try {
        build_into(ctx, G, data, offsets, k, data_on_device, false, true);
        if (ctx->stats.async_rounds > 0) ctx->plan_slack = std::max(1.0, ctx->plan_slack * 0.97);
    } catch (const Retry& r) {
        if (!r.levels) ctx->plan_slack = std::min(4.0, ctx->plan_slack * 1.6);
        // the rounds planned from the previous build did not fit: round by round
        sync(ctx);
        free_grammar_now(G);
        G = nullptr;
        kt_reset(ctx);
        G = new_grammar(ctx);
        build_into(ctx, G, data, offsets, k, data_on_device, false, false);
        ctx->stats.redone = 1;
    }
    ctx->stats.plan_slack = ctx->plan_slack;
    sync(ctx);
    kt_collect(ctx);
    *out = G;
    return LCG_OK;
    }
    catch (const Fail& f) {
        cudaStreamSynchronize(ctx->st);
        free_grammar_now(G);
        return f.code;
    }
    catch (const std::bad_alloc&) {
        ctx->err = "host allocation failed";
        cudaStreamSynchronize(ctx->st);
        free_grammar_now(G);
        return LCG_ENOMEM;
    }
}

int lcg_build_into(lcg_ctx* ctx, lcg_grammar* resident, const uint8_t* data, const uint64_t* offsets, uint32_t k,
                   int data_on_device) {
    if (!ctx || !resident) return LCG_EINVAL;
    const Range range("lcg_build_into");
    if (resident->tag != ctx->tag) {
        ctx->err = "resident grammar of another hash family";
        return LCG_EMISMATCH;
    }
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    kt_reset(ctx);
    reset_status(ctx);
    // what the grammar goes back to when the build fails: the rounds that were done have
    // appended rules, whose places are then free again
    const u32 k0 = resident->k;
    std::vector<std::pair<u64, u64>> sizes;
    for (const Level& L : resident->lv) sizes.emplace_back(L.g, L.G);
    try {
        build_into(ctx, resident, data, offsets, k, data_on_device, true, false);
    } catch (...) {
        resident->k = k0;
        while (resident->lv.size() > sizes.size()) pop_level(ctx, resident);
        for (size_t i = 0; i < sizes.size(); i++) {
            Level& L = resident->lv[i];
            L.g = sizes[i].first;
            L.G = sizes[i].second;
            L.rvalid = false;  // (the table may hold rules past them)
        }
        throw;
    }
    sync(ctx);
    kt_collect(ctx);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_merge(lcg_ctx* ctx, lcg_grammar* a, const lcg_grammar* b) {
    if (!ctx || !a || !b) return LCG_EINVAL;
    const Range range("lcg_merge");
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    kt_reset(ctx);
    reset_status(ctx);
    merge(ctx, a, b);
    kt_collect(ctx);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_decompress(lcg_ctx* ctx, const lcg_grammar* G, uint32_t j, uint8_t* out, uint64_t cap, uint64_t* out_len,
                   int out_on_device) {
    if (!ctx || !G || !out_len) return LCG_EINVAL;
    const Range range("lcg_decompress");
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    decompress(ctx, G, j, out, cap, out_len, out_on_device);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_decompress_static(lcg_ctx* ctx, const lcg_grammar* G, uint32_t j, uint8_t* out_dev, uint64_t cap,
                          uint64_t* out_len) {
    if (!ctx || !G || !out_dev || !out_len) return LCG_EINVAL;
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    decompress_static(ctx, G, j, out_dev, cap, out_len);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_selftest_blocks(lcg_ctx* ctx, uint32_t most) {
    if (!ctx) return LCG_EINVAL;
    ctx->blocks_max = most;
    destroy_graph(ctx);  // (captured with another number)
    return LCG_OK;
}

int lcg_selftest_alloc_failure(lcg_ctx* ctx, uint64_t nth) {
    if (!ctx) return LCG_EINVAL;
    ctx->fail_alloc = nth;
    return LCG_OK;
}

int lcg_selftest_wait_timeout(lcg_ctx* ctx) {
    if (!ctx) return LCG_EINVAL;
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    kt_reset(ctx);
    reset_status(ctx);
    // A scan of two tiles whose tile counter is read one ahead: the first block
    // takes tile 1 and waits for a tile 0 that no block takes.  Every block
    // stays in bounds (tiles 1 and 2 of the three look-back slots sized below; tile
    // 2 returns at once), and the wait ends with kErrTimeout.
    const u64 n = 16384;  // two tiles of the scan
    const u64 tiles = scan2_tiles_for(n);
    ensure_lb(ctx, &ctx->lb2, &ctx->lb2_tiles, tiles + 1, scan2_lb_bytes(tiles + 1));
    u32* in = dalloc<u32>(ctx, n);
    u64* out = dalloc<u64>(ctx, n);
    ck(ctx, cudaMemsetAsync(in, 0, n * sizeof(u32), ctx->st), "memset");
    ck(ctx, cudaMemsetAsync(ctx->ds, 0, sizeof(DevStatus), ctx->st), "reset status");
    u64 grid = 0;
    ck(ctx, launch_scan2(in, nullptr, n, out, nullptr, ctx->scratch + 1, ctx->lb2, ++ctx->epoch, ctx->ctr,
                         ctx->ctr_val - 1, ctx->ds, ctx->st, &grid, nullptr),
       "scan");
    ctx->ctr_val += grid;
    dfree(ctx, in);
    dfree(ctx, out);
    const DevStatus st = read_status(ctx);
    check_device_status(ctx, st);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_grammar_shape(const lcg_grammar* G, uint32_t* k, uint32_t* nlevels) {
    if (!G) return LCG_EINVAL;
    if (k) *k = G->k;
    if (nlevels) *nlevels = (uint32_t)G->lv.size();
    return LCG_OK;
}

int lcg_level_size(const lcg_grammar* G, uint32_t level, uint64_t* g, uint64_t* Gsz) {
    if (!G || level < 1 || level > G->lv.size()) return LCG_EINVAL;
    if (g) *g = G->lv[level - 1].g;
    if (Gsz) *Gsz = G->lv[level - 1].G;
    return LCG_OK;
}

int lcg_export_level(lcg_ctx* ctx, const lcg_grammar* G, uint32_t level, uint64_t* rhs_off, uint32_t* rhs,
                     uint32_t* F) {
    if (!ctx || !G || level < 1 || level > G->lv.size()) return LCG_EINVAL;
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    const Level& L = G->lv[level - 1];
    if (rhs_off)
        ck(ctx, cudaMemcpyAsync(rhs_off, L.rhs_off, (L.g + 1) * 8, cudaMemcpyDeviceToHost, ctx->st), "export");
    if (rhs && L.G) ck(ctx, cudaMemcpyAsync(rhs, L.rhs, L.G * 4, cudaMemcpyDeviceToHost, ctx->st), "export");
    if (F && L.g) ck(ctx, cudaMemcpyAsync(F, L.F, L.g * 4, cudaMemcpyDeviceToHost, ctx->st), "export");
    sync(ctx);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_export_start(lcg_ctx* ctx, const lcg_grammar* G, uint32_t* F0, uint32_t* c_level, uint32_t* c_rank) {
    if (!ctx || !G) return LCG_EINVAL;
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    if (F0) ck(ctx, cudaMemcpyAsync(F0, G->F0, 256 * 4, cudaMemcpyDeviceToHost, ctx->st), "export");
    if (c_level && G->k)
        ck(ctx, cudaMemcpyAsync(c_level, G->c_level, G->k * 4, cudaMemcpyDeviceToHost, ctx->st), "export");
    if (c_rank && G->k)
        ck(ctx, cudaMemcpyAsync(c_rank, G->c_rank, G->k * 4, cudaMemcpyDeviceToHost, ctx->st), "export");
    sync(ctx);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_import(lcg_ctx* ctx, uint32_t k, uint32_t nlevels, const uint64_t* g, const uint64_t* const* rhs_off,
               const uint32_t* const* rhs, const uint32_t* const* F, const uint32_t* c_level, const uint32_t* c_rank,
               lcg_grammar** out) {
    if (!ctx || !out) return LCG_EINVAL;
    *out = nullptr;
    if (nlevels && (!g || !rhs_off || !rhs || !F)) return LCG_EINVAL;
    if (k && (!c_level || !c_rank)) return LCG_EINVAL;
    lcg_grammar* G = nullptr;
    try {
        ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
        kt_reset(ctx);
        fail_if(ctx, nlevels >= ctx->levels, LCG_ELEVELS, "grammar has more levels than the hash family has functions");
        // host checks: offsets, symbol ranges and C entries name existing rules
        for (u32 i = 1; i <= nlevels; i++) {
            const u64 gi = g[i - 1];
            fail_if(ctx, gi > kMaxRank, LCG_EOVERFLOW, "level with 2^31 rules or more");
            fail_if(ctx, rhs_off[i - 1] == nullptr || (gi && (rhs[i - 1] == nullptr || F[i - 1] == nullptr)),
                    LCG_EINVAL, "missing array of level " + std::to_string(i));
            const uint64_t* ro = rhs_off[i - 1];
            fail_if(ctx, ro[0] != 0, LCG_EINVAL, "rhs_off of level " + std::to_string(i) + " does not start at 0");
            for (u64 r = 0; r < gi; r++)
                fail_if(ctx, ro[r + 1] <= ro[r], LCG_EINVAL,
                        "rule " + std::to_string(r) + " of level " + std::to_string(i) + " is empty or misplaced");
            const u64 prev = (i == 1) ? 256 : g[i - 2];
            const uint32_t* x = rhs[i - 1];
            for (u64 y = 0; y < ro[gi]; y++)
                fail_if(ctx, x[y] >= prev, LCG_EINVAL,
                        "level " + std::to_string(i) + " names a symbol outside level " + std::to_string(i - 1));
        }
        for (u32 j = 0; j < k; j++) {
            const u32 lvl = c_level[j];
            fail_if(ctx, lvl > nlevels, LCG_EINVAL, "C entry " + std::to_string(j) + " names a missing level");
            const u64 lim = (lvl == 0) ? 256 : g[lvl - 1];
            fail_if(ctx, c_rank[j] >= lim, LCG_EINVAL, "C entry " + std::to_string(j) + " names a missing rule");
        }
        reset_status(ctx);
        G = new_grammar(ctx);
        if (k) {
            grow_c(ctx, G, k);
            ck(ctx, cudaMemcpyAsync(G->c_level, c_level, (u64)k * 4, cudaMemcpyHostToDevice, ctx->st), "import");
            ck(ctx, cudaMemcpyAsync(G->c_rank, c_rank, (u64)k * 4, cudaMemcpyHostToDevice, ctx->st), "import");
            G->k = k;
        }
        for (u32 i = 1; i <= nlevels; i++) {
            const u64 gi = g[i - 1], Gi = rhs_off[i - 1][gi];
            G->lv.emplace_back();
            Level& L = G->lv.back();
            grow_level(ctx, L, gi, Gi);
            ck(ctx, cudaMemcpyAsync(L.rhs_off, rhs_off[i - 1], (gi + 1) * 8, cudaMemcpyHostToDevice, ctx->st), "import");
            if (Gi) ck(ctx, cudaMemcpyAsync(L.rhs, rhs[i - 1], Gi * 4, cudaMemcpyHostToDevice, ctx->st), "import");
            if (gi) ck(ctx, cudaMemcpyAsync(L.F, F[i - 1], gi * 4, cudaMemcpyHostToDevice, ctx->st), "import");
            L.g = gi;
            L.G = Gi;
            L.rvalid = false;
        }
        std::vector<void*> temps;
        check_fingerprints(ctx, G, temps);
        for (void* p : temps) dfree(ctx, p);
        const DevStatus st = read_status(ctx);
        fail_if(ctx, st.error == kErrMismatch, LCG_EMISMATCH,
                "imported fingerprints differ from those of this context's hash family");
        check_device_status(ctx, st);
        *out = G;
        return LCG_OK;
    } catch (const Fail& f) {
        cudaStreamSynchronize(ctx->st);
        free_grammar_now(G);
        return f.code;
    } catch (const std::bad_alloc&) {
        ctx->err = "host allocation failed";
        cudaStreamSynchronize(ctx->st);
        free_grammar_now(G);
        return LCG_ENOMEM;
    }
}

int lcg_string_roots(lcg_ctx* ctx, const lcg_grammar* G, uint32_t j0, uint32_t count, uint32_t* level,
                     uint32_t* rank, uint32_t* fp) {
    if (!ctx || !G || (count && (!level || !rank || !fp))) return LCG_EINVAL;
    if ((u64)j0 + count > G->k) {
        ctx->err = "string index out of range";
        return LCG_EINVAL;
    }
    if (count == 0) return LCG_OK;
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    fail_if(ctx, G->lv.size() > 64, LCG_ELEVELS, "grammar with more than 64 levels");
    FTable ft{};
    ft.F[0] = G->F0;
    for (u32 i = 1; i <= G->lv.size(); i++) ft.F[i] = G->lv[i - 1].F;
    ft.n = (u32)G->lv.size() + 1;
    u32* d = dalloc<u32>(ctx, 3ull * count);
    ck(ctx, launch_roots(G->c_level, G->c_rank, j0, count, ft, d, ctx->st), "k_roots");
    std::vector<u32> h(3ull * count);
    fetch(ctx, {{h.data(), d, h.size() * 4}});
    dfree(ctx, d);
    for (u32 x = 0; x < count; x++) {
        level[x] = h[3 * x];
        rank[x] = h[3 * x + 1];
        fp[x] = h[3 * x + 2];
    }
    return LCG_OK;
    LCG_GUARD_END
}

// ---- packed form: one buffer, every section 8-byte aligned ----------------

constexpr u64 kPackMagic = 0x4C434753ull;  // "LCGS"

static u64 pad8(u64 b) { return (b + 7) & ~7ull; }

static u64 packed_bytes(const lcg_grammar* G) {
    const u64 nl = G->lv.size();
    u64 b = 8 * (3 + 2 * nl);
    for (const Level& L : G->lv) b += 8 * (L.g + 1) + pad8(4 * L.G) + pad8(4 * L.g);
    return b + 2 * pad8(4ull * G->k) + 4 * 256;
}

int lcg_packed_size(const lcg_grammar* G, uint64_t* bytes) {
    if (!G || !bytes) return LCG_EINVAL;
    *bytes = packed_bytes(G);
    return LCG_OK;
}

constexpr u64 kPackGather = 65536;

int lcg_export_packed(lcg_ctx* ctx, const lcg_grammar* G, void* out, uint64_t cap) {
    if (!ctx || !G || !out) return LCG_EINVAL;
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    fail_if(ctx, ((uintptr_t)out & 7) != 0, LCG_EINVAL, "packed buffer must be 8-byte aligned");
    fail_if(ctx, cap < packed_bytes(G), LCG_EINVAL, "packed buffer too small");
    unsigned char* o = (unsigned char*)out;
    u64* head = (u64*)o;
    const u64 nl = G->lv.size();
    head[0] = kPackMagic;
    head[1] = G->k;
    head[2] = nl;
    for (u64 i = 0; i < nl; i++) {
        head[3 + 2 * i] = G->lv[i].g;
        head[4 + 2 * i] = G->lv[i].G;
    }
    // Columns in the order of the form.  Neighbours of at most kPackGather bytes (the
    // upper levels) are put next to each other on the device by one launch and copied
    // together: a copy of its own takes 3 us however short it is (a string of 20 kB has
    // 34 columns of 60 kB in all: its build, roots and export 347 us so, 326 us now).
    struct Col {
        const void* src;
        u64 bytes, span, pos;
    };
    std::vector<Col> cols;
    u64 pos = 8 * (3 + 2 * nl);
    auto add = [&](const void* src, u64 bytes) {
        cols.push_back(Col{src, bytes, pad8(bytes), pos});
        pos += pad8(bytes);
    };
    for (const Level& L : G->lv) {
        add(L.rhs_off, 8 * (L.g + 1));
        add(L.rhs, 4 * L.G);
        add(L.F, 4 * L.g);
    }
    add(G->c_level, 4ull * G->k);
    add(G->c_rank, 4ull * G->k);
    add(G->F0, 4 * 256);
    auto copy = [&](const Col& x) {
        if (x.bytes) ck(ctx, cudaMemcpyAsync(o + x.pos, x.src, x.bytes, cudaMemcpyDeviceToHost, ctx->st), "export");
        if (x.span > x.bytes) std::memset(o + x.pos + x.bytes, 0, x.span - x.bytes);
    };
    for (size_t c = 0; c < cols.size();) {
        size_t e = c;
        while (e < cols.size() && cols[e].bytes <= kPackGather) e++;
        if (e < c + 2) {
            copy(cols[c++]);
            continue;
        }
        const u64 from = cols[c].pos, bytes = cols[e - 1].pos + cols[e - 1].span - from;
        void* stage = nullptr;
        if (alloc_async(ctx, &stage, bytes) != cudaSuccess) {  // (the form needs no device memory)
            cudaGetLastError();
            for (; c < e; c++) copy(cols[c]);
            continue;
        }
        std::vector<void*> temps{stage};
        try {
            Copies gather;
            for (; c < e; c++) gather.add((u8*)stage + (cols[c].pos - from), cols[c].src, cols[c].bytes / 4, true);
            gather.run(ctx, temps);
            ck(ctx, cudaMemcpyAsync(o + from, stage, bytes, cudaMemcpyDeviceToHost, ctx->st), "export");
        } catch (...) {
            for (void* p : temps) dfree(ctx, p);
            throw;
        }
        for (void* p : temps) dfree(ctx, p);
    }
    sync(ctx);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_import_packed(lcg_ctx* ctx, const void* buf, uint64_t size, lcg_grammar** out) {
    if (!ctx || !buf || !out) return LCG_EINVAL;
    *out = nullptr;
    auto bad = [&](const char* why) {
        ctx->err = std::string("packed grammar: ") + why;
        return LCG_EINVAL;
    };
    if (((uintptr_t)buf & 7) != 0) return bad("buffer must be 8-byte aligned");
    const unsigned char* b = (const unsigned char*)buf;
    const u64* head = (const u64*)b;
    if (size < 24 || head[0] != kPackMagic) return bad("not a packed grammar");
    const u64 k = head[1], nl = head[2];
    if (k > 0xffffffffull || nl > 4096 || size < 8 * (3 + 2 * nl)) return bad("malformed header");
    std::vector<uint64_t> g(nl), Gs(nl);
    std::vector<const uint64_t*> ro(nl);
    std::vector<const uint32_t*> rhs(nl), F(nl);
    u64 pos = 8 * (3 + 2 * nl);
    for (u64 i = 0; i < nl; i++) {
        g[i] = head[3 + 2 * i];
        Gs[i] = head[4 + 2 * i];
        if (g[i] > kMaxRank || Gs[i] > (1ull << 40)) return bad("malformed level sizes");
        const u64 need = 8 * (g[i] + 1) + pad8(4 * Gs[i]) + pad8(4 * g[i]);
        if (pos + need > size) return bad("truncated");
        ro[i] = (const uint64_t*)(b + pos);
        rhs[i] = (const uint32_t*)(b + pos + 8 * (g[i] + 1));
        F[i] = (const uint32_t*)(b + pos + 8 * (g[i] + 1) + pad8(4 * Gs[i]));
        if (ro[i][g[i]] != Gs[i]) return bad("level sizes disagree with the offsets");
        pos += need;
    }
    if (pos + 2 * pad8(4 * k) + 4 * 256 != size) return bad("wrong size");
    const uint32_t* cl = (const uint32_t*)(b + pos);
    const uint32_t* cr = (const uint32_t*)(b + pos + pad8(4 * k));
    const uint32_t* F0 = (const uint32_t*)(b + pos + 2 * pad8(4 * k));
    lcg_grammar* G = nullptr;
    const int rc = lcg_import(ctx, (uint32_t)k, (uint32_t)nl, g.data(), ro.data(), rhs.data(), F.data(), cl, cr, &G);
    if (rc != LCG_OK) return rc;
    // F^0 must be the context's too
    uint32_t mine[256];
    if (cudaMemcpyAsync(mine, G->F0, sizeof(mine), cudaMemcpyDeviceToHost, ctx->st) != cudaSuccess ||
        cudaStreamSynchronize(ctx->st) != cudaSuccess) {
        free_grammar_now(G);
        ctx->err = "read F0";
        return LCG_EDEVICE;
    }
    if (std::memcmp(mine, F0, sizeof(mine)) != 0) {
        free_grammar_now(G);
        ctx->err = "packed grammar: F0 of another hash family";
        return LCG_EMISMATCH;
    }
    *out = G;
    return LCG_OK;
}

// ---- VByte form (Sec. 4, resource usage) ---------------------------------

constexpr u64 kVbMagic = 0x4C434756ull;  // "LCGV"

static int sm_count(lcg_ctx* ctx) {
    int sms = 0;
    ck(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device), "device attribute");
    return sms > 0 ? sms : 1;
}

// Exclusive scan of `cnt` (u32) into `off` (u64); the sum goes to totals[0].
static void vb_scan(lcg_ctx* ctx, const u32* cnt, u64 tiles, u64* off, u64* totals) {
    if (tiles == 0) return;
    u64 grid = 0;
    const u64 stiles = std::max<u64>(1, scan2_tiles_for(tiles));
    ensure_lb(ctx, &ctx->lb2, &ctx->lb2_tiles, stiles, scan2_lb_bytes(stiles));
    const int h = kt_begin(ctx, "k_scan2", 12.0 * (double)tiles);
    ck(ctx, launch_scan2(cnt, nullptr, tiles, off, nullptr, totals, ctx->lb2, ++ctx->epoch, ctx->ctr, ctx->ctr_val,
                         ctx->ds, ctx->st, &grid),
       "scan");
    kt_end(ctx, h);
    ctx->ctr_val += grid;
    ctx->launches++;
}

// Encode step 1: stream bytes per tile of one column (the u32 array `vals`,
// or the rule lengths of `offs`), scanned into tile offsets; the column's
// stream length goes to totals[0] (device).
static void vb_count_col(lcg_ctx* ctx, const u32* vals, const u64* offs, u64 n, u32* tile_bytes, u64* tile_off,
                         u64* totals) {
    const u64 tiles = vb_encode_tiles(n);
    if (tiles == 0) return;
    const int h = kt_begin(ctx, "k_vb_tile_bytes", (offs ? 8.0 : 4.0) * (double)n);
    ck(ctx, launch_vb_tile_bytes(vals, offs, n, tile_bytes, ctx->st), "k_vb_tile_bytes");
    kt_end(ctx, h);
    ctx->launches++;
    vb_scan(ctx, tile_bytes, tiles, tile_off, totals);
}

// Encode step 2: the column's stream at dst (nb bytes in all).
static void vb_write_col(lcg_ctx* ctx, const u32* vals, const u64* offs, u64 n, const u64* tile_off, u8* dst, bool pad,
                         u64 nb) {
    if (n == 0) return;
    const int h = kt_begin(ctx, "k_vb_write", (offs ? 8.0 : 4.0) * (double)n + (double)nb);
    ck(ctx, launch_vb_write(vals, offs, n, tile_off, dst, pad, ctx->st), "k_vb_write");
    kt_end(ctx, h);
    ctx->launches++;
}

// Scratch of the decode of one column: tile counts and offsets.
struct VbTemps {
    u32* cnt = nullptr;
    u64* off = nullptr;
};

// Decode nb bytes into exactly n values in [lo, hi) at vals.
static void vb_decode_col(lcg_ctx* ctx, const u8* src, u64 nb, u64 n, u64 lo, u64 hi, u32* vals, const VbTemps& t,
                          u64* totals) {
    const u64 tiles = vb_decode_tiles(nb);
    if (tiles == 0) return;
    int h = kt_begin(ctx, "k_vb_tile_ends", (double)nb);
    ck(ctx, launch_vb_tile_ends(src, nb, t.cnt, ctx->st), "k_vb_tile_ends");
    kt_end(ctx, h);
    ctx->launches++;
    vb_scan(ctx, t.cnt, tiles, t.off, totals);
    h = kt_begin(ctx, "k_vb_dwrite", (double)nb + 4.0 * (double)n);
    ck(ctx, launch_vb_dwrite(src, nb, n, lo, hi, t.off, vals, ctx->ds, ctx->st), "k_vb_dwrite");
    kt_end(ctx, h);
    ctx->launches++;
}

// Bytes of each level's two VByte streams: [2 i] rule lengths, [2 i + 1]
// right-hand sides of level i + 1.
static std::vector<u64> vb_section_bytes(lcg_ctx* ctx, const lcg_grammar* G) {
    const u64 nl = G->lv.size();
    std::vector<u64> nb(2 * nl, 0);
    if (nl == 0) return nb;
    u64* d = dalloc<u64>(ctx, 2 * nl);
    ck(ctx, cudaMemsetAsync(d, 0, 16 * nl, ctx->st), "memset");
    const int sms = sm_count(ctx);
    for (u64 i = 0; i < nl; i++) {
        const Level& L = G->lv[i];
        ck(ctx, launch_vb_count(nullptr, L.rhs_off, L.g, d + 2 * i, sms, ctx->st), "k_vb_count");
        ck(ctx, launch_vb_count(L.rhs, nullptr, L.G, d + 2 * i + 1, sms, ctx->st), "k_vb_count");
        ctx->launches += (L.g != 0) + (L.G != 0);
    }
    fetch(ctx, {{nb.data(), d, 16 * nl}});
    dfree(ctx, d);
    return nb;
}

static u64 vb_total_bytes(const lcg_grammar* G, const std::vector<u64>& nb) {
    const u64 nl = G->lv.size();
    u64 b = 24 + 32 * nl;
    for (u64 i = 0; i < nl; i++) b += pad8(nb[2 * i]) + pad8(nb[2 * i + 1]) + pad8(4 * G->lv[i].g);
    return b + 2 * pad8(4ull * G->k) + 4 * 256;
}

int lcg_vbyte_encode(lcg_ctx* ctx, const uint32_t* in, uint64_t n, uint8_t* out, uint64_t cap, uint64_t* out_bytes) {
    if (!ctx || !out_bytes || (n && (!in || !out))) return LCG_EINVAL;
    const Range range("lcg_vbyte_encode");
    u32* cnt = nullptr;
    u64* off = nullptr;
    try {
        ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
        kt_reset(ctx);
        reset_status(ctx);
        *out_bytes = 0;
        if (n == 0) return LCG_OK;
        const u64 tiles = vb_encode_tiles(n);
        cnt = dalloc<u32>(ctx, tiles);
        off = dalloc<u64>(ctx, tiles);
        vb_count_col(ctx, in, nullptr, n, cnt, off, ctx->scratch + 1);
        u64 nb = 0;
        // a buffer that holds any stream of n values need not wait for this one's size
        // (which a timed launch is recorded with)
        const bool fits = cap / 5 >= n && ctx->ktime == 0;
        if (!fits) {
            fetch(ctx, {{&nb, ctx->scratch + 1, 8}});
            *out_bytes = nb;
            fail_if(ctx, cap < nb, LCG_EINVAL, "output buffer too small");
        }
        vb_write_col(ctx, in, nullptr, n, off, out, false, nb);
        dfree(ctx, cnt);
        dfree(ctx, off);
        cnt = nullptr;
        off = nullptr;
        const DevStatus st = fits ? read_status(ctx, &nb, ctx->scratch + 1, 8) : read_status(ctx);
        *out_bytes = nb;
        kt_collect(ctx);
        check_device_status(ctx, st);
        return LCG_OK;
    } catch (const Fail& f) {
        cudaStreamSynchronize(ctx->st);
        if (cnt) cudaFree(cnt);
        if (off) cudaFree(off);
        return f.code;
    }
}

int lcg_vbyte_decode(lcg_ctx* ctx, const uint8_t* in, uint64_t nbytes, uint32_t* out, uint64_t n) {
    if (!ctx || (nbytes && !in) || (n && !out)) return LCG_EINVAL;
    const Range range("lcg_vbyte_decode");
    VbTemps t;
    try {
        ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
        kt_reset(ctx);
        fail_if(ctx, nbytes < n || nbytes > 5 * n, LCG_EINVAL, "stream length does not fit the value count");
        if (n == 0) return LCG_OK;
        reset_status(ctx);
        const u64 tiles = vb_decode_tiles(nbytes);
        t.cnt = dalloc<u32>(ctx, tiles);
        t.off = dalloc<u64>(ctx, tiles);
        vb_decode_col(ctx, in, nbytes, n, 0, 1ull << 32, out, t, ctx->scratch + 1);
        dfree(ctx, t.cnt);
        dfree(ctx, t.off);
        t = VbTemps{};
        const DevStatus st = read_status(ctx);
        kt_collect(ctx);
        check_device_status(ctx, st);
        return LCG_OK;
    } catch (const Fail& f) {
        cudaStreamSynchronize(ctx->st);
        if (t.cnt) cudaFree(t.cnt);
        if (t.off) cudaFree(t.off);
        return f.code;
    }
}

int lcg_vbyte_size(lcg_ctx* ctx, const lcg_grammar* G, uint64_t* bytes) {
    if (!ctx || !G || !bytes) return LCG_EINVAL;
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    fail_if(ctx, G->device != ctx->device, LCG_EINVAL, "grammar on another device");
    *bytes = vb_total_bytes(G, vb_section_bytes(ctx, G));
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_export_vbyte(lcg_ctx* ctx, const lcg_grammar* G, void* out, uint64_t cap, int out_on_device,
                     uint64_t* bytes) {
    if (!ctx || !G || !out) return LCG_EINVAL;
    const Range range("lcg_export_vbyte");
    std::vector<void*> temps;
    try {
        ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
        fail_if(ctx, G->device != ctx->device, LCG_EINVAL, "grammar on another device");
        fail_if(ctx, ((uintptr_t)out & 7) != 0, LCG_EINVAL, "VByte buffer must be 8-byte aligned");
        kt_reset(ctx);
        reset_status(ctx);
        const u64 nl = G->lv.size();
        // columns: [2 i] rule lengths, [2 i + 1] right-hand sides of level i + 1;
        // one launch per step over all of them
        const u32 ncols = (u32)(2 * nl);
        fail_if(ctx, ncols > (u32)kVbMaxCols, LCG_EINVAL, "too many levels");
        std::vector<VbEncCol> cols(ncols + 1, VbEncCol{nullptr, nullptr, 0, 0, nullptr});
        u64 T = 0;
        for (u32 c = 0; c < ncols; c++) {
            const Level& L = G->lv[c / 2];
            cols[c] = (c % 2) ? VbEncCol{L.rhs, nullptr, L.G, T, nullptr} : VbEncCol{nullptr, L.rhs_off, L.g, T, nullptr};
            T += vb_encode_tiles(cols[c].n);
        }
        cols[ncols].tile0 = T;
        double in_bytes = 0, out_bytes = 0;
        for (u32 c = 0; c < ncols; c++) in_bytes += (c % 2 ? 4.0 : 8.0) * (double)cols[c].n;
        VbEncCol* dcols = dalloc<VbEncCol>(ctx, ncols + 1);
        temps.push_back(dcols);
        u32* cnt = dalloc<u32>(ctx, T);
        temps.push_back(cnt);
        u64* off = dalloc<u64>(ctx, T);
        temps.push_back(off);
        u64* colb = dalloc<u64>(ctx, ncols + 1);
        temps.push_back(colb);
        ck(ctx, cudaMemsetAsync(colb, 0, 8 * (ncols + 1), ctx->st), "memset");
        ck(ctx, cudaMemcpyAsync(dcols, cols.data(), sizeof(VbEncCol) * (ncols + 1), cudaMemcpyHostToDevice, ctx->st),
           "columns");
        if (T) {
            const int h = kt_begin(ctx, "k_vb_tile_bytes", in_bytes);
            ck(ctx, launch_vb_tile_bytes_all(dcols, ncols, T, cnt, colb, ctx->st), "k_vb_tile_bytes");
            kt_end(ctx, h);
            ctx->launches++;
            vb_scan(ctx, cnt, T, off, ctx->scratch + 1);
        }
        std::vector<u64> nb(ncols + 1);
        fetch(ctx, {{nb.data(), colb, 8 * (ncols + 1)}});
        for (u32 c = 0; c < ncols; c++) out_bytes += (double)nb[c];
        const u64 total = vb_total_bytes(G, nb);
        if (bytes) *bytes = total;
        fail_if(ctx, cap < total, LCG_EINVAL, "VByte buffer too small");
        u8* dst = (u8*)out;
        if (!out_on_device) {
            dst = dalloc<u8>(ctx, total);
            temps.push_back(dst);
        }
        std::vector<u64> head(3 + 4 * nl);
        head[0] = kVbMagic;
        head[1] = G->k;
        head[2] = nl;
        for (u64 i = 0; i < nl; i++) {
            head[3 + 4 * i] = G->lv[i].g;
            head[4 + 4 * i] = G->lv[i].G;
            head[5 + 4 * i] = nb[2 * i];
            head[6 + 4 * i] = nb[2 * i + 1];
        }
        ck(ctx, cudaMemcpyAsync(dst, head.data(), 8 * head.size(), cudaMemcpyHostToDevice, ctx->st), "header");
        u64 pos = 8 * head.size();
        Copies copies;
        auto copy_u32 = [&](const u32* src, u64 n) {
            copies.add(dst + pos, src, n, true);
            pos += pad8(4 * n);
        };
        for (u64 i = 0; i < nl; i++) {
            const Level& L = G->lv[i];
            cols[2 * i].dst = dst + pos;
            pos += pad8(nb[2 * i]);
            cols[2 * i + 1].dst = dst + pos;
            pos += pad8(nb[2 * i + 1]);
            copy_u32(L.F, L.g);
        }
        if (T) {
            ck(ctx, cudaMemcpyAsync(dcols, cols.data(), sizeof(VbEncCol) * (ncols + 1), cudaMemcpyHostToDevice,
                                    ctx->st),
               "columns");
            const int h = kt_begin(ctx, "k_vb_write", in_bytes + out_bytes);
            ck(ctx, launch_vb_write_all(dcols, ncols, T, off, ctx->st), "k_vb_write");
            kt_end(ctx, h);
            ctx->launches++;
        }
        copy_u32(G->c_level, G->k);
        copy_u32(G->c_rank, G->k);
        copy_u32(G->F0, 256);
        copies.run(ctx, temps);
        fail_if(ctx, pos != total, LCG_EDEVICE, "VByte layout");
        if (!out_on_device) ck(ctx, cudaMemcpyAsync(out, dst, total, cudaMemcpyDeviceToHost, ctx->st), "export");
        for (void* p : temps) dfree(ctx, p);
        temps.clear();
        const DevStatus st = read_status(ctx);
        kt_collect(ctx);
        check_device_status(ctx, st);
        return LCG_OK;
    } catch (const Fail& f) {
        cudaStreamSynchronize(ctx->st);
        for (void* p : temps) cudaFree(p);
        return f.code;
    } catch (const std::bad_alloc&) {
        ctx->err = "host allocation failed";
        cudaStreamSynchronize(ctx->st);
        for (void* p : temps) cudaFree(p);
        return LCG_ENOMEM;
    }
}

// Largest level of an imported grammar that shares an allocation with others.
constexpr u64 kImportSlabRules = 65536, kImportSlabSymbols = 262144;

// F^0[s] on the host.
static u32 host_h0(const lcg_ctx* ctx, u32 s) {
    const LevelHash h = level_hash(ctx, 0);
    return (u32)((u64)(((unsigned __int128)h.a * s + h.b) % kP61) & h.mmask);
}

int lcg_import_vbyte(lcg_ctx* ctx, const void* buf, uint64_t size, int buf_on_device, lcg_grammar** out) {
    if (!ctx || !buf || !out) return LCG_EINVAL;
    *out = nullptr;
    const Range range("lcg_import_vbyte");
    lcg_grammar* G = nullptr;
    u8* staging = nullptr;
    std::vector<void*> temps;
    try {
        ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
        kt_reset(ctx);
        fail_if(ctx, ((uintptr_t)buf & 7) != 0, LCG_EINVAL, "VByte buffer must be 8-byte aligned");
        fail_if(ctx, size < 24, LCG_EINVAL, "not a VByte grammar");
        const u8* b = (const u8*)buf;
        auto read_host = [&](void* dst, u64 off, u64 n) {
            if (n == 0) return;
            if (buf_on_device) {
                fetch(ctx, {{dst, b + off, n}});
            } else {
                std::memcpy(dst, b + off, n);
            }
        };
        // the fixed header and the level headers of most grammars in one read
        u64 first[3 + 4 * 64];
        const u64 got = std::min<u64>(size & ~7ull, sizeof(first));
        read_host(first, 0, got);
        const u64* h3 = first;
        fail_if(ctx, h3[0] != kVbMagic, LCG_EINVAL, "not a VByte grammar");
        const u64 k = h3[1], nl = h3[2];
        fail_if(ctx, k > 0xffffffffull || nl > 4096 || size < 24 + 32 * nl, LCG_EINVAL, "malformed VByte header");
        fail_if(ctx, nl >= ctx->levels, LCG_ELEVELS, "grammar has more levels than the hash family has functions");
        std::vector<u64> hd(4 * nl);
        if (24 + 32 * nl <= got) std::memcpy(hd.data(), first + 3, 32 * nl);
        else read_host(hd.data(), 24, 32 * nl);
        std::vector<u64> off_len(nl), off_rhs(nl), off_F(nl);
        u64 pos = 24 + 32 * nl;
        for (u64 i = 0; i < nl; i++) {
            const u64 g = hd[4 * i], Gs = hd[4 * i + 1], nbl = hd[4 * i + 2], nbr = hd[4 * i + 3];
            fail_if(ctx, g > kMaxRank || Gs > (1ull << 40) || Gs < g || (g == 0) != (Gs == 0), LCG_EINVAL,
                    "malformed level sizes");
            fail_if(ctx, nbl < g || nbl > 5 * g || nbr < Gs || nbr > 5 * Gs, LCG_EINVAL,
                    "stream lengths do not fit the level sizes");
            off_len[i] = pos;
            pos += pad8(nbl);
            off_rhs[i] = pos;
            pos += pad8(nbr);
            off_F[i] = pos;
            pos += pad8(4 * g);
            fail_if(ctx, pos > size, LCG_EINVAL, "truncated");
        }
        const u64 off_cl = pos, off_cr = pos + pad8(4 * k), off_F0 = pos + 2 * pad8(4 * k);
        fail_if(ctx, off_F0 + 4 * 256 != size, LCG_EINVAL, "wrong size");
        // C entries name existing rules
        std::vector<uint32_t> tail((size - off_cl) / 4);
        read_host(tail.data(), off_cl, size - off_cl);
        const uint32_t *cl = tail.data(), *cr = cl + (off_cr - off_cl) / 4, *theirs = cl + (off_F0 - off_cl) / 4;
        for (u64 j = 0; j < k; j++) {
            fail_if(ctx, cl[j] > nl, LCG_EINVAL, "C entry " + std::to_string(j) + " names a missing level");
            const u64 lim = cl[j] == 0 ? 256 : hd[4 * (cl[j] - 1)];
            fail_if(ctx, cr[j] >= lim, LCG_EINVAL, "C entry " + std::to_string(j) + " names a missing rule");
        }
        const u8* src = b;
        if (!buf_on_device) {
            staging = dalloc<u8>(ctx, size);
            ck(ctx, cudaMemcpyAsync(staging, buf, size, cudaMemcpyHostToDevice, ctx->st), "upload");
            src = staging;
        }
        reset_status(ctx);
        G = new_grammar(ctx);
        Copies copies;
        if (k) {
            grow_c(ctx, G, (u32)k);
            copies.add(G->c_level, src + off_cl, k);
            copies.add(G->c_rank, src + off_cr, k);
            G->k = (u32)k;
        }
        // the levels' arrays, and one decode over all columns: every level's
        // rule lengths (into one array, scanned into the offsets afterwards)
        // and right-hand sides
        u64 sum_g = 0, max_g = 0;
        for (u64 i = 0; i < nl; i++) {
            sum_g += hd[4 * i];
            max_g = std::max<u64>(max_g, hd[4 * i]);
        }
        // small levels share one allocation (a level that grows leaves its part unused)
        auto in_slab = [&](u64 i) {
            return hd[4 * i] > 0 && hd[4 * i] <= kImportSlabRules && hd[4 * i + 1] <= kImportSlabSymbols;
        };
        Parts parts;
        for (u64 i = 0; i < nl; i++)
            if (in_slab(i)) {
                parts.take((hd[4 * i] + 1) * sizeof(u64));
                parts.take(hd[4 * i] * sizeof(u32));
                parts.take(hd[4 * i + 1] * sizeof(u32));
            }
        unsigned char* slab = nullptr;
        if (parts.size) {
            slab = dalloc<unsigned char>(ctx, parts.size);
            G->slabs.push_back(slab);
        }
        parts = Parts{};
        u32* lens = dalloc<u32>(ctx, sum_g);
        temps.push_back(lens);
        std::vector<VbDecCol> cols;
        std::vector<VbLevelOff> lvo;
        u64 T = 0, gbase = 0;
        for (u64 i = 0; i < nl; i++) {
            const u64 g = hd[4 * i], Gs = hd[4 * i + 1];
            G->lv.emplace_back();
            Level& L = G->lv.back();
            if (in_slab(i)) {
                L.rhs_off = (u64*)(slab + parts.take((g + 1) * sizeof(u64)));
                L.F = (u32*)(slab + parts.take(g * sizeof(u32)));
                L.rhs = (u32*)(slab + parts.take(Gs * sizeof(u32)));
                L.cap_g = g;
                L.cap_G = Gs;
                L.shared_rules = L.shared_rhs = true;
            } else {
                grow_level(ctx, L, g, Gs);
            }
            L.g = g;
            L.G = Gs;
            L.rvalid = false;
            if (g == 0) continue;
            const u64 prev = i == 0 ? 256 : hd[4 * (i - 1)];
            cols.push_back(VbDecCol{src + off_len[i], hd[4 * i + 2], g, 1, 1ull << 32, lens + gbase, T});
            T += vb_decode_tiles(hd[4 * i + 2]);
            cols.push_back(VbDecCol{src + off_rhs[i], hd[4 * i + 3], Gs, 0, prev, L.rhs, T});
            T += vb_decode_tiles(hd[4 * i + 3]);
            lvo.push_back(VbLevelOff{L.rhs_off, g, Gs, gbase});
            gbase += g;
            copies.add(L.F, src + off_F[i], g);
        }
        const u32 ncols = (u32)cols.size();
        fail_if(ctx, ncols > (u32)kVbMaxCols, LCG_EINVAL, "too many levels");
        cols.push_back(VbDecCol{nullptr, 0, 0, 0, 0, nullptr, T});
        if (T) {
            VbDecCol* dcols = dalloc<VbDecCol>(ctx, cols.size());
            temps.push_back(dcols);
            VbLevelOff* dlvo = dalloc<VbLevelOff>(ctx, lvo.size());
            temps.push_back(dlvo);
            u32* cnt = dalloc<u32>(ctx, T);
            temps.push_back(cnt);
            u64* off = dalloc<u64>(ctx, T);
            temps.push_back(off);
            u64* gscan = dalloc<u64>(ctx, sum_g);
            temps.push_back(gscan);
            ck(ctx, cudaMemcpyAsync(dcols, cols.data(), sizeof(VbDecCol) * cols.size(), cudaMemcpyHostToDevice,
                                    ctx->st),
               "columns");
            ck(ctx, cudaMemcpyAsync(dlvo, lvo.data(), sizeof(VbLevelOff) * lvo.size(), cudaMemcpyHostToDevice,
                                    ctx->st),
               "levels");
            double nbytes = 0, nvals = 0;
            for (u32 c = 0; c < ncols; c++) {
                nbytes += (double)cols[c].nb;
                nvals += (double)cols[c].n;
            }
            int h = kt_begin(ctx, "k_vb_tile_ends", nbytes);
            ck(ctx, launch_vb_tile_ends_all(dcols, ncols, T, cnt, ctx->st), "k_vb_tile_ends");
            kt_end(ctx, h);
            vb_scan(ctx, cnt, T, off, ctx->scratch + 1);
            h = kt_begin(ctx, "k_vb_dwrite", nbytes + 4.0 * nvals);
            ck(ctx, launch_vb_dwrite_all(dcols, ncols, T, off, ctx->ds, ctx->st), "k_vb_dwrite");
            kt_end(ctx, h);
            vb_scan(ctx, lens, sum_g, gscan, ctx->scratch + 1);
            h = kt_begin(ctx, "k_vb_offsets", 12.0 * (double)sum_g);
            ck(ctx, launch_vb_offsets_all(dlvo, (u32)lvo.size(), max_g, gscan, ctx->scratch + 1, ctx->ds, ctx->st),
               "k_vb_offsets");
            kt_end(ctx, h);
            ctx->launches += 3;
        }
        copies.run(ctx, temps);
        // (does nothing after a stream that is malformed)
        check_fingerprints(ctx, G, temps);
        dfree(ctx, staging);
        staging = nullptr;
        for (void* p : temps) dfree(ctx, p);
        temps.clear();
        const DevStatus st = read_status(ctx);
        kt_collect(ctx);
        fail_if(ctx, st.error == kErrFormat, LCG_EINVAL, "malformed VByte form");
        fail_if(ctx, st.error == kErrMismatch, LCG_EMISMATCH,
                "imported fingerprints differ from those of this context's hash family");
        check_device_status(ctx, st);
        for (u32 c = 0; c < 256; c++)
            fail_if(ctx, theirs[c] != host_h0(ctx, c), LCG_EMISMATCH, "VByte grammar: F0 of another hash family");
        *out = G;
        return LCG_OK;
    } catch (const Fail& f) {
        cudaStreamSynchronize(ctx->st);
        if (staging) cudaFree(staging);
        for (void* p : temps) cudaFree(p);
        free_grammar_now(G);
        return f.code;
    } catch (const std::bad_alloc&) {
        ctx->err = "host allocation failed";
        cudaStreamSynchronize(ctx->st);
        if (staging) cudaFree(staging);
        for (void* p : temps) cudaFree(p);
        free_grammar_now(G);
        return LCG_ENOMEM;
    }
}

void lcg_grammar_free(lcg_grammar* G) { free_grammar_now(G); }

int lcg_postprocess(lcg_ctx* ctx, const lcg_grammar* G, lcg_pp** out) {
    if (!ctx || !G || !out) return LCG_EINVAL;
    *out = nullptr;
    const Range range("lcg_postprocess");
    LCG_GUARD_BEGIN
    ck(ctx, cudaSetDevice(ctx->device), "cudaSetDevice");
    fail_if(ctx, G->device != ctx->device, LCG_EINVAL, "grammar on another device");
    *out = postprocess(ctx, G);
    return LCG_OK;
    LCG_GUARD_END
}

int lcg_pp_stats_of(const lcg_pp* pp, lcg_pp_stats* out) {
    if (!pp || !out) return LCG_EINVAL;
    *out = pp->stats;
    return LCG_OK;
}

int lcg_pp_export(const lcg_pp* pp, uint8_t* kind, uint64_t* rhs_off, uint32_t* rhs, uint32_t* c) {
    if (!pp || !kind || !rhs_off || (!rhs && pp->size) || (!c && pp->k)) return LCG_EINVAL;
    if (cudaSetDevice(pp->device) != cudaSuccess) return LCG_EDEVICE;
    bool ok = cudaMemcpy(kind, pp->kind, pp->rules, cudaMemcpyDeviceToHost) == cudaSuccess &&
              cudaMemcpy(rhs_off, pp->rhs_off, 8 * (pp->rules + 1), cudaMemcpyDeviceToHost) == cudaSuccess;
    if (ok && pp->size) ok = cudaMemcpy(rhs, pp->rhs, 4 * pp->size, cudaMemcpyDeviceToHost) == cudaSuccess;
    if (ok && pp->k) ok = cudaMemcpy(c, pp->c, 4ull * pp->k, cudaMemcpyDeviceToHost) == cudaSuccess;
    return ok ? LCG_OK : LCG_EDEVICE;
}

void lcg_pp_free(lcg_pp* pp) { free_pp(pp); }

}  // extern "C"
