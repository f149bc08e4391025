// Kernels of one BuildGram round (Sec. 3.3) over all active strings of a
// batch, and their host-side launchers.
//
// A round i reads the sequence T^i (bytes in round 1, uint32 ids later) of
// the active strings, laid out back to back with offsets soff[0..k], and the
// fingerprints of its symbols (F^0 of the bytes in round 1; afterwards the
// fingerprint stream the previous round's parse wrote).  It runs:
//   k_tile_strings  per block step of k_breaks, the string holding its first
//                   position, and the bitmap of string starts
//   k_breaks   RandLMSPar break bits (Eq. rand_types) as a bitmap, 32
//              positions per thread; the phrases of every parse unit; the
//              first phrase of every string
//   k_scan2    unit phrase counts -> global phrase indices (single pass)
//   k_strings  per-string phrase ranges; strings that become one phrase retire
//   k_parse    per unit: the phrase starts (from the bitmap), a key per phrase
//              (its symbols when short, else a hash of its Eq. fast_hash
//              polynomial and its position), its fingerprint F^i and its slot
//              in the round's phrase table, whose value is the smallest phrase
//              index of the content (content-confirmed, never by hash alone);
//              T^{i+1} gets the slot's id and the fingerprint, retired strings
//              left out
//   k_mark, k_popscan, k_rank
//              first-occurrence naming: the first occurrences of the new
//              phrases are marked in a bitmap over phrase indices, and a
//              phrase's rank is the number of marks before its own
//   k_rule_offs  rule lengths -> right-hand-side offsets
//   k_rules    the level-i rules in rank order: rhs (ids translated to ranks)
//              and F^i, and the ranks of the retired strings' roots
// The sequence between the rounds holds ids (slots), not ranks, and the parse
// computes a phrase's fingerprint from the stream it reads anyway.  Before,
// a rewrite pass followed the naming and read (F^i, rank) of every phrase
// from an array indexed by slot: one random DRAM sector per phrase in the
// rounds whose table is beyond L2 (4 x 3.1 Gbp: 42.3 ms of 218 ms).
// The short rounds at a build's end (and the whole of a small build) run in two
// cooperative launches: k_parse_small and k_naming_small, further down.
// Every kernel of the round starts with pdl_wait(): it is launched with
// programmatic dependent launch after the one before it.
#include <algorithm>
#include <type_traits>
#include <utility>

#include "lcg_dev.cuh"
#include "lcg_internal.h"
#include "per_device.h"
#include "table.cuh"

namespace lcg {

// Sizes of a round: from the device when the round was enqueued without a
// host synchronisation, else from the arguments.
__device__ __forceinline__ u64 round_n(const RoundArgs& a) { return a.d_n ? *a.d_n : a.n; }
__device__ __forceinline__ u32 round_k(const RoundArgs& a) { return a.d_k ? (u32)*a.d_k : a.k; }

// A round stops as soon as it, or the round before it, has failed (an error,
// or a phrase table past its load limit): its inputs and buffers can no longer
// be trusted, and the host discards or reruns it.  Called by every thread of a
// block; the answer is the same for the whole block.
__device__ bool round_halted(const RoundArgs& a) {
    __shared__ int s_halt;
    __syncthreads();
    if (threadIdx.x == 0) {
        // (four reads in flight together)
        const DevStatus* before = a.ds_prev ? a.ds_prev : a.ds;
        const u32 h0 = vload(&a.ds->error), h1 = vload(&a.ds->overflow);
        const u32 h2 = vload(&before->error), h3 = vload(&before->overflow);
        s_halt = (h0 | h1 | h2 | h3) != 0 ? 1 : 0;
    }
    __syncthreads();
    return s_halt != 0;
}

// A read of the round's input.  The short rounds' launches (kLive) read what their own
// earlier steps wrote, for which the non-coherent path is not defined: it is for data
// that nothing writes while the kernel runs.
template <bool kLive, typename T>
__device__ __forceinline__ T ld_in(const T* p) {
    if constexpr (kLive) return *p;
    else return __ldg(p);
}

// index of the string holding position `pos`: largest j with soff[j] <= pos
template <bool kLive>
__device__ __forceinline__ u32 string_of(const u64* soff, u32 k, u64 pos) {
    u32 lo = 0, hi = k;  // answer in [lo, hi)
    while (hi - lo > 1) {
        const u32 mid = (lo + hi) >> 1;
        if (ld_in<kLive>(soff + mid) <= pos) lo = mid; else hi = mid;
    }
    return lo;
}

// --------------------------------------------------------------------------
// k_parse
// --------------------------------------------------------------------------
//
// The warps of a persistent grid take units of U positions (an eighth of
// lcg_tuning.parse_tile: 128, 256 or 512) and never wait for one another.  A
// warp copies its next unit's symbols (and kHalo more) to shared memory while
// it parses the current one, and lists the unit's phrase starts from the
// break bitmap.  Each phrase gets a key: its symbols packed exactly when they
// fit in 124 bits, else a hash of its polynomial H (Eq. fast_hash) with its
// length and position, confirmed by comparing contents.  It is looked up
// first in the resident level (when parsing against a resident grammar and
// all its symbols are resident), then in the round's table, where a new
// content is claimed; the slot says the claim's number (the id) and the
// fingerprint F^i.  Phrase p of the round goes to place p of T^{i+1}, less the
// retired strings' phrases before it.
//
// Most phrases are answered with one read: in rank rounds of their home slot,
// in byte rounds of a per-block cache of packed phrases.  What that read does not answer goes to the warp's queue,
// with all that the long path needs (so the queue outlives the unit), and the
// long path runs on 32 queued phrases at a time: fingerprint, probing, claim.
//
// What bounds it: the byte round instruction issue, the rank rounds random
// 32-byte DRAM reads (one slot per phrase) and, with many new phrases, the
// chain slot read -> compare-and-swap -> store of the long path.

constexpr int kParseThreads = 32 * (int)kParseWarps;
constexpr int kUnitMin = 128, kUnitMax = 512;
// Warps of a k_parse block.  A byte round's blocks fill their SM, so that its warps
// share one phrase cache of 8192 places instead of four of 2048 (round 1 of 4 x 3.1
// Gbp, 22 k phrases: 39.6 ms, now 37.2; 64 x 5 Mbp 1.06 ms, 0.97).  Three probes in
// it: text, whose phrases fill any cache, takes 0.72 ms so and 0.76 with eight.
template <typename T>
constexpr int parse_warps = sizeof(T) == 1 ? 32 : (int)kParseWarps;
template <int W>
constexpr int parse_blocks = W >= 32 ? 1 : W >= 16 ? 2 : (int)kParseBlocksMax;
constexpr int kHalo = 64;  // symbols staged past the unit's end

// Unit order of the rank rounds' parse: with `stripes` = k > 1
// the round's tiles are cut into k equal stripes and taken interleaved
// (stripe 0's first tile, stripe 1's first tile, ..., then every stripe's
// second tile), so that strings which are near-copies of one another at the
// same offsets (k assemblies of one genome) are parsed side by side and the
// later copies find the first copy's new table entries still in L2.  Logical
// tile l in [0, k * ceil(T / k)) names tile (l % k) * ceil(T / k) + l / k, or
// nothing (>= T).  Phrases keep their indices, so the result does not depend
// on the order.
__device__ __forceinline__ u64 stripe_tiles(u64 ntiles, u32 stripes) {
    if (stripes <= 1) return ntiles;
    const u64 per = (ntiles + stripes - 1) / stripes;
    return per * stripes;
}
__device__ __forceinline__ u64 stripe_tile(u64 l, u64 ntiles, u32 stripes) {
    if (stripes <= 1) return l;
    const u64 per = (ntiles + stripes - 1) / stripes;
    return (l % stripes) * per + l / stripes;
}
constexpr int kCacheProbes = 3;
// Byte rounds: so many misses among a warp's 32 phrases are looked up in the table
// at once (text, whose phrases are too many for the cache); fewer go to the
// queue, where a full warp takes the long path.  Round 1 of 32 x 2 MB of text:
// 1.06 ms with the queue alone, 0.72 ms with 8 to 16 here, 0.84 ms with 24.
constexpr int kByteFind = 16;
// A cache entry's value: bits 58..63 an exponent x, bits 32..57 the id, the low
// half F^1.  The phrase's first occurrence is known to be before 2^x, so a
// phrase at place 2^x or later needs nothing more; the warps of a block are at
// different places, and one before that takes the long path, which keeps the
// first occurrence right.

// Long phrases (hashed keys) in rank rounds: symbols per round trip when a
// match is confirmed by content (byte rounds take one at a time).
constexpr int kCompareBatchR = 4;
// Phrases longer than kLongLen (N-runs of DNA, repeated text) are hashed and
// compared by a whole warp after the unit's other phrases: a thread alone
// would spend a round trip per symbol on them while its warp waits.
constexpr int kLongLen = 32;

// --------------------------------------------------------------------------
// k_breaks: the round's break bitmap (Eq. rand_types)
// --------------------------------------------------------------------------
//
// A phrase starts at x when x starts a string, or f[x-1] > f[x] and x has
// type S: the first fingerprint right of x (within the string) that differs
// from f[x] is larger than f[x].  Thread t of a block step owns the 32
// positions of bitmap word t and works on bit masks: gt / lt mark positions
// whose right neighbour (in the string) is larger / smaller, stop marks
// positions whose right neighbour starts a string (or is past the end).  A
// position's type is decided by the first of these at or above it, so the S
// mask is gt spread down over the undecided positions (five doubling steps).
// Positions above the thread's last decision take the type of the next
// thread's first position, found through per-thread summaries; past the block
// step, the type of the next step's first position.  Then breaks = starts |
// ((lt << 1) & S), bit 0 using f of the position before.
//
// A run of equal fingerprints can span many block steps (N-runs of DNA).
// Block steps are therefore taken in decreasing order from a counter, and
// each publishes the type of its first position (its "head") as soon as its
// masks are known: decided, or "open" when the whole step is one run.  A step
// whose last position is undecided reads the heads of the steps after it,
// skipping open ones, until one is decided (a look-ahead over steps that were
// all taken before it, so every wait ends); an open step then publishes the
// type it found as its head.  Each step reads its own positions once, however
// long the run.

constexpr int kBrkThreads = 256;
constexpr u64 kBrkSpan = (u64)kBrkThreads * 32;  // positions per block step
static_assert(kUnitMax <= 32 * 32, "a warp of k_breaks covers whole parse units");

// Head of block step b in the look-ahead words: (epoch << 8) | (state << 2) |
// type, state 1 = open, 2 = decided.  The word is all that passes between steps, so
// it needs no order with other accesses (as a release the store held the block's warps
// at the barrier after it).
__device__ __forceinline__ void brk_publish(u64* heads, u64 b, u64 epoch, u32 state, u32 type) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(heads + b), "l"((epoch << 8) | (state << 2) | type)
                 : "memory");
}

// Type of the first position of step j (the run continues into it), looking
// further right past open steps.  `none` is the type past the last step.
__device__ u32 brk_lookahead(const u64* heads, u64 j, u64 nsteps, u64 epoch, u32 none, DevStatus* ds) {
    for (; j < nsteps; j++) {
        u64 it = 0;
        u32 backoff = 32;
        while (true) {
            u64 w;
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(heads + j) : "memory");
            if ((w >> 8) == epoch) {
                if (((w >> 2) & 3u) == 2u) return (u32)(w & 3u);
                break;  // open: one run throughout, look at the next step
            }
            if (++it > kSpinLimit || vload(&ds->error) != 0) {
                set_error(ds, kErrTimeout);
                return none;
            }
            __nanosleep(backoff);
            if (backoff < 256) backoff <<= 1;
        }
    }
    return none;
}

// Spread the bits of `src` down over the positions of `pass` (positions that
// take the value of the position above): bit i of the result is src[j] for
// the first j >= i with pass[j] == 0, when that j is at most 31.
__device__ __forceinline__ u32 spread_down(u32 src, u32 pass) {
    u32 y = src, m = pass;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        y |= (y >> k) & m;
        m &= m >> k;
    }
    return y;
}

// Kernel bodies are device functions: k_X launches body_X on a grid, and the
// short rounds' cooperative kernels (k_parse_small, k_naming_small) run several of
// them in one launch.
// `own_step`: block b takes the steps nblocks - 1 - b, nblocks - 1 - b - gridDim.x, ...
// (a launch whose blocks are all resident, mostly more than steps): no counter, and the
// steps after the one that a block waits for are done or another block's, so it ends.
template <typename T, bool own_step = false>
__device__ __forceinline__ void body_breaks(const RoundArgs& a, u64 nblocks) {
    pdl_wait();
    constexpr bool kByte = sizeof(T) == 1;
    constexpr u32 kTypeU = 0, kTypeS = 1, kTypeL = 2, kUndecided = 3;
    constexpr int SW = kBrkThreads;  // string-start words of a step
    __shared__ u32 sF0[kByte ? 256 : 1];
    __shared__ u32 sst[SW + 1];      // string starts at base .. base + kBrkSpan
    __shared__ u32 sfirst[kBrkThreads];  // type of each thread's first position
    __shared__ u32 s_bits[kBrkThreads], s_pre[kBrkThreads];
    __shared__ u64 s_step[2];
    __shared__ u32 s_open, s_carry;
    if (round_halted(a)) return;
    const T* S = (const T*)a.S;
    const u32* Sf = a.Sf;
    const u64 n = round_n(a);
    const int tid = threadIdx.x, lane = tid & 31;
    if constexpr (kByte)
        for (int x = tid; x < 256; x += kBrkThreads) sF0[x] = a.Fprev[x];
    auto fpos = [&](u64 x) -> u32 {  // fingerprint of position x < n
        if constexpr (kByte) return sF0[S[x]]; else return ld_in<own_step>(Sf + x);
    };
    const bool aligned = kByte ? (reinterpret_cast<unsigned long long>(S) & 15) == 0
                               : (reinterpret_cast<unsigned long long>(Sf) & 15) == 0;
    nblocks = min(nblocks, (n + kBrkSpan - 1) / kBrkSpan);
    if (blockIdx.x >= nblocks && blockIdx.x > 0) return;  // more blocks than steps: no counter traffic
    u64* heads = a.heads;
    const int warp = tid >> 5;
    // Block steps in decreasing order (the counter starts at 0 every round).  In the
    // rounds over ranks, with many steps a block, the step after the next is asked for
    // and the next one's string starts are read while a step is worked on (rounds 2 and
    // 3 of 4 x 3.1 Gbp: 4.29 and 1.39 ms, now 3.68 and 1.22); with few, a step that a
    // block holds back would be one that another could have begun.  Not so the byte
    // round, whose steps more often end in a run and wait for the next one's head (10.2
    // ms, 10.0 without).
    const bool ahead = !kByte && !own_step && nblocks > 4 * (u64)gridDim.x;
    auto step_of = [&](u64 t) { return t < nblocks ? nblocks - 1 - t : ~0ull; };
    u64 own = blockIdx.x;
    auto ticket = [&]() {
        if constexpr (own_step) {
            const u64 t = own;
            own += gridDim.x;
            return step_of(t);
        } else {
            return step_of(atomicAdd(&a.ds->aux[0], 1ull));
        }
    };
    // string starts of a step (bitmap of k_tile_strings; n counts as one): this
    // thread's word, and the one past the step
    auto starts = [&](u64 b, u32 w) {
        const u64 gw = b * (kBrkSpan / 32) + (u64)w;
        return b != ~0ull && gw < a.sbm_words ? ld_in<own_step>(a.sbm + gw) : 0u;
    };
    if (tid == 0) {
        s_step[0] = ticket();
        s_step[1] = ahead ? ticket() : ~0ull;
    }
    __syncthreads();  // also: sF0 loaded
    u64 b = s_step[0], b_next = s_step[1];
    u32 my_starts = starts(b, (u32)tid), end_starts = tid == 0 ? starts(b, SW) : 0u;
    for (u32 it = 0; b != ~0ull; it++) {
        u64 asked = ~0ull;
        if (ahead && tid == 0) asked = ticket();
        const u32 next_starts = ahead ? starts(b_next, (u32)tid) : 0u,
                  next_end = ahead && tid == 0 ? starts(b_next, SW) : 0u;
        const u64 base = b * kBrkSpan;
        const u64 bend = min(base + kBrkSpan, n);
        sst[tid] = my_starts;
        if (tid == 0) sst[SW] = end_starts;
        const u64 x0 = base + 32ull * (u64)tid;
        u32 f[32];
        if (aligned && x0 + 32 <= n) {
            if constexpr (kByte) {
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const uint4 v = __ldcs(reinterpret_cast<const uint4*>(S + x0 + 16 * h));
                    const u32 w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int i = 0; i < 16; i++) f[16 * h + i] = sF0[(w[i >> 2] >> (8 * (i & 3))) & 0xFFu];
                }
            } else {
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const uint4 v = __ldcs(reinterpret_cast<const uint4*>(Sf + x0 + 4 * q));
                    f[4 * q] = v.x;
                    f[4 * q + 1] = v.y;
                    f[4 * q + 2] = v.z;
                    f[4 * q + 3] = v.w;
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 32; i++) f[i] = (x0 + i < n) ? fpos(x0 + i) : 0u;
        }
        // f of the position after the thread's last, and of the one before its first
        u32 fnext = __shfl_down_sync(0xffffffffu, f[0], 1);
        u32 fprev = __shfl_up_sync(0xffffffffu, f[31], 1);
        if (lane == 31 && x0 + 32 < n) fnext = fpos(x0 + 32);
        if (lane == 0 && x0 > 0 && x0 - 1 < n) fprev = fpos(x0 - 1);
        __syncthreads();  // sst loaded
        const u32 st = sst[tid];                      // starts at x0 .. x0 + 31
        const u32 st_next = (sst[tid + 1] & 1u);      // start at x0 + 32
        // masks over the thread's positions: right neighbour larger, smaller,
        // or a string start / the end of the sequence
        const u32 stop = (st >> 1) | (st_next << 31);
        u32 gt = 0, lt = 0;
#pragma unroll
        for (int i = 0; i < 31; i++) {
            gt |= (u32)(f[i + 1] > f[i]) << i;
            lt |= (u32)(f[i + 1] < f[i]) << i;
        }
        gt |= (u32)(fnext > f[31]) << 31;
        lt |= (u32)(fnext < f[31]) << 31;
        gt &= ~stop;
        lt &= ~stop;
        const u32 dec = gt | lt | stop;  // positions whose type is decided here
        u32 sm = spread_down(gt, ~dec);
        u32 lm = spread_down(lt, ~dec);
        // type of the thread's first position (or undecided: one run throughout)
        sfirst[tid] = dec == 0 ? kUndecided : (sm & 1u) ? kTypeS : (lm & 1u) ? kTypeL : kTypeU;
        const bool open = dec != (u32)~0u && ((dec >> 31) & 1u) == 0;  // positions above the last decision
        if (tid == kBrkThreads - 1) s_open = open ? 1u : 0u;
        __syncthreads();
        if (warp == 0) {
            // the step's head: the type of the first thread whose first position is decided
            u32 head = kUndecided;
            for (int c = 0; c < kBrkThreads / 32; c++) {
                const u32 v = sfirst[c * 32 + lane];
                const unsigned m = __ballot_sync(0xffffffffu, v != kUndecided);
                if (m) {
                    head = __shfl_sync(0xffffffffu, v, __ffs(m) - 1);
                    break;
                }
            }
            if (lane == 0) {
                brk_publish(heads, b, a.brk_epoch, head == kUndecided ? 1u : 2u, head == kUndecided ? 0u : head);
                // type of the next step's first position (the last thread's run goes on there)
                u32 carry = kTypeU;
                if (bend < n && s_open) carry = brk_lookahead(heads, b + 1, nblocks, a.brk_epoch, kTypeU, a.ds);
                if (head == kUndecided) brk_publish(heads, b, a.brk_epoch, 2u, carry);
                s_carry = carry;
            }
        }
        __syncthreads();
        if (open) {
            // positions above the last decision take the type of position x0 + 32:
            // the first decided thread after this one, else the next step's head
            u32 carry = s_carry;
            for (int t = tid + 1; t < kBrkThreads; t++) {
                const u32 c = sfirst[t];
                if (c != kUndecided) {
                    carry = c;
                    break;
                }
            }
            const int hi = 31 - __clz(dec | 1u);  // highest decided position (or 0)
            const u32 top = dec == 0 ? ~0u : ~((2u << hi) - 1u);
            if (carry == kTypeS) sm |= top;
            if (carry == kTypeL) lm |= top;
        }
        u32 bits = st | ((lt << 1) & sm);
        if (fprev > f[0] && (sm & 1u)) bits |= 1u;
        if (x0 < bend) {
            if (bend - x0 < 32) bits &= (1u << (bend - x0)) - 1u;
            a.brk[x0 >> 5] = bits;
        } else {
            bits = 0;
        }
        // phrases of each parse unit (a unit is a.tp / 32 lanes of one warp)
        const u32 lpu = a.tp / 32;
        u32 ucnt = (u32)__popc(bits);
        for (u32 o = 1; o < lpu; o <<= 1) ucnt += __shfl_xor_sync(0xffffffffu, ucnt, (int)o);
        if ((lane & (int)(lpu - 1)) == 0 && x0 < bend) a.tile_cnt[x0 / a.tp] = ucnt;
        // the first phrase of every string that starts in the step: its index
        // among its unit's phrases
        if (tid == 0) s_step[it & 1] = ahead ? asked : ticket();
        if (__syncthreads_or((int)(st & bits))) {
            u32 pre = (u32)__popc(bits);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u32 y = __shfl_up_sync(0xffffffffu, pre, o);
                if (lane >= o) pre += y;
            }
            pre -= (u32)__popc(bits);
            s_bits[tid] = bits;
            s_pre[tid] = pre - __shfl_sync(0xffffffffu, pre, lane & ~(int)(lpu - 1));
            __syncthreads();
            const u32 kact = round_k(a);
            // (the rounds of one launch have no table of the steps' strings)
            const u32 j0 = a.step_str != nullptr ? a.step_str[b] : string_of<own_step>(a.soff, kact, base);
            for (u32 jj = j0 + (u32)tid;; jj += kBrkThreads) {
                const u64 s = jj < kact ? ld_in<own_step>(a.soff + jj) : ~0ull;
                if (s >= base && s < bend) {
                    const u32 x = (u32)(s - base);
                    a.string_first[jj] = s / a.tp * a.tp + s_pre[x >> 5] +
                                         __popc(s_bits[x >> 5] & ((1u << (x & 31)) - 1u));
                }
                if (__shfl_sync(0xffffffffu, s < bend ? 1u : 0u, 31) == 0) break;
            }
        }
        const u64 fresh = s_step[it & 1];
        if (ahead) {
            b = b_next;
            b_next = fresh;
            my_starts = next_starts;
            end_starts = next_end;
        } else {
            b = fresh;
            my_starts = starts(b, (u32)tid);
            end_starts = tid == 0 ? starts(b, SW) : 0u;
        }
    }
}

// What the parse's functions take from RoundArgs, in shared memory (they are not
// inlined, and a kernel's parameters passed by reference are read through
// generic addresses).
struct ParseArgs {
    const void* S;
    const u32* Sf;
    u32* Tnext;
    u32* Fnext;
    u64 n, T_cap, retired;
    LevelHash lh;
    RoundTable table;
    u64 rtab_cap;
    const RoundArgs* all;  // for what is seldom needed
    u32 sym_w, inline_most, find_inline, id_base, prev_base;
};

// Shared memory of a k_parse block (dynamic).  A warp's part holds its unit's
// symbols (and those of the unit it takes next), phrase starts and queue.
template <typename T, int U, int W>
struct ParseSmem {
    static constexpr bool kByte = sizeof(T) == 1;
    static constexpr int kCacheBits = W >= 32 ? 13 : W >= 16 ? 12 : 11;
    static constexpr int kCacheSlots = 1 << kCacheBits;
    static constexpr int kSP = U + kHalo;            // staged symbols
    // phrase starts: a phrase has two symbols or more unless it is a string's
    // first, and a string in a round two or more, so at most two phrases start
    // in three positions; one more entry for the end of the last
    static constexpr int kStarts = (2 * U / 3 + 2 + 7) / 8 * 8;
    struct Warp {
        __align__(16) T sym[2][kSP];  // (packed byte keys read whole 8-byte words past a phrase)
        ulonglong2 queue[32 + 31];
        u64 claims, claim_len;  // what the warp claimed
        unsigned short start[kStarts];
    };
    Warp w[W];
    ClaimIds ids;
    ParseArgs args;
    // byte rounds: the block's phrase cache, packed bytes -> CacheVal
    u64 ckey[kByte ? kCacheSlots : 1];
    u64 cval[kByte ? kCacheSlots : 1];
    u32 sF[kByte ? 256 : 1];  // byte rounds: F^0
    u64 cpow[kLongLen];       // c^j mod p
};

// A queued phrase: where it starts in S, its length, what is known of its home
// slot, and the cache slot it may take (0: none); with its index p.
constexpr int kPosBits = 44;  // positions and phrase indices are below 2^44
__device__ __forceinline__ ulonglong2 queue_entry(u64 pos, u32 len, u32 home, u32 cache, u64 p) {
    return make_ulonglong2(pos | ((u64)len << kPosBits) | ((u64)home << (kPosBits + 6)), p | ((u64)cache << kPosBits));
}
static_assert(kLongLen < 64, "queue entry");

// First index with R_phr >= p (the phrases of the strings that retire, ascending).
__device__ __noinline__ u64 retired_before(const RoundArgs& a, u64 p) {
    u64 lo = 0, hi = a.rc->retired;
    while (lo < hi) {
        const u64 mid = (lo + hi) >> 1;
        if (a.R_phr[mid] < p) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Phrase p becomes a symbol of T^{i+1}, or the root of its string, when
// strings retire this round (or there is no room).
__device__ __noinline__ void emit_slow(const RoundArgs& a, u64 p, u32 id, u32 F) {
    const u64 lo = retired_before(a, p);
    if (lo < a.rc->retired && a.R_phr[lo] == p) {
        a.c_level[a.R_sid[lo]] = a.level;
        a.c_rank[a.R_sid[lo]] = id;  // k_rules makes it a rank
        return;
    }
    if (p - lo >= a.T_cap) {
        set_error(a.ds, kErrCapacity);
        return;
    }
    __stcs(a.Tnext + (p - lo), id);
    __stcs(a.Fnext + (p - lo), F);
}

template <typename T, int U, int W>
__device__ __forceinline__ ParseSmem<T, U, W>& parse_smem() {
    static_assert((sizeof(ParseSmem<T, U, W>) + 1024) * parse_blocks<W> <= 228 * 1024, "shared memory of an SM");
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    return *reinterpret_cast<ParseSmem<T, U, W>*>(dyn_smem);
}

// The resident rank of a phrase given its key (a hashed key names the
// phrase's position in S), or ~0.
template <typename T>
__device__ __noinline__ u64 find_resident(const RoundArgs& a, const Key128& key) {
    const T* S = (const T*)a.S;
    const u64 len = key_len(key), pos = key.lo;
    return table_find(ContentTable{(Slot*)a.rtab, a.rtab_cap}, key, key_is_hashed(key), [&](u64 rank) {
        const u64 o = a.rrhs_off[rank];
        for (u64 j = 0; j < len; j++)
            if ((u32)S[pos + j] != a.rrhs[o + j]) return false;
        return true;
    });
}

// The phrase that a hashed key names (at pos) against the one at ref, kBatch
// symbols per round trip.
template <typename T, int kBatch>
__device__ __noinline__ bool same_content(const T* S, u64 pos, u64 len, u64 ref) {
    for (u64 j = 0; j < len; j += kBatch) {
        T x[kBatch], y[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; u++) {
            const bool in = j + u < len;
            x[u] = in ? S[ref + j + u] : (T)0;
            y[u] = in ? S[pos + j + u] : (T)0;
        }
#pragma unroll
        for (int u = 0; u < kBatch; u++)
            if (x[u] != y[u]) return false;
    }
    return true;
}

// The inline key of a phrase of len <= kInlineMax bytes at offset st of the
// 8-byte words s64: its bytes as one little-endian number B, B mod 2^60 (with
// the length above) in hi and B >> 60 in lo (the layout of key_inline for
// 8-bit symbols).
__device__ __forceinline__ Key128 byte_key_of(u64 b0, u64 b1, u32 len) {
    if (len < 8) {
        b0 &= (1ull << (8 * len)) - 1;
        b1 = 0;
    } else if (len < 16) {
        b1 &= (1ull << (8 * (len - 8))) - 1;
    }
    return Key128{(b0 >> 60) | (b1 << 4), (b0 & ((1ull << 60) - 1)) | ((u64)len << 60)};
}
__device__ __forceinline__ Key128 byte_key(const u64* s64, u32 st, u32 len) {
    const u32 sh = (st & 7) * 8;
    s64 += st >> 3;
    const u64 x0 = s64[0], x1 = s64[1], x2 = s64[2];
    return byte_key_of(sh ? (x0 >> sh) | (x1 << (64 - sh)) : x0, sh ? (x1 >> sh) | (x2 << (64 - sh)) : x1, len);
}

// Byte rounds: a phrase found or claimed enters the cache at its free place
// `cache` - 1 (0: none; then it is not short either), valid from a place
// after its first occurrence (at or before `first`) on.
template <int U, int W>
__device__ __forceinline__ void cache_put(u32 cache, const Key128& key, u32 len, u32 id, u32 F, u64 first) {
    ParseSmem<unsigned char, U, W>& sm = parse_smem<unsigned char, U, W>();
    if (cache == 0 || id >= (1u << 26)) return;
    const u64 ck = ((u64)len << 56) | (key.hi & ((1ull << (8 * len)) - 1));
    if (atomicCAS((unsigned long long*)&sm.ckey[cache - 1], (unsigned long long)kEmpty, (unsigned long long)ck) == kEmpty)
        *(volatile u64*)&sm.cval[cache - 1] = ((u64)(64 - __clzll((long long)first)) << 58) | ((u64)id << 32) | F;
}

// A phrase of more than kLongLen symbols at `pos`, by the whole warp: the
// fingerprint polynomial H (Eq. fast_hash) and the content comparisons of its
// hashed key are spread over the lanes.
template <typename T, int U, int W, bool kLive>
__device__ __noinline__ void parse_long(u64 pos, u64 len, u64 p) {
    ParseSmem<T, U, W>& sm = parse_smem<T, U, W>();
    const RoundArgs& a = *sm.args.all;
    const T* S = (const T*)a.S;
    const u32 lane = threadIdx.x & 31;
    auto& w = sm.w[threadIdx.x >> 5];
    if (len > kMaxPhraseLen) {
        if (lane == 0) set_error(a.ds, kErrPhraseLong);
        return;
    }
    const u64 H = warp_poly61([&](u64 j) -> u64 {
        if constexpr (sizeof(T) == 1) return sm.sF[S[pos + j]];
        else return ld_in<kLive>(a.Sf + pos + j);
    }, len, a.lh.c);
    const u32 F = finish_hash(a.lh, H);
    const Key128 key = key_hashed(H, len, pos);
    const ContentTable rt{(Slot*)a.rtab, a.rtab_cap};
    u64 r = ~0ull;
    if (rt.cap)
        r = table_find_warp(rt, key, [&](u64 rank) {
            const u64 o = a.rrhs_off[rank];
            return warp_equal([&](u64 j) { return (u32)S[pos + j]; }, [&](u64 j) { return a.rrhs[o + j]; }, len);
        });
    u64 pub = kNoPub;
    if (r == ~0ull) {
        ClaimSum sum{0, 0};
        pub = table_resolve_warp(sm.args.table, &sm.ids, sum, key, p, F, [&](u64 ref) {
            return warp_equal([&](u64 j) { return S[ref + j]; }, [&](u64 j) { return S[pos + j]; }, len);
        });
        __syncwarp();
        if (lane == 0) {
            w.claims += sum.count;
            w.claim_len += sum.len;
        }
        __syncwarp();
    }
    if (lane == 0) {
        if (r != ~0ull) emit_slow(a, p, (u32)r, F);
        else if (pub != kNoPub) emit_slow(a, p, a.id_base + (u32)pub, (u32)(pub >> 32));
    }
}

// The long path on the warp's queued phrases first .. first + take - 1 (at
// most 32): fingerprint, resident lookup, find or claim, and the symbol of
// T^{i+1}.  Not inlined, so that the loop over the units keeps its registers.
template <typename T, int U, int W, bool kLive>
__device__ __noinline__ void parse_queued(u32 first, u32 take) {
    ParseSmem<T, U, W>& sm = parse_smem<T, U, W>();
    const ParseArgs& a = sm.args;
    constexpr bool kByte = sizeof(T) == 1;
    const T* S = (const T*)a.S;
    const u32 lane = threadIdx.x & 31;
    auto& w = sm.w[threadIdx.x >> 5];
    const bool act = lane < take;
    ulonglong2 e = make_ulonglong2(0ull, 0ull);
    if (act) e = w.queue[first + lane];
    constexpr u64 kPosMask = (1ull << kPosBits) - 1;
    const u64 pos = e.x & kPosMask, p = e.y & kPosMask;
    const u32 plen = (u32)(e.x >> kPosBits) & 63u, home = (u32)(e.x >> (kPosBits + 6)) & 3u;
    Key128 k;
    u64 H = 0;
    bool res = a.rtab_cap != 0;  // a phrase with a symbol that is new in this build is no resident rule
    if constexpr (kByte) {
        // up to 16 bytes with three aligned 8-byte reads
        const u64 adr = reinterpret_cast<unsigned long long>(S + pos);
        const bool words = plen <= 16 && pos >= 8 && pos + 24 <= a.n;
        u64 b0 = 0, b1 = 0;
        if (words) {
            const u64* q = reinterpret_cast<const u64*>(adr & ~7ull);
            const u32 sh = (u32)(adr & 7) * 8;
            const u64 x0 = __ldg(q), x1 = __ldg(q + 1), x2 = __ldg(q + 2);
            b0 = sh ? (x0 >> sh) | (x1 << (64 - sh)) : x0;
            b1 = sh ? (x1 >> sh) | (x2 << (64 - sh)) : x1;
        } else if (plen <= 16) {
            for (u32 j = 0; j < plen; j++) {
                const u64 x = (u64)S[pos + j] << (8 * (j & 7));
                if (j < 8) b0 |= x; else b1 |= x;
            }
        }
        PolySum ps;
        for (u32 j = 0; j < plen;) {
            const u64 x = j < 8 ? b0 : b1;
            const u32 end = min(plen, j + 8);
            for (u32 sh = 0; j < end; j++, sh += 8) {
                const u32 v = plen <= 16 ? (u32)(x >> sh) & 0xFFu : (u32)S[pos + j];
                ps.add(sm.sF[v], sm.cpow[j]);
            }
            ps.fold();
        }
        H = ps.h;
        k = plen <= (u32)kInlineMax ? byte_key_of(b0, b1, plen) : key_hashed(H, plen, pos);
    } else {
        // four symbols from the last on at a time: H, and the packed symbols
        PackedSyms ps;
        PolySum poly;
        for (u32 j = plen; j > 0;) {
            const u32 m = min(j, 4u);
            u32 v[4], f[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                v[u] = f[u] = 0;
                if ((u32)u < m) {
                    v[u] = (u32)ld_in<kLive>(S + pos + j - 1 - u);
                    f[u] = ld_in<kLive>(a.Sf + pos + j - 1 - u);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; u++)
                if ((u32)u < m) {
                    res = res && v[u] < a.prev_base;
                    ps.push(v[u], a.sym_w);
                    poly.add(f[u], sm.cpow[j - 1 - u]);
                }
            poly.fold();
            j -= m;
        }
        H = poly.h;
        k = plen <= a.inline_most ? ps.key(plen) : key_hashed(H, plen, pos);
    }
    const u32 F = finish_hash(a.lh, H);
    u64 r = ~0ull;
    if (act && res) r = find_resident<T>(*a.all, k);
    u64 first_occ = r != ~0ull ? 0 : p;  // a bound of its first occurrence
    ClaimSum sum{0, 0};
    const u64 pub = table_resolve(a.table, &sm.ids, sum, act && r == ~0ull, home, k, p, F, first_occ, [&](u64 ref) {
        return same_content<T, kByte ? 1 : kCompareBatchR>(S, k.lo, key_len(k), ref);
    });
    const u32 count = __reduce_add_sync(0xffffffffu, sum.count), len = __reduce_add_sync(0xffffffffu, sum.len);
    if (lane == 0) {
        w.claims += count;
        w.claim_len += len;
    }
    if (act && (r != ~0ull || pub != kNoPub)) {
        const u32 id = r != ~0ull ? (u32)r : a.id_base + (u32)pub;
        if constexpr (kByte) {
            cache_put<U, W>((u32)(e.y >> kPosBits), k, plen, id, F, first_occ);
        }
        if (a.retired == 0 && p < a.T_cap) {
            __stcs(a.Tnext + p, id);
            __stcs(a.Fnext + p, F);
        } else {
            emit_slow(*a.all, p, id, F);
        }
    }
    __syncwarp();
}

// The first read for the phrases of a unit from q0 on: cache or home slot.
// What that does not answer joins the warp's nq queued phrases; stops when 32
// are queued.  `span`: q0 | (the unit's phrases) << 16.  Returns the next
// phrase, the queue's length (bits 10..17) and whether there was a long phrase
// (bit 18).  Not inlined, and without calls: this loop keeps every value in
// registers (inlined beside the long path it spilled: the byte round of
// 4 x 3.1 Gbp took 52.7 ms, now 37.1).  One phrase per thread at a time: with
// two in flight round 2 of the same took 45.2 ms (44.4), with four 52.2: the
// rounds with large tables are bound by random sectors, not by their latency.
template <typename T, int U, int W>
__device__ __noinline__ u32 parse_unit_find(u32 buf, u64 t0, u64 p0, u64 out, u32 span, u32 nq, bool direct) {
    using Smem = ParseSmem<T, U, W>;
    Smem& sm = parse_smem<T, U, W>();
    const ParseArgs& a = sm.args;
    constexpr bool kByte = Smem::kByte;
    const u32 lane = threadIdx.x & 31;
    typename Smem::Warp& w = sm.w[threadIdx.x >> 5];
    const T* sym = w.sym[buf];
    volatile u64* ckey = sm.ckey;
    volatile u64* cval = sm.cval;
    const u32 find_inline = a.find_inline, id_base = a.id_base;
    const int sym_w = (int)a.sym_w;
    Slot* const slots = a.table.slots;
    const u64 cap = a.table.cap;
    u32* Tn = a.Tnext + out;
    u32* Fn = a.Fnext + out;
    auto emit = [&](u32 q, u32 id, u32 F) {
        __stcs(Tn + q, id);
        __stcs(Fn + q, F);
    };
    constexpr u32 kDone = 3, kLong = 4;  // else the home state of a phrase to be queued
    const u32 cnt = span >> 16;
    u32 q0 = span & 0xFFFFu, longs = 0;
    for (; q0 < cnt && nq < 32; q0 += 32) {
        const u32 q = q0 + lane;
        u32 state = kDone, cache = 0, st = 0, len = 0;
        if (q < cnt) {
            st = w.start[q];
            len = w.start[q + 1] - st;
            state = len > (u32)kLongLen ? kLong : kHomeUnknown;
            if constexpr (kByte) {
                if (len <= 7 && direct) {
                    // the packed bytes of the phrase
                    const u64* s64 = reinterpret_cast<const u64*>(sym) + (st >> 3);
                    const u32 sh = (st & 7) * 8;
                    const u64 lo = s64[0], hi = s64[1];
                    const u64 v = sh ? (lo >> sh) | (hi << (64 - sh)) : lo;
                    const u64 k = ((u64)len << 56) | (v & ((1ull << (8 * len)) - 1));
                    u32 h = (u32)((k * 0x9E3779B97F4A7C15ull) >> (64 - Smem::kCacheBits));
                    for (int probe = 0; probe < kCacheProbes; probe++) {
                        const u64 ck = ckey[h];
                        if (ck == k) {
                            const u64 cv = cval[h];
                            // (not yet written, or first seen after this place: the long path)
                            if (cv != ~0ull && ((p0 + q) >> (cv >> 58)) != 0) {
                                state = kDone;
                                emit(q, (u32)(cv >> 32) & ((1u << 26) - 1), (u32)cv);
                            }
                            break;
                        }
                        if (ck == kEmpty) {
                            cache = h + 1;
                            break;
                        }
                        h = (h + 1) & (Smem::kCacheSlots - 1);
                    }
                }
            }
        }
        // the home slot: every phrase in rank rounds, in byte rounds when enough
        // lanes of the warp missed the cache
        auto look = [&]() {
            const Key128 key = kByte ? byte_key(reinterpret_cast<const u64*>(sym), st, len)
                                     : key_inline32(reinterpret_cast<const u32*>(sym) + st, len, sym_w);
            const Slot c = ld_slot_relaxed(&slots[key_home(key, cap)]);
            if (c.key.hi == key.hi && c.key.lo == key.lo && c.pub != kUnpublished && c.val <= p0 + q) {
                const u32 id = id_base + (u32)c.pub, F = (u32)(c.pub >> 32);
                state = kDone;
                emit(q, id, F);
                if constexpr (kByte) cache_put<U, W>(cache, key, len, id, F, c.val);
            } else if (c.key.hi == kEmptyHi) {
                state = kHomeEmpty;
            } else if (c.key.hi != key.hi) {
                state = kHomeOther;
            }
            // else: another key, one being written, or a first occurrence
            // that may be here: the long path reads the slot again
        };
        if constexpr (!kByte)
            if (state == kHomeUnknown && len <= find_inline && direct) look();
        unsigned m = __ballot_sync(0xffffffffu, state < kDone);
        if (kByte && __popc(m) >= kByteFind) {
            if (state == kHomeUnknown && len <= find_inline && direct) look();
            m = __ballot_sync(0xffffffffu, state < kDone);
        }
        if (state < kDone)
            w.queue[nq + __popc(m & ((1u << lane) - 1u))] =
                queue_entry(t0 + st, len, state, cache, p0 + q);
        nq += (u32)__popc(m);
        longs |= __ballot_sync(0xffffffffu, state == kLong);
        __syncwarp();
    }
    return min(q0, cnt) | (nq << 10) | ((longs ? 1u : 0u) << 18);
}

template <typename T, int U, int W, bool kLive = false>
__device__ __forceinline__ void body_parse(const RoundArgs& a, u64 nunits) {
    pdl_wait();
    using Smem = ParseSmem<T, U, W>;
    constexpr bool kByte = Smem::kByte;
    constexpr int kSP = Smem::kSP;
    constexpr int kWords = U / 32;  // break words of a unit
    constexpr int kBits = U / 32;   // positions per lane in the phrase list
    static_assert(kWords + kHalo / 32 <= 32 && kHalo % 32 == 0 && kBits <= 32, "a unit's break words fit one per lane");
    static_assert(kHalo > kLongLen, "a phrase that is not long lies in the staged symbols");
    Smem& sm = parse_smem<T, U, W>();
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    typename Smem::Warp& w = sm.w[warp];

    const T* S = (const T*)a.S;
    // After a planned round that outgrew its next sequence *d_n is the number of
    // symbols that there should have been.  Such a round is halted, but the first unit
    // is fetched before its status is known, so all that is read lies within the
    // buffers whatever the status.
    const u64 n = min(round_n(a), min(a.n_cap, nunits * (u64)U));
    const u64 nwords = (n + 31) / 32;  // words of the break bitmap
    nunits = min(nunits, (n + U - 1) / U);
    const u64 nr = a.rc->retired;
    u32 nq = 0;  // the warp's queued phrases
    // The warps of the grid take units in turn (rank rounds in stripes when
    // asked) and wait for no other: unit lt of the logical order.
    const u32 stripes = kByte ? 1u : a.stripes;
    const u32 nlog = (u32)stripe_tiles(nunits, stripes), step = gridDim.x * W;
    // A unit's symbols go to buffer b; its break words (one per lane) and first
    // phrase index to registers.
    u32 nx_bits = 0;
    u64 nx_p0 = 0;
    auto fetch = [&](u32 lt, u32 b) {
        const u64 unit = lt < nlog ? stripe_tile(lt, nunits, stripes) : ~0ull;
        if (unit < nunits) {
            const u64 f0 = unit * (u64)U;
            const u32 ns = (u32)(min(f0 + (u64)kSP, n) - f0);
            const T* src = S + f0;
            constexpr u32 PER = 16 / sizeof(T);
            const bool vec = (reinterpret_cast<unsigned long long>(src) & 15) == 0;
            for (u32 x = lane * PER; x < ns; x += 32 * PER) {
                if (x + PER <= ns && vec) {
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                     (u32)__cvta_generic_to_shared(&w.sym[b][x])),
                                 "l"(src + x)
                                 : "memory");
                } else {
                    T v[PER];
#pragma unroll
                    for (u32 e = 0; e < PER; e++) v[e] = x + e < ns ? src[x + e] : (T)0;
#pragma unroll
                    for (u32 e = 0; e < PER; e++) w.sym[b][x + e] = v[e];  // (kSP is a multiple of PER)
                }
            }
            const u64 gw = f0 / 32 + lane;
            nx_bits = (lane < kWords + kHalo / 32 && gw < nwords) ? ld_in<kLive>(a.brk + gw) : 0u;
            nx_p0 = a.tile_pfx[unit];
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    u32 lt = blockIdx.x * W + warp;
    fetch(lt, 0);  // (its reads run beside the set-up)
    if constexpr (kByte) {
        for (int x = threadIdx.x; x < 256; x += 32 * W) sm.sF[x] = a.Fprev[x];
        for (int x = threadIdx.x; x < Smem::kCacheSlots; x += 32 * W) {
            sm.ckey[x] = kEmpty;
            sm.cval[x] = ~0ull;
        }
    }
    if (threadIdx.x == 0) {
        ParseArgs& pa = sm.args;
        pa.S = a.S;
        pa.Sf = a.Sf;
        pa.Tnext = a.Tnext;
        pa.Fnext = a.Fnext;
        pa.n = n;
        pa.T_cap = a.T_cap;
        pa.retired = nr;
        pa.lh = a.lh;
        pa.table = RoundTable{(Slot*)a.tab, a.tab_cap, a.minpos, (ClaimRec*)a.crec, a.id_cap, a.id_chunk,
                              kLive ? a.tab_cap : kMaxProbes, a.ds};  // (a short round's table is never too full)
        pa.rtab_cap = a.rtab_cap;
        pa.all = &a;
        pa.sym_w = (u32)a.sym_w;
        pa.inline_most = (u32)inline_max(a.sym_w);
        pa.find_inline = a.rtab_cap ? 0u : pa.inline_most;  // phrases looked up in the table at once
        pa.id_base = a.id_base;
        pa.prev_base = a.prev_base;
    }
    if (threadIdx.x < (u32)kLongLen) sm.cpow[threadIdx.x] = powmod61(a.lh.c, threadIdx.x);
    if (threadIdx.x == 0) sm.ids = ClaimIds{0, 0, 0};
    if (lane == 0) {
        w.claims = w.claim_len = 0;
    }
    __syncthreads();

    for (u32 iter = 0;; lt += step, iter++) {
        const bool have = lt < nlog;  // past the last unit: the queue is emptied
        if (!have && nq == 0) break;
        // a round that has failed stops early
        if ((iter & 15) == 0) {
            u32 h = 0;
            if (lane == 0) {
                const DevStatus* before = a.ds_prev ? a.ds_prev : a.ds;
                const u32 h0 = vload(&a.ds->error), h1 = vload(&a.ds->overflow);
                const u32 h2 = vload(&before->error), h3 = vload(&before->overflow);
                h = h0 | h1 | h2 | h3;
            }
            if (__shfl_sync(0xffffffffu, h, 0)) break;
        }
        const u64 unit = have ? stripe_tile(lt, nunits, stripes) : ~0ull;
        const u32 bits = nx_bits;
        const u64 p0 = nx_p0;  // the unit's first phrase
        fetch(lt + step, (iter + 1) & 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const u64 t0 = unit * (u64)U;

        // 1. phrase starts of the unit, in order, kBits positions per lane
        u32 cnt = 0;
        u64 tail = 0;  // end of the last phrase
        if (unit < nunits) {  // (none in a gap of the striped order)
            const u32 nt = (u32)(min(t0 + (u64)U, n) - t0);
            u32 part = __shfl_sync(0xffffffffu, bits, (int)(lane * kBits / 32)) >> (lane * kBits % 32);
            if (kBits < 32) part &= (1u << (kBits & 31)) - 1u;
            const u32 x0 = lane * kBits;
            if (x0 >= nt) part = 0;
            else if (nt - x0 < (u32)kBits) part &= (1u << (nt - x0)) - 1u;
            u32 o = (u32)__popc(part);
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const u32 y = __shfl_up_sync(0xffffffffu, o, d);
                if (lane >= (u32)d) o += y;
            }
            cnt = __shfl_sync(0xffffffffu, o, 31);
            o -= (u32)__popc(part);
            if (cnt >= (u32)Smem::kStarts) {  // not reached: a phrase but a string's first has two symbols
                if (lane == 0) set_error(a.ds, kErrCapacity);
                cnt = part = 0;
            }
            for (; part; part &= part - 1) w.start[o++] = (unsigned short)(x0 + (u32)__ffs(part) - 1);
            // the first phrase start at or after the unit's end: in the break
            // words after the unit, else further on in the bitmap
            const u32 h0 = __shfl_sync(0xffffffffu, bits, kWords), h1 = __shfl_sync(0xffffffffu, bits, kWords + 1);
            if (nt < (u32)U) tail = nt;
            else if (h0) tail = (u64)U + (u32)__ffs(h0) - 1;
            else if (h1) tail = (u64)U + 32 + (u32)__ffs(h1) - 1;
            else {
                tail = n - t0;
                for (u64 gw = t0 / 32 + kWords + 2; gw < nwords; gw += 32) {
                    const u32 x = gw + lane < nwords ? ld_in<kLive>(a.brk + gw + lane) : 0u;
                    const unsigned m = __ballot_sync(0xffffffffu, x != 0);
                    if (m) {
                        const int l = __ffs(m) - 1;
                        tail = (gw + (u64)l) * 32 + (u32)__ffs(__shfl_sync(0xffffffffu, x, l)) - 1 - t0;
                        break;
                    }
                }
            }
            if (lane == 0) w.start[cnt] = (unsigned short)min(tail, (u64)0xFFFF);
        }
        __syncwarp();

        // 2. lookups: what the cache or the home slot does not answer is queued
        //    (with all that the long path needs, so the queue outlives the
        //    unit), and whenever 32 phrases are queued the warp runs the long
        //    path on them.
        // Where the unit's phrases go in T^{i+1}; a unit in which a string
        // retires (or that does not fit) leaves all of them to the long path,
        // which looks each place up.
        u64 out = p0;
        bool direct = true;
        if (nr) {
            const u64 r0 = retired_before(a, p0);
            direct = r0 == nr || a.R_phr[r0] >= p0 + cnt;
            out -= r0;
        }
        direct = direct && out + cnt <= a.T_cap;
        bool longs = false;
        for (u32 q0 = 0;;) {
            if (q0 < cnt) {
                const u32 r = parse_unit_find<T, U, W>(iter & 1, t0, p0, out, q0 | (cnt << 16), nq, direct);
                q0 = r & 0x3FFu;
                nq = (r >> 10) & 0xFFu;
                longs = longs || (r >> 18) != 0;
            }
            if (nq < 32 && (have || nq == 0)) break;  // (the whole unit has been looked at)
            const u32 take = min(nq, 32u);
            nq -= take;
            parse_queued<T, U, W, kLive>(nq, take);
        }

        // 3. long phrases, one at a time by the whole warp
        if (longs) {
            for (u32 q0 = 0; q0 < cnt; q0 += 32) {
                const u32 q = q0 + lane;
                u32 m = __ballot_sync(0xffffffffu, q < cnt && w.start[q + 1] - w.start[q] > kLongLen);
                for (; m; m &= m - 1) {
                    const u32 x = q0 + (u32)__ffs(m) - 1;
                    const u64 st = w.start[x], en = x + 1 < cnt ? (u64)w.start[x + 1] : tail;
                    parse_long<T, U, W, kLive>(t0 + st, en - st, p0 + x);
                }
            }
        }
        __syncwarp();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (lane == 0 && w.claims) {
        atomicAdd(&a.ds->claims, w.claims);
        atomicAdd(&a.ds->claim_len, w.claim_len);
    }
}

// Per block step of k_breaks: the string that holds its first position.
__device__ __forceinline__ void body_tile_strings(const RoundArgs& a, u64 tiles) {
    pdl_wait();
    const u64 n = round_n(a);
    const u32 k = round_k(a);
    const u64 nt = (n + a.tp - 1) / a.tp;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.d_tiles = nt;
        if (a.ds_prev && (vload(&a.ds_prev->error) != 0 || vload(&a.ds_prev->overflow) != 0))
            set_error(a.ds, kErrHalted);
        else if (nt > tiles)
            set_error(a.ds, kErrCapacity);
    }
    if (round_halted(a)) return;
    const u64 steps = (min(tiles * a.tp, n) + kBrkSpan - 1) / kBrkSpan;
    if (a.step_str != nullptr)
        for (u64 t = blockIdx.x * (u64)blockDim.x + threadIdx.x; t < steps; t += (u64)gridDim.x * blockDim.x)
            a.step_str[t] = string_of<false>(a.soff, k, t * kBrkSpan);
    // bitmap of string starts (and of n), zeroed by the host
    for (u64 j = blockIdx.x * (u64)blockDim.x + threadIdx.x; j <= k; j += (u64)gridDim.x * blockDim.x) {
        const u64 s0 = __ldg(a.soff + j);
        if ((s0 >> 5) < a.sbm_words) atomicOr(a.sbm + (s0 >> 5), 1u << (s0 & 31));
    }
}

// --------------------------------------------------------------------------
// k_strings: per-string phrase ranges, retirement, next offsets (one block)
// --------------------------------------------------------------------------

// The first phrase of string j of k, and whether the string has no other.
__device__ __forceinline__ bool string_retires(const RoundArgs& a, u32 j, u32 k, u64 P, u64& first) {
    auto index_of = [&](u64 ok) { return a.tile_pfx[ok / a.tp] + ok % a.tp; };
    first = index_of(a.string_first[j]);
    return ((j + 1 < k) ? index_of(a.string_first[j + 1]) : P) - first == 1;
}

// Strings lo .. hi - 1 of the round's k, by one block; `carry`: the strings before them
// that retire.  Returns those and its own.
__device__ __forceinline__ u64 strings_range(const RoundArgs& a, u64 P, u32 k, u32 lo, u32 hi, u64 carry) {
    for (u32 j0 = lo; j0 < hi; j0 += blockDim.x) {
        const u32 j = j0 + threadIdx.x;
        u64 first = 0;
        const bool retire = j < hi && string_retires(a, j, k, P, first);
        u64 tot;
        const u64 rb = block_excl_scan(retire ? 1ull : 0ull, tot) + carry;
        if (j < hi) {
            if (retire) {
                a.R_phr[rb] = first;
                a.R_sid[rb] = a.sid[j];
            } else {
                const u64 s0 = first - rb;
                a.soff_next[j - rb] = s0;
                a.sid_next[j - rb] = a.sid[j];
                if (a.sbm_next != nullptr && (s0 >> 5) < a.sbm_next_words)
                    atomicOr(a.sbm_next + (s0 >> 5), 1u << (s0 & 31));
            }
        }
        carry += tot;
    }
    return carry;
}

// After all strings (one thread): the end of the next sequence and the round's counts;
// `carry`: the strings that retire.
__device__ __forceinline__ void strings_end(const RoundArgs& a, u64 P, u32 k, u64 carry) {
    const u64 s0 = P - carry;
    a.soff_next[k - carry] = s0;
    if (a.sbm_next != nullptr && (s0 >> 5) < a.sbm_next_words) atomicOr(a.sbm_next + (s0 >> 5), 1u << (s0 & 31));
    a.rc->phrases = P;
    a.rc->retired = carry;
    a.rc->k_next = k - carry;
    a.rc->n_next = P - carry;
}

__device__ __forceinline__ void body_strings(const RoundArgs& a) {
    pdl_wait();
    if (round_halted(a)) return;
    const u64 P = *a.total;
    const u32 k = round_k(a);
    const u64 retired = strings_range(a, P, k, 0, k, 0);
    if (threadIdx.x == 0) strings_end(a, P, k, retired);
}

// --------------------------------------------------------------------------
// first-occurrence naming over the claimed entries
// --------------------------------------------------------------------------

// Number of new rules of the round, bounded by the naming arrays.
__device__ __forceinline__ u64 round_gnew(const RoundArgs& a) {
    const u64 g = *a.d_gnew;
    if (g > a.r_cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_error(a.ds, kErrCapacity);
        return a.r_cap;
    }
    return g;
}

// Whether the new rules fit the level's arrays.
__device__ __forceinline__ bool rules_fit(const RoundArgs& a) {
    if (a.g_base + min(*a.d_gnew, a.r_cap) <= a.cap_g && a.G_base + *a.d_Gnew <= a.cap_G) return true;
    if (blockIdx.x == 0 && threadIdx.x == 0) set_error(a.ds, kErrCapacity);
    return false;
}

// Mark the first occurrence of every new phrase in a bitmap over phrase
// indices.  Claims are numbered about in the order of their positions, so the
// marks of a warp fall close together.
__device__ __forceinline__ void body_mark(const RoundArgs& a) {
    pdl_wait();
    if (round_halted(a)) return;
    const u64 ids = min(*a.d_ids, a.id_cap);
    const u64 phrases = a.first_words * 32;  // phrase indices the bitmap covers
    for (u64 c = blockIdx.x * (u64)blockDim.x + threadIdx.x; c < ids; c += (u64)gridDim.x * blockDim.x) {
        const u64 m = a.minpos[c];
        if (m == ~0ull) continue;  // a number that no claim used
        if (m >= phrases) {
            set_error(a.ds, kErrCapacity);
            continue;
        }
        atomicOr(&a.first[m >> 5].x, 1u << (m & 31));
    }
}

constexpr int kPopThreads = 512;
constexpr int kPopItems = 8;  // pairs of words of a thread, 32 pairs apart
constexpr int kPopTile = kPopThreads * kPopItems * 2;

// Exclusive prefix of the popcounts of the bitmap words (single pass).  Word
// and prefix lie side by side, so that k_rank reads both with one sector.  Lanes take
// neighbouring pairs of words (see k_rule_offs): 113 M
// words 0.83 ms before, 0.51 now.
__global__ void __launch_bounds__(kPopThreads) k_popscan(const RoundArgs a) {
    __shared__ u32 s_sum[kPopThreads / 32];
    pdl_wait();
    const u64 tile = dynamic_tile(a.ctr, a.ctr_base);
    const u64 nw = min(a.first_words, (*a.total + 31) / 32);
    if (tile > 0 && tile * (u64)kPopTile >= nw) return;  // beyond the count read on the device
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u64 w0 = tile * (u64)kPopTile + (u64)warp * (64 * kPopItems) + 2 * lane;
    const bool pairs = (reinterpret_cast<unsigned long long>(a.first) & 15) == 0;
    u32 x[kPopItems], y[kPopItems], at[kPopItems];
#pragma unroll
    for (int i = 0; i < kPopItems; i++) {
        const u64 w = w0 + 64 * i;
        if (pairs && w + 2 <= nw) {
            const uint4 v = *reinterpret_cast<const uint4*>(a.first + w);
            x[i] = v.x, y[i] = v.z;
        } else {
            x[i] = w < nw ? a.first[w].x : 0u;
            y[i] = w + 1 < nw ? a.first[w + 1].x : 0u;
        }
    }
    u32 sum = 0;
#pragma unroll
    for (int i = 0; i < kPopItems; i++) {
        const u32 c = (u32)(__popc(x[i]) + __popc(y[i]));
        u32 e = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u32 z = __shfl_up_sync(0xffffffffu, e, o);
            if (lane >= (u32)o) e += z;
        }
        at[i] = sum + e - c;
        sum += __shfl_sync(0xffffffffu, e, 31);
    }
    if (lane == 0) s_sum[warp] = sum;
    __syncthreads();
    u64 before = 0, tot = 0;
#pragma unroll
    for (u32 w = 0; w < kPopThreads / 32; w++) {
        before += w < warp ? s_sum[w] : 0;
        tot += s_sum[w];
    }
    u64 agg[1] = {tot}, excl[1];
    block_lookback<1>((LBSlot<1>*)a.lb1, tile, a.epoch, agg, excl, a.ds);
    before += excl[0];
#pragma unroll
    for (int i = 0; i < kPopItems; i++) {
        const u64 w = w0 + 64 * i;
        const u32 e0 = (u32)before + at[i], e1 = e0 + (u32)__popc(x[i]);
        if (pairs && w + 2 <= nw) {
            *reinterpret_cast<uint4*>(a.first + w) = make_uint4(x[i], e0, y[i], e1);
        } else {
            if (w < nw) a.first[w].y = e0;
            if (w + 1 < nw) a.first[w + 1].y = e1;
        }
    }
}

// Rank of every new phrase: the marks before its first occurrence.  Its
// record moves to its rank's place.
__device__ __forceinline__ void body_rank(const RoundArgs& a) {
    pdl_wait();
    if (round_halted(a)) return;
    const u64 g_new = round_gnew(a), ids = min(*a.d_ids, a.id_cap);
    const ClaimRec* crec = (const ClaimRec*)a.crec;
    ClaimRec* rrec = (ClaimRec*)a.rrec;
    for (u64 c = blockIdx.x * (u64)blockDim.x + threadIdx.x; c < ids; c += (u64)gridDim.x * blockDim.x) {
        const u64 m = a.minpos[c];
        const ClaimRec rec = crec[c];
        if (m >= a.first_words * 32) continue;  // no claim (or k_mark flagged it)
        const uint2 f = a.first[m >> 5];
        const u64 r = f.y + __popc(f.x & ((1u << (m & 31)) - 1u));
        if (r >= g_new) { set_error(a.ds, kErrCapacity); continue; }
        a.rank_of[c] = (u32)(a.g_base + r);
        rrec[r] = rec;
    }
}

constexpr int kRoThreads = 512;
constexpr int kRoItems = 16;  // rules of a thread, 32 apart
constexpr int kRoTile = kRoThreads * kRoItems;

// Right-hand-side offsets of the new rules, straight from their keys' lengths
// (single pass).  The lanes of a warp take neighbouring records, whose sectors are read
// as whole lines; with a thread's records next to each other (and its lanes 256 bytes
// apart) they were read one by one at the rate of random sectors.  14.6 M rules: 0.36 ms so
// in tiles of 2048, 0.30 with neighbouring lanes, 0.20 in tiles of 8192.
__global__ void __launch_bounds__(kRoThreads) k_rule_offs(const RoundArgs a) {
    __shared__ u64 s_sum[kRoThreads / 32];
    pdl_wait();
    const u64 tile = dynamic_tile(a.ctr, a.ctr_base);
    if (!rules_fit(a)) return;  // the same answer for every block
    const u64 n = min(*a.d_gnew, a.r_cap);
    if (tile * (u64)kRoTile >= n && tile > 0) return;
    const ClaimRec* rec = (const ClaimRec*)a.rrec;
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u64 r0 = tile * (u64)kRoTile + warp * (32 * kRoItems) + lane;
    u32 len[kRoItems];
    u32 most = 0;
#pragma unroll
    for (int i = 0; i < kRoItems; i++) {
        // the length is in the key's high half
        const Key128 k{0, r0 + 32 * i < n ? rec[r0 + 32 * i].key.hi : 0ull};
        len[i] = (u32)key_len(k);
    }
#pragma unroll
    for (int i = 0; i < kRoItems; i++) most |= len[i];
    // places within the warp: in 32 bits unless a length alone takes more than 20
    u64 at[kRoItems], sum = 0;
    const bool wide = __any_sync(0xffffffffu, most >> 20) != 0;
#pragma unroll
    for (int i = 0; i < kRoItems; i++) {
        if (wide) {
            u64 x = len[i];
            for (int o = 1; o < 32; o <<= 1) {
                const u64 y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= (u32)o) x += y;
            }
            at[i] = sum + x - len[i];
            sum += __shfl_sync(0xffffffffu, x, 31);
        } else {
            u32 x = len[i];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u32 y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= (u32)o) x += y;
            }
            at[i] = sum + (x - len[i]);
            sum += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    if (lane == 0) s_sum[warp] = sum;
    __syncthreads();
    u64 before = 0, tot = 0;
#pragma unroll
    for (u32 w = 0; w < kRoThreads / 32; w++) {
        before += w < warp ? s_sum[w] : 0;
        tot += s_sum[w];
    }
    u64 agg[1] = {tot}, excl[1];
    block_lookback<1>((LBSlot<1>*)a.lb1, tile, a.epoch, agg, excl, a.ds);
    before += excl[0] + a.G_base;
    u64* off = a.rhs_off + a.g_base;
#pragma unroll
    for (int i = 0; i < kRoItems; i++)
        if (r0 + 32 * i < n) off[r0 + 32 * i] = before + at[i];
    if ((tile + 1) * (u64)kRoTile >= n && threadIdx.x == 0) off[n] = a.G_base + excl[0] + tot;
}

// The rank of a symbol of T^i (ids; bytes name themselves).
template <typename T, bool kLive>
__device__ __forceinline__ u32 sym_rank(const RoundArgs& a, u32 v) {
    if constexpr (sizeof(T) == 1) return v;
    return v < a.prev_base ? v : ld_in<kLive>(a.rank_prev + (v - a.prev_base));
}

// The new rules first, first + stride, ... below `end` of this thread (in rank
// order; a warp's 32 threads take consecutive ones): right-hand sides (ids
// translated to ranks) and F^i; their offsets are written.
template <typename T, bool kLive = false>
__device__ __forceinline__ void rules_range(const RoundArgs& a, u64 first, u64 stride, u64 end) {
    const T* S = (const T*)a.S;
    const ContentTable rw{(Slot*)a.rtab_w, a.rtab_w_cap};
    // whole warps step through the ranks, so that a warp can take its long
    // rules (more than kLongLen symbols) together after its short ones
    const u32 lane = threadIdx.x & 31;
    const ClaimRec* rec = (const ClaimRec*)a.rrec;
    for (u64 r0 = first - lane; r0 < end; r0 += stride) {
        const u64 r = r0 + lane;
        bool longr = false;
        if (r < end) {
            const Key128 k = rec[r].key;
            const u64 len = key_len(k);
            const bool hashed = key_is_hashed(k);
            const u64 rank = a.g_base + r;
            const u64 off = a.rhs_off[rank];
            a.F[rank] = rec[r].fp;
            if (len > (u64)kLongLen) {
                longr = true;
            } else {
                // four symbols at a time: their reads (and the translation's) are issued together
                for (u64 j = 0; j < len; j += 4) {
                    u32 v[4];
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        v[u] = j + u < len ? (hashed ? (u32)S[k.lo + j + u] : key_sym(k, j + u, a.sym_w)) : 0u;
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (j + u < len) v[u] = sym_rank<T, kLive>(a, v[u]);
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (j + u < len) a.rhs[off + j + u] = v[u];
                }
                if (rw.cap) {
                    auto get = [&](u64 j) -> u32 { return a.rhs[off + j]; };
                    const int w = sizeof(T) == 1 ? 8 : kRankBits;
                    u64 H = 0;
                    if (len > inline_max(w))
                        for (u64 j = len; j-- > 0;) H = addmod61(mulmod61(H, a.lh.c), (u64)ld_in<kLive>(a.Fprev + get(j)));
                    table_put(rw, rule_key(get, len, w, H, rank), rank, a.ds);
                }
            }
        }
        // long rules (hashed keys: the content is read at the first occurrence
        // k.lo), one at a time by the whole warp
        unsigned m = __ballot_sync(0xffffffffu, longr);
        while (m) {
            const u64 rr = r0 + (u64)(__ffs(m) - 1);
            m &= m - 1;
            const Key128 k = rec[rr].key;
            const u64 len = key_len(k);
            const u64 off = a.rhs_off[a.g_base + rr];
            // (eight symbols a lane at a time: the N-runs of 4 x 3.1 Gbp took 1.66 ms one by one, 0.46 so)
            for (u64 j0 = lane; j0 < len; j0 += 256) {
                u32 v[8];
#pragma unroll
                for (int u = 0; u < 8; u++) v[u] = j0 + 32 * u < len ? (u32)S[k.lo + j0 + 32 * u] : 0u;
#pragma unroll
                for (int u = 0; u < 8; u++)
                    if (j0 + 32 * u < len) v[u] = sym_rank<T, kLive>(a, v[u]);
#pragma unroll
                for (int u = 0; u < 8; u++)
                    if (j0 + 32 * u < len) a.rhs[off + j0 + 32 * u] = v[u];
            }
            if (rw.cap) {
                __syncwarp();
                const u64 H = warp_poly61([&](u64 j) -> u64 { return ld_in<kLive>(a.Fprev + a.rhs[off + j]); }, len, a.lh.c);
                if (lane == 0) table_put(rw, key_hashed(H, len, a.g_base + rr), a.g_base + rr, a.ds);
            }
        }
    }
}

// The new rules of level i in rank order: right-hand sides (ids translated to
// ranks) and F^i.  When the grammar keeps a table of its rules, the new rules
// enter it.  The roots of the retired strings get their ranks.
template <typename T>
__device__ __forceinline__ void body_rules(const RoundArgs& a) {
    pdl_wait();
    if (round_halted(a)) return;
    const u64 g_new = round_gnew(a);
    if (!rules_fit(a)) return;
    for (u64 x = blockIdx.x * (u64)blockDim.x + threadIdx.x; x < a.rc->retired; x += (u64)gridDim.x * blockDim.x) {
        const u32 id = a.c_rank[a.R_sid[x]];
        if (id < a.id_base) continue;
        if (id - a.id_base < a.id_cap) a.c_rank[a.R_sid[x]] = a.rank_of[id - a.id_base];
        else set_error(a.ds, kErrCapacity);
    }
    rules_range<T>(a, blockIdx.x * (u64)blockDim.x + threadIdx.x, (u64)gridDim.x * blockDim.x, g_new);
}

// --------------------------------------------------------------------------
// round 0 helpers: strings of length one, and gathering the active strings
// --------------------------------------------------------------------------

__global__ void k_level0(const unsigned char* __restrict__ data, const u64* __restrict__ pos,
                         const u32* __restrict__ ids, u32 cnt, u32* c_level, u32* c_rank) {
    pdl_wait();
    const u32 x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < cnt) {
        c_level[ids[x]] = 0;
        c_rank[ids[x]] = data[pos[x]];
    }
}

__global__ void k_gather_strings(const unsigned char* __restrict__ data, const u64* __restrict__ src_off,
                                 const u64* __restrict__ dst_off, u32 k, unsigned char* __restrict__ out) {
    pdl_wait();
    for (u32 j = blockIdx.x; j < k; j += gridDim.x) {
        const u64 s = src_off[j], d = dst_off[j], len = dst_off[j + 1] - dst_off[j];
        for (u64 x = threadIdx.x; x < len; x += blockDim.x) out[d + x] = data[s + x];
    }
}

// --------------------------------------------------------------------------
// host launchers
// --------------------------------------------------------------------------

// --------------------------------------------------------------------------
// the round's kernels, and the short rounds' cooperative kernels
// --------------------------------------------------------------------------

template <typename T>
// Blocks per SM: six in the byte round (10.0 ms for 12.4 GB; 10.2 with five, 10.5 with
// four), four over ranks, whose steps read four times as much (3.7 ms for 3.6 G
// symbols; 4.4 with three, 4.3 with five).
__global__ void __launch_bounds__(kBrkThreads, sizeof(T) == 1 ? 6 : 4) k_breaks(const RoundArgs a, u64 nblocks) { body_breaks<T>(a, nblocks); }
template <typename T, int U>
__global__ void __launch_bounds__(32 * parse_warps<T>, parse_blocks<parse_warps<T>>)
    k_parse(const __grid_constant__ RoundArgs a, u64 nunits) {
    body_parse<T, U, parse_warps<T>>(a, nunits);
}
__global__ void k_tile_strings(const RoundArgs a, u64 tiles) { body_tile_strings(a, tiles); }
__global__ void __launch_bounds__(1024) k_strings(const RoundArgs a) { body_strings(a); }
__global__ void k_mark(const RoundArgs a) { body_mark(a); }
__global__ void k_rank(const RoundArgs a) { body_rank(a); }
template <typename T>
__global__ void k_rules(const RoundArgs a) { body_rules<T>(a); }

// --------------------------------------------------------------------------
// the short rounds: all that are left of a build in two launches
// --------------------------------------------------------------------------
//
// Once a round has at most kTailSymbols symbols, it and every round after it
// run in one cooperative launch for their phrases and parses (k_parse_small)
// and one for their naming (k_naming_small): no later round reads a round's
// ranks (the sequences hold ids), so the naming of all of them can wait.  The
// last rounds, of at most kSoloSymbols symbols, are one block's (solo_rounds).
// What bounds such rounds is latency: before, each took two cooperative
// launches of its own with 3 and 4 grid barriers (55-95 us a round; a string of
// 20 kB has 10 rounds and nothing else); now a round has two barriers and all
// namings share four.  Their buffers need no plan and cannot be outgrown: a round
// of n symbols in k strings has at most (n + k) / 2 phrases.  (The levels' arrays, which
// the grammar keeps, may be planned smaller.)
// Why 524288: six builds of 12 MB into a growing grammar take 8.66 ms when the
// short rounds begin at 131072 symbols, 8.27 at 262144, 7.94 at 524288 and 7.82 at
// 1048576; a build of 8 x 1 MB 947, 948, 917 and 916 us; the larger builds do not
// tell them apart.  The buffers, some 200 bytes a symbol, grow with it.

constexpr int kSmallThreads = kParseThreads;
static_assert(kSmallThreads == kBrkThreads, "one block shape");

// Exclusive prefix of get(0 .. n) by one block: put(i, prefix) for every i;
// returns the sum (every thread).
constexpr int kSmallItems = 4;
template <typename Get, typename Put>
__device__ __forceinline__ u64 block_scan_small(Get get, u64 n, Put put) {
    u64 carry = 0;
    for (u64 base = 0; base < n; base += (u64)kSmallThreads * kSmallItems) {
        const u64 p0 = base + (u64)threadIdx.x * kSmallItems;
        u32 v[kSmallItems];
        u64 sum = 0;
#pragma unroll
        for (int i = 0; i < kSmallItems; i++) {
            v[i] = p0 + i < n ? get(p0 + i) : 0u;
            sum += v[i];
        }
        u64 tot;
        u64 e = block_excl_scan(sum, tot) + carry;
#pragma unroll
        for (int i = 0; i < kSmallItems; i++) {
            if (p0 + i < n) put(p0 + i, e);
            e += v[i];
        }
        carry += tot;
    }
    __syncthreads();
    return carry;
}

// The rounds of at most kSoloSymbols symbols, by block 0 alone with everything
// in its shared memory (the last 7 or 8 rounds of a build; through global
// memory and the round's general steps each took about 25 us of round trips).
// Phrases are compared by content in a small table, and numbered in the order
// of their first occurrences, so a claim's number is its rank already.
constexpr int kSoloWords = (int)kSoloSymbols / 32;
constexpr int kSoloStrings = (int)kSoloSymbols / 2;                 // two symbols each, at least
constexpr int kSoloPhrases = ((int)kSoloSymbols + kSoloStrings) / 2;
constexpr int kSoloSlots = 2048;
static_assert(kSoloWords == 32, "a warp takes a word per lane");

struct SoloSmem {
    u32 T[2][kSoloSymbols], F[2][kSoloSymbols];  // the round's sequence and the next
    u32 sid[2][kSoloStrings];
    unsigned short soff[2][kSoloStrings + 1];
    unsigned short sfirst[kSoloStrings + 1];     // first phrase of each string
    unsigned short start[kSoloPhrases + 1];      // of each phrase
    unsigned short slot_of[kSoloPhrases];
    u32 pF[kSoloPhrases];                        // its fingerprint
    u32 slot[kSoloSlots];                        // a phrase with the slot's content (~0: none), later its id
    u32 first[kSoloSlots];                       // the first such phrase
    u32 st[kSoloWords], gt[kSoloWords], lt[kSoloWords], stop[kSoloWords], bits[kSoloWords], pre[kSoloWords];
    u32 ret[kSoloWords], rpre[kSoloWords];       // phrases that are whole strings, and how many before each word
    u32 phrases;
};

template <bool kByte>
__device__ __noinline__ void solo_rounds(const TailArgs& t, u32 r) {
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    SoloSmem& sm = *reinterpret_cast<SoloSmem*>(dyn_smem);
    const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr u32 NT = kSmallThreads, NW = NT / 32;
    if (round_halted(t.r[r])) return;
    u32 n, k;
    {
        const RoundArgs& a = t.r[r];
        n = (u32)round_n(a);
        k = round_k(a);
        if (n > min(a.n_cap, a.tiles_bound * a.tp) || k > (u32)kSoloStrings) {  // more than the buffers were sized for
            if (tid == 0) set_error(a.ds, kErrCapacity);
            return;
        }
        for (u32 x = tid; x < n; x += NT) {
            if (kByte && r == 0) {
                const u32 s = ((const unsigned char*)a.S)[x];
                sm.T[0][x] = s;
                sm.F[0][x] = a.Fprev[s];
            } else {
                sm.T[0][x] = ((const u32*)a.S)[x];
                sm.F[0][x] = a.Sf[x];
            }
        }
        for (u32 j = tid; j <= k; j += NT) sm.soff[0][j] = (unsigned short)a.soff[j];
        for (u32 j = tid; j < k; j += NT) sm.sid[0][j] = a.sid[j];
    }
    for (u32 cur = 0; r < t.rounds && k > 0; r++, cur ^= 1) {
        const RoundArgs& a = t.r[r];
        const u32* T = sm.T[cur];
        const u32* F = sm.F[cur];
        const unsigned short* soff = sm.soff[cur];
        const u32 nw = (n + 31) / 32;
        for (u32 x = tid; x < (u32)kSoloSlots; x += NT) sm.slot[x] = sm.first[x] = ~0u;
        if (tid < (u32)kSoloWords) sm.st[tid] = sm.ret[tid] = 0;
        __syncthreads();
        // string starts (and the end of the sequence, when a word holds it)
        for (u32 j = tid; j <= k; j += NT)
            if (soff[j] < kSoloSymbols) atomicOr(&sm.st[soff[j] >> 5], 1u << (soff[j] & 31));
        __syncthreads();
        // right neighbour larger, smaller, or in no string (see k_breaks)
        for (u32 w = warp; w < nw; w += NW) {
            const u32 x = w * 32 + lane, x1 = x + 1;
            const bool end = x1 >= n || ((sm.st[x1 >> 5] >> (x1 & 31)) & 1u);
            const u32 f0 = x < n ? F[x] : 0u, f1 = x1 < n ? F[x1] : 0u;
            const u32 g = __ballot_sync(0xffffffffu, !end && f1 > f0), l = __ballot_sync(0xffffffffu, !end && f1 < f0);
            const u32 s = __ballot_sync(0xffffffffu, end);
            if (lane == 0) sm.gt[w] = g, sm.lt[w] = l, sm.stop[w] = s;
        }
        __syncthreads();
        if (warp == 0) {
            // one word per lane: types, breaks and the phrases before the word
            const u32 g = lane < nw ? sm.gt[lane] : 0u, l = lane < nw ? sm.lt[lane] : 0u;
            const u32 dec = lane < nw ? g | l | sm.stop[lane] : ~0u;
            u32 s = spread_down(g, ~dec);
            const unsigned decided = __ballot_sync(0xffffffffu, dec != 0);
            const u32 later = lane < 31 ? decided >> (lane + 1) : 0u;
            // is the first position of the next decided word of type S?
            const u32 from = later ? lane + (u32)__ffs(later) : lane;
            const u32 next_s = __shfl_sync(0xffffffffu, s & 1u, (int)from);
            if (!(dec >> 31) && later && next_s) {
                const int hi = 31 - __clz(dec | 1u);
                s |= dec == 0 ? ~0u : ~((2u << hi) - 1u);
            }
            const u32 lp = __shfl_up_sync(0xffffffffu, l, 1);
            u32 b = sm.st[lane] | (((l << 1) | (lane ? lp >> 31 : 0u)) & s);
            if (lane * 32 >= n) b = 0;
            else if (n - lane * 32 < 32) b &= (1u << (n - lane * 32)) - 1u;
            u32 o = (u32)__popc(b);
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const u32 y = __shfl_up_sync(0xffffffffu, o, d);
                if (lane >= (u32)d) o += y;
            }
            sm.bits[lane] = b;
            sm.pre[lane] = o - (u32)__popc(b);
            if (lane == 31) {
                sm.phrases = o;
                if (o <= (u32)kSoloPhrases) sm.start[o] = (unsigned short)n;
            }
        }
        __syncthreads();
        const u32 P = sm.phrases;
        if (P > (u32)kSoloPhrases) {  // not reached: a phrase but a string's first has two symbols
            if (tid == 0) set_error(a.ds, kErrCapacity);
            return;
        }
        for (u32 w = warp; w < nw; w += NW) {
            const u32 b = sm.bits[w];
            if ((b >> lane) & 1u)
                sm.start[sm.pre[w] + __popc(b & ((1u << lane) - 1u))] = (unsigned short)(w * 32 + lane);
        }
        for (u32 j = tid; j < k; j += NT) {
            const u32 x = soff[j];
            sm.sfirst[j] = (unsigned short)(sm.pre[x >> 5] + __popc(sm.bits[x >> 5] & ((1u << (x & 31)) - 1u)));
        }
        if (tid == 0) sm.sfirst[k] = (unsigned short)P;
        __syncthreads();
        // the strings that become one phrase, and the others' places
        constexpr u32 kPer = kSoloStrings / NT;
        static_assert(kPer * NT == kSoloStrings, "strings per thread");
        u32 one = 0;
#pragma unroll
        for (u32 i = 0; i < kPer; i++) {
            const u32 j = tid * kPer + i;
            if (j < k && sm.sfirst[j + 1] - sm.sfirst[j] == 1) one |= 1u << i;
        }
        u64 retired;
        u32 rb = (u32)block_excl_scan((u64)__popc(one), retired);
#pragma unroll
        for (u32 i = 0; i < kPer; i++) {
            const u32 j = tid * kPer + i;
            if (j >= k) continue;
            const u32 q = sm.sfirst[j];
            if ((one >> i) & 1u) {
                a.R_phr[rb] = q;
                a.R_sid[rb] = sm.sid[cur][j];
                atomicOr(&sm.ret[q >> 5], 1u << (q & 31));
                rb++;
            } else {
                sm.soff[cur ^ 1][j - rb] = (unsigned short)(q - rb);
                sm.sid[cur ^ 1][j - rb] = sm.sid[cur][j];
            }
        }
        const u32 k1 = k - (u32)retired, n1 = P - (u32)retired;
        if (tid == 0) sm.soff[cur ^ 1][k1] = (unsigned short)n1;
        // fingerprints, and equal phrases to one slot
        auto same = [&](u32 q0, u32 q1) {
            const u32 s0 = sm.start[q0], s1 = sm.start[q1], len = sm.start[q0 + 1] - s0;
            if (sm.start[q1 + 1] - s1 != len) return false;
            for (u32 j = 0; j < len; j++)
                if (T[s0 + j] != T[s1 + j]) return false;
            return true;
        };
        auto poly = [&](u32 q) -> u64 {
            u64 H = 0;
            for (u32 x = sm.start[q + 1]; x-- > sm.start[q];) H = addmod61(mulmod61(H, a.lh.c), (u64)F[x]);
            return H;
        };
        for (u32 q = tid; q < P; q += NT) {
            const u32 f = finish_hash(a.lh, poly(q));
            sm.pF[q] = f;
            u32 s = (f * 0x9E3779B1u) >> 21;
            while (true) {
                const u32 old = atomicCAS(&sm.slot[s], ~0u, q);
                if (old == ~0u || same(old, q)) break;
                s = (s + 1) & (kSoloSlots - 1);
            }
            sm.slot_of[q] = (unsigned short)s;
            atomicMin(&sm.first[s], q);
        }
        static_assert(kSoloSlots == 1 << 11 && kSoloPhrases < kSoloSlots, "a slot for every phrase");
        __syncthreads();
        // ids: resident rules, and the new ones in the order of their first occurrences
        constexpr u32 kPerQ = (kSoloPhrases + NT - 1) / NT;
        u32 fresh = 0;
        u64 len_sum = 0;
        for (u32 i = 0; i < kPerQ; i++) {
            const u32 q = tid * kPerQ + i;
            if (q >= P || sm.first[sm.slot_of[q]] != q) continue;
            const u32 st = sm.start[q], len = sm.start[q + 1] - st;
            u64 rank = ~0ull;
            if (a.rtab_cap) {
                bool res = true;
                if (a.sym_bytes != 1)
                    for (u32 j = 0; j < len; j++) res = res && T[st + j] < a.prev_base;
                if (res) {
                    const bool hashed = len > (u32)inline_max(a.sym_w);
                    const Key128 key = hashed ? key_hashed(poly(q), len, st) : key_inline32(T + st, len, a.sym_w);
                    rank = table_find(ContentTable{(Slot*)a.rtab, a.rtab_cap}, key, hashed, [&](u64 rk) {
                        const u64 o = a.rrhs_off[rk];
                        for (u32 j = 0; j < len; j++)
                            if (T[st + j] != a.rrhs[o + j]) return false;
                        return true;
                    });
                }
            }
            if (rank == ~0ull) {
                fresh |= 1u << i;
                len_sum += len;
            } else {
                sm.slot[sm.slot_of[q]] = (u32)rank;
            }
        }
        u64 g_new, G_new;
        u32 c = (u32)block_excl_scan((u64)__popc(fresh), g_new);
        block_excl_scan(len_sum, G_new);
        for (u32 i = 0; i < kPerQ; i++) {
            if (!((fresh >> i) & 1u)) continue;
            const u32 q = tid * kPerQ + i, st = sm.start[q], len = sm.start[q + 1] - st;
            const Key128 key = len > (u32)inline_max(a.sym_w) ? key_hashed(poly(q), len, st)
                                                              : key_inline32(T + st, len, a.sym_w);
            ((ClaimRec*)a.crec)[c] = ClaimRec{key, sm.pF[q], {0u, 0u, 0u}};
            a.minpos[c] = q;
            sm.slot[sm.slot_of[q]] = a.id_base + c;
            c++;
        }
        if (warp == 0) {
            u32 o = (u32)__popc(sm.ret[lane]);
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const u32 y = __shfl_up_sync(0xffffffffu, o, d);
                if (lane >= (u32)d) o += y;
            }
            sm.rpre[lane] = o - (u32)__popc(sm.ret[lane]);
        }
        __syncthreads();
        // the next sequence (in global memory too: long rules are read there), and the roots
        for (u32 q = tid; q < P; q += NT) {
            const u32 id = sm.slot[sm.slot_of[q]];
            const u32 w = q >> 5, before = sm.rpre[w] + __popc(sm.ret[w] & ((1u << (q & 31)) - 1u));
            if ((sm.ret[w] >> (q & 31)) & 1u) {
                const u32 j = a.R_sid[before];
                a.c_level[j] = a.level;
                a.c_rank[j] = id;  // k_naming_small makes it a rank
            } else {
                sm.T[cur ^ 1][q - before] = id;
                sm.F[cur ^ 1][q - before] = sm.pF[q];
                a.Tnext[q - before] = id;
            }
        }
        if (tid == 0) {
            a.rc->phrases = P;
            a.rc->retired = retired;
            a.rc->k_next = k1;
            a.rc->n_next = n1;
            *a.total = P;
            a.ds->claims = g_new;
            a.ds->claim_len = G_new;
            a.ds->aux[1] = g_new;
        }
        n = n1;
        k = k1;
        __syncthreads();
    }
}

// The phrases and the parse of the rounds t.r[0 .. t.rounds), until no string
// is left.
// Strings of a round, at most, that one block takes (in the barrier); more are shared
// out, for two barriers more (some 6 us, what one block takes for 800 strings).  100,000
// strings of 5 bytes: 1443 us in this kernel with one block for all strings, 200 so; the
// build 5.90 ms, 4.47 so.
constexpr u32 kStringsAlone = 2048;

// (one block per SM: without the bound the compiler may settle on 80 registers and spill)
template <bool kByte>
__global__ void __launch_bounds__(kSmallThreads, 1) k_parse_small(const __grid_constant__ TailArgs t) {
    pdl_wait();
    u64 idx = 0;
    for (u32 r = 0; r < t.rounds; r++) {
        const RoundArgs& a = t.r[r];
        const u64 n = round_n(a);
        if (n == 0) break;
        if (n <= kSoloSymbols) {
            if (blockIdx.x == 0) solo_rounds<kByte>(t, r);
            return;
        }
        const u32 k = round_k(a);
        auto barrier = [&](auto work) { grid_barrier_work(t.bar, idx++, a.ds, work); };
        if (r == 0) {
            body_tile_strings(a, a.tiles_bound);
            barrier([] {});
        }
        const u64 steps = (n + kBrkSpan - 1) / kBrkSpan;
        if (kByte && r == 0) body_breaks<unsigned char, true>(a, steps);
        else body_breaks<u32, true>(a, steps);
        // places of the units' phrases; the strings, and their starts in T^{i+1}
        barrier([&] {
            const u64 units = min((n + a.tp - 1) / a.tp, a.tiles_bound);
            const u64 P = block_scan_small([&](u64 i) { return a.tile_cnt[i]; }, units,
                                           [&](u64 i, u64 e) { a.tile_pfx[i] = e; });
            if (threadIdx.x == 0) *a.total = P;
            __syncthreads();
            if (k <= kStringsAlone) body_strings(a);
        });
        if (k > kStringsAlone) {
            // each block its share of the strings: how many retire, then their places
            const u64 P = *a.total;
            const u32 share = (k + gridDim.x - 1) / gridDim.x;
            const u32 lo = min(k, blockIdx.x * share), hi = min(k, lo + share);
            const bool ok = !round_halted(a);
            u64 mine = 0, sum;
            for (u32 j = lo + threadIdx.x; ok && j < hi; j += blockDim.x) {
                u64 first;
                mine += string_retires(a, j, k, P, first) ? 1 : 0;
            }
            block_excl_scan(mine, sum);
            if (threadIdx.x == 0) t.retired[blockIdx.x] = sum;
            barrier([] {});
            u64 before = 0;
            for (u32 b = threadIdx.x; b < blockIdx.x; b += blockDim.x) before += t.retired[b];
            block_excl_scan(before, sum);
            const u64 upto = ok ? strings_range(a, P, k, lo, hi, sum) : 0;
            if (ok && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) strings_end(a, P, k, upto);
            barrier([] {});
        }
        if (kByte && r == 0) body_parse<unsigned char, kUnitMin, kParseWarps, true>(a, a.tiles_bound);
        else body_parse<u32, kUnitMin, kParseWarps, true>(a, a.tiles_bound);
        barrier([] {});
    }
}

// The naming of the same rounds: marks, popcount prefixes (a round's by one
// block), ranks, then the rules in chunks of kRuleChunk: the chunks' lengths,
// and each chunk's offsets and right-hand sides by one block.
constexpr u32 kRuleChunk = 512;

template <bool kByte>
__global__ void __launch_bounds__(kSmallThreads) k_naming_small(const __grid_constant__ TailArgs t) {
    pdl_wait();
    __shared__ u32 s_chunk0[kTailRounds + 1];  // first chunk of each round
    __shared__ u64 s_ids[kTailRounds], s_g[kTailRounds], s_words[kTailRounds], s_retired[kTailRounds];
    __shared__ u32 s_halt;
    const u64 gthreads = (u64)gridDim.x * blockDim.x, gtid = blockIdx.x * (u64)blockDim.x + threadIdx.x;
    if (threadIdx.x == 0) s_halt = 0;
    __syncthreads();
    if (threadIdx.x < t.rounds) {
        const RoundArgs& a = t.r[threadIdx.x];
        const u64 g = *a.d_gnew;
        if (vload(&a.ds->error) || vload(&a.ds->overflow)) s_halt = 1;
        if (threadIdx.x == 0 && a.ds_prev && (vload(&a.ds_prev->error) || vload(&a.ds_prev->overflow))) s_halt = 1;
        if (g > a.r_cap || a.g_base + g > a.cap_g || a.G_base + *a.d_Gnew > a.cap_G) {
            set_error(a.ds, kErrCapacity);  // a level that outgrew its plan
            s_halt = 1;
        }
        s_g[threadIdx.x] = g;
        s_ids[threadIdx.x] = min(*a.d_ids, a.id_cap);
        s_words[threadIdx.x] = g ? min(a.first_words, (*a.total + 31) / 32) : 0;
        s_retired[threadIdx.x] = a.rc->retired;
    }
    __syncthreads();
    // (the answer is the same in every block: the rounds are over, and a
    // capacity that a block finds exceeded is exceeded for all)
    if (s_halt) return;
    if (threadIdx.x == 0) {
        u32 c = 0;
        for (u32 r = 0; r < t.rounds; r++) {
            s_chunk0[r] = c;
            c += (u32)((s_g[r] + kRuleChunk - 1) / kRuleChunk);
        }
        s_chunk0[t.rounds] = c;
    }
    // 1. marks
    for (u32 r = 0; r < t.rounds; r++) {
        const RoundArgs& a = t.r[r];
        for (u64 c = gtid; c < s_ids[r]; c += gthreads) {
            const u64 m = a.minpos[c];
            if (m < a.first_words * 32) atomicOr(&a.first[m >> 5].x, 1u << (m & 31));
        }
    }
    DevStatus* ds = t.r[0].ds;
    grid_barrier(t.bar + 2, 0, ds);
    // 2. popcount prefixes
    for (u32 r = blockIdx.x; r < t.rounds; r += gridDim.x) {
        const RoundArgs& a = t.r[r];
        block_scan_small([&](u64 w) { return (u32)__popc(a.first[w].x); }, s_words[r],
                         [&](u64 w, u64 e) { a.first[w].y = (u32)e; });
    }
    grid_barrier(t.bar + 2, 1, ds);
    // 3. ranks
    for (u32 r = 0; r < t.rounds; r++) {
        const RoundArgs& a = t.r[r];
        const ClaimRec* crec = (const ClaimRec*)a.crec;
        ClaimRec* rrec = (ClaimRec*)a.rrec;
        for (u64 c = gtid; c < s_ids[r]; c += gthreads) {
            const u64 m = a.minpos[c];
            const ClaimRec rec = crec[c];
            if (m >= a.first_words * 32) continue;  // no claim
            const uint2 f = a.first[m >> 5];
            const u64 rank = f.y + __popc(f.x & ((1u << (m & 31)) - 1u));
            if (rank >= s_g[r]) continue;  // not reached
            a.rank_of[c] = (u32)(a.g_base + rank);
            a.F[a.g_base + rank] = rec.fp;  // (read below by the level above's rules)
            rrec[rank] = rec;
        }
    }
    grid_barrier(t.bar + 2, 2, ds);
    // 4. symbols of each chunk of rules
    const u32 chunks = s_chunk0[t.rounds];
    auto round_of = [&](u32 ch) {
        u32 r = 0;
        while (s_chunk0[r + 1] <= ch) r++;
        return r;
    };
    for (u32 ch = blockIdx.x; ch < chunks; ch += gridDim.x) {
        const u32 r = round_of(ch);
        const ClaimRec* rec = (const ClaimRec*)t.r[r].rrec;
        const u64 r0 = (u64)(ch - s_chunk0[r]) * kRuleChunk, r1 = min(s_g[r], r0 + kRuleChunk);
        u64 sum = 0, tot;
        for (u64 x = r0 + threadIdx.x; x < r1; x += blockDim.x) sum += key_len(rec[x].key);
        block_excl_scan(sum, tot);
        if (threadIdx.x == 0) t.chunk_len[ch] = tot;
    }
    // the retired strings' roots
    for (u32 r = 0; r < t.rounds; r++) {
        const RoundArgs& a = t.r[r];
        for (u64 x = gtid; x < s_retired[r]; x += gthreads) {
            const u32 id = a.c_rank[a.R_sid[x]];
            if (id >= a.id_base && id - a.id_base < a.id_cap) a.c_rank[a.R_sid[x]] = a.rank_of[id - a.id_base];
        }
    }
    grid_barrier(t.bar + 2, 3, ds);
    // 5. offsets and right-hand sides
    for (u32 ch = blockIdx.x; ch < chunks; ch += gridDim.x) {
        const u32 r = round_of(ch);
        const RoundArgs& a = t.r[r];
        const ClaimRec* rec = (const ClaimRec*)a.rrec;
        const u64 r0 = (u64)(ch - s_chunk0[r]) * kRuleChunk, r1 = min(s_g[r], r0 + kRuleChunk);
        u64 before = 0, base;
        for (u32 x = s_chunk0[r] + threadIdx.x; x < ch; x += blockDim.x) before += t.chunk_len[x];
        block_excl_scan(before, base);
        u64* off = a.rhs_off + a.g_base;
        const u64 len = block_scan_small([&](u64 x) { return (u32)key_len(rec[r0 + x].key); }, r1 - r0,
                                         [&](u64 x, u64 e) { off[r0 + x] = a.G_base + base + e; });
        if (r1 == s_g[r] && threadIdx.x == 0) off[r1] = a.G_base + base + len;
        __syncthreads();
        if (kByte && r == 0) rules_range<unsigned char, true>(a, r0 + threadIdx.x, blockDim.x, r1);
        else rules_range<u32, true>(a, r0 + threadIdx.x, blockDim.x, r1);
        __syncthreads();
    }
}

static unsigned grid_for(u64 n, u64 cap = 152ull * 32) {
    u64 b = (n + 255) / 256;
    if (b == 0) b = 1;
    return (unsigned)(b < cap ? b : cap);
}

constexpr u32 kWarps = kParseWarps;
bool parse_tile_valid(u32 tp) { return tp == 1024 || tp == 2048 || tp == 4096; }
u32 parse_unit(u32 tile) { return tile / kWarps; }
static_assert(1024 / kWarps == kUnitMin && 4096 / kWarps == kUnitMax, "units of the accepted tiles");
size_t claim_rec_bytes() { return sizeof(ClaimRec); }
u64 breaks_steps(u64 tiles, u32 tp) { return (tiles * (u64)tp + kBrkSpan - 1) / kBrkSpan + 1; }

u64 popscan_tiles_for(u64 nw) { return (nw + kPopTile - 1) / kPopTile; }

cudaError_t launch_tile_strings(const RoundArgs& a, cudaStream_t st) {
    return launch_pdl(k_tile_strings, grid_for(a.tiles_bound), 256, st, a, a.tiles_bound);
}

// What the current device can hold of a kernel with `smem` bytes of dynamic shared
// memory, whose limit is raised there (CUDA keeps it per device).
struct Fit {
    int per_sm = 0;  // resident blocks of an SM
    int sms = 0;
};
template <typename Kernel>
static cudaError_t fit_of(PerDevice<Fit>& known, Kernel* kernel, int threads, size_t smem, Fit& out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return known.get(dev, out, [&](Fit& f) {
        cudaError_t err = cudaDeviceGetAttribute(&f.sms, cudaDevAttrMultiProcessorCount, dev);
        if (err == cudaSuccess && smem > 0)
            err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (err == cudaSuccess)
            err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f.per_sm, kernel, threads, smem);
        if (err == cudaSuccess && (f.per_sm < 1 || f.sms < 1)) err = cudaErrorInvalidConfiguration;
        return err;
    });
}

template <typename T, int U>
static cudaError_t parse_fit(Fit& out) {
    static PerDevice<Fit> known;
    return fit_of(known, k_parse<T, U>, 32 * parse_warps<T>, sizeof(ParseSmem<T, U, parse_warps<T>>), out);
}

// Persistent grid: `per_sm` blocks per SM (0 or more than fit: as many as fit).
template <typename T>
static unsigned persistent_grid(const Fit& fit, u64 units, u32 per_sm) {
    const u64 fits = std::min<u64>((u64)fit.per_sm, parse_blocks<parse_warps<T>>);
    const u64 b = (per_sm == 0 || per_sm > fits) ? fits : (u64)per_sm;
    const u64 g = b * (u64)fit.sms, most = (units + parse_warps<T> - 1) / parse_warps<T>;
    return (unsigned)(most < g ? (most ? most : 1) : g);
}

u64 parse_blocks_most(int sym_bytes, u64 units, u64 sms) {
    const u64 warps = sym_bytes == 1 ? parse_warps<unsigned char> : parse_warps<u32>;
    const u64 per_sm = sym_bytes == 1 ? parse_blocks<parse_warps<unsigned char>> : parse_blocks<parse_warps<u32>>;
    return std::max<u64>(1, std::min(per_sm * sms, (units + warps - 1) / warps));
}

// Most k_parse blocks that fit on an SM of the current device, over every unit size
// (at least 1).
template <typename T>
static int parse_max_blocks_t() {
    int most = 1;
    for (auto fit : {parse_fit<T, 128>, parse_fit<T, 256>, parse_fit<T, 512>}) {
        Fit f;
        if (fit(f) == cudaSuccess) most = std::max(most, f.per_sm);
    }
    return most;
}
int parse_max_blocks(int sym_bytes) {
    return sym_bytes == 1 ? parse_max_blocks_t<unsigned char>() : parse_max_blocks_t<u32>();
}

template <typename T>
static cudaError_t launch_breaks_t(const RoundArgs& a, cudaStream_t st) {
    static PerDevice<Fit> known;
    Fit fit;
    const cudaError_t e = fit_of(known, k_breaks<T>, kBrkThreads, 0, fit);
    if (e != cudaSuccess) return e;
    const u64 steps = (a.tiles_bound * (u64)a.tp + kBrkSpan - 1) / kBrkSpan;
    const u64 blocks = std::max<u64>(1, std::min<u64>(steps, (u64)fit.per_sm * (u64)fit.sms));
    return launch_pdl(k_breaks<T>, (unsigned)blocks, kBrkThreads, st, a, steps);
}

cudaError_t launch_breaks(const RoundArgs& a, cudaStream_t st) {
    return a.sym_bytes == 1 ? launch_breaks_t<unsigned char>(a, st) : launch_breaks_t<u32>(a, st);
}

template <typename T, int U>
static cudaError_t launch_parse_tp(const RoundArgs& a, cudaStream_t st) {
    const u64 tiles = a.tiles_bound;
    Fit fit;
    const cudaError_t e = parse_fit<T, U>(fit);
    if (e != cudaSuccess) return e;
    return launch_pdl_smem(k_parse<T, U>, persistent_grid<T>(fit, tiles, a.parse_blocks), 32 * parse_warps<T>,
                           sizeof(ParseSmem<T, U, parse_warps<T>>), st, a, tiles);
}

template <typename T>
static cudaError_t launch_parse_t(const RoundArgs& a, cudaStream_t st) {
    switch (a.tp) {
        case 128: return launch_parse_tp<T, 128>(a, st);
        case 256: return launch_parse_tp<T, 256>(a, st);
        case 512: return launch_parse_tp<T, 512>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_parse(const RoundArgs& a, cudaStream_t st) {
    if (a.sym_bytes == 1) return launch_parse_t<unsigned char>(a, st);
    return launch_parse_t<u32>(a, st);
}

// Blocks of the short rounds' launches: a warp per unit, at most one block per SM (all
// of them resident at once: one fits an SM).
static u32 tail_grid(const Fit& fit, u64 units, u32 most) {
    const u64 blocks = std::min<u64>((u64)fit.sms, std::max<u64>(1, (units + kWarps - 1) / kWarps));
    return (u32)(most ? std::min<u64>(blocks, most) : blocks);
}

template <bool kByte>
static cudaError_t launch_parse_small_t(const TailArgs& t, u32 most, cudaStream_t st) {
    using T0 = std::conditional_t<kByte, unsigned char, u32>;
    constexpr size_t smem = std::max({sizeof(ParseSmem<T0, kUnitMin, kParseWarps>), sizeof(ParseSmem<u32, kUnitMin, kParseWarps>), sizeof(SoloSmem)});
    static PerDevice<Fit> known;
    Fit fit;
    const cudaError_t e = fit_of(known, k_parse_small<kByte>, kSmallThreads, smem, fit);
    if (e != cudaSuccess) return e;
    return launch_coop(k_parse_small<kByte>, tail_grid(fit, t.r[0].tiles_bound, most), kSmallThreads, smem, st, t);
}

template <bool kByte>
static cudaError_t launch_naming_small_t(const TailArgs& t, u32 most, cudaStream_t st) {
    static PerDevice<Fit> known;
    Fit fit;
    const cudaError_t e = fit_of(known, k_naming_small<kByte>, kSmallThreads, 0, fit);
    if (e != cudaSuccess) return e;
    return launch_coop(k_naming_small<kByte>, tail_grid(fit, t.r[0].tiles_bound, most), kSmallThreads, 0, st, t);
}

cudaError_t launch_parse_small(const TailArgs& t, u32 most, cudaStream_t st) {
    return t.r[0].sym_bytes == 1 ? launch_parse_small_t<true>(t, most, st) : launch_parse_small_t<false>(t, most, st);
}

cudaError_t launch_naming_small(const TailArgs& t, u32 most, cudaStream_t st) {
    return t.r[0].sym_bytes == 1 ? launch_naming_small_t<true>(t, most, st) : launch_naming_small_t<false>(t, most, st);
}

u64 rule_chunks(u64 g) { return (g + kRuleChunk - 1) / kRuleChunk; }

cudaError_t launch_strings(const RoundArgs& a, cudaStream_t st) {
    return launch_pdl(k_strings, 1, 1024, st, a);
}

cudaError_t launch_mark(const RoundArgs& a, u64 g_grid, cudaStream_t st) {
    return launch_pdl(k_mark, grid_for(g_grid), 256, st, a);
}

cudaError_t launch_popscan(const RoundArgs& a, cudaStream_t st) {
    u64 tiles = popscan_tiles_for(a.first_words);
    if (tiles == 0) tiles = 1;
    return launch_pdl(k_popscan, (unsigned)tiles, kPopThreads, st, a);
}

u64 rule_offs_tiles(u64 g) { return std::max<u64>(1, (g + kRoTile - 1) / kRoTile); }

cudaError_t launch_rule_offs(const RoundArgs& a, u64 g_grid, cudaStream_t st) {
    return launch_pdl(k_rule_offs, (unsigned)rule_offs_tiles(g_grid), kRoThreads, st, a);
}

cudaError_t launch_rank(const RoundArgs& a, u64 g_grid, cudaStream_t st) {
    return launch_pdl(k_rank, grid_for(g_grid), 256, st, a);
}

cudaError_t launch_rules(const RoundArgs& a, u64 g_grid, cudaStream_t st) {
    if (a.sym_bytes == 1) return launch_pdl(k_rules<unsigned char>, grid_for(g_grid), 256, st, a);
    return launch_pdl(k_rules<u32>, grid_for(g_grid), 256, st, a);
}

cudaError_t launch_level0(const unsigned char* data, const u64* pos, const u32* ids, u32 cnt, u32* c_level,
                          u32* c_rank, cudaStream_t st) {
    if (cnt == 0) return cudaSuccess;
    k_level0<<<(cnt + 255) / 256, 256, 0, st>>>(data, pos, ids, cnt, c_level, c_rank);
    return cudaGetLastError();
}

cudaError_t launch_gather_strings(const unsigned char* data, const u64* src_off, const u64* dst_off, u32 k,
                                  unsigned char* out, cudaStream_t st) {
    if (k == 0) return cudaSuccess;
    const unsigned blocks = k < 152 * 8 ? k : 152 * 8;
    k_gather_strings<<<blocks, 256, 0, st>>>(data, src_off, dst_off, k, out);
    return cudaGetLastError();
}

size_t lb1_bytes(u64 tiles) { return tiles * sizeof(LBSlot<1>); }
size_t slot_bytes() { return sizeof(Slot); }

}  // namespace lcg
