// Content-addressed phrase tables (one per level and round).
//
// A table maps the content of a phrase (a sequence of level-(i-1) symbols) to
// a value: during a round's parse the value is the smallest phrase index among
// the phrase's occurrences, which decides first-occurrence naming; in the
// table of a resident grammar it is the rule's rank.
//
// Keys are 128 bits.  Short phrases are stored exactly ("inline" keys): the
// top 4 bits of `hi` hold the length q, and the symbols are packed from bit 0
// upwards in the 124 bits left, w bits each (8 for bytes; for ranks the width
// of the level below, at most 31), so q <= min(14, 124 / w).  Two inline keys
// of one width are equal exactly when the phrases are.  The length field is
// at most 14, so no key has hi == ~0, the mark of an empty slot (tables are
// cleared to all ones): with 15 bytes a phrase of 0xFF bytes would have
// packed to exactly that mark.  A longer phrase gets a "hashed" key: top 4
// bits 0, its length in bits 32..59 of `hi` and a 32-bit hash below, with `lo`
// naming where its content can be read; a hashed-key match is confirmed by
// comparing the contents symbol by symbol.  Slots are claimed with one 128-bit compare-and-swap.
// The home slot is the high half of mix(key) * cap, so any capacity works;
// the polynomial fingerprint H = sum_j F[Q_j] c^{j-1} mod p of a phrase is
// only needed for hashed keys.
#pragma once

#include "lcg_dev.cuh"

namespace lcg {

struct __align__(16) Key128 {
    u64 lo, hi;
};

// A slot holds its 128-bit key, its 64-bit value and what a round's lookups
// take from it in one 32-byte sector, so that a lookup touches one sector.
struct __align__(32) Slot {
    Key128 key;
    u64 val;  // round tables: the smallest phrase index seen (a filter: minpos decides); resident tables: the rank
    u64 pub;  // round tables: (F^i << 32) | number of the claim; ~0 until the claiming thread has stored it
};
static_assert(sizeof(Slot) == 32, "one sector per slot");
constexpr u64 kUnpublished = ~0ull;

struct ContentTable {
    Slot* slots;
    u64 cap;  // 0: no table
};

constexpr u64 kEmptyHi = ~0ull;
constexpr int kHiBits = 60;
constexpr u64 kMaxPhraseLen = (1ull << 28) - 1;  // longest phrase a hashed key can describe

// Bits per symbol in inline keys: 8 for bytes; for ranks a width w with every
// rank of the level below < 2^w.  A round's own table uses the smallest such w
// (so that more phrases fit inline); tables that outlive a round (resident
// grammars, merges) use kRankBits.
constexpr int kRankBits = 31;
constexpr int kInlineMax = 14;
__device__ __forceinline__ u64 inline_max(int w) {
    const int m = 124 / w;
    return m < kInlineMax ? (u64)m : (u64)kInlineMax;
}

__device__ __forceinline__ u64 get_bits(u64 hi, u64 lo, int pos, int b) {
    const u64 m = (1ull << b) - 1;
    if (pos + b <= kHiBits) return (hi >> pos) & m;
    if (pos >= kHiBits) return (lo >> (pos - kHiBits)) & m;
    const u64 low = (hi >> pos) & ((1ull << (kHiBits - pos)) - 1);
    return (low | (lo << (kHiBits - pos))) & m;
}

// The inline key of get(0..len-1): the symbols form the number
// V = sum_j get(j) 2^(j b) (at most 124 bits), accumulated from the last
// symbol with a 128-bit shift per symbol (no branch on where a symbol falls);
// bits 0..59 of V go to hi under the length, bits 60..123 to lo.  This is the
// layout key_sym reads.
template <typename Get>
__device__ __forceinline__ Key128 key_inline(Get get, u64 len, int b) {
    u64 vlo = 0, vhi = 0;  // V, 128 bits
    for (u64 j = len; j-- > 0;) {
        vhi = (vhi << b) | (vlo >> (64 - b));  // b in 1..31: both shifts defined
        vlo = (vlo << b) | (u64)get(j);
    }
    const u64 hi = (len << kHiBits) | (vlo & ((1ull << kHiBits) - 1));
    const u64 lo = (vlo >> kHiBits) | (vhi << (64 - kHiBits));
    return Key128{lo, hi};
}

// The same key, built from 32-bit symbols pushed from the last to the first
// (b in 1..31): four words and a funnel shift each.
struct PackedSyms {
    u32 w0 = 0, w1 = 0, w2 = 0, w3 = 0;
    __device__ __forceinline__ void push(u32 v, int b) {
        w3 = __funnelshift_l(w2, w3, b);
        w2 = __funnelshift_l(w1, w2, b);
        w1 = __funnelshift_l(w0, w1, b);
        w0 = (w0 << b) | v;
    }
    __device__ __forceinline__ Key128 key(u32 len) const {
        const u32 lo0 = __funnelshift_r(w1, w2, 28), lo1 = __funnelshift_r(w2, w3, 28);
        const u32 hi1 = (w1 & ((1u << (kHiBits - 32)) - 1)) | (len << (kHiBits - 32));
        return Key128{((u64)lo1 << 32) | lo0, ((u64)hi1 << 32) | w0};
    }
};

__device__ __forceinline__ Key128 key_inline32(const u32* sym, u32 len, int b) {
    PackedSyms ps;
#pragma unroll 1
    for (u32 j = len; j-- > 0;) ps.push(sym[j], b);
    return ps.key(len);
}

__device__ __forceinline__ Key128 key_hashed(u64 H, u64 len, u64 ref) {
    const u32 h = (u32)fmix64(H ^ (len * 0x9E3779B97F4A7C15ull));
    return Key128{ref, (len << 32) | (u64)h};
}

__device__ __forceinline__ bool key_is_hashed(const Key128& k) { return (k.hi >> kHiBits) == 0; }

__device__ __forceinline__ u64 key_len(const Key128& k) {
    const u64 l = k.hi >> kHiBits;
    return l ? l : ((k.hi >> 32) & kMaxPhraseLen);
}

// symbol j of an inline key
__device__ __forceinline__ u32 key_sym(const Key128& k, u64 j, int b) {
    return (u32)get_bits(k.hi, k.lo, (int)j * b, b);
}

// Home slot of a key: the high half of mix(key) * cap.  An inline key is the
// content itself; a hashed key's high half carries the length and a hash of
// the phrase's fingerprint (its low half names a location, not content).  The
// mix is a multiply-xorshift of both halves (two 64-bit products).
__device__ __forceinline__ u64 key_home(const Key128& k, u64 cap) {
    const u64 lo = key_is_hashed(k) ? 0ull : k.lo;
    u64 m = (lo ^ (k.hi * 0x9E3779B97F4A7C15ull)) * 0xD6E8FEB86659FD93ull;
    m ^= m >> 32;
    return __umul64hi(m, cap);
}

__device__ __forceinline__ Key128 ld_key_relaxed(const Key128* p) {
    Key128 k;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(k.lo), "=l"(k.hi) : "l"(p) : "memory");
    return k;
}

// A slot with one 32-byte load (one request for the sector).  The four words
// need not be read at one instant: the key is checked by the caller, the value
// only used as an upper bound of the stored value, which never increases, and
// pub is written once.
__device__ __forceinline__ Slot ld_slot_relaxed(const Slot* p) {
    Slot s;
    asm volatile("ld.relaxed.gpu.global.v4.u64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(s.key.lo), "=l"(s.key.hi), "=l"(s.val), "=l"(s.pub)
                 : "l"(p)
                 : "memory");
    return s;
}

__device__ __forceinline__ Key128 cas_key(Key128* p, Key128 cmp, Key128 val) {
    Key128 old;
    asm volatile(
        "{\n\t"
        ".reg .b128 c, n, d;\n\t"
        "mov.b128 c, {%2, %3};\n\t"
        "mov.b128 n, {%4, %5};\n\t"
        "atom.relaxed.gpu.global.cas.b128 d, [%6], c, n;\n\t"
        "mov.b128 {%0, %1}, d;\n\t"
        "}"
        : "=l"(old.lo), "=l"(old.hi)
        : "l"(cmp.lo), "l"(cmp.hi), "l"(val.lo), "l"(val.hi), "l"(p)
        : "memory");
    return old;
}

// Longest probe sequence of a claim: far beyond what a table under its load
// limit shows, so reaching it means the table is (nearly) full.
constexpr u64 kMaxProbes = 4096;

// Rounds: find or claim the slot of a key in a table that other threads are
// filling, 32 keys of a warp side by side.
//
// A slot read as empty is claimed with a compare-and-swap (it may have been
// claimed since: the swap then returns its key; one read as taken stays so, as
// keys are never removed).  Claims are numbered from ranges that a block takes
// from the round's counter (ClaimIds), and a claiming thread then stores what
// the slot's finders need in one 16-byte store: (F << 32) | number.  A finder
// that comes before that store reads the slot again: the claiming thread waits
// for no other, so the wait ends (bounded all the same).  The
// phrase's first occurrence is kept by claim number in minpos; the slot's
// value is a copy that tells most finders that they come later.
struct __align__(32) ClaimRec {
    Key128 key;
    u32 fp;  // F^i of the phrase
    u32 pad[3];
};
static_assert(sizeof(ClaimRec) == 32, "one sector per claim");

struct RoundTable {
    Slot* slots;
    u64 cap;
    u64* minpos;     // claim -> smallest phrase index
    ClaimRec* crec;  // claim -> key and fingerprint
    u64 id_cap;      // claim numbers that fit
    u32 id_chunk;    // claim numbers a block takes at a time
    u64 max_probes;  // slots that a phrase tries before the table counts as too full
    DevStatus* ds;   // aux[1] (the counter of claim numbers), overflow, error
};

// A block's claim numbers, in shared memory: [next, next + left) are its own.
// The counter is one address for the whole grid, and its atomics come one
// after another (about 7 ns each: with a warp taking its own numbers, 12 K of
// them for 0.38 M claims, such a round took 100 us instead of 45), so a block
// takes id_chunk numbers at a time.  What is left at the kernel's end stays
// unused (minpos ~0), at most id_chunk numbers per block.
struct ClaimIds {
    u64 next;
    u32 left;
    u32 lock;
};

// Claim numbers for the lanes of mask m (non-empty, uniform); every lane of
// the warp calls it.  The lock is held by one warp's lane 0, which waits for
// nothing but the counter, so every wait for it ends.
__device__ __forceinline__ u64 take_ids(const RoundTable& t, ClaimIds* ids, unsigned m) {
    const u32 lane = threadIdx.x & 31;
    const u32 need = (u32)__popc(m), mine = (u32)__popc(m & ((1u << lane) - 1u));
    u64 first = 0, base = 0;
    u32 had = 0;
    if (lane == 0) {
        u32 it = 0;
        while (atomicCAS(&ids->lock, 0u, 1u) != 0u) {
            if (++it > (u32)kSpinLimit) {
                set_error(t.ds, kErrTimeout);
                break;
            }
        }
        volatile ClaimIds* v = ids;
        first = v->next;
        had = min(v->left, need);
        if (had == need) {
            v->next = first + need;
            v->left = v->left - need;
        } else {
            const u32 more = need - had, size = more > t.id_chunk ? more : t.id_chunk;
            base = atomicAdd(&t.ds->aux[1], (u64)size);
            v->next = base + more;
            v->left = size - more;
        }
        __threadfence_block();
        atomicExch(&ids->lock, 0u);
    }
    first = __shfl_sync(0xffffffffu, first, 0);
    base = __shfl_sync(0xffffffffu, base, 0);
    had = __shfl_sync(0xffffffffu, had, 0);
    return mine < had ? first + mine : base + (mine - had);
}

// What a thread's claims add up to: their number and their phrases' lengths.
struct ClaimSum {
    u32 count;
    u32 len;
};

// Store what a claim leaves for the round's later kernels and for the slot's
// finders.  False when the round has made too many claims.
__device__ __forceinline__ bool publish_claim(const RoundTable& t, u64 s, u64 c, const Key128& k, u64 p, u32 F) {
    if (c >= t.id_cap) {
        atomicExch(&t.ds->overflow, 1u);
        return false;
    }
    atomicMin(&t.minpos[c], p);  // ~0 before; a finder may come first
    t.crec[c] = ClaimRec{k, F, {0u, 0u, 0u}};
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(&t.slots[s].val), "l"(p),
                 "l"(((u64)F << 32) | c)
                 : "memory");
    return true;
}

// A finder at phrase index p of a published slot (value val): its first
// occurrence is lowered when the value does not rule that out.
__device__ __forceinline__ void lower_first(const RoundTable& t, u64 s, u64 val, u64 pub, u64 p) {
    if (val > p) {
        atomicMin(&t.slots[s].val, p);
        atomicMin(&t.minpos[(u32)pub], p);
    }
}

constexpr u64 kNoPub = ~0ull;

// What is known of a key's home slot before table_resolve.
constexpr u32 kHomeUnknown = 0, kHomeEmpty = 1, kHomeOther = 2;

// Every lane of a warp calls it; lanes with act = false only take part in the
// votes.  `same(ref)` compares the content stored at `ref` with the phrase
// (hashed keys only).  Returns the slot's pub word ((F << 32) | claim number),
// or kNoPub when the table is over its limits (overflow is then set, and the
// host regrows the table and reruns) or a wait ran out.  `home`: kHomeEmpty
// tries to claim the home slot without reading it first, kHomeOther starts at
// the slot after it.  `first` is lowered to the slot's first occurrence as far
// as it is known.
template <typename Same>
__device__ __forceinline__ u64 table_resolve(const RoundTable& t, ClaimIds* ids, ClaimSum& sum, bool act, u32 home,
                                             const Key128& k, u64 p, u32 F, u64& first, Same same) {
    const Key128 empty{~0ull, ~0ull};
    const bool hashed = key_is_hashed(k);
    u64 s = act ? key_home(k, t.cap) : 0;
    if (home == kHomeOther) s = (s + 1 == t.cap) ? 0 : s + 1;
    bool known_empty = home == kHomeEmpty;
    u64 res = kNoPub;
    bool done = !act;
    const u64 limit = t.cap < t.max_probes ? t.cap : t.max_probes;
    u64 probe = 0;
    for (u32 it = 1; !__all_sync(0xffffffffu, done); it++) {
        bool won = false;
        Slot c;
        if (!done) {
            if (known_empty) c.key = empty;
            else c = ld_slot_relaxed(&t.slots[s]);
            known_empty = false;
            if (c.key.hi == kEmptyHi) {
                const Key128 old = cas_key(&t.slots[s].key, empty, k);
                if (old.hi == kEmptyHi) {
                    won = true;
                } else {
                    c.key = old;
                    c.pub = kUnpublished;
                }
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, won);
        if (m) {
            const u64 n = take_ids(t, ids, m);
            if (won) {
                if (publish_claim(t, s, n, k, p, F)) res = ((u64)F << 32) | n;
                sum.count++;
                sum.len += (u32)key_len(k);
                done = true;
            }
        }
        if (!done) {
            bool match = false;
            if (c.key.hi == k.hi) {
                // a pair read while being written shows the empty low half: read it again atomically
                if (c.key.lo == ~0ull) c.key = cas_key(&t.slots[s].key, empty, empty);
                match = hashed ? same(c.key.lo) : c.key.lo == k.lo;
            }
            if (!match) {
                s = (s + 1 == t.cap) ? 0 : s + 1;
                if (++probe >= limit) {
                    atomicExch(&t.ds->overflow, 1u);
                    done = true;
                }
            } else if (c.pub != kUnpublished) {
                lower_first(t, s, c.val, c.pub, p);
                first = min(first, c.val);
                res = c.pub;
                done = true;
            }
            // (matched but not yet published: read it again)
        }
        // once the table is over its limits the pass is rerun: stop early
        if ((it & 15) == 0) {
            if (vload(&t.ds->overflow) || vload(&t.ds->error)) done = true;
            if (it > (u32)kSpinLimit) {
                set_error(t.ds, kErrTimeout);
                done = true;
            }
        }
    }
    return res;
}

// table_resolve by a whole warp for one hashed key (a long phrase): every lane
// calls it with the same arguments.  Lane 0 reads and claims the slots, in the
// same probe order; `same(ref)` is a warp-wide content comparison run by all
// lanes.  Every lane returns the pub word; lane 0 counts the claim.
template <typename SameWarp>
__device__ u64 table_resolve_warp(const RoundTable& t, ClaimIds* ids, ClaimSum& sum, const Key128& k, u64 p, u32 F,
                                  SameWarp same) {
    const u32 lane = threadIdx.x & 31;
    u64 s = key_home(k, t.cap);
    const Key128 empty{~0ull, ~0ull};
    const u64 limit = t.cap < t.max_probes ? t.cap : t.max_probes;
    for (u64 probe = 0; probe < limit; probe++) {
        Slot c{Key128{0, 0}, 0, 0};
        u64 mine = kNoPub;
        int took = 0, stop = 0;
        if (lane == 0) {
            if ((probe & 15) == 15 && vload(&t.ds->overflow)) stop = 1;
            if (!stop) {
                c = ld_slot_relaxed(&t.slots[s]);
                if (c.key.hi == kEmptyHi) {
                    const Key128 old = cas_key(&t.slots[s].key, empty, k);
                    if (old.hi == kEmptyHi) took = 1;
                    c.key = old;
                }
                if (!took && c.key.hi == k.hi && c.key.lo == ~0ull) c.key = cas_key(&t.slots[s].key, empty, empty);
            }
        }
        stop = __shfl_sync(0xffffffffu, stop, 0);
        if (stop) return kNoPub;
        took = __shfl_sync(0xffffffffu, took, 0);
        if (took) {
            const u64 n = take_ids(t, ids, 1u);
            if (lane == 0) {
                if (publish_claim(t, s, n, k, p, F)) mine = ((u64)F << 32) | n;
                sum.count++;
                sum.len += (u32)key_len(k);
            }
            return __shfl_sync(0xffffffffu, mine, 0);
        }
        c.key.lo = __shfl_sync(0xffffffffu, c.key.lo, 0);
        c.key.hi = __shfl_sync(0xffffffffu, c.key.hi, 0);
        if (c.key.hi == k.hi && same(c.key.lo)) {
            if (lane == 0) {
                // wait until the claiming thread has stored the slot's pub word
                u32 it = 0;
                while (true) {
                    c = ld_slot_relaxed(&t.slots[s]);
                    if (c.pub != kUnpublished) {
                        lower_first(t, s, c.val, c.pub, p);
                        mine = c.pub;
                        break;
                    }
                    if ((++it & 15) == 0 && (vload(&t.ds->overflow) || vload(&t.ds->error))) break;
                    if (it > (u32)kSpinLimit) {
                        set_error(t.ds, kErrTimeout);
                        break;
                    }
                }
            }
            return __shfl_sync(0xffffffffu, mine, 0);
        }
        s = (s + 1 == t.cap) ? 0 : s + 1;
    }
    if (lane == 0) atomicExch(&t.ds->overflow, 1u);
    return kNoPub;
}

// table_find by a whole warp for one hashed key; `same(lo)` is a warp-wide
// comparison.  Every lane returns the value, or ~0 when absent.
template <typename SameWarp>
__device__ u64 table_find_warp(const ContentTable& t, const Key128& k, SameWarp same) {
    u64 s = key_home(k, t.cap);
    for (u64 probe = 0; probe < t.cap; probe++) {
        const Key128 cur = t.slots[s].key;  // the same address on every lane
        if (cur.hi == kEmptyHi) return ~0ull;
        if (cur.hi == k.hi && same(cur.lo)) return t.slots[s].val;
        s = (s + 1 == t.cap) ? 0 : s + 1;
    }
    return ~0ull;
}

// Look a key up in a table that nobody writes during the call.  `same(lo)`
// confirms hashed keys.  Returns the slot's value, or ~0 when absent.
template <typename Same>
__device__ u64 table_find(const ContentTable& t, const Key128& k, bool hashed, Same same) {
    u64 s = key_home(k, t.cap);
    for (u64 probe = 0; probe < t.cap; probe++) {
        const Key128 cur = t.slots[s].key;
        if (cur.hi == kEmptyHi) return ~0ull;
        if (cur.hi == k.hi && (hashed ? same(cur.lo) : (cur.lo == k.lo))) return t.slots[s].val;
        s = (s + 1 == t.cap) ? 0 : s + 1;
    }
    return ~0ull;
}

// Claim a free slot for a key known to be absent (rules of a level are
// distinct) and store `val`.
__device__ __forceinline__ void table_put(ContentTable t, const Key128& k, u64 val, DevStatus* ds) {
    u64 s = key_home(k, t.cap);
    const Key128 empty{~0ull, ~0ull};
    for (u64 probe = 0; probe < t.cap; probe++) {
        const Key128 old = cas_key(&t.slots[s].key, empty, k);
        if (old.hi == kEmptyHi) {
            t.slots[s].val = val;
            return;
        }
        s = (s + 1 == t.cap) ? 0 : s + 1;
    }
    set_error(ds, kErrTableFull);
}

// Key of a rule of level `level` whose right-hand side is get(0..len-1)
// (bytes at level 1), with polynomial fingerprint H, for a table whose values
// are ranks: hashed keys name the rank.
template <typename Get>
__device__ __forceinline__ Key128 rule_key(Get get, u64 len, int w, u64 H, u64 rank) {
    if (len <= inline_max(w)) return key_inline(get, len, w);
    return key_hashed(H, len, rank);
}

}  // namespace lcg
