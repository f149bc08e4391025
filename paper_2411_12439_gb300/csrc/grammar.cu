// Kernels that work on finished grammars: MergeGrams (Sec. 3.6), the
// expansion exp(C[j]) (Sec. 2.2), and a generic two-column exclusive scan.
#include "lcg_dev.cuh"
#include "lcg_internal.h"
#include "per_device.h"
#include "table.cuh"

namespace lcg {

// Large tiles: the tiles of a first wave find no prefix to end their look-back at and
// walk back to the first, 32 tiles a round trip.  3.4 M values: 45 us with tiles of
// 2048, 31 us with these.
constexpr int kScanThreads = 512;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

// --------------------------------------------------------------------------
// exclusive scan of two uint32 columns into uint64 (single pass)
// --------------------------------------------------------------------------

// kScanItems consecutive values of a column from p0 (16-byte loads when the
// whole run is inside the column and aligned), zero past n or for no column.
__device__ __forceinline__ void scan_load(const u32* in, u64 p0, u64 n, u32 (&v)[kScanItems]) {
    if (in != nullptr && p0 + kScanItems <= n && (reinterpret_cast<unsigned long long>(in + p0) & 15) == 0) {
#pragma unroll
        for (int q = 0; q < kScanItems / 4; q++) {
            const uint4 x = reinterpret_cast<const uint4*>(in + p0)[q];
            v[4 * q] = x.x, v[4 * q + 1] = x.y, v[4 * q + 2] = x.z, v[4 * q + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int it = 0; it < kScanItems; it++) v[it] = (in != nullptr && p0 + it < n) ? in[p0 + it] : 0u;
    }
}

// out[p0 ...) = e, e + v[0], ... (two at a time when they may be stored so).
__device__ __forceinline__ void scan_store(u64* out, u64 p0, u64 n, const u32 (&v)[kScanItems], u64 e) {
    if (p0 + kScanItems <= n && (reinterpret_cast<unsigned long long>(out + p0) & 15) == 0) {
#pragma unroll
        for (int it = 0; it < kScanItems; it += 2) {
            reinterpret_cast<ulonglong2*>(out + p0)[it / 2] = make_ulonglong2(e, e + v[it]);
            e += (u64)v[it] + v[it + 1];
        }
    } else {
#pragma unroll
        for (int it = 0; it < kScanItems; it++) {
            if (p0 + it < n) out[p0 + it] = e;
            e += v[it];
        }
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan2(const u32* __restrict__ in0, const u32* __restrict__ in1,
                                                        u64 n, u64* __restrict__ out0, u64* __restrict__ out1,
                                                        u64* __restrict__ totals, LBSlot<2>* lb, u64 epoch, u64* ctr,
                                                        u64 ctr_base, DevStatus* ds, const u64* n_dev, u64* end0) {
    pdl_wait();
    const u64 tile = dynamic_tile(ctr, ctr_base);
    if (n_dev != nullptr) n = min(*n_dev, n);
    if (tile > 0 && tile * (u64)kScanTile >= n) return;  // beyond the count read on the device
    const u64 p0 = tile * (u64)kScanTile + (u64)threadIdx.x * kScanItems;
    u32 a[kScanItems], b[kScanItems];
    scan_load(in0, p0, n, a);
    scan_load(in1, p0, n, b);
    u64 sa = 0, sb = 0;
#pragma unroll
    for (int it = 0; it < kScanItems; it++) {
        sa += a[it];
        sb += b[it];
    }
    u64 ta, tb;
    u64 ea = block_excl_scan(sa, ta);
    u64 eb = block_excl_scan(sb, tb);
    u64 agg[2] = {ta, tb}, excl[2];
    block_lookback<2>(lb, tile, epoch, agg, excl, ds);
    ea += excl[0];
    eb += excl[1];
    scan_store(out0, p0, n, a, ea);
    if (out1 != nullptr) scan_store(out1, p0, n, b, eb);
    if ((tile + 1) * (u64)kScanTile >= n && threadIdx.x == 0) {
        totals[0] = excl[0] + ta;
        if (end0 != nullptr) *end0 = excl[0] + ta;
        totals[1] = excl[1] + tb;
    }
}

u64 scan2_tiles_for(u64 n) { return (n + kScanTile - 1) / kScanTile; }
size_t scan2_lb_bytes(u64 tiles) { return scan2_lb_bytes_static(tiles); }

cudaError_t launch_scan2(const u32* in0, const u32* in1, u64 n, u64* out0, u64* out1, u64* totals, void* lb,
                         u64 epoch, u64* ctr, u64 ctr_base, DevStatus* ds, cudaStream_t st, u64* grid_out,
                         const u64* n_dev, u64* end0) {
    u64 tiles = scan2_tiles_for(n);
    if (tiles == 0) tiles = 1;
    *grid_out = tiles;
    return launch_pdl(k_scan2, (unsigned)tiles, kScanThreads, st, in0, in1, n, out0, out1, totals, (LBSlot<2>*)lb,
                      epoch, ctr, ctr_base, ds, n_dev, end0);
}

// --------------------------------------------------------------------------
// MergeGrams
// --------------------------------------------------------------------------

// Three launches per large level: the lookup reads G_b's symbols through Mprev (no
// rewritten copy of G_b), the append takes the totals of the scan from device memory,
// enters the new rules in G_a's table and renames G_b's roots.  Bound by random
// sectors: the table's slots in DRAM, ranks and fingerprints in L2.  (Tiles of 1024
// rules with their symbols in shared memory and four rules a thread, and claiming the
// slots in the lookup, were slower: 543 + 223 us against 267 + 342.)
//
// A rule of more than kRuleLong symbols (an N-run of DNA) is read, hashed and
// compared by a whole warp, after the 32 rules of its threads: a thread alone
// takes a round trip per symbol.
constexpr u64 kRuleLong = 32;

// Calls `one(r, s, len)` for the rules r of [r_first, r_end) that are this thread's
// (s: where their symbols start; block `block` of `blocks` takes 256 at a time) and
// `whole(r, s, len)` with the whole warp for the long ones.
template <typename One, typename Whole>
__device__ __forceinline__ void for_rules(const u64* off, u64 r_first, u64 r_end, u64 block, u64 blocks, One one,
                                          Whole whole) {
    const u32 lane = threadIdx.x & 31;
    for (u64 r0 = r_first + block * blockDim.x + (threadIdx.x & ~31u); r0 < r_end; r0 += blocks * blockDim.x) {
        const u64 r = r0 + lane;
        const u64 s = r < r_end ? off[r] : 0, e = r < r_end ? off[r + 1] : 0;
        if (r < r_end && e - s <= kRuleLong) one(r, s, e - s);
        __syncwarp();
        for (unsigned m = __ballot_sync(0xffffffffu, e - s > kRuleLong); m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const u64 ws = __shfl_sync(0xffffffffu, s, l), we = __shfl_sync(0xffffffffu, e, l);
            whole(r0 + l, ws, we - ws);
            __syncwarp();
        }
    }
}

// H of a rule whose symbol j is get(j), by one thread, four fingerprints in
// flight at a time.
template <typename Get>
__device__ __forceinline__ u64 rule_poly(Get get, u64 len, const u32* F, u64 c) {
    u64 H = 0;
    for (u64 j = len; j > 0;) {
        u32 f[4];
        const u64 m = j < 4 ? j : 4;
#pragma unroll
        for (int u = 0; u < 4; u++) f[u] = (u64)u < m ? F[get(j - 1 - u)] : 0u;
#pragma unroll
        for (int u = 0; u < 4; u++)
            if ((u64)u < m) H = addmod61(mulmod61(H, c), (u64)f[u]);
        j -= m;
    }
    return H;
}

// Key of a rule of at most kRuleLong symbols for a table whose values are ranks
// (see rule_key); H is only computed when the key needs it.
template <bool kByte, typename Get>
__device__ __forceinline__ Key128 rank_key(Get get, u64 len, const u32* Fprev, u64 c, u64 rank) {
    constexpr int w = kByte ? 8 : kRankBits;
    if (len <= inline_max(w)) return key_inline(get, len, w);
    return key_hashed(rule_poly(get, len, Fprev, c), len, rank);
}

// Rules r0 .. r0+cnt-1 of a level enter its table (values: ranks).
template <bool kByte>
__global__ void __launch_bounds__(256) k_resident_build(const u32* __restrict__ rhs, const u64* __restrict__ rhs_off,
                                                        u64 r0, u64 cnt, const u32* __restrict__ Fprev, LevelHash lh,
                                                        ContentTable t, DevStatus* ds) {
    pdl_wait();
    for_rules(rhs_off, r0, r0 + cnt, blockIdx.x, gridDim.x,
              [&](u64 r, u64 s, u64 len) {
                  table_put(t, rank_key<kByte>([&](u64 j) { return __ldg(rhs + s + j); }, len, Fprev, lh.c, r), r, ds);
              },
              [&](u64 r, u64 s, u64 len) {
                  const u64 H = warp_poly61([&](u64 j) -> u64 { return __ldg(Fprev + __ldg(rhs + s + j)); }, len, lh.c);
                  if ((threadIdx.x & 31) == 0) table_put(t, key_hashed(H, len, r), r, ds);
              });
}

// Symbol x of G_b's right-hand sides in G_a's ranks.  (What a merge itself writes --
// ranks, rules, fingerprints -- is read by plain loads: k_merge_small reads it in the
// launch that wrote it.)
template <bool kByte>
__device__ __forceinline__ u32 merge_sym(const MergeLevel& m, u64 x) {
    const u32 v = __ldg(m.brhs + x);
    if constexpr (kByte) return v;
    else return m.Mprev[v];
}

// An earlier level's failure: what this one would read may not have been written.
__device__ __forceinline__ bool merge_failed(const MergeLevel& m) {
    return vload(&m.ds->error) != 0 || vload(&m.ds->overflow) != 0;
}

// For every rule of G_b: its rank in G_a when G_a has the same right-hand side
// (G_b's symbols through Mprev are G_a's ranks; looked up in G_a's table of the
// level, hashed keys confirmed by comparing contents), else a miss.  Bound by the
// round trips of a thread's rule: its bounds, its symbols, their ranks, the slot.
template <bool kByte, typename Put>
__device__ __forceinline__ void merge_lookup(const MergeLevel& m, u64 r_first, u64 r_end, u64 block, u64 blocks, Put put) {
    const ContentTable at{(Slot*)m.slots, m.cap};
    for_rules(m.boff, r_first, r_end, block, blocks,
              [&](u64 r, u64 s, u64 len) {
                  const Key128 key = rank_key<kByte>([&](u64 j) { return merge_sym<kByte>(m, s + j); }, len, m.aFprev,
                                                     m.lh.c, 0);
                  put(r, len, table_find(at, key, key_is_hashed(key), [&](u64 ra) {
                          const u64 o = m.aoff[ra];
                          for (u64 x = 0; x < len; x++)
                              if (m.arhs[o + x] != merge_sym<kByte>(m, s + x)) return false;
                          return true;
                      }));
              },
              [&](u64 r, u64 s, u64 len) {
                  const u64 H = warp_poly61([&](u64 j) -> u64 { return m.aFprev[merge_sym<kByte>(m, s + j)]; }, len,
                                            m.lh.c);
                  const u64 found = table_find_warp(at, key_hashed(H, len, 0), [&](u64 ra) {
                      const u64 o = m.aoff[ra];
                      return warp_equal([&](u64 x) { return m.arhs[o + x]; },
                                        [&](u64 x) { return merge_sym<kByte>(m, s + x); }, len);
                  });
                  if ((threadIdx.x & 31) == 0) put(r, len, found);
              });
}

template <bool kByte>
__global__ void __launch_bounds__(256) k_merge_lookup(const __grid_constant__ MergeLevel m) {
    pdl_wait();
    if (merge_failed(m)) return;
    merge_lookup<kByte>(m, 0, m.gb, blockIdx.x, gridDim.x, [&](u64 r, u64 len, u64 found) {
        if (found != ~0ull) {
            if (m.aF[found] != m.bF[r]) set_error(m.ds, kErrMismatch);
            m.M[r] = (u32)found;
        }
        m.miss[r] = found == ~0ull ? 1u : 0u;
        m.mlen[r] = found == ~0ull ? (u32)len : 0u;
    });
}

// Append the missed rules of G_b to G_a in G_b's rank order (totals: their number
// and symbols, read here so that the host need not wait for them) and to G_a's
// table, and give G_b's roots of this level their ranks in G_a.
template <bool kByte>
__global__ void __launch_bounds__(256) k_merge_append(const __grid_constant__ MergeLevel m) {
    pdl_wait();
    if (merge_failed(m)) return;
    const ContentTable at{(Slot*)m.slots, m.cap};
    if (blockIdx.x == 0 && threadIdx.x == 0) m.aoff[m.ga + m.totals[0]] = m.Ga + m.totals[1];
    for (u32 j = blockIdx.x * blockDim.x + threadIdx.x; j < m.kb; j += gridDim.x * blockDim.x)
        if (m.c_level[j] == m.level) {
            const u32 r = m.c_rank[j];
            m.c_out[j] = m.miss[r] ? (u32)(m.ga + m.xrank[r]) : m.M[r];
        }
    for_rules(m.boff, 0, m.gb, blockIdx.x, gridDim.x,
              [&](u64 r, u64 s, u64 len) {
                  if (!m.miss[r]) return;
                  const u64 nr = m.ga + m.xrank[r], o = m.Ga + m.xlen[r];
                  m.aoff[nr] = o;
                  m.aF[nr] = m.bF[r];
                  m.M[r] = (u32)nr;
                  for (u64 x = 0; x < len; x++) m.arhs[o + x] = merge_sym<kByte>(m, s + x);
                  table_put(at, rank_key<kByte>([&](u64 j) { return merge_sym<kByte>(m, s + j); }, len, m.aFprev,
                                                m.lh.c, nr),
                            nr, m.ds);
              },
              [&](u64 r, u64 s, u64 len) {
                  if (!m.miss[r]) return;  // (the same for the whole warp)
                  const u32 lane = threadIdx.x & 31;
                  const u64 nr = m.ga + m.xrank[r], o = m.Ga + m.xlen[r];
                  for (u64 x = lane; x < len; x += 32) m.arhs[o + x] = merge_sym<kByte>(m, s + x);
                  const u64 H = warp_poly61([&](u64 j) -> u64 { return m.aFprev[merge_sym<kByte>(m, s + j)]; },
                                            len, m.lh.c);
                  if (lane == 0) {
                      m.aoff[nr] = o;
                      m.aF[nr] = m.bF[r];
                      m.M[r] = (u32)nr;
                      table_put(at, key_hashed(H, len, nr), nr, m.ds);
                  }
              });
}

// --------------------------------------------------------------------------
// the small levels of a merge: all of them in one cooperative launch
// --------------------------------------------------------------------------
//
// Launch by launch a level of a few thousand rules takes eight launches and copies in
// a row, 45 us, whatever its size; two grammars of 3.5 M rules have eleven such levels
// of 15.  Here G_a's tables and grown arrays of all of them are filled at once, and a
// level then takes two barriers: each block looks its part of G_b's rules up and
// counts what is new, then appends it after what the blocks before it counted.
// All eleven in 231 us (32768 rules a level at most, both grammars together: 2.48 ms
// for importing, merging and exporting the two, 131072: 2.42, 262144: 2.40, 655360:
// 2.40, none: 2.64).

constexpr u32 kNoRank = 0xffffffffu;

template <bool kByte>
__device__ __forceinline__ void merge_build(const MergeLevel& m) {
    const ContentTable t{(Slot*)m.slots, m.cap};
    for_rules(m.aoff, 0, m.ga, blockIdx.x, gridDim.x,
              [&](u64 r, u64 s, u64 len) {
                  table_put(t, rank_key<kByte>([&](u64 j) { return m.arhs[s + j]; }, len, m.aFprev, m.lh.c, r), r, m.ds);
              },
              [&](u64 r, u64 s, u64 len) {
                  const u64 H = warp_poly61([&](u64 j) -> u64 { return m.aFprev[m.arhs[s + j]]; }, len, m.lh.c);
                  if ((threadIdx.x & 31) == 0) table_put(t, key_hashed(H, len, r), r, m.ds);
              });
}

// Part `block` of G_b's rules: M[r] their ranks, kNoRank for new ones, whose number and
// symbols go to counts[2 block], counts[2 block + 1].
template <bool kByte>
__device__ __forceinline__ void merge_part_lookup(const MergeLevel& m, u64 lo, u64 hi, u64* counts) {
    u64 n = 0, G = 0;
    merge_lookup<kByte>(m, lo, hi, 0, 1, [&](u64 r, u64 len, u64 found) {
        if (found != ~0ull) {
            if (m.aF[found] != m.bF[r]) set_error(m.ds, kErrMismatch);
        } else {
            n++;
            G += len;
        }
        m.M[r] = found == ~0ull ? kNoRank : (u32)found;
    });
    u64 tn, tG;
    block_excl_scan(n, tn);
    block_excl_scan(G, tG);
    if (threadIdx.x == 0) {
        counts[2 * blockIdx.x] = tn;
        counts[2 * blockIdx.x + 1] = tG;
    }
}

template <bool kByte>
__device__ __forceinline__ void merge_part_append(const MergeLevel& m, u64 lo, u64 hi, const u64* counts, u64* totals) {
    const u32 lane = threadIdx.x & 31;
    const ContentTable at{(Slot*)m.slots, m.cap};
    u64 bn = 0, bG = 0, an = 0, aG = 0;  // new rules and symbols before this part, and in all
    for (u32 b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
        const u64 x = counts[2 * b], y = counts[2 * b + 1];
        an += x;
        aG += y;
        if (b < blockIdx.x) bn += x, bG += y;
    }
    u64 t;
    block_excl_scan(bn, t);
    u64 nr0 = m.ga + t;
    block_excl_scan(bG, t);
    u64 o0 = m.Ga + t;
    block_excl_scan(an, t);
    an = t;
    block_excl_scan(aG, t);
    aG = t;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        totals[0] = an;
        totals[1] = aG;
        m.aoff[m.ga + an] = m.Ga + aG;
    }
    for (u64 base = lo; base < hi; base += blockDim.x) {
        const u64 r = base + threadIdx.x;
        const bool miss = r < hi && m.M[r] == kNoRank;
        const u64 s = miss ? m.boff[r] : 0, len = miss ? m.boff[r + 1] - s : 0;
        u64 tot;  // lengths are below 2^28, new rules of a turn at most 1024
        const u64 e = block_excl_scan(len << 16 | (miss ? 1u : 0u), tot);
        const u64 nr = nr0 + (e & 0xffffu), o = o0 + (e >> 16);
        if (miss) {
            m.aoff[nr] = o;
            m.aF[nr] = m.bF[r];
            m.M[r] = (u32)nr;
            if (len <= kRuleLong) {
                for (u64 x = 0; x < len; x++) m.arhs[o + x] = merge_sym<kByte>(m, s + x);
                table_put(at, rank_key<kByte>([&](u64 j) { return merge_sym<kByte>(m, s + j); }, len, m.aFprev, m.lh.c,
                                              nr),
                          nr, m.ds);
            }
        }
        __syncwarp();
        for (unsigned q = __ballot_sync(0xffffffffu, len > kRuleLong); q; q &= q - 1) {
            const int l = __ffs(q) - 1;
            const u64 ws = __shfl_sync(0xffffffffu, s, l), wl = __shfl_sync(0xffffffffu, len, l),
                      wo = __shfl_sync(0xffffffffu, o, l), wr = __shfl_sync(0xffffffffu, nr, l);
            for (u64 x = lane; x < wl; x += 32) m.arhs[wo + x] = merge_sym<kByte>(m, ws + x);
            const u64 H = warp_poly61([&](u64 j) -> u64 { return m.aFprev[merge_sym<kByte>(m, ws + j)]; }, wl, m.lh.c);
            if (lane == 0) table_put(at, key_hashed(H, wl, wr), wr, m.ds);
            __syncwarp();
        }
        nr0 += tot & 0xffffu;
        o0 += tot >> 16;
    }
}

__global__ void __launch_bounds__(kMergeSmallThreads) k_merge_small(const __grid_constant__ MergeSmall a) {
    pdl_wait();
    u64 barriers = 0;
    const u64 t0 = (u64)blockIdx.x * blockDim.x + threadIdx.x, stride = (u64)gridDim.x * blockDim.x;
    for (u32 i = 0; i < a.levels; i++) {
        const MergeLevel& m = a.lv[i];
        const MergeOld& o = a.old[i];
        if (o.off != nullptr) {
            for (u64 x = t0; x <= m.ga; x += stride) m.aoff[x] = o.off[x];
            for (u64 x = t0; x < m.ga; x += stride) m.aF[x] = o.F[x];
        }
        if (o.first && t0 == 0) m.aoff[0] = 0;
        if (o.rhs != nullptr)
            for (u64 x = t0; x < m.Ga; x += stride) m.arhs[x] = o.rhs[x];
        if (o.fresh)
            for (u64 x = t0; x < 2 * m.cap; x += stride)
                reinterpret_cast<uint4*>(m.slots)[x] = make_uint4(~0u, ~0u, ~0u, ~0u);
    }
    DevStatus* const ds = a.lv[0].ds;
    if (merge_failed(a.lv[0])) return;  // (by an earlier launch: the same for every block)
    grid_barrier(a.bar, barriers++, ds);
    for (u32 i = 0; i < a.levels; i++) {
        const MergeLevel& m = a.lv[i];
        if (!a.old[i].fresh) continue;
        if (m.level == 1) merge_build<true>(m);
        else merge_build<false>(m);
    }
    grid_barrier(a.bar, barriers++, ds);
    for (u32 i = 0; i < a.levels; i++) {
        const MergeLevel& m = a.lv[i];
        const u64 part = (m.gb + gridDim.x - 1) / gridDim.x;
        const u64 lo = min(m.gb, blockIdx.x * part), hi = min(m.gb, lo + part);
        if (m.level == 1) merge_part_lookup<true>(m, lo, hi, a.counts);
        else merge_part_lookup<false>(m, lo, hi, a.counts);
        grid_barrier(a.bar, barriers++, ds);
        if (m.level == 1) merge_part_append<true>(m, lo, hi, a.counts, a.totals[i]);
        else merge_part_append<false>(m, lo, hi, a.counts, a.totals[i]);
        grid_barrier(a.bar, barriers++, ds);
    }
    const u32 kb = a.lv[0].kb;
    for (u64 j = t0; j < kb; j += stride) {
        const u32 lvl = a.lv[0].c_level[j];
        if (lvl >= a.lv[0].level)
            for (u32 i = 0; i < a.levels; i++)
                if (a.lv[i].level == lvl) a.lv[0].c_out[j] = a.lv[i].M[a.lv[0].c_rank[j]];
    }
}

// F^0[s] = h^0(s) = ((a_0 s + b_0) mod p) mod m for every byte s (Sec. 3.2).
__global__ void k_h0(LevelHash h0, u32* __restrict__ F0) {
    pdl_wait();
    const u32 s = threadIdx.x;
    if (s < 256) F0[s] = (u32)(addmod61(mulmod61(h0.a, (u64)s), h0.b) & h0.mmask);
}

cudaError_t launch_h0(LevelHash h0, u32* F0, cudaStream_t st) {
    return launch_pdl(k_h0, 1, 256, st, h0, F0);
}

// The entry of a list whose blocks (from blk0 on, ascending) contain block b.
template <typename T>
__device__ __forceinline__ u32 owner_of(const T* list, u32 n, u64 b) {
    u32 lo = 0, hi = n - 1;
    while (lo < hi) {
        const u32 mid = (lo + hi + 1) / 2;
        if (list[mid].blk0 <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// A grammar's columns copied in one launch: as copies of their own, 2 us each
// however short, the 17 of a grammar of 15 levels took 50 us.
constexpr u32 kCopyEach = 16;  // words per thread
__global__ void __launch_bounds__(256) k_copy_cols(const CopyCol* __restrict__ cols, u32 ncols) {
    pdl_wait();
    const CopyCol c = cols[owner_of(cols, ncols, blockIdx.x)];
    const u64 x0 = (blockIdx.x - c.blk0) * (256ull * kCopyEach);
    const u32 m = (u32)min((u64)256 * kCopyEach, c.n - x0);
    if (c.pad && x0 == 0 && threadIdx.x == 0) c.dst[c.n] = 0;
    if (((reinterpret_cast<uintptr_t>(c.dst) | reinterpret_cast<uintptr_t>(c.src)) & 7) == 0) {
        // (x0 is even: pairs stay aligned)
        for (u32 x = threadIdx.x; x < m / 2; x += 256)
            reinterpret_cast<uint2*>(c.dst + x0)[x] = __ldg(reinterpret_cast<const uint2*>(c.src + x0) + x);
        if (threadIdx.x == 0 && (m & 1)) c.dst[x0 + m - 1] = c.src[x0 + m - 1];
    } else {
        for (u32 x = threadIdx.x; x < m; x += 256) c.dst[x0 + x] = __ldg(c.src + x0 + x);
    }
}

u64 copy_blocks(u64 n) { return (n + 256 * kCopyEach - 1) / (256 * kCopyEach); }

cudaError_t launch_copy_cols(const CopyCol* cols, u32 ncols, u64 blocks, cudaStream_t st) {
    if (blocks == 0) return cudaSuccess;
    return launch_pdl(k_copy_cols, (unsigned)blocks, 256, st, cols, ncols);
}

// Imported rules: F^i[r] must be h^i of the rule's right-hand side
// (Eq. fast_hash over F^{i-1}); a difference means the grammar was built with
// another hash family (or was altered).  All levels in one launch: block b has
// 256 rules of the level whose blocks start at blk0 <= b.
__global__ void __launch_bounds__(256) k_check_fp(const FpLevel* __restrict__ lv, u32 nl, DevStatus* ds) {
    pdl_wait();
    if (vload(&ds->error) != 0) return;  // (a malformed stream: an earlier launch's)
    const FpLevel L = lv[owner_of(lv, nl, blockIdx.x)];
    for_rules(L.off, 0, L.g, blockIdx.x - L.blk0, 1ull << 32,
              [&](u64 r, u64 s, u64 len) {
                  const u64 H = rule_poly([&](u64 j) { return __ldg(L.rhs + s + j); }, len, L.Fprev, L.lh.c);
                  if (finish_hash(L.lh, H) != L.F[r]) set_error(ds, kErrMismatch);
              },
              [&](u64 r, u64 s, u64 len) {
                  const u64 H =
                      warp_poly61([&](u64 j) -> u64 { return __ldg(L.Fprev + __ldg(L.rhs + s + j)); }, len, L.lh.c);
                  if ((threadIdx.x & 31) == 0 && finish_hash(L.lh, H) != L.F[r]) set_error(ds, kErrMismatch);
              });
}

cudaError_t launch_check_fp(const FpLevel* lv, u32 nl, u64 blocks, DevStatus* ds, cudaStream_t st) {
    if (blocks == 0) return cudaSuccess;
    return launch_pdl(k_check_fp, (unsigned)blocks, 256, st, lv, nl, ds);
}

// Root of strings j0 .. j0+cnt-1: C[j] = (level, rank) and the fingerprint
// F^level[rank] of exp(T_j) (Eq. fast_hash: it depends on the content only).
__global__ void k_roots(const u32* __restrict__ c_level, const u32* __restrict__ c_rank, u32 j0, u32 cnt, FTable ft,
                        u32* __restrict__ out) {
    for (u32 x = blockIdx.x * blockDim.x + threadIdx.x; x < cnt; x += gridDim.x * blockDim.x) {
        const u32 lvl = c_level[j0 + x], r = c_rank[j0 + x];
        out[3 * x] = lvl;
        out[3 * x + 1] = r;
        out[3 * x + 2] = lvl < ft.n ? __ldg(ft.F[lvl] + r) : 0u;
    }
}

cudaError_t launch_roots(const u32* c_level, const u32* c_rank, u32 j0, u32 cnt, const FTable& ft, u32* out,
                         cudaStream_t st) {
    if (cnt == 0) return cudaSuccess;
    k_roots<<<(cnt + 255) / 256 < 1024 ? (cnt + 255) / 256 : 1024, 256, 0, st>>>(c_level, c_rank, j0, cnt, ft, out);
    return cudaGetLastError();
}

static unsigned grid_for(u64 n, unsigned cap = 152 * 32) {
    u64 b = (n + 255) / 256;
    if (b == 0) b = 1;
    return (unsigned)(b < cap ? b : cap);
}

cudaError_t launch_resident_build(const u32* rhs, const u64* rhs_off, u64 r0, u64 cnt, bool bytes, const u32* Fprev,
                                  LevelHash lh, void* slots, u64 cap, DevStatus* ds, cudaStream_t st) {
    if (cnt == 0) return cudaSuccess;
    const ContentTable t{(Slot*)slots, cap};
    return launch_pdl(bytes ? k_resident_build<true> : k_resident_build<false>, grid_for(cnt), 256, st, rhs, rhs_off,
                      r0, cnt, Fprev, lh, t, ds);
}

cudaError_t launch_merge_lookup(const MergeLevel& m, bool bytes, cudaStream_t st) {
    if (m.gb == 0) return cudaSuccess;
    return launch_pdl(bytes ? k_merge_lookup<true> : k_merge_lookup<false>, grid_for(m.gb), 256, st, m);
}

cudaError_t launch_merge_small(const MergeSmall& a, u32 blocks, cudaStream_t st) {
    return launch_coop(k_merge_small, blocks, kMergeSmallThreads, 0, st, a);
}

cudaError_t launch_merge_append(const MergeLevel& m, bool bytes, cudaStream_t st) {
    if (m.gb == 0) return cudaSuccess;
    return launch_pdl(bytes ? k_merge_append<true> : k_merge_append<false>, grid_for(m.gb), 256, st, m);
}

// --------------------------------------------------------------------------
// exp(C[j]): top-down expansion, one level per step
// --------------------------------------------------------------------------
//
// A short expansion (every level of at most kExpandSmall symbols) is one block's,
// all levels in one launch, its symbols in shared memory.  A longer one goes on
// from there level by level: k_expand_count and a scan give the tiles' places
// (and the host the length of the next sequence), and k_expand_tiles copies the
// right-hand sides and, at level 1, writes the bytes themselves.  Before, a
// level took three kernels (lengths, scan, copy) with the lengths and their
// 64-bit offsets in between, and the last level's symbols were written as words
// and then narrowed: 4 x 200 Mbp 14.1 ms of kernels, and 0.39 ms for a string
// of 20 kB, whose ten levels each waited for the host.

constexpr int kExpThreads = 1024;
constexpr u64 kExpandCopyAlone = 32;  // rules up to this length are copied by one thread

// Rules too long for one thread, listed for the block.
struct LongCopy {
    u64 src, dst;
    u32 len;
};
constexpr u32 kLongCopies = 512;

struct ExpandSmem {
    u32 sym[2][kExpandSmall];
    LongCopy longs[kLongCopies];
    u32 nlong;
};

__global__ void __launch_bounds__(kExpThreads) k_expand_small(const __grid_constant__ ExpandLevels lv,
                                                              const u32* __restrict__ c_level,
                                                              const u32* __restrict__ c_rank, u32 j,
                                                              unsigned char* __restrict__ out, u64 cap,
                                                              u32* __restrict__ rest, ExpandState* state) {
    extern __shared__ __align__(16) unsigned char exp_smem[];
    ExpandSmem& sm = *reinterpret_cast<ExpandSmem*>(exp_smem);
    constexpr u32 kPer = kExpandSmall / kExpThreads;  // symbols per thread
    u32 level = c_level[j], cnt = 1, cur = 0;
    if (threadIdx.x == 0) sm.sym[0][0] = c_rank[j];
    __syncthreads();
    u64 total = 1;
    bool done = level == 0;
    while (level >= 1) {
        const u64* __restrict__ off = lv.off[level - 1];
        const u32* __restrict__ rhs = lv.rhs[level - 1];
        const u32* src = sm.sym[cur];
        u32* dst = sm.sym[cur ^ 1];
        if (threadIdx.x == 0) sm.nlong = 0;
        // consecutive symbols per thread, as few as cover the sequence
        const u32 per = (cnt + kExpThreads - 1) / kExpThreads;
        const u32 x0 = threadIdx.x * per;
        u64 from[kPer];
        u32 len[kPer];
        u64 sum = 0;
#pragma unroll
        for (u32 i = 0; i < kPer; i++) {
            const u32 x = x0 + i;
            from[i] = 0;
            len[i] = 0;
            if (i < per && x < cnt) {
                const u32 r = src[x];
                from[i] = off[r];
                len[i] = (u32)(off[r + 1] - from[i]);
            }
        }
#pragma unroll
        for (u32 i = 0; i < kPer; i++) sum += len[i];
        u64 o = block_excl_scan(sum, total);
        const bool bytes = level == 1;
        if (bytes ? (total > kExpandSmallBytes || total > cap) : total > (u64)kExpandSmall) break;
        auto put = [&](u64 at, u32 v) {
            if (bytes) out[at] = (unsigned char)v;
            else dst[at] = v;
        };
#pragma unroll
        for (u32 i = 0; i < kPer; i++) {
            if (len[i] > kExpandCopyAlone) {
                const u32 l = atomicAdd(&sm.nlong, 1u);
                if (l < kLongCopies) {
                    sm.longs[l] = LongCopy{from[i], o, len[i]};
                    o += len[i];
                    continue;
                }
            }
            for (u32 y = 0; y < len[i]; y++) put(o + y, __ldg(rhs + from[i] + y));
            o += len[i];
        }
        __syncthreads();
        const u32 nl = min(sm.nlong, kLongCopies);
        for (u32 l = 0; l < nl; l++) {
            const LongCopy c = sm.longs[l];
            for (u32 y = threadIdx.x; y < c.len; y += kExpThreads) put(c.dst + y, __ldg(rhs + c.src + y));
        }
        __syncthreads();
        cur ^= 1;
        cnt = (u32)total;
        level--;
        done = level == 0;
    }
    if (done && c_level[j] == 0 && cap >= 1 && threadIdx.x == 0) out[0] = (unsigned char)sm.sym[0][0];
    if (!done)
        for (u32 x = threadIdx.x; x < cnt; x += kExpThreads) rest[x] = sm.sym[cur][x];
    if (threadIdx.x == 0) {
        state->count = cnt;
        state->level = level;
        state->which = 2;
    }
}

// The levels after that, down to level 2, while they have at most kExpandMid symbols:
// one cooperative launch, two grid barriers a level.  A block counts what its part of
// the sequence expands to, then copies it after what the blocks before it counted.
// Level by level each of them took three launches and a wait of the host, some 41 us for
// 10 us of work (4 x 200 Mbp, six such levels a string: 4.89 ms, now 4.46).
constexpr int kEmThreads = 512;

__global__ void __launch_bounds__(kEmThreads) k_expand_mid(const __grid_constant__ ExpandLevels lv, const u32* first,
                                                           u32* mid, u64* counts, u64* bar, ExpandState* state,
                                                           DevStatus* ds) {
    pdl_wait();
    const u32 lane = threadIdx.x & 31;
    u32 level = state->level, which = 2;  // of mid's two halves, or `first`
    u64 cnt = state->count, barriers = 0;
    const u32* src = first;
    while (level >= 2) {
        const u64* __restrict__ off = lv.off[level - 1];
        const u32* __restrict__ rhs = lv.rhs[level - 1];
        const u64 part = (cnt + gridDim.x - 1) / gridDim.x;
        const u64 lo = min(cnt, blockIdx.x * part), hi = min(cnt, lo + part);
        u64 sum = 0, t;
        for (u64 x = lo + threadIdx.x; x < hi; x += kEmThreads) {
            const u32 r = src[x];
            sum += __ldg(off + r + 1) - __ldg(off + r);
        }
        block_excl_scan(sum, t);
        if (threadIdx.x == 0) counts[blockIdx.x] = t;
        grid_barrier(bar, barriers++, ds);
        u64 before = 0, all = 0;
        for (u32 b = threadIdx.x; b < gridDim.x; b += kEmThreads) {
            const u64 c = vload(counts + b);
            all += c;
            if (b < blockIdx.x) before += c;
        }
        block_excl_scan(before, t);
        u64 o0 = t;
        block_excl_scan(all, t);
        const u64 total = t;
        if (total > kExpandMid) break;  // (the same for every block)
        which = which == 0 ? 1 : 0;
        u32* dst = mid + which * kExpandMid;
        for (u64 base = lo; base < hi; base += kEmThreads) {
            const u64 x = base + threadIdx.x;
            u64 from = 0;
            u32 len = 0;
            if (x < hi) {
                const u32 r = src[x];
                from = __ldg(off + r);
                len = (u32)(__ldg(off + r + 1) - from);
            }
            const u64 o = o0 + block_excl_scan((u64)len, t);
            o0 += t;
            if (len <= (u32)kExpandCopyAlone) {
                for (u32 y = 0; y < len; y += 4) {
                    u32 v[4];
#pragma unroll
                    for (u32 u = 0; u < 4; u++) v[u] = y + u < len ? __ldg(rhs + from + y + u) : 0u;
#pragma unroll
                    for (u32 u = 0; u < 4; u++)
                        if (y + u < len) dst[o + y + u] = v[u];
                }
            }
            __syncwarp();
            for (unsigned q = __ballot_sync(0xffffffffu, len > (u32)kExpandCopyAlone); q; q &= q - 1) {
                const int l = __ffs(q) - 1;
                const u64 wf = __shfl_sync(0xffffffffu, from, l), wo = __shfl_sync(0xffffffffu, o, l);
                const u32 wl = __shfl_sync(0xffffffffu, len, l);
                for (u32 y = lane; y < wl; y += 32) dst[wo + y] = __ldg(rhs + wf + y);
            }
        }
        grid_barrier(bar, barriers++, ds);
        src = dst;
        cnt = total;
        level--;
    }
    if (barriers > 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        state->count = cnt;
        state->level = level;
        state->which = which;
    }
}

constexpr int kEtThreads = 256;
constexpr int kEtItems = 4;
constexpr int kEtTile = kEtThreads * kEtItems;

// Symbols [x0, x0 + kEtItems) of cur and their rules' places: from[i], len[i] (0
// past the end).
__device__ __forceinline__ void et_load(const u32* __restrict__ cur, u64 cnt, const u64* __restrict__ off, u64 x0,
                                        u64 (&from)[kEtItems], u32 (&len)[kEtItems]) {
    u32 r[kEtItems];
    if (x0 + kEtItems <= cnt) {  // (cur is 16-byte aligned: an allocation of its own)
#pragma unroll
        for (int q = 0; q < kEtItems / 4; q++) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(cur + x0) + q);
            r[4 * q] = v.x, r[4 * q + 1] = v.y, r[4 * q + 2] = v.z, r[4 * q + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kEtItems; i++) r[i] = x0 + i < cnt ? cur[x0 + i] : 0u;
    }
#pragma unroll
    for (int i = 0; i < kEtItems; i++) {
        const bool in = x0 + i < cnt;
        from[i] = in ? __ldg(off + r[i]) : 0ull;
        len[i] = in ? (u32)(__ldg(off + r[i] + 1) - from[i]) : 0u;
    }
}

// The symbols that each tile of kEtTile symbols expands to: their low and high
// halves (k_scan2 makes them the tiles' places).
__global__ void __launch_bounds__(kEtThreads) k_expand_count(const u32* __restrict__ cur, u64 cnt,
                                                             const u64* __restrict__ off, u32* __restrict__ lo,
                                                             u32* __restrict__ hi) {
    __shared__ u64 s_w[kEtThreads / 32];
    u64 from[kEtItems];
    u32 len[kEtItems];
    et_load(cur, cnt, off, blockIdx.x * (u64)kEtTile + (u64)threadIdx.x * kEtItems, from, len);
    u64 s = 0;
#pragma unroll
    for (int i = 0; i < kEtItems; i++) s += len[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        u64 t = 0;
        for (int w = 0; w < kEtThreads / 32; w++) t += s_w[w];
        lo[blockIdx.x] = (u32)t;
        hi[blockIdx.x] = (u32)(t >> 32);
    }
}

// One level of an expansion: a block scans the lengths of a tile's symbols, copies
// their right-hand sides to shared memory as they will lie in the output (to
// within 16 bytes) and stores them with 16-byte stores.  A tile that does not
// fit there (long rules) is copied straight to the output; rules too long for
// one thread are copied by the whole block.  Out: u32 symbols of the level
// below, or bytes.  The tiles' places are scanned beforehand: with a look-back
// in this kernel its blocks waited for one another (4 x 200 Mbp: 9.6 ms; now
// 2.6 ms, with the count's 0.8 ms and the scan's 0.2 ms).  Four symbols per
// thread and 64 registers: with eight and 116, 5.6 ms in all, now 3.8.
constexpr u32 kEtStageBytes = 18 * 1024;
constexpr u32 kEtLongs = 256;
constexpr u32 kEtBatch = 4;  // symbols of a rule read together

// In is u32 (the level's right-hand sides) or, at level 1 of a long string, u8 (the
// same packed by k_expand_pack: a rule of up to 8 bytes is three 4-byte reads).
template <typename In, typename Out>
__global__ void __launch_bounds__(kEtThreads, 4) k_expand_tiles(const u32* __restrict__ cur, u64 cnt,
                                                             const u64* __restrict__ off,
                                                             const In* __restrict__ rhs,
                                                             const u64* __restrict__ lo, const u64* __restrict__ hi,
                                                             Out* __restrict__ out) {
    constexpr u32 kStage = (sizeof(Out) == 1 ? kEtStageBytes / 3 : kEtStageBytes) / sizeof(Out);
    __shared__ __align__(16) Out stage[kStage];
    __shared__ LongCopy s_long[kEtLongs];
    __shared__ u32 s_nlong;
    if (threadIdx.x == 0) s_nlong = 0;
    const u64 place = lo[blockIdx.x] + (hi[blockIdx.x] << 32);
    u64 from[kEtItems];
    u32 len[kEtItems];
    et_load(cur, cnt, off, blockIdx.x * (u64)kEtTile + (u64)threadIdx.x * kEtItems, from, len);
    u64 sum = 0;
#pragma unroll
    for (int i = 0; i < kEtItems; i++) sum += len[i];
    // the first symbols of every rule are read before the scan
    constexpr bool kPacked = sizeof(In) == 1;
    constexpr u32 kFirst = kPacked ? 8 : kEtBatch;  // symbols of them
    u32 v[kEtItems][kPacked ? 3 : kEtBatch];
#pragma unroll
    for (int i = 0; i < kEtItems; i++) {
        if constexpr (kPacked) {
            const u32* w = reinterpret_cast<const u32*>(rhs) + (from[i] >> 2);
            const u32 end = ((u32)from[i] & 3u) + len[i];  // bytes from the word's start
            v[i][0] = len[i] ? __ldg(w) : 0u;
            v[i][1] = end > 4 ? __ldg(w + 1) : 0u;
            v[i][2] = end > 8 ? __ldg(w + 2) : 0u;
        } else {
#pragma unroll
            for (u32 y = 0; y < kEtBatch; y++) v[i][y] = y < len[i] ? (u32)__ldg(rhs + from[i] + y) : 0u;
        }
    }
    u64 total;
    u64 o = block_excl_scan(sum, total);
    Out* dst = out + place;
    constexpr u32 kPer16 = 16 / sizeof(Out);
    // the output's place within its 16 bytes
    const u32 skew = (u32)((reinterpret_cast<unsigned long long>(dst) & 15) / sizeof(Out));
    const bool staged = total + skew <= (u64)kStage;  // the same for the whole block
    Out* to = staged ? stage + skew : dst;
#pragma unroll
    for (int i = 0; i < kEtItems; i++) {
        bool listed = false;
        if (len[i] > (u32)kExpandCopyAlone) {
            const u32 l = atomicAdd(&s_nlong, 1u);
            listed = l < kEtLongs;
            if (listed) s_long[l] = LongCopy{from[i], o, len[i]};
        }
        if (!listed) {
            if constexpr (kPacked) {
                const u32 sh = ((u32)from[i] & 3u) * 8;
                const u64 b = ((u64)__funnelshift_r(v[i][1], v[i][2], sh) << 32) | __funnelshift_r(v[i][0], v[i][1], sh);
#pragma unroll
                for (u32 y = 0; y < kFirst; y++)
                    if (y < len[i]) to[o + y] = (Out)(b >> (8 * y));
            } else {
#pragma unroll
                for (u32 y = 0; y < kFirst; y++)
                    if (y < len[i]) to[o + y] = (Out)v[i][y];
            }
            for (u32 y = kFirst; y < len[i]; y++) to[o + y] = (Out)__ldg(rhs + from[i] + y);
        }
        o += len[i];
    }
    __syncthreads();
    const u32 nl = min(s_nlong, kEtLongs);
    for (u32 l = 0; l < nl; l++) {
        const LongCopy c = s_long[l];
        for (u32 y = threadIdx.x; y < c.len; y += kEtThreads) to[c.dst + y] = (Out)__ldg(rhs + c.src + y);
    }
    if (!staged) return;
    __syncthreads();
    // whole 16-byte words; the first and the last, shared with other tiles, by entries
    const u32 end = skew + (u32)total;
    Out* base = dst - skew;  // 16-byte aligned
    const u32 w0 = (skew + kPer16 - 1) / kPer16, w1 = end / kPer16;
    for (u32 w = w0 + threadIdx.x; w < w1; w += kEtThreads)
        reinterpret_cast<uint4*>(base)[w] = reinterpret_cast<const uint4*>(stage)[w];
    const u32 head = min(w0 * kPer16, end);
    for (u32 x = skew + threadIdx.x; x < head; x += kEtThreads) base[x] = stage[x];
    for (u32 x = max(w1 * kPer16, head) + threadIdx.x; x < end; x += kEtThreads) base[x] = stage[x];
}

cudaError_t launch_expand_small(const ExpandLevels& lv, const u32* c_level, const u32* c_rank, u32 j,
                                unsigned char* out, u64 cap, u32* rest, ExpandState* state, cudaStream_t st) {
    static PerDevice<bool> raised;  // (the limit of dynamic shared memory is each device's own)
    int dev = 0;
    bool set = false;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = raised.get(dev, set, [](bool& b) {
            b = true;
            return cudaFuncSetAttribute(k_expand_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)sizeof(ExpandSmem));
        });
    if (e != cudaSuccess) return e;
    k_expand_small<<<1, kExpThreads, sizeof(ExpandSmem), st>>>(lv, c_level, c_rank, j, out, cap, rest, state);
    return cudaGetLastError();
}

cudaError_t launch_expand_mid(const ExpandLevels& lv, const u32* first, u32* mid, u64* counts, u64* bar,
                              ExpandState* state, DevStatus* ds, u32 blocks, cudaStream_t st) {
    return launch_coop(k_expand_mid, blocks, kEmThreads, 0, st, lv, first, mid, counts, bar, state, ds);
}

u64 expand_tiles_for(u64 cnt) { return std::max<u64>(1, (cnt + kEtTile - 1) / kEtTile); }

cudaError_t launch_expand_count(const u32* cur, u64 cnt, const u64* off, u32* lo, u32* hi, cudaStream_t st) {
    k_expand_count<<<(unsigned)expand_tiles_for(cnt), kEtThreads, 0, st>>>(cur, cnt, off, lo, hi);
    return cudaGetLastError();
}

cudaError_t launch_expand_tiles(const u32* cur, u64 cnt, const u64* off, const u32* rhs, const u8* packed,
                                const u64* lo, const u64* hi, u32* next, u8* bytes, cudaStream_t st) {
    const unsigned g = (unsigned)expand_tiles_for(cnt);
    if (packed) k_expand_tiles<u8, u8><<<g, kEtThreads, 0, st>>>(cur, cnt, off, packed, lo, hi, bytes);
    else if (bytes) k_expand_tiles<u32, u8><<<g, kEtThreads, 0, st>>>(cur, cnt, off, rhs, lo, hi, bytes);
    else k_expand_tiles<u32, u32><<<g, kEtThreads, 0, st>>>(cur, cnt, off, rhs, lo, hi, next);
    return cudaGetLastError();
}

// The n bytes that level 1's right-hand sides hold as words.
__global__ void __launch_bounds__(256) k_expand_pack(const u32* __restrict__ rhs, u64 n, u8* __restrict__ out) {
    for (u64 x = 4 * (blockIdx.x * 256ull + threadIdx.x); x < n; x += 4 * 256ull * gridDim.x) {
        u32 w = 0;
#pragma unroll
        for (int i = 0; i < 4; i++) w |= (x + i < n ? __ldg(rhs + x + i) & 0xFFu : 0u) << (8 * i);
        reinterpret_cast<u32*>(out)[x >> 2] = w;
    }
}

cudaError_t launch_expand_pack(const u32* rhs, u64 n, u8* out, cudaStream_t st) {
    k_expand_pack<<<(unsigned)std::min<u64>((n + 1023) / 1024 + 1, 152 * 16), 256, 0, st>>>(rhs, n, out);
    return cudaGetLastError();
}

// The steps of lcg_decompress_static, which brings its own scratch.
__global__ void k_rule_lens(const u32* __restrict__ cur, u64 cnt, const u64* __restrict__ rhs_off,
                            u32* __restrict__ lens) {
    for (u64 x = blockIdx.x * (u64)blockDim.x + threadIdx.x; x < cnt; x += (u64)gridDim.x * blockDim.x) {
        const u32 r = cur[x];
        lens[x] = (u32)(rhs_off[r + 1] - rhs_off[r]);
    }
}

__global__ void k_expand(const u32* __restrict__ cur, u64 cnt, const u64* __restrict__ offs,
                         const u64* __restrict__ rhs_off, const u32* __restrict__ rhs, u32* __restrict__ next) {
    for (u64 x = blockIdx.x * (u64)blockDim.x + threadIdx.x; x < cnt; x += (u64)gridDim.x * blockDim.x) {
        const u32 r = cur[x];
        const u64 s = rhs_off[r], e = rhs_off[r + 1], o = offs[x];
        for (u64 y = s; y < e; y++) next[o + (y - s)] = rhs[y];
    }
}

__global__ void k_to_bytes(const u32* __restrict__ cur, u64 cnt, unsigned char* __restrict__ out) {
    for (u64 x = blockIdx.x * (u64)blockDim.x + threadIdx.x; x < cnt; x += (u64)gridDim.x * blockDim.x)
        out[x] = (unsigned char)cur[x];
}

cudaError_t launch_rule_lens(const u32* cur, u64 cnt, const u64* rhs_off, u32* lens, cudaStream_t st) {
    k_rule_lens<<<grid_for(cnt), 256, 0, st>>>(cur, cnt, rhs_off, lens);
    return cudaGetLastError();
}

cudaError_t launch_expand(const u32* cur, u64 cnt, const u64* offs, const u64* rhs_off, const u32* rhs, u32* next,
                          cudaStream_t st) {
    k_expand<<<grid_for(cnt), 256, 0, st>>>(cur, cnt, offs, rhs_off, rhs, next);
    return cudaGetLastError();
}

cudaError_t launch_to_bytes(const u32* cur, u64 cnt, unsigned char* out, cudaStream_t st) {
    k_to_bytes<<<grid_for(cnt), 256, 0, st>>>(cur, cnt, out);
    return cudaGetLastError();
}

}  // namespace lcg
