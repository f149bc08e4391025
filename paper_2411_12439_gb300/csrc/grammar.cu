// Kernels that work on finished grammars: MergeGrams (Sec. 3.6), the
// expansion exp(C[j]) (Sec. 2.2), and a generic two-column exclusive scan.
#include "lcg_dev.cuh"
#include "lcg_internal.h"
#include "table.cuh"

namespace lcg {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
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

__global__ void __launch_bounds__(kScanThreads) k_scan2(const u32* __restrict__ in0, const u32* __restrict__ in1,
                                                        u64 n, u64* __restrict__ out0, u64* __restrict__ out1,
                                                        u64* __restrict__ totals, LBSlot<2>* lb, u64 epoch, u64* ctr,
                                                        u64 ctr_base, DevStatus* ds, const u64* n_dev) {
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
#pragma unroll
    for (int it = 0; it < kScanItems; it++) {
        const u64 p = p0 + it;
        if (p < n) {
            out0[p] = ea;
            if (out1 != nullptr) out1[p] = eb;
        }
        ea += a[it];
        eb += b[it];
    }
    if ((tile + 1) * (u64)kScanTile >= n && threadIdx.x == 0) {
        totals[0] = excl[0] + ta;
        totals[1] = excl[1] + tb;
    }
}

u64 scan2_tiles_for(u64 n) { return (n + kScanTile - 1) / kScanTile; }
size_t scan2_lb_bytes(u64 tiles) { return scan2_lb_bytes_static(tiles); }

cudaError_t launch_scan2(const u32* in0, const u32* in1, u64 n, u64* out0, u64* out1, u64* totals, void* lb,
                         u64 epoch, u64* ctr, u64 ctr_base, DevStatus* ds, cudaStream_t st, u64* grid_out,
                         const u64* n_dev) {
    u64 tiles = scan2_tiles_for(n);
    if (tiles == 0) tiles = 1;
    *grid_out = tiles;
    return launch_pdl(k_scan2, (unsigned)tiles, kScanThreads, st, in0, in1, n, out0, out1, totals, (LBSlot<2>*)lb,
                      epoch, ctr, ctr_base, ds, n_dev);
}

// --------------------------------------------------------------------------
// MergeGrams
// --------------------------------------------------------------------------

// out[x] = M[in[x]]: rewrite right-hand sides of G_b into G_a's ranks.
__global__ void k_remap(const u32* __restrict__ in, u64 n, const u32* __restrict__ M, u32* __restrict__ out) {
    for (u64 x = blockIdx.x * (u64)blockDim.x + threadIdx.x; x < n; x += (u64)gridDim.x * blockDim.x)
        out[x] = M[in[x]];
}

// For every rule of G_b (right-hand side already over G_a's ranks): its rank
// in G_a when G_a has the same right-hand side (looked up in G_a's table of
// the level, hashed keys confirmed by comparing contents), else a miss.
template <bool kByte>
__global__ void k_merge_lookup(const u32* __restrict__ brhs, const u64* __restrict__ brhs_off,
                               const u32* __restrict__ bF, u64 gb, const u32* __restrict__ aFprev, LevelHash lh,
                               ContentTable at, const u32* __restrict__ arhs, const u64* __restrict__ arhs_off,
                               const u32* __restrict__ aF, u32* __restrict__ M, u32* __restrict__ miss,
                               u32* __restrict__ mlen, DevStatus* ds) {
    for (u64 r = blockIdx.x * (u64)blockDim.x + threadIdx.x; r < gb; r += (u64)gridDim.x * blockDim.x) {
        const u64 s = brhs_off[r], e = brhs_off[r + 1], len = e - s;
        u64 H = 0;
        for (u64 x = e; x-- > s;) H = addmod61(mulmod61(H, lh.c), (u64)__ldg(aFprev + brhs[x]));
        const int w = kByte ? 8 : kRankBits;
        const bool hashed = len > inline_max(w);
        const Key128 key = hashed ? key_hashed(H, len, 0) : key_inline([&](u64 j) { return brhs[s + j]; }, len, w);
        u64 found = ~0ull;
        if (at.cap) {
            found = table_find(at, key, hashed, [&](u64 ra) {
                const u64 o = arhs_off[ra];
                if (arhs_off[ra + 1] - o != len) return false;
                for (u64 x = 0; x < len; x++)
                    if (arhs[o + x] != brhs[s + x]) return false;
                return true;
            });
        }
        if (found != ~0ull) {
            if (aF[found] != bF[r]) set_error(ds, kErrMismatch);
            M[r] = (u32)found;
            miss[r] = 0;
            mlen[r] = 0;
        } else {
            miss[r] = 1;
            mlen[r] = (u32)len;
        }
    }
}

// Append the missed rules of G_b to G_a in G_b's rank order.
__global__ void k_merge_append(const u32* __restrict__ brhs, const u64* __restrict__ brhs_off,
                               const u32* __restrict__ bF, u64 gb, const u32* __restrict__ miss,
                               const u64* __restrict__ xrank, const u64* __restrict__ xlen, u64 ga, u64 Ga,
                               u32* __restrict__ arhs, u64* __restrict__ arhs_off, u32* __restrict__ aF,
                               u32* __restrict__ M) {
    for (u64 r = blockIdx.x * (u64)blockDim.x + threadIdx.x; r < gb; r += (u64)gridDim.x * blockDim.x) {
        if (!miss[r]) continue;
        const u64 nr = ga + xrank[r], o = Ga + xlen[r];
        const u64 s = brhs_off[r], e = brhs_off[r + 1];
        arhs_off[nr] = o;
        for (u64 x = s; x < e; x++) arhs[o + (x - s)] = brhs[x];
        aF[nr] = bF[r];
        M[r] = (u32)nr;
    }
}

__global__ void k_set_u64(u64* p, u64 v) { *p = v; }

// F^0[s] = h^0(s) = ((a_0 s + b_0) mod p) mod m for every byte s (Sec. 3.2).
__global__ void k_h0(LevelHash h0, u32* __restrict__ F0) {
    pdl_wait();
    const u32 s = threadIdx.x;
    if (s < 256) F0[s] = (u32)(addmod61(mulmod61(h0.a, (u64)s), h0.b) & h0.mmask);
}

cudaError_t launch_h0(LevelHash h0, u32* F0, cudaStream_t st) {
    return launch_pdl(k_h0, 1, 256, st, h0, F0);
}

// C_b entries of level `level` move to G_a's ranks.
// Imported rules: F^i[r] must be h^i of the rule's right-hand side
// (Eq. fast_hash over F^{i-1}); a difference means the grammar was built with
// another hash family (or was altered).
__global__ void k_check_fp(const u32* __restrict__ rhs, const u64* __restrict__ rhs_off, u64 g,
                           const u32* __restrict__ Fprev, LevelHash lh, const u32* __restrict__ F, DevStatus* ds) {
    for (u64 r = blockIdx.x * (u64)blockDim.x + threadIdx.x; r < g; r += (u64)gridDim.x * blockDim.x) {
        const u64 s = rhs_off[r], e = rhs_off[r + 1];
        u64 H = 0;
        for (u64 y = e; y-- > s;) H = addmod61(mulmod61(H, lh.c), (u64)__ldg(Fprev + rhs[y]));
        if (finish_hash(lh, H) != F[r]) set_error(ds, kErrMismatch);
    }
}

cudaError_t launch_check_fp(const u32* rhs, const u64* rhs_off, u64 g, const u32* Fprev, LevelHash lh, const u32* F,
                            DevStatus* ds, cudaStream_t st) {
    if (g == 0) return cudaSuccess;
    const u64 b = (g + 255) / 256;
    k_check_fp<<<(unsigned)(b < 152 * 16 ? b : 152 * 16), 256, 0, st>>>(rhs, rhs_off, g, Fprev, lh, F, ds);
    return cudaGetLastError();
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

__global__ void k_remap_c(const u32* __restrict__ c_level, u32* __restrict__ c_rank, u32 k, u32 level,
                          const u32* __restrict__ M) {
    for (u32 j = blockIdx.x * blockDim.x + threadIdx.x; j < k; j += gridDim.x * blockDim.x)
        if (c_level[j] == level) c_rank[j] = M[c_rank[j]];
}

static unsigned grid_for(u64 n, unsigned cap = 152 * 32) {
    u64 b = (n + 255) / 256;
    if (b == 0) b = 1;
    return (unsigned)(b < cap ? b : cap);
}

cudaError_t launch_remap(const u32* in, u64 n, const u32* M, u32* out, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    k_remap<<<grid_for(n), 256, 0, st>>>(in, n, M, out);
    return cudaGetLastError();
}

cudaError_t launch_merge_lookup(const u32* brhs, const u64* brhs_off, const u32* bF, u64 gb, bool bytes,
                                const u32* aFprev, LevelHash lh, void* aslots, u64 acap, const u32* arhs,
                                const u64* arhs_off, const u32* aF, u32* M, u32* miss, u32* mlen, DevStatus* ds,
                                cudaStream_t st) {
    if (gb == 0) return cudaSuccess;
    const ContentTable at{(Slot*)aslots, acap};
    if (bytes)
        k_merge_lookup<true><<<grid_for(gb), 256, 0, st>>>(brhs, brhs_off, bF, gb, aFprev, lh, at, arhs, arhs_off, aF,
                                                           M, miss, mlen, ds);
    else
        k_merge_lookup<false><<<grid_for(gb), 256, 0, st>>>(brhs, brhs_off, bF, gb, aFprev, lh, at, arhs, arhs_off,
                                                            aF, M, miss, mlen, ds);
    return cudaGetLastError();
}

cudaError_t launch_merge_append(const u32* brhs, const u64* brhs_off, const u32* bF, u64 gb, const u32* miss,
                                const u64* xrank, const u64* xlen, u64 ga, u64 Ga, u32* arhs, u64* arhs_off,
                                u32* aF, u32* M, u64 ga_new, u64 Ga_new, cudaStream_t st) {
    if (gb > 0)
        k_merge_append<<<grid_for(gb), 256, 0, st>>>(brhs, brhs_off, bF, gb, miss, xrank, xlen, ga, Ga, arhs,
                                                     arhs_off, aF, M);
    k_set_u64<<<1, 1, 0, st>>>(arhs_off + ga_new, Ga_new);
    return cudaGetLastError();
}

cudaError_t launch_remap_c(const u32* c_level, u32* c_rank, u32 k, u32 level, const u32* M, cudaStream_t st) {
    if (k == 0) return cudaSuccess;
    k_remap_c<<<grid_for(k, 152), 256, 0, st>>>(c_level, c_rank, k, level, M);
    return cudaGetLastError();
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
    static const cudaError_t attr = cudaFuncSetAttribute(k_expand_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         (int)sizeof(ExpandSmem));
    if (attr != cudaSuccess) return attr;
    k_expand_small<<<1, kExpThreads, sizeof(ExpandSmem), st>>>(lv, c_level, c_rank, j, out, cap, rest, state);
    return cudaGetLastError();
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
