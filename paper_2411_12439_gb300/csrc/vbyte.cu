// VByte codec of the grammar's arrays (Sec. 4, resource usage: rules stored
// with VBytes instead of 32-bit cells).  A value is cut into groups of 7 bits,
// least significant group first, one group per byte; the high bit of a byte
// is set when another byte of the same value follows (the LEB128 / varint
// layout).
//
// Both directions run in three independent streaming steps, with no wait of
// one tile on another:
//   encode: k_vb_tile_bytes (stream bytes of each tile of 2048 values), an
//     exclusive scan of those counts (k_scan2), k_vb_write (each tile
//     re-reads its values, assembles its bytes in shared memory and stores
//     them at its offset with 16-byte stores, the edges byte by byte).  An
//     export needs the counts anyway to lay out its sections.
//   decode: k_vb_tile_ends (values ending in each tile of 4096 stream bytes),
//     a scan of those counts, k_vb_dwrite (every byte without the high bit
//     ends a value; a thread per value takes the bytes since the end before).
//     Malformed streams (a value of more than 32 bits or 5 bytes, a stream that
//     ends inside a value, a value outside the allowed range, another number of
//     values) set kErrFormat; no write leaves the output.
// The writing kernels are bound by instruction issue, not by memory, so they are
// laid out for few instructions per value and lanes that do the same.
// k_vb_count sizes a column without writing it (lcg_vbyte_size).
#include "lcg_dev.cuh"
#include "lcg_internal.h"

namespace lcg {

constexpr int kVbThreads = 256;
constexpr int kVbItems = 8;                         // values per thread (encode)
constexpr int kVbTile = kVbThreads * kVbItems;      // 2048 values
constexpr int kVbBytes = 16;                        // stream bytes per thread (decode)
constexpr int kVbDecTile = kVbThreads * kVbBytes;   // 4096 bytes
constexpr int kVbPer = 4;                           // tiles of a column that a counting block takes

__device__ __forceinline__ u32 vb_len(u32 v) {
    return ((38u - (u32)__clz((int)(v | 1u))) * 37u) >> 8;  // ceil(bits / 7), bits 1 .. 32
}

// Exclusive scan of one count per thread over the block (totals below 2^32), with
// one barrier; s_w may not be reused before the next one.
__device__ __forceinline__ u32 vb_block_scan(u32 x, u32* s_w, u32& total) {
    const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    u32 incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 y = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += y;
    }
    if (lane == 31) s_w[wid] = incl;
    __syncthreads();
    u32 before = 0;
    total = 0;
#pragma unroll
    for (u32 w = 0; w < kVbThreads / 32; w++) {
        const u32 t = s_w[w];
        before += w < wid ? t : 0u;
        total += t;
    }
    return before + incl - x;
}

// Sums of kVbPer counts per thread over the block, each below 2^16, to out[0 ..
// min(kVbPer, left)).
__device__ __forceinline__ void vb_block_sums(const u32 (&c)[kVbPer], u32* s_w, u64 left, u32* out) {
    static_assert(kVbPer == 4, "two sums a word");
    const u32 a = __reduce_add_sync(0xffffffffu, c[0] | c[1] << 16), b = __reduce_add_sync(0xffffffffu, c[2] | c[3] << 16);
    if ((threadIdx.x & 31) == 0) {
        s_w[2 * (threadIdx.x >> 5)] = a;
        s_w[2 * (threadIdx.x >> 5) + 1] = b;
    }
    __syncthreads();
    if (threadIdx.x < kVbPer && threadIdx.x < left) {
        u32 t = 0;
        for (u32 w = 0; w < kVbThreads / 32; w++)
            t += (s_w[2 * w + threadIdx.x / 2] >> (threadIdx.x % 2 ? 16 : 0)) & 0xffffu;
        out[threadIdx.x] = t;
    }
}

__host__ __device__ __forceinline__ u64 vb_div(u64 n, u64 per) { return (n + per - 1) / per; }

// Value p of the column: a u32 array, or the lengths rhs_off[p+1] - rhs_off[p].
template <bool kLens>
__device__ __forceinline__ u32 vb_value(const u32* vals, const u64* offs, u64 p) {
    if (kLens) return (u32)(__ldg(offs + p + 1) - __ldg(offs + p));
    return __ldg(vals + p);
}

// --------------------------------------------------------------------------
// byte count of a column (sizes the sections of an export)
// --------------------------------------------------------------------------

template <bool kLens>
__global__ void __launch_bounds__(kVbThreads) k_vb_count(const u32* __restrict__ vals, const u64* __restrict__ offs,
                                                         u64 n, u64* __restrict__ total) {
    pdl_wait();
    u64 s = 0;
    for (u64 p = blockIdx.x * (u64)blockDim.x + threadIdx.x; p < n; p += (u64)gridDim.x * blockDim.x)
        s += vb_len(vb_value<kLens>(vals, offs, p));
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    __shared__ u64 s_w[kVbThreads / 32];
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        u64 t = 0;
        for (int w = 0; w < kVbThreads / 32; w++) t += s_w[w];
        if (t) atomicAdd(reinterpret_cast<unsigned long long*>(total), (unsigned long long)t);
    }
}

// --------------------------------------------------------------------------
// encode: bytes per tile, (scan of the tile counts), write
// --------------------------------------------------------------------------

// Values of this thread (kVbItems from p0; 0 past n).
template <bool kLens>
__device__ __forceinline__ void vb_load(const u32* vals, const u64* offs, u64 n, u64 p0, u32 (&v)[kVbItems]) {
    if (!kLens && p0 + kVbItems <= n && (reinterpret_cast<uintptr_t>(vals + p0) & 15) == 0) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(vals + p0));
        const uint4 b = __ldg(reinterpret_cast<const uint4*>(vals + p0) + 1);
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else if (kLens) {
        u64 prev = (p0 < n) ? __ldg(offs + p0) : 0;
#pragma unroll
        for (int it = 0; it < kVbItems; it++) {
            const u64 nx = (p0 + it < n) ? __ldg(offs + p0 + it + 1) : prev;
            v[it] = (u32)(nx - prev);
            prev = nx;
        }
    } else {
#pragma unroll
        for (int it = 0; it < kVbItems; it++) v[it] = (p0 + it < n) ? __ldg(vals + p0 + it) : 0u;
    }
}

template <bool kLens>
__device__ __forceinline__ u32 vb_thread_bytes(const u32 (&v)[kVbItems], u64 n, u64 p0) {
    const u32 c = n > p0 ? (u32)min(n - p0, (u64)kVbItems) : 0u;
    u32 b = 0;
#pragma unroll
    for (int it = 0; it < kVbItems; it++) b += vb_len(v[it]);
    return b - ((u32)kVbItems - c);  // (values past n are zeros: a byte each)
}

// tile_bytes[t] = bytes of the VByte stream of values [t * kVbTile, ...).  A block
// takes kVbPer tiles, whose loads are in flight together (200 MB in 45 us with one).
template <bool kLens>
__global__ void __launch_bounds__(kVbThreads) k_vb_tile_bytes(const u32* __restrict__ vals,
                                                              const u64* __restrict__ offs, u64 n,
                                                              u32* __restrict__ tile_bytes) {
    __shared__ u32 s_w[2 * kVbThreads / 32];
    pdl_wait();
    const u64 t0 = blockIdx.x * (u64)kVbPer;
    u32 v[kVbPer][kVbItems], b[kVbPer];
#pragma unroll
    for (int u = 0; u < kVbPer; u++)
        vb_load<kLens>(vals, offs, n, (t0 + u) * kVbTile + (u64)threadIdx.x * kVbItems, v[u]);
#pragma unroll
    for (int u = 0; u < kVbPer; u++)
        b[u] = vb_thread_bytes<kLens>(v[u], n, (t0 + u) * kVbTile + (u64)threadIdx.x * kVbItems);
    vb_block_sums(b, s_w, vb_div(n, kVbTile) - t0, tile_bytes + t0);
}

// A tile's stream bytes, at the offset of their place in a 16-byte line of the
// output, so that whole lines are copied as they are.
constexpr u32 kVbOutWords = (kVbTile * 5 + 16) / 4 + 3;
struct __align__(16) VbOut {
    u32 w[(kVbOutWords + 3) / 4 * 4];
    u32 sums[kVbThreads / 32];
};

// Bytes on their way to shared memory: those that do not fill a word yet.
struct VbPack {
    u32* w;    // the word they belong to
    u32 part;  // the word so far
    u32 bits;  // 8 times its bytes
    __device__ __forceinline__ void put(u32 y, u32 ybits) {  // ybits <= 32, y < 2^ybits
        const u32 over = __funnelshift_l(y, 0u, bits);
        part |= y << bits;
        bits += ybits;
        if (bits >= 32) {
            *w++ = part;
            part = over;
        }
        bits &= 31;
    }
};

// Assembles the tile's values (`left` values from its first to the column's end) and
// stores its bytes at dst (mine: this thread's bytes).  A value's groups are spread over the bytes of a word,
// the continuation bits added, and the bytes shifted into a register that goes to
// shared memory word by word; what a thread has left over at its end it adds to the
// word that the next thread has begun.  Some 40 instructions a value and no loop;
// byte by byte in a loop it was 121 us for 50 M values of 116 MB, 89 us now.
__device__ __forceinline__ u32 vb_put_tile(VbOut& sm, const u32 (&v)[kVbItems], u64 left, u32 mine, u8* dst) {
    const u32 a = (u32)(reinterpret_cast<uintptr_t>(dst) & 15);
    u32 tb;
    const u32 o = a + vb_block_scan(mine, sm.sums, tb);
    VbPack p{sm.w + (o >> 2), 0, 8 * (o & 3)};
    const u32 here = (u32)min(left, (u64)kVbTile), t0 = threadIdx.x * kVbItems;
    const bool all = t0 + kVbItems <= here;
    if (all) {
#pragma unroll
        for (int it = 0; it < kVbItems; it++) {
            const u32 x = v[it], l = min(vb_len(x), 4u);
            u32 y = (x & 0x3fffu) | ((x << 2) & 0x3fff0000u);     // 14 bits per half word
            y = (y & 0x007f007fu) | ((y << 1) & 0x7f007f00u);     // 7 bits per byte
            y |= 0x00808080u >> (32u - 8u * l);
            if (x >> 28) {
                p.put(y | 0x80000000u, 32u);
                p.put(x >> 28, 8u);
            } else {
                p.put(y, 8u * l);
            }
        }
    }
    __syncthreads();
    // (eight values are two words or more: the next thread with eight has begun the word)
    if (all && p.bits) {
        if (t0 + 2 * kVbItems <= here) *p.w |= p.part;
        else *p.w = p.part;
    }
    if (here < (u32)kVbTile) {  // the end of the column: its last few values byte by byte
        __syncthreads();
        if (!all) {
            u8* by = reinterpret_cast<u8*>(sm.w) + o;
#pragma unroll
            for (int it = 0; it < kVbItems; it++) {
                if (t0 + it >= here) continue;
                u32 x = v[it];
                for (; x >= 0x80u; x >>= 7) *by++ = (u8)(x | 0x80u);
                *by++ = (u8)x;
            }
        }
    }
    __syncthreads();
    u8* line = dst - a;
    const u8* by = reinterpret_cast<const u8*>(sm.w);
    const u32 lines = (a + tb) / 16;
    for (u32 l = (a ? 1u : 0u) + threadIdx.x; l < lines; l += kVbThreads)
        reinterpret_cast<uint4*>(line)[l] = reinterpret_cast<const uint4*>(sm.w)[l];
    if (a && threadIdx.x < 16 && threadIdx.x >= a && threadIdx.x < a + tb) line[threadIdx.x] = by[threadIdx.x];
    if ((lines >= 1 || a == 0) && threadIdx.x < a + tb - 16 * lines)
        line[16 * lines + threadIdx.x] = by[16 * lines + threadIdx.x];
    return tb;
}

// Writes the VByte stream of the n values to out[0 ..): tile t at its
// offset tile_off[t] (exclusive scan of k_vb_tile_bytes), assembled in shared
// memory and stored by 16-byte lines.  With `pad`, the last tile adds zeros up to
// the next multiple of 8 bytes (section padding).
template <bool kLens>
__global__ void __launch_bounds__(kVbThreads) k_vb_write(const u32* __restrict__ vals, const u64* __restrict__ offs,
                                                         u64 n, const u64* __restrict__ tile_off,
                                                         u8* __restrict__ out, bool pad) {
    __shared__ VbOut sm;
    pdl_wait();
    const u64 tile = blockIdx.x;
    const u64 p0 = tile * (u64)kVbTile + (u64)threadIdx.x * kVbItems;
    const u64 base = tile_off[tile];
    u32 v[kVbItems];
    vb_load<kLens>(vals, offs, n, p0, v);
    const u32 tb = vb_put_tile(sm, v, n - tile * kVbTile, vb_thread_bytes<kLens>(v, n, p0), out + base);
    if (pad && tile == gridDim.x - 1 && threadIdx.x == 0)
        for (u64 z = base + tb; z & 7; z++) out[z] = 0;
}

// --------------------------------------------------------------------------
// decode: values per tile, (scan of the tile counts), write
// --------------------------------------------------------------------------

// High bit of each byte of a little-endian word: bit q = bit 7 of byte q (the four
// bits gathered into the top ones by one multiplication).
__device__ __forceinline__ u32 vb_high_bits(u32 w) { return ((w & 0x80808080u) * 0x00204081u) >> 28; }

// Bytes [p0, p0 + 16) of the stream as little-endian words; past nb bytes that do
// not end a value.
__device__ __forceinline__ void vb_load16(const u8* in, u64 nb, u64 p0, u32 (&w)[4]) {
    if (p0 + kVbBytes <= nb && (reinterpret_cast<uintptr_t>(in + p0) & 7) == 0) {
        const uint2 a = __ldg(reinterpret_cast<const uint2*>(in + p0)), b = __ldg(reinterpret_cast<const uint2*>(in + p0) + 1);
        w[0] = a.x, w[1] = a.y, w[2] = b.x, w[3] = b.y;
    } else if (p0 > 0 && p0 + kVbBytes + 4 <= nb) {
        // inside an unaligned stream: the aligned words around them (byte by byte a stream
        // of 260 kB took 47 us to decode, 41 so)
        const uintptr_t at = reinterpret_cast<uintptr_t>(in + p0);
        const u32* const word = reinterpret_cast<const u32*>(at & ~(uintptr_t)3);
        const u32 sh = 8 * (u32)(at & 3);
        u32 x[5];
#pragma unroll
        for (int q = 0; q < 5; q++) x[q] = __ldg(word + q);
#pragma unroll
        for (int q = 0; q < 4; q++) w[q] = __funnelshift_r(x[q], x[q + 1], sh);
    } else {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            w[q] = 0;
#pragma unroll
            for (int j = 0; j < 4; j++)
                w[q] |= ((p0 + 4 * q + j < nb) ? (u32)__ldg(in + p0 + 4 * q + j) : 0x80u) << (8 * j);
        }
    }
}

// How many of the 16 bytes end a value (high bit clear).
__device__ __forceinline__ u32 vb_ends(const u32 (&w)[4]) {
    constexpr u32 m = 0x80808080u;
    return 16u - __popc((w[0] & m) | ((w[1] & m) >> 1) | ((w[2] & m) >> 2) | ((w[3] & m) >> 3));
}

// tile_cnt[t] = values that end in bytes [t * kVbDecTile, ...) of the stream.  A
// block takes kVbPer tiles, whose loads are in flight together (116 MB in 32 us with
// one).
__global__ void __launch_bounds__(kVbThreads) k_vb_tile_ends(const u8* __restrict__ in, u64 nb,
                                                             u32* __restrict__ tile_cnt) {
    __shared__ u32 s_w[2 * kVbThreads / 32];
    pdl_wait();
    const u64 t0 = blockIdx.x * (u64)kVbPer;
    u32 c[kVbPer];
#pragma unroll
    for (int u = 0; u < kVbPer; u++) {
        u32 w[4];
        vb_load16(in, nb, (t0 + u) * kVbDecTile + (u64)threadIdx.x * kVbBytes, w);
        c[u] = vb_ends(w);
    }
    vb_block_sums(c, s_w, vb_div(nb, kVbDecTile) - t0, tile_cnt + t0);
}

struct VbIn {
    u32 v[kVbDecTile];  // the tile's values
    u32 sums[kVbThreads / 32];
    uint2 tail[kVbThreads / 32];  // each warp's last 8 bytes
};

// The groups of four bytes, least significant first, as one number of 28 bits.
__device__ __forceinline__ u32 vb_groups(u32 y) {
    y = (y & 0x007f007fu) | ((y >> 1) & 0x3f803f80u);
    return (y & 0x3fffu) | ((y >> 2) & 0x0fffc000u);
}

// One tile of a stream (bytes [t0, t0 + 4096) of src, nb bytes in all) into
// out[base ...).  Each thread takes its 16 bytes one after the other, from the groups
// of the value that the bytes before them began: every byte adds its group, and one
// that ends a value gives it to the tile's values, which are then stored coalesced.
// Every lane does the same for every byte, some ten instructions; a loop over the
// values that end in a thread's bytes left the lanes waiting for the one with the
// most: 252 us for 50 M values of 116 MB, 100 us now (138 with a thread per value over
// a list of their ends).  `last`: the stream's last tile, which checks that n values
// were found.
__device__ __forceinline__ void vb_decode_tile(const u8* __restrict__ src, u64 nb, u64 n, u64 lo, u64 hi, u64 t0,
                                               u64 base, bool last, u32* __restrict__ out, VbIn& sm,
                                               DevStatus* ds) {
    const u64 p0 = t0 + (u64)threadIdx.x * kVbBytes;
    const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // loads issued together: the 8 bytes before the tile (thread 0; zeros, which end a
    // value, before the stream), the thread's 16 bytes
    uint2 before = make_uint2(0, 0);
    if (threadIdx.x == 0 && t0 > 0) {
        if ((reinterpret_cast<uintptr_t>(src + t0 - 8) & 7) == 0) {
            before = __ldg(reinterpret_cast<const uint2*>(src + t0 - 8));
        } else {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                before.x |= (u32)__ldg(src + t0 - 8 + q) << (8 * q);
                before.y |= (u32)__ldg(src + t0 - 4 + q) << (8 * q);
            }
        }
    }
    u32 w[4];
    vb_load16(src, nb, p0, w);
    uint2 b8;  // the 8 bytes before p0
    b8.x = __shfl_up_sync(0xffffffffu, w[2], 1);
    b8.y = __shfl_up_sync(0xffffffffu, w[3], 1);
    if (lane == 31) sm.tail[wid] = make_uint2(w[2], w[3]);
    u32 cnt;
    const u32 first = vb_block_scan(vb_ends(w), sm.sums, cnt);  // its barrier also publishes the tails
    if (lane == 0) b8 = wid > 0 ? sm.tail[wid - 1] : before;
    // continuation bytes: bits 0 .. 7 of the 8 before, 8 .. 23 of the thread's
    const u32 c = vb_high_bits(b8.x) | vb_high_bits(b8.y) << 4 | vb_high_bits(w[0]) << 8 | vb_high_bits(w[1]) << 12 |
                  vb_high_bits(w[2]) << 16 | vb_high_bits(w[3]) << 20;
    // (bytes past the stream are continuation bytes here)
    const u32 here = p0 >= nb ? 0u : (nb - p0 < kVbBytes ? (1u << (u32)(nb - p0)) - 1u : 0xffffu);
    const u32 c4 = c & (c << 1) & (c << 2) & (c << 3);                      // bytes up to here: four continuations
    bool bad = ((c4 << 1) & c & (here << 8)) != 0;                          // and a fifth: a sixth byte follows
    u32 five = (c4 << 1) & ~c & (here << 8);                                // the fifth byte of a value
    for (; five; five &= five - 1) {
        const u32 q = (u32)__ffs((int)five) - 9;
        const u32 x = (q < 8 ? (q < 4 ? w[0] : w[1]) : (q < 12 ? w[2] : w[3])) >> (8 * (q & 3));
        bad = bad || (x & 0x70u) != 0;                                      // more than 32 bits
    }
    // the stream must end with a value's last byte
    if (p0 < nb && nb - p0 <= kVbBytes && ((c >> (u32)(nb - p0 + 7)) & 1u)) bad = true;
    // the value begun before: its r <= 4 bytes (more is an error)
    const u32 r = min(4u, (u32)__clz((int)~(c << 24)));
    u32 x = r ? vb_groups(b8.y >> (32 - 8 * r)) : 0u, scale = 1u << (7 * r);
    u32* to = sm.v + first;
#pragma unroll
    for (int q = 0; q < kVbBytes; q++) {
        const u32 byte = w[q / 4] >> (8 * (q % 4));
        x += (byte & 0x7fu) * scale;
        scale <<= 7;
        if (!(byte & 0x80u)) {
            *to++ = x;
            x = 0;
            scale = 1;
        }
    }
    __syncthreads();
    const u32 room = base < n ? (u32)min(n - base, (u64)cnt) : 0u;  // (too many values: an error of the last tile)
    if (lo == 0 && hi == (1ull << 32)) {
        for (u32 k = threadIdx.x; k < room; k += kVbThreads) out[base + k] = sm.v[k];
    } else {
        // lo <= 1 and hi <= 2^32; nothing is allowed when hi is 0
        const u32 least = (u32)lo, most = (u32)(hi - 1);
        bad = bad || (hi == 0 && cnt > 0);
        for (u32 k = threadIdx.x; k < room; k += kVbThreads) {
            const u32 y = sm.v[k];
            bad = bad || y < least || y > most;
            out[base + k] = y;
        }
    }
    if (bad) set_error(ds, kErrFormat);
    if (last && threadIdx.x == 0 && base + cnt != n) set_error(ds, kErrFormat);
}

// Decodes the nb-byte stream into exactly n values with lo <= v < hi: the
// values ending in tile t go to vals[cnt_off[t] ...) (cnt_off: exclusive
// scan of k_vb_tile_ends).
__global__ void __launch_bounds__(kVbThreads) k_vb_dwrite(const u8* __restrict__ in, u64 nb, u64 n, u64 lo, u64 hi,
                                                          const u64* __restrict__ cnt_off, u32* __restrict__ vals,
                                                          DevStatus* ds) {
    __shared__ VbIn sm;
    pdl_wait();
    const u64 tile = blockIdx.x;
    vb_decode_tile(in, nb, n, lo, hi, tile * (u64)kVbDecTile, cnt_off[tile], tile == gridDim.x - 1, vals, sm, ds);
}

// --------------------------------------------------------------------------
// every column of a grammar in one launch per step
// --------------------------------------------------------------------------
//
// Tile t of a launch belongs to column c with cols[c].tile0 <= t <
// cols[c + 1].tile0 (the last entry is a sentinel holding the launch's tile
// count); a block finds its column by binary search over the tile0 values,
// loaded into shared memory.

template <typename Col>
__device__ __forceinline__ u32 vb_column_of(const Col* cols, u32 ncols, u64 t, u64* s_t0) {
    for (u32 c = threadIdx.x; c <= ncols; c += blockDim.x) s_t0[c] = cols[c].tile0;
    __syncthreads();
    u32 lo = 0, hi = ncols;  // s_t0[lo] <= t < s_t0[hi]
    while (hi - lo > 1) {
        const u32 mid = (lo + hi) / 2;
        if (s_t0[mid] <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(kVbThreads) k_vb_tile_bytes_all(const VbEncCol* __restrict__ cols, u32 ncols,
                                                                  u32* __restrict__ tile_bytes,
                                                                  u64* __restrict__ col_bytes) {
    __shared__ u64 s_t0[kVbMaxCols + 1];
    __shared__ u32 s_w[kVbThreads / 32];
    pdl_wait();
    const u64 t = blockIdx.x;
    const u32 c = vb_column_of(cols, ncols, t, s_t0);
    const VbEncCol col = cols[c];
    const u64 p0 = (t - col.tile0) * (u64)kVbTile + (u64)threadIdx.x * kVbItems;
    u32 v[kVbItems];
    u32 b;
    if (col.offs) {
        vb_load<true>(col.vals, col.offs, col.n, p0, v);
        b = vb_thread_bytes<true>(v, col.n, p0);
    } else {
        vb_load<false>(col.vals, col.offs, col.n, p0, v);
        b = vb_thread_bytes<false>(v, col.n, p0);
    }
    for (int o = 16; o > 0; o >>= 1) b += __shfl_down_sync(0xffffffffu, b, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = b;
    __syncthreads();
    if (threadIdx.x == 0) {
        u32 sum = 0;
        for (int w = 0; w < kVbThreads / 32; w++) sum += s_w[w];
        tile_bytes[t] = sum;
        if (sum) atomicAdd(reinterpret_cast<unsigned long long*>(col_bytes + c), (unsigned long long)sum);
    }
}

// Tile t of column c goes to cols[c].dst + tile_off[t] - tile_off[cols[c].tile0];
// the last tile of each column zero-pads it to a multiple of 8 bytes.
__global__ void __launch_bounds__(kVbThreads) k_vb_write_all(const VbEncCol* __restrict__ cols, u32 ncols,
                                                             const u64* __restrict__ tile_off) {
    __shared__ u64 s_t0[kVbMaxCols + 1];
    __shared__ VbOut sm;
    pdl_wait();
    const u64 t = blockIdx.x;
    const u32 c = vb_column_of(cols, ncols, t, s_t0);
    const VbEncCol col = cols[c];
    const u64 base = tile_off[t] - tile_off[col.tile0];
    const bool last = (t + 1 == s_t0[c + 1]);
    const u64 p0 = (t - col.tile0) * (u64)kVbTile + (u64)threadIdx.x * kVbItems;
    u32 v[kVbItems];
    u32 mine;
    if (col.offs) {
        vb_load<true>(col.vals, col.offs, col.n, p0, v);
        mine = vb_thread_bytes<true>(v, col.n, p0);
    } else {
        vb_load<false>(col.vals, col.offs, col.n, p0, v);
        mine = vb_thread_bytes<false>(v, col.n, p0);
    }
    const u32 tb = vb_put_tile(sm, v, col.n - (t - col.tile0) * kVbTile, mine, col.dst + base);
    if (last && threadIdx.x == 0)
        for (u64 z = base + tb; z & 7; z++) col.dst[z] = 0;
}

__global__ void __launch_bounds__(kVbThreads) k_vb_tile_ends_all(const VbDecCol* __restrict__ cols, u32 ncols,
                                                                 u32* __restrict__ tile_cnt) {
    __shared__ u64 s_t0[kVbMaxCols + 1];
    __shared__ u32 s_w[kVbThreads / 32];
    pdl_wait();
    const u64 t = blockIdx.x;
    const u32 c = vb_column_of(cols, ncols, t, s_t0);
    const VbDecCol col = cols[c];
    const u64 p0 = (t - col.tile0) * (u64)kVbDecTile + (u64)threadIdx.x * kVbBytes;
    u32 w[4];
    vb_load16(col.src, col.nb, p0, w);
    u32 n = vb_ends(w);
    for (int o = 16; o > 0; o >>= 1) n += __shfl_down_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = n;
    __syncthreads();
    if (threadIdx.x == 0) {
        u32 sum = 0;
        for (int w = 0; w < kVbThreads / 32; w++) sum += s_w[w];
        tile_cnt[t] = sum;
    }
}

__global__ void __launch_bounds__(kVbThreads) k_vb_dwrite_all(const VbDecCol* __restrict__ cols, u32 ncols,
                                                              const u64* __restrict__ cnt_off, DevStatus* ds) {
    __shared__ u64 s_t0[kVbMaxCols + 1];
    __shared__ VbIn sm;
    pdl_wait();
    const u64 t = blockIdx.x;
    const u32 c = vb_column_of(cols, ncols, t, s_t0);
    const VbDecCol col = cols[c];
    const bool last = (t + 1 == s_t0[c + 1]);
    const u64 base = cnt_off[t] - cnt_off[col.tile0];
    const u64 t0 = (t - col.tile0) * (u64)kVbDecTile;
    vb_decode_tile(col.src, col.nb, col.n, col.lo, col.hi, t0, base, last, col.out, sm, ds);
}

// Offsets of every level from the scan of all levels' rule lengths (levels
// with rules only, in order): rhs_off[r] = scan[gbase + r] - scan[gbase],
// rhs_off[g] = the level's length sum, which must be G (else kErrFormat).
// blockIdx.y = level; *total = the sum of all lengths.
__global__ void k_vb_offsets_all(const VbLevelOff* __restrict__ lv, const u64* __restrict__ scan,
                                 const u64* __restrict__ total, u32 nlv, DevStatus* ds) {
    pdl_wait();
    const VbLevelOff L = lv[blockIdx.y];
    const u64 s0 = scan[L.gbase];
    const u64 s1 = (blockIdx.y + 1 < nlv) ? scan[lv[blockIdx.y + 1].gbase] : *total;
    for (u64 r = blockIdx.x * (u64)blockDim.x + threadIdx.x; r <= L.g; r += (u64)gridDim.x * blockDim.x)
        L.rhs_off[r] = (r < L.g ? scan[L.gbase + r] : s1) - s0;
    if (blockIdx.x == 0 && threadIdx.x == 0 && s1 - s0 != L.G) set_error(ds, kErrFormat);
}

// --------------------------------------------------------------------------
// launchers
// --------------------------------------------------------------------------

u64 vb_encode_tiles(u64 n) { return vb_div(n, kVbTile); }
u64 vb_decode_tiles(u64 nb) { return vb_div(nb, kVbDecTile); }

cudaError_t launch_vb_count(const u32* vals, const u64* offs, u64 n, u64* total, int sms, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const unsigned grid = (unsigned)std::min<u64>((n + kVbThreads - 1) / kVbThreads, (u64)sms * 8);
    if (offs) return launch_pdl(k_vb_count<true>, grid, kVbThreads, st, vals, offs, n, total);
    return launch_pdl(k_vb_count<false>, grid, kVbThreads, st, vals, offs, n, total);
}

cudaError_t launch_vb_tile_bytes(const u32* vals, const u64* offs, u64 n, u32* tile_bytes, cudaStream_t st) {
    const unsigned grid = (unsigned)vb_div(vb_encode_tiles(n), kVbPer);
    if (grid == 0) return cudaSuccess;
    if (offs) return launch_pdl(k_vb_tile_bytes<true>, grid, kVbThreads, st, vals, offs, n, tile_bytes);
    return launch_pdl(k_vb_tile_bytes<false>, grid, kVbThreads, st, vals, offs, n, tile_bytes);
}

cudaError_t launch_vb_write(const u32* vals, const u64* offs, u64 n, const u64* tile_off, u8* out, bool pad,
                            cudaStream_t st) {
    const unsigned grid = (unsigned)vb_encode_tiles(n);
    if (grid == 0) return cudaSuccess;
    if (offs) return launch_pdl(k_vb_write<true>, grid, kVbThreads, st, vals, offs, n, tile_off, out, pad);
    return launch_pdl(k_vb_write<false>, grid, kVbThreads, st, vals, offs, n, tile_off, out, pad);
}

cudaError_t launch_vb_tile_ends(const u8* in, u64 nb, u32* tile_cnt, cudaStream_t st) {
    const unsigned grid = (unsigned)vb_div(vb_decode_tiles(nb), kVbPer);
    if (grid == 0) return cudaSuccess;
    return launch_pdl(k_vb_tile_ends, grid, kVbThreads, st, in, nb, tile_cnt);
}

cudaError_t launch_vb_dwrite(const u8* in, u64 nb, u64 n, u64 lo, u64 hi, const u64* cnt_off, u32* vals,
                             DevStatus* ds, cudaStream_t st) {
    const unsigned grid = (unsigned)vb_decode_tiles(nb);
    if (grid == 0) return cudaSuccess;
    return launch_pdl(k_vb_dwrite, grid, kVbThreads, st, in, nb, n, lo, hi, cnt_off, vals, ds);
}

cudaError_t launch_vb_tile_bytes_all(const VbEncCol* cols, u32 ncols, u64 tiles, u32* tile_bytes, u64* col_bytes,
                                     cudaStream_t st) {
    if (tiles == 0) return cudaSuccess;
    return launch_pdl(k_vb_tile_bytes_all, (unsigned)tiles, kVbThreads, st, cols, ncols, tile_bytes, col_bytes);
}

cudaError_t launch_vb_write_all(const VbEncCol* cols, u32 ncols, u64 tiles, const u64* tile_off, cudaStream_t st) {
    if (tiles == 0) return cudaSuccess;
    return launch_pdl(k_vb_write_all, (unsigned)tiles, kVbThreads, st, cols, ncols, tile_off);
}

cudaError_t launch_vb_tile_ends_all(const VbDecCol* cols, u32 ncols, u64 tiles, u32* tile_cnt, cudaStream_t st) {
    if (tiles == 0) return cudaSuccess;
    return launch_pdl(k_vb_tile_ends_all, (unsigned)tiles, kVbThreads, st, cols, ncols, tile_cnt);
}

cudaError_t launch_vb_dwrite_all(const VbDecCol* cols, u32 ncols, u64 tiles, const u64* cnt_off, DevStatus* ds,
                                 cudaStream_t st) {
    if (tiles == 0) return cudaSuccess;
    return launch_pdl(k_vb_dwrite_all, (unsigned)tiles, kVbThreads, st, cols, ncols, cnt_off, ds);
}

cudaError_t launch_vb_offsets_all(const VbLevelOff* lv, u32 nlv, u64 max_g, const u64* scan, const u64* total,
                                  DevStatus* ds, cudaStream_t st) {
    if (nlv == 0) return cudaSuccess;
    // (a few blocks per SM for the largest level: blocks of the small ones only exit, and
    // 4096 a level took 39 us for 15 levels of 3.3 M rules)
    const unsigned gx = (unsigned)std::min<u64>((max_g + 1 + kVbThreads - 1) / kVbThreads, 4 * 152);
    return launch_pdl(k_vb_offsets_all, dim3(gx, nlv), dim3(kVbThreads), st, lv, scan, total, nlv, ds);
}

}  // namespace lcg
