// Compaction, sort, merge, top-k and export of count tables.
//
// After the counting kernel the global hash tables hold each distinct word
// once with its exact count (Sec. 3.3's reduced dictionary).  This file turns
// them into the sorted output.  A table of at most kBktMaxCap slots whose counts
// are below 2^48 goes through the bucket sort of wc_bucket.cuh, straight from the
// hash tables.  Other tables (and the allocation-free entry point, whose fixed
// scratch has no room for it) are compacted and then sorted by an LSD radix sort over a
// permutation: 10 byte-digits of the packed prefix and up to 8 digits of the
// complemented count (count descending).  Either is followed by a fix-up that
// orders long words sharing count and 16-letter prefix by their remaining
// bytes, so the final order is (count desc, word asc).  Radix digits that are
// equal for every element are skipped, detected on the device from one
// histogram pass; those the host's bounds already show constant (count bytes
// above the token bound, document bytes above the document count) are not
// launched at all.
#include <algorithm>
#include <vector>

#include "wc_bucket.cuh"
#include "wc_internal.h"

namespace wc {

constexpr int kSortTile = (int)kSortTileElems;  // elements per block in a radix pass
constexpr int kSortThreads = 256;
constexpr int kItems = kSortTile / kSortThreads;  // 16
constexpr int kPasses = kSortPasses;
constexpr int kPassesSeg = kSortPassesSeg;

__device__ __forceinline__ unsigned long long be64(uint32_t x, uint32_t y) {
    return ((unsigned long long)__byte_perm(x, 0, 0x0123) << 32) | __byte_perm(y, 0, 0x0123);
}
__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

size_t sort_scratch_bytes(uint64_t cap) {
    uint64_t ntiles = (cap + kSortTile - 1) / kSortTile;
    return cap * (8 + 8 + 8 + 8 + 4 + 4 + 4 + 4 + 4) + 4 * kPassesSeg * 256 + 4 * 256 * ntiles + 4 * 32 +
           2 * 4 * 256 * (ntiles <= kSortFusedMaxTiles ? sort_group_stride(ntiles) : 1) + 4096 +
           2 * (4 * 256 * ntiles + 256) + 256;
}

void sort_scratch_carve(SortScratch &s, void *base, uint64_t cap) {
    uint64_t ntiles = (cap + kSortTile - 1) / kSortTile;
    uint8_t *p = static_cast<uint8_t *>(base);
    auto take = [&](size_t n) { uint8_t *r = p; p += (n + 255) & ~(size_t)255; return r; };
    s.cap = cap;
    s.khi = reinterpret_cast<unsigned long long *>(take(cap * 8));
    s.klo = reinterpret_cast<unsigned long long *>(take(cap * 8));
    s.cnt = reinterpret_cast<unsigned long long *>(take(cap * 8));
    s.pk = reinterpret_cast<unsigned long long *>(take(cap * 8));
    s.pk2 = reinterpret_cast<uint32_t *>(take(cap * 4));
    s.lref = reinterpret_cast<uint32_t *>(take(cap * 4));
    s.perm[0] = reinterpret_cast<uint32_t *>(take(cap * 4));
    s.perm[1] = reinterpret_cast<uint32_t *>(take(cap * 4));
    s.doc = reinterpret_cast<uint32_t *>(take(cap * 4));
    s.hist_all = reinterpret_cast<uint32_t *>(take(4 * kPassesSeg * 256));
    s.tile_hist = reinterpret_cast<uint32_t *>(take(4 * 256 * ntiles));
    s.cur = reinterpret_cast<uint32_t *>(take(4 * 32));
    s.group_stride = (uint32_t)(ntiles <= kSortFusedMaxTiles ? sort_group_stride(ntiles) : 1);
    s.group_hist[0] = reinterpret_cast<uint32_t *>(take(2 * 4 * 256 * (size_t)s.group_stride));  // both, adjacent
    s.group_hist[1] = s.group_hist[0] + 256 * (size_t)s.group_stride;
    s.look[0] = reinterpret_cast<uint32_t *>(take(4 * 256 * ntiles));
    s.look[1] = reinterpret_cast<uint32_t *>(take(4 * 256 * ntiles));
    s.tile_ctr = reinterpret_cast<uint32_t *>(take(4 * 2));
}

// ---------------------------------------------------------------- compaction
// The sort's key for an entry: the 16-letter prefix packed 5 bits a letter
// (80 bits: pk low 64, pk2 high 16) and the count inverted (descending), and
// the counts of each of their digits in a block's histogram h (one row of 256
// per pass), from which a pass with a single digit value is skipped.
__device__ __forceinline__ void sort_key_prep(const SortScratch &s, unsigned long long i, unsigned long long khi,
                                              unsigned long long klo, unsigned long long cnt, uint32_t *h) {
    const unsigned long long ph = pack5(khi), pl = pack5(klo), c = ~cnt;
    const unsigned long long lo = (ph << 40) | pl;  // the 80-bit code: ph:pl
    const uint32_t hi = (uint32_t)(ph >> 24);
    s.perm[0][i] = (uint32_t)i;
    s.pk[i] = lo;
    s.pk2[i] = hi;
#pragma unroll
    for (int b = 0; b < 8; b++) {
        atomicAdd(&h[b * 256 + ((lo >> (8 * b)) & 0xFF)], 1u);
        atomicAdd(&h[(kSortKeyPasses + b) * 256 + ((c >> (8 * b)) & 0xFF)], 1u);
    }
    atomicAdd(&h[8 * 256 + (hi & 0xFF)], 1u);
    atomicAdd(&h[9 * 256 + ((hi >> 8) & 0xFF)], 1u);
}

// One entry of a compaction, with its sort keys (digit counts into the block histogram h).
__device__ __forceinline__ void emit_entry(const SortScratch &ss, unsigned long long pos, unsigned long long khi,
                                           unsigned long long klo, unsigned long long cnt, uint32_t lref, uint32_t *h) {
    ss.khi[pos] = khi;
    ss.klo[pos] = klo;
    ss.cnt[pos] = cnt;
    ss.lref[pos] = lref;
    sort_key_prep(ss, pos, khi, klo, cnt, h);
}

// Occupied 16-byte-key slots -> entries (big-endian key halves); block bid of nb.
__device__ __forceinline__ void compact_short_body(const GSlot *slots, unsigned long long cap, const SortScratch &ss,
                                                   unsigned long long *meta, unsigned bid, unsigned nb,
                                                   uint32_t *h) {
    __shared__ BlockTake sh;
    const unsigned long long step = (unsigned long long)nb * blockDim.x * kScanUnroll;
    for (unsigned long long b = (unsigned long long)bid * blockDim.x * kScanUnroll; b < cap; b += step) {
        uint4 k[kScanUnroll];
        unsigned long long c[kScanUnroll], tok = 0;
        uint32_t mine = 0;
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            const unsigned long long i = b + (unsigned long long)u * blockDim.x + threadIdx.x;
            k[u] = make_uint4(0, 0, 0, 0);
            c[u] = 0;
            if (i < cap) {
                k[u] = slots[i].key;
                c[u] = slots[i].cnt;
            }
            if (!key_zero(k[u])) {
                mine++;
                tok += c[u];
            }
        }
        unsigned long long pos = block_take(sh, mine, tok, &meta[0], &meta[3], &meta[6]);
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            if (key_zero(k[u])) continue;
            emit_entry(ss, pos, be64(k[u].x, k[u].y), be64(k[u].z, k[u].w), c[u], 0u, h);
            pos++;
        }
    }
}

// Occupied 8-byte-key slots -> entries; block bid of nb.
__device__ __forceinline__ void compact8_body(const G8Slot *slots, unsigned long long cap, const SortScratch &ss,
                                              unsigned long long *meta, unsigned bid, unsigned nb,
                                              uint32_t *h) {
    __shared__ BlockTake sh;
    const unsigned long long step = (unsigned long long)nb * blockDim.x * kScanUnroll;
    for (unsigned long long b = (unsigned long long)bid * blockDim.x * kScanUnroll; b < cap; b += step) {
        ulonglong2 v[kScanUnroll];
        unsigned long long tok = 0;
        uint32_t mine = 0;
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            const unsigned long long i = b + (unsigned long long)u * blockDim.x + threadIdx.x;
            v[u] = i < cap ? *reinterpret_cast<const ulonglong2 *>(&slots[i]) : make_ulonglong2(0ull, 0ull);
            if (v[u].x) {
                mine++;
                tok += v[u].y;
            }
        }
        unsigned long long pos = block_take(sh, mine, tok, &meta[0], &meta[3], &meta[5]);
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            const unsigned long long key = v[u].x;
            if (!key) continue;
            emit_entry(ss, pos, be64((uint32_t)key, (uint32_t)(key >> 32)), 0ull, v[u].y, 0u, h);
            pos++;
        }
    }
}

// Byte i (0..15) of 16 bytes held as a uint4 (little-endian words).
__device__ __forceinline__ uint32_t byte16(uint4 v, uint32_t i) {
    const uint32_t w = i < 8u ? (i < 4u ? v.x : v.y) : (i < 12u ? v.z : v.w);
    return (w >> (8u * (i & 3u))) & 0xFFu;
}

// One lane per long-word slot: a warp's occupied slots take their long-word
// indices and arena bytes with one atomic each.  Each word is copied
// (lowercased, followed by one 0 byte so a run in the arena ends where the word
// ends) into the arena, by its own lane up to 64 bytes and by the whole warp
// beyond; then emit(slot, rank, occupied, khi, klo, count, lref, nocc, length) runs in every lane
// (rank: among the warp's nocc occupied slots).  A word of at most 32 letters
// whose slot holds its first and last 16 letters (kLongReady) is written from
// the slot, without reading its occurrence in the text.
template <class Emit>
__device__ __forceinline__ void long_slots_body(const LSlot *ls, unsigned long long lcap, const DevTable &out,
                                                unsigned bid, unsigned nb, Emit &&emit) {
    const int lane = threadIdx.x & 31;
    const unsigned long long nw = ((unsigned long long)nb * blockDim.x) >> 5;
    unsigned long long *meta = out.d_meta;
    for (unsigned long long w0 = (((unsigned long long)bid * blockDim.x + threadIdx.x) >> 5) * 32; w0 < lcap;
         w0 += nw * 32) {
        const unsigned long long w = w0 + lane;
        unsigned long long h = 0, addr = 0, len = 0, c = 0, lr = 0;
        uint4 f = make_uint4(0u, 0u, 0u, 0u), l = f;
        if (w < lcap) {
            h = ls[w].h;
            addr = ls[w].addr;
            lr = ls[w].len;
            len = long_len(lr);
            c = ls[w].cnt;
        }
        const bool occ = !(h == 0 && addr == 0);
        const uint32_t m = __ballot_sync(kFull, occ);
        if (!m) continue;
        const bool from_slot = occ && (lr & kLongReady) && len <= 32;
        if (from_slot) {
            f = ls[w].f;
            l = ls[w].l;
        }
        const unsigned long long rank = __popc(m & lanemask_lt()), nocc = __popc(m);
        const unsigned long long bytes = occ ? len + 1 : 0ull;
        unsigned long long incl = bytes;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long t = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += t;
        }
        const unsigned long long total = __shfl_sync(kFull, incl, 31);
        unsigned long long boff = 0, blidx = 0;
        if (lane == 0) {
            boff = atomicAdd(&meta[2], total);
            blidx = atomicAdd(&meta[1], nocc);
        }
        const unsigned long long off = __shfl_sync(kFull, boff, 0) + incl - bytes;
        const unsigned long long lidx = __shfl_sync(kFull, blidx, 0) + rank;
        // The arena or the long index is full: the table fails (status), but
        // the entry slot taken above is still filled (prefix key, no long
        // reference) so that the sort that follows reads only valid entries.
        const bool full = occ && (off + len + 1 > out.arena_cap || lidx >= out.lcap);
        const uint8_t *src = reinterpret_cast<const uint8_t *>(addr);
        if (from_slot && !full)  // word byte j: f[j] below 16, else l[j - (len - 16)]
            for (uint32_t j = 0; j < (uint32_t)len; j++)
                out.arena[off + j] = (uint8_t)(j < 16u ? byte16(f, j) : byte16(l, j + 16u - (uint32_t)len));
        else if (occ && !full && len <= 64)
            for (unsigned long long j = 0; j < len; j++) out.arena[off + j] = (uint8_t)(src[j] | 0x20u);
        uint32_t big = __ballot_sync(kFull, occ && !full && len > 64);
        while (big) {
            const int l = __ffs(big) - 1;
            big &= big - 1;
            const uint8_t *bs = reinterpret_cast<const uint8_t *>(__shfl_sync(kFull, addr, l));
            const unsigned long long bo = __shfl_sync(kFull, off, l), bl = __shfl_sync(kFull, len, l);
            for (unsigned long long j = lane; j < bl; j += 32) out.arena[bo + j] = (uint8_t)(bs[j] | 0x20u);
        }
        unsigned long long hi = 0, lo = 0;
        if (occ) {
            if (full) {
                atomicOr(out.d_status, ST_ARENA_FULL);
            } else {
                out.arena[off + len] = 0;
                out.loff[lidx] = off;
                out.llen[lidx] = len;
            }
            if (from_slot) {  // f holds the first 16 letters, lowercased, little-endian words
                hi = ((unsigned long long)__byte_perm(f.x, 0, 0x0123) << 32) | __byte_perm(f.y, 0, 0x0123);
                lo = ((unsigned long long)__byte_perm(f.z, 0, 0x0123) << 32) | __byte_perm(f.w, 0, 0x0123);
            } else {
                for (int j = 0; j < 8; j++) hi = (hi << 8) | (unsigned long long)(src[j] | 0x20u);
                for (int j = 8; j < 16; j++) lo = (lo << 8) | (unsigned long long)(src[j] | 0x20u);
            }
        }
        emit(w, (uint32_t)rank, occ, hi, lo, c, full ? 0u : (uint32_t)(lidx + 1), (uint32_t)nocc, len);
    }
}
__device__ __forceinline__ void compact_long_body(const LSlot *ls, unsigned long long lcap, const SortScratch &ss,
                                                  const DevTable &out, unsigned bid, unsigned nb, uint32_t *hist) {
    const int lane = threadIdx.x & 31;
    long_slots_body(ls, lcap, out, bid, nb, [&](unsigned long long, uint32_t rank, bool occ, unsigned long long hi,
                                                unsigned long long lo, unsigned long long c, uint32_t lref, uint32_t nocc,
                                                unsigned long long) {
        unsigned long long tok = occ ? c : 0ull, pos = 0;
        for (int d = 16; d; d >>= 1) tok += __shfl_xor_sync(kFull, tok, d);
        if (lane == 0) {
            pos = atomicAdd(&out.d_meta[0], (unsigned long long)nocc);
            atomicAdd(&out.d_meta[3], tok);
        }
        pos = __shfl_sync(kFull, pos, 0) + rank;
        if (occ) emit_entry(ss, pos, hi, lo, c, lref, hist);
    });
}

// All three tables' occupied slots -> entries in one launch: blocks
// [0, nb8) scan the 8-byte table, the next nb16 the 16-byte table and the
// rest the long-word table.  The per-kind entry counts go to meta[5] (8-byte)
// and meta[6] (16-byte).  The entries' radix keys and the digit histograms of
// the passes are prepared here as well.
__global__ void __launch_bounds__(256) k_compact_all(GTable g, unsigned long long cap8, unsigned long long cap16,
                                                     unsigned long long lcap, SortScratch ss, DevTable out,
                                                     unsigned nb8, unsigned nb16) {
    __shared__ uint32_t h[kPasses * 256];
    grid_dependency_wait();
    grid_dependency_trigger();
    for (int i = threadIdx.x; i < kPasses * 256; i += blockDim.x) h[i] = 0u;
    __syncthreads();
    const unsigned b = blockIdx.x;
    if (b < nb8) compact8_body(g.slots8, cap8, ss, out.d_meta, b, nb8, h);
    else if (b < nb8 + nb16) compact_short_body(g.slots, cap16, ss, out.d_meta, b - nb8, nb16, h);
    else compact_long_body(g.lslots, lcap, ss, out, b - nb8 - nb16, gridDim.x - nb8 - nb16, h);
    __syncthreads();
    for (int i = threadIdx.x; i < kPasses * 256; i += blockDim.x)
        if (h[i]) atomicAdd(&ss.hist_all[i], h[i]);
}

// ---------------------------------------------------------------- radix sort
__device__ __forceinline__ uint32_t sort_digit(const SortScratch &s, uint32_t idx, int p) {
    if (p >= kPasses) return (s.doc[idx] >> (8 * (p - kPasses))) & 0xFFu;
    if (p < 8) return (uint32_t)(s.pk[idx] >> (8 * p)) & 0xFFu;
    if (p < kSortKeyPasses) return (s.pk2[idx] >> (8 * (p - 8))) & 0xFFu;
    return (uint32_t)(~s.cnt[idx] >> (8 * (p - kSortKeyPasses))) & 0xFFu;
}

// Packs the prefix keys, and takes the histograms of all digit positions
// (for skipping constant digits) and the identity permutation.
__global__ void k_hist_all(SortJob job, int passes) {
    const SortScratch &s = job.s;
    const unsigned long long *meta = job.meta;
    __shared__ uint32_t h[kPassesSeg * 256];
    for (int i = threadIdx.x; i < kPassesSeg * 256; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const unsigned long long n = meta[0];
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        sort_key_prep(s, i, s.khi[i], s.klo[i], s.cnt[i], h);
        if (passes > kPasses) {
            const uint32_t d = s.doc[i];
#pragma unroll
            for (int b = 0; b < 4; b++) atomicAdd(&h[(kPasses + b) * 256 + ((d >> (8 * b)) & 0xFF)], 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += blockDim.x)
        if (h[i]) atomicAdd(&s.hist_all[i], h[i]);
}

// A pass is skipped when one digit value holds every element.
__device__ __forceinline__ bool pass_skipped(const SortScratch &s, int p, unsigned long long n) {
    bool mine = false;
    for (int d = threadIdx.x; d < 256; d += blockDim.x) mine |= (s.hist_all[p * 256 + d] == n);
    return __syncthreads_or(mine) != 0;
}

__global__ void __launch_bounds__(kSortThreads) k_pass_count(SortJob job, int p, int e, int fused) {
    const SortScratch &s = job.s;
    const unsigned long long *meta = job.meta;
    __shared__ uint32_t h[256];
    const unsigned long long n = meta[0];
    const unsigned long long ntiles = (n + kSortTile - 1) / kSortTile;
    if (blockIdx.x >= ntiles) return;
    if (pass_skipped(s, p, n)) return;
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t *in = s.perm_buf(s.cur[e]);
    const unsigned long long t0 = (unsigned long long)blockIdx.x * kSortTile + threadIdx.x;
    // all loads first (16 independent gathers in flight per thread), then the histogram
    uint32_t dig[kItems];
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const unsigned long long i = t0 + (unsigned long long)it * kSortThreads;
        dig[it] = i < n ? in[i] : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int it = 0; it < kItems; it++)
        if (dig[it] != 0xFFFFFFFFu) dig[it] = sort_digit(s, dig[it], p);
#pragma unroll
    for (int it = 0; it < kItems; it++)
        if (dig[it] != 0xFFFFFFFFu) atomicAdd(&h[dig[it]], 1u);
    __syncthreads();
    const uint32_t c = h[threadIdx.x];
    s.tile_hist[(unsigned long long)threadIdx.x * ntiles + blockIdx.x] = c;
    if (fused && c)
        atomicAdd(&s.group_buf((uint32_t)e & 1u)[(unsigned long long)threadIdx.x * s.group_stride +
                                                 blockIdx.x / sort_group_tiles(ntiles)],
                  c);
}

// Sorts of more than kSortFusedMaxTiles tiles: exclusive scan of the
// digit-major tile histogram: block d scans digit d's
// row of tile counts, starting from the number of elements with a smaller
// digit (from the all-pass histogram).  256 blocks of 256 threads.
__global__ void __launch_bounds__(256) k_pass_scan(SortJob job, int p, int e, int last) {
    const SortScratch &s = job.s;
    const unsigned long long *meta = job.meta;
    __shared__ uint32_t part[256];
    __shared__ uint32_t base_s;
    const unsigned long long n = meta[0];
    const bool skip = pass_skipped(s, p, n) || n == 0;
    if (skip) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            s.cur[e + 1] = s.cur[e];
            if (last) s.cur[kCurFinal] = s.cur[e];
        }
        return;
    }
    const uint32_t d = blockIdx.x, t = threadIdx.x;
    // base = elements whose digit is below d
    part[t] = t < d ? s.hist_all[p * 256 + t] : 0u;
    __syncthreads();
    for (int w = 128; w; w >>= 1) {
        if (t < (uint32_t)w) part[t] += part[t + w];
        __syncthreads();
    }
    if (t == 0) base_s = part[0];
    __syncthreads();
    uint32_t run = base_s;
    const unsigned long long ntiles = (n + kSortTile - 1) / kSortTile;
    uint32_t *row = s.tile_hist + (unsigned long long)d * ntiles;
    for (unsigned long long c0 = 0; c0 < ntiles; c0 += 256) {
        const unsigned long long i = c0 + t;
        const uint32_t v = i < ntiles ? row[i] : 0u;
        __syncthreads();
        part[t] = v;
        __syncthreads();
        for (int w = 1; w < 256; w <<= 1) {
            uint32_t x = t >= (uint32_t)w ? part[t - w] : 0u;
            __syncthreads();
            part[t] += x;
            __syncthreads();
        }
        if (i < ntiles) row[i] = run + part[t] - v;
        run += part[255];
    }
    if (d == 0 && t == 0) {
        s.cur[e + 1] = 1u - s.cur[e];
        if (last) s.cur[kCurFinal] = 1u - s.cur[e];
    }
}

// Stable scatter: warp w ranks its 512 consecutive elements in order with
// match_any; warps are combined in order, so equal digits keep their order.
__global__ void __launch_bounds__(kSortThreads) k_pass_scatter(SortJob job, int p, int e, int fused, int last) {
    const SortScratch &s = job.s;
    const unsigned long long *meta = job.meta;
    constexpr int WARPS = kSortThreads / 32;
    static_assert(kSortThreads == 256, "one thread per digit");
    __shared__ uint32_t wcount[WARPS][256];
    __shared__ uint32_t wtot[WARPS];
    const unsigned long long n = meta[0];
    const unsigned long long ntiles = (n + kSortTile - 1) / kSortTile;
    const bool skip = pass_skipped(s, p, n);
    if (fused) {  // (the scan pass does both otherwise)
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            const uint32_t c = skip ? s.cur[e] : 1u - s.cur[e];
            s.cur[e + 1] = c;
            if (last) s.cur[kCurFinal] = c;
        }
        // the next pass's group counts start from zero (this pass's are in the other buffer)
        uint32_t *gn = s.group_buf(((uint32_t)e + 1u) & 1u);
        for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
             i < 256ull * s.group_stride; i += (unsigned long long)gridDim.x * blockDim.x)
            gn[i] = 0u;
    }
    if (skip || blockIdx.x >= ntiles) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < WARPS * 256; i += kSortThreads) (&wcount[0][0])[i] = 0;
    // This tile's first position for digit d = threadIdx.x: scanned by the
    // scan pass, or (fused) the entries with a smaller digit, then digit d's
    // entries in the earlier tile groups and in the earlier tiles of this
    // tile's group.
    const int d = threadIdx.x;
    uint32_t run;
    if (fused) {
        const uint32_t own = s.hist_all[p * 256 + d];
        uint32_t incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) wtot[warp] = incl;
        run = incl - own;
        const uint32_t G = (uint32_t)sort_group_tiles(ntiles), g = blockIdx.x / G;
        const uint32_t *gb = s.group_buf((uint32_t)e & 1u) + (unsigned long long)d * s.group_stride;
#pragma unroll 4
        for (uint32_t q = 0; q < g; q++) run += gb[q];
        const uint32_t *tb = s.tile_hist + (unsigned long long)d * ntiles;
#pragma unroll 4
        for (uint32_t t2 = g * G; t2 < blockIdx.x; t2++) run += tb[t2];
    } else {
        run = s.tile_hist[(unsigned long long)d * ntiles + blockIdx.x];
    }
    __syncthreads();
    if (fused)
        for (int w = 0; w < warp; w++) run += wtot[w];
    const uint32_t cur = s.cur[e];
    const uint32_t *in = s.perm_buf(cur);
    uint32_t *out = s.perm_buf(1 - cur);
    const unsigned long long t0 = (unsigned long long)blockIdx.x * kSortTile + (unsigned long long)warp * (kSortTile / WARPS);
    uint32_t idx[kItems], dig[kItems], rank[kItems];
    // all loads first (independent gathers in flight), then the in-order ranking
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const unsigned long long i = t0 + it * 32 + lane;
        idx[it] = i < n ? in[i] : 0u;
    }
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const unsigned long long i = t0 + it * 32 + lane;
        dig[it] = i < n ? sort_digit(s, idx[it], p) : 256u + lane;  // invalid lanes never match real digits
    }
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const unsigned long long i = t0 + it * 32 + lane;
        const bool valid = i < n;
        uint32_t peers = __match_any_sync(kFull, dig[it]);
        int leader = __ffs(peers) - 1;
        uint32_t before = 0;
        if (lane == leader && valid) {
            before = wcount[warp][dig[it]];
            wcount[warp][dig[it]] = before + __popc(peers);
        }
        before = __shfl_sync(kFull, before, leader);
        rank[it] = before + __popc(peers & lanemask_lt());
    }
    __syncthreads();
    // exclusive prefix over warps, per digit (thread d handles digit d)
    {
        for (int w = 0; w < WARPS; w++) {
            uint32_t v = wcount[w][d];
            wcount[w][d] = run;
            run += v;
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        unsigned long long i = t0 + it * 32 + lane;
        if (i < n) out[wcount[warp][dig[it]] + rank[it]] = idx[it];
    }
}

// One radix pass in one launch, with a decoupled look-back for the tile
// offsets.  Blocks take tiles in launch order from a counter (so every tile
// a block waits for belongs to a block that is already running), rank their
// entries per digit as k_pass_scatter does, publish their per-digit counts
// (flag "aggregate"), and learn the counts of all earlier tiles by walking
// back over the published values until one carries a complete prefix (flag
// "inclusive"), which they then publish for their own tile.  Each wait is
// bounded: a look-back that gives up records kCurSortError (reported as a
// timeout by the finish) instead of hanging.  The block also zeroes its row
// of the other parity's look-back buffer and block 0 the other tile counter,
// for the next pass.
constexpr uint32_t kLookAgg = 1u << 30, kLookInc = 2u << 30, kLookVal = kLookAgg - 1u;
constexpr uint32_t kLookSpins = 1u << 22;  // look-back rounds before giving up
constexpr int kLookWin = 8;                // earlier tiles read per round
// A published word carries its flag and value together, and nothing else is
// read on its account (the next pass is ordered by the kernel boundary), so
// relaxed GPU-scope accesses suffice.
__device__ __forceinline__ void st_relaxed_u32(uint32_t *p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__global__ void __launch_bounds__(kSortThreads) k_pass_one(SortJob job, int p, int e, int last) {
    grid_dependency_wait();
    grid_dependency_trigger();
    const SortScratch &s = job.s;
    const unsigned long long *meta = job.meta;
    constexpr int WARPS = kSortThreads / 32;
    __shared__ uint32_t wcount[WARPS][256];
    __shared__ uint32_t wtot[WARPS];
    __shared__ uint32_t tile_sh;
    const unsigned long long n = meta[0];
    // loads that do not depend on n go out with it: digit d's count over all
    // entries (thread d) and the order this pass reads
    const int d = threadIdx.x;
    const uint32_t own = s.hist_all[p * 256 + d];
    const uint32_t cur = s.cur[e];
    const unsigned long long ntiles = (n + kSortTile - 1) / kSortTile;
    // the grid is sized by capacity: blocks past the entries leave at once
    // (block 0 stays: it records this pass's order even for an empty table)
    if (blockIdx.x >= ntiles && blockIdx.x != 0) return;
    const uint32_t par = (uint32_t)e & 1u;
    // the tile is taken before the skip test is known (a skipped pass's count
    // is zeroed by the next pass like any other)
    if (blockIdx.x < ntiles && threadIdx.x == 0) tile_sh = atomicAdd(&s.tile_ctr[par], 1u);
    if (blockIdx.x < ntiles) s.look_buf(par ^ 1u)[(unsigned long long)blockIdx.x * 256 + threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) s.tile_ctr[par ^ 1u] = 0u;
    // a pass is skipped when one digit value holds every entry
    const bool skip = __syncthreads_or(own == n) != 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const uint32_t c = skip ? cur : 1u - cur;
        s.cur[e + 1] = c;
        if (last) s.cur[kCurFinal] = c;
    }
    if (skip || blockIdx.x >= ntiles) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < WARPS * 256; i += kSortThreads) (&wcount[0][0])[i] = 0;
    __syncthreads();
    const uint32_t tile = tile_sh;
    const uint32_t *in = s.perm_buf(cur);
    uint32_t *out = s.perm_buf(1 - cur);
    const unsigned long long t0 = (unsigned long long)tile * kSortTile + (unsigned long long)warp * (kSortTile / WARPS);
    uint32_t idx[kItems], dig[kItems], rank[kItems];
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const unsigned long long i = t0 + it * 32 + lane;
        idx[it] = i < n ? in[i] : 0u;
    }
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const unsigned long long i = t0 + it * 32 + lane;
        dig[it] = i < n ? sort_digit(s, idx[it], p) : 256u + lane;  // invalid lanes never match real digits
    }
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const unsigned long long i = t0 + it * 32 + lane;
        const bool valid = i < n;
        const uint32_t peers = __match_any_sync(kFull, dig[it]);
        const int leader = __ffs(peers) - 1;
        uint32_t before = 0;
        if (lane == leader && valid) {
            before = wcount[warp][dig[it]];
            wcount[warp][dig[it]] = before + __popc(peers);
        }
        before = __shfl_sync(kFull, before, leader);
        rank[it] = before + __popc(peers & lanemask_lt());
    }
    __syncthreads();
    // thread d: this tile's count of digit d, published, then the look-back
    uint32_t cnt = 0;
#pragma unroll
    for (int w = 0; w < WARPS; w++) cnt += wcount[w][d];
    uint32_t *look = s.look_buf(par);
    uint32_t excl = 0;
    if (tile == 0) {
        st_relaxed_u32(&look[d], kLookInc | cnt);
    } else {
        st_relaxed_u32(&look[(unsigned long long)tile * 256 + d], kLookAgg | cnt);
        // look back kLookWin tiles per round trip: add published counts from
        // the nearest tile down until one carries a complete prefix; a tile not
        // yet published ends the round, and the next round starts from it
        long long t = (long long)tile - 1;
        uint32_t rounds = 0;
        bool done = false;
        while (!done) {
            uint32_t v[kLookWin];
#pragma unroll
            for (int j = 0; j < kLookWin; j++)
                v[j] = t - j >= 0 ? ld_relaxed_u32(&look[(unsigned long long)(t - j) * 256 + d]) : 0u;
            int j = 0;
#pragma unroll
            for (; j < kLookWin; j++) {
                if (!(v[j] & (kLookAgg | kLookInc))) break;
                excl += v[j] & kLookVal;
                if (v[j] & kLookInc) { done = true; break; }
            }
            if (done) break;
            t -= j;
            if (++rounds >= kLookSpins) {  // gave up: recorded, the order is not used
                atomicOr(&s.cur[kCurSortError], 1u);
                break;
            }
        }
        st_relaxed_u32(&look[(unsigned long long)tile * 256 + d], kLookInc | (excl + cnt));
    }
    // this tile's first position for digit d: the entries with a smaller
    // digit (the all-pass histogram) plus digit d's entries in earlier tiles
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    uint32_t run = incl - own + excl;
    for (int w = 0; w < warp; w++) run += wtot[w];
    for (int w = 0; w < WARPS; w++) {
        const uint32_t v = wcount[w][d];
        wcount[w][d] = run;
        run += v;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const unsigned long long i = t0 + it * 32 + lane;
        if (i < n) out[wcount[warp][dig[it]] + rank[it]] = idx[it];
    }
}

__device__ __forceinline__ bool tail_less(const LongView &v, uint32_t a, uint32_t b) {
    return lref_less(v, v.lref[a], v.lref[b]);
}

// After the last pass, entries are in (document, count desc, 16-letter prefix
// asc) order; only a long word can share its prefix with another word, so
// the runs left to order are the entries of one document with equal count
// and prefix that hold a long word, ordered here by their full bytes.  The
// first long entry of such a run sorts it by insertion; the runs are tiny.
__device__ __forceinline__ bool same_run(const SortScratch &s, uint32_t a, uint32_t b, bool seg) {
    return s.khi[a] == s.khi[b] && s.klo[a] == s.klo[b] && s.cnt[a] == s.cnt[b] && (!seg || s.doc[a] == s.doc[b]);
}
__global__ void k_fix_long(SortJob job, int passes) {
    grid_dependency_wait();
    grid_dependency_trigger();
    const SortScratch &s = job.s;
    const LongView &v = job.v;
    const unsigned long long *meta = job.meta;
    const unsigned long long n = meta[0];
    if (meta[1] == 0) return;
    const bool seg = passes > kPasses;
    uint32_t *perm = s.perm_buf(s.cur[kCurFinal]);
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t e = perm[i];
        if (v.lref[e] == 0u) continue;
        unsigned long long lo = i;
        bool leader = true;
        while (lo > 0) {
            const uint32_t q = perm[lo - 1];
            if (!same_run(s, q, e, seg)) break;
            if (v.lref[q] != 0u) { leader = false; break; }  // an earlier long entry sorts the run
            lo--;
        }
        if (!leader) continue;
        unsigned long long j = i + 1;
        while (j < n && same_run(s, perm[j], e, seg)) j++;
        if (j - lo < 2) continue;
        const unsigned long long i0 = lo;
        for (unsigned long long a = i0 + 1; a < j; a++) {
            uint32_t x = perm[a];
            unsigned long long b = a;
            while (b > i0 && tail_less(v, x, perm[b - 1])) { perm[b] = perm[b - 1]; b--; }
            perm[b] = x;
        }
    }
}

__device__ __forceinline__ unsigned long long short_len(unsigned long long hi, unsigned long long lo) {
    if (lo) return 16 - (__ffsll((long long)lo) - 1) / 8;
    return 8 - (__ffsll((long long)hi) - 1) / 8;
}

__global__ void k_gather_final(SortJob job) {
    grid_dependency_wait();
    grid_dependency_trigger();
    const SortScratch &s = job.s;
    const DevTable &out = job.out;
    const unsigned long long n = out.d_meta[0];
    if (blockIdx.x == 0 && threadIdx.x == 0 && s.cur[kCurSortError]) atomicOr(out.d_status, ST_TIMEOUT);
    const uint32_t *perm = s.perm_buf(s.cur[kCurFinal]);
    unsigned long long bytes = 0;
    // kScanUnroll entries a thread per step, all gathers issued before the stores
    const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x * kScanUnroll;
    for (unsigned long long b = (unsigned long long)blockIdx.x * blockDim.x * kScanUnroll; b < n; b += step) {
        uint32_t e[kScanUnroll];
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            const unsigned long long i = b + (unsigned long long)u * blockDim.x + threadIdx.x;
            e[u] = i < n ? perm[i] : 0u;
        }
        unsigned long long hi[kScanUnroll], lo[kScanUnroll], c[kScanUnroll];
        uint32_t r[kScanUnroll];
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            hi[u] = s.khi[e[u]];
            lo[u] = s.klo[e[u]];
            c[u] = s.cnt[e[u]];
            r[u] = s.lref[e[u]];
        }
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            const unsigned long long i = b + (unsigned long long)u * blockDim.x + threadIdx.x;
            if (i >= n) continue;
            out.khi[i] = hi[u];
            out.klo[i] = lo[u];
            out.lref[i] = r[u];
            if (out.count_bits == 32) static_cast<uint32_t *>(out.cnt)[i] = (uint32_t)c[u];
            else static_cast<unsigned long long *>(out.cnt)[i] = c[u];
            bytes += r[u] ? out.llen[r[u] - 1] : short_len(hi[u], lo[u]);
        }
    }
    for (int d = 16; d; d >>= 1) bytes += __shfl_xor_sync(kFull, bytes, d);
    if ((threadIdx.x & 31) == 0 && bytes) atomicAdd(&out.d_meta[4], bytes);
}

static int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

static int grid_for(unsigned long long n, int threads, int max_blocks) {
    unsigned long long g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > (unsigned long long)max_blocks) g = max_blocks;
    return (int)g;
}

// ---------------------------------------------------------------- radix finish
int sort_entries_launches(int passes, uint64_t cap, uint32_t skip) {
    const bool fused = (cap + kSortTile - 1) / kSortTile <= kSortFusedMaxTiles;
    const uint32_t mask = passes >= 32 ? ~0u : ((1u << passes) - 1u);
    const int per = cap < (1ull << 30) ? 1 : (fused ? 2 : 3);
    return 1 + 1 + per * (passes - __builtin_popcount(skip & mask));
}

// The passes of one sort; keyed: the compaction has prepared the sort keys
// and histograms already.
static void launch_sort(const SortJob &job, int passes, uint32_t skip, cudaStream_t st, bool keyed = false) {
    const int sms = sm_count();
    const uint64_t cap = job.s.cap;
    if (!keyed) k_hist_all<<<grid_for(cap, 256, sms * 2), 256, 0, st>>>(job, passes);
    const int ntiles = (int)((cap + kSortTile - 1) / kSortTile);
    const int fused = (uint64_t)ntiles <= kSortFusedMaxTiles;
    int lastp = -1;
    for (int p = 0; p < passes; p++)
        if (!((skip >> p) & 1u)) lastp = p;
    // e counts the launched passes: pass e reads its order from cur[e].
    // Counts below 2^30 fit the look-back words: one launch a pass; larger
    // sorts count, (scan) and scatter in separate launches.
    const bool onesweep = cap < (1ull << 30);
    for (int p = 0, e = 0; p < passes; p++) {
        if ((skip >> p) & 1u) continue;
        const int last = p == lastp;
        if (onesweep) {  // overlaps its launch with the tail of the kernel before
            launch_dependent(k_pass_one, dim3(ntiles), dim3(kSortThreads), 0, st, job, p, e, last);
        } else {
            k_pass_count<<<ntiles, kSortThreads, 0, st>>>(job, p, e, fused);
            if (!fused) k_pass_scan<<<256, 256, 0, st>>>(job, p, e, last);
            k_pass_scatter<<<ntiles, kSortThreads, 0, st>>>(job, p, e, fused, last);
        }
        e++;
    }
    launch_dependent(k_fix_long, dim3(grid_for(cap, 256, sms * 4)), dim3(256), 0, st, job, passes);
}

// LSD radix sort of the entries in ss (count n = meta[0]) into ss.perm_buf(ss.cur[passes]).
cudaError_t sort_entries(SortScratch &ss, const unsigned long long *meta, const LongView &v, int passes,
                         cudaStream_t st, uint32_t skip) {
    launch_sort(SortJob{ss, meta, v, DevTable{}}, passes, skip, st);
    return cudaGetLastError();
}

uint32_t sort_skip_mask(uint64_t max_count, uint64_t ndocs) {
    auto bytes_of = [](uint64_t x) {
        int b = 0;
        while (x) { b++; x >>= 8; }
        return b;
    };
    uint32_t m = 0;
    for (int b = bytes_of(max_count); b < 8; b++) m |= 1u << (kSortKeyPasses + b);
    const int db = std::max(1, bytes_of(ndocs ? ndocs - 1 : 0));
    for (int b = db; b < 4; b++) m |= 1u << (kPasses + b);
    return m;
}

// Zeroes a sort's state in one launch: the digit histograms, the pass
// order words, the group histograms, the first look-back buffer and the tile
// counters (the second look-back buffer is zeroed by the first pass).
__global__ void k_sort_reset(SortScratch ss, uint64_t nlook) {
    const uint64_t n0 = (uint64_t)kPassesSeg * 256, n1 = n0 + 32, n2 = n1 + 2ull * 256 * ss.group_stride,
                   n3 = n2 + nlook, n4 = n3 + 2;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (uint64_t)gridDim.x * blockDim.x) {
        if (i < n0) ss.hist_all[i] = 0u;
        else if (i < n1) ss.cur[i - n0] = 0u;
        else if (i < n2) ss.group_hist[0][i - n1] = 0u;
        else if (i < n3) ss.look[0][i - n2] = 0u;
        else ss.tile_ctr[i - n3] = 0u;
    }
}

void sort_state_reset(SortScratch &ss, cudaStream_t st) {
    const uint64_t ntiles = (ss.cap + kSortTile - 1) / kSortTile;
    const uint64_t n = (uint64_t)kPassesSeg * 256 + 32 + 2ull * 256 * ss.group_stride + 256 * ntiles + 2;
    k_sort_reset<<<grid_for(n, 256, sm_count() * 2), 256, 0, st>>>(ss, 256 * ntiles);
}

// reset + compaction (with the sort keys) + passes + long-word fix-up + gather
static void finish_by_radix(const GTable &g, uint64_t gcap8, uint64_t gcap, uint64_t glcap, SortScratch &ss,
                            DevTable &out, cudaStream_t st, uint32_t skip) {
    const int sms = sm_count();
    sort_state_reset(ss, st);
    const int nb8 = grid_for(gcap8, 256 * kScanUnroll, sms * 8), nb16 = grid_for(gcap, 256 * kScanUnroll, sms * 8),
              nbl = grid_for(glcap, 256, sms * 8);
    launch_dependent(k_compact_all, dim3(nb8 + nb16 + nbl), dim3(256), 0, st, g, (unsigned long long)gcap8,
                     (unsigned long long)gcap, (unsigned long long)glcap, ss, out, (unsigned)nb8, (unsigned)nb16);
    const SortJob job{ss, out.d_meta, LongView{ss.lref, out.loff, out.llen, out.arena}, out};
    launch_sort(job, kPasses, skip, st, true);
    launch_dependent(k_gather_final, dim3(grid_for(ss.cap, 256 * kScanUnroll, sms * 8)), dim3(256), 0, st, job);
}

// ---------------------------------------------------------------- bucket finish
size_t bucket_scratch_bytes(uint64_t cap) {
    BucketScratch s{};
    bucket_scratch_carve(s, nullptr, cap);
    return (size_t)reinterpret_cast<uintptr_t>(s.big_lref) + 4 * cap + 256;
}

void bucket_scratch_carve(BucketScratch &s, void *base, uint64_t cap) {
    uintptr_t p = reinterpret_cast<uintptr_t>(base);
    auto take = [&](size_t n) { void *r = reinterpret_cast<void *>(p); p += (n + 255) & ~(size_t)255; return r; };
    s.groups = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(kBktGroups, (cap + kBktProbes - 1) / kBktProbes));
    s.rank_blocks = s.groups;  // two keys a warp
    s.tree = 2;
    while (s.tree <= s.splits()) s.tree *= 2;
    const size_t keep = (size_t)s.groups * kBktKeep, split = s.splits();
    // twice the slots: tables are at most about half full, so a bucket may
    // hold four times its share before entries spill; batches' large tables,
    // mostly sized by estimates, are emptier still and make do with their slots
    s.slots = kOneSlot ? cap / 16 : (cap <= (1ull << 24) ? 2 * cap : cap);  // (the one-slot test build spills)
    s.kept = static_cast<ulonglong2 *>(take(keep * 16));
    s.split = static_cast<ulonglong2 *>(take(split * 16));
    s.kept_tie = static_cast<uint32_t *>(take(keep * 4));
    s.split_tie = static_cast<uint32_t *>(take(split * 4));
    s.found = static_cast<uint2 *>(take(s.groups * sizeof(uint2)));
    s.count = static_cast<uint32_t *>(take((split + 1) * kBktStride * 4));
    s.first = static_cast<uint32_t *>(take((split + 1) * 4));
    s.state = static_cast<uint32_t *>(take(64));
    s.key = static_cast<ulonglong2 *>(take(s.slots * 16));
    s.lref = static_cast<uint32_t *>(take(s.slots * 4));
    s.spill_key = static_cast<ulonglong2 *>(take(cap * 16));
    s.spill_lref = static_cast<uint32_t *>(take(cap * 4));
    s.spill_bucket = static_cast<uint32_t *>(take(cap * 4));
    s.big_key = static_cast<ulonglong2 *>(take(cap * 16));
    s.big_lref = static_cast<uint32_t *>(take(cap * 4));
}

// One table's finish; the kernels take it as their parameter (OneFinish) or
// several tables' from a device array, table blockIdx.y (FinishList): a batch's
// class and global tables are finished by one launch a step.
struct FinishJob {
    GTable g;
    unsigned long long cap8, cap16, lcap;
    BucketScratch s;
    DevTable out;
};
struct OneFinish {
    FinishJob j;
    __device__ __forceinline__ const FinishJob &get() const { return j; }
};
struct FinishList {
    const FinishJob *j;
    __device__ __forceinline__ const FinishJob &get() const { return j[blockIdx.y]; }
};

// The slots of the three hash tables, one after another.
struct TableSource {
    const FinishJob &j;
    __device__ __forceinline__ unsigned long long cap() const { return j.cap8 + j.cap16 + j.lcap; }
    __device__ __forceinline__ bool get(unsigned long long i, Key128 &k, uint32_t &tie) const {
        tie = 0u;
        if (i < j.cap8) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(&j.g.slots8[i]);
            if (!v.x) return false;
            k = count_key(v.y, be_half((uint32_t)v.x, (uint32_t)(v.x >> 32)), 0ull);
            return true;
        }
        i -= j.cap8;
        if (i < j.cap16) {
            const uint4 w = j.g.slots[i].key;
            if (key_zero(w)) return false;
            k = count_key(j.g.slots[i].cnt, be_half(w.x, w.y), be_half(w.z, w.w));
            return true;
        }
        i -= j.cap16;
        const LSlot &l = j.g.lslots[i];
        if (l.h == 0ull && l.addr == 0ull) return false;
        const uint4 f = (l.len & kLongReady) ? l.f : load_run16(reinterpret_cast<const uint8_t *>(l.addr), 16);
        k = count_key(l.cnt, be_half(f.x, f.y), be_half(f.z, f.w));
        tie = (uint32_t)i + 1u;  // 0: the short words'
        return true;
    }
};

template <class J>
__global__ void __launch_bounds__(kBktThreads) k_bucket_sample(J job) {
    grid_dependency_wait();
    grid_dependency_trigger();
    const FinishJob &j = job.get();
    if (blockIdx.x >= j.s.groups) return;
    bucket_sample(j.s, TableSource{j});
}

template <class J>
__global__ void __launch_bounds__(kRankThreads) k_bucket_rank(J job) {
    extern __shared__ __align__(16) uint8_t bsm[];
    grid_dependency_wait();
    grid_dependency_trigger();
    const FinishJob &j = job.get();
    if (blockIdx.x < j.s.rank_blocks) bucket_rank(j.s, bsm, TableSource{j}.cap());
}

// Scans the three tables once: every entry goes to its bucket, long words'
// bytes to the arena, the totals to the metadata.  Bound by L2 (the tables are
// read once, 20 bytes an entry written) and by the splitter search (11 steps of
// 16 bytes from shared memory an entry).
constexpr int kScatterThreads = 512;
constexpr int kScatterPerSm = 2;
template <class J>
__global__ void __launch_bounds__(kScatterThreads, kScatterPerSm) k_bucket_scatter(J job) {
    extern __shared__ __align__(16) uint8_t bsm[];
    __shared__ unsigned long long tot[6];  // entries (8-byte, 16-byte, long), tokens, word bytes
    grid_dependency_wait();
    grid_dependency_trigger();
    const FinishJob &j = job.get();
    if (threadIdx.x < 6) tot[threadIdx.x] = 0ull;
    SlotQueue q = slot_queue(bsm);
    const Splitters sp = load_splitters(j.s, bsm + slot_queue_smem(kScatterThreads));
    const unsigned long long step = (unsigned long long)gridDim.x * kScatterThreads * kScanUnroll;
    const unsigned long long b0 = (unsigned long long)blockIdx.x * kScatterThreads * kScanUnroll;
    unsigned long long n8 = 0, n16 = 0, nl = 0, tok = 0, bytes = 0;
    auto make = [&](const uint4 &k, unsigned long long c) -> Key128 {
        const unsigned long long khi = be_half(k.x, k.y), klo = be_half(k.z, k.w);
        if (klo) n16++;
        else n8++;
        tok += c;
        bytes += short_len(khi, klo);
        return count_key(c, khi, klo);
    };
    for (unsigned long long b = b0; b < j.cap8; b += step) {  // block-uniform
        ulonglong2 v[kScanUnroll];
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            const unsigned long long i = b + (unsigned long long)u * kScatterThreads + threadIdx.x;
            v[u] = i < j.cap8 ? *reinterpret_cast<const ulonglong2 *>(&j.g.slots8[i]) : make_ulonglong2(0ull, 0ull);
        }
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++)
            q.push(j.s, sp, v[u].x != 0ull, make_uint4((uint32_t)v[u].x, (uint32_t)(v[u].x >> 32), 0u, 0u), v[u].y, make);
    }
    for (unsigned long long b = b0; b < j.cap16; b += step) {
        uint4 k[kScanUnroll];
        unsigned long long c[kScanUnroll];
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) {
            const unsigned long long i = b + (unsigned long long)u * kScatterThreads + threadIdx.x;
            k[u] = make_uint4(0, 0, 0, 0);
            c[u] = 0;
            if (i < j.cap16) {
                k[u] = j.g.slots[i].key;
                c[u] = j.g.slots[i].cnt;
            }
        }
#pragma unroll
        for (int u = 0; u < kScanUnroll; u++) q.push(j.s, sp, !key_zero(k[u]), k[u], c[u], make);
    }
    q.flush(j.s, sp, make);
    long_slots_body(j.g.lslots, j.lcap, j.out, blockIdx.x, gridDim.x,
                    [&](unsigned long long slot, uint32_t, bool occ, unsigned long long khi, unsigned long long klo,
                        unsigned long long c, uint32_t lref, uint32_t, unsigned long long len) {
                        if (!occ) return;
                        nl++;
                        tok += c;
                        bytes += len;
                        bucket_put(j.s, sp, count_key(c, khi, klo), (uint32_t)slot + 1u, lref);
                    });
    for (int d = 16; d; d >>= 1) {
        n8 += __shfl_xor_sync(kFull, n8, d);
        n16 += __shfl_xor_sync(kFull, n16, d);
        nl += __shfl_xor_sync(kFull, nl, d);
        tok += __shfl_xor_sync(kFull, tok, d);
        bytes += __shfl_xor_sync(kFull, bytes, d);
    }
    if ((threadIdx.x & 31) == 0) {
        if (n8) atomicAdd(&tot[0], n8);
        if (n16) atomicAdd(&tot[1], n16);
        if (nl) atomicAdd(&tot[2], nl);
        if (tok) atomicAdd(&tot[3], tok);
        if (bytes) atomicAdd(&tot[4], bytes);
    }
    __syncthreads();
    if (threadIdx.x == 0 && tot[0] + tot[1] + tot[2]) {
        unsigned long long *meta = j.out.d_meta;
        atomicAdd(&meta[0], tot[0] + tot[1] + tot[2]);
        atomicAdd(&meta[3], tot[3]);
        atomicAdd(&meta[4], tot[4]);
        if (tot[0]) atomicAdd(&meta[5], tot[0]);
        if (tot[1]) atomicAdd(&meta[6], tot[1]);
    }
    bucket_close(j.s);
}

__device__ __forceinline__ void put_row(const DevTable &out, unsigned long long row, const Key128 &k, uint32_t lref) {
    unsigned long long khi, klo;
    key_prefix(k, khi, klo);
    out.khi[row] = khi;
    out.klo[row] = klo;
    out.lref[row] = lref;
    if (out.count_bits == 32) static_cast<uint32_t *>(out.cnt)[row] = (uint32_t)key_count(k);
    else static_cast<unsigned long long *>(out.cnt)[row] = key_count(k);
}

template <class J>
__global__ void __launch_bounds__(kBktSortThreads, kBktSortPerSm) k_bucket_sort(J job) {
    extern __shared__ __align__(16) uint8_t bsm[];
    grid_dependency_wait();
    grid_dependency_trigger();
    const FinishJob &j = job.get();
    if (blockIdx.x >= j.s.buckets()) return;
    bucket_sort(
        j.s, *reinterpret_cast<BucketShared *>(bsm),
        [&](unsigned long long base, uint32_t m, auto &&row) {
            for (uint32_t i = threadIdx.x; i < m; i += kBktSortThreads) {
                Key128 k;
                uint32_t r;
                row(i, k, r);
                put_row(j.out, base + i, k, r);
            }
        },
        [&](unsigned long long row, const Key128 &k, uint32_t r) { put_row(j.out, row, k, r); });
}

// Runs of equal count and prefix (only words of 17+ letters, and one of 16,
// share a prefix) ordered by their remaining bytes: the rows of a run differ
// in lref alone.  The first long row of a run sorts it by insertion; returns
// at once when the bucket sort saw no two equal keys.
template <class J>
__global__ void k_fix_rows(J job) {
    grid_dependency_wait();
    grid_dependency_trigger();
    const FinishJob &j = job.get();
    if (!j.s.state[kBktTied]) return;
    const DevTable &t = j.out;
    const unsigned long long n = t.d_meta[0];
    const LongView v{t.lref, t.loff, t.llen, t.arena};
    auto same = [&](unsigned long long a, unsigned long long b) {
        if (t.khi[a] != t.khi[b] || t.klo[a] != t.klo[b]) return false;
        return t.count_bits == 32 ? static_cast<const uint32_t *>(t.cnt)[a] == static_cast<const uint32_t *>(t.cnt)[b]
                                  : static_cast<const unsigned long long *>(t.cnt)[a] ==
                                        static_cast<const unsigned long long *>(t.cnt)[b];
    };
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        // the last row of a run sorts it (a run holds at most one row without a long reference)
        if (i == 0 || (i + 1 < n && same(i, i + 1)) || !same(i - 1, i)) continue;
        unsigned long long lo = i - 1;
        while (lo > 0 && same(lo - 1, i)) lo--;
        for (unsigned long long a = lo + 1; a <= i; a++) {
            const uint32_t x = t.lref[a];
            unsigned long long b = a;
            while (b > lo && lref_less(v, x, t.lref[b - 1])) { t.lref[b] = t.lref[b - 1]; b--; }
            t.lref[b] = x;
        }
    }
}

// sample, rank, scatter, sort, fix-up
constexpr int kBucketLaunches = 5;

// most: the largest table's scratch.
template <class J>
static cudaError_t launch_buckets(const J &job, const BucketScratch &most, uint64_t cap, int ntab, cudaStream_t st) {
    const int sms = sm_count();
    const size_t smem = splitters_smem(most);
    const uint32_t groups = most.groups;
    cudaError_t e = ensure_smem_limit((const void *)k_bucket_rank<J>, (int)kept_smem(kBktGroups));
    if (e == cudaSuccess) e = ensure_smem_limit((const void *)k_bucket_scatter<J>, (int)(kSplittersMax + slot_queue_smem(kScatterThreads)));
    if (e == cudaSuccess) e = ensure_smem_limit((const void *)k_bucket_sort<J>, (int)sizeof(BucketShared));
    if (e != cudaSuccess) return e;
    launch_dependent(k_bucket_sample<J>, dim3(groups, ntab), dim3(kBktThreads), 0, st, job);
    launch_dependent(k_bucket_rank<J>, dim3(groups, ntab), dim3(kRankThreads), kept_smem(groups), st, job);
    launch_dependent(k_bucket_scatter<J>, dim3(grid_for(cap, kScatterThreads * kScanUnroll, sms * kScatterPerSm), ntab),
                     dim3(kScatterThreads), smem + slot_queue_smem(kScatterThreads), st, job);
    launch_dependent(k_bucket_sort<J>, dim3(most.buckets(), ntab), dim3(kBktSortThreads), sizeof(BucketShared), st, job);
    launch_dependent(k_fix_rows<J>, dim3(grid_for(cap, 256, sms), ntab), dim3(256), 0, st, job);
    return cudaGetLastError();
}

bool finish_by_buckets(const BucketScratch &bs, uint32_t skip) {
    return bs.key && ((skip >> (kSortKeyPasses + 6)) & 3u) == 3u;
}

int finish_table_launches(const SortScratch &ss, const BucketScratch &bs, uint32_t skip) {
    if (finish_by_buckets(bs, skip)) return kBucketLaunches;
    return 2 + sort_entries_launches(kPasses, ss.cap, skip) - 1 + 1;
}

cudaError_t finish_table(const GTable &g, uint64_t gcap8, uint64_t gcap, uint64_t glcap, SortScratch &ss,
                         const BucketScratch &bs, DevTable &out, cudaStream_t st, uint32_t skip) {
    if (finish_by_buckets(bs, skip))
        return launch_buckets(OneFinish{FinishJob{g, gcap8, gcap, glcap, bs, out}}, bs, gcap8 + gcap + glcap, 1, st);
    finish_by_radix(g, gcap8, gcap, glcap, ss, out, st, skip);
    return cudaGetLastError();
}

size_t finish_tables_job_bytes(int n) { return sizeof(FinishJob) * (size_t)(n > 0 ? n : 1); }

int finish_tables_launches(const FinishSpec *spec, int n, uint32_t skip) {
    int k = 0;
    bool buckets = false;
    for (int t = 0; t < n; t++) {
        if (finish_by_buckets(*spec[t].bs, skip)) buckets = true;
        else k += finish_table_launches(*spec[t].ss, *spec[t].bs, skip);
    }
    return k + (buckets ? kBucketLaunches : 0);
}

cudaError_t finish_tables(const FinishSpec *spec, int n, void *d_jobs, cudaStream_t st, uint32_t skip) {
    std::vector<FinishJob> jobs;
    uint64_t cap = 0;
    const BucketScratch *most = nullptr;
    for (int t = 0; t < n; t++) {
        const FinishSpec &f = spec[t];
        if (!finish_by_buckets(*f.bs, skip)) {
            const cudaError_t e = finish_table(f.g, f.gcap8, f.gcap, f.glcap, *f.ss, *f.bs, *f.out, st, skip);
            if (e != cudaSuccess) return e;
            continue;
        }
        jobs.push_back(FinishJob{f.g, f.gcap8, f.gcap, f.glcap, *f.bs, *f.out});
        cap = std::max<uint64_t>(cap, f.gcap8 + f.gcap + f.glcap);
        if (!most || f.bs->groups > most->groups) most = f.bs;
    }
    if (jobs.empty()) return cudaSuccess;
    const cudaError_t e =
        cudaMemcpyAsync(d_jobs, jobs.data(), sizeof(FinishJob) * jobs.size(), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    return launch_buckets(FinishList{static_cast<const FinishJob *>(d_jobs)}, *most, cap, (int)jobs.size(), st);
}

// ---------------------------------------------------------------- merge
__global__ void k_merge_insert(const MergeSrc *src, const unsigned long long *chunk_start, uint32_t nsrc, GTable g) {
    // table t owns blocks [chunk_start[t], chunk_start[t+1])
    uint32_t lo = 0, hi = nsrc;
    const unsigned long long b = blockIdx.x;
    while (hi - lo > 1) {
        uint32_t mid = (lo + hi) / 2;
        if (chunk_start[mid] <= b) lo = mid; else hi = mid;
    }
    const MergeSrc t = src[lo];
    const unsigned long long n = t.meta[0];
    const unsigned long long i0 = (b - chunk_start[lo]) * kMergeChunk;
    for (unsigned long long ib = i0 + (threadIdx.x & ~31u); ib < i0 + kMergeChunk && ib < n; ib += blockDim.x) {
        const unsigned long long i = ib + (threadIdx.x & 31);  // whole warps iterate together
        const bool valid = i < i0 + kMergeChunk && i < n;
        unsigned long long c = 0;
        uint32_t r = 0;
        if (valid) {
            c = t.count_bits == 32 ? static_cast<const uint32_t *>(t.cnt)[i]
                                   : static_cast<const unsigned long long *>(t.cnt)[i];
            r = t.lref[i];
        }
        if (valid && r == 0) {
            unsigned long long hi8 = t.khi[i], lo8 = t.klo[i];
            uint4 k;
            k.x = __byte_perm((uint32_t)(hi8 >> 32), 0, 0x0123);
            k.y = __byte_perm((uint32_t)hi8, 0, 0x0123);
            k.z = __byte_perm((uint32_t)(lo8 >> 32), 0, 0x0123);
            k.w = __byte_perm((uint32_t)lo8, 0, 0x0123);
            table_insert_key(g, k, c);
        }
        if (valid && r != 0)
            long_insert(g, t.arena + t.loff[r - 1], t.llen[r - 1], c, nullptr, nullptr);
    }
}

cudaError_t launch_merge_insert(const MergeSrc *d_src, const uint64_t *d_chunk_start, uint32_t nsrc,
                                uint64_t total_chunks, const GTable &g, cudaStream_t s) {
    if (total_chunks == 0) return cudaSuccess;
    k_merge_insert<<<(unsigned)total_chunks, 256, 0, s>>>(d_src, reinterpret_cast<const unsigned long long *>(d_chunk_start), nsrc, g);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- top-k
__global__ void k_topk_copy(DevTable in, unsigned long long k, DevTable out) {
    const unsigned long long n = in.d_meta[0];
    const unsigned long long m = n < k ? n : k;
    const unsigned long long nl = in.d_meta[1], ab = in.d_meta[2];
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) {
        out.d_meta[0] = m;
        out.d_meta[1] = nl;
        out.d_meta[2] = ab;
        *out.d_status = *in.d_status;
    }
    // meta[1] keeps the length of the long words' list, all of which is copied; the
    // rows' own kinds are counted (a merge sizes its tables by them)
    unsigned long long tok = 0, bytes = 0, n8 = 0, n16 = 0;
    for (unsigned long long i = t; i < m; i += stride) {
        const unsigned long long klo = in.klo[i];
        out.khi[i] = in.khi[i];
        out.klo[i] = klo;
        uint32_t r = in.lref[i];
        n8 += !r && !klo ? 1u : 0u;
        n16 += !r && klo ? 1u : 0u;
        out.lref[i] = r;
        unsigned long long c;
        if (in.count_bits == 32) c = static_cast<const uint32_t *>(in.cnt)[i];
        else c = static_cast<const unsigned long long *>(in.cnt)[i];
        if (out.count_bits == 32) static_cast<uint32_t *>(out.cnt)[i] = (uint32_t)c;
        else static_cast<unsigned long long *>(out.cnt)[i] = c;
        tok += c;
        bytes += r ? in.llen[r - 1] : short_len(in.khi[i], klo);
    }
    for (unsigned long long i = t; i < nl; i += stride) {
        out.loff[i] = in.loff[i];
        out.llen[i] = in.llen[i];
    }
    for (unsigned long long i = t; i < ab; i += stride) out.arena[i] = in.arena[i];
    for (int d = 16; d; d >>= 1) {
        tok += __shfl_xor_sync(kFull, tok, d);
        bytes += __shfl_xor_sync(kFull, bytes, d);
        n8 += __shfl_xor_sync(kFull, n8, d);
        n16 += __shfl_xor_sync(kFull, n16, d);
    }
    if ((threadIdx.x & 31) == 0) {
        if (tok) atomicAdd(&out.d_meta[3], tok);
        if (bytes) atomicAdd(&out.d_meta[4], bytes);
        if (n8) atomicAdd(&out.d_meta[5], n8);
        if (n16) atomicAdd(&out.d_meta[6], n16);
    }
}

cudaError_t launch_topk_copy(const DevTable &in, uint64_t k, DevTable &out, cudaStream_t s) {
    uint64_t work = in.cap > in.arena_cap ? in.cap : in.arena_cap;
    k_topk_copy<<<grid_for(work, 256, sm_count() * 8), 256, 0, s>>>(in, k, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- export
constexpr int kScanBlock = 1024;  // elements per scan block (256 threads x 4)

size_t export_scratch_bytes(uint64_t cap) {
    uint64_t nb = (cap + kScanBlock - 1) / kScanBlock;
    return (nb + 8) * 8 + 256;
}

__global__ void k_export_lens(DevTable t, unsigned long long *offs, unsigned long long *blocksum) {
    __shared__ unsigned long long part[256];
    const unsigned long long n = t.d_meta[0];
    const unsigned long long b0 = (unsigned long long)blockIdx.x * kScanBlock;
    if (b0 >= n && !(n == 0 && blockIdx.x == 0)) return;
    unsigned long long v[4], sum = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        unsigned long long i = b0 + threadIdx.x * 4 + j;
        unsigned long long len = 0;
        if (i < n) {
            uint32_t r = t.lref[i];
            len = r ? t.llen[r - 1] : short_len(t.khi[i], t.klo[i]);
        }
        v[j] = len;
        sum += len;
    }
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int d = 1; d < 256; d <<= 1) {
        unsigned long long x = threadIdx.x >= (unsigned)d ? part[threadIdx.x - d] : 0ull;
        __syncthreads();
        part[threadIdx.x] += x;
        __syncthreads();
    }
    unsigned long long run = part[threadIdx.x] - sum;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        unsigned long long i = b0 + threadIdx.x * 4 + j;
        if (i < n) offs[i] = run;
        run += v[j];
    }
    if (threadIdx.x == 255) blocksum[blockIdx.x] = part[255];
}

// Exclusive scan of the scan blocks' byte counts, in one block: each thread
// sums a contiguous run of them, the run totals are scanned in shared
// memory, and each thread writes its run's prefixes.
constexpr int kBlockSumThreads = 1024;
__global__ void __launch_bounds__(kBlockSumThreads) k_export_blocksums(const DevTable t, unsigned long long *blocksum,
                                                                       unsigned long long *offs) {
    __shared__ unsigned long long part[kBlockSumThreads];
    const unsigned long long n = t.d_meta[0];
    const unsigned long long nb = (n + kScanBlock - 1) / kScanBlock;
    const unsigned long long per = (nb + kBlockSumThreads - 1) / kBlockSumThreads;
    const unsigned long long lo = threadIdx.x * per, hi = lo + per < nb ? lo + per : nb;
    unsigned long long own = 0;
    for (unsigned long long b = lo; b < hi; b++) own += blocksum[b];
    part[threadIdx.x] = own;
    __syncthreads();
    for (int o = 1; o < kBlockSumThreads; o <<= 1) {
        const unsigned long long x = threadIdx.x >= (unsigned)o ? part[threadIdx.x - o] : 0ull;
        __syncthreads();
        part[threadIdx.x] += x;
        __syncthreads();
    }
    unsigned long long run = part[threadIdx.x] - own;
    for (unsigned long long b = lo; b < hi; b++) {
        const unsigned long long v = blocksum[b];
        blocksum[b] = run;
        run += v;
    }
    if (threadIdx.x == kBlockSumThreads - 1) offs[n] = part[kBlockSumThreads - 1];
}

__global__ void k_export_write(DevTable t, unsigned long long *offs, const unsigned long long *blocksum, uint8_t *words) {
    const unsigned long long n = t.d_meta[0];
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        unsigned long long o = offs[i] + blocksum[i / kScanBlock];
        offs[i] = o;
        uint32_t r = t.lref[i];
        if (r) {
            const uint8_t *p = t.arena + t.loff[r - 1];
            unsigned long long len = t.llen[r - 1];
            for (unsigned long long j = 0; j < len; j++) words[o + j] = p[j];
        } else {
            unsigned long long hi = t.khi[i], lo = t.klo[i];
            unsigned long long len = short_len(hi, lo);
            for (unsigned long long j = 0; j < len; j++)
                words[o + j] = (uint8_t)((j < 8 ? hi >> (56 - 8 * j) : lo >> (56 - 8 * (j - 8))) & 0xFF);
        }
    }
}

// A table of at most kExportSmall rows in one block: lengths, their scan and the
// bytes, a thread its rows' words of up to 64 letters, the whole warp each longer
// one.  One launch for three, but one block writes slowly: tables of more than
// 16 KB of letters, or of more than 24 a row, go to the grid.  Export, us, one
// block | grid: 100 words of 8 letters 36 | 44, of 30 40 | 43, of 40 50 | 44; 1,000 of
// 14 39 | 44, of 20 50 | 44; 2,000 of 7 38 | 44, of 14 51 | 44; 4,000 of 4 38 | 43, of 7
// 50 | 43.
constexpr int kExportSmall = 4096, kExportSmallThreads = 1024;
__global__ void __launch_bounds__(kExportSmallThreads) k_export_small(DevTable t, uint32_t n, unsigned long long *offs,
                                                                      uint8_t *words) {
    constexpr int kPer = kExportSmall / kExportSmallThreads;
    __shared__ unsigned long long wsum[kExportSmallThreads / 32];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, i0 = threadIdx.x * kPer;
    unsigned long long hi[kPer], lo[kPer], len[kPer], own = 0;
    uint32_t r[kPer];
#pragma unroll
    for (int q = 0; q < kPer; q++) {
        const uint32_t i = i0 + q;
        r[q] = i < n ? t.lref[i] : 0u;
        hi[q] = i < n ? t.khi[i] : 0ull;
        lo[q] = i < n ? t.klo[i] : 0ull;
    }
#pragma unroll
    for (int q = 0; q < kPer; q++) {
        len[q] = i0 + q >= n ? 0ull : (r[q] ? t.llen[r[q] - 1] : short_len(hi[q], lo[q]));
        own += len[q];
    }
    unsigned long long incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long x = __shfl_up_sync(kFull, incl, o);
        if (lane >= (uint32_t)o) incl += x;
    }
    if (lane == 31u) wsum[warp] = incl;
    __syncthreads();
    unsigned long long run = incl - own;
    for (uint32_t w = 0; w < warp; w++) run += wsum[w];
#pragma unroll
    for (int q = 0; q < kPer; q++) {
        const uint32_t i = i0 + q;
        const bool have = i < n, warp_word = have && len[q] > 64;  // (such words by the whole warp)
        const uint8_t *p = r[q] ? t.arena + t.loff[r[q] - 1] : nullptr;
        if (have) offs[i] = run;
        if (have && !warp_word)
            for (unsigned long long j = 0; j < len[q]; j++)
                words[run + j] = p ? p[j] : (uint8_t)((j < 8 ? hi[q] >> (56 - 8 * j) : lo[q] >> (56 - 8 * (j - 8))) & 0xFF);
        for (uint32_t m = __ballot_sync(kFull, warp_word); m; m &= m - 1u) {
            const int l = __ffs((int)m) - 1;
            const unsigned long long src = __shfl_sync(kFull, (unsigned long long)reinterpret_cast<uintptr_t>(p), l);
            const unsigned long long to = __shfl_sync(kFull, run, l), letters = __shfl_sync(kFull, len[q], l);
            for (unsigned long long j = lane; j < letters; j += 32) words[to + j] = reinterpret_cast<const uint8_t *>(src)[j];
        }
        run += len[q];
    }
    if (threadIdx.x == kExportSmallThreads - 1) offs[n] = run;
}

cudaError_t launch_export(const DevTable &t, uint64_t n, uint64_t word_bytes, void *scratch, uint8_t *d_words,
                          unsigned long long *d_offs, cudaStream_t s) {
    if (n <= (uint64_t)kExportSmall && word_bytes <= (16u << 10) && word_bytes <= 24 * n) {
        k_export_small<<<1, kExportSmallThreads, 0, s>>>(t, (uint32_t)n, d_offs, d_words);
        return cudaGetLastError();
    }
    unsigned long long *blocksum = static_cast<unsigned long long *>(scratch);
    const int nb = (int)((n + kScanBlock - 1) / kScanBlock);  // (n = 0 has no letters: above)
    k_export_lens<<<nb, 256, 0, s>>>(t, d_offs, blocksum);
    k_export_blocksums<<<1, kBlockSumThreads, 0, s>>>(t, blocksum, d_offs);
    k_export_write<<<grid_for(n, 256, sm_count() * 8), 256, 0, s>>>(t, d_offs, blocksum, d_words);
    return cudaGetLastError();
}

}  // namespace wc
