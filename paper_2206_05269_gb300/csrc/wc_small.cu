// One short document counted, sorted and written by one block.
//
// A text of a few kilobytes is a few hundred words: counting it by the general
// path was a dozen launches (tables cleared, counted, sampled, scattered, sorted,
// fixed), each mostly its own latency.  Here the text sits in shared memory and
// everything refers to it by position: the distinct words are found with a hash
// table of word numbers (equality is always decided on the bytes, whatever the
// length), ordered by count and bytes (order_by_parts; words of 17+ letters that
// share count and prefix compare their remaining bytes there and then), and the
// rows are written to the table.  Bound by latency: about ten block barriers.
//   us          general path, here: count + size (host clock)
//   2 KB, 16 KB ordinary words   131, 36    142, 48
//   2 KB, 16 KB distinct words   140, 41    164, 88
//   16 KB of 17+ letter words with equal counts and prefixes   11,500, 180
//   2 KB, count + top 100 read back: 152, 109; the kernel itself 9.7
// The limit is the shared memory's: 204 KB at 16 KB of text (a key an entry).
#include <algorithm>

#include "wc_bucket.cuh"
#include "wc_internal.h"

namespace wc {

constexpr int kSmallThreads = 1024;
constexpr uint32_t kSmallText = (uint32_t)kSmallCountMax;
constexpr uint32_t kSmallChunks = kSmallText / 16 + 1;  // 16-byte pieces of a text at any alignment
constexpr uint32_t kSmallWords = kSmallText / 2 + 8;    // words at most (one letter, one separator)
// Distinct words at most: 26 of one letter (2 bytes each), 676 of two (3), the
// rest at least 4 bytes each.
constexpr uint32_t kSmallDistinct = (26 + 676 + (kSmallText - 26 * 2 - 676 * 3) / 4 + 8 + 7) & ~7u;
constexpr uint32_t kSmallSlots = 8192, kSmallParts = 256;
static_assert(kSmallDistinct < kSmallSlots * 3 / 4 && kSmallText < 65536, "the table is never full; 16-bit positions");

struct SmallShared {
    uint8_t text[(kSmallChunks + 2) * 16];  // spaces around the text
    uint32_t word[kSmallWords];             // position | length << 16
    ulonglong2 key[kSmallDistinct];
    uint32_t row[kSmallDistinct];           // the entry's word
    union {
        struct {
            uint32_t slot[kSmallSlots];  // 1 + word number
            uint32_t count[kSmallSlots];
        } tab;
        struct {
            uint16_t found[kSmallDistinct], prow[kSmallDistinct], byparts[kSmallDistinct];
            ulonglong2 coarse[kBktCoarse + 1];
            KeyRange range[kBktCoarse];
            uint32_t pcount[kSmallParts];
        } sort;
    };
    uint16_t mask[kSmallChunks + 2];  // letters of each piece
    uint32_t nword, nent, n16, nlong;
    uint32_t bytes, arena;
};
static_assert(sizeof(SmallShared) <= 227 * 1024 - 64, "one block's shared memory");

__global__ void __launch_bounds__(kSmallThreads) k_count_small(const uint8_t *text, uint32_t nbytes, DevTable out) {
    extern __shared__ __align__(16) uint8_t smem[];
    SmallShared &sh = *reinterpret_cast<SmallShared *>(smem);
    const uint32_t t = threadIdx.x, lane = t & 31u;
    const uintptr_t vb = reinterpret_cast<uintptr_t>(text), ve = vb + nbytes, base = vb & ~(uintptr_t)15;
    const uint32_t chunks = (uint32_t)((ve - base + 15) >> 4);
    // slots: at least twice the distinct words a text of this size usually has,
    // and more than it can have
    uint32_t nslot = 1024;
    while (nslot < kSmallSlots && nslot < nbytes / 2) nslot <<= 1;
    if (t == 0) {
        sh.nword = sh.nent = sh.n16 = sh.nlong = 0u;
        sh.bytes = sh.arena = 0u;
    }
    for (uint32_t i = t; i < nslot; i += kSmallThreads) {
        sh.tab.slot[i] = 0u;
        sh.tab.count[i] = 0u;
    }
    // ---- the text, one 16-byte piece in front of it, and its letters
    for (uint32_t c = t; c < chunks + 2; c += kSmallThreads) {
        uint4 v = make_uint4(0x20202020u, 0x20202020u, 0x20202020u, 0x20202020u);
        if (c >= 1 && c <= chunks) {
            const uintptr_t a = base + 16 * (uintptr_t)(c - 1);
            v = mask_outside_doc(ld_stream16(reinterpret_cast<const void *>(a)), a, vb, ve);
        }
        reinterpret_cast<uint4 *>(sh.text)[c] = v;
        sh.mask[c] = (uint16_t)letter_mask16(v);
    }
    __syncthreads();
    // ---- words: every start with its length, in any order of pieces
    for (uint32_t c0 = 1; c0 <= chunks; c0 += kSmallThreads) {
        const uint32_t c = c0 + t;
        uint32_t m = 0, s = 0;
        if (c <= chunks) {
            m = sh.mask[c];
            s = m & ~((m << 1) | ((uint32_t)sh.mask[c - 1] >> 15)) & 0xFFFFu;
        }
        const uint32_t own = __popc(s);
        uint32_t incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(kFull, incl, o);
            if (lane >= (uint32_t)o) incl += x;
        }
        uint32_t at = 0;
        if (lane == 31u) at = atomicAdd(&sh.nword, incl);
        at = __shfl_sync(kFull, at, 31) + incl - own;
        while (s) {
            const uint32_t j = (uint32_t)__ffs((int)s) - 1u;
            s &= s - 1u;
            uint32_t len = (uint32_t)__ffs((int)~(m >> j)) - 1u;  // letters of this piece from j (bits past 15 are 0)
            if (j + len == 16u)
                for (uint32_t d = c + 1;; d++) {  // the last piece (spaces) ends any word
                    const uint32_t x = sh.mask[d];
                    if (x == 0xFFFFu) {
                        len += 16u;
                        continue;
                    }
                    len += (uint32_t)__ffs((int)~x) - 1u;
                    break;
                }
            sh.word[at++] = (16u * c + j) | (len << 16);
        }
    }
    __syncthreads();
    // ---- distinct words
    const uint32_t nword = sh.nword;
    auto key_at = [&](uint32_t w, uint32_t j) {  // letters [j, j + 16) of a word, 0 past its end
        const uint32_t left = (w >> 16) - j;
        return load_key16(sh.text, (w & 0xFFFFu) + j, left < 16u ? left : 16u);
    };
    auto key16 = [&](uint32_t w) { return key_at(w, 0u); };
    auto last16 = [&](uint32_t w) { return load_key16(sh.text, (w & 0xFFFFu) + (w >> 16) - 16u, 16u); };
    for (uint32_t i = t; i < nword; i += kSmallThreads) {
        const uint32_t w = sh.word[i], len = w >> 16;
        const uint4 k = key16(w);
        uint32_t h = k.x * 0x9E3779B1u + k.y * 0x85EBCA77u + k.z * 0xC2B2AE3Du + k.w * 0x27D4EB2Fu;
        if (len > 16u) {
            const uint4 l = last16(w);
            h += l.x * 0x165667B1u + l.y * 0xD3A2646Du + l.z * 0xFD7046C5u + l.w * 0xB55A4F09u + len;
        }
        h ^= h >> 15;
        h *= 0x2C1B3C6Du;
        uint32_t s = kOneSlot ? 0u : (h >> 10) & (nslot - 1u);
        for (uint32_t probe = 0; probe < nslot; probe++) {
            uint32_t cur = *reinterpret_cast<volatile uint32_t *>(&sh.tab.slot[s]);
            if (cur == 0u) cur = atomicCAS(&sh.tab.slot[s], 0u, i + 1u);
            bool same = cur == 0u;
            if (!same) {
                const uint32_t o = sh.word[cur - 1u];
                same = (o >> 16) == len && key_eq(key16(o), k);
                for (uint32_t j = 16; same && j < len; j += 16) same = key_eq(key_at(o, j), key_at(w, j));
            }
            if (same) {
                atomicAdd(&sh.tab.count[s], 1u);
                break;
            }
            s = (s + 1u) & (nslot - 1u);
        }
    }
    __syncthreads();
    // ---- entries with their keys (count, 16-letter prefix)
    uint32_t bytes = 0, n16 = 0;
    for (uint32_t s0 = 0; s0 < nslot; s0 += kSmallThreads) {
        const uint32_t cur = sh.tab.slot[s0 + t];
        const uint32_t m = __ballot_sync(kFull, cur != 0u);
        uint32_t at = 0;
        if (lane == 0u && m) at = atomicAdd(&sh.nent, (uint32_t)__popc(m));
        at = __shfl_sync(kFull, at, 0) + __popc(m & ((1u << lane) - 1u));
        if (cur) {
            const uint32_t w = sh.word[cur - 1u];
            const uint4 k = key16(w);
            const unsigned long long ph = pack5(be_half(k.x, k.y)), pl = pack5(be_half(k.z, k.w));
            sh.key[at] = make_ulonglong2(((0xFFFFull - sh.tab.count[s0 + t]) << 48) | (ph << 8) | (pl >> 32), pl << 32);
            sh.row[at] = w;
            bytes += w >> 16;
            n16 += (w >> 16) > 8u && (w >> 16) <= 16u ? 1u : 0u;
        }
    }
    bytes = __reduce_add_sync(kFull, bytes);
    n16 = __reduce_add_sync(kFull, n16);
    if (lane == 0u && bytes) {
        atomicAdd(&sh.bytes, bytes);
        atomicAdd(&sh.n16, n16);
    }
    __syncthreads();
    // ---- order (the table's memory becomes the lists')
    const uint32_t n = sh.nent;
    for (uint32_t e = t; e < n; e += kSmallThreads) sh.sort.found[e] = (uint16_t)e;
    for (uint32_t i = t; i < kSmallParts; i += kSmallThreads) sh.sort.pcount[i] = 0u;
    __syncthreads();
    const uint16_t *order = order_by_parts<kSmallThreads, kSmallParts>(
        n, sh.sort.found, sh.sort.prow, sh.sort.byparts, sh.sort.coarse, sh.sort.range, sh.sort.pcount,
        [&](uint32_t e) { return sh.key[e]; },
        [&](uint32_t x, uint32_t y) {  // equal counts and prefixes: words of 17+ letters, and at most one of 16
            const uint32_t a = sh.row[x], b = sh.row[y], la = a >> 16, lb = b >> 16, l = la < lb ? la : lb;
            for (uint32_t j = 16; j < l; j += 16) {
                const uint4 p = key_at(a, j), q = key_at(b, j);
                if (!key_eq(p, q)) {
                    const unsigned long long ph = be_half(p.x, p.y), qh = be_half(q.x, q.y);
                    return ph != qh ? ph < qh : be_half(p.z, p.w) < be_half(q.z, q.w);
                }
            }
            return la < lb;
        });
    // ---- rows; a long word's bytes are copied by its warp, followed by one 0
    for (uint32_t i0 = 0; i0 < n; i0 += kSmallThreads) {
        const uint32_t i = i0 + t;
        uint32_t w = 0, off = 0, lref = 0;
        if (i < n) {
            const uint32_t e = order[i], cnt = 0xFFFFu - (uint32_t)(sh.key[e].x >> 48);
            w = sh.row[e];
            const uint4 k = key16(w);
            out.khi[i] = be_half(k.x, k.y);
            out.klo[i] = be_half(k.z, k.w);
            if (out.count_bits == 32) static_cast<uint32_t *>(out.cnt)[i] = cnt;
            else static_cast<unsigned long long *>(out.cnt)[i] = cnt;
            if ((w >> 16) > 16u) {
                lref = atomicAdd(&sh.nlong, 1u) + 1u;
                off = atomicAdd(&sh.arena, (w >> 16) + 1u);
                out.loff[lref - 1u] = off;
                out.llen[lref - 1u] = w >> 16;
            }
            out.lref[i] = lref;
        }
        for (uint32_t m = __ballot_sync(kFull, lref != 0u); m; m &= m - 1u) {
            const int l = __ffs((int)m) - 1;
            const uint32_t lw = __shfl_sync(kFull, w, l), lo = __shfl_sync(kFull, off, l);
            for (uint32_t j = lane; j <= lw >> 16; j += 32u)
                out.arena[lo + j] = j < lw >> 16 ? (uint8_t)(sh.text[(lw & 0xFFFFu) + j] | 0x20u) : (uint8_t)0;
        }
    }
    __syncthreads();
    if (t == 0) {
        unsigned long long *meta = out.d_meta;
        meta[0] = n;
        meta[1] = sh.nlong;
        meta[2] = sh.arena;
        meta[3] = nword;
        meta[4] = sh.bytes;
        meta[5] = n - sh.n16 - sh.nlong;
        meta[6] = sh.n16;
        meta[7] = 0ull;
        *out.d_status = 0u;
    }
}

void small_count_caps(uint64_t nbytes, uint64_t *cap, uint64_t *lcap, uint64_t *arena) {
    *cap = std::min<uint64_t>(nbytes / 2 + 1, kSmallDistinct);
    *lcap = nbytes / 18 + 1;  // 17 letters and a separator
    *arena = nbytes + *lcap + 16;
}

cudaError_t launch_count_small(const uint8_t *d_text, uint64_t nbytes, DevTable &out, cudaStream_t s) {
    const cudaError_t e = ensure_smem_limit((const void *)k_count_small, (int)sizeof(SmallShared));
    if (e != cudaSuccess) return e;
    k_count_small<<<1, kSmallThreads, sizeof(SmallShared), s>>>(d_text, (uint32_t)nbytes, out);
    return cudaGetLastError();
}

}  // namespace wc
