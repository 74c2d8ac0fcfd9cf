// Bucket sort of table entries by one 128-bit key each.
//
// Key of an entry: 48 bits that order first (a table: the count complemented,
// so that larger counts come first; a batch's (document, word) rows: the
// document, then the count complemented), then the 16-letter prefix packed 5
// bits a letter (80 bits: integer order is word order, a proper prefix first).
// Keys tie only among words of 17+ letters that share their prefix; those runs
// are ordered by their remaining bytes afterwards.
//
// The entries sit unordered in hash tables.  Four launches order them:
//   sample    blocks read evenly spread table slots and keep, in order, some of the keys
//             they find (the slots are in hash order: a random sample);
//   rank      each kept key's place among all of them is the sum of its places in
//             the blocks' lists; evenly spaced ones are the splitters (about
//             every fourth: buckets of more than four times their share are
//             then about 1 in 10^4 ... 10^5);
//   scatter   the tables are scanned once; each entry finds its bucket by
//             bisection among the splitters and is appended to it;
//   sort      one block a bucket: it splits its few hundred entries again
//             by keys of its own, ranks each part by counting, and writes the
//             finished rows at their place (the bucket's first row is the sum of
//             the buckets before it).
// No kernel waits for another block, and nothing is moved twice.  (Before: the
// entries compacted, 13-14 radix passes or a run sort and 8-10 merge rounds,
// then a gather by index.)
#pragma once
#include "wc_internal.h"

namespace wc {

struct Key128 {
    unsigned long long hi, lo;
};
__device__ __forceinline__ bool key_less(const Key128 &a, const Key128 &b) { return a.hi != b.hi ? a.hi < b.hi : a.lo < b.lo; }
__device__ __forceinline__ bool key_same(const Key128 &a, const Key128 &b) { return a.hi == b.hi && a.lo == b.lo; }

// (first: the 48 bits that order first; khi, klo: the big-endian halves of the first 16 letters.)
__device__ __forceinline__ Key128 bucket_key(unsigned long long first, unsigned long long khi, unsigned long long klo) {
    const unsigned long long ph = pack5(khi), pl = pack5(klo);
    return Key128{(first << 16) | (ph >> 24), (ph << 40) | pl};
}
constexpr unsigned long long kFirstMask = (1ull << 48) - 1;
__device__ __forceinline__ Key128 count_key(unsigned long long cnt, unsigned long long khi, unsigned long long klo) {
    return bucket_key(~cnt & kFirstMask, khi, klo);
}
__device__ __forceinline__ void key_prefix(const Key128 &k, unsigned long long &khi, unsigned long long &klo) {
    khi = unpack5(((k.hi & 0xFFFFull) << 24) | (k.lo >> 40));
    klo = unpack5(k.lo & 0xFFFFFFFFFFull);
}
__device__ __forceinline__ unsigned long long key_count(const Key128 &k) { return ~(k.hi >> 16) & kFirstMask; }

// The big-endian key halves of 16 key bytes.
__device__ __forceinline__ unsigned long long be_half(uint32_t x, uint32_t y) {
    return ((unsigned long long)__byte_perm(x, 0, 0x0123) << 32) | __byte_perm(y, 0, 0x0123);
}

// Compares two words whose 16-byte prefixes are equal (given by their long
// references) by the bytes after the prefix (a word that fits the prefix is a proper prefix of a longer one).
__device__ __forceinline__ bool lref_less(const LongView &v, uint32_t ra, uint32_t rb) {
    if (ra == 0) return rb != 0;   // the 16-letter (or shorter) word is a prefix
    if (rb == 0) return false;
    const uint8_t *pa = v.arena + v.loff[ra - 1], *pb = v.arena + v.loff[rb - 1];
    unsigned long long la = v.llen[ra - 1], lb = v.llen[rb - 1];
    unsigned long long m = la < lb ? la : lb;
    for (unsigned long long i = 16; i < m; i++)
        if (pa[i] != pb[i]) return pa[i] < pb[i];
    return la < lb;
}

__device__ __forceinline__ bool row_less(const ulonglong2 &a, uint32_t ra, const ulonglong2 &b, uint32_t rb) {
    return a.x != b.x ? a.x < b.x : (a.y != b.y ? a.y < b.y : ra < rb);
}

// ---------------------------------------------------------------- sample
constexpr int kBktThreads = 256;
constexpr int kBktProbes = 512;  // slots a sample block reads

// Source: cap slots; get(i, key, tie): whether slot i holds an entry, its key
// and a number that tells entries of equal keys apart (all of them: two equal
// samples would take one rank and leave the next, maybe a splitter, unwritten).
template <class Source>
__device__ __forceinline__ void bucket_sample(const BucketScratch &s, const Source &src) {
    __shared__ uint32_t nv;
    const uint32_t g = blockIdx.x, t = threadIdx.x;
    for (uint32_t i = g * kBktThreads + t; i < s.buckets(); i += s.groups * kBktThreads) s.count[i * kBktStride] = 0u;
    if (g == 0 && t < 8) s.state[t] = 0u;
    if (t == 0) nv = 0u;
    __syncthreads();
    const unsigned long long cap = src.cap(), all = (unsigned long long)s.groups * kBktProbes, probes = cap < all ? cap : all;
    constexpr int kPer = kBktProbes / kBktThreads;
    Key128 k[kPer];
    uint32_t e[kPer], at[kPer];
#pragma unroll
    for (int r = 0; r < kPer; r++) {
        const unsigned long long q = (unsigned long long)(r * kBktThreads + t) * s.groups + g;
        at[r] = ~0u;
        if (q < probes && src.get(probes == cap ? q : q * cap / probes, k[r], e[r])) at[r] = 0u;
    }
#pragma unroll
    for (int r = 0; r < kPer; r++)
        if (at[r] == 0u) at[r] = atomicAdd(&nv, 1u);
    __syncthreads();
    // four keys for kBktMean entries of this block's share of the table
    const uint32_t v = nv;
    const unsigned long long share = probes ? (unsigned long long)v * cap / probes : 0ull;
    uint32_t keep = share * 4ull / kBktMean >= (unsigned long long)kBktKeep ? (uint32_t)kBktKeep : (uint32_t)(share * 4ull / kBktMean);
    if (keep < 4u) keep = 4u;
    if (keep > v) keep = v;
    __shared__ ulonglong2 key[kBktKeep];
    __shared__ uint32_t tie[kBktKeep];
    // evenly spaced among those found, each block's starting at its own phase:
    // where the slots are rows in order (a vocabulary's source), the blocks' kept
    // places together are spread evenly too (golden-ratio steps: neighbouring
    // blocks read neighbouring slots)
    const uint32_t phase = ((g * 0x9E3779B9u >> 16) * v) >> 16;
#pragma unroll
    for (int r = 0; r < kPer; r++)
        if (at[r] < v) {
            const uint32_t x = at[r] * keep + phase, m = x / v;
            if (x < keep || (x - keep) / v != m) {
                const uint32_t i = m - (phase < keep ? 0u : 1u);
                key[i] = make_ulonglong2(k[r].hi, k[r].lo);
                tie[i] = e[r];
            }
        }
    if (t == 0) s.found[g] = make_uint2(v, keep);
    __syncthreads();
    constexpr uint32_t kLanes = kBktThreads / kBktKeep;  // threads that rank one key
    const uint32_t i = t / kLanes;
    uint32_t r = 0;
    const ulonglong2 x = i < keep ? key[i] : make_ulonglong2(0ull, 0ull);
    const uint32_t xe = i < keep ? tie[i] : 0u;
    if (i < keep)
        for (uint32_t j = t % kLanes; j < keep; j += kLanes) r += row_less(key[j], tie[j], x, xe) ? 1u : 0u;
    for (int o = kLanes / 2; o; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
    if (i < keep && t % kLanes == 0u) {
        s.kept[g * kBktKeep + r] = x;
        s.kept_tie[g * kBktKeep + r] = xe;
    }
}

// ---------------------------------------------------------------- rank
constexpr int kRankThreads = 1024;
constexpr int kListPad = kBktKeep + 1;  // a list a row: 32 lanes at one position of 32 lists hit different banks
// One warp a key: lane l bisects lists l, l + 32, ...  smem: kept_smem(groups)
// bytes; s.rank_blocks blocks.
__device__ __forceinline__ void bucket_rank(const BucketScratch &s, uint8_t *smem, unsigned long long cap) {
    const uint32_t n = s.groups * kBktKeep, t = threadIdx.x, lane = t & 31u;
    ulonglong2 *sk = reinterpret_cast<ulonglong2 *>(smem);
    uint32_t *st = reinterpret_cast<uint32_t *>(sk + s.groups * kListPad), *sn = st + s.groups * kListPad;
    __shared__ uint32_t sum[2];  // keys kept, entries found
    if (t < 2) sum[t] = 0u;
    {   // every load issued before the first store
        constexpr int kPer = kBktGroups * kBktKeep / kRankThreads;
        ulonglong2 k[kPer];
        uint32_t e[kPer];
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const uint32_t i = t + (uint32_t)q * kRankThreads;
            k[q] = i < n ? s.kept[i] : make_ulonglong2(0ull, 0ull);
            e[q] = i < n ? s.kept_tie[i] : 0u;
        }
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const uint32_t i = t + (uint32_t)q * kRankThreads;
            if (i < n) {
                const uint32_t at = i / kBktKeep * kListPad + i % kBktKeep;
                sk[at] = k[q];
                st[at] = e[q];
            }
        }
    }
    __syncthreads();
    if (t < s.groups) {
        const uint2 f = s.found[t];
        sn[t] = f.y;
        atomicAdd(&sum[0], f.y);
        atomicAdd(&sum[1], f.x);
    }
    __syncthreads();
    const uint32_t kept = sum[0];
    // splitters: one for kBktMean entries, at least kBktApart kept keys apart
    const unsigned long long all = (unsigned long long)s.groups * kBktProbes, probes = cap < all ? cap : all;
    const unsigned long long entries = probes ? (unsigned long long)sum[1] * cap / probes : 0ull;
    uint32_t want = (uint32_t)(entries / kBktMean) + 1u, every = kept / want;
    if (every < (uint32_t)kBktApart) every = kBktApart;
    for (uint32_t w = blockIdx.x * (kRankThreads / 32) + t / 32; w < n; w += s.rank_blocks * (kRankThreads / 32)) {
        const uint32_t g = w / kBktKeep, i = w % kBktKeep;
        if (i >= sn[g]) continue;
        const ulonglong2 x = sk[g * kListPad + i];
        const uint32_t xe = st[g * kListPad + i];
        uint32_t r = 0;
        for (uint32_t l = lane; l < s.groups; l += 32) {
            uint32_t lo = 0, hi = sn[l];
            const uint32_t b = l * kListPad;
            while (lo < hi) {
                const uint32_t m = (lo + hi) >> 1;
                if (row_less(sk[b + m], st[b + m], x, xe)) lo = m + 1;
                else hi = m;
            }
            r += lo;
        }
        r = __reduce_add_sync(kFull, r);
        if (lane == 0u && r % every == every - 1u) {
            s.split[r / every] = x;
            s.split_tie[r / every] = xe;
        }
    }
    if (blockIdx.x == 0 && t == 0) {
        s.state[kBktSplits] = kept / every;
        s.state[kBktRoom] = (uint32_t)(s.slots / (kept / every + 1u));
    }
}
inline size_t kept_smem(uint32_t groups) { return (size_t)groups * (kListPad * 20 + 4); }

// ---------------------------------------------------------------- scatter
// The splitters in shared memory, searched by every entry: the high halves down
// a search tree in level order (8 bytes a step; a plain bisection's power-of-two
// strides put a warp's loads in one bank), then the few splitters of an equal high
// half in order (their low halves are read from global memory).
struct Splitters {
    const unsigned long long *tree;  // tree[1 .. 2^levels - 1]
    const unsigned long long *hi;
    const ulonglong2 *split;
    const uint32_t *tie;
    uint32_t n;
    int levels;
    uint32_t room;
    __device__ __forceinline__ bool not_above(uint32_t i, const Key128 &k, uint32_t e) const {
        if (hi[i] != k.hi) return false;
        const unsigned long long lo = split[i].y;
        return lo != k.lo ? lo < k.lo : tie[i] <= e;
    }
    // How many splitters are not above (k, e): the entry's bucket.
    __device__ __forceinline__ uint32_t find(const Key128 &k, uint32_t e) const {
        uint32_t p = 1;
        for (int q = 0; q < levels; q++) p = 2u * p + (tree[p] < k.hi ? 1u : 0u);
        p -= 1u << levels;
        for (int q = 0; q < 4; q++) {
            if (p >= n || !not_above(p, k, e)) return p;
            p++;
        }
        uint32_t end = n;  // many of one high half: the first above
        while (p < end) {
            const uint32_t m = (p + end) >> 1;
            if (not_above(m, k, e)) p = m + 1;
            else end = m;
        }
        return p;
    }
};
constexpr uint32_t kTreeMax = 4096;
static_assert(kBktGroups * kBktKeep / kBktApart < (int)kTreeMax, "the splitters fit the tree");
__device__ __forceinline__ Splitters load_splitters(const BucketScratch &s, uint8_t *smem) {
    const uint32_t n = s.state[kBktSplits];
    const int levels = 32 - __clz((int)n);  // 2^levels > n
    unsigned long long *tree = reinterpret_cast<unsigned long long *>(smem), *h = tree + s.tree;
    for (uint32_t i = threadIdx.x; i + 1u < (1u << levels); i += blockDim.x) {
        unsigned long long k = ~0ull;
        if (i < n) {
            k = s.split[i].x;
            h[i] = k;
        }
        const int up = __ffs((int)(i + 1u));  // its height from the leaves, from 1
        tree[(1u << (levels - up)) + ((i + 1u) >> up)] = k;
    }
    __syncthreads();
    return Splitters{tree, h, s.split, s.split_tie, n, levels, s.state[kBktRoom]};
}
inline size_t splitters_smem(const BucketScratch &s) { return ((size_t)s.tree + s.splits()) * 8; }
constexpr size_t kSplittersMax = ((size_t)kTreeMax + kBktGroups * kBktKeep / kBktApart) * 8;

__device__ __forceinline__ void bucket_store(const BucketScratch &s, uint32_t room, uint32_t b, uint32_t p, const Key128 &k,
                                             uint32_t lref) {
    if (p < room) {
        const unsigned long long at = (unsigned long long)b * room + p;
        s.key[at] = make_ulonglong2(k.hi, k.lo);
        s.lref[at] = lref;
    } else {  // a bucket far larger than the sample promised
        const uint32_t o = atomicAdd(&s.state[kBktSpilled], 1u);
        s.spill_key[o] = make_ulonglong2(k.hi, k.lo);
        s.spill_lref[o] = lref;
        s.spill_bucket[o] = b;
    }
}
__device__ __forceinline__ void bucket_put(const BucketScratch &s, const Splitters &sp, const Key128 &k, uint32_t tie,
                                           uint32_t lref) {
    const uint32_t b = sp.find(k, tie);
    bucket_store(s, sp.room, b, atomicAdd(&s.count[b * kBktStride], 1u), k, lref);
}
// Two entries without long references, their searches and appends overlapped.
__device__ __forceinline__ void bucket_put2(const BucketScratch &s, const Splitters &sp, const Key128 &k0, const Key128 &k1) {
    const uint32_t b0 = sp.find(k0, 0u), b1 = sp.find(k1, 0u);
    const uint32_t p0 = atomicAdd(&s.count[b0 * kBktStride], 1u), p1 = atomicAdd(&s.count[b1 * kBktStride], 1u);
    bucket_store(s, sp.room, b0, p0, k0, 0u);
    bucket_store(s, sp.room, b1, p1, k1, 0u);
}

// A warp's occupied slots queued until 64 are there, two a lane, so that the
// search and the append run with all lanes on (tables are a third full: without
// the queue two lanes of three idled).  Word: 16 key bytes and the count.
// make(key bytes, count) gives the entry's key.
struct SlotQueue {
    static constexpr int kRoom = 96;
    uint4 *key;
    unsigned long long *cnt;
    uint32_t n = 0;  // warp-uniform, below 64 between calls
    template <class Make>
    __device__ __forceinline__ void push(const BucketScratch &s, const Splitters &sp, bool have, const uint4 &k,
                                         unsigned long long c, Make &&make) {
        const uint32_t m = __ballot_sync(kFull, have), lane = threadIdx.x & 31u;
        if (have) {
            const uint32_t i = n + __popc(m & ((1u << lane) - 1u));
            key[i] = k;
            cnt[i] = c;
        }
        n += __popc(m);
        __syncwarp();
        if (n >= 64u) {
            n -= 64u;
            bucket_put2(s, sp, make(key[n + lane], cnt[n + lane]), make(key[n + 32u + lane], cnt[n + 32u + lane]));
            __syncwarp();
        }
    }
    template <class Make>
    __device__ __forceinline__ void flush(const BucketScratch &s, const Splitters &sp, Make &&make) {
        for (uint32_t i = threadIdx.x & 31u; i < n; i += 32u) bucket_put(s, sp, make(key[i], cnt[i]), 0u, 0u);
        n = 0u;
        __syncwarp();
    }
};
__host__ __device__ constexpr size_t slot_queue_smem(int threads) { return (size_t)(threads / 32) * SlotQueue::kRoom * 24; }
__device__ __forceinline__ SlotQueue slot_queue(uint8_t *smem) {
    const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    SlotQueue q;
    q.key = reinterpret_cast<uint4 *>(smem) + warp * SlotQueue::kRoom;
    q.cnt = reinterpret_cast<unsigned long long *>(smem + (size_t)warps * SlotQueue::kRoom * 16) + warp * SlotQueue::kRoom;
    return q;
}

// The last block of a scatter kernel to finish writes each bucket's first row.
__device__ __forceinline__ void bucket_close(const BucketScratch &s) {
    __shared__ uint32_t wsum[32];
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&s.state[kBktTicket], 1u) == gridDim.x - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const uint32_t n = s.state[kBktSplits] + 1u, per = (n + blockDim.x - 1u) / blockDim.x, t = threadIdx.x, lane = t & 31u;
    uint32_t own = 0;
    for (uint32_t i = t * per; i < n && i < (t + 1u) * per; i++) own += __ldcg(&s.count[i * kBktStride]);
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(kFull, incl, o);
        if (lane >= (uint32_t)o) incl += x;
    }
    if (lane == 31u) wsum[t >> 5] = incl;
    __syncthreads();
    uint32_t run = incl - own;
    for (uint32_t w = 0; w < (t >> 5); w++) run += wsum[w];
    for (uint32_t i = t * per; i < n && i < (t + 1u) * per; i++) {
        s.first[i] = run;
        run += __ldcg(&s.count[i * kBktStride]);
    }
}

// ---------------------------------------------------------------- sort
constexpr int kBktSortThreads = 512, kBktSortPerSm = 3;
// Entries a block sorts in shared memory (three blocks an SM).  The one-slot
// test build sorts nearly every bucket in global memory, and spills.
constexpr int kBktFast = kOneSlot ? 64 : 2560;
constexpr int kBktParts = 1024;
constexpr int kBktCoarse = 32;
// The keys between two given ones mapped evenly to `parts` numbers: the 64 bits
// from the first bit in which the two differ, scaled.  Monotone for any keys
// between them.
struct KeyRange {
    unsigned long long w0;
    uint32_t scale;
    uint8_t z, up, high;
    __device__ __forceinline__ unsigned long long window(const ulonglong2 &k) const {
        return high ? (z ? (k.x << z) | (k.y >> (64 - z)) : k.x) : k.y << z;
    }
    __device__ __forceinline__ void set(const ulonglong2 &from, const ulonglong2 &to, uint32_t parts) {
        high = from.x != to.x ? 1 : 0;
        z = (uint8_t)(high ? __clzll((long long)(from.x ^ to.x)) : (from.y != to.y ? __clzll((long long)(from.y ^ to.y)) : 0));
        w0 = window(from);
        const unsigned long long span = window(to) - w0;
        up = (uint8_t)(span ? __clzll((long long)span) : 0);
        const unsigned long long top = (span << up) >> 32;
        // at most parts * 2^32 / (top + 1): the last number is below parts (parts < 2^16)
        scale = span ? (parts << 16) / ((uint32_t)(top >> 16) + 1u) : 0u;
    }
    __device__ __forceinline__ uint32_t operator()(const ulonglong2 &k) const {
        return __umulhi((uint32_t)(((window(k) - w0) << up) >> 32), scale);
    }
};
struct BucketShared {
    ulonglong2 key[kBktFast];
    uint32_t lref[kBktFast];
    uint32_t at[kBktFast];  // part and place of each entry; then the order (uint16_t)
    uint16_t part[kBktFast];
    uint32_t pstart[kBktParts + 1];
    uint32_t wsum[kBktSortThreads / 32];
    ulonglong2 cand[kBktCoarse], coarse[kBktCoarse + 1];  // coarse[c], coarse[c + 1]: around coarse part c
    KeyRange range[kBktCoarse];
};

// Sorts this block's bucket and calls write(base, m, row) once for the block's
// rows [base, base + m), row(i) giving the key and lref of row base + i; for a
// bucket too large for shared memory put(row, key, lref) instead, row by row.
template <class Write, class Put>
__device__ __forceinline__ void bucket_sort(const BucketScratch &s, BucketShared &sh, Write &&write, Put &&put) {
    const uint32_t b = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t nsplit = s.state[kBktSplits], room = s.state[kBktRoom], m = b <= nsplit ? s.count[b * kBktStride] : 0u;
    if (m == 0u) return;
    const unsigned long long base = s.first[b];
    const ulonglong2 *key = s.key + (unsigned long long)b * room;
    const uint32_t *lref = s.lref + (unsigned long long)b * room;
    // words of one prefix and first key may lie on both sides of the next splitter
    const ulonglong2 next = b < nsplit ? s.split[b] : make_ulonglong2(~0ull, ~0ull);
    bool tied = false;
    if (m > (uint32_t)kBktFast || m > room) {
        // more than fits: sorted in global memory, the entries past the
        // bucket's room collected first
        if (t == 0) {
            sh.pstart[0] = atomicAdd(&s.state[kBktBig], m);
            sh.pstart[1] = 0u;
        }
        __syncthreads();
        ulonglong2 *bk = s.big_key + sh.pstart[0];
        uint32_t *br = s.big_lref + sh.pstart[0];
        const uint32_t in = m < room ? m : room, ns = s.state[kBktSpilled];
        for (uint32_t i = t; i < in; i += kBktSortThreads) {
            bk[i] = key[i];
            br[i] = lref[i];
        }
        if (m > room)
            for (uint32_t j = t; j < ns; j += kBktSortThreads) {
                if (s.spill_bucket[j] != b) continue;
                const uint32_t i = in + atomicAdd(&sh.pstart[1], 1u);
                bk[i] = s.spill_key[j];
                br[i] = s.spill_lref[j];
            }
        __syncthreads();
        // bitonic, every merge ascending (its first stage against the mirrored
        // position), so that pairs reaching past m never swap
        for (uint32_t w = 2; (w >> 1) < m; w <<= 1)
            for (uint32_t d = w >> 1; d; d >>= 1) {
                for (uint32_t p = t;; p += kBktSortThreads) {
                    const uint32_t i = 2 * p - (p & (d - 1)), q = d == (w >> 1) ? (i ^ (w - 1)) : i + d;
                    if (i >= m) break;
                    if (q >= m) continue;
                    const ulonglong2 x = bk[i], y = bk[q];
                    const uint32_t rx = br[i], ry = br[q];
                    if (row_less(y, ry, x, rx)) {
                        bk[i] = y;
                        bk[q] = x;
                        br[i] = ry;
                        br[q] = rx;
                    }
                }
                __syncthreads();
            }
        for (uint32_t i = t; i < m; i += kBktSortThreads) {
            const ulonglong2 x = bk[i], y = i + 1 < m ? bk[i + 1] : next;
            if (x.x == y.x && x.y == y.y) tied = true;
            put(base + i, Key128{x.x, x.y}, br[i]);
        }
        if (tied) s.state[kBktTied] = 1u;
        return;
    }
    // Parts of two to four entries: 32 coarse ones between evenly spaced entries
    // of the bucket itself, which follow its distribution, each split evenly by
    // interpolation.  (Interpolation over the whole bucket alone left the
    // buckets of large counts, whose keys are far from even, in a few parts:
    // 127 us for five class tables instead of 40.)
    uint32_t fine = 1;
    while (fine < (uint32_t)(kBktParts / kBktCoarse) && fine * kBktCoarse * 3u < m) fine <<= 1;
    const uint32_t parts = fine * kBktCoarse;
    if (t + 1 < (uint32_t)kBktCoarse) sh.cand[t] = key[(t + 1) * m / kBktCoarse];
    for (uint32_t i = t; i < parts; i += kBktSortThreads) sh.pstart[i] = 0u;
    __syncthreads();
    {   // the coarse splitters in order: sixteen threads rank one
        constexpr uint32_t kLanes = kBktSortThreads / kBktCoarse;
        const uint32_t i = t / kLanes;
        uint32_t r = 0;
        if (i + 1 < (uint32_t)kBktCoarse) {
            const ulonglong2 k = sh.cand[i];
            for (uint32_t j = t % kLanes; j + 1 < (uint32_t)kBktCoarse; j += kLanes) r += row_less(sh.cand[j], j, k, i) ? 1u : 0u;
        }
        for (uint32_t o = kLanes / 2; o; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
        if (t % kLanes == 0u) {
            if (i + 1 < (uint32_t)kBktCoarse) sh.coarse[r + 1] = sh.cand[i];
            else sh.coarse[0] = b ? s.split[b - 1] : make_ulonglong2(0ull, 0ull);
        }
        if (t == 0) sh.coarse[kBktCoarse] = next;
    }
    __syncthreads();
    if (t < (uint32_t)kBktCoarse) sh.range[t].set(sh.coarse[t], sh.coarse[t + 1], fine);
    __syncthreads();
    auto part_of = [&](const ulonglong2 &k) -> uint32_t {
        uint32_t c = 0;
#pragma unroll
        for (uint32_t step = kBktCoarse / 2; step; step >>= 1) {
            const ulonglong2 v = sh.coarse[c + step];
            if (v.x != k.x ? v.x < k.x : v.y <= k.y) c += step;
        }
        return c * fine + sh.range[c](k);
    };
    // every entry's part and place in it
    for (uint32_t i = t; i < m; i += kBktSortThreads) {
        const uint32_t p = part_of(key[i]);
        sh.at[i] = (p << 16) | atomicAdd(&sh.pstart[p], 1u);
    }
    __syncthreads();
    {   // part starts: each thread a run of parts
        constexpr int kPer = kBktParts / kBktSortThreads;
        uint32_t c[kPer], own = 0;
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const uint32_t i = t * kPer + q;
            c[q] = i < parts ? sh.pstart[i] : 0u;
            own += c[q];
        }
        uint32_t incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(kFull, incl, o);
            if (lane >= (uint32_t)o) incl += x;
        }
        if (lane == 31u) sh.wsum[warp] = incl;
        __syncthreads();
        uint32_t run = incl - own;
        for (uint32_t w = 0; w < warp; w++) run += sh.wsum[w];
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            const uint32_t i = t * kPer + q;
            if (i <= parts) sh.pstart[i] = run;
            run += c[q];
        }
        if (t == kBktSortThreads - 1) sh.pstart[kBktParts] = run;
    }
    __syncthreads();
    for (uint32_t i = t; i < m; i += kBktSortThreads) {
        const uint32_t a = sh.at[i], p = a >> 16, j = sh.pstart[p] + (a & 0xFFFFu);
        sh.key[j] = key[i];
        sh.lref[j] = lref[i];
        sh.part[j] = (uint16_t)p;
    }
    __syncthreads();
    // rank within the part by counting
    uint16_t *order = reinterpret_cast<uint16_t *>(sh.at);
    for (uint32_t j = t; j < m; j += kBktSortThreads) {
        const ulonglong2 x = sh.key[j];
        const uint32_t p = sh.part[j], lo = sh.pstart[p], hi = sh.pstart[p + 1];
        uint32_t rank = lo;
#pragma unroll 2
        for (uint32_t i = lo; i < hi; i++) {
            const ulonglong2 o = sh.key[i];
            bool less = o.x < x.x;
            if (o.x == x.x) {
                less = o.y < x.y;
                if (o.y == x.y && i != j) {
                    tied = true;
                    less = sh.lref[i] < sh.lref[j];
                }
            }
            rank += less ? 1u : 0u;
        }
        if (x.x == next.x && x.y == next.y) tied = true;
        order[rank] = (uint16_t)j;
    }
    if (tied) s.state[kBktTied] = 1u;
    __syncthreads();
    write(base, m, [&](uint32_t i, Key128 &kk, uint32_t &rr) {
        const uint32_t j = order[i];
        kk = Key128{sh.key[j].x, sh.key[j].y};
        rr = sh.lref[j];
    });
}

// Orders n entries of one block in shared memory: found[0, n) (entry ids) becomes
// their ids in ascending key order.  Parts of a few entries (32 coarse ones
// between evenly spaced entries, each split evenly by interpolation), then each
// entry's place is its part's first place plus the part's entries before it.
// About 200 instructions an entry; a bitonic network over the list took 500 (200
// entries) to 1,800 (6,000) and a block barrier a stage.  key_of(id): the entry's
// key, with a count below 2^16 complemented in the top 16 bits; before(x, y):
// whether entry x goes before entry y of an equal key.  prow, byparts: n ids of
// room each (byparts also holds 31 keys); coarse: 33, range: 32, pcount: PARTS
// zeros.  Every thread of the block calls it, after a barrier.
template <int BLOCK, uint32_t PARTS, class KeyOf, class Before>
__device__ __forceinline__ uint16_t *order_by_parts(uint32_t n, uint16_t *found, uint16_t *prow, uint16_t *byparts,
                                                    ulonglong2 *coarse, KeyRange *range, uint32_t *pcount,
                                                    KeyOf &&key_of, Before &&before) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t fine = 1;
    while (fine < PARTS / kBktCoarse && fine * kBktCoarse * 3u < n) fine <<= 1;
    {
        ulonglong2 *cand = reinterpret_cast<ulonglong2 *>(byparts);
        constexpr uint32_t kLanes = BLOCK / kBktCoarse;  // threads that rank one candidate
        if (threadIdx.x + 1 < (uint32_t)kBktCoarse && n) cand[threadIdx.x] = key_of(found[(threadIdx.x + 1) * n / kBktCoarse]);
        __syncthreads();
        const uint32_t i = threadIdx.x / kLanes;
        uint32_t r = 0;
        if (i + 1 < (uint32_t)kBktCoarse) {
            const ulonglong2 k = cand[i];
            for (uint32_t j = threadIdx.x % kLanes; j + 1 < (uint32_t)kBktCoarse; j += kLanes)
                r += row_less(cand[j], j, k, i) ? 1u : 0u;
        }
#pragma unroll
        for (uint32_t o = kLanes / 2; o; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
        if (threadIdx.x % kLanes == 0u) {
            if (i + 1 < (uint32_t)kBktCoarse) coarse[r + 1] = cand[i];
            else coarse[0] = make_ulonglong2(0ull, 0ull);
        }
        if (threadIdx.x == 0) coarse[kBktCoarse] = make_ulonglong2((0xFFFFull << 48) - 1ull, ~0ull);  // counts are at least 1
    }
    __syncthreads();
    if (threadIdx.x < (uint32_t)kBktCoarse) range[threadIdx.x].set(coarse[threadIdx.x], coarse[threadIdx.x + 1], fine);
    __syncthreads();
    for (uint32_t e = threadIdx.x; e < n; e += BLOCK) {
        const ulonglong2 k = key_of(found[e]);
        uint32_t c = 0;
#pragma unroll
        for (uint32_t step = kBktCoarse / 2; step; step >>= 1) {
            const ulonglong2 v = coarse[c + step];
            if (v.x != k.x ? v.x < k.x : v.y <= k.y) c += step;
        }
        const uint32_t q = c * fine + range[c](k);
        prow[e] = (uint16_t)q;
        atomicAdd(&pcount[q], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // counts -> first rows
        constexpr int kPer = PARTS / 32;
        uint32_t c[kPer], own = 0;
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            c[q] = pcount[lane * kPer + q];
            own += c[q];
        }
        uint32_t incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(kFull, incl, o);
            if (lane >= (uint32_t)o) incl += x;
        }
        uint32_t run = incl - own;
#pragma unroll
        for (int q = 0; q < kPer; q++) {
            pcount[lane * kPer + q] = run;
            run += c[q];
        }
    }
    __syncthreads();
    for (uint32_t e = threadIdx.x; e < n; e += BLOCK) byparts[atomicAdd(&pcount[prow[e]], 1u)] = found[e];
    __syncthreads();
    // pcount[q] is now the first row after part q.  Thread and place agree (not
    // thread and entry), so that a warp's lanes rank within the same few parts
    // and a long part holds up only the warps that own it.
    for (uint32_t j = threadIdx.x; j < n; j += BLOCK) {
        uint32_t q = 0;
#pragma unroll
        for (uint32_t step = PARTS / 2; step; step >>= 1)
            if (pcount[q + step - 1] <= j) q += step;
        const uint32_t lo = q ? pcount[q - 1] : 0u, hi = pcount[q], mine = byparts[j];
        const ulonglong2 k = key_of(mine);
        uint32_t rank = lo;
        for (uint32_t i = lo; i < hi; i++) {
            const ulonglong2 o = key_of(byparts[i]);
            rank += (o.x != k.x ? o.x < k.x : (o.y != k.y ? o.y < k.y : i != j && before(byparts[i], mine))) ? 1u : 0u;
        }
        found[rank] = (uint16_t)mine;  // (the entries as found are not read any more)
    }
    __syncthreads();
    return found;
}

}  // namespace wc
