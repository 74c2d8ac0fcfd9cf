// Host-side declarations shared by the library's translation units.
#pragma once
#include <cstdint>
#include <utility>
#include <cuda_runtime.h>

#include "wc_device.cuh"

namespace wc {

// Raises kernel `func`'s dynamic shared-memory limit to `bytes` on the
// calling thread's current device.  The attribute belongs to that device's
// context, so it is set once per (kernel, device, size): a process that
// counts on several devices sets it on each.  Safe to call from several host
// threads at once.
cudaError_t ensure_smem_limit(const void *func, int bytes);

// ---------------------------------------------------------------- counting
struct CountLaunch {
    const uint8_t *text;     // document bytes are text[lo, hi); long words may
                             // match representatives anywhere in text[0, hi)
    uint64_t lo, hi;
    GTable g;
    int grid;                // 0 = one persistent block per SM
    void *head_scratch;      // head_scratch_bytes() or null (no shared-memory head)
    cudaEvent_t main_ev[2];  // recorded (when non-null) right before the main counting kernel
    int head_mode;           // 0: build a head for texts >= count_global_head_min(); 1: reuse the
                             // head an earlier launch built in head_scratch; 2: no head; 3: build one
    int no_level1;           // 1: no shared-memory level-1 table at all (measurement)
};
// Tokenises and counts text[lo, hi) into g (8-byte, 16-byte and long tables).
cudaError_t launch_count_global(const CountLaunch &c, cudaStream_t s);
uint64_t count_global_head_min();
// Head scratch (also where long words wait) pays for itself in texts from here on.
uint64_t count_global_scratch_min();
// One block runs the counting kernel's bounded barrier wait (see wc_selftest_wait).
cudaError_t launch_wait_selftest(uint32_t *d_status, uint32_t polls, int arrive, cudaStream_t s);
// Kernel launches of one launch_count_global: head selection when it builds a
// head, the counting kernel, and the deferred long-word
// inserts when head scratch is given (`scratch`).
int count_global_launches(uint64_t nbytes, bool builds_head, bool scratch);
size_t head_scratch_bytes();

// Texts of at most kSmallCountMax bytes: the whole table by one block, no scratch
// (wc_small.cu).  small_count_caps: sizes of `out` that always suffice.
constexpr uint64_t kSmallCountMax = 16384;
void small_count_caps(uint64_t nbytes, uint64_t *cap, uint64_t *lcap, uint64_t *arena);

// ---------------------------------------------------------------- dependent launches
// A kernel launched with launch_dependent may have its blocks scheduled
// before the previous kernel in the stream has finished; it must call
// grid_dependency_wait() before touching anything that kernel (or earlier
// work) reads or writes.  grid_dependency_trigger() lets the next dependent
// launch start once every block of the calling kernel has called it.  Both
// are no-ops for ordinary launches.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                             Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// ---------------------------------------------------------------- numeric MapReduce
// Blocks of the series sum for n terms, and its two launches (exact per-block
// sums into part[nb], then their sum rounded once).
int series_blocks(unsigned long long n);
cudaError_t launch_series(int series, unsigned long long n, ulonglong2 *part, int nb, double *d_out, cudaStream_t s);

// Row sums of a row-major uint32 matrix (the hybrid pipeline's reduce).
cudaError_t launch_row_sums(const uint32_t *m, unsigned long long rows, unsigned long long cols,
                            unsigned long long *out, cudaStream_t s);

// ---------------------------------------------------------------- tables
// A compacted, sorted table in device memory.  Entry i: big-endian key
// halves (first 16 letters), count, and lref (0 = word fits the key, else
// 1 + index into loff/llen of a long word whose bytes are in arena).
struct DevTable {
    uint64_t cap;            // entry capacity of the arrays below
    uint64_t lcap;           // long-word entry capacity
    uint64_t arena_cap;
    int count_bits;          // 32 or 64
    unsigned long long *d_meta;   // [0] n entries, [1] n long, [2] arena bytes used, [3] tokens
    uint32_t *d_status;
    unsigned long long *khi, *klo;
    void *cnt;               // uint32_t or unsigned long long [cap]
    uint32_t *lref;
    unsigned long long *loff, *llen;
    uint8_t *arena;
};

// Counts d_text[0, nbytes) into `out` (metadata and status written too); nbytes
// in 1 .. kSmallCountMax.
cudaError_t launch_count_small(const uint8_t *d_text, uint64_t nbytes, DevTable &out, cudaStream_t s);

// Scratch for compaction + sort of up to `cap` entries.
// Radix passes of the entry sort: 10 byte digits of the packed 16-letter
// prefix (5 bits a letter, 80 bits), 8 digits of the complemented count, and
// 4 document digits when a batch is sorted per document.
constexpr int kSortKeyPasses = 10;
constexpr int kSortPasses = kSortKeyPasses + 8;
constexpr int kSortPassesSeg = kSortPasses + 4;

// A radix pass sorts tiles of kSortTileElems entries.  A small sort (at most
// kSortFusedMaxTiles tiles by capacity) needs no scan pass: each tile finds
// its digit offsets from the counts of the tile groups before its own group
// and of the tiles before it in its group, in groups of sort_group_tiles(t)
// tiles for t tiles (a power of two of at least sqrt(t)), so at most
// sort_group_stride(capacity tiles) groups.  Larger sorts scan the tile
// counts in a pass of their own.
constexpr uint64_t kSortTileElems = 4096;
constexpr uint64_t kSortFusedMaxTiles = 1024;
__host__ __device__ constexpr uint64_t sort_group_tiles(uint64_t ntiles) {
    uint64_t g = 1;
    while (g * g < ntiles) g <<= 1;
    return g;
}
constexpr uint64_t sort_group_stride(uint64_t ntiles_cap) {
    uint64_t r = 1;
    while (r * r < ntiles_cap) r++;
    return r + 1;
}

struct SortScratch {
    uint64_t cap;
    unsigned long long *khi, *klo, *cnt;
    unsigned long long *pk;  // packed prefix, low 64 bits (written by the sort)
    uint32_t *pk2;           // packed prefix, high 16 bits
    uint32_t *lref;
    uint32_t *perm[2];
    uint32_t *doc;           // document of each entry (segmented sorts)
    uint32_t *hist_all;      // 24 x 256
    uint32_t *tile_hist;     // 256 x ntiles
    uint32_t *cur;           // 25
    uint32_t *group_hist[2]; // 256 x group_stride each: digit counts per tile group, by pass parity
    uint32_t group_stride;
    uint32_t *look[2];       // 256 x ntiles each: per-tile digit counts published for the look-back, by pass parity
    uint32_t *tile_ctr;      // [2]: tiles taken in launch order, by pass parity
    // permutation buffer c (0 or 1), selected without indexing the parameter array
    __device__ __forceinline__ uint32_t *perm_buf(uint32_t c) const { return c ? perm[1] : perm[0]; }
    __device__ __forceinline__ uint32_t *group_buf(uint32_t c) const { return c ? group_hist[1] : group_hist[0]; }
    __device__ __forceinline__ uint32_t *look_buf(uint32_t c) const { return c ? look[1] : look[0]; }
};
// Slot of SortScratch::cur where a radix pass records a look-back that gave
// up waiting (the finish then reports WC_ERR_TIMEOUT).
constexpr int kCurSortError = 30;
size_t sort_scratch_bytes(uint64_t cap);
void sort_scratch_carve(SortScratch &s, void *base, uint64_t cap);
// Zeroes what a sort accumulates into (digit histograms, pass cursors, group
// counts, the first pass's look-back buffer and the tile counters): every
// sort of a scratch starts with this (stream-ordered memsets).
void sort_state_reset(SortScratch &ss, cudaStream_t st);

// Word bytes of table entries for ordering long words that share a prefix.
struct LongView {
    const uint32_t *lref;
    const unsigned long long *loff, *llen;
    const uint8_t *arena;
};
// Slot of SortScratch::cur naming the permutation buffer that holds a
// finished sort's order.
constexpr int kCurFinal = 31;
// Radix passes the host knows to be constant, not launched at all: the count
// digits above the bytes of `max_count` (a bound on every count) and the
// document digits above those of `ndocs - 1` (bit p: pass p skipped).
uint32_t sort_skip_mask(uint64_t max_count, uint64_t ndocs);
// Stable LSD radix sort of ss's n = meta[0] entries by (count desc, word asc);
// with passes == kSortPassesSeg the document is the most significant key.
// The result is the permutation ss.perm_buf(ss.cur[kCurFinal]) (device value).
cudaError_t sort_entries(SortScratch &ss, const unsigned long long *meta, const LongView &v, int passes,
                         cudaStream_t st, uint32_t skip = 0);
int sort_entries_launches(int passes, uint64_t cap, uint32_t skip = 0);

// Scratch of the bucket sort (wc_bucket.cuh) of up to `cap` entries: about 84
// bytes an entry.
constexpr int kBktGroups = 128;  // sample blocks at most
constexpr int kBktKeep = 64;     // sampled keys a sample block keeps at most
constexpr int kBktApart = 3;     // sampled keys between two splitters at least
constexpr int kBktMean = 384;    // entries a bucket is meant to hold
constexpr int kBktStride = 8;    // words between two buckets' counters
constexpr int kBktSplits = 0, kBktRoom = 1, kBktSpilled = 2, kBktTied = 3, kBktBig = 4, kBktTicket = 5;  // BucketScratch::state
// Tables of more slots are radix sorted.  There are at most 2,730 splitters (54 KB
// of shared memory in the scatter kernels); past 1,500 entries a bucket more and
// more buckets hold over 2,560 and are sorted in global memory, while the radix
// passes' cost an entry stays the same.  Finish of N words, ms, bucket | radix:
// 1 M 0.13 | 0.20-0.25; 2 M (8.5 M slots) 0.31-0.33 | 0.34-0.41; 4 M (16.8 M
// slots) 0.74-0.79 | 0.67-0.80; 8 M 2.3-2.4 | 1.4-1.7; 12 M (2 x 2^24 slots) 4.0-4.3 |
// 2.2-2.5.
//   Batches: the (document, word) tables have several times the slots of their rows
// where documents are large, and class and global tables are sized for a quarter of
// the documents' rows, so the rows to expect decide, up to the slots that the
// scratch is meant for.  Plans, ms: documents of 94 KB of a 500,000-word vocabulary,
// 2.5 M rows (1.8 M expected) 0.77 | 1.00, 5 M (3.6 M) 2.13 | 1.98, 10 M (7.2 M)
// 5.1-5.4 | 4.12; log-normal documents, 20,000 (1.5 M expected) 1.37 | 1.62, 60,000
// (5.0 M) 3.95 | 4.21.
constexpr uint64_t kBktMaxCap = 10ull << 20;
constexpr uint64_t kBktMaxRows = 5000000, kBktMaxSparse = 1ull << 26;
struct BucketScratch {
    uint32_t groups;              // sample blocks
    unsigned long long slots;     // entries `key` and `lref` hold, shared out evenly to the buckets
    ulonglong2 *kept, *split;     // sampled keys, splitters in order (high and low halves)
    uint32_t *kept_tie, *split_tie;
    uint2 *found;                 // per sample block: entries found, keys kept
    uint32_t rank_blocks;         // blocks of the rank kernel
    uint32_t tree;                // words of the scatter kernels' search tree: a power of two above splits()
    uint32_t *count;              // entries a bucket got, kBktStride words apart
    uint32_t *first;              // a bucket's first row
    uint32_t *state;
    ulonglong2 *key;              // null: no bucket scratch
    uint32_t *lref;
    ulonglong2 *spill_key;        // entries past their bucket's room
    uint32_t *spill_lref, *spill_bucket;
    ulonglong2 *big_key;          // buckets too large for shared memory are sorted here
    uint32_t *big_lref;
    __host__ __device__ __forceinline__ uint32_t splits() const { return groups * kBktKeep / kBktApart; }
    __host__ __device__ __forceinline__ uint32_t buckets() const { return splits() + 1; }
};
size_t bucket_scratch_bytes(uint64_t cap);
void bucket_scratch_carve(BucketScratch &s, void *base, uint64_t cap);

// Turns the global hash tables into the sorted table `out` (long words copied
// into out.arena): by the bucket sort when `bs` is carved and `skip` shows every
// count below 2^48 (the count's two high digits skipped), else compaction
// into `ss` and the radix sort.  finish_table_launches(...) kernels are launched.
bool finish_by_buckets(const BucketScratch &bs, uint32_t skip);
int finish_table_launches(const SortScratch &ss, const BucketScratch &bs, uint32_t skip = 0);
cudaError_t finish_table(const GTable &g, uint64_t gcap8, uint64_t gcap, uint64_t glcap, SortScratch &ss,
                         const BucketScratch &bs, DevTable &out, cudaStream_t s, uint32_t skip = 0);

// Compaction scans read kScanUnroll slots a thread per step (independent
// loads in flight) and reserve output positions with one atomic per block
// and step: block_take returns the first of `mine` positions reserved for
// the calling thread and adds the block's `tok` to *tokens and its count of
// positions to *kind (either may be null).
// Every thread of the block must call it (the loops step block-uniformly).
constexpr int kScanUnroll = 4;
struct BlockTake {
    uint32_t wsum[32];
    unsigned long long tok[32];
    unsigned long long base;
};
__device__ __forceinline__ unsigned long long block_take(BlockTake &sh, uint32_t mine, unsigned long long tok,
                                                         unsigned long long *counter, unsigned long long *tokens,
                                                         unsigned long long *kind = nullptr) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    uint32_t incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += t;
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) tok += __shfl_xor_sync(0xFFFFFFFFu, tok, d);
    if (lane == 31) sh.wsum[warp] = incl;
    if (lane == 0) sh.tok[warp] = tok;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        unsigned long long tt = 0;
        for (int w = 0; w < nw; w++) {
            const uint32_t v = sh.wsum[w];
            sh.wsum[w] = run;
            run += v;
            tt += sh.tok[w];
        }
        sh.base = run ? atomicAdd(counter, (unsigned long long)run) : 0ull;
        if (tokens && tt) atomicAdd(tokens, tt);
        if (kind && run) atomicAdd(kind, (unsigned long long)run);
    }
    __syncthreads();
    const unsigned long long pos = sh.base + sh.wsum[warp] + incl - mine;
    __syncthreads();
    return pos;
}

// One radix sort's arguments.
struct SortJob {
    SortScratch s;
    const unsigned long long *meta;
    LongView v;
    DevTable out;
};
// finish_table for n tables at once: every step of those with bucket scratch as
// one launch over them all (grid.y), the others one by one.  d_jobs: device
// memory of finish_tables_job_bytes(n), alive until the stream has run the
// launches.
struct FinishSpec {
    GTable g;
    uint64_t gcap8, gcap, glcap;
    SortScratch *ss;
    BucketScratch *bs;
    DevTable *out;
};
size_t finish_tables_job_bytes(int n);
int finish_tables_launches(const FinishSpec *spec, int n, uint32_t skip = 0);
cudaError_t finish_tables(const FinishSpec *spec, int n, void *d_jobs, cudaStream_t s, uint32_t skip = 0);

// Entries of finished tables re-inserted into a global hash table (merge).
struct MergeSrc {
    const unsigned long long *meta;
    const unsigned long long *khi, *klo;
    const void *cnt;
    const uint32_t *lref;
    const unsigned long long *loff, *llen;
    const uint8_t *arena;
    int count_bits;
    uint64_t cap;
    uint64_t arena_cap;
};
cudaError_t launch_merge_insert(const MergeSrc *d_src, const uint64_t *h_chunk_start, uint32_t nsrc,
                                uint64_t total_chunks, const GTable &g, cudaStream_t s);
constexpr int kMergeChunk = 256;  // rows a merge block inserts, one a thread

cudaError_t launch_topk_copy(const DevTable &in, uint64_t k, DevTable &out, cudaStream_t s);

// Export of a table's n rows of word_bytes letters: word lengths -> offsets -> bytes, on the device.
size_t export_scratch_bytes(uint64_t n);
cudaError_t launch_export(const DevTable &t, uint64_t n, uint64_t word_bytes, void *scratch, uint8_t *d_words,
                          unsigned long long *d_offs, cudaStream_t s);

}  // namespace wc
