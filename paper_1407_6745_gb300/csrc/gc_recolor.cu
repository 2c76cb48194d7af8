// gc_recolor.cu -- iterative recoloring on one GPU.
//
// Culberson's iterated greedy (Sec. 2.1) as synchronous recoloring RC
// (Sec. 3): the classes of the previous coloring are taken one after the
// other in a class permutation (RV, NI, ND or RAND, Sec. 3) and every vertex
// takes the smallest color not used by a neighbor of an earlier class.  A
// class is an independent set, so all its vertices can choose at once and
// the result equals the sequential greedy run in class order (Sec. 3).
//
// One iteration = three launches, with no host round trip:
//   k_rc_hist     histogram of (class, degree bucket) pairs (first iteration
//                 only; later ones get it from the previous recoloring);
//   k_rc_order    the class permutation, computed on the device (one block):
//                 present classes, RV/NI/ND order or a Fisher-Yates shuffle,
//                 rank of every color, segment starts and tile counts;
//   k_rc_scatter  counting sort of the vertices into class-major,
//                 bucket-minor segments; new[v] = -(rank(v) + 1);
//   k_rc_recolor  the class steps, as one cooperative launch: warp tiles are
//                 dealt out statically in class order; a neighbor u of an
//                 earlier class whose new color is not yet written (still
//                 negative) is waited for, with a bounded spin; a neighbor of
//                 a later class (negative, rank above v's) is ignored.  The
//                 alternative form launches one grid per class and needs no
//                 waits.
// The negative encoding makes one 4-byte gather per edge serve both "is u
// earlier than v" and "what color did u take".  Rows longer than
// rc_warp_max_deg are cut into chunks of 256 neighbors handled by different
// warps; the chunks OR their forbidden colors into a per-row bitmap and the
// warp that finishes the last chunk waits for the row's nearest classes and
// picks the color.
#include <algorithm>
#include <cstring>
#include <vector>

#include "gc_internal.h"

namespace gc {

constexpr int32_t kMaxInputColor = 1 << 28;
constexpr int kOrderThreads = 1024;
constexpr int kShuffleSmem = 4096;
constexpr int32_t kChunk = 256;   // neighbors per chunk of a split (heavy) row (measured best on R-MAT)

// A chunk of a split row leaves its in-flight neighbors of the kNearClasses
// classes before its own to the row's last chunk, through a list of kRowPend
// entries a row (see defer_near; both measured there).
constexpr int32_t kNearClasses = 2;
constexpr int32_t kRowPend = 256;
static_assert(kRowPend == 256, "8 entries per lane of the warp that takes them");

// An isolated vertex (no neighbor) takes color 1 in every iteration and no
// vertex waits on it: it gets bucket kIsoBucket, no list entry and no tile;
// the scatter writes its color and it is counted in iso_cnt (class sizes
// only).  (R-MAT 24: 47 % of the vertices; the recoloring kernel went from
// 5.07 to 4.91 ms per iteration.)
constexpr int kIsoBucket = 8;

// The recoloring phase's buckets: 0 split rows, 1 a warp per row (bucket_of's 1
// and 2, which the row's length tells apart: see kBitsDeg), 2..5 groups of
// 16/8/4/2 lanes, and 6: rows of up to
// kOneLaneDeg entries, a lane each (its gathers are one batch), where the
// 2-lane threshold allows it.  Such rows are most of a skewed graph's and all
// of a 7-point mesh's; with 2 lanes a warp tile held 16 of them (recoloring
// launch, 2 lanes -> 1: 7-point mesh of 1 M vertices 53 -> 40 us, a batch of
// 512 graphs 0.74 -> 0.66 ms, RMAT-Bad 22 0.56 -> 0.53, R-MAT 24 within 3 %).
// No more than 7: the (class, bucket) tables of the largest input color are
// then within 32-bit indices (an eighth bucket's were not).
constexpr int kRcNB = 7;
constexpr int32_t kOneLaneDeg = 8;
constexpr int32_t kBitsDeg = 63;  // rows of up to this many entries: their color is among the first 64
static_assert((static_cast<int64_t>(kMaxInputColor) + 1) * kRcNB <= INT32_MAX, "32-bit (class, bucket) indices");
// Entries of the (class, bucket) tables for the colors [1, cap] (0: beyond 32-bit indices).
inline int64_t class_entries(int32_t cap) {
    const int64_t ent = (static_cast<int64_t>(cap) + 1) * kRcNB;
    return ent <= INT32_MAX ? ent : 0;
}
__device__ __forceinline__ int rc_bucket_of(int32_t deg, const Tuning& t) {
    if (deg == 0) return kIsoBucket;
    if (deg <= min(kOneLaneDeg, t.g2_max_deg)) return 6;
    const int b = bucket_of(deg, 1, t);
    return b < 2 ? b : b - 1;
}

// Lanes per row (log2) of a bucket's warp tiles, and rows (bucket 0: row
// chunks) per tile.
__host__ __device__ constexpr int lanes_log2(int b) { return b < 2 ? 5 : 6 - b; }
__host__ __device__ constexpr int warp_tile(int b) { return 32 >> lanes_log2(b); }

struct RcCtrl {
    int32_t k;            // present classes this iteration
    int32_t total_tiles;  // warp tiles this iteration
    int32_t hub_next;     // next free split-row slot
    int32_t max_in;       // max input color (validation)
    int32_t n_heavy;      // rows in bucket 0 (split into chunks)
    uint32_t err;
    int32_t hot_sg;       // the largest segment of single-entry vertices (scatter)
    uint32_t over;        // a vertex took a color above cap (only where the CSR is not symmetric)
    unsigned long long edges;
};

struct RcArgs {
    Graph g;
    Tuning tune;
    uint64_t seed;
    int32_t perm;
    int32_t iteration;
    int32_t cap;          // colors are in [1, cap]
    const int32_t* old_c;
    int32_t* new_c;
    uint8_t* bucket;
    int32_t* cls_cnt;     // (cap + 1) * kRcNB vertices per (class, bucket)
    int32_t* cls_units;   // cap + 1: row chunks of the bucket-0 vertices per class
    int32_t* nxt_cnt;     // the same two histograms of the new colors, filled by
    int32_t* nxt_units;   //   the recoloring kernel for the next iteration
    int32_t* iso_cnt;     // cap + 1 (batch: per (graph, color)): isolated vertices per class
    int32_t* nxt_iso;     // the same of the new colors, filled by the scatter (one graph)
    int32_t* present;     // cap + 1
    int32_t* psize;       // cap + 1
    int32_t* order;       // cap + 1 (class order, colors)
    int32_t* jtab;        // cap + 1 (shuffle indices)
    int32_t* rank_of;     // cap + 1
    int32_t* seg_start;   // (cap + 1) * kRcNB + 1, in list entries
    int32_t* tile_prefix; // (cap + 1) * kRcNB + 1, in warp tiles
    int32_t* fill;        // (cap + 1) * kRcNB
    WorkItem* list;       // list entries in class-major order
    int32_t* ncolors;     // iterations + 1
    int32_t* hub_v;       // split rows: vertex, chunk count, finished chunks,
    int32_t* hub_nch;     //   and a forbidden-color bitmap of hub_words words
    int32_t* hub_done;
    uint32_t* hub_bm;
    int32_t hub_words;
    int32_t* hub_pcnt;    // neighbors left to the row's last chunk: count, kRowPend entries
    int32_t* hub_pend;
    RcCtrl* ctrl;
    // batches (nullptr for one graph): graph of every vertex, descriptors,
    // and the start of each graph's colors in the (graph, color) tables
    // cls_cnt / cls_units / rank_of / g*
    const int32_t* graph_of;
    const BatchDesc* desc;
    const int64_t* cls_base;
    int32_t ngraphs;
    int32_t fuse_hist;    // 1: the recoloring kernel fills nxt_cnt (one graph only)
    int32_t scatter_segs; // segments the scatter counts in shared memory
    int32_t hist_smem;    // entries of its dynamic shared-memory histogram (0: global)
    int32_t* gpresent;    // per (graph, color): present colors, sizes, order, shuffle
    int32_t* gpsize;
    int32_t* gorder;
    int32_t* gjtab;
    int32_t* seg_cnt;     // list entries per global segment (rank, bucket)
};

__device__ __forceinline__ int32_t ld_relaxed(const int32_t* p) {
    int32_t x;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(x) : "l"(p));
    return x;
}
__device__ __forceinline__ void st_relaxed(int32_t* p, int32_t x) {
    asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}

__device__ __forceinline__ int32_t chunks_of(int32_t deg) { return (deg + kChunk - 1) / kChunk; }

// ---------------------------------------------------------------------------
// Per-call set-up: degree buckets (X = 1).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock) k_rc_bucket(RcArgs a) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kBlock;
    int32_t heavy = 0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x; i < a.g.n; i += stride) {
        int64_t beg;
        int32_t deg;
        row_of(a.g, static_cast<int32_t>(i), beg, deg, &a.ctrl->err);
        const int b = rc_bucket_of(deg, a.tune);
        a.bucket[i] = static_cast<uint8_t>(b);
        heavy += b == 0;
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) heavy += __shfl_xor_sync(kFull, heavy, d);
    if (lane_id() == 0 && heavy) atomicAdd(&a.ctrl->n_heavy, heavy);
}

// Max color of a coloring known to be proper (colors outside [1, max input
// color] still flag it improper).
__global__ void __launch_bounds__(kBlock) k_rc_maxin(RcArgs a) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kBlock;
    int32_t my_max = 0;
    for (int64_t v = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x; v < a.g.n; v += stride) {
        const int32_t cv = a.old_c[v];
        if (cv < 1 || cv > kMaxInputColor) atomicOr(&a.ctrl->err, kErrImproper);
        else my_max = max(my_max, cv);
    }
    warp_max(&a.ctrl->max_in, my_max);
}

// ---------------------------------------------------------------------------
// Histogram of (class, bucket); bucket-0 rows also count their chunks
// ---------------------------------------------------------------------------
constexpr int kHistSmem = 8192;

constexpr int kIsoSmem = 1024;  // isolated vertices per class, colors below this counted in shared memory

// kBucket: it also sets the buckets (k_rc_bucket's part, where nothing has to
// be known of them before).
template <bool kBucket>
__global__ void __launch_bounds__(kBlock) k_rc_hist(RcArgs a) {
    __shared__ int32_t sh[kHistSmem];
    __shared__ int32_t s_iso[kIsoSmem];
    const int32_t entries = (a.cap + 1) * kRcNB;
    const bool local = entries <= kHistSmem;
    for (int i = threadIdx.x; i < kIsoSmem; i += kBlock) s_iso[i] = 0;
    if (local)
        for (int i = threadIdx.x; i < entries; i += kBlock) sh[i] = 0;
    __syncthreads();
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kBlock;
    for (int64_t v = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x; v < a.g.n; v += stride) {
        const int32_t c = a.old_c[v];
        int b;
        if (kBucket) {
            int64_t beg;
            int32_t deg;
            row_of(a.g, static_cast<int32_t>(v), beg, deg, &a.ctrl->err);
            b = rc_bucket_of(deg, a.tune);
            a.bucket[v] = static_cast<uint8_t>(b);
            if (b == 0 && !a.ctrl->n_heavy) atomicOr(&a.ctrl->n_heavy, 1);  // (only whether there are any is asked)
        } else {
            b = a.bucket[v];
        }
        if (c < 1 || c > a.cap) {
            atomicOr(&a.ctrl->err, kErrImproper);
            continue;
        }
        if (b == kIsoBucket) {
            if (c < kIsoSmem) atomicAdd(&s_iso[c], 1);
            else atomicAdd(&a.iso_cnt[c], 1);
            continue;
        }
        const int32_t key = c * kRcNB + b;
        const unsigned act = __activemask();
        const unsigned peers = __match_any_sync(act, key);
        if (lane_id() == __ffs(peers) - 1) {
            if (local) atomicAdd(&sh[key], __popc(peers));
            else atomicAdd(&a.cls_cnt[key], __popc(peers));
        }
        if (b == 0) {
            int64_t beg;
            int32_t deg;
            row_of(a.g, static_cast<int32_t>(v), beg, deg, &a.ctrl->err);
            atomicAdd(&a.cls_units[c], chunks_of(deg));
        }
    }
    __syncthreads();
    if (local)
        for (int i = threadIdx.x; i < entries; i += kBlock)
            if (sh[i]) atomicAdd(&a.cls_cnt[i], sh[i]);
    for (int i = threadIdx.x; i < kIsoSmem && i <= a.cap; i += kBlock)
        if (s_iso[i]) atomicAdd(&a.iso_cnt[i], s_iso[i]);
}

// ---------------------------------------------------------------------------
// Class order (one block of 1024 threads)
// ---------------------------------------------------------------------------
struct OrderShared {
    int32_t wsum[kOrderThreads / 32];
    int32_t carry;
    unsigned long long best[kOrderThreads / 32];
    int32_t shuffle[kShuffleSmem];
};

// Exclusive scan over the block; returns the prefix, writes the total.
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t x, OrderShared& s, int32_t& total) {
    const int l = lane_id(), w = threadIdx.x >> 5;
    const int32_t incl = static_cast<int32_t>(warp_inclusive_scan(static_cast<uint32_t>(x)));
    if (l == 31) s.wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int32_t y = s.wsum[l];
        const int32_t yi = static_cast<int32_t>(warp_inclusive_scan(static_cast<uint32_t>(y)));
        s.wsum[l] = yi - y;
        if (l == 31) s.carry = yi;
    }
    __syncthreads();
    const int32_t r = s.wsum[w] + incl - x;
    total = s.carry;
    __syncthreads();
    return r;
}

// Segment starts (list entries) and tile prefix (warp tiles) of the k
// ranks x kRcNB buckets, class-major; units(sg) gives a segment's entries.
template <class Units>
__device__ __forceinline__ void build_segments(const RcArgs& a, int32_t k, OrderShared& s, Units&& units) {
    const int t = threadIdx.x;
    const int32_t nseg = k * kRcNB;
    int32_t vbase = 0, tbase = 0;
    unsigned long long best = 0;  // (entries << 32) | segment, over the single-entry buckets
    for (int32_t s0 = 0; s0 < nseg; s0 += kOrderThreads) {
        const int32_t sg = s0 + t;
        int32_t cnt = 0, tiles = 0;
        if (sg < nseg) {
            const int b = sg % kRcNB;
            cnt = units(sg);
            tiles = (cnt + warp_tile(b) - 1) / warp_tile(b);
            a.fill[sg] = 0;
            if (b != 0) {
                const unsigned long long key = (static_cast<unsigned long long>(cnt) << 32) | static_cast<uint32_t>(sg);
                best = key > best ? key : best;
            }
        }
        int32_t vt, tt;
        const int32_t vp = block_exclusive_scan(cnt, s, vt);
        const int32_t tp = block_exclusive_scan(tiles, s, tt);
        if (sg < nseg) {
            a.seg_start[sg] = vbase + vp;
            a.tile_prefix[sg] = tbase + tp;
        }
        vbase += vt;
        tbase += tt;
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(kFull, best, d);
        best = o > best ? o : best;
    }
    if (lane_id() == 0) s.best[t >> 5] = best;
    __syncthreads();
    if (t == 0) {
        for (int w = 0; w < kOrderThreads / 32; ++w) best = s.best[w] > best ? s.best[w] : best;
        a.seg_start[nseg] = vbase;
        a.tile_prefix[nseg] = tbase;
        a.ctrl->k = k;
        a.ctrl->total_tiles = tbase;
        a.ctrl->hub_next = 0;
        a.ctrl->hot_sg = (best >> 32) ? static_cast<int32_t>(best & 0xffffffffu) : -1;
    }
}

__global__ void __launch_bounds__(kOrderThreads) k_rc_order(RcArgs a) {
    __shared__ OrderShared s;
    const int t = threadIdx.x;
    const uint32_t over = t == 0 ? __ldcg(&a.ctrl->over) : 0u;  // (used last: its latency is in no one's way)
    // present classes in ascending color, with their sizes
    int32_t k = 0;
    for (int32_t c0 = 1; c0 <= a.cap; c0 += kOrderThreads) {
        const int32_t c = c0 + t;
        int32_t size = 0;
        if (c <= a.cap) {
            for (int b = 0; b < kRcNB; ++b) size += a.cls_cnt[c * kRcNB + b];
            size += a.iso_cnt[c];
        }
        int32_t total;
        const int32_t pos = block_exclusive_scan(size > 0 ? 1 : 0, s, total);
        if (size > 0) {
            a.present[k + pos] = c;
            a.psize[k + pos] = size;
        }
        k += total;
    }
    __syncthreads();
    if (a.ncolors && a.iteration == 0 && t == 0) a.ncolors[0] = k > 0 ? a.present[k - 1] : 0;

    // the permutation (Sec. 3) of this iteration (Sec. 4.2.1 schedules)
    const int32_t perm = perm_at(a.perm, a.iteration);
    if (perm == 0) {  // RV
        for (int32_t i = t; i < k; i += kOrderThreads) a.order[i] = a.present[k - 1 - i];
    } else if (perm == 1 || perm == 2) {  // NI / ND, ties to the smaller color
        const bool noninc = perm == 1;
        for (int32_t i = t; i < k; i += kOrderThreads) {
            const int32_t si = a.psize[i];
            int32_t r = 0;
            for (int32_t j = 0; j < k; ++j) {
                const int32_t sj = a.psize[j];
                const bool before = noninc ? (sj > si || (sj == si && j < i))
                                           : (sj < si || (sj == si && j < i));
                r += before;
            }
            a.order[r] = a.present[i];
        }
    } else {  // RAND: Fisher-Yates from the ascending list, i = k-1 .. 1
        for (int32_t i = t; i < k; i += kOrderThreads) {
            a.jtab[i] = i == 0 ? 0
                               : static_cast<int32_t>(scale_index(perm_word(a.seed, i, a.iteration),
                                                                  static_cast<uint32_t>(i + 1)));
            if (k <= kShuffleSmem) s.shuffle[i] = a.present[i];
            else a.order[i] = a.present[i];
        }
        __syncthreads();
        if (t == 0) {
            int32_t* L = k <= kShuffleSmem ? s.shuffle : a.order;
            for (int32_t i = k - 1; i >= 1; --i) {
                const int32_t j = a.jtab[i];
                const int32_t x = L[i];
                L[i] = L[j];
                L[j] = x;
            }
        }
        __syncthreads();
        if (k <= kShuffleSmem)
            for (int32_t i = t; i < k; i += kOrderThreads) a.order[i] = s.shuffle[i];
    }
    __syncthreads();

    // rank of every present color; segments (class-major, bucket-minor) in
    // list entries and in warp tiles
    for (int32_t p = t; p < k; p += kOrderThreads) a.rank_of[a.order[p]] = p;
    build_segments(a, k, s, [&](int32_t sg) {
        const int b = sg % kRcNB;
        const int32_t c = a.order[sg / kRcNB];
        return b == 0 ? a.cls_units[c] : a.cls_cnt[c * kRcNB + b];
    });
    if (over) atomicOr(&a.ctrl->err, kErrImproper);  // the tables hold the colors up to cap: no iteration on others
}

// ---------------------------------------------------------------------------
// Counting-sort scatter into class-major segments.  Each block counts the
// list entries of its vertices per segment in shared memory, reserves its
// ranges with one global atomic per (block, segment), then places them.  A
// bucket-0 row takes one entry per chunk and a split-row slot.  (Order inside
// a segment is free: a class is an independent set.)
// ---------------------------------------------------------------------------
constexpr int kScatterSegs = 6144;  // segments counted in (dynamic) shared memory: 48 KB

struct ScatterInfo {
    int32_t rank;
    int32_t b;
    int32_t sg;
    int32_t units;
    int64_t beg;
    int32_t deg;
};

// What the scatter reads of a vertex, loaded an iteration ahead of its use.
// (The rows were checked when the buckets were set.)
template <bool kBatch>
struct ScatterRow {
    int32_t b, c, gi;
    int64_t beg, end;
    __device__ __forceinline__ void load(const RcArgs& a, int64_t v, bool offsets) {
        b = a.bucket[v];
        c = a.old_c[v];
        if (kBatch) gi = a.graph_of[v];
        if (offsets) {
            beg = __ldg(a.g.off + v);
            end = __ldg(a.g.off + v + 1);
        }
    }
    // The rank of its class, or -1: a batch's finished graph (keeps its colors), -2: isolated.
    __device__ __forceinline__ int32_t rank(const RcArgs& a) const {
        int64_t key = c;
        if (kBatch) {  // the graph's own class ranks
            if (a.iteration >= a.desc[gi].iterations) return -1;
            key += a.cls_base[gi];
        }
        return b == kIsoBucket ? -2 : a.rank_of[key];
    }
    __device__ __forceinline__ int32_t deg() const { return static_cast<int32_t>(end - beg); }
    __device__ __forceinline__ int32_t units() const { return b == 0 ? chunks_of(deg()) : 1; }
};

// A vertex without a list entry: a finished graph's (rank -1) keeps its color,
// an isolated one (-2) takes color 1 and is counted in `iso`.
__device__ __forceinline__ void place_unlisted(const RcArgs& a, int32_t v, int32_t rank, int32_t& iso) {
    if (rank == -2) {
        a.new_c[v] = 1;
        ++iso;
    } else {
        a.new_c[v] = a.old_c[v];
    }
}

// The isolated vertices placed by a block: counted in the next iteration's
// class 1 (one graph), and the iteration's max color is at least 1.  The
// entries of the others' rows are the ones this iteration examines.
__device__ __forceinline__ void flush_placed(const RcArgs& a, int32_t iso, unsigned long long edges) {
    warp_add(&a.ctrl->edges, edges);
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) iso += __shfl_xor_sync(kFull, iso, d);
    if (lane_id() == 0 && iso > 0) {
        if (a.nxt_iso) atomicAdd(&a.nxt_iso[1], iso);
        if (a.ncolors) atomicMax(&a.ncolors[a.iteration + 1], 1);
    }
}

__device__ __forceinline__ void place(const RcArgs& a, int32_t v, const ScatterInfo& si, int32_t pos) {
    a.new_c[v] = -(si.rank + 1);
    if (si.b != 0) {
        store_item(a.list + pos, si.beg, v, si.deg);
        return;
    }
    const int32_t slot = atomicAdd(&a.ctrl->hub_next, 1);
    a.hub_v[slot] = v;
    a.hub_nch[slot] = si.units;
    a.hub_pcnt[slot] = 0;
    a.hub_done[slot] = -si.units;  // counted up to 0 by the chunks
    for (int32_t w = 0; w < a.hub_words; ++w) a.hub_bm[static_cast<int64_t>(slot) * a.hub_words + w] = 0u;
    for (int32_t c = 0; c < si.units; ++c) {
        const int32_t len = min(kChunk, si.deg - c * kChunk);
        store_item(a.list + pos + c, si.beg + static_cast<int64_t>(c) * kChunk, -(slot + 1), len);
    }
}

// Reserve `units` entries of segment sg from a counter (warp-aggregated
// when all peers reserve one entry).
__device__ __forceinline__ int32_t reserve(int32_t* counter_base, const ScatterInfo& si) {
    if (si.units != 1) return atomicAdd(&counter_base[si.sg], si.units);
    const unsigned act = __activemask();
    const unsigned peers = __match_any_sync(act, si.sg);
    const int leader = __ffs(peers) - 1;
    int32_t base = 0;
    if (lane_id() == leader) base = atomicAdd(&counter_base[si.sg], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + __popc(peers & ((1u << lane_id()) - 1u));
}

// Reserve `units` entries of s_cnt[sg]: the active lanes whose segment is
// `hot` share one atomic (ballot, not a match), the others take their own.
__device__ __forceinline__ int32_t hot_or_own(int32_t* s_cnt, int32_t sg, int32_t units, int32_t hot) {
    const unsigned act = __activemask();
    const bool is_hot = sg == hot && units == 1;
    const unsigned hm = __ballot_sync(act, is_hot);
    if (!is_hot) return atomicAdd(&s_cnt[sg], units);
    const int l = lane_id();
    const int leader = __ffs(hm) - 1;
    int32_t base = 0;
    if (l == leader) base = atomicAdd(&s_cnt[sg], __popc(hm));
    base = __shfl_sync(hm, base, leader);
    return base + __popc(hm & ((1u << l) - 1u));
}

// A vertex's loads are issued an iteration ahead of their use (the kernel
// waits for memory latency, not bandwidth).  On one graph a block takes every
// grid-th group of vertices: skewed graphs have their hubs at neighboring
// ids, and the block whose slice held them placed their chunks alone.  A batch
// keeps slices (a block then looks up few graphs' class ranks).  Per iteration,
// before / with the loads ahead / and strided: R-MAT 24 0.445 / 0.399 / 0.207
// ms, R-MAT 22 0.104 / 0.097 / 0.060, stencil 128^3 27 / 25 / 23 us, a batch
// of 512 graphs 0.18 / 0.109 / 0.126 ms.  A graph without split rows keeps
// slices too once its colors outgrow what L2 serves at full rate: the lists
// are then in the order of the ids, and a graph whose ids are local gathers
// locally (2048 graphs as one of 304 M vertices: 48 / 29 instead of 61 / 61 ms
// of cooperative / stepwise recoloring; the shuffled stencil, whose 8 MB of
// colors need no order, would lose 3 %).
constexpr int64_t kSliceMin = int64_t(16) << 20;
template <bool kBatch>
__global__ void __launch_bounds__(kBlock) k_rc_scatter(RcArgs a) {
    extern __shared__ int32_t s_cnt[];  // a.scatter_segs counts, then as many bases
    int32_t* const s_base = s_cnt + a.scatter_segs;
    if (a.ctrl->err & (kErrImproper | kErrBadGraph)) return;
    const int32_t nseg = a.ctrl->k * kRcNB;
    const bool slices = kBatch || (a.g.n > kSliceMin && a.ctrl->n_heavy == 0);
    const int64_t slice = (static_cast<int64_t>(a.g.n) + gridDim.x - 1) / gridDim.x;
    const int64_t first = static_cast<int64_t>(blockIdx.x) * (slices ? slice : kBlock) + threadIdx.x;
    const int64_t hi = slices ? min(static_cast<int64_t>(a.g.n), (blockIdx.x + 1) * slice) : a.g.n;
    const int64_t stride = slices ? kBlock : static_cast<int64_t>(gridDim.x) * kBlock;
    const bool many = nseg > a.scatter_segs;  // many classes: global atomics
    const int32_t hot = a.ctrl->hot_sg;
    if (!many) {
        for (int i = threadIdx.x; i < nseg; i += kBlock) s_cnt[i] = 0;
        __syncthreads();
        // count: the segment and, for a split row, its chunk count (no row read
        // for the others); shared-memory atomics, positions inside a segment are
        // free (a class is an independent set).  The lanes of a warp that fall
        // into the largest segment (on a skewed graph most vertices do) take
        // their entries with one atomic.
        ScatterRow<kBatch> row{}, next{};
        if (first < hi) next.load(a, first, false);
        for (int64_t i = first; i < hi; i += stride) {
            row = next;
            if (i + stride < hi) next.load(a, i + stride, false);
            const int32_t rank = row.rank(a);
            if (rank < 0) continue;
            int32_t units = 1;
            if (row.b == 0) units = chunks_of(static_cast<int32_t>(__ldg(a.g.off + i + 1) - __ldg(a.g.off + i)));
            hot_or_own(s_cnt, rank * kRcNB + row.b, units, hot);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nseg; i += kBlock) {
            const int32_t c = s_cnt[i];
            if (c) s_base[i] = a.seg_start[i] + atomicAdd(&a.fill[i], c);
            s_cnt[i] = 0;
        }
        __syncthreads();
    }
    int32_t iso = 0;
    unsigned long long edges = 0;
    ScatterRow<kBatch> row{}, next{};
    if (first < hi) next.load(a, first, true);
    for (int64_t i = first; i < hi; i += stride) {
        row = next;
        if (i + stride < hi) next.load(a, i + stride, true);
        const int32_t v = static_cast<int32_t>(i);
        ScatterInfo si;
        si.rank = row.rank(a);
        if (si.rank < 0) {
            place_unlisted(a, v, si.rank, iso);
            continue;
        }
        si.b = row.b;
        si.sg = si.rank * kRcNB + si.b;
        si.units = row.units();
        si.beg = row.beg;
        si.deg = row.deg();
        edges += static_cast<unsigned long long>(si.deg);
        const int32_t pos = many ? a.seg_start[si.sg] + reserve(a.fill, si)
                                 : s_base[si.sg] + hot_or_own(s_cnt, si.sg, si.units, hot);
        place(a, v, si, pos);
    }
    flush_placed(a, iso, edges);
}

// ---------------------------------------------------------------------------
// The class steps
// ---------------------------------------------------------------------------
// Color of neighbor u as seen by a vertex of class rank p (< 1 = ignore).
//
// In the dataflow form an entry of new_c changes once in the launch, from
// -(rank + 1) to the final color, so a stale copy can only be the negative
// placeholder.  On graphs with split (hub) rows the first read is an
// L1-cached weak load: millions of light rows read the same few hub colors,
// which as GPU-scope loads all queue at the few L2 lines holding them
// (R-MAT scale 24: 6.14 -> 5.17 ms per iteration).  A positive value read
// that way is final; a negative one of an earlier class is read again from
// L2 (relaxed) while waiting.  Without hub rows the gathers are scattered
// and gain nothing from L1 (the shuffled stencil: 0.325 -> 0.335 ms), so they
// stay GPU-scope loads.
__device__ __forceinline__ int32_t ld_weak_l1(const int32_t* p) {
    int32_t x;
    asm volatile("ld.global.ca.s32 %0, [%1];" : "=r"(x) : "l"(p));
    return x;
}

template <bool kDataflow>
struct RecolorFetch {
    int32_t* new_c;
    int32_t p;
    int32_t spin_limit;
    uint32_t* err;
    bool cached;  // first read through L1 (dataflow form, graphs with hub rows)
    __device__ __forceinline__ int32_t raw(int32_t u) const {
        if (!kDataflow) return __ldcg(new_c + u);
        return cached ? ld_weak_l1(new_c + u) : ld_relaxed(new_c + u);
    }
    __device__ __forceinline__ int32_t resolve(int32_t u, int32_t x) const {
        if (x > 0) return x;
        if (!kDataflow || -x - 1 >= p) return 0;  // later class: not recolored yet
        // Earlier class, still in flight: bounded wait.  Once any wait of the
        // launch has run out, every other wait gives up at once, so a launch
        // never spends more than about one spin_limit in waits.
        unsigned ns = 32;
        for (int32_t it = 0; it < spin_limit; ++it) {
            __nanosleep(ns);
            if (ns < 256) ns <<= 1;
            x = ld_relaxed(new_c + u);
            if (x > 0) return x;
            if ((it & 63) == 0 &&
                (ld_relaxed(reinterpret_cast<const int32_t*>(err)) & static_cast<int32_t>(kErrTimeout)))
                return 0;
        }
        atomicOr(err, kErrTimeout);
        return 0;
    }
};

// Histogram of the new colors for the next iteration: counts in dynamic
// shared memory sized to the colors (up to 1169 colors), flushed once per
// block; beyond that, global counts, where the lanes of a warp that add to
// the same (color, bucket) are merged into one atomic (most vertices of a
// skewed graph take the same few colors, and unmerged adds to one global
// counter serialise in L2).
constexpr int kRcHistSmem = 8192;

struct NextHist {
    int32_t* sh;     // nullptr: count in global memory
    int32_t* glob;
    int32_t* units;
    int32_t cap;
    uint32_t* over;
    __device__ __forceinline__ void add(int32_t c, int b, int32_t chunks) const {
        if (c < 1 || c > cap) {
            if (over) atomicOr(over, 1u);
            return;
        }
        const int32_t key = c * kRcNB + b;
        if (sh) {
            atomicAdd(&sh[key], 1);
        } else {
            const unsigned act = __activemask();
            const unsigned peers = __match_any_sync(act, key);
            if (lane_id() == __ffs(peers) - 1) atomicAdd(&glob[key], __popc(peers));
        }
        if (b == 0) atomicAdd(&units[c], chunks);
    }
};

// A neighbor that is not there: later than every class.
constexpr int32_t kNoNeighbor = -0x7fffffff;

// A neighbor that was read as -(rank + 1), of a class rank below `horizon`:
// earlier and still in flight.  (A color, 1 or more, gives a huge number.)
__device__ __forceinline__ bool in_flight(int32_t x, int32_t horizon) {
    return static_cast<uint32_t>(~x) < static_cast<uint32_t>(horizon);
}

// Colors of up to 8 neighbors per lane (u[i] < 0: none), all loads in flight
// together.
template <bool kDataflow>
__device__ __forceinline__ void load8(const RecolorFetch<kDataflow>& f, const int32_t (&u)[8], int32_t (&x)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        x[i] = kNoNeighbor;
        if (u[i] >= 0) x[i] = f.raw(u[i]);
    }
}

// Waits until no neighbor of a class before `horizon` is in flight (bounded;
// once any wait of the launch has run out, every other one gives up at once,
// so a launch never spends more than about one spin_limit in waits).  Each
// lane polls its pending neighbor of the latest class; when it is there, the
// others mostly are too and all are read again.  A poll is one load and a
// few instructions per lane, so it does not back off: with sleeps of up to
// 256 ns the class chain (which every poll is a link of) was 10-20 % slower
// (R-MAT 22 1.33 -> 1.27 ms per iteration, R-MAT 18 0.51 -> 0.48), and with
// all of a lane's pending neighbors in every poll R-MAT 24 lost 4 %.  The
// whole warp calls it.
template <bool kDataflow>
__device__ __forceinline__ void wait8(const RecolorFetch<kDataflow>& f, const int32_t (&u)[8], int32_t (&x)[8],
                                      int32_t horizon) {
    for (int32_t it = 0; kDataflow;) {
        int32_t q = -1, r = -1;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (in_flight(x[i], horizon) && ~x[i] > r) {
                r = ~x[i];
                q = u[i];
            }
        bool there = q < 0;
        if (__all_sync(kFull, there)) return;
        for (;; ++it) {
            if (it >= f.spin_limit) {
                if (!there) atomicOr(f.err, kErrTimeout);
                return;
            }
            if (!there) there = ld_relaxed(f.new_c + q) > 0;
            if (__all_sync(kFull, there)) break;
            // (a vote: a lane that left alone would be missed by the others)
            if ((it & 63) == 0 &&
                __any_sync(kFull, ld_relaxed(reinterpret_cast<const int32_t*>(f.err)) & static_cast<int32_t>(kErrTimeout)))
                return;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (in_flight(x[i], f.p)) x[i] = ld_relaxed(f.new_c + u[i]);
    }
}

// What a warp keeps in shared memory: the work items of its current and next
// tile, the ids of its next tile (kStageIds over the tile's rows), the two
// tiles' segments and entry counts, and a bitmap of forbidden colors.
constexpr int kStageIds = 384;
struct __align__(16) WarpStage {
    WorkItem item[2][32];
    int32_t ids[kStageIds];
    int4 meta[2];  // class rank, bucket, entries
    uint32_t bm[kWarpBitmapWords];
    uint32_t have[kWarpBitmapWords];  // a chunk's row: its merged bits, as read with the chunk
    int32_t win_t[32], win_s[32];     // tile prefix and start of the segments sought next
};

__device__ __forceinline__ void stage_copy16(void* smem, const void* gmem, int bytes) {
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;" ::"r"(sa), "l"(gmem), "r"(bytes),
                 "l"(policy_evict_first())
                 : "memory");
}

__device__ __forceinline__ void stage_copy4(void* smem, const void* gmem) {
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}

// The ids that the tile's lanes take first (8 per lane: the whole row except
// for 4-lane rows above 32 entries and warp rows above 256), as aligned
// 16-byte pieces, into each row's part of the stage.
__device__ __forceinline__ void stage_ids(const RcArgs& a, WarpStage& w, int slot) {
    if (!a.g.vec) return;
    const int4 m = w.meta[slot];
    const int lg = lanes_log2(m.y), G = 1 << lg;
    const int gi = lane_id() >> lg, gl = lane_id() & (G - 1);
    if (gi >= m.z) return;
    const WorkItem it = w.item[slot][gi];
    int32_t* dst = w.ids + gi * (kStageIds >> (5 - lg));
    const int64_t e0 = it.beg & ~static_cast<int64_t>(3);
    const int32_t nch = (static_cast<int32_t>(it.beg & 3) + min(it.deg, 8 << lg) + 3) >> 2;
    for (int32_t c = gl; c < nch; c += G) {
        const int64_t e = e0 + 4 * static_cast<int64_t>(c);
        stage_copy16(dst + 4 * c, a.g.idx + e, static_cast<int>(min(static_cast<int64_t>(16), 4 * (a.g.nnz - e))));
    }
}

// Skewed graphs have hundreds of classes that hold hub rows only, and a
// hub waits for hubs of the class just before its own: the launch is a chain
// of as many links, each the time from one hub's color to the next one's.
// Were every chunk to wait for its own neighbors, a link would be poll,
// merge into the row's bitmap, counting atomic (with its fence), bitmap
// read and pick, about 4 us.  Instead a chunk waits only for classes more
// than kNearClasses before its own, merges and counts at once, and leaves the
// nearer neighbors still in flight to the row's last chunk: that one holds the
// merged bitmap while it polls them, so a link is poll, pick and store.  A
// chunk that finds the row's list full waits for its own.  (ms per iteration,
// no deferral / 1 / 2 / 4 classes: R-MAT 22 1.30 / 1.10 / 0.98 / 1.00, R-MAT 18
// 0.50 / 0.40 / 0.34 / 0.33, RMAT-Bad 22 0.61 / 0.58 / 0.56 / 0.55, R-MAT 24
// 3.43 / 3.30 / 3.21 / 3.27; a list of 128 entries overflowed: R-MAT 24 4.3.)
//
// Ends: the smallest-class unfinished row has all its tiles dealt before any
// that waits for it, and their owners can only be waiting for rows of still
// smaller classes.
__device__ __forceinline__ void defer_near(const RcArgs& a, const RecolorFetch<true>& f, int32_t slot,
                                           const int32_t (&u)[8], int32_t (&x)[8]) {
    const int l = lane_id();
    uint32_t mine = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) mine += in_flight(x[i], f.p);
    const uint32_t incl = warp_inclusive_scan(mine);
    const int32_t total = static_cast<int32_t>(__shfl_sync(kFull, incl, 31));
    if (total == 0) return;
    int32_t base = 0;
    if (l == 0) base = atomicAdd(a.hub_pcnt + slot, total);
    base = __shfl_sync(kFull, base, 0);
    int32_t* pend = a.hub_pend + static_cast<int64_t>(slot) * kRowPend;
    int32_t pos = base + static_cast<int32_t>(incl - mine);
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (in_flight(x[i], f.p)) {
            if (pos < kRowPend) pend[pos] = u[i];
            ++pos;
        }
    if (base + total > kRowPend) wait8<true>(f, u, x, f.p);
}
__device__ __forceinline__ void defer_near(const RcArgs&, const RecolorFetch<false>&, int32_t, const int32_t (&)[8],
                                           int32_t (&)[8]) {}

// One warp tile whose items and ids are staged: its rows' lanes gather the
// neighbors' colors 8 at a time.  A row of up to kBitsDeg entries keeps its
// forbidden colors in 64 register bits; a longer warp row or a chunk of a split row
// keeps colors 1..32 in a register (most neighbors of a hub carry one of the
// lowest colors, and as shared atomics they would all hit one word) and the
// others in a shared bitmap.
//
// A chunk's forbidden colors are OR-ed into the row's bitmap; the warp
// finishing the last chunk picks the First-Fit color.  Ordering: the lanes'
// OR-s into the row's bitmap precede a warp barrier, and lane 0 then counts
// the chunk with one acquire-release atomic.  Its release covers the warp's
// OR-s (the barrier orders them before it); the last chunk's acquire reads
// the end of the counter's chain of increments, so it sees every chunk's
// OR-s, and the barrier after it orders the lanes' bitmap reads after it.
template <bool kDataflow, class Ahead>
__device__ __forceinline__ void recolor_tile(const RcArgs& a, const NextHist& nh, WarpStage& w, int slot, bool cached,
                                             int32_t& my_max, Ahead&& stage_ahead) {
    const int l = lane_id();
    const int4 m = w.meta[slot];
    const int32_t p = m.x;
    const int b = m.y;
    const int lg = lanes_log2(b), G = 1 << lg;
    const int gi = l >> lg, gl = l & (G - 1);
    const bool valid = gi < m.z;
    WorkItem it{0, 0, 0};
    if (valid) it = w.item[slot][gi];
    const RecolorFetch<kDataflow> f{a.new_c, p, a.tune.spin_limit, &a.ctrl->err, cached};

    int32_t u[8], x[8];
    bool bad = false;
    {
        const int32_t* ids = w.ids + gi * (kStageIds >> (5 - lg)) + (it.beg & 3);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int32_t k = gl + (i << lg);
            u[i] = -1;
            if (k < it.deg) {
                u[i] = a.g.vec ? ids[k] : ld_stream(a.g.idx + it.beg + k);
                if (static_cast<uint32_t>(u[i]) >= static_cast<uint32_t>(a.g.n)) {
                    bad = true;
                    u[i] = -1;
                }
            }
        }
    }
    __syncwarp();   // the slot and the staged ids are read: the next tiles' may land there
    stage_ahead();

    const bool bits = b >= 2 || (b == 1 && it.deg <= kBitsDeg);  // (the same for the whole warp)
    uint32_t lo = 0, hi = 0;
    if (!bits) {
        w.bm[l] = 0u;
        w.bm[l + 32] = 0u;
        if (b == 0) {
            // the row's bits already merged (read in the shadow of the gathers): a word
            // adding no new bit is not merged again; bits are only ever set during the launch
            if (4 * l < min(a.hub_words, kWarpBitmapWords))
                stage_copy16(&w.have[4 * l], a.hub_bm + static_cast<int64_t>(-it.v - 1) * a.hub_words + 4 * l, 16);
            cp_async_commit();
        }
        __syncwarp();
    }
    for (int32_t k0 = 0;;) {
        load8<kDataflow>(f, u, x);
        wait8<kDataflow>(f, u, x, b == 0 ? max(p - kNearClasses, 0) : p);
        if (b == 0 && kDataflow) defer_near(a, f, -it.v - 1, u, x);
        if (bits) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                lo |= bit_or_none(x[i] - 1);
                hi |= bit_or_none(x[i] - 33);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                lo |= bit_or_none(x[i] - 1);
                if (x[i] > 32 && x[i] <= 32 * kWarpBitmapWords) atomicOr(&w.bm[(x[i] - 1) >> 5], 1u << ((x[i] - 1) & 31));
            }
        }
        k0 += 8 << lg;
        if (!__any_sync(kFull, k0 < it.deg)) break;
#pragma unroll
        for (int i = 0; i < 8; ++i) {  // longer rows: the rest is not staged
            const int32_t k = k0 + gl + (i << lg);
            u[i] = k < it.deg ? load_nbr(a.g, it.beg + k, &a.ctrl->err) : -1;
        }
    }
    if (bad) atomicOr(&a.ctrl->err, kErrBadGraph);

    if (bits) {
        for (int d = G >> 1; d >= 1; d >>= 1) {
            lo |= __shfl_xor_sync(kFull, lo, d);
            hi |= __shfl_xor_sync(kFull, hi, d);
        }
        if (valid && gl == 0) {
            const int32_t c = ~lo ? __ffs(~lo) : 32 + __ffs(~hi);  // a free one: deg < 64
            st_relaxed(a.new_c + it.v, c);
            my_max = max(my_max, c);
            nh.add(c, b, 0);
        }
        return;
    }
    lo = __reduce_or_sync(kFull, lo);
    __syncwarp();
    uint32_t w0 = w.bm[l], w1 = w.bm[l + 32];
    if (l == 0) w0 |= lo;
    if (b == 1) {
        const uint32_t any0 = __ballot_sync(kFull, ~w0 != 0u), any1 = __ballot_sync(kFull, ~w1 != 0u);
        int32_t c;
        if (any0 | any1) {
            const int src = __ffs(any0 ? any0 : any1) - 1;
            const uint32_t fw = __shfl_sync(kFull, ~(any0 ? w0 : w1), src);
            c = ((any0 ? 0 : 32) + src) * 32 + __ffs(fw);
        } else {  // every color of the window is taken
            c = choose_warp<4>(a.g, it.beg, it.deg, 0u, f, w.bm, &a.ctrl->err);
        }
        if (l == 0) {
            st_relaxed(a.new_c + it.v, c);
            my_max = max(my_max, c);
            nh.add(c, 1, 0);
        }
        return;
    }
    static_assert(kWarpBitmapWords == 64, "two bitmap words per lane");
    uint32_t* hb = a.hub_bm + static_cast<int64_t>(-it.v - 1) * a.hub_words;
    cp_async_wait<0>();  // (the next tiles' copies are in the same queue: they had the gathers' time)
    __syncwarp();
    if (l < a.hub_words && (w0 & ~w.have[l])) atomicOr(&hb[l], w0);
    if (l + 32 < a.hub_words && (w1 & ~w.have[l + 32])) atomicOr(&hb[l + 32], w1);
    for (int32_t s0 = kWarpBitmapWords; s0 < a.hub_words; s0 += kWarpBitmapWords) {  // colors beyond the first window
        __syncwarp();
        w.bm[l] = 0u;
        w.bm[l + 32] = 0u;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int32_t d = x[i] - 1 - 32 * s0;
            if (x[i] > 0 && d >= 0 && d < 32 * kWarpBitmapWords) atomicOr(&w.bm[d >> 5], 1u << (d & 31));
        }
        __syncwarp();
        if (s0 + l < a.hub_words && w.bm[l]) atomicOr(&hb[s0 + l], w.bm[l]);
        if (s0 + l + 32 < a.hub_words && w.bm[l + 32]) atomicOr(&hb[s0 + l + 32], w.bm[l + 32]);
    }
    __syncwarp();
    int last = 0;
    if (l == 0) last = add_acq_rel(a.hub_done - it.v - 1) == -1;  // counts up from minus the chunks
    last = __shfl_sync(kFull, last, 0);
    __syncwarp();
    if (!last) return;
    // The neighbors left to this chunk, then First Fit over the merged bitmap.
    // Everything it takes is loaded at once (the list's words past its count
    // are dropped); with one window w.bm still holds this chunk's bits, which
    // are the row's too.
    uint32_t h0 = l < a.hub_words ? __ldcg(hb + l) : ~0u;
    uint32_t h1 = l + 32 < a.hub_words ? __ldcg(hb + l + 32) : ~0u;
    const int32_t hv = l == 0 ? __ldg(a.hub_v - it.v - 1) : 0;
    int32_t left = 0;
    if (kDataflow) {
        const int32_t* pend = a.hub_pend + static_cast<int64_t>(-it.v - 1) * kRowPend;
        left = __ldcg(a.hub_pcnt - it.v - 1);
#pragma unroll
        for (int i = 0; i < 8; ++i) u[i] = __ldcg(pend + l + 32 * i);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (l + 32 * i >= left) u[i] = -1;
        if (left > 0) {
            load8<kDataflow>(f, u, x);
            wait8<kDataflow>(f, u, x, p);
        }
    }
    for (int32_t s0 = 0; s0 < a.hub_words; s0 += kWarpBitmapWords) {
        if (a.hub_words > kWarpBitmapWords) {
            __syncwarp();
            w.bm[l] = 0u;
            w.bm[l + 32] = 0u;
            __syncwarp();
        }
        if (left > 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int32_t d = x[i] - 1 - 32 * s0;
                if (x[i] > 0 && d >= 0 && d < 32 * kWarpBitmapWords) atomicOr(&w.bm[d >> 5], 1u << (d & 31));
            }
        }
        __syncwarp();
        if (s0 > 0) {
            h0 = s0 + l < a.hub_words ? __ldcg(hb + s0 + l) : ~0u;
            h1 = s0 + l + 32 < a.hub_words ? __ldcg(hb + s0 + l + 32) : ~0u;
        }
        const uint32_t f0 = ~(h0 | w.bm[l]), f1 = ~(h1 | w.bm[l + 32]);
        const uint32_t any0 = __ballot_sync(kFull, f0 != 0u), any1 = __ballot_sync(kFull, f1 != 0u);
        if (any0 | any1) {
            const int src = __ffs(any0 ? any0 : any1) - 1;
            const uint32_t fw = __shfl_sync(kFull, any0 ? f0 : f1, src);
            const int32_t c = (s0 + (any0 ? 0 : 32) + src) * 32 + __ffs(fw);
            if (l == 0) {
                st_relaxed(a.new_c + hv, c);
                my_max = max(my_max, c);
                nh.add(c, 0, __ldg(a.hub_nch - it.v - 1));
            }
            return;
        }
    }
    // every color of the bitmap is taken (not on a symmetric CSR): a color
    // all the same, above cap, since others wait for the row
    if (l == 0) {
        const int32_t c = 32 * a.hub_words + 1;
        st_relaxed(a.new_c + hv, c);
        my_max = max(my_max, c);
        nh.add(c, 0, 0);
    }
}

// A warp's tiles t, t + step, ... below `end`, in order.  A tile is reached
// through four dependent reads (segment table, work items, ids, colors); the
// launch is bound by that latency (R-MAT 22 before: 5 % of DRAM, 30 % of the
// L1 rate, long-scoreboard stalls), so the first three run ahead: while a
// tile's colors are gathered, the ids of the next tile and the items of the
// one after are on their way to shared memory (cp.async, no registers) and
// the segment table's words for the third.  Together with one code path for
// all buckets, branch-free marks and 4 blocks per SM (64 registers, none
// spilled; a fifth block's 48 spilled 144 bytes: R-MAT 24 4.29 ms, stencil
// 0.293) an iteration takes, before -> after: 27-point stencil 128^3 315 ->
// 254 us (its 53.6 M scattered gathers alone take about 190 us at one L1TEX
// sector per clock and SM), R-MAT 24 4.25 -> 3.21 ms, R-MAT 22 1.72 -> 0.98,
// RMAT-Bad 22 0.95 -> 0.56, R-MAT 18 0.75 -> 0.34, a batch of 512 graphs 1.22
// -> 0.66 (the deferral of defer_near and the 1-lane rows included).
template <bool kDataflow>
__device__ __forceinline__ void recolor_tiles(const RcArgs& a, const NextHist& nh, WarpStage& w, uint32_t t,
                                              uint32_t end, uint32_t step, int32_t nseg, bool cached,
                                              int32_t& my_max) {
    if (t >= end) return;
    const int l = lane_id();
    int32_t sg = 0;
    auto load_window = [&]() {
        const int32_t i = min(sg + l, nseg);
        stage_copy4(&w.win_t[l], a.tile_prefix + i);
        stage_copy4(&w.win_s[l], a.seg_start + i);
    };
    // the items of tile tt, whose segment is sought from sg on, into a slot
    auto stage_items = [&](uint32_t tt, int slot) {
        int32_t win_t = w.win_t[l], win_s = w.win_s[l];
        int n;
        for (;;) {
            n = __popc(__ballot_sync(kFull, static_cast<uint32_t>(win_t) <= tt));
            if (n < 32) break;
            sg += 31;
            win_t = __ldg(a.tile_prefix + min(sg + l, nseg));
            win_s = __ldg(a.seg_start + min(sg + l, nseg));
        }
        sg += n - 1;
        const int32_t seg_t = __shfl_sync(kFull, win_t, n - 1), seg_s = __shfl_sync(kFull, win_s, n - 1);
        const int32_t seg_e = __shfl_sync(kFull, win_s, n);
        const int32_t rank = sg / kRcNB, bucket = sg - rank * kRcNB;
        const int tile = warp_tile(bucket);
        const int32_t first = seg_s + static_cast<int32_t>(tt - static_cast<uint32_t>(seg_t)) * tile;
        const int32_t cnt = min(tile, seg_e - first);
        if (l < cnt) stage_copy16(&w.item[slot][l], a.list + first + l, 16);
        if (l == 0) w.meta[slot] = make_int4(rank, bucket, cnt, 0);
    };
    sg = find_segment(a.tile_prefix, nseg, static_cast<int32_t>(t));
    load_window();
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
    stage_items(t, 0);
    load_window();
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
    stage_ids(a, w, 0);
    if (end - t > step) stage_items(t + step, 1);
    load_window();
    cp_async_commit();
    for (int slot = 0;; slot ^= 1) {
        cp_async_wait<0>();
        __syncwarp();
        const uint32_t left = end - t;  // tiles t + step, t + 2 step exist if left exceeds step, 2 step
        recolor_tile<kDataflow>(a, nh, w, slot, cached, my_max, [&]() {
            if (left > step) {
                stage_ids(a, w, slot ^ 1);
                if (left - step > step) stage_items(t + 2 * step, slot);
            }
            load_window();
            cp_async_commit();
        });
        if (left <= step) break;
        t += step;
    }
}

// Blocks of the dataflow launch: about one per 200 adjacency entries per
// color class, at least 16, at most all that fit.  An iteration is bound by
// its class chain when the classes are small (each class waits for the ones
// before it, and more warps only add pollers) and by throughput when they
// are large.  Per iteration with one block per 800 / 400 / 200 / 100 / 50
// entries: R-MAT 18 428 / 340 / 312 / 316 / 352 us, R-MAT 20 718 / 633 / 608 /
// 608 / 607 us, R-MAT 22 1.14 / 0.98 / 0.98 / 0.98 / 0.98 ms, G(10^4, 16) 29 /
// 23 / 23 / 24 / 24 us; a least grid of 8, 16, 32 or 64 blocks makes no
// difference there.
inline int coop_grid(int64_t nnz, int32_t classes, int capacity) {
    const int64_t want = nnz / (200 * static_cast<int64_t>(std::max(classes, 1)));
    return static_cast<int>(std::max<int64_t>(std::min<int64_t>(16, capacity), std::min<int64_t>(want, capacity)));
}

// Dataflow form, cooperative launch (every block resident): warp w takes the
// warp tiles w, w + W, w + 2W, ... in class order, W = all warps of the
// grid.  A tile waits only on tiles before it, and the owner of the first
// unfinished tile has finished all its earlier tiles, so it is working on
// that tile: the waits always end.
__device__ __forceinline__ NextHist setup_next_hist(const RcArgs& a, int32_t* s_hist) {
    if (!a.fuse_hist) return NextHist{nullptr, nullptr, nullptr, 0, nullptr};  // cap 0: add() is a no-op
    const bool local = a.hist_smem > 0;  // (cap + 1) * kRcNB entries of dynamic shared memory
    if (local)
        for (int i = threadIdx.x; i < a.hist_smem; i += kBlock) s_hist[i] = 0;
    return NextHist{local ? s_hist : nullptr, a.nxt_cnt, a.nxt_units, a.cap, &a.ctrl->over};
}

__device__ __forceinline__ void flush_next_hist(const RcArgs& a, const NextHist& nh) {
    if (!nh.sh) return;
    __syncthreads();
    const int32_t entries = (a.cap + 1) * kRcNB;
    for (int i = threadIdx.x; i < entries; i += kBlock)
        if (nh.sh[i]) atomicAdd(&a.nxt_cnt[i], nh.sh[i]);
}

__global__ void __launch_bounds__(kBlock, 4) k_rc_recolor_coop(RcArgs a) {
    __shared__ WarpStage s_stage[kWarps];
    extern __shared__ int32_t s_hist[];
    if (a.ctrl->err & (kErrImproper | kErrBadGraph)) return;
    const NextHist nh = setup_next_hist(a, s_hist);
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    int32_t my_max = 0;
    recolor_tiles<true>(a, nh, s_stage[warp], blockIdx.x * kWarps + warp, a.ctrl->total_tiles, gridDim.x * kWarps,
                        a.ctrl->k * kRcNB, a.ctrl->n_heavy > 0, my_max);
    warp_max(&a.ncolors[a.iteration + 1], my_max);
    flush_next_hist(a, nh);
}

// Stepwise form: one launch per class over its warp tiles [t0, t1).
__global__ void __launch_bounds__(kBlock, 4) k_rc_recolor_step(RcArgs a, int32_t t0, int32_t t1) {
    __shared__ WarpStage s_stage[kWarps];
    extern __shared__ int32_t s_hist[];
    if (a.ctrl->err & (kErrImproper | kErrBadGraph)) return;
    const NextHist nh = setup_next_hist(a, s_hist);
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    int32_t my_max = 0;
    recolor_tiles<false>(a, nh, s_stage[warp], t0 + blockIdx.x * kWarps + warp, t1, gridDim.x * kWarps,
                         a.ctrl->k * kRcNB, false, my_max);
    warp_max(&a.ncolors[a.iteration + 1], my_max);
    flush_next_hist(a, nh);
}

// ---------------------------------------------------------------------------
// Class ranks of a coloring (for aRC): the histogram and permutation kernels
// of one iteration, without the scatter and the class steps.
// ---------------------------------------------------------------------------
gc_status class_ranks_device(const Graph& g, const int32_t* colors, bool trusted, int32_t perm,
                             int32_t iteration, uint64_t seed, int32_t* rank_out, int32_t* maxc_out,
                             cudaStream_t s) {
    const int64_t n = g.n;
    *maxc_out = 0;
    if (n == 0) return GC_OK;
    if (!trusted && !rank_out) return check_input_device(g, colors, kMaxInputColor, maxc_out, s);
    const Tuning tune = recolor_tuning(current_tuning());
    const int grid = persistent_grid(tune);
    const int vgrid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n + kBlock - 1) / kBlock, grid)));
    RcArgs a;
    std::memset(&a, 0, sizeof(a));
    ScratchSet sc_rows, sc;
    sc_rows.want(&a.ctrl, sizeof(RcCtrl));
    sc_rows.want(&a.bucket, n);
    if (!sc_rows.alloc(s)) return GC_ERR_OOM;
    a.g = g;
    a.tune = tune;
    a.seed = seed;
    a.perm = perm;
    a.iteration = iteration;
    a.old_c = colors;
    cudaMemsetAsync(a.ctrl, 0, sizeof(RcCtrl), s);
    GC_LAUNCH(KID_RC_BUCKET, s, k_rc_bucket<<<vgrid, kBlock, 0, s>>>(a));
    int32_t max_checked = 0;
    gc_status st = GC_OK;
    if (!trusted) st = check_input_device(g, colors, kMaxInputColor, &max_checked, s);
    else GC_LAUNCH(KID_RC_VALIDATE, s, k_rc_maxin<<<vgrid, kBlock, 0, s>>>(a));
    if (st != GC_OK && st != GC_ERR_IMPROPER_INPUT) return st;
    RcCtrl h;
    cudaError_t ce = cudaMemcpyAsync(&h, a.ctrl, sizeof(RcCtrl), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_status(ce);
    if (h.err & kErrBadGraph) return GC_ERR_BAD_GRAPH;
    if (st != GC_OK || (h.err & kErrImproper)) return GC_ERR_IMPROPER_INPUT;
    if (!trusted) h.max_in = max_checked;
    *maxc_out = h.max_in;
    if (!rank_out) return GC_OK;
    const int32_t cap = std::max(h.max_in, 1);
    const int64_t ent = class_entries(cap);
    if (ent == 0) return GC_ERR_OOM;
    const int64_t c4 = static_cast<int64_t>(cap + 1) * 4, hist_bytes = ent * 4 + 2 * c4;
    sc.want(&a.cls_cnt, hist_bytes);
    sc.want(&a.present, c4);
    sc.want(&a.psize, c4);
    sc.want(&a.order, c4);
    sc.want(&a.jtab, c4);
    sc.want(&a.seg_start, (ent + 1) * 4);
    sc.want(&a.tile_prefix, (ent + 1) * 4);
    sc.want(&a.fill, ent * 4);
    if (!sc.alloc(s)) return GC_ERR_OOM;
    a.cap = cap;
    a.rank_of = rank_out;
    a.cls_units = a.cls_cnt + ent;
    a.iso_cnt = a.cls_units + cap + 1;
    cudaMemsetAsync(a.cls_cnt, 0, hist_bytes, s);
    cudaMemsetAsync(rank_out, 0, (cap + 1) * 4, s);
    GC_LAUNCH(KID_RC_HIST, s, k_rc_hist<false><<<vgrid, kBlock, 0, s>>>(a));
    GC_LAUNCH(KID_RC_ORDER, s, k_rc_order<<<1, kOrderThreads, 0, s>>>(a));
    ce = cudaMemcpyAsync(&h, a.ctrl, sizeof(RcCtrl), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_status(ce);
    return status_from_err_bits(h.err);
}

// ---------------------------------------------------------------------------
// Batches: per-graph class histograms and orders, global (rank, bucket)
// segments.  A vertex waits only on neighbors of its own graph of a smaller
// rank, and ranks are global segment keys, so the cooperative launch above
// serves the whole batch unchanged.
// ---------------------------------------------------------------------------
// A block's slice of consecutive vertices belongs to few graphs, and these
// own consecutive class tables, so the slice is counted in shared memory where
// the tables it spans fit (small graphs' in any case spread over many
// counters).  A batch of 512 graphs (11 M vertices): 47 us instead of 79 with
// a global atomic per warp and key, nearly all on the few counters of the
// graph at hand; 69 while a vertex's reads were not issued together.
constexpr int32_t kBrcSlice = 2048;
constexpr int32_t kBrcClasses = 512;
__global__ void __launch_bounds__(kBlock) k_brc_hist(RcArgs a) {
    __shared__ int32_t s_cnt[kBrcClasses * kRcNB];
    __shared__ int32_t s_iso[kBrcClasses];
    for (int64_t c0 = static_cast<int64_t>(blockIdx.x) * kBrcSlice; c0 < a.g.n;
         c0 += static_cast<int64_t>(gridDim.x) * kBrcSlice) {
        const int64_t c1 = min(c0 + kBrcSlice, static_cast<int64_t>(a.g.n));
        const int64_t k0 = a.cls_base[a.graph_of[c0]];
        const int64_t classes = a.cls_base[a.graph_of[c1 - 1] + 1] - k0;
        const bool local = classes <= kBrcClasses;
        if (local) {
            for (int i = threadIdx.x; i < classes * kRcNB; i += kBlock) s_cnt[i] = 0;
            for (int i = threadIdx.x; i < classes; i += kBlock) s_iso[i] = 0;
        }
        __syncthreads();
        constexpr int U = kBrcSlice / kBlock;
        int32_t gv[U], cv[U];
        uint8_t bv[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int64_t v = min(c0 + i * kBlock + threadIdx.x, c1 - 1);
            gv[i] = __ldg(a.graph_of + v);
            cv[i] = __ldg(a.old_c + v);
            bv[i] = __ldg(a.bucket + v);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int64_t v = c0 + i * kBlock + threadIdx.x;
            if (v >= c1) break;
            const int32_t gi = gv[i], c = cv[i], b = bv[i];
            if (a.iteration >= a.desc[gi].iterations) continue;
            const int64_t base = a.cls_base[gi];
            const int32_t maxc = static_cast<int32_t>(a.cls_base[gi + 1] - base - 1);
            if (c < 1 || c > maxc) {
                atomicOr(&a.ctrl->err, kErrImproper);
                continue;
            }
            const int64_t key = base + c;
            if (local) {
                if (b == kIsoBucket) atomicAdd(&s_iso[key - k0], 1);
                else atomicAdd(&s_cnt[(key - k0) * kRcNB + b], 1);
            } else {
                int32_t* at = b == kIsoBucket ? &a.iso_cnt[key] : &a.cls_cnt[key * kRcNB + b];
                const unsigned peers = __match_any_sync(__activemask(), reinterpret_cast<unsigned long long>(at));
                if (lane_id() == __ffs(peers) - 1) atomicAdd(at, __popc(peers));
            }
            if (b == 0) {
                int64_t rb;
                int32_t deg;
                row_of(a.g, static_cast<int32_t>(v), rb, deg, &a.ctrl->err);
                atomicAdd(&a.cls_units[key], chunks_of(deg));
            }
        }
        __syncthreads();
        if (local) {
            for (int i = threadIdx.x; i < classes * kRcNB; i += kBlock)
                if (s_cnt[i]) atomicAdd(&a.cls_cnt[k0 * kRcNB + i], s_cnt[i]);
            for (int i = threadIdx.x; i < classes; i += kBlock)
                if (s_iso[i]) atomicAdd(&a.iso_cnt[k0 + i], s_iso[i]);
            __syncthreads();
        }
    }
}

// One warp per graph: present classes, the graph's permutation (the rules of
// k_rc_order), the rank of each color, and the global segment counts.
__global__ void __launch_bounds__(kBlock) k_brc_order(RcArgs a) {
    const int l = lane_id();
    const int32_t warps = gridDim.x * kWarps;
    for (int32_t gi = blockIdx.x * kWarps + (threadIdx.x >> 5); gi < a.ngraphs; gi += warps) {
        const BatchDesc d = a.desc[gi];
        if (a.iteration >= d.iterations) continue;
        const int64_t base = a.cls_base[gi];
        const int32_t maxc = static_cast<int32_t>(a.cls_base[gi + 1] - base - 1);
        int32_t* present = a.gpresent + base;
        int32_t* psize = a.gpsize + base;
        int32_t* order = a.gorder + base;
        int32_t k = 0;
        for (int32_t c0 = 1; c0 <= maxc; c0 += 32) {
            const int32_t c = c0 + l;
            int32_t size = 0;
            if (c <= maxc) {
                for (int b = 0; b < kRcNB; ++b) size += a.cls_cnt[(base + c) * kRcNB + b];
                size += a.iso_cnt[base + c];
            }
            const uint32_t bal = __ballot_sync(kFull, size > 0);
            if (size > 0) {
                const int32_t pos = k + __popc(bal & ((1u << l) - 1u));
                present[pos] = c;
                psize[pos] = size;
            }
            k += __popc(bal);
        }
        __syncwarp();
        const int32_t perm = perm_at(d.perm, a.iteration);
        if (perm == 0) {
            for (int32_t i = l; i < k; i += 32) order[i] = present[k - 1 - i];
        } else if (perm == 1 || perm == 2) {
            const bool noninc = perm == 1;
            for (int32_t i = l; i < k; i += 32) {
                const int32_t si = psize[i];
                int32_t r = 0;
                for (int32_t j = 0; j < k; ++j) {
                    const int32_t sj = psize[j];
                    r += noninc ? (sj > si || (sj == si && j < i)) : (sj < si || (sj == si && j < i));
                }
                order[r] = present[i];
            }
        } else {
            int32_t* jtab = a.gjtab + base;
            for (int32_t i = l; i < k; i += 32) {
                jtab[i] = i == 0 ? 0
                                 : static_cast<int32_t>(scale_index(perm_word(d.perm_seed, i, a.iteration),
                                                                    static_cast<uint32_t>(i + 1)));
                order[i] = present[i];
            }
            __syncwarp();
            if (l == 0)
                for (int32_t i = k - 1; i >= 1; --i) {
                    const int32_t j = jtab[i];
                    const int32_t x = order[i];
                    order[i] = order[j];
                    order[j] = x;
                }
        }
        __syncwarp();
        for (int32_t p = l; p < k; p += 32) {
            const int32_t c = order[p];
            a.rank_of[base + c] = p;
            for (int b = 0; b < kRcNB; ++b) {
                const int32_t u = b == 0 ? a.cls_units[base + c] : a.cls_cnt[(base + c) * kRcNB + b];
                if (u) atomicAdd(&a.seg_cnt[p * kRcNB + b], u);
            }
        }
        if (l == 0) atomicMax(&a.ctrl->k, k);
    }
}

__global__ void __launch_bounds__(kOrderThreads) k_brc_segments(RcArgs a) {
    __shared__ OrderShared s;
    const int32_t k = a.ctrl->k;
    build_segments(a, k, s, [&](int32_t sg) { return a.seg_cnt[sg]; });
}

// ---------------------------------------------------------------------------
// Host driver
// ---------------------------------------------------------------------------
// The scatter's shared segment counters (sized to the classes, so that small
// tables leave the SM to more blocks and to L1) and its resident grid.
static int scatter_launch(RcArgs& a, const void* kernel, int32_t cap, const Tuning& tune, size_t* dyn) {
    a.scatter_segs = static_cast<int32_t>(std::min<int64_t>(static_cast<int64_t>(cap) * kRcNB, kScatterSegs));
    *dyn = static_cast<size_t>(a.scatter_segs) * 2 * sizeof(int32_t);
    const int64_t blocks = (static_cast<int64_t>(a.g.n) + kBlock - 1) / kBlock;
    const int64_t fit = tune.grid_blocks > 0 ? tune.grid_blocks
                                             : sm_count() * occupancy_of(kernel, kBlock, *dyn);
    return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(blocks, fit)));
}

gc_status recolor_device(const Graph& g, const int32_t* colors_in, int32_t maxc_in, int32_t max_deg, bool trusted,
                         int32_t perm, int32_t iterations, uint64_t seed, int32_t* colors_out,
                         int32_t* ncolors_per_iter, gc_stats* stats, cudaStream_t s) {
    const int64_t n = g.n;
    if (stats) std::memset(stats, 0, sizeof(*stats));
    const Tuning tune = recolor_tuning(current_tuning());
    const int grid = persistent_grid(tune);
    const int vgrid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n + kBlock - 1) / kBlock, grid)));
    cudaError_t ce;

    // (before anything else is allocated: the gathers of the check ran at 427 us
    // on R-MAT 22 with the buckets' array in front of its own, at 327 without)
    if (!trusted) {
        const gc_status input = check_input_device(g, colors_in, kMaxInputColor, &maxc_in, s);
        if (input != GC_OK) return input;
    }
    if (n == 0) {
        if (ncolors_per_iter)
            for (int32_t i = 0; i <= iterations; ++i) ncolors_per_iter[i] = 0;
        return GC_OK;
    }
    if (iterations == 0) {
        if (colors_out != colors_in)
            cudaMemcpyAsync(colors_out, colors_in, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, s);
        ce = cudaStreamSynchronize(s);
        if (ncolors_per_iter) ncolors_per_iter[0] = maxc_in;
        if (stats) stats->max_color = maxc_in;
        return ce == cudaSuccess ? GC_OK : cuda_status(ce);
    }

    RcArgs a;
    std::memset(&a, 0, sizeof(a));
    ScratchSet sc_rows, sc;
    const int64_t ctrl_bytes = sizeof(RcCtrl) + (static_cast<int64_t>(iterations) + 1) * 4;  // and the color counts
    sc_rows.want(&a.ctrl, ctrl_bytes);
    sc_rows.want(&a.bucket, n);
    if (!sc_rows.alloc(s)) return GC_ERR_OOM;
    a.ncolors = reinterpret_cast<int32_t*>(a.ctrl + 1);
    a.g = g;
    a.tune = tune;
    a.seed = seed;
    a.perm = perm;
    a.old_c = colors_in;
    cudaMemsetAsync(a.ctrl, 0, ctrl_bytes, s);
    RcCtrl h;
    std::memset(&h, 0, sizeof(h));
    // A trusted input (our own coloring) has a known max color and longest
    // row; the split rows are then sized by a bound (a bucket-0 row has more
    // than max(rc_warp_max_deg, 63) entries; none if the longest row is no
    // longer) instead of a read-back, when the bound's scratch is small.
    const int64_t heavy_min = std::max<int64_t>(tune.warp_max_deg, 63) + 1;
    const int64_t heavy_bound = max_deg < heavy_min ? 0 : std::min<int64_t>(n, static_cast<int64_t>(g.nnz) / heavy_min);
    const int64_t bound_words = (static_cast<int64_t>(std::max(maxc_in, 1)) + 1 + 31) / 32 + kRowPend;
    const bool read_back = !trusted || heavy_bound * bound_words * 4 > (int64_t(64) << 20);
    if (read_back) {
        GC_LAUNCH(KID_RC_BUCKET, s, k_rc_bucket<<<vgrid, kBlock, 0, s>>>(a));
        ce = cudaMemcpyAsync(&h, a.ctrl, sizeof(RcCtrl), cudaMemcpyDeviceToHost, s);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
        if (ce != cudaSuccess) return cuda_status(ce);
        if (h.err & kErrBadGraph) return GC_ERR_BAD_GRAPH;
    } else {
        h.n_heavy = static_cast<int32_t>(heavy_bound);
    }

    // Colors stay within [1, maxc_in]: a vertex of the class of rank p takes
    // at most color p + 1 <= k <= maxc_in.
    const int32_t cap = std::max(maxc_in, 1);
    const int64_t ent = class_entries(cap);
    if (ent == 0) return GC_ERR_OOM;
    const int32_t hub_words = ((cap + 1 + 31) / 32 + 3) & ~3;  // 16-byte rows
    const int64_t hubs = std::max<int64_t>(1, h.n_heavy);
    // list entries: one per vertex, one per chunk of a bucket-0 row
    const int64_t list_len = n + (static_cast<int64_t>(g.nnz) / kChunk) + h.n_heavy;
    const int64_t c4 = static_cast<int64_t>(cap + 1) * 4, hist_bytes = ent * 4 + 2 * c4;
    int32_t *hist = nullptr, *alt = nullptr;  // hist: this iteration's and the next one's class tables
    sc.want(&hist, 2 * hist_bytes);
    sc.want(&a.present, c4);
    sc.want(&a.psize, c4);
    sc.want(&a.order, c4);
    sc.want(&a.jtab, c4);
    sc.want(&a.rank_of, c4);
    sc.want(&a.seg_start, (ent + 1) * 4);
    sc.want(&a.tile_prefix, (ent + 1) * 4);
    sc.want(&a.fill, ent * 4);
    sc.want(&a.list, list_len * static_cast<int64_t>(sizeof(WorkItem)));
    sc.want(&alt, n * 4);
    sc.want(&a.hub_v, hubs * 4);
    sc.want(&a.hub_nch, hubs * 4);
    sc.want(&a.hub_done, hubs * 4);
    sc.want(&a.hub_pcnt, hubs * 4);
    sc.want(&a.hub_bm, hubs * hub_words * 4);
    sc.want(&a.hub_pend, hubs * kRowPend * 4);
    if (!sc.alloc(s)) return GC_ERR_OOM;
    a.cap = cap;
    a.hub_words = hub_words;
    a.fuse_hist = 1;
    const int32_t hist_entries = static_cast<int32_t>(ent);
    const size_t hist_dyn = hist_entries <= kRcHistSmem ? static_cast<size_t>(hist_entries) * 4 : 0;
    a.hist_smem = hist_dyn ? hist_entries : 0;
    if (hist_dyn > 16 * 1024)  // beyond 48 KB with the warps' stages
        for (const void* k : {reinterpret_cast<const void*>(k_rc_recolor_coop), reinterpret_cast<const void*>(k_rc_recolor_step)})
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kRcHistSmem * 4);
    size_t sc_dyn = 0;
    const int grid_sc = scatter_launch(a, reinterpret_cast<const void*>(k_rc_scatter<false>), cap, tune, &sc_dyn);
    const int coop_capacity =
        sm_count() * occupancy_of(reinterpret_cast<const void*>(k_rc_recolor_coop), kBlock, hist_dyn);
    const int grid_rc = tune.grid_blocks > 0 ? std::min(tune.grid_blocks, coop_capacity)
                                             : coop_grid(g.nnz, cap, coop_capacity);
    const int step_capacity =
        sm_count() * occupancy_of(reinterpret_cast<const void*>(k_rc_recolor_step), kBlock, hist_dyn);
    const int grid_step = tune.grid_blocks > 0 ? tune.grid_blocks : step_capacity;
    cudaMemsetAsync(hist, 0, 2 * hist_bytes, s);

    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    const int32_t* cur = colors_in;
    gc_status st = GC_OK;
    std::vector<int32_t> tp;
    for (int32_t it = 0; it < iterations && st == GC_OK; ++it) {
        int32_t* dst = (it % 2 == 0) ? alt : colors_out;
        a.iteration = it;
        a.old_c = cur;
        a.new_c = dst;
        // histograms: of the input (iteration 0), else filled by the previous
        // iteration's recoloring kernel
        const int64_t set = hist_bytes / 4;
        a.cls_cnt = hist + (it % 2) * set;
        a.cls_units = a.cls_cnt + ent;
        a.iso_cnt = a.cls_units + cap + 1;
        a.nxt_cnt = hist + (1 - it % 2) * set;
        a.nxt_units = a.nxt_cnt + ent;
        a.nxt_iso = a.nxt_units + cap + 1;
        if (it > 0) {
            cudaMemsetAsync(a.nxt_cnt, 0, hist_bytes, s);
        } else if (read_back) {
            GC_LAUNCH(KID_RC_HIST, s, k_rc_hist<false><<<vgrid, kBlock, 0, s>>>(a));
        } else {
            GC_LAUNCH(KID_RC_HIST, s, k_rc_hist<true><<<vgrid, kBlock, 0, s>>>(a));
        }
        GC_LAUNCH(KID_RC_ORDER, s, k_rc_order<<<1, kOrderThreads, 0, s>>>(a));
        GC_LAUNCH(KID_RC_SCATTER, s, k_rc_scatter<false><<<grid_sc, kBlock, sc_dyn, s>>>(a));
        if (tune.recolor_mode == 0) {
            void* args[] = {&a};
            cudaError_t le;
            GC_LAUNCH(KID_RC_RECOLOR, s,
                      le = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_rc_recolor_coop),
                                                       dim3(grid_rc), dim3(kBlock), args, hist_dyn, s));
            if (le != cudaSuccess) { st = cuda_status(le); break; }
        } else {
            RcCtrl hc;
            ce = cudaMemcpyAsync(&hc, a.ctrl, sizeof(RcCtrl), cudaMemcpyDeviceToHost, s);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
            if (ce != cudaSuccess) { st = cuda_status(ce); break; }
            tp.resize(static_cast<size_t>(hc.k) * kRcNB + 1);
            ce = cudaMemcpyAsync(tp.data(), a.tile_prefix, tp.size() * 4, cudaMemcpyDeviceToHost, s);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
            if (ce != cudaSuccess) { st = cuda_status(ce); break; }
            for (int32_t p = 0; p < hc.k; ++p) {
                const int32_t t0 = tp[p * kRcNB], t1 = tp[(p + 1) * kRcNB];
                if (t1 <= t0) continue;
                const int g2 = std::min(grid_step, (t1 - t0 + kWarps - 1) / kWarps);
                GC_LAUNCH(KID_RC_STEP, s, k_rc_recolor_step<<<g2, kBlock, hist_dyn, s>>>(a, t0, t1));
            }
        }
        cur = dst;
    }
    if (st == GC_OK && cur != colors_out)
        cudaMemcpyAsync(colors_out, cur, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, s);
    cudaEventRecord(e1, s);
    std::vector<char> back(static_cast<size_t>(ctrl_bytes));
    ce = cudaMemcpyAsync(back.data(), a.ctrl, back.size(), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    std::vector<int32_t> nc(static_cast<size_t>(iterations) + 1);
    if (ce == cudaSuccess) {
        std::memcpy(&h, back.data(), sizeof(RcCtrl));
        std::memcpy(nc.data(), back.data() + sizeof(RcCtrl), nc.size() * 4);
    }
    if (ce != cudaSuccess && st == GC_OK) st = cuda_status(ce);
    if (st == GC_OK) st = status_from_err_bits(h.err);
    if (ncolors_per_iter) std::copy(nc.begin(), nc.end(), ncolors_per_iter);
    if (stats) {
        stats->iterations = iterations;
        stats->max_color = nc[iterations];
        stats->edges_examined = static_cast<int64_t>(h.edges);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        stats->ms_recolor = ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}

// Batch recoloring: every graph recolored with its own permutation, seed and
// iteration count; a graph past its count keeps its colors.
// Iterations [it_begin, it_end) of every graph (it_end < 0: to the largest
// count); a graph whose count is reached keeps its colors.  Running the
// iterations in several calls gives the same colors as one call: an
// iteration's class order depends only on the colors it starts from and its
// own number.
static gc_status recolor_batch_impl(const Graph& g, const gc_batch_graph* graphs, int32_t ng,
                                    const int32_t* colors_in, bool trusted, const int32_t* max_in,
                                    int32_t* colors_out, int32_t* max_color_out, gc_stats* stats,
                                    cudaStream_t s, int32_t it_begin = 0, int32_t it_end = -1) {
    int32_t max_x = 1;
    gc_status st = batch_layout(g, graphs, ng, &max_x);
    if (st != GC_OK) return st;
    const int64_t n = g.n;
    if (stats) std::memset(stats, 0, sizeof(*stats));
    int32_t iters = 0;
    for (int32_t i = 0; i < ng; ++i) iters = std::max(iters, graphs[i].iterations);
    if (it_end >= 0) iters = std::min(iters, it_end);
    it_begin = std::max(it_begin, 0);
    if (iters < it_begin) iters = it_begin;
    const Tuning tune = recolor_tuning(current_tuning());
    const int grid = persistent_grid(tune);
    const int vgrid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n + kBlock - 1) / kBlock, grid)));
    const int coop_capacity = sm_count() * occupancy_of(reinterpret_cast<const void*>(k_rc_recolor_coop), kBlock);
    const int grid_step = resident_grid(k_rc_recolor_step, tune);
    const int grid_go = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((ng + kWarps - 1) / kWarps, grid)));
    cudaError_t ce;

    RcArgs a;
    std::memset(&a, 0, sizeof(a));
    ScratchSet sc_rows, sc;
    BatchDesc* desc = nullptr;
    int32_t* graph_of = nullptr;
    sc_rows.want(&a.ctrl, sizeof(RcCtrl));
    sc_rows.want(&a.bucket, n);
    sc_rows.want(&desc, static_cast<int64_t>(ng) * static_cast<int64_t>(sizeof(BatchDesc)));
    sc_rows.want(&graph_of, n * 4);
    if (!sc_rows.alloc(s)) return GC_ERR_OOM;
    ce = cudaMemcpyAsync(desc, graphs, static_cast<size_t>(ng) * sizeof(BatchDesc), cudaMemcpyHostToDevice, s);
    if (ce != cudaSuccess) return cuda_status(ce);
    a.g = g;
    a.tune = tune;
    a.old_c = colors_in;
    a.desc = desc;
    a.graph_of = graph_of;
    a.ngraphs = ng;
    batch_graph_of(g, desc, ng, graph_of, s);
    cudaMemsetAsync(a.ctrl, 0, sizeof(RcCtrl), s);
    if (n > 0) {
        GC_LAUNCH(KID_RC_BUCKET, s, k_rc_bucket<<<vgrid, kBlock, 0, s>>>(a));
    }
    gc_status input = GC_OK;
    if (!trusted) {
        int32_t max_checked = 0;
        input = check_input_device(g, colors_in, kMaxInputColor, &max_checked, s);
        if (input != GC_OK && input != GC_ERR_IMPROPER_INPUT) return input;
    }
    RcCtrl h;
    ce = cudaMemcpyAsync(&h, a.ctrl, sizeof(RcCtrl), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_status(ce);
    if (h.err & kErrBadGraph) return GC_ERR_BAD_GRAPH;
    if (input != GC_OK) return input;
    // each graph's max input color sizes its rows of the (graph, color) tables
    std::vector<int32_t> gmax(ng, 0);
    if (trusted && max_in) {
        std::copy(max_in, max_in + ng, gmax.begin());
    } else {
        st = batch_max_colors(g, a.graph_of, colors_in, nullptr, ng, gmax.data(), nullptr, s);
        if (st != GC_OK) return st;
    }
    std::vector<int64_t> base(static_cast<size_t>(ng) + 1, 0);
    int32_t cap = 1;
    for (int32_t i = 0; i < ng; ++i) {
        base[i + 1] = base[i] + gmax[i] + 1;
        cap = std::max(cap, gmax[i]);
    }
    const int64_t T = base[ng];
    if (iters == it_begin || n == 0) {
        if (colors_out != colors_in && n > 0)
            cudaMemcpyAsync(colors_out, colors_in, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, s);
        if (max_color_out) std::copy(gmax.begin(), gmax.end(), max_color_out);
        return cuda_status(cudaStreamSynchronize(s));
    }
    const int64_t ent = class_entries(cap);
    if (ent == 0) return GC_ERR_OOM;
    const int32_t hub_words = ((cap + 1 + 31) / 32 + 3) & ~3;  // 16-byte rows
    const int64_t hubs = std::max<int64_t>(1, h.n_heavy);
    const int64_t list_len = n + (static_cast<int64_t>(g.nnz) / kChunk) + h.n_heavy;
    const int grid_rc = tune.grid_blocks > 0 ? std::min(tune.grid_blocks, coop_capacity)
                                             : coop_grid(g.nnz, cap, coop_capacity);
    int64_t* cls_base = nullptr;
    int32_t *alt = nullptr;
    const int64_t t4 = T * 4, hist_bytes = (kRcNB + 2) * t4 + ent * 4;
    sc.want(&cls_base, (static_cast<int64_t>(ng) + 1) * 8);
    sc.want(&a.cls_cnt, hist_bytes);
    sc.want(&a.rank_of, t4);
    sc.want(&a.gpresent, t4);
    sc.want(&a.gpsize, t4);
    sc.want(&a.gorder, t4);
    sc.want(&a.gjtab, t4);
    sc.want(&a.seg_start, (ent + 1) * 4);
    sc.want(&a.tile_prefix, (ent + 1) * 4);
    sc.want(&a.fill, ent * 4);
    sc.want(&a.list, list_len * static_cast<int64_t>(sizeof(WorkItem)));
    sc.want(&alt, n * 4);
    sc.want(&a.ncolors, (static_cast<int64_t>(iters) + 1) * 4);
    sc.want(&a.hub_v, hubs * 4);
    sc.want(&a.hub_nch, hubs * 4);
    sc.want(&a.hub_done, hubs * 4);
    sc.want(&a.hub_pcnt, hubs * 4);
    sc.want(&a.hub_bm, hubs * hub_words * 4);
    sc.want(&a.hub_pend, hubs * kRowPend * 4);
    if (!sc.alloc(s)) return GC_ERR_OOM;
    ce = cudaMemcpyAsync(cls_base, base.data(), (ng + 1) * 8, cudaMemcpyHostToDevice, s);
    if (ce != cudaSuccess) return cuda_status(ce);
    a.cap = cap;
    a.cls_base = cls_base;
    a.cls_units = a.cls_cnt + T * kRcNB;
    a.iso_cnt = a.cls_units + T;
    a.seg_cnt = a.iso_cnt + T;
    a.hub_words = hub_words;
    a.fuse_hist = 0;
    size_t sc_dyn = 0;
    const int grid_sc = scatter_launch(a, reinterpret_cast<const void*>(k_rc_scatter<true>), cap, tune, &sc_dyn);
    cudaMemsetAsync(a.ncolors, 0, (iters + 1) * 4, s);

    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    const int32_t* cur = colors_in;
    std::vector<int32_t> tp;
    for (int32_t it = it_begin; it < iters && st == GC_OK; ++it) {
        int32_t* dst = ((it - it_begin) % 2 == 0) ? alt : colors_out;
        a.iteration = it;
        a.old_c = cur;
        a.new_c = dst;
        cudaMemsetAsync(a.cls_cnt, 0, hist_bytes, s);
        cudaMemsetAsync(&a.ctrl->k, 0, sizeof(int32_t), s);
        GC_LAUNCH(KID_BRC_HIST, s, k_brc_hist<<<vgrid, kBlock, 0, s>>>(a));
        GC_LAUNCH(KID_BRC_ORDER, s, k_brc_order<<<grid_go, kBlock, 0, s>>>(a));
        GC_LAUNCH(KID_BRC_SEGMENTS, s, k_brc_segments<<<1, kOrderThreads, 0, s>>>(a));
        GC_LAUNCH(KID_RC_SCATTER, s, k_rc_scatter<true><<<grid_sc, kBlock, sc_dyn, s>>>(a));
        if (tune.recolor_mode == 0) {
            void* args[] = {&a};
            cudaError_t le;
            GC_LAUNCH(KID_RC_RECOLOR, s,
                      le = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_rc_recolor_coop),
                                                       dim3(grid_rc), dim3(kBlock), args, 0, s));
            if (le != cudaSuccess) { st = cuda_status(le); break; }
        } else {
            RcCtrl hc;
            ce = cudaMemcpyAsync(&hc, a.ctrl, sizeof(RcCtrl), cudaMemcpyDeviceToHost, s);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
            if (ce != cudaSuccess) { st = cuda_status(ce); break; }
            tp.resize(static_cast<size_t>(hc.k) * kRcNB + 1);
            ce = cudaMemcpyAsync(tp.data(), a.tile_prefix, tp.size() * 4, cudaMemcpyDeviceToHost, s);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
            if (ce != cudaSuccess) { st = cuda_status(ce); break; }
            for (int32_t p = 0; p < hc.k; ++p) {
                const int32_t t0 = tp[p * kRcNB], t1 = tp[(p + 1) * kRcNB];
                if (t1 <= t0) continue;
                const int g2 = std::min(grid_step, (t1 - t0 + kWarps - 1) / kWarps);
                GC_LAUNCH(KID_RC_STEP, s, k_rc_recolor_step<<<g2, kBlock, 0, s>>>(a, t0, t1));
            }
        }
        cur = dst;
    }
    if (st == GC_OK && cur != colors_out)
        cudaMemcpyAsync(colors_out, cur, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, s);
    cudaEventRecord(e1, s);
    ce = cudaMemcpyAsync(&h, a.ctrl, sizeof(RcCtrl), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess && st == GC_OK) st = cuda_status(ce);
    if (st == GC_OK) st = status_from_err_bits(h.err);
    if (st == GC_OK && max_color_out)
        st = batch_max_colors(g, a.graph_of, colors_out, nullptr, ng, max_color_out, nullptr, s);
    if (stats) {
        stats->iterations = iters - it_begin;
        stats->edges_examined = static_cast<int64_t>(h.edges);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        stats->ms_recolor = ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}

gc_status recolor_batch_range(const Graph& g, const gc_batch_graph* graphs, int32_t ng, int32_t* colors,
                              const int32_t* max_in, int32_t it_begin, int32_t it_end,
                              int32_t* max_color_out, cudaStream_t s) {
    return recolor_batch_impl(g, graphs, ng, colors, true, max_in, colors, max_color_out, nullptr, s,
                              it_begin, it_end);
}

gc_status recolor_batch_device(const Graph& g, const gc_batch_graph* graphs, int32_t ng,
                               const int32_t* colors_in, int32_t* colors_out, int32_t* max_color_out,
                               gc_stats* stats, cudaStream_t s) {
    return recolor_batch_impl(g, graphs, ng, colors_in, false, nullptr, colors_out, max_color_out,
                              stats, s);
}

gc_status color_recolor_batch_device(const Graph& g, const gc_batch_graph* graphs, int32_t ng,
                                     int32_t* colors_out, int32_t* rounds_out, int32_t* max_color_out,
                                     gc_stats* stats, cudaStream_t s) {
    std::vector<int32_t> cmax(std::max(ng, 1));
    gc_stats cs;
    gc_status st = color_batch_device(g, graphs, ng, colors_out, rounds_out, cmax.data(), &cs, s);
    if (st != GC_OK) return st;
    gc_stats rs;
    st = recolor_batch_impl(g, graphs, ng, colors_out, true, cmax.data(), colors_out, max_color_out,
                            &rs, s);
    if (stats) {
        *stats = cs;
        stats->iterations = rs.iterations;
        stats->edges_examined = cs.edges_examined + rs.edges_examined;
        stats->ms_recolor = rs.ms_recolor;
    }
    return st;
}

}  // namespace gc
