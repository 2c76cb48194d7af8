// gc_color.cu -- speculative distance-1 coloring on one GPU.
//
// The rounds of Sec. 2.2 in a data-parallel (Jacobi) form: in round r every
// vertex of the work set W_r chooses a tentative color against the colors
// fixed before the round (First Fit, Alg. 1 / Sec. 2.1, or Random-X Fit,
// Sec. 3.2); then every vertex of W_r compares its tentative color with its
// neighbors' and loses if one of them has the same color and a larger
// (priority, id) -- the random total order of Sec. 2.2.  Winners keep their
// color, losers form W_{r+1}.  The vertex of W_r with the largest (priority,
// id) always wins, so the loop ends within |V| rounds.
//
// Layout in HBM: a color word per vertex holds its tentative color with bit
// 31 set until it is fixed and the color alone afterwards, so one gather tells
// a neighbor's color and whether it is fixed; the priority stands beside it
// or in an array of its own (see color_word).  Two work lists of 16-byte items
// are used as ping-pong buffers, each cut into degree-bucket regions whose
// starts are fixed by the set-up (a loser stays in its bucket, so a region
// never overflows).
//
// No row is read to choose a tentative color: a vertex fixed at color c walks
// its row once and sets bit c - 1 in the mask of each neighbor -- 64 bits for
// a light row (degree + X <= 64: its color is among the first 64), a bitmap
// for a heavy one -- so the choice is the j-th clear bit of the mask.  Each
// row is pushed once in a run instead of being gathered in every round
// (G(10^6, 24) First Fit: 24 M pushes instead of 128 M gathers).  Where
// Random-X Fit has few losers in round 0, these gather its colors instead
// (late_of).  Pushes need a symmetric CSR; the rounds of another one end by
// k_pull_choose.
//
// The conflict test of a light row reads the row a few neighbors at a time and
// ends at the first one it loses to (most vertices of an early round lose to
// one of the first).  A heavy row keeps a list of its neighbors above it in
// the total order that were not fixed at its last look, built from the row
// in round 0; only those can beat it.
//
// All rounds (after such a round 0: the others) run in one cooperative launch
// with a grid barrier between the phases of a round (choice, test, and where there are any the long lists left
// open and the long rows' pushes); a barrier takes about 1.2 us.
//
// What it replaced -- three launches a round in a CUDA graph, every light row
// gathered again for every choice and every test, an 8-byte key per gather, a
// block per row beyond 1024 entries -- spent its time on the launches and
// their gaps (20 us a round where there is little to do), on gathers, and on
// a block waiting through one dependent load after the other for a row that
// then lost at once.  Coloring, set-up included, before -> after: R-MAT 24
// First Fit 87.0 -> 41.2 ms (524 rounds), R-MAT 22 Random-4 Fit 12.1 -> 7.5,
// RMAT-Bad 22 14.6 -> 7.3, R-MAT 20 11.4 -> 7.6, G(10^6, 24) 1.68 -> 1.12, the
// 27-point stencil 128^3 with Random-8 Fit 1.12 -> 0.90, a batch of 512 graphs
// 3.99 -> 3.73, G(10^4, 16) 0.22 -> 0.14 (kernels).
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <type_traits>

#include "gc_internal.h"

namespace gc {

struct SpecCtrl {
    int32_t cnt[2][kNB];    // bucket counts of the work list of parity p (0: heavy rows)
    int32_t init_cnt[kNB];  // round-0 bucket sizes (0: heavy rows)
    int32_t round;
    int32_t active;         // |W| for the coming round
    int32_t max_color;
    int32_t max_deg;
    uint32_t err;
    uint32_t setup_err;     // malformed offsets (written by the set-up only: see k_spec_rounds)
    uint32_t barrier;       // arrivals at the grid barrier
    int32_t mark_cnt;       // row pieces to be pushed (round 0: to be tested) by the whole grid
    int32_t open_cnt;       // list pieces left open
    int32_t open_rows;
    int32_t stuck;          // a round had no winner (see k_pull_choose)
    unsigned long long edges;
    unsigned long long conflicts;
    unsigned long long lose16;  // Random-X: 16 x the entries of the rows expected to lose round 0 (set-up)
    long long heavy_entries;  // list entries over all heavy rows
    long long heavy_words;    // bitmap words over all heavy rows
};

// Heavy rows (degree + X > 64), in the order of their region of the round-0
// list: each one's list (start, length; bit 31: it lost round 0), its
// forbidden bitmap (start, words), which the pushing vertices reach through
// bref, and the queues of row and list pieces.
struct HeavyRows {
    int64_t* h_pbeg;
    int32_t* h_pcnt;
    int32_t* pend;
    uint32_t* hbm;
    uint64_t* bref;      // per heavy vertex: bitmap_ref of its row
    WorkItem* mark;      // row pieces: start, color (round 0: heavy row index), length
    WorkItem* open;      // list pieces: start, index of the open row, length
    WorkItem* open_row;  // open rows: the row's work item
    int32_t* open_done;  // pieces done, counted up from minus their number
    int32_t* open_lost;
    int64_t mark_cap, open_cap, open_rows_cap;
};

constexpr int32_t kPiece = 128;         // entries of a row piece (one warp, 4 per lane)
constexpr int32_t kRound0Piece = 256;   // of a row piece of round 0 (8 per lane)
constexpr int32_t kOpenPiece = 256;     // entries of a list piece (8 per lane)
constexpr uint8_t kBucketFixed = 0xFE;  // bucket byte of a fixed vertex (pushes skip it)

struct SpecArgs {
    Graph g;
    int32_t X;
    uint64_t seed;
    Tuning tune;
    int32_t* color;    // the output
    uint32_t* prio;    // priorities, or (wide) 8-byte words: priority, tentative color | kUnfixed / fixed color
    uint32_t* mlo;     // colors 1..32 and 33..64 of the fixed neighbors (light rows)
    uint32_t* mhi;
    uint8_t* bucket;   // degree bucket per vertex (0: heavy)
    WorkItem* list0;   // work lists (ping-pong), bucket regions, the heavy rows' first
    WorkItem* list1;
    SpecCtrl* ctrl;
    int32_t round_limit;
    int32_t max_rounds;   // rounds of this launch
    float late_share;     // round 0 leaves its marks to k_late_marks below this share of losers (see late_of)
    int32_t chosen;       // the first round's choice has been made (k_pull_choose)
    // batches: graph of every vertex and the graphs' descriptors (nullptr for
    // one graph), and the round in which every vertex kept its color
    const int32_t* graph_of;
    const BatchDesc* desc;
    int32_t* win_round;
    HeavyRows heavy;
    // priority rule: 0 the random order; 1 Largest First (degree first);
    // 2 aRC (rank of the vertex's previous class first, from prio_rank[prio_old[v]])
    int32_t prio_kind;
    const int32_t* prio_rank;
    const int32_t* prio_old;
};

constexpr int32_t kUnfixed = INT32_MIN;
__device__ __forceinline__ int32_t tent_of(int32_t x) { return x & INT32_MAX; }

// A vertex's color word (tentative color | kUnfixed, or the fixed color) and
// priority.  Up to kWideMax vertices they share an 8-byte word, so that the
// test of a light row takes one gather; beyond, the words, the masks and the
// streamed rows would crowd each other out of L2, and the
// color words (the output array) and the priorities are arrays of their own,
// the priorities gathered only where a color matches.  (Coloring with shared /
// separate words: G(3 10^6, 6) First Fit 0.80 / 0.82 ms, G(10^7, 6) 3.8 / 3.4,
// G(10^7, 24) Random-8 Fit 7.4 / 6.0, RMAT-ER 23 First Fit 6.4 / 6.0, R-MAT 22
// First Fit 16.6 / 16.0.)
constexpr int64_t kWideMax = 15 << 18;
template <bool kWide>
__device__ __forceinline__ int32_t* color_word(const SpecArgs& a, int32_t v) {
    return kWide ? reinterpret_cast<int32_t*>(a.prio) + 2 * static_cast<int64_t>(v) + 1 : a.color + v;
}
template <bool kWide>
__device__ __forceinline__ uint32_t prio_word(const SpecArgs& a, int32_t v) {
    return __ldg(a.prio + (kWide ? 2 * static_cast<int64_t>(v) : static_cast<int64_t>(v)));
}

// A vertex-visit key (16 bits, clamped) above the upper half of the random
// priority; equal keys still fall back to the id.
__device__ __forceinline__ uint32_t ordered_prio(int64_t first_key, uint32_t p) {
    const uint32_t k = static_cast<uint32_t>(first_key < 0 ? 0 : first_key > 65535 ? 65535 : first_key);
    return (k << 16) | (p >> 16);
}

// u is above v in the random total order of Sec. 2.2: the larger priority,
// then the larger id.
__device__ __forceinline__ bool above(uint32_t pu, int32_t u, uint32_t pv, int32_t v) {
    return pu > pv || (pu == pv && u > v);
}

// Bitmap words of a heavy row: colors 1 .. 32 * words, at least deg + 64.
__host__ __device__ __forceinline__ int32_t heavy_words(int32_t deg) { return (deg + 64) / 32 + 2; }

// Reference to a heavy row's bitmap: (first word << 24) | words, the words
// clamped to 2^24 - 1 on the pushing and the reading side alike.
constexpr uint32_t kRefWords = (1u << 24) - 1u;
__device__ __forceinline__ uint64_t bitmap_ref(long long first_word, long long words) {
    return (static_cast<uint64_t>(first_word) << 24) |
           static_cast<uint32_t>(words < kRefWords ? words : kRefWords);
}

// Random-X index of v in `round`: the graph's own seed, X and local id.
__device__ __forceinline__ uint32_t draw_index(const SpecArgs& a, int32_t v, int32_t round) {
    if (a.graph_of) {
        const BatchDesc& d = a.desc[a.graph_of[v]];
        if (d.X <= 1) return 0u;
        return scale_index(rxf_word(d.seed, static_cast<int32_t>(v - d.base), round),
                           static_cast<uint32_t>(d.X));
    }
    return scale_index(rxf_word(a.seed, v, round), static_cast<uint32_t>(a.X));
}

// ---------------------------------------------------------------------------
// Set-up: priorities, round-0 tentative colors (nothing is colored yet, so
// the j-th permissible color is j + 1 with no row read), bucket sizes, and
// the heavy rows' region of the round-0 list.  (The light rows of round 0
// are taken in id order and need no list.)
// ---------------------------------------------------------------------------
// Chance that a row of deg entries loses round 0: about Poisson(deg / X)
// neighbors draw its color, and it wins over k of them with chance 1 / (k + 1).
__device__ __forceinline__ float lose_chance(float deg, int32_t X) {
    if (X <= 1) return deg / (deg + 1.0f);
    const float m = deg / static_cast<float>(X);
    return m < 0.01f ? 0.5f * m : 1.0f - (1.0f - expf(-m)) / m;
}

template <bool kWide>
__global__ void __launch_bounds__(kBlock) k_spec_setup(SpecArgs a) {
    __shared__ int32_t s_cnt[kNB];
    if (threadIdx.x < kNB) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kBlock;
    int32_t my_max_deg = 0;
    unsigned long long lose16 = 0;
    for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * kBlock; i0 < a.g.n; i0 += stride) {
        const int64_t i = i0 + threadIdx.x;
        const bool valid = i < a.g.n;
        const int32_t v = static_cast<int32_t>(i);
        int64_t beg = 0;
        int32_t deg = 0, b = kNB;
        if (valid) {
            row_of(a.g, v, beg, deg, &a.ctrl->setup_err);
            my_max_deg = max(my_max_deg, deg);
            int32_t X = a.X, vl = v;
            uint64_t seed = a.seed;
            if (a.graph_of) {
                const BatchDesc& d = a.desc[a.graph_of[v]];
                X = d.X;
                seed = d.seed;
                vl = static_cast<int32_t>(v - d.base);
            }
            b = bucket_of(deg, X, a.tune);
            if (b == 1) b = 0;
            a.bucket[v] = static_cast<uint8_t>(b);
            uint32_t p = prio_of(seed, vl);
            if (a.prio_kind == 1) p = ordered_prio(deg, p);
            else if (a.prio_kind == 2) p = ordered_prio(65535 - static_cast<int64_t>(a.prio_rank[a.prio_old[v]]), p);
            const uint32_t j0 = (a.graph_of || a.X > 1) ? draw_index(a, v, 0) : 0u;
            if (a.late_share > 0.f) lose16 += static_cast<unsigned long long>(16.0f * static_cast<float>(deg) * lose_chance(static_cast<float>(deg), X));
            const int32_t c0 = static_cast<int32_t>(j0 + 1u) | kUnfixed;
            if (kWide) {
                reinterpret_cast<uint2*>(a.prio)[v] = make_uint2(p, static_cast<uint32_t>(c0));
            } else {
                a.prio[v] = p;
                a.color[v] = c0;
            }
            a.mlo[v] = 0u;
            a.mhi[v] = 0u;
        }
        warp_append(b == 0, beg, v, deg, &a.ctrl->init_cnt[0], a.list0, 0);
        for (int q = 2; q < kNB; ++q) {
            const uint32_t m = __ballot_sync(kFull, b == q);
            if (m && lane_id() == 0) atomicAdd(&s_cnt[q], __popc(m));
        }
    }
    warp_max(&a.ctrl->max_deg, my_max_deg);
    warp_add(&a.ctrl->lose16, lose16);
    __syncthreads();
    if (threadIdx.x >= 2 && threadIdx.x < kNB && s_cnt[threadIdx.x])
        atomicAdd(&a.ctrl->init_cnt[threadIdx.x], s_cnt[threadIdx.x]);
}

constexpr int kHeavyThreads = 1024;
constexpr int kHeavyChunk = 8 * kHeavyThreads;  // rows per block of the two set-up kernels

__device__ __forceinline__ void heavy_sizes(const SpecArgs& a, int32_t h, int32_t nh, WorkItem& it,
                                            long long& e, long long& wd) {
    it = WorkItem{0, 0, 0};
    e = 0;
    wd = 0;
    if (h < nh) {
        it = load_item(a.list0 + h);
        e = (static_cast<long long>(it.deg) + 3) & ~3ll;  // 16-byte aligned list starts
        wd = heavy_words(it.deg);
    }
}

// Block sums of the list entries and bitmap words of its chunk of rows.
__global__ void __launch_bounds__(kHeavyThreads) k_heavy_sums(SpecArgs a, int32_t nh, long long* sums) {
    __shared__ long long s_e[kHeavyThreads / 32], s_w[kHeavyThreads / 32];
    const int l = lane_id(), w = threadIdx.x >> 5;
    long long te = 0, tw = 0;
    const int64_t lo = static_cast<int64_t>(blockIdx.x) * kHeavyChunk;
    const int64_t hi = min(static_cast<int64_t>(nh), lo + kHeavyChunk);
    for (int64_t h = lo + threadIdx.x; h < hi; h += kHeavyThreads) {
        WorkItem it;
        long long e, wd;
        heavy_sizes(a, static_cast<int32_t>(h), nh, it, e, wd);
        te += e;
        tw += wd;
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        te += __shfl_xor_sync(kFull, te, d);
        tw += __shfl_xor_sync(kFull, tw, d);
    }
    if (l == 0) {
        s_e[w] = te;
        s_w[w] = tw;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long be = 0, bw = 0;
        for (int k = 0; k < kHeavyThreads / 32; ++k) {
            be += s_e[k];
            bw += s_w[k];
        }
        sums[2 * blockIdx.x] = be;
        sums[2 * blockIdx.x + 1] = bw;
        atomicAdd(reinterpret_cast<unsigned long long*>(&a.ctrl->heavy_entries), static_cast<unsigned long long>(be));
        atomicAdd(reinterpret_cast<unsigned long long*>(&a.ctrl->heavy_words), static_cast<unsigned long long>(bw));
    }
}

// Heavy rows: list and bitmap offsets (exclusive scans over their region of
// the round-0 list), a chunk of rows per block, based at the sums of the
// chunks before it; and the row pieces of round 0.
__global__ void __launch_bounds__(kHeavyThreads) k_heavy_setup(SpecArgs a, int32_t nh, const long long* sums) {
    __shared__ long long s_e[kHeavyThreads / 32], s_w[kHeavyThreads / 32];
    __shared__ long long s_base_e, s_base_w;
    const int l = lane_id(), w = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        long long be = 0, bw = 0;
        for (uint32_t b = 0; b < blockIdx.x; ++b) {
            be += sums[2 * b];
            bw += sums[2 * b + 1];
        }
        s_base_e = be;
        s_base_w = bw;
    }
    __syncthreads();
    const int64_t lo = static_cast<int64_t>(blockIdx.x) * kHeavyChunk;
    const int64_t hi = min(static_cast<int64_t>(nh), lo + kHeavyChunk);
    const HeavyRows& hr = a.heavy;
    for (int64_t h0 = lo; h0 < hi; h0 += kHeavyThreads) {
        const int64_t h = h0 + threadIdx.x;
        WorkItem it;
        long long e, wd;
        heavy_sizes(a, h < hi ? static_cast<int32_t>(h) : nh, nh, it, e, wd);
        const int32_t np = (it.deg + kRound0Piece - 1) / kRound0Piece;
        long long ie = e, iw = wd;  // warp inclusive scans
        int32_t ip = np;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const long long ye = __shfl_up_sync(kFull, ie, d), yw = __shfl_up_sync(kFull, iw, d);
            const int32_t yp = __shfl_up_sync(kFull, ip, d);
            if (l >= d) {
                ie += ye;
                iw += yw;
                ip += yp;
            }
        }
        int32_t pbase = 0;
        if (l == 31 && ip) pbase = atomicAdd(&a.ctrl->mark_cnt, ip);
        pbase = __shfl_sync(kFull, pbase, 31) + ip - np;
        for (int32_t q = 0; q < np && pbase + q < hr.mark_cap; ++q)
            store_item(hr.mark + pbase + q, it.beg + static_cast<int64_t>(q) * kRound0Piece, static_cast<int32_t>(h),
                       min(kRound0Piece, it.deg - q * kRound0Piece));
        if (l == 31) {
            s_e[w] = ie;
            s_w[w] = iw;
        }
        __syncthreads();
        long long be = s_base_e, bw = s_base_w, te = 0, tw = 0;
        for (int k = 0; k < kHeavyThreads / 32; ++k) {
            if (k < w) {
                be += s_e[k];
                bw += s_w[k];
            }
            te += s_e[k];
            tw += s_w[k];
        }
        if (h < hi) {
            hr.h_pbeg[h] = be + ie - e;
            hr.h_pcnt[h] = 0;
            hr.bref[it.v] = bitmap_ref(bw + iw - wd, wd);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            s_base_e += te;
            s_base_w += tw;
        }
        __syncthreads();
    }
}

// Random-X with few losers in round 0 (a large X, a sparse graph): most rows
// would push their whole row for few that still read their masks.  Round 0
// then pushes nothing and ends its launch, the losers gather the colors fixed
// in it from their own rows (k_late_marks), and the rounds go on as ever.
// A gather for each of the losers' entries takes the place of a push for each
// of the winners', so late_share, the share of the entries that the losers are
// expected to hold (the set-up sums it) up to which this is done, is larger the
// more a push costs against a gather: with heavy rows (it looks up the kind of
// the neighbor and its bitmap) and beyond what L2 holds; on light graphs that
// L2 holds a push costs no more.  Coloring with the pushes / without:
// G(10^6, 40) Random-32 Fit (heavy) 1.87 / 1.55 ms, RMAT-Good 23 Random-8 5.8 /
// 4.7, G(10^7, 24) Random-5 7.3 / 6.4, Random-32 7.5 / 3.6; light: the 27-point
// mesh 100^3 Random-32 0.32 / 0.35, G(6 10^6, 24) Random-8 2.6 / 2.8.
// Below kLateMin entries the read-back and launches more cost what is saved
// (200,000 x 12 with 5 % of the rows heavy, Random-32: 0.25 / 0.27 ms), below
// half of it also where most rows are heavy (Random-70: 0.45 / 0.36).
constexpr int64_t kLateMin = 11 << 18;
inline float late_share_limit(int64_t n, int64_t nnz, int64_t heavy_rows) {
    if (nnz < (2 * heavy_rows > n ? kLateMin / 2 : kLateMin)) return 0.f;
    if (n <= kWideMax) return heavy_rows ? 0.7f : 0.f;
    return heavy_rows || n > (int64_t(9) << 20) ? 0.92f : 0.6f;
}
__device__ __forceinline__ bool late_of(const SpecArgs& a) {
    return a.late_share > 0.f &&
           static_cast<float>(a.ctrl->lose16) < a.late_share * 16.0f * static_cast<float>(a.g.nnz);
}

// ---------------------------------------------------------------------------
// The rounds
// ---------------------------------------------------------------------------
// Grid barrier of the cooperative launch: every block adds one arrival and
// polls until all have (bounded: false, and kErrTimeout, once the limit has
// run out; the blocks then all leave by the same limit).
constexpr int32_t kBarrierPolls = 1 << 24;

struct GridBarrier {
    uint32_t target = 0;
    __device__ __forceinline__ bool sync(SpecCtrl* c) {
        __shared__ bool s_ok;
        __syncthreads();
        if (threadIdx.x == 0) {
            target += gridDim.x;
            __threadfence();
            atomicAdd(&c->barrier, 1u);
            bool ok = false;
            for (int32_t i = 0; i < kBarrierPolls && !ok; ++i) {
                uint32_t x;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(&c->barrier) : "memory");
                ok = static_cast<int32_t>(x - target) >= 0;
            }
            if (!ok) atomicOr(&c->err, kErrTimeout);
            __threadfence();
            s_ok = ok;
        }
        __syncthreads();
        return s_ok;
    }
};

// Items of the work lists are rewritten during the launch: no read-only loads.
__device__ __forceinline__ WorkItem load_item_rw(const WorkItem* p) {
    int4 r;
    asm volatile("ld.global.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "l"(p));
    WorkItem w;
    w.beg = (static_cast<int64_t>(static_cast<uint32_t>(r.y)) << 32) | static_cast<uint32_t>(r.x);
    w.v = r.z;
    w.deg = r.w;
    return w;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}

// The same for what a pass reads once (ids, items): first out of L2.  (Light
// forms only: large light graphs run 3 to 6 % faster, R-MAT 24 with Random-8 1 %
// slower.)
__device__ __forceinline__ void cp_async16_stream(void* smem, const void* gmem) {
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(sa), "l"(gmem),
                 "l"(policy_evict_first())
                 : "memory");
}

template <bool kHeavy>
__device__ __forceinline__ void cp_async16_rows(void* smem, const void* gmem) {
    if constexpr (kHeavy) cp_async16(smem, gmem);
    else cp_async16_stream(smem, gmem);
}

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 8, %2;" ::"r"(sa), "l"(gmem),
                 "l"(policy_evict_first())
                 : "memory");
}

constexpr int kHead = 128;              // list entries a warp looks at first, 4 per lane
constexpr int kRefill = 8;             // dead ones among them that are worth replacing
constexpr int32_t kLongList = 1024;     // longer lists are left open to the grid
constexpr int32_t kPushInline = 128;    // longer winners' rows are pushed by the grid

// What a warp keeps in shared memory: the heads of its current and next heavy
// row's lists, or the items and ids of its current and next tile of light
// rows; and the losers it has not yet written to the next list.  kOut of them:
// a counter update by all warps of the grid goes to one word, and pushes wait
// behind it (G(10^7, 6) First Fit with 32: round 0 1.94 ms, 0.86 with no
// update at all); large graphs of light rows trade staged ids for more (G(2 10^7,
// 6) First Fit 8.7 -> 8.1 ms; with heavy rows too, RMAT-Good 24 lost 1 to 2 %).
template <bool kHeavy, bool kWide>
struct __align__(16) WarpRounds {
    static constexpr int kIds = kHeavy || kWide ? 512 : 448;  // per row with 2 lanes: 32, 28
    static constexpr int kOut = kHeavy || kWide ? 64 : 96;
    union {
        int32_t head[2][kHead];
        struct {
            WorkItem item[2][16];
            int32_t ids[2][kIds];
        } light;
    };
    WorkItem out[kOut];
};

// State of a warp over the launch.  Lane b keeps the count of bucket b's work
// list and the start of its region.
template <bool kHeavy, bool kWide>
struct Rounds {
    const SpecArgs& a;
    WarpRounds<kHeavy, kWide>& w;
    int32_t lane_start, lane_cnt;
    int32_t round;
    int32_t par;
    int32_t out_n;         // buffered losers
    int32_t out_at;        // lane 0: their places in the next list, once asked for
    int32_t my_max;
    unsigned long long edges;
    __device__ __forceinline__ int32_t start(int b) const { return __shfl_sync(kFull, lane_start, b); }
    __device__ __forceinline__ int32_t cnt(int b) const { return __shfl_sync(kFull, lane_cnt, b); }
};

template <bool kHeavy, bool kWide>
__device__ __forceinline__ WorkItem* next_list(const Rounds<kHeavy, kWide>& r) { return r.par ? r.a.list0 : r.a.list1; }
template <bool kHeavy, bool kWide>
__device__ __forceinline__ const WorkItem* this_list(const Rounds<kHeavy, kWide>& r) { return r.par ? r.a.list1 : r.a.list0; }

// The buffered losers of bucket b ask for their places in the next list once
// the next 16 may not fit any more, and are written there when these come (the
// answer takes its time).
template <bool kHeavy, bool kWide>
__device__ __forceinline__ bool losers_asked(const Rounds<kHeavy, kWide>& r) { return r.out_n > WarpRounds<kHeavy, kWide>::kOut - 16; }
template <bool kHeavy, bool kWide>
__device__ __forceinline__ void ask_places(Rounds<kHeavy, kWide>& r, int b) {
    if (lane_id() == 0) r.out_at = atomicAdd(&r.a.ctrl->cnt[r.par ^ 1][b], r.out_n);
}
template <bool kHeavy, bool kWide>
__device__ __forceinline__ void write_losers(Rounds<kHeavy, kWide>& r, int b) {
    const int32_t base = __shfl_sync(kFull, r.out_at, 0) + r.start(b);
    for (int32_t i = lane_id(); i < r.out_n; i += 32) {
        const WorkItem x = r.w.out[i];
        store_item(next_list(r) + base + i, x.beg, x.v, x.deg);
    }
    __syncwarp();
    r.out_n = 0;
}
template <bool kHeavy, bool kWide>
__device__ __forceinline__ void flush_losers(Rounds<kHeavy, kWide>& r, int b) {
    if (r.out_n == 0) return;
    if (!losers_asked(r)) ask_places(r, b);
    write_losers(r, b);
}

// The lanes with `want` (16 at most) add their row to the losers of bucket b
// (one bucket at a time is buffered).  The whole warp calls it.
template <bool kHeavy, bool kWide>
__device__ __forceinline__ void add_losers(Rounds<kHeavy, kWide>& r, int b, bool want, int64_t beg, int32_t v, int32_t deg) {
    const uint32_t m = __ballot_sync(kFull, want);
    if (m == 0) return;
    if (losers_asked(r)) write_losers(r, b);
    if (want) r.w.out[r.out_n + __popc(m & ((1u << lane_id()) - 1u))] = WorkItem{beg, v, deg};
    r.out_n += __popc(m);
    __syncwarp();
    if (losers_asked(r)) ask_places(r, b);
}

// A vertex fixed at color c sets its bit in the mask of each neighbor not yet
// fixed, where it stays forbidden for the neighbor's later rounds.  Lanes
// lane0, lane0 + stride, ... take the row's entries.  Without heavy rows the
// bit is set with no look at the neighbor (a fixed one's mask is not read any
// more); with them the bucket byte tells the kind (L2-resident), and a
// bitmap's bit that is there already is not written again.
template <bool kHeavy>
__device__ __forceinline__ void push4(const SpecArgs& a, const int32_t (&u)[4], int32_t c) {
    const uint32_t bit = static_cast<uint32_t>(c - 1);
    const uint32_t mask = 1u << (bit & 31u);
    uint32_t* const light = bit < 32u ? a.mlo : a.mhi;
    if constexpr (!kHeavy) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (u[i] >= 0) atomicOr(light + u[i], mask);
    } else {
        uint32_t b[4];
        uint64_t ref[4];
        uint32_t* w[4];
        uint32_t have[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = u[i] >= 0 ? __ldcg(a.bucket + u[i]) : kBucketFixed;
#pragma unroll
        for (int i = 0; i < 4; ++i) ref[i] = b[i] == 0 ? __ldg(a.heavy.bref + u[i]) : 0ull;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            w[i] = nullptr;
            if (b[i] == 0) {
                if (bit < 32u * static_cast<uint32_t>(ref[i] & kRefWords)) w[i] = a.heavy.hbm + (ref[i] >> 24) + (bit >> 5);
            } else if (b[i] != kBucketFixed && bit < 64u) {
                atomicOr(light + u[i], mask);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) have[i] = w[i] ? __ldcg(w[i]) : mask;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (!(have[i] & mask)) atomicOr(w[i], mask);
    }
}

// A heavy row (or a piece of one), 4 entries per lane at a time.
__device__ __forceinline__ void push_row(const SpecArgs& a, int64_t beg, int32_t deg, int32_t c) {
    for (int32_t k0 = lane_id(); k0 < deg; k0 += 128) {
        int32_t u[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) u[i] = k0 + 32 * i < deg ? load_nbr(a.g, beg + k0 + 32 * i, &a.ctrl->err) : -1;
        push4<true>(a, u, c);
    }
}

// Fixes v at color c (one lane calls it).  A row is examined twice in every
// round that its vertex is in the work set (the method's choice and test;
// the choice of round 0 is counted for all rows by the host).
template <bool kHeavy, bool kWide>
__device__ __forceinline__ void fix_color(Rounds<kHeavy, kWide>& r, int32_t v, int32_t c, int32_t deg) {
    r.a.color[v] = c;
    if (kWide) *color_word<true>(r.a, v) = c;
    if (kHeavy) r.a.bucket[v] = kBucketFixed;
    r.my_max = max(r.my_max, c);
    if (r.a.win_round) r.a.win_round[v] = r.round;
    r.edges += static_cast<unsigned long long>(deg) * (2ull * static_cast<unsigned long long>(r.round) + 1ull);
}

// ---------------------------------------------------------------------------
// Tentative colors of W_r against the masks of the colors fixed before it
// ---------------------------------------------------------------------------
// Colors fixed before the round, for the full-row fallback.
template <bool kWide>
struct SnapshotFetch {
    const SpecArgs& a;
    __device__ __forceinline__ int32_t raw(int32_t u) const { return __ldcg(color_word<kWide>(a, u)); }
    __device__ __forceinline__ int32_t resolve(int32_t, int32_t x) const { return x; }  // negative: not fixed
};

// The j-th clear bit of a bitmap (bit b = color b + 1), one warp; -1: past it.
__device__ __forceinline__ int32_t choose_from_bitmap(const uint32_t* bm, int32_t words, uint32_t j) {
    const int l = lane_id();
    for (int32_t w0 = 0; w0 < words; w0 += 32) {
        const int32_t wi = w0 + l;
        const uint32_t f = wi < words ? ~__ldcg(bm + wi) : 0u;
        const uint32_t cnt_f = static_cast<uint32_t>(__popc(f));
        const uint32_t incl = warp_inclusive_scan(cnt_f);
        const uint32_t total = __shfl_sync(kFull, incl, 31);
        if (j < total) {
            const uint32_t excl = incl - cnt_f;
            const bool mine = j >= excl && j < incl;
            const int owner = __ffs(__ballot_sync(kFull, mine)) - 1;
            int32_t color = 0;
            if (mine) color = 32 * wi + select_bit32(f, j - excl) + 1;
            return __shfl_sync(kFull, color, owner);
        }
        j -= total;
    }
    return -1;
}

// A heavy row's choice (the whole warp): the j-th clear bit of its bitmap.
template <bool kWide>
__device__ __forceinline__ int32_t choose_heavy(Rounds<true, kWide>& r, int32_t v, uint32_t j, uint64_t ref) {
    const SpecArgs& a = r.a;
    int32_t c = choose_from_bitmap(a.heavy.hbm + (ref >> 24), static_cast<int32_t>(ref & kRefWords), j);
    if (c < 0) {  // past the bitmap's free colors (Random-X with a large X): the row in full
        int64_t beg;
        int32_t deg;
        row_of(a.g, v, beg, deg, &a.ctrl->err);
        c = choose_warp<4>(a.g, beg, deg, j, SnapshotFetch<kWide>{a}, reinterpret_cast<uint32_t*>(r.w.head), &a.ctrl->err);
    }
    return c;
}

// A light row takes a thread (its color is among the first 64); a heavy one's
// bitmap is searched.
template <bool kRXF, bool kHeavy, bool kWide>
__device__ __forceinline__ void choose_phase(Rounds<kHeavy, kWide>& r) {
    const SpecArgs& a = r.a;
    const WorkItem* list = this_list(r);
    if constexpr (kHeavy) {
        // Threads of a warp start on a row each: its first words, for First
        // Fit from the word of its last choice on (a row's forbidden colors
        // only grow, so its choice never gets smaller).  The rows whose color
        // lies beyond take the whole warp.  (R-MAT 24's first choices: 300 ->
        // 50 us and less a round.)
        // (Fewer rows than warps take a warp each at once.)
        const uint32_t n = r.cnt(0);
        const uint32_t step = gridDim.x * kBlock;
        if (n <= gridDim.x * kWarps) {
            const uint32_t k = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
            if (k < n) {
                const int32_t v = load_item_rw(list + k).v;
                const int32_t c = choose_heavy<kWide>(r, v, kRXF ? draw_index(a, v, r.round) : 0u, __ldg(a.heavy.bref + v));
                if (lane_id() == 0) *color_word<kWide>(a, v) = c | kUnfixed;
            }
        } else for (uint32_t k0 = blockIdx.x * kBlock + (threadIdx.x & ~31u); k0 < n; k0 += step) {
            const uint32_t k = k0 + lane_id();
            int32_t v = 0, c = -1;
            uint32_t j = 0;
            uint64_t ref = 0;
            if (k < n) {
                v = load_item_rw(list + k).v;
                ref = __ldg(a.heavy.bref + v);
                const int32_t words = static_cast<int32_t>(ref & kRefWords);
                const uint32_t* bm = a.heavy.hbm + (ref >> 24);
                int32_t w = 0;
                if (kRXF) j = draw_index(a, v, r.round);
                else w = (tent_of(__ldcg(color_word<kWide>(a, v))) - 1) >> 5;
                uint32_t left = j;
#pragma unroll
                for (int q = 0; q < 2; ++q, w += 2) {
                    const uint32_t f0 = w < words ? ~__ldcg(bm + w) : 0u;
                    const uint32_t f1 = w + 1 < words ? ~__ldcg(bm + w + 1) : 0u;
                    const uint64_t f = (static_cast<uint64_t>(f1) << 32) | f0;
                    const uint32_t cnt = static_cast<uint32_t>(__popcll(f));
                    if (left < cnt) {
                        c = 32 * w + 1 + (left ? select_bit64(f, left) : __ffsll(static_cast<long long>(f)) - 1);
                        break;
                    }
                    left -= cnt;
                }
            }
            for (uint32_t m = __ballot_sync(kFull, k < n && c < 0); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const int32_t vs = __shfl_sync(kFull, v, src);
                const uint32_t js = __shfl_sync(kFull, j, src);
                const uint64_t rs = __shfl_sync(kFull, ref, src);
                const int32_t cs = choose_heavy<kWide>(r, vs, js, rs);
                if (lane_id() == src) c = cs;
            }
            if (k < n) *color_word<kWide>(a, v) = c | kUnfixed;
        }
    }
    for (int b = 2; b < kNB; ++b) {
        const int32_t n = r.cnt(b);
        const WorkItem* lst = list + r.start(b);
        for (uint32_t k = blockIdx.x * kBlock + threadIdx.x; k < static_cast<uint32_t>(n); k += gridDim.x * kBlock) {
            const int32_t v = load_item_rw(lst + k).v;
            const uint32_t lo = ~__ldcg(a.mlo + v);
            int32_t c;
            if (kRXF) {
                const uint64_t f = (static_cast<uint64_t>(~__ldcg(a.mhi + v)) << 32) | lo;
                c = select_bit64(f, draw_index(a, v, r.round)) + 1;
            } else {
                c = lo ? __ffs(lo) : 32 + __ffs(~__ldcg(a.mhi + v));
            }
            *color_word<kWide>(a, v) = c | kUnfixed;
        }
    }
}

// ---------------------------------------------------------------------------
// Conflict test of the light rows, G lanes each
// ---------------------------------------------------------------------------
// Of 4 ids, the first of them k places into the row, the row's own; a bad
// one is flagged and dropped (-1).
__device__ __forceinline__ void in_row(const Graph& g, int32_t k, int32_t deg, int32_t (&u)[4], uint32_t* err) {
    bool bad = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool mine = static_cast<uint32_t>(k + i) < static_cast<uint32_t>(deg);
        const bool fits = static_cast<uint32_t>(u[i]) < static_cast<uint32_t>(g.n);
        bad |= mine && !fits;
        if (!mine || !fits) u[i] = -1;
    }
    if (bad) atomicOr(err, kErrBadGraph);
}

// The 4 ids of piece c of a row (aligned 16-byte pieces, or single reads), -1
// where the row has none.
__device__ __forceinline__ void row_piece(const Graph& g, int64_t beg, int32_t deg, int32_t c, int32_t (&u)[4],
                                          uint32_t* err) {
    const int32_t k = 4 * c - (g.vec ? static_cast<int32_t>(beg & 3) : 0);
    const int64_t e0 = beg + k, end = beg + deg;
    if (g.vec && e0 + 4 <= g.nnz) {
        const int4 q = ld_stream4(g.idx + e0);
        u[0] = q.x;
        u[1] = q.y;
        u[2] = q.z;
        u[3] = q.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) u[i] = e0 + i < end ? ld_stream(g.idx + e0 + i) : -1;
    }
    in_row(g, k, deg, u, err);
}
__device__ __forceinline__ int32_t row_pieces(const Graph& g, int64_t beg, int32_t deg) {
    return ((g.vec ? static_cast<int32_t>(beg & 3) : 0) + deg + 3) >> 2;
}

// Does one of the 4 neighbors u have v's tentative color tv and stand above
// v?  With `all` every neighbor's color matches (First Fit's round 0).
// Bit i of `live`: u[i] is not fixed yet.
template <bool kWide>
__device__ __forceinline__ bool beaten(const SpecArgs& a, const int32_t (&u)[4], int32_t v, int32_t tv, bool all,
                                       uint32_t& live) {
    bool lose = false;
    live = 0;
    if constexpr (kWide) {
        const uint2* key = reinterpret_cast<const uint2*>(a.prio);
        uint2 x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = u[i] >= 0 ? key[u[i]] : make_uint2(0u, 0u);
        const uint32_t pv = prio_word<true>(a, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            lose |= u[i] >= 0 && (all || tent_of(static_cast<int32_t>(x[i].y)) == tv) && above(x[i].x, u[i], pv, v);
            live |= (x[i].y >> 31) << i;
        }
    } else {
        bool match[4];
        if (all) {
#pragma unroll
            for (int i = 0; i < 4; ++i) match[i] = u[i] >= 0;
            live = 15u;
        } else {
            int32_t x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = u[i] >= 0 ? a.color[u[i]] : 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                match[i] = u[i] >= 0 && tent_of(x[i]) == tv;
                live |= (static_cast<uint32_t>(x[i]) >> 31) << i;
            }
        }
        uint32_t p[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i] = match[i] ? prio_word<false>(a, u[i]) : 0u;
        if (match[0] || match[1] || match[2] || match[3]) {
            const uint32_t pv = prio_word<false>(a, v);
#pragma unroll
            for (int i = 0; i < 4; ++i) lose |= match[i] && above(p[i], u[i], pv, v);
        }
    }
    return lose;
}

// The lanes with `want` add their light row to the losers (of bucket b;
// round 0: of its own).
template <bool kRound0, bool kHeavy, bool kWide>
__device__ __forceinline__ void light_losers(Rounds<kHeavy, kWide>& r, int b, bool want, const WorkItem& it) {
    if (!kRound0) {
        add_losers(r, b, want, it.beg, it.v, it.deg);
        return;
    }
    const int own = bucket_of(it.deg, 1, r.a.tune);  // (a light row's bucket does not depend on X)
    add_losers(r, kNB - 1, want && own == kNB - 1, it.beg, it.v, it.deg);
    for (int q = 2; q < kNB - 1; ++q)
        warp_append(want && own == q, it.beg, it.v, it.deg, &r.a.ctrl->cnt[1][q], r.a.list1, r.start(q));
}

// The light rows of bucket b, or (round 0) all of them in id order, where
// consecutive rows are consecutive in the adjacency: a warp takes 32 / G rows
// at a time.  A row's group tests one piece per lane first (most rows of an
// early round lose to one of the first neighbors), then two at a time, until
// it has found a neighbor that the row loses to.  The items (round 0: offsets
// and buckets) of the tile after the next and the ids of the next are on
// their way to shared memory meanwhile.  Round 0 looks at every id, for the
// checks of the adjacency; colors and priorities are gathered until the row
// has lost.
template <int G, bool kRXF, bool kHeavy, bool kWide, bool kRound0>
__device__ __forceinline__ void light_rows(Rounds<kHeavy, kWide>& r, int b) {
    const SpecArgs& a = r.a;
    constexpr int R = 32 / G;
    constexpr int kRow = WarpRounds<kHeavy, kWide>::kIds / R;  // ids of a row in the stage
    static_assert(R <= 16 && kRow % 4 == 0, "16-byte rows");
    const int l = lane_id(), gi = l / G, gl = l % G;
    const int32_t cnt = kRound0 ? a.g.n : r.cnt(b);
    const int32_t tiles = cnt / R + (cnt % R != 0);
    const int32_t W = gridDim.x * kWarps;
    int32_t t = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (t >= tiles) return;
    const WorkItem* lst = kRound0 ? nullptr : this_list(r) + r.start(b);
    const bool late = kRXF && kRound0 && late_of(a);
    auto& st = r.w.light;
    auto stage_items = [&](int32_t tt, int slot) {
        if (kRound0) {  // the R + 1 offsets
            int64_t* off = reinterpret_cast<int64_t*>(st.item[slot]);
            if (l <= min(R, cnt - tt * R)) cp_async8(off + l, a.g.off + tt * R + l);
        } else if (l < min(R, cnt - tt * R)) {
            cp_async16_rows<kHeavy>(&st.item[slot][l], lst + tt * R + l);
        }
    };
    auto item = [&](int32_t tt, int slot) {
        WorkItem it{0, 0, 0};
        if (gi < cnt - tt * R) {
            if (kRound0) {
                const int64_t* off = reinterpret_cast<const int64_t*>(st.item[slot]);
                const int64_t len = off[gi + 1] - off[gi];  // checked by the set-up
                if (len < 64) it = WorkItem{off[gi], tt * R + gi, static_cast<int32_t>(len)};
            } else {
                it = st.item[slot][gi];
            }
        }
        return it;
    };
    // Round 0: the rows of a tile are consecutive in the adjacency, and are
    // staged as one run where that fits (else, and later, a part for each row:
    // most rows of a skewed graph are short, and the few longer than their
    // part were read id by id).  First place of the run, -1: it does not fit.
    auto run_of = [&](int32_t tt, int slot, int64_t& end) -> int64_t {
        if (!kRound0) return -1;
        const int64_t* off = reinterpret_cast<const int64_t*>(st.item[slot]);
        const int64_t base = off[0] & ~static_cast<int64_t>(3);
        end = off[min(R, cnt - tt * R)];
        return end - base <= WarpRounds<kHeavy, kWide>::kIds ? base : -1;
    };
    auto stage_ids = [&](int32_t tt, int slot) {
        if (!a.g.vec) return;
        int64_t end = 0;
        const int64_t base = run_of(tt, slot, end);
        if (kRound0 && base >= 0) {
            for (int64_t e = base + 4 * l; e < end; e += 128)
                if (e + 4 <= a.g.nnz) cp_async16_rows<kHeavy>(&st.ids[slot][e - base], a.g.idx + e);
            return;
        }
        const WorkItem it = item(tt, slot);
        const int32_t np = min(row_pieces(a.g, it.beg, it.deg), kRow / 4);
        for (int32_t c = gl; c < np; c += G) {
            const int64_t e = (it.beg & ~static_cast<int64_t>(3)) + 4 * static_cast<int64_t>(c);
            if (e + 4 <= a.g.nnz) cp_async16_rows<kHeavy>(&st.ids[slot][gi * kRow + 4 * c], a.g.idx + e);
        }
    };
    stage_items(t, 0);
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
    stage_ids(t, 0);
    if (tiles - t > W) stage_items(t + W, 1);
    cp_async_commit();
    int next_bucket = b;
    if (kRound0 && kHeavy) next_bucket = gi < cnt - t * R ? a.bucket[t * R + gi] : 0;
    for (int slot = 0;; slot ^= 1) {
        const int bucket = next_bucket;
        if (kRound0 && kHeavy && tiles - t > W) next_bucket = gi < cnt - (t + W) * R ? a.bucket[(t + W) * R + gi] : 0;
        cp_async_wait<0>();
        __syncwarp();
        const WorkItem it = item(t, slot);
        const int32_t shift = static_cast<int32_t>(it.beg & 3);
        int64_t run_end = 0;
        const int64_t run = run_of(t, slot, run_end);
        // where the row's pieces are staged, and how many of them
        const int32_t at0 = run >= 0 ? static_cast<int32_t>(it.beg - shift - run) : gi * kRow;
        const int32_t staged = a.g.vec ? static_cast<int32_t>(min(static_cast<int64_t>(run >= 0 ? INT32_MAX : kRow / 4),
                                                                  (a.g.nnz - it.beg + shift) >> 2)) : 0;
        __syncwarp();  // the slot's items are read: the ones after the next tile's may land there
        const bool valid = gi < cnt - t * R && (!kRound0 || !kHeavy || bucket != 0);
        const int32_t left = tiles - t;
        if (left > W) {
            stage_ids(t + W, slot ^ 1);
            if (left - W > W) stage_items(t + 2 * W, slot);
        }
        cp_async_commit();

        auto piece = [&](int32_t c, int32_t (&u)[4]) {
            if (c < staged) {
                const int4 q = *reinterpret_cast<const int4*>(&st.ids[slot][at0 + 4 * c]);
                u[0] = q.x;
                u[1] = q.y;
                u[2] = q.z;
                u[3] = q.w;
                in_row(a.g, 4 * c - shift, it.deg, u, &a.ctrl->err);
            } else {
                row_piece(a.g, it.beg, it.deg, c, u, &a.ctrl->err);
            }
        };
        const bool all = kRound0 && !kRXF;
        const int32_t tv = !valid ? 0 : all ? 1 : tent_of(*color_word<kWide>(a, it.v));
        const int32_t np = valid ? row_pieces(a.g, it.beg, it.deg) : 0;
        bool lost = false, loop = false;
        uint64_t live = 0;  // of this lane's first 16 pieces, 4 bits each: neighbors not fixed yet
        int at = 0;
        // A tile of short rows takes the up to two pieces per lane at once
        // (7-point mesh of 1 M vertices: 180 -> 161 us of rounds), others a piece first: taking both
        // there cost a batch of 512 graphs 3 %, half a piece G(10^6, 24) 4 %.
        bool two = __all_sync(kFull, np <= 2 * G);
        for (int32_t c0 = 0;; c0 += two ? 2 * G : G, two = true) {
            const bool on = c0 < np && (kRound0 || !lost);
            if (!__any_sync(kFull, on)) break;
            int32_t u[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int i = 0; i < 4; ++i) u[q][i] = -1;
                const int32_t c = c0 + q * G + gl;
                if (on && c < np && (q == 0 || two)) piece(c, u[q]);
                if (kRound0) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (u[q][i] == it.v && valid) {  // uncolorable (Sec. 1): reported as a malformed graph
                            loop = true;
                            u[q][i] = -1;
                        }
                        if (lost) u[q][i] = -1;
                    }
                }
            }
            uint32_t lv;
            bool lose = beaten<kWide>(a, u[0], it.v, tv, all, lv);
            live |= static_cast<uint64_t>(lv) << at;
            at += 4;
            if (two) {
                lose |= beaten<kWide>(a, u[1], it.v, tv, all, lv);
                live |= static_cast<uint64_t>(lv) << at;
                at += 4;
            }
            lost |= group_any<G>(lose);
        }
        if (kRound0 && loop) atomicOr(&a.ctrl->err, kErrBadGraph);
        light_losers<kRound0>(r, b, valid && lost && gl == 0, it);
        if (valid && !lost) {
            if (gl == 0) fix_color<kHeavy, kWide>(r, it.v, tv, it.deg);
            for (int32_t c = gl, q = 0; c < np && !late; c += G, ++q) {
                int32_t u[4];
                piece(c, u);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (q < 16 && !(live >> (4 * q + i) & 1u)) u[i] = -1;
                push4<kHeavy>(a, u, tv);
            }
        }
        if (left <= W) break;
        t += W;
    }
    cp_async_wait<0>();
    __syncwarp();
    flush_losers(r, kRound0 ? kNB - 1 : b);
}

// ---------------------------------------------------------------------------
// Conflict test of the heavy rows, a warp each
// ---------------------------------------------------------------------------
// ListItem: the work item of a heavy row holds its list, not its row: beg =
// the list's start in pend, deg = its length.

// A heavy winner (the whole warp): fixed, and its row pushed or queued for
// the whole grid.
template <bool kWide>
__device__ __forceinline__ void heavy_win(Rounds<true, kWide>& r, int32_t v, int32_t c, int64_t beg, int32_t deg) {
    const SpecArgs& a = r.a;
    const int l = lane_id();
    if (l == 0) fix_color<true, kWide>(r, v, c, deg);
    if (deg <= kPushInline) {
        push_row(a, beg, deg, c);
        return;
    }
    const int32_t np = (deg + kPiece - 1) / kPiece;
    int32_t pos = 0;
    if (l == 0) pos = atomicAdd(&a.ctrl->mark_cnt, np);
    pos = __shfl_sync(kFull, pos, 0);
    for (int32_t q = l; q < np && pos + q < a.heavy.mark_cap; q += 32)  // (the capacity holds every piece of every row)
        store_item(a.heavy.mark + pos + q, beg + static_cast<int64_t>(q) * kPiece, c, min(kPiece, deg - q * kPiece));
}

// The lanes with `want` queue the pieces of their row for the whole grid.
__device__ __forceinline__ void queue_losers(const SpecArgs& a, bool want, const WorkItem& it) {
    const int l = lane_id();
    const uint32_t np = want ? (static_cast<uint32_t>(it.deg) + kPiece - 1) / kPiece : 0u;
    const uint32_t incl = warp_inclusive_scan(np);
    int32_t base = 0;
    if (l == 31 && incl) base = atomicAdd(&a.ctrl->mark_cnt, static_cast<int32_t>(incl));
    base = __shfl_sync(kFull, base, 31) + static_cast<int32_t>(incl - np);
    for (uint32_t m = __ballot_sync(kFull, np != 0); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const int64_t beg = __shfl_sync(kFull, it.beg, src);
        const int32_t deg = __shfl_sync(kFull, it.deg, src), v = __shfl_sync(kFull, it.v, src);
        const int32_t pos = __shfl_sync(kFull, base, src), n = static_cast<int32_t>(__shfl_sync(kFull, np, src));
        for (int32_t q = l; q < n && pos + q < a.heavy.mark_cap; q += 32)  // (the capacity holds every piece of every row)
            store_item(a.heavy.mark + pos + q, beg + static_cast<int64_t>(q) * kPiece, v, min(kPiece, deg - q * kPiece));
    }
}

// Round 0, a piece of a heavy row (the whole warp): its share of the test,
// and the row's list -- the neighbors above it in the total order, the only
// ones that can beat it in a later round (their order is free, so the pieces
// of a row just take places; a row of one piece needs none).  Bound by the
// latency of its dependent reads: a shared word gives priority and color at
// once (separate ones: the color of those above only; with all R-MAT 24
// Random-8 Fit took 24.6 ms, 22.8 without).  Random-70 Fit, round 0, with the
// places of all rows counted and the words read one after the other / now:
// G(20,000, 1500) 234 / 198 us, G(2 10^6, 60) 1.45 / 1.23 ms, G(3 10^7, 6) 20.4 /
// 16.8.
template <bool kRXF, bool kWide>
__device__ __forceinline__ void heavy_round0_piece(Rounds<true, kWide>& r, const WorkItem& it) {
    const SpecArgs& a = r.a;
    const int l = lane_id();
    const int32_t h = it.v;
    const WorkItem row = load_item_rw(a.list0 + h);
    int32_t* dst = a.heavy.pend + __ldg(a.heavy.h_pbeg + h);
    int32_t u[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int32_t k = 32 * i + l;
        u[i] = k < it.deg ? load_nbr(a.g, it.beg + k, &a.ctrl->err) : -1;
    }
    uint32_t p[8];
    int32_t x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        p[i] = 0u;
        x[i] = 0;
        if (u[i] < 0) continue;
        if (kRXF && kWide) {
            const uint2 w = reinterpret_cast<const uint2*>(a.prio)[u[i]];
            p[i] = w.x;
            x[i] = static_cast<int32_t>(w.y);
        } else {
            p[i] = prio_word<kWide>(a, u[i]);
        }
    }
    const uint32_t pv = prio_word<kWide>(a, row.v);
    const int32_t tv = kRXF ? tent_of(*color_word<kWide>(a, row.v)) : 1;
    bool lose = false, loop = false;
    uint32_t keep[8];
    int32_t total = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        loop |= u[i] == row.v;
        const bool up = u[i] >= 0 && u[i] != row.v && above(p[i], u[i], pv, row.v);
        if (kRXF && !kWide && up) x[i] = *color_word<kWide>(a, u[i]);
        lose |= up && (!kRXF || tent_of(x[i]) == tv);
        keep[i] = __ballot_sync(kFull, up);
        total += __popc(keep[i]);
    }
    const bool single = row.deg <= kRound0Piece;
    int32_t pos = 0;
    if (!single) {
        if (l == 0 && total) pos = atomicAdd(a.heavy.h_pcnt + h, total) & INT32_MAX;
        pos = __shfl_sync(kFull, pos, 0);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (keep[i] >> l & 1u) dst[pos + __popc(keep[i] & ((1u << l) - 1u))] = u[i];
        pos += __popc(keep[i]);
    }
    if (loop) atomicOr(&a.ctrl->err, kErrBadGraph);
    lose = __any_sync(kFull, lose);
    if (l == 0) {
        if (single) a.heavy.h_pcnt[h] = total | (lose ? INT32_MIN : 0);
        else if (lose) atomicOr(a.heavy.h_pcnt + h, INT32_MIN);
    }
}

// Round 0, once every piece is done: winners and losers (32 rows per warp).
template <bool kRXF, bool kWide>
__device__ __forceinline__ void heavy_round0_close(Rounds<true, kWide>& r) {
    const SpecArgs& a = r.a;
    const int l = lane_id();
    const int32_t nh = a.ctrl->init_cnt[0];
    const int64_t step = static_cast<int64_t>(gridDim.x) * kBlock;
    const bool late = kRXF && late_of(a);
    for (int64_t h0 = (static_cast<int64_t>(blockIdx.x) * kWarps + (threadIdx.x >> 5)) * 32; h0 < nh; h0 += step) {
        const int64_t h = h0 + l;
        WorkItem it{0, 0, 0};
        int32_t pc = 0, c = 0;
        int64_t pb = 0;
        if (h < nh) {
            it = load_item_rw(a.list0 + h);
            pc = __ldcg(a.heavy.h_pcnt + h);
            pb = __ldg(a.heavy.h_pbeg + h);
            c = tent_of(*color_word<kWide>(a, it.v));
        }
        const bool lost = h < nh && pc < 0, won = h < nh && pc >= 0;
        warp_append(lost, pb, it.v, pc & INT32_MAX, &a.ctrl->cnt[1][0], a.list1, 0);
        if (late) {
            if (won) fix_color<true>(r, it.v, c, it.deg);
            queue_losers(a, lost, it);
            continue;
        }
        for (uint32_t m = __ballot_sync(kFull, won); m; m &= m - 1) {
            const int src = __ffs(m) - 1;
            heavy_win(r, __shfl_sync(kFull, it.v, src), __shfl_sync(kFull, c, src), __shfl_sync(kFull, it.beg, src),
                      __shfl_sync(kFull, it.deg, src));
        }
    }
}

// Is one of the list entries [k0, k0 + 256) of the lane's tentative color tv?
// (An entry was above v and unfixed at the last look; one fixed before the
// round never matches, the color was chosen against it.)
template <bool kWide>
__device__ __forceinline__ bool list_hit(const SpecArgs& a, const int32_t* lst, int32_t k0, int32_t len, int32_t tv) {
    int32_t u[8], x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int32_t k = k0 + 32 * i + lane_id();
        u[i] = k < len ? __ldcg(lst + k) : -1;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = u[i] >= 0 ? *color_word<kWide>(a, u[i]) : 0;
    bool hit = false;
#pragma unroll
    for (int i = 0; i < 8; ++i) hit |= tent_of(x[i]) == tv;  // tv >= 1
    return hit;
}

// A long list none of whose first entries beat its row is left to the whole
// grid, in pieces.
template <bool kWide>
__device__ __forceinline__ void leave_open(const Rounds<true, kWide>& r, const WorkItem& it) {
    const SpecArgs& a = r.a;
    const int l = lane_id();
    const int32_t np = (it.deg + kOpenPiece - 1) / kOpenPiece;
    int32_t slot = 0, pos = 0;
    if (l == 0) {
        slot = atomicAdd(&a.ctrl->open_rows, 1);
        pos = atomicAdd(&a.ctrl->open_cnt, np);
        store_item(a.heavy.open_row + slot, it.beg, it.v, it.deg);
        a.heavy.open_done[slot] = -np;
        a.heavy.open_lost[slot] = 0;
    }
    slot = __shfl_sync(kFull, slot, 0);
    pos = __shfl_sync(kFull, pos, 0);
    for (int32_t q = l; q < np; q += 32)
        store_item(a.heavy.open + pos + q, it.beg + static_cast<int64_t>(q) * kOpenPiece, slot,
                   min(kOpenPiece, it.deg - q * kOpenPiece));
}

template <int N>
using Int = std::integral_constant<int, N>;

// Rounds from 1 on.  The first 32 entries of a list come first, then the rest
// of the first kHead (both at once where there are fewer rows than warps, and
// a row waits for its latency only): most rows of a dense core lose in every
// round (98 % of the visits to R-MAT 24's rows beyond 1024 entries), nearly
// always to one of the first 32 (R-MAT 24, all rounds, with the choice
// above: 50.5 -> 40.5 ms).  The items and the heads of a warp's next rows are on their
// way while it tests one.  A list seen in full is compacted in place; on a
// longer one the entries seen that were fixed since are replaced by the
// list's last ones once there are kRefill, so that the head stays alive and
// the list shrinks without a pass over it (it stays a superset of the
// neighbors above v not fixed; its order is free).
template <bool kWide>
__device__ __forceinline__ void heavy_rows(Rounds<true, kWide>& r) {
    const SpecArgs& a = r.a;
    const WorkItem* list = this_list(r);
    const int l = lane_id();
    const int32_t n = r.cnt(0);
    const int32_t W = gridDim.x * kWarps;
    int32_t k = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (k >= n) return;
    auto stage = [&](const WorkItem& it, int slot) {
        if (4 * l < it.deg) cp_async16(&r.w.head[slot][4 * l], a.heavy.pend + it.beg + 4 * l);
    };
    const bool many = n > W;
    WorkItem it = load_item_rw(list + k), nx{0, 0, 0};
    if (k + W < n) nx = load_item_rw(list + k + W);
    stage(it, 0);
    cp_async_commit();
    for (int slot = 0;; slot ^= 1) {
        int looked = 0;
        cp_async_wait<0>();
        __syncwarp();
        const bool more = n - k > W;
        if (more) stage(nx, slot ^ 1);
        cp_async_commit();
        WorkItem after{0, 0, 0};
        if (more && n - k - W > W) after = load_item_rw(list + k + 2 * W);

        const int32_t pc = it.deg;
        int32_t* lst = a.heavy.pend + it.beg;
        const int32_t* head = r.w.head[slot];
        const int32_t tv = tent_of(*color_word<kWide>(a, it.v));
        int32_t u[4] = {0, 0, 0, 0}, x[4] = {kUnfixed, kUnfixed, kUnfixed, kUnfixed};
        uint32_t dead[4] = {0, 0, 0, 0};
        int32_t nd = 0;
        bool lost = false;
        auto look = [&](auto from, auto to) {  // at entries [32 from, 32 to)
            bool mine = false;
#pragma unroll
            for (int i = from; i < to; ++i)
                if (32 * i + l < pc) {
                    u[i] = head[32 * i + l];
                    x[i] = *color_word<kWide>(a, u[i]);
                }
#pragma unroll
            for (int i = from; i < to; ++i) {
                mine |= tent_of(x[i]) == tv;
                dead[i] = __ballot_sync(kFull, x[i] >= 0);
                nd += __popc(dead[i]);
            }
            lost = __any_sync(kFull, mine);
            looked = to;
        };
        if (many) {
            look(Int<0>{}, Int<1>{});
            if (!lost && pc > 32) look(Int<1>{}, Int<4>{});
        } else {
            look(Int<0>{}, Int<4>{});
        }
        int32_t len = pc;
        if (pc <= 32 * looked) {  // seen in full: compacted in place
            if (lost && nd) {
                int32_t kept = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t live = __ballot_sync(kFull, i < looked && 32 * i + l < pc && x[i] < 0);
                    if (live >> l & 1u) lst[kept + __popc(live & ((1u << l) - 1u))] = u[i];
                    kept += __popc(live);
                }
                len = kept;
            }
        } else if (nd >= kRefill) {  // the dead ones seen make room for the list's last entries
            const int32_t moved = min(nd, pc - 32 * looked);
            int32_t d = 0;  // rank of the entry among the dead ones
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int32_t rank = d + __popc(dead[i] & ((1u << l) - 1u));
                if ((dead[i] >> l & 1u) && rank < moved) lst[32 * i + l] = __ldcg(lst + pc - 1 - rank);
                d += __popc(dead[i]);
            }
            len = pc - moved;
        }
        bool open = false;
        if (!lost && pc > kHead) {
            // (a refill left the entries it moved in their old places, which are tested here)
            if (pc <= kLongList) {
                for (int32_t k0 = kHead; k0 < pc && !lost; k0 += 256) lost = __any_sync(kFull, list_hit<kWide>(a, lst, k0, pc, tv));
            } else {
                open = true;  // (the shortened list holds every live entry)
                leave_open(r, WorkItem{it.beg, it.v, len});
            }
        }
        add_losers(r, 0, l == 0 && lost, it.beg, it.v, len);
        if (!lost && !open) {
            int64_t beg;
            int32_t deg;
            row_of(a.g, it.v, beg, deg, &a.ctrl->err);
            heavy_win(r, it.v, tv, beg, deg);
        }
        if (!more) break;
        it = nx;
        nx = after;
        k += W;
    }
    flush_losers(r, 0);
}

// The open lists' pieces: the warp that finishes a row's last piece closes
// the row (acquire-release on the row's counter orders the other pieces'
// findings before it).
template <bool kWide>
__device__ __forceinline__ void open_phase(Rounds<true, kWide>& r) {
    const SpecArgs& a = r.a;
    const int l = lane_id();
    const int32_t n = __ldcg(&a.ctrl->open_cnt);
    const int32_t W = gridDim.x * kWarps;
    for (uint32_t k = blockIdx.x * kWarps + (threadIdx.x >> 5); k < static_cast<uint32_t>(n); k += W) {
        const WorkItem it = load_item_rw(a.heavy.open + k);
        const WorkItem row = load_item_rw(a.heavy.open_row + it.v);  // beside the piece's entries
        const int32_t* lst = a.heavy.pend + it.beg;
        int32_t u[8], x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) u[i] = 32 * i + l < it.deg ? __ldcg(lst + 32 * i + l) : -1;
        const int32_t tv = tent_of(*color_word<kWide>(a, row.v));  // and the row beside their colors
        int64_t beg;
        int32_t deg;
        row_of(a.g, row.v, beg, deg, &a.ctrl->err);
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = u[i] >= 0 ? *color_word<kWide>(a, u[i]) : 0;
        bool hit = false;
#pragma unroll
        for (int i = 0; i < 8; ++i) hit |= tent_of(x[i]) == tv;
        if (__any_sync(kFull, hit) && l == 0) atomicExch(a.heavy.open_lost + it.v, 1);
        __syncwarp();
        int last = 0;
        if (l == 0) last = add_acq_rel(a.heavy.open_done + it.v) == -1;
        if (!__shfl_sync(kFull, last, 0)) continue;
        __syncwarp();
        if (__ldcg(a.heavy.open_lost + it.v)) {
            if (l == 0) {
                const int32_t pos = atomicAdd(&a.ctrl->cnt[r.par ^ 1][0], 1);
                store_item(next_list(r) + pos, row.beg, row.v, row.deg);
            }
        } else {
            heavy_win(r, row.v, tv, beg, deg);
        }
    }
}

// The long winners' rows, in pieces.
__device__ __forceinline__ void push_phase(const SpecArgs& a) {
    const int32_t n = static_cast<int32_t>(min(static_cast<int64_t>(__ldcg(&a.ctrl->mark_cnt)), a.heavy.mark_cap));
    const int32_t W = gridDim.x * kWarps;
    for (uint32_t k = blockIdx.x * kWarps + (threadIdx.x >> 5); k < static_cast<uint32_t>(n); k += W) {
        const WorkItem it = load_item_rw(a.heavy.mark + k);
        push_row(a, it.beg, it.deg, it.v);
    }
}

template <bool kRXF, bool kHeavy, bool kWide>
__device__ __forceinline__ void test_phase(Rounds<kHeavy, kWide>& r) {
    const SpecArgs& a = r.a;
    if (r.round == 0) {
        if constexpr (kHeavy) {
            const int32_t np = static_cast<int32_t>(min(static_cast<int64_t>(a.ctrl->mark_cnt), a.heavy.mark_cap));
            const int32_t W = gridDim.x * kWarps;
            uint32_t k = blockIdx.x * kWarps + (threadIdx.x >> 5);
            WorkItem it{0, 0, 0};
            if (k < static_cast<uint32_t>(np)) it = load_item_rw(a.heavy.mark + k);
            for (; k < static_cast<uint32_t>(np); k += W) {
                WorkItem nx{0, 0, 0};
                if (k + W < static_cast<uint32_t>(np)) nx = load_item_rw(a.heavy.mark + k + W);
                heavy_round0_piece<kRXF, kWide>(r, it);
                it = nx;
            }
        }
        light_rows<2, kRXF, kHeavy, kWide, true>(r, 0);
        return;
    }
    if constexpr (kHeavy) heavy_rows<kWide>(r);
    for (int b = 2; b < kNB; ++b) {
        if (r.cnt(b) == 0) continue;
        switch (b) {
        case 2: light_rows<32, kRXF, kHeavy, kWide, false>(r, 2); break;
        case 3: light_rows<16, kRXF, kHeavy, kWide, false>(r, 3); break;
        case 4: light_rows<8, kRXF, kHeavy, kWide, false>(r, 4); break;
        case 5: light_rows<4, kRXF, kHeavy, kWide, false>(r, 5); break;
        default: light_rows<2, kRXF, kHeavy, kWide, false>(r, 6); break;
        }
    }
}

// kHeavy: the graph has heavy rows (the form without them returns at once on
// such a graph, and is launched before the host knows).
//
// The grid barriers need every block, so whether a launch runs is decided on
// words that no launch writes: the set-up's errors and bucket counts.  `err`
// is not among them -- a block of round 0 may have flagged an id in it before
// another has started, and one that left on it would be waited for by the
// others until their polls run out.
template <bool kRXF, bool kHeavy, bool kWide>
__global__ void __launch_bounds__(kBlock, 4) k_spec_rounds(const __grid_constant__ SpecArgs a) {
    __shared__ WarpRounds<kHeavy, kWide> s_w[kWarps];
    static_assert(sizeof(WarpRounds<kHeavy, kWide>::head) >= kWarpBitmapWords * 4, "the full-row fallback's bitmap");
    SpecCtrl* const c = a.ctrl;
    if (c->setup_err || (!kHeavy && c->init_cnt[0] > 0)) return;
    const int warp = threadIdx.x >> 5;
    const int l = lane_id();
    const int32_t mine = l < kNB && l != 1 ? c->init_cnt[l] : 0;
    Rounds<kHeavy, kWide> r{a, s_w[warp],
             static_cast<int32_t>(warp_inclusive_scan(static_cast<uint32_t>(mine))) - mine,
             l < kNB ? c->cnt[c->round & 1][l] : 0, c->round, 0, 0, 0, 0, 0ull};
    GridBarrier bar;
    unsigned long long conflicts = 0;
    int32_t total = 0;
    bool ok = true;
    for (int32_t done = 0; done < a.max_rounds; ++done) {
        r.par = r.round & 1;
        if (r.round > 0) {
            if (done > 0 || !a.chosen) choose_phase<kRXF, kHeavy, kWide>(r);
            if (blockIdx.x == 0 && threadIdx.x < kNB) c->cnt[r.par ^ 1][threadIdx.x] = 0;
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                c->mark_cnt = 0;
                c->open_cnt = 0;
                c->open_rows = 0;
            }
            if (!(ok = bar.sync(c))) break;
        }
        test_phase<kRXF, kHeavy, kWide>(r);
        if (!(ok = bar.sync(c))) break;
        if constexpr (kHeavy) {
            if (r.round == 0) {
                if (blockIdx.x == 0 && threadIdx.x == 0) c->mark_cnt = 0;
                if (!(ok = bar.sync(c))) break;
                heavy_round0_close<kRXF>(r);
                if (!(ok = bar.sync(c))) break;
            }
            if (__ldcg(&c->open_cnt) > 0) {
                open_phase<kWide>(r);
                if (!(ok = bar.sync(c))) break;
            }
            if (!(kRXF && r.round == 0 && late_of(a)) && __ldcg(&c->mark_cnt) > 0) {
                push_phase(a);
                if (!(ok = bar.sync(c))) break;
            }
        }
        const int32_t before = __reduce_add_sync(kFull, r.lane_cnt);  // (0 in round 0)
        r.lane_cnt = l < kNB ? __ldcg(&c->cnt[r.par ^ 1][l]) : 0;
        total = __reduce_add_sync(kFull, r.lane_cnt);
        conflicts += static_cast<unsigned long long>(total);
        ++r.round;
        if (total == 0) break;
        if (total == before) {  // no winner: see k_pull_choose
            if (blockIdx.x == 0 && threadIdx.x == 0) c->stuck = 1;
            break;
        }
        if (kRXF && r.round == 1 && late_of(a)) break;  // k_late_marks comes next
        if (r.round >= a.round_limit) {
            if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&c->err, kErrRoundLimit);
            break;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->round = r.round;
        c->active = total;
        c->conflicts += conflicts;
    }
    warp_add(&c->edges, r.edges);
    warp_max(&c->max_color, r.my_max);
}

// Start of bucket b's region of the work lists.
__device__ __forceinline__ int32_t region_start(const SpecCtrl* c, int b) {
    int32_t s = 0;
    for (int q = 0; q < b; ++q) s += q != 1 ? c->init_cnt[q] : 0;
    return s;
}

// The marks that a late round 0 left out (see late_of): of every light loser
// by 2 or 8 lanes, of the heavy ones by queued pieces.  (A kernel of its own:
// with this code in theirs the rounds ran up to 7 % slower.)
template <int G, bool kWide>
__device__ __forceinline__ void late_light(const SpecArgs& a, const WorkItem* lst, int32_t cnt) {
    constexpr int R = 32 / G;
    const int l = lane_id(), gi = l / G, gl = l % G;
    const uint32_t step = gridDim.x * kWarps * R;
    uint32_t k = (blockIdx.x * kWarps + (threadIdx.x >> 5)) * R + gi;
    WorkItem nx{0, 0, 0};
    if (k < static_cast<uint32_t>(cnt)) nx = load_item(lst + k);
    while (__any_sync(kFull, k < static_cast<uint32_t>(cnt))) {
        const WorkItem it = nx;
        const bool valid = k < static_cast<uint32_t>(cnt);
        k += step;
        nx = WorkItem{0, 0, 0};
        if (k < static_cast<uint32_t>(cnt)) nx = load_item(lst + k);
        const int32_t np = valid ? row_pieces(a.g, it.beg, it.deg) : 0;
        uint32_t lo = 0, hi = 0;
        for (int32_t c0 = gl; c0 < np; c0 += 2 * G) {
            int32_t u[2][4], x[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int i = 0; i < 4; ++i) u[q][i] = -1;
                if (c0 + q * G < np) row_piece(a.g, it.beg, it.deg, c0 + q * G, u[q], &a.ctrl->err);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) x[q][i] = u[q][i] >= 0 ? *color_word<kWide>(a, u[q][i]) : kUnfixed;
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) {  // (a word with kUnfixed set: no bit)
                    lo |= bit_or_none(x[q][i] - 1);
                    hi |= bit_or_none(x[q][i] - 33);
                }
        }
#pragma unroll
        for (int d = G / 2; d >= 1; d >>= 1) {
            lo |= __shfl_xor_sync(kFull, lo, d);
            hi |= __shfl_xor_sync(kFull, hi, d);
        }
        if (valid && gl == 0) {
            a.mlo[it.v] = lo;
            a.mhi[it.v] = hi;
        }
    }
}

template <bool kWide>
__global__ void __launch_bounds__(kBlock) k_late_marks(const __grid_constant__ SpecArgs a) {
    SpecCtrl* const c = a.ctrl;
    if (blockIdx.x == 0 && threadIdx.x == 0) c->barrier = 0;  // of the next launch
    if (c->round != 1 || c->active == 0 || !late_of(a)) return;
    for (int b = 2; b < kNB; ++b) {
        const int32_t n = c->cnt[1][b];
        if (n == 0) continue;
        const WorkItem* lst = a.list1 + region_start(c, b);
        if (b <= 4) late_light<8, kWide>(a, lst, n);
        else late_light<2, kWide>(a, lst, n);
    }
    if (c->init_cnt[0] == 0) return;
    const int32_t n = static_cast<int32_t>(min(static_cast<int64_t>(c->mark_cnt), a.heavy.mark_cap));
    for (uint32_t k = blockIdx.x * kWarps + (threadIdx.x >> 5); k < static_cast<uint32_t>(n); k += gridDim.x * kWarps) {
        const WorkItem it = load_item(a.heavy.mark + k);
        const uint64_t ref = __ldg(a.heavy.bref + it.v);
        int32_t u[4], x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int32_t e = lane_id() + 32 * i;
            u[i] = e < it.deg ? load_nbr(a.g, it.beg + e, &c->err) : -1;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = u[i] >= 0 ? *color_word<kWide>(a, u[i]) : kUnfixed;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t bit = static_cast<uint32_t>(x[i] - 1);
            if (x[i] <= 0 || bit >= 32u * static_cast<uint32_t>(ref & kRefWords)) continue;
            uint32_t* const w = a.heavy.hbm + (ref >> 24) + (bit >> 5);
            if (!(__ldcg(w) >> (bit & 31u) & 1u)) atomicOr(w, 1u << (bit & 31u));
        }
    }
}

// The choice of a whole round from the rows, a warp each.  The row of the
// work set above all others wins a round unless a neighbor fixed before has
// its color, so a round without a winner means that a neighbor did not push
// it: the CSR is not symmetric, or a bad id was dropped.  The launch then
// ends, and the rounds left are run one by one with this choice.
template <bool kWide>
__global__ void __launch_bounds__(kBlock) k_pull_choose(const __grid_constant__ SpecArgs a) {
    __shared__ uint32_t s_bm[kWarps][kWarpBitmapWords];
    SpecCtrl* const c = a.ctrl;
    if (blockIdx.x == 0 && threadIdx.x == 0) c->barrier = 0;  // of the next launch
    const int par = c->round & 1;
    const WorkItem* list = par ? a.list1 : a.list0;
    for (int b = 0; b < kNB; ++b) {
        const uint32_t n = b != 1 ? c->cnt[par][b] : 0;
        const WorkItem* lst = list + region_start(c, b);
        for (uint32_t k = blockIdx.x * kWarps + (threadIdx.x >> 5); k < n; k += gridDim.x * kWarps) {
            const int32_t v = load_item(lst + k).v;
            int64_t beg;
            int32_t deg;
            row_of(a.g, v, beg, deg, &c->err);
            const uint32_t j = a.graph_of || a.X > 1 ? draw_index(a, v, c->round) : 0u;
            const int32_t color = choose_warp<4>(a.g, beg, deg, j, SnapshotFetch<kWide>{a}, s_bm[threadIdx.x >> 5], &c->err);
            if (lane_id() == 0) *color_word<kWide>(a, v) = color | kUnfixed;
        }
    }
}

__global__ void __launch_bounds__(kBlock) k_priorities(uint64_t seed, int64_t n, uint32_t* out) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kBlock;
    for (int64_t v = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x; v < n; v += stride)
        out[v] = prio_of(seed, static_cast<int32_t>(v));
}

gc_status priorities_device(uint64_t seed, int64_t n, uint32_t* out, cudaStream_t s) {
    if (n == 0) return GC_OK;
    const int grid = static_cast<int>(std::min<int64_t>((n + kBlock - 1) / kBlock,
                                                        persistent_grid(current_tuning())));
    GC_LAUNCH(KID_PRIORITIES, s, k_priorities<<<grid, kBlock, 0, s>>>(seed, n, out));
    return cuda_status(cudaStreamSynchronize(s));
}

// ---------------------------------------------------------------------------
// Host driver
// ---------------------------------------------------------------------------
struct PrioRule {
    int32_t kind = 0;
    const int32_t* rank = nullptr;
    const int32_t* old = nullptr;
};

namespace {
template <bool kWide>
const void* rounds_kernel_of(bool rxf, bool heavy) {
    if (rxf) return heavy ? reinterpret_cast<const void*>(k_spec_rounds<true, true, kWide>)
                          : reinterpret_cast<const void*>(k_spec_rounds<true, false, kWide>);
    return heavy ? reinterpret_cast<const void*>(k_spec_rounds<false, true, kWide>)
                 : reinterpret_cast<const void*>(k_spec_rounds<false, false, kWide>);
}

// The rounds: one cooperative launch (spec_graph 1), or one per round; two
// with the marks of round 0 in between where it pushed nothing (late_of).  h
// receives the final control block.  heavy_rows: 0 for the form without them.
gc_status run_rounds(SpecArgs& a, bool rxf, int32_t heavy_rows, SpecCtrl* h, cudaStream_t s) {
    const bool heavy = heavy_rows > 0;
    const bool wide = a.g.n <= kWideMax;
    const void* k = wide ? rounds_kernel_of<true>(rxf, heavy) : rounds_kernel_of<false>(rxf, heavy);
    const auto late = wide ? k_late_marks<true> : k_late_marks<false>;
    const auto pull = wide ? k_pull_choose<true> : k_pull_choose<false>;
    const int fit = sm_count() * occupancy_of(k, kBlock);
    // a block per tile of round 0 at most: on small graphs more blocks would only lengthen the barriers
    const int64_t tiles = heavy ? fit : (static_cast<int64_t>(a.g.n) * 2 + kBlock - 1) / kBlock;
    const int64_t want = a.tune.grid_blocks > 0 ? a.tune.grid_blocks : std::max<int64_t>(1, tiles);
    const int grid = static_cast<int>(std::min<int64_t>(fit, want));
    a.late_share = rxf ? late_share_limit(a.g.n, a.g.nnz, heavy_rows) : 0.f;
    a.max_rounds = a.tune.spec_graph ? INT32_MAX : 1;
    a.chosen = 0;
    const auto launch = [&]() {
        void* args[] = {&a};
        cudaError_t e;
        GC_LAUNCH(KID_SPEC_ROUNDS, s, e = cudaLaunchCooperativeKernel(k, dim3(grid), dim3(kBlock), args, 0, s));
        return e;
    };
    for (;;) {
        cudaError_t e = launch();
        if (e == cudaSuccess) e = cudaMemcpyAsync(h, a.ctrl, sizeof(SpecCtrl), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_status(e);
        if (h->err | h->setup_err) return status_from_err_bits(h->err | h->setup_err);
        if ((!heavy && h->init_cnt[0] > 0) || h->active == 0) return GC_OK;
        if (h->stuck) {
            a.chosen = 1;
            a.max_rounds = 1;
            GC_LAUNCH(KID_SPEC_PULL, s, pull<<<resident_grid(pull, a.tune), kBlock, 0, s>>>(a));
        } else if (a.late_share > 0.f && h->round == 1) {
            GC_LAUNCH(KID_SPEC_LATE, s, late<<<resident_grid(late, a.tune), kBlock, 0, s>>>(a));
        } else {
            e = cudaMemsetAsync(&a.ctrl->barrier, 0, sizeof(uint32_t), s);
            if (e != cudaSuccess) return cuda_status(e);
        }
    }
}
}  // namespace

// The speculative coloring; with graph_of / desc / win_round set, a batch.
static gc_status color_impl(const Graph& g, int32_t X, uint64_t seed, const int32_t* graph_of,
                            const BatchDesc* desc, int32_t* win_round, const PrioRule& rule,
                            int32_t* colors_out, gc_stats* stats, cudaStream_t s, int32_t* max_deg = nullptr) {
    if (max_deg) *max_deg = 0;
    if (g.n == 0) {
        if (stats) { std::memset(stats, 0, sizeof(*stats)); }
        return GC_OK;
    }
    const int64_t n = g.n;
    const bool wide = n <= kWideMax;
    SpecArgs a;
    std::memset(&a, 0, sizeof(a));
    ScratchSet sc;
    sc.want(&a.ctrl, sizeof(SpecCtrl));
    sc.want(&a.prio, n * (wide ? 8 : 4));
    sc.want(&a.mlo, n * 4);
    sc.want(&a.mhi, n * 4);
    sc.want(&a.list0, n * static_cast<int64_t>(sizeof(WorkItem)));
    sc.want(&a.list1, n * static_cast<int64_t>(sizeof(WorkItem)));
    sc.want(&a.bucket, n);
    if (!sc.alloc(s)) return GC_ERR_OOM;
    a.g = g;
    a.X = X;
    a.seed = seed;
    a.tune = current_tuning();
    a.color = colors_out;
    a.graph_of = graph_of;
    a.desc = desc;
    a.win_round = win_round;
    a.prio_kind = rule.kind;
    a.prio_rank = rule.rank;
    a.prio_old = rule.old;
    a.round_limit = static_cast<int32_t>(std::min<int64_t>(n + 2, INT32_MAX));

    struct Events {
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        Events() {
            cudaEventCreate(&e0);
            cudaEventCreate(&e1);
        }
        ~Events() {
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
        }
    } ev;
    cudaEventRecord(ev.e0, s);
    cudaMemsetAsync(a.ctrl, 0, sizeof(SpecCtrl), s);
    a.late_share = X > 1 && g.nnz >= kLateMin / 2 ? 1.f : 0.f;  // (the set-up counts; the rounds take their own limit)
    const auto setup = wide ? k_spec_setup<true> : k_spec_setup<false>;
    const int setup_grid = static_cast<int>(std::min<int64_t>((n + kBlock - 1) / kBlock, resident_grid(setup, a.tune)));
    GC_LAUNCH(KID_SPEC_SETUP, s, setup<<<setup_grid, kBlock, 0, s>>>(a));
    SpecCtrl h{};
    gc_status st = run_rounds(a, X > 1, 0, &h, s);
    ScratchSet sc_heavy, sc_queues;
    if (st == GC_OK && h.init_cnt[0] > 0) {
        // heavy rows: their lists and bitmaps (sizes read back), then the rounds
        const int32_t nh = h.init_cnt[0];
        const int hblocks = static_cast<int>((static_cast<int64_t>(nh) + kHeavyChunk - 1) / kHeavyChunk);
        HeavyRows& hr = a.heavy;
        long long* sums = nullptr;
        sc_heavy.want(&hr.h_pbeg, static_cast<int64_t>(nh) * 8);
        sc_heavy.want(&hr.h_pcnt, static_cast<int64_t>(nh) * 4);
        sc_heavy.want(&hr.bref, n * 8);
        sc_heavy.want(&sums, static_cast<int64_t>(hblocks) * 16);
        if (!sc_heavy.alloc(s)) return GC_ERR_OOM;
        GC_LAUNCH(KID_SPEC_FILL, s, k_heavy_sums<<<hblocks, kHeavyThreads, 0, s>>>(a, nh, sums));
        cudaError_t ce = cudaMemcpyAsync(&h, a.ctrl, sizeof(SpecCtrl), cudaMemcpyDeviceToHost, s);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
        if (ce != cudaSuccess) return cuda_status(ce);
        hr.mark_cap = h.heavy_entries / kPiece + nh;  // every piece of every row
        hr.open_rows_cap = h.heavy_entries / kLongList + 1;
        hr.open_cap = h.heavy_entries / kOpenPiece + hr.open_rows_cap;
        constexpr int64_t kItem = sizeof(WorkItem);
        sc_queues.want(&hr.pend, h.heavy_entries * 4);
        sc_queues.want(&hr.hbm, h.heavy_words * 4);
        sc_queues.want(&hr.mark, hr.mark_cap * kItem);
        sc_queues.want(&hr.open, hr.open_cap * kItem);
        sc_queues.want(&hr.open_row, hr.open_rows_cap * kItem);
        sc_queues.want(&hr.open_done, hr.open_rows_cap * 4);
        sc_queues.want(&hr.open_lost, hr.open_rows_cap * 4);
        if (!sc_queues.alloc(s)) return GC_ERR_OOM;
        ce = cudaMemsetAsync(hr.hbm, 0, static_cast<size_t>(h.heavy_words) * 4, s);
        if (ce != cudaSuccess) return cuda_status(ce);
        GC_LAUNCH(KID_SPEC_FILL, s,
                  k_heavy_setup<<<hblocks, kHeavyThreads, 0, s>>>(a, nh, sums));
        st = run_rounds(a, X > 1, nh, &h, s);
    }
    cudaEventRecord(ev.e1, s);
    if (max_deg) *max_deg = h.max_deg;
    if (stats) {
        std::memset(stats, 0, sizeof(*stats));
        stats->rounds = h.round;
        stats->max_color = h.max_color;
        stats->edges_examined = static_cast<int64_t>(h.edges) + g.nnz;  // round 0's choice: every row once
        stats->conflicts = static_cast<int64_t>(h.conflicts);
        float ms = 0.f;
        cudaEventSynchronize(ev.e1);
        cudaEventElapsedTime(&ms, ev.e0, ev.e1);
        stats->ms_color = ms;
    }
    return st;
}

gc_status color_device(const Graph& g, int32_t X, uint64_t seed, int32_t* colors_out,
                       gc_stats* stats, cudaStream_t s, int32_t* max_deg) {
    return color_impl(g, X, seed, nullptr, nullptr, nullptr, PrioRule{}, colors_out, stats, s, max_deg);
}

gc_status color_lf_device(const Graph& g, int32_t X, uint64_t seed, int32_t* colors_out,
                          gc_stats* stats, cudaStream_t s) {
    PrioRule r;
    r.kind = 1;
    return color_impl(g, X, seed, nullptr, nullptr, nullptr, r, colors_out, stats, s);
}

// aRC (Sec. 3): every iteration colors the graph again by the speculative
// First-Fit rounds, the vertices of earlier classes (in the iteration's
// permutation of the previous coloring's classes) winning their conflicts.
gc_status recolor_async_device(const Graph& g, const int32_t* colors_in, int32_t perm, int32_t iterations,
                               uint64_t seed, int32_t* colors_out, int32_t* ncolors_per_iter,
                               gc_stats* stats, cudaStream_t s) {
    const int64_t n = g.n;
    if (stats) std::memset(stats, 0, sizeof(*stats));
    Scratch sc_old;
    if (!sc_old.alloc(n * 4, s)) return GC_ERR_OOM;
    int32_t* old = sc_old.as<int32_t>();
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    gc_status st = GC_OK;
    int32_t maxc = 0;
    // the input: proper, and its max color (no iteration: copied through)
    st = class_ranks_device(g, colors_in, false, perm, 0, seed, nullptr, &maxc, s);
    if (st == GC_OK && ncolors_per_iter) ncolors_per_iter[0] = n > 0 ? maxc : 0;
    const int32_t* cur = colors_in;
    for (int32_t it = 0; it < iterations && st == GC_OK && n > 0; ++it) {
        cudaError_t ce = cudaMemcpyAsync(old, cur, n * 4, cudaMemcpyDeviceToDevice, s);
        if (ce != cudaSuccess) { st = cuda_status(ce); break; }
        Scratch sc_rank;
        if (!sc_rank.alloc((static_cast<int64_t>(maxc) + 1) * 4, s)) { st = GC_ERR_OOM; break; }
        int32_t m = 0;
        st = class_ranks_device(g, old, true, perm, it, seed, sc_rank.as<int32_t>(), &m, s);
        if (st != GC_OK) break;
        PrioRule r;
        r.kind = 2;
        r.rank = sc_rank.as<int32_t>();
        r.old = old;
        gc_stats cs;
        st = color_impl(g, 1, seed, nullptr, nullptr, nullptr, r, colors_out, &cs, s);
        if (st != GC_OK) break;
        maxc = cs.max_color;
        if (ncolors_per_iter) ncolors_per_iter[it + 1] = maxc;
        if (stats) {
            stats->rounds += cs.rounds;
            stats->edges_examined += cs.edges_examined;
            stats->conflicts += cs.conflicts;
        }
        cur = colors_out;
    }
    if (st == GC_OK && iterations == 0 && n > 0 && colors_out != colors_in) {
        const cudaError_t ce = cudaMemcpyAsync(colors_out, colors_in, n * 4, cudaMemcpyDeviceToDevice, s);
        if (ce != cudaSuccess) st = cuda_status(ce);
    }
    if (st == GC_OK && n == 0 && ncolors_per_iter)
        for (int32_t i = 0; i <= iterations; ++i) ncolors_per_iter[i] = 0;
    cudaEventRecord(e1, s);
    const cudaError_t ce = cudaEventSynchronize(e1);
    if (st == GC_OK && ce != cudaSuccess) st = cuda_status(ce);
    if (stats) {
        stats->iterations = iterations;
        stats->max_color = maxc;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        stats->ms_recolor = ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}

// ---------------------------------------------------------------------------
// Batches
// ---------------------------------------------------------------------------
// Graph of every vertex, by binary search over the graphs' first vertices.
// The graphs of a slice of consecutive vertices lie between those of its
// first and last one, so only these two are searched for among all graphs.
// (With the statistics' read before each atomic: 150 us a call on a batch of
// 512 graphs, 11 M vertices, for 340.)
constexpr int32_t kGraphSlice = 2048;
__global__ void __launch_bounds__(kBlock) k_graph_of(int64_t n, const BatchDesc* desc, int32_t ng,
                                                     int32_t* graph_of) {
    __shared__ int32_t s_range[2];
    const auto search = [&](int64_t v, int lo, int hi) {
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (desc[mid].base <= v) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    for (int64_t c0 = static_cast<int64_t>(blockIdx.x) * kGraphSlice; c0 < n;
         c0 += static_cast<int64_t>(gridDim.x) * kGraphSlice) {
        const int64_t c1 = min(c0 + kGraphSlice, n);
        if (threadIdx.x % 32 == 0 && threadIdx.x < 64) s_range[threadIdx.x / 32] = search(threadIdx.x ? c1 - 1 : c0, 0, ng - 1);
        __syncthreads();
        const int lo = s_range[0], hi = s_range[1];
        for (int64_t v = c0 + threadIdx.x; v < c1; v += kBlock) graph_of[v] = search(v, lo, hi);
        __syncthreads();
    }
}

// Per-graph max of a color array and of the winning rounds (+1); graphs are
// contiguous, so a warp mostly covers one or two of them.
__global__ void __launch_bounds__(kBlock) k_batch_stats(int64_t n, const int32_t* graph_of,
                                                        const int32_t* colors, const int32_t* win_round,
                                                        int32_t* g_maxc, int32_t* g_rounds) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kBlock;
    for (int64_t v = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x; v < n; v += stride) {
        const int32_t gi = graph_of[v];
        int32_t c = colors[v];
        int32_t r = win_round ? win_round[v] + 1 : 0;
        const unsigned act = __activemask();
        const unsigned peers = __match_any_sync(act, gi);
        c = __reduce_max_sync(peers, c);
        r = __reduce_max_sync(peers, r);
        if (lane_id() == __ffs(peers) - 1) {
            // (a read through L1 first: a value no larger than the current
            // one, which is all that a skipped atomic needs)
            if (c > __ldca(&g_maxc[gi])) atomicMax(&g_maxc[gi], c);
            if (g_rounds && r > __ldca(&g_rounds[gi])) atomicMax(&g_rounds[gi], r);
        }
    }
}

gc_status batch_layout(const Graph& g, const gc_batch_graph* graphs, int32_t ng, int32_t* max_x) {
    if (ng < 1 || !graphs) return GC_ERR_INVALID_ARG;
    int64_t next = 0;
    int32_t mx = 1;
    for (int32_t i = 0; i < ng; ++i) {
        const gc_batch_graph& d = graphs[i];
        if (d.vertex_base != next || d.n < 0 || d.X < 1 || d.iterations < 0 || !perm_valid(d.perm))
            return GC_ERR_INVALID_ARG;
        next += d.n;
        mx = std::max(mx, d.X);
    }
    if (next != g.n) return GC_ERR_INVALID_ARG;
    *max_x = mx;
    return GC_OK;
}

gc_status batch_graph_of(const Graph& g, const BatchDesc* d_desc, int32_t ng, int32_t* graph_of,
                         cudaStream_t s) {
    if (g.n == 0) return GC_OK;
    const int grid = static_cast<int>(std::min<int64_t>((static_cast<int64_t>(g.n) + kBlock - 1) / kBlock,
                                                        persistent_grid(current_tuning())));
    GC_LAUNCH(KID_BATCH, s, k_graph_of<<<grid, kBlock, 0, s>>>(g.n, d_desc, ng, graph_of));
    return GC_OK;
}

gc_status batch_max_colors(const Graph& g, const int32_t* graph_of, const int32_t* colors,
                           const int32_t* win_round, int32_t ng, int32_t* max_color_out,
                           int32_t* rounds_out, cudaStream_t s) {
    Scratch sm, sr;
    if (!sm.alloc(ng * 4, s) || !sr.alloc(ng * 4, s)) return GC_ERR_OOM;
    cudaMemsetAsync(sm.p, 0, ng * 4, s);
    cudaMemsetAsync(sr.p, 0, ng * 4, s);
    if (g.n > 0) {
        const int grid = static_cast<int>(std::min<int64_t>((static_cast<int64_t>(g.n) + kBlock - 1) / kBlock,
                                                            persistent_grid(current_tuning())));
        GC_LAUNCH(KID_BATCH, s,
                  k_batch_stats<<<grid, kBlock, 0, s>>>(g.n, graph_of, colors, win_round,
                                                         sm.as<int32_t>(), win_round ? sr.as<int32_t>() : nullptr));
    }
    cudaError_t e = cudaSuccess;
    if (max_color_out) e = cudaMemcpyAsync(max_color_out, sm.p, ng * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && rounds_out)
        e = cudaMemcpyAsync(rounds_out, sr.p, ng * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return cuda_status(e);
}

gc_status color_batch_device(const Graph& g, const gc_batch_graph* graphs, int32_t ng,
                             int32_t* colors_out, int32_t* rounds_out, int32_t* max_color_out,
                             gc_stats* stats, cudaStream_t s) {
    int32_t max_x = 1;
    gc_status st = batch_layout(g, graphs, ng, &max_x);
    if (st != GC_OK) return st;
    static_assert(sizeof(BatchDesc) == sizeof(gc_batch_graph), "descriptor layout");
    Scratch sd, sgo, swr;
    if (!sd.alloc(static_cast<size_t>(ng) * sizeof(BatchDesc), s) || !sgo.alloc(static_cast<int64_t>(g.n) * 4 + 4, s) ||
        !swr.alloc(static_cast<int64_t>(g.n) * 4 + 4, s))
        return GC_ERR_OOM;
    cudaError_t e = cudaMemcpyAsync(sd.p, graphs, static_cast<size_t>(ng) * sizeof(BatchDesc),
                                    cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_status(e);
    const BatchDesc* d_desc = sd.as<BatchDesc>();
    int32_t* graph_of = sgo.as<int32_t>();
    batch_graph_of(g, d_desc, ng, graph_of, s);
    st = color_impl(g, max_x, 0, graph_of, d_desc, swr.as<int32_t>(), PrioRule{}, colors_out, stats, s);
    if (st != GC_OK) return st;
    if (rounds_out || max_color_out)
        st = batch_max_colors(g, graph_of, colors_out, swr.as<int32_t>(), ng, max_color_out, rounds_out, s);
    return st;
}

}  // namespace gc
