// gc_util.cu -- validation of a coloring (the definition of Sec. 1:
// C(u) != C(v) on every edge, #colors = max_u C(u)) and the CSR structure
// check, each one pass over the adjacency.
#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>

#include "gc_internal.h"
#include "gc_steps.h"

namespace gc {

struct ValCtrl {
    unsigned long long conflicts;
    unsigned long long uncolored;
    unsigned long long bad_rank;  // n minus the first bad vertex; 0: none
    int32_t max_color;
    uint32_t err;
    unsigned long long distinct;
    int32_t big_colors;     // vertices with a color >= kPresColors
    int32_t pad;
};

constexpr int kValG = 4;                 // lanes per light row (measured: 8 -> 4 saves 30 us on the stencil)
constexpr int32_t kHeavyDeg = 256;       // heavier rows: one block each (gc_validate_noalloc)
// The blocks of an SM that the pass over the entries is limited for (R-MAT 24 /
// 22 with 3: 1.73 / 0.38 ms, with 4: 2.03 / 0.37, with 5: 2.06 / 0.39).
constexpr int kValBlocks = 3;
constexpr int kPresWords = 2048;         // presence bitmap of colors < 65536
constexpr int32_t kPresColors = kPresWords * 32;

struct ValArgs {
    Graph g;
    const int32_t* colors;
    ValCtrl* c;
    uint32_t* pres;    // kPresWords
    uint8_t* low;      // gc_validate: the low byte of every color
    int32_t* first;    // gc_validate: the row each step of kValChunk begins in
    int64_t steps;     // length of `first`
    int32_t max_allowed;  // a recoloring input: the row of a vertex whose color is outside [1, max_allowed]
                          // is not read; 0: a validation, which reads every row
};

// Count of neighbors with v's color in this lane's stripe.
template <int UC>
__device__ __forceinline__ int32_t same_color(const ValArgs& a, int64_t beg, int32_t deg, int32_t cv,
                                              int32_t lane0, int32_t stride) {
    int32_t cnt = 0;
    for_each_nbr<UC, int32_t, true>(
        a.g, beg, deg, lane0, stride, [&](int32_t u) { return __ldg(a.colors + u); },
        [&](int32_t, int32_t x) { cnt += x == cv; }, &a.c->err);
    return cnt;
}

__device__ __forceinline__ void account(const ValArgs& a, int32_t v, int32_t cv, int32_t same,
                                        uint32_t* s_pres, unsigned long long& conf,
                                        unsigned long long& unc, int32_t& my_max) {
    conf += static_cast<unsigned long long>(same);
    if (cv < 1) ++unc;
    if (cv < 1 || same > 0) atomicMax(&a.c->bad_rank, static_cast<unsigned long long>(a.g.n) - static_cast<unsigned long long>(v));
    my_max = max(my_max, cv);
    if (cv >= 1 && cv < kPresColors) {
        // (a read first: atomics of a warp on one word take turns; R-MAT 24 112 -> 97 us)
        if (!(*reinterpret_cast<volatile uint32_t*>(&s_pres[cv >> 5]) >> (cv & 31) & 1u))
            atomicOr(&s_pres[cv >> 5], 1u << (cv & 31));
    } else if (cv >= kPresColors) {
        atomicAdd(&a.c->big_colors, 1);
    }
}

__device__ __forceinline__ void flush_presence(const ValArgs& a, uint32_t* s_pres) {
    __syncthreads();
    for (int i = threadIdx.x; i < kPresWords; i += kBlock)
        if (s_pres[i]) atomicOr(&a.pres[i], s_pres[i]);
}

// Steps of a row that its own thread writes (more: its warp).  Both ways are a
// few stores; the warp's turns cost where many rows have some (R-MAT 22 with 4,
// 32, 128: 42, 33, 31 us of row pass; a star of 10^7 vertices 187 -> 52 us).
constexpr int32_t kOwnSteps = 128;

// One pass over the vertices: a vertex's own accounting, the low byte of its
// color, and which row each step of the pass over the entries begins in.
// Steps are cut on the count of rows plus entries (row v covers
// [v + off[v], v + 1 + off[v + 1]) of it, less off[0]), so that neither a
// long row nor a long run of empty rows falls to one block (and the step
// starts inside a long row are written by a warp, not by a thread).
__global__ void __launch_bounds__(kBlock) k_validate_rows(ValArgs a) {
    __shared__ uint32_t s_pres[kPresWords];
    for (int i = threadIdx.x; i < kPresWords; i += kBlock) s_pres[i] = 0u;
    __syncthreads();
    int32_t my_max = 0;
    unsigned long long conf = 0, unc = 0;
    const int64_t off0 = __ldg(a.g.off);
    const bool narrow = a.g.n + a.g.nnz < int64_t(1) << 31;
    constexpr int U = 4;  // vertices of a thread whose loads are in flight together
    const int64_t all = static_cast<int64_t>(gridDim.x) * kBlock;
    for (int64_t b0 = static_cast<int64_t>(blockIdx.x) * kBlock; b0 < a.g.n; b0 += U * all) {
        const int64_t b = b0 + threadIdx.x;
        int64_t beg[U];
        int32_t deg[U], cv[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int64_t v = min(b + i * all, static_cast<int64_t>(a.g.n) - 1);
            row_of(a.g, static_cast<int32_t>(v), beg[i], deg[i], &a.c->err);
            cv[i] = __ldg(a.colors + v);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int64_t v = b + i * all;
            int64_t k0 = 0, k1 = -1;
            if (v < a.g.n) {
                account(a, static_cast<int32_t>(v), cv[i], 0, s_pres, conf, unc, my_max);
                a.low[v] = static_cast<uint8_t>(cv[i]);
                row_steps(v + beg[i] - off0, deg[i], a.steps, narrow, k0, k1);
            }
            // a row's steps: its own thread writes a few, its warp those of a longer row
            const bool own = k1 - k0 < kOwnSteps;
            if (own)
                for (; k0 <= k1; ++k0) a.first[k0] = static_cast<int32_t>(v);
            for (uint32_t m = __ballot_sync(kFull, !own); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const int64_t last = __shfl_sync(kFull, k1, src);
                const int32_t row = static_cast<int32_t>(__shfl_sync(kFull, v, src));
                for (int64_t k = __shfl_sync(kFull, k0, src) + lane_id(); k <= last; k += 32) a.first[k] = row;
            }
        }
    }
    warp_add(&a.c->uncolored, unc);
    warp_max(&a.c->max_color, my_max);
    flush_presence(a, s_pres);
}

// The ids of a step in the lane's 8 slots (a0: 16-byte aligned), those of
// slots outside [e0, e1) unspecified.
__device__ __forceinline__ void step_ids(const Graph& g, int64_t a0, int64_t e1, int32_t (&u)[8]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t e = a0 + 4 * (h * 32 + lane_id());
        int4 q = make_int4(0, 0, 0, 0);
        if (g.vec && e + 4 <= g.nnz) {
            if (e < e1) q = ld_stream4(g.idx + e);
        } else {
            if (e < e1) q.x = ld_stream(g.idx + e);
            if (e + 1 < e1) q.y = ld_stream(g.idx + e + 1);
            if (e + 2 < e1) q.z = ld_stream(g.idx + e + 2);
            if (e + 3 < e1) q.w = ld_stream(g.idx + e + 3);
        }
        u[4 * h] = q.x, u[4 * h + 1] = q.y, u[4 * h + 2] = q.z, u[4 * h + 3] = q.w;
    }
}

// One pass over the entries, flat: every lane takes 8 entries of a warp's
// step whatever rows they belong to, so none waits for a longer row; the
// next step's ids are read meanwhile.  Whose an entry is: a bit where a row
// begins, the row's color beside it; an entry's row is the last bit at or
// before it.  The low bytes are gathered, and a color only where its byte
// equals the row's: four times as many vertices stay in L1, where a random
// gather takes a third of the time it takes from L2 (800 against 280 G/s
// measured).  Bound by the gathers: both passes take 0.41 ms on R-MAT 22
// (128 M entries) and 1.83 ms on R-MAT 24 (522 M), where 4 lanes a short
// row, a warp or blocks a longer one, and 4-byte gathers took 0.69 and 2.63;
// bytes alone 0.69 and 2.62; this with a block's steps and its barriers 0.52
// and 2.23.  On a stencil of shuffled vertices, where nothing stays in L1,
// 241 us for 230.  A step inside one row skips the bits, and a step's row is
// read a step before its ids, which wait for it (this pass: R-MAT 22 376 ->
// 327 us, K_4000 39 -> 34).
// kInput: a recoloring input, with max_allowed.
template <bool kInput>
__global__ void __launch_bounds__(kBlock, kValBlocks) k_validate(ValArgs a) {
    constexpr int kWords = kValSlots / 32;
    __shared__ uint32_t s_bits_[kWarps][kWords];
    __shared__ int32_t s_color_[kWarps][kValSlots];  // of the row that begins at the slot
    const int w = threadIdx.x >> 5, l = lane_id();
    uint32_t* s_bits = s_bits_[w];
    int32_t* s_color = s_color_[w];
    // malformed offsets: the steps mean nothing (a vote: an id found bad meanwhile stops whole warps)
    if (__any_sync(kFull, *reinterpret_cast<volatile uint32_t*>(&a.c->err) != 0u)) return;
    const int32_t n = a.g.n;
    const int64_t off0 = __ldg(a.g.off);
    const int64_t total = n + __ldg(a.g.off + n) - off0;
    const int64_t nsteps = (total + kValChunk - 1) / kValChunk;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kWarps;
    uint32_t conf = 0;
    int64_t k = static_cast<int64_t>(blockIdx.x) * kWarps + w;
    // rows [v0, v1], entries [e0, e1)
    int32_t v0 = 0, v1 = 0;
    int64_t e0 = 0, e1 = 0;
    int32_t u[8];
    int32_t f0 = 0, f1 = 0;  // v0, v1 of the step staged next, read a step before its ids
    const auto rows_of = [&](int64_t step) {
        if (step >= nsteps) return;
        f0 = __ldg(a.first + step);
        f1 = step + 1 < nsteps ? __ldg(a.first + step + 1) : n;
    };
    rows_of(k);
    const auto stage = [&](int64_t step) {
        v0 = f0;
        v1 = f1;
        e0 = step * kValChunk - v0 + off0;
        e1 = min((step + 1) * kValChunk, total) - v1 + off0;
        step_ids(a.g, e0 & ~int64_t(3), e1, u);
        rows_of(step + stride);
    };
    if (k < nsteps) stage(k);
    for (; k < nsteps; k += stride) {
        const int64_t a0 = e0 & ~int64_t(3);
        const int32_t first_row = v0, last_row = min(v1, n - 1);
        const int32_t lo = static_cast<int32_t>(e0 - a0), hi = static_cast<int32_t>(e1 - a0);  // slots
        const bool inside = first_row == last_row;  // of a long row: its entries have one color
        const int32_t row_color = inside ? __ldg(a.colors + first_row) : 0;
        if (!inside) {
            if (l < kWords) s_bits[l] = 0u;
            __syncwarp();
            for (int32_t r = first_row; r <= last_row; r += 32) {
                const int32_t v = r + l;
                if (v <= last_row) {
                    const int64_t b = max(__ldg(a.g.off + v), e0), e = min(__ldg(a.g.off + v + 1), e1);
                    if (b < e) {
                        const int32_t at = static_cast<int32_t>(b - a0);
                        s_color[at] = __ldg(a.colors + v);
                        atomicOr(&s_bits[at >> 5], 1u << (at & 31));
                    }
                }
            }
        }
        uint32_t invalid = 0;  // slots of the lane with an id outside [0, n)
        uint32_t low[8];
        int32_t x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int32_t at = 4 * ((i >> 2) * 32 + l) + (i & 3);
            x[i] = u[i];
            low[i] = 256u;  // no entry: equals no byte
            if (at >= lo && at < hi) {
                if (static_cast<uint32_t>(x[i]) < static_cast<uint32_t>(n)) low[i] = __ldg(a.low + x[i]);
                else invalid |= 1u << i;
            }
        }
        if (k + stride < nsteps) stage(k + stride);
        int32_t bad = INT_MAX;
        // entry i of the lane, of the row that begins at slot `row` and has color cv
        const auto look_at = [&](int i, int32_t cv, int32_t row) {
            if (kInput && (cv < 1 || cv > a.max_allowed)) return;
            if (invalid >> i & 1u) {
                atomicOr(&a.c->err, kErrBadGraph);
            } else if (__ldg(a.colors + x[i]) == cv) {
                ++conf;
                bad = min(bad, row);
            }
        };
        if (inside) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if ((invalid >> i & 1u) || low[i] == (static_cast<uint32_t>(row_color) & 255u)) look_at(i, row_color, lo);
        } else {
            __syncwarp();
            // the last row start before each word
            const uint32_t wb = l < kWords ? s_bits[l] : 0u;
            int32_t m = wb ? 32 * l + 31 - __clz(wb) : -1;
#pragma unroll
            for (int d = 1; d < kWords; d <<= 1) {
                const int32_t o = __shfl_up_sync(kFull, m, d);
                if (l >= d) m = max(m, o);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int wi = 4 * h + (l >> 3);
                const int at = 4 * (h * 32 + l);
                const int32_t before = __shfl_sync(kFull, m, wi ? wi - 1 : 0);
                const uint32_t word = __shfl_sync(kFull, wb, wi);
                const uint32_t upto = word & (0xffffffffu >> (31 - (at & 31)));
                int32_t row = upto ? (at & ~31) + 31 - __clz(upto) : wi ? before : -1;
                const uint32_t begins = word >> (at & 31);
                int32_t cv = row >= 0 ? s_color[row] : 0;
                int32_t cvs[4];
                uint32_t look = invalid >> (4 * h) & 15u;  // entries to look at again
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j && (begins >> j & 1u)) cv = s_color[at + j];
                    cvs[j] = cv;
                    look |= static_cast<uint32_t>(low[4 * h + j] == (static_cast<uint32_t>(cv) & 255u)) << j;
                }
                if (look == 0) continue;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j && (begins >> j & 1u)) row = at + j;
                    if (look >> j & 1u) look_at(4 * h + j, cvs[j], row);
                }
            }
        }
        bad = __reduce_min_sync(kFull, bad);
        if (bad != INT_MAX && l == 0) {
            // the row that begins at the slot: the last one at or before that entry
            const int64_t e = a0 + bad;
            int32_t p = first_row, q = last_row;
            while (p < q) {
                const int32_t mid = p + (q - p + 1) / 2;
                if (__ldg(a.g.off + mid) <= e) p = mid;
                else q = mid - 1;
            }
            const unsigned long long rank = static_cast<unsigned long long>(n) - static_cast<unsigned long long>(p);
            if (rank > *reinterpret_cast<volatile unsigned long long*>(&a.c->bad_rank)) atomicMax(&a.c->bad_rank, rank);
        }
        __syncwarp();
    }
    warp_add(&a.c->conflicts, static_cast<unsigned long long>(conf));
}

__global__ void __launch_bounds__(kBlock) k_mark_present(int64_t n, const int32_t* colors,
                                                         uint32_t* bits) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kBlock;
    for (int64_t v = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x; v < n; v += stride) {
        const int32_t cv = colors[v];
        if (cv >= 1) atomicOr(&bits[cv >> 5], 1u << (cv & 31));
    }
}

__global__ void __launch_bounds__(kBlock) k_count_bits(int64_t words, const uint32_t* bits,
                                                       ValCtrl* c) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kBlock;
    unsigned long long s = 0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x; i < words; i += stride)
        s += __popc(bits[i]);
    warp_add(&c->distinct, s);
}

// The scratch of one validation, its pass over the rows and that over the entries.
struct ValRun {
    ScratchSet sc;
    ValArgs a{};
    gc_status start(const Graph& g, const int32_t* colors, int32_t max_allowed, const Tuning& t, cudaStream_t s) {
        a = ValArgs{g, colors, nullptr, nullptr, nullptr, nullptr, 0, max_allowed};
        a.steps = (static_cast<int64_t>(g.n) + g.nnz) / kValChunk + 1;
        static_assert(sizeof(ValCtrl) % 8 == 0, "the bitmap follows it");
        sc.want(&a.c, sizeof(ValCtrl) + kPresWords * 4);
        sc.want(&a.low, static_cast<int64_t>(g.n));
        sc.want(&a.first, a.steps * 4);
        if (!sc.alloc(s)) return GC_ERR_OOM;
        a.pres = reinterpret_cast<uint32_t*>(a.c + 1);
        cudaMemsetAsync(a.c, 0, sizeof(ValCtrl) + kPresWords * 4, s);
        const bool input = max_allowed != 0;
        // (four vertices a thread, but a block per SM first: K_4000 10.6 -> 5.2 us)
        const int64_t row_blocks = std::max<int64_t>((static_cast<int64_t>(g.n) + 4 * kBlock - 1) / (4 * kBlock),
                                                     std::min<int64_t>((static_cast<int64_t>(g.n) + kBlock - 1) / kBlock, sm_count()));
        const int rows = static_cast<int>(std::min<int64_t>(row_blocks, resident_grid(k_validate_rows, t)));
        GC_LAUNCH(input ? KID_RC_VALIDATE : KID_VALIDATE_ROWS, s, k_validate_rows<<<rows, kBlock, 0, s>>>(a));
        const auto entries = input ? k_validate<true> : k_validate<false>;
        const int grid = static_cast<int>(std::min<int64_t>((a.steps + kWarps - 1) / kWarps, resident_grid(entries, t)));
        GC_LAUNCH(input ? KID_RC_VALIDATE : KID_VALIDATE, s, entries<<<grid, kBlock, 0, s>>>(a));
        return GC_OK;
    }
};

// The input of a recoloring call: proper (Sec. 1), colors in [1,
// max_allowed].  The validation's passes instead of a warp per row, which
// left one warp walking each hub row: R-MAT 18 742 -> 41 us.
gc_status check_input_device(const Graph& g, const int32_t* colors, int32_t max_allowed, int32_t* max_color,
                             cudaStream_t s) {
    *max_color = 0;
    if (g.n == 0) return GC_OK;
    ValRun run;
    const gc_status st = run.start(g, colors, max_allowed, current_tuning(), s);
    if (st != GC_OK) return st;
    ValCtrl h;
    cudaError_t ce = cudaMemcpyAsync(&h, run.a.c, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_status(ce);
    if (h.err & kErrBadGraph) return GC_ERR_BAD_GRAPH;
    if (h.conflicts || h.uncolored || h.max_color > max_allowed) return GC_ERR_IMPROPER_INPUT;
    *max_color = h.max_color;
    return GC_OK;
}

gc_status validate_device(const Graph& g, const int32_t* colors, gc_validation* out,
                          cudaStream_t s) {
    std::memset(out, 0, sizeof(*out));
    out->first_bad_vertex = -1;
    if (g.n == 0) return GC_OK;
    const Tuning t = current_tuning();
    const int grid = persistent_grid(t);
    ValRun run;
    const gc_status st = run.start(g, colors, 0, t, s);
    if (st != GC_OK) return st;
    const ValArgs& a = run.a;
    ValCtrl h;
    GC_LAUNCH(KID_COUNT_BITS, s, k_count_bits<<<8, kBlock, 0, s>>>(kPresWords, a.pres, a.c));
    cudaError_t ce = cudaMemcpyAsync(&h, a.c, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_status(ce);
    if (h.err & kErrBadGraph) return GC_ERR_BAD_GRAPH;
    int64_t distinct = static_cast<int64_t>(h.distinct);
    if (h.big_colors > 0) {
        // colors beyond the shared bitmap: one bit per color up to the max
        const int64_t words = (static_cast<int64_t>(h.max_color) >> 5) + 1;
        Scratch sb;
        if (!sb.alloc(words * 4, s)) return GC_ERR_OOM;
        cudaMemsetAsync(sb.p, 0, words * 4, s);
        cudaMemsetAsync(&a.c->distinct, 0, sizeof(unsigned long long), s);
        const int vg = static_cast<int>(std::min<int64_t>((static_cast<int64_t>(g.n) + kBlock - 1) / kBlock, grid));
        GC_LAUNCH(KID_MARK_PRESENT, s, k_mark_present<<<vg, kBlock, 0, s>>>(g.n, colors, sb.as<uint32_t>()));
        const int wg = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((words + kBlock - 1) / kBlock, grid)));
        GC_LAUNCH(KID_COUNT_BITS, s, k_count_bits<<<wg, kBlock, 0, s>>>(words, sb.as<uint32_t>(), a.c));
        ce = cudaMemcpyAsync(&h, a.c, sizeof(h), cudaMemcpyDeviceToHost, s);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
        if (ce != cudaSuccess) return cuda_status(ce);
        distinct = static_cast<int64_t>(h.distinct);
    }
    out->n_conflicts = static_cast<int64_t>(h.conflicts);
    out->n_uncolored = static_cast<int64_t>(h.uncolored);
    out->max_color = h.max_color;
    out->n_distinct = static_cast<int32_t>(distinct);
    out->first_bad_vertex = h.bad_rank == 0 ? -1 : static_cast<int64_t>(g.n) - static_cast<int64_t>(h.bad_rank);
    return GC_OK;
}

// ---------------------------------------------------------------------------
// Validation without allocation (gc_validate_noalloc).  For callers that
// cannot allocate device memory: a process whose own caching allocator has
// reserved the device's memory up front (a cudaMalloc would fail or fragment
// it), a caller checking a result after an out-of-memory error, or a
// latency-critical path that must not wait on the driver's allocator.  Its
// scratch is a file-scope device array, held by every device that loads the
// library until the process exits; every call shares it, so two calls that
// overlap on the GPU (e.g. on two streams) race on it and must be serialised
// by the caller.  The call reads its result back and synchronizes the
// caller's stream.  The presence bitmap covers colors below kPresColors
// (65536); a coloring with a larger color is rejected, since counting its
// distinct colors would need scratch beyond the array.
// ---------------------------------------------------------------------------
struct NoAllocScratch {
    ValCtrl ctrl;
    uint32_t pres[kPresWords];
};

static __device__ __align__(256) NoAllocScratch g_validate_scratch;

// Clears what every call must start from: counters, the first bad vertex and
// the presence bitmap.
__global__ void __launch_bounds__(kBlock) k_validate_na_clear(NoAllocScratch* sc) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->ctrl.conflicts = 0;
        sc->ctrl.uncolored = 0;
        sc->ctrl.bad_rank = 0;
        sc->ctrl.max_color = 0;
        sc->ctrl.err = 0;
        sc->ctrl.distinct = 0;
        sc->ctrl.big_colors = 0;
    }
    for (int i = blockIdx.x * kBlock + threadIdx.x; i < kPresWords; i += gridDim.x * kBlock)
        sc->pres[i] = 0u;
}

// Light rows, kValG lanes per vertex; heavy rows are left to the next kernel
// (which finds them again by degree instead of through a list).
__global__ void __launch_bounds__(kBlock) k_validate_na_light(ValArgs a) {
    __shared__ uint32_t s_pres[kPresWords];
    for (int i = threadIdx.x; i < kPresWords; i += kBlock) s_pres[i] = 0u;
    __syncthreads();
    const int gi = threadIdx.x / kValG, gl = threadIdx.x % kValG;
    const int64_t groups = static_cast<int64_t>(gridDim.x) * (kBlock / kValG);
    int32_t my_max = 0;
    unsigned long long conf = 0, unc = 0;
    const int64_t n_pad = (a.g.n + groups - 1) / groups * groups;
    for (int64_t v = static_cast<int64_t>(blockIdx.x) * (kBlock / kValG) + gi; v < n_pad; v += groups) {
        const bool valid = v < a.g.n;
        int64_t beg = 0;
        int32_t deg = 0, cv = 0;
        bool heavy = false;
        if (valid) {
            row_of(a.g, static_cast<int32_t>(v), beg, deg, &a.c->err);
            cv = a.colors[v];
            heavy = deg > kHeavyDeg;
        }
        int32_t same = same_color<1>(a, beg, heavy ? 0 : deg, cv, gl, kValG);
#pragma unroll
        for (int d = kValG / 2; d >= 1; d >>= 1) same += __shfl_xor_sync(kFull, same, d);
        if (valid && gl == 0 && !heavy) account(a, static_cast<int32_t>(v), cv, same, s_pres, conf, unc, my_max);
    }
    warp_add(&a.c->conflicts, conf);
    warp_add(&a.c->uncolored, unc);
    warp_max(&a.c->max_color, my_max);
    flush_presence(a, s_pres);
}

// Heavy rows (degree > kHeavyDeg), one block per row, found by a scan of the
// degrees.
__global__ void __launch_bounds__(kBlock) k_validate_na_heavy(ValArgs a) {
    __shared__ uint32_t s_pres[kPresWords];
    __shared__ int32_t s_sum[kWarps];
    for (int i = threadIdx.x; i < kPresWords; i += kBlock) s_pres[i] = 0u;
    __syncthreads();
    int32_t my_max = 0;
    unsigned long long conf = 0, unc = 0;
    for (int64_t v0 = static_cast<int64_t>(blockIdx.x) * kBlock; v0 < a.g.n;
         v0 += static_cast<int64_t>(gridDim.x) * kBlock) {
        // the block's threads look at kBlock vertices, then walk the heavy ones
        const int64_t mine = v0 + threadIdx.x;
        bool heavy = false;
        if (mine < a.g.n) {
            const int64_t b = a.g.off[mine], e = a.g.off[mine + 1];
            heavy = e - b > kHeavyDeg;
        }
        uint32_t mask = __ballot_sync(kFull, heavy);
        __shared__ uint32_t s_mask[kWarps];
        if (lane_id() == 0) s_mask[threadIdx.x >> 5] = mask;
        __syncthreads();
        for (int w = 0; w < kWarps; ++w) {
            uint32_t m = s_mask[w];
            while (m) {
                const int bit = __ffs(m) - 1;
                m &= m - 1;
                const int32_t v = static_cast<int32_t>(v0 + w * 32 + bit);
                int64_t beg;
                int32_t deg;
                row_of(a.g, v, beg, deg, &a.c->err);
                const int32_t cv = a.colors[v];
                int32_t same = same_color<1>(a, beg, deg, cv, threadIdx.x, kBlock);
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1) same += __shfl_xor_sync(kFull, same, d);
                if (lane_id() == 0) s_sum[threadIdx.x >> 5] = same;
                __syncthreads();
                if (threadIdx.x == 0) {
                    int32_t tot = 0;
                    for (int q = 0; q < kWarps; ++q) tot += s_sum[q];
                    account(a, v, cv, tot, s_pres, conf, unc, my_max);
                }
                __syncthreads();
            }
        }
        __syncthreads();
    }
    warp_add(&a.c->conflicts, conf);
    warp_add(&a.c->uncolored, unc);
    warp_max(&a.c->max_color, my_max);
    flush_presence(a, s_pres);
}

namespace {
constexpr int kNoAllocDevices = 64;
std::mutex g_na_mu;
NoAllocScratch* g_na_ptr[kNoAllocDevices] = {};

// Device address of the scratch array on the current device, looked up once
// per device (the array's name is only a host-side stand-in).
gc_status noalloc_scratch(NoAllocScratch** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return GC_ERR_CUDA;
    if (dev < 0 || dev >= kNoAllocDevices) return GC_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g_na_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_validate_scratch);
        if (e != cudaSuccess || !p) return GC_ERR_CUDA;
        g_na_ptr[dev] = static_cast<NoAllocScratch*>(p);
    }
    *out = g_na_ptr[dev];
    return GC_OK;
}

int noalloc_grid(const void* kernel) {
    int dev = 0, sms = 1, per_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    return std::max(1, sms) * per_sm;
}
}  // namespace

gc_status validate_noalloc_device(const Graph& g, const int32_t* colors, gc_validation* out,
                                  cudaStream_t s) {
    std::memset(out, 0, sizeof(*out));
    out->first_bad_vertex = -1;
    if (g.n == 0) return GC_OK;
    NoAllocScratch* sc = nullptr;
    gc_status st = noalloc_scratch(&sc);
    if (st != GC_OK) return st;
    ValArgs a{g, colors, &sc->ctrl, sc->pres, nullptr, nullptr, 0, 0};
    // Each launch is checked before the next is enqueued: a clear that failed
    // to launch must not let the read-back return the previous call's counts.
    // (Not bracketed by the profiling events, which would create events.)
    cudaError_t ce;
    k_validate_na_clear<<<8, kBlock, 0, s>>>(sc);
    note_launches(1);
    if ((ce = cudaGetLastError()) != cudaSuccess) return cuda_status(ce);
    k_validate_na_light<<<noalloc_grid(reinterpret_cast<const void*>(k_validate_na_light)), kBlock, 0, s>>>(a);
    note_launches(1);
    if ((ce = cudaGetLastError()) != cudaSuccess) return cuda_status(ce);
    k_validate_na_heavy<<<noalloc_grid(reinterpret_cast<const void*>(k_validate_na_heavy)), kBlock, 0, s>>>(a);
    note_launches(1);
    if ((ce = cudaGetLastError()) != cudaSuccess) return cuda_status(ce);
    k_count_bits<<<8, kBlock, 0, s>>>(kPresWords, sc->pres, &sc->ctrl);
    note_launches(1);
    if ((ce = cudaGetLastError()) != cudaSuccess) return cuda_status(ce);
    ValCtrl h;
    ce = cudaMemcpyAsync(&h, &sc->ctrl, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_status(ce);
    if (h.err & kErrBadGraph) return GC_ERR_BAD_GRAPH;
    if (h.big_colors > 0) return GC_ERR_INVALID_ARG;  // a color >= 65536: beyond the scratch
    out->n_conflicts = static_cast<int64_t>(h.conflicts);
    out->n_uncolored = static_cast<int64_t>(h.uncolored);
    out->max_color = h.max_color;
    out->n_distinct = static_cast<int32_t>(h.distinct);
    out->first_bad_vertex = h.bad_rank == 0 ? -1 : static_cast<int64_t>(g.n) - static_cast<int64_t>(h.bad_rank);
    return GC_OK;
}

// ---------------------------------------------------------------------------
// CSR structure check
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock) k_check_graph(Graph g, long long* first_bad) {
    const int w = (blockIdx.x * kBlock + threadIdx.x) >> 5;
    const int nw = (gridDim.x * kBlock) >> 5;
    const int l = lane_id();
    for (int64_t v = w; v < g.n; v += nw) {
        const int64_t beg = g.off[v], end = g.off[v + 1];
        bool bad = beg < 0 || end < beg || end > g.nnz || (v == 0 && beg != 0) ||
                   (v == g.n - 1 && end != g.nnz);
        if (!bad) {
            for (int64_t e = beg + l; e < end; e += 32) {
                const int32_t u = g.idx[e];
                if (u < 0 || u >= g.n || u == v) bad = true;
            }
        }
        if (__any_sync(kFull, bad) && l == 0) atomicMin(first_bad, static_cast<long long>(v));
    }
}

gc_status check_graph_device(const Graph& g, int64_t* first_bad, cudaStream_t s) {
    if (first_bad) *first_bad = -1;
    if (g.n == 0) return g.nnz == 0 ? GC_OK : GC_ERR_BAD_GRAPH;
    Scratch sc;
    if (!sc.alloc(sizeof(long long), s)) return GC_ERR_OOM;
    long long h = LLONG_MAX;
    cudaMemcpyAsync(sc.p, &h, sizeof(h), cudaMemcpyHostToDevice, s);
    GC_LAUNCH(KID_CHECK_GRAPH, s,
              k_check_graph<<<persistent_grid(current_tuning()), kBlock, 0, s>>>(g, sc.as<long long>()));
    cudaError_t ce = cudaMemcpyAsync(&h, sc.p, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    if (ce != cudaSuccess) return cuda_status(ce);
    if (h == LLONG_MAX) return GC_OK;
    if (first_bad) *first_bad = static_cast<int64_t>(h);
    return GC_ERR_BAD_GRAPH;
}

}  // namespace gc
