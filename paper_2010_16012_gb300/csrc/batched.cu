// batched.cu -- many personalised PageRank vectors and multi-source BFS runs
// over several graphs in one persistent launch (replayed from a CUDA graph).
//
// Personalised PageRank (Section 3.1 formula with a one-hot teleport vector
// s = e_seed per vector): for each graph the K iterates are one row-major
// matrix X[n][K], so the pull sweep (Algorithm 1, pulling) gathers neighbour
// rows -- one coalesced read per in-edge instead of K scattered 4-byte reads:
//     Y[v][j] = (1-d) [v == seed_j] + d * sum_{u in in(v)} w_uv inv_deg[u] X[u][j]
// The work is cut into jobs: one graph and a slice of KS consecutive columns,
// KS the widest of 128, 64 or 32 (at most K) for which the slice of both
// iterates fits the L2 budget, so every gathered row segment (KS * 4 bytes, a whole number of
// 128-byte lines) comes from L2 for the job's whole run.  Jobs run one after
// another over the whole grid; each sweeps its slice to convergence.  Every
// vector (column) starts at its seed's one-hot vector (or at 1/n), has its own
// L1 residual, reduced in FP64, and stops at its first sweep below tol; its
// column is then carried forward unchanged.
//
// Multi-source BFS (Section 3.3 / Algorithm 3 with ready = 1, up to 64 sources
// at once): F[v], V[v] and N[v] are 64-bit masks (bit j = search j).  Each
// graph chooses per level between top-down (frontier vertices OR their masks
// into their out-neighbours' N with 64-bit atomics) and bottom-up (every vertex
// not yet reached by all searches ORs the frontier masks of its in-neighbours,
// stopping once every missing search is covered), by the rule of the single
// search: bottom-up when the frontier's out-edges times alpha exceed the
// in-edges of vertices still missing a search, back to top-down when the
// frontier shrinks below n / beta.  An owner-only update then advances V, F and
// the levels.
//
// Both kernels are cooperative launches whose phases are separated by a grid
// barrier with a bounded spin-wait (on expiry an error flag is set, every
// block returns and the host reports GP_ERR_TIMEOUT).
#include <algorithm>
#include <cstring>
#include <initializer_list>
#include <vector>

#include "gp_internal.cuh"

namespace gp {

constexpr int BT_THREADS = 512;  // threads per block of the persistent kernels
#ifndef GP_BT_MINB
#define GP_BT_MINB 2
#endif
constexpr int BT_SEG = 8;        // vertices per warp work unit (light rows)
constexpr int BT_MAX_KS = 128;   // widest column slice of one PageRank job (a float4 per lane)

struct BGraph {  // per-graph device descriptor
    int64_t n;
    const int64_t *csc_off;
    const int32_t *csc_idx;
    const float *csc_w;
    const int64_t *csr_off;
    const int32_t *csr_idx;
    const float *inv_deg;
    float *X0, *X1;          // PPR iterates [n][K]; X0 doubles as the output
    uint64_t *F, *V, *N;     // MS-BFS masks
    int32_t *levels;         // MS-BFS output [n][64]
    int64_t chunk0, nchunk;  // in-edge chunks of its vertices of big in-degree in the chunk list
    int64_t ochunk0, nochunk;  // out-edge chunks of the vertices of big out-degree (the in-edge ones where the orders are one)
};

struct BChunk {  // warp work item: a piece of a big vertex's edge list
    int64_t beg;
    int32_t len;
    int32_t v;
    int32_t r;    // in-edge chunks: the vertex's place among the big ones,
    int32_t nch;  // and its chunks
};

struct BJob {  // one graph and the column slice [c0, c0 + 32 * kpl)
    int32_t graph;
    int32_t c0;
    int32_t kpl;
    int32_t pad;
};

struct BPend {  // a PageRank column a job left iterating, for a packed job
    int32_t graph;
    int32_t col;    // its column in the graph's iterates
    int32_t kdone;  // sweeps it has had
    int32_t pad;
};

struct BatchDev {
    int ngraphs, K, nsrc;
    float d, one_minus_d;
    double tol;
    int iters;
    int64_t big_min;        // in-degree above which a vertex's in-edges are split into chunks
    int32_t one_hot_start;  // PPR iterates start at e_seed (else 1/n)
    float alpha, beta;      // MS-BFS direction rule
    const BGraph *graphs;
    const BJob *jobs;
    int njobs;
    const int64_t *bcstart; // [big vertices + 1] chunk range of each big vertex, grouped by graph
    const BChunk *chunks;
    unsigned *bdone;        // [big vertices] chunks of each big vertex summed in this sweep
    float *part;            // [max chunks of one graph][K] chunk partial rows
    double *res_acc;        // [3][K] per-sweep column residuals (a ring)
    const int32_t *seeds;   // [ngraphs][K]
    int32_t *iters_done;    // [ngraphs][K]
    const int32_t *sources; // [ngraphs][64] (MS-BFS)
    int32_t *const *lev_out;  // [ngraphs] where this call's levels go (MS-BFS)
    int32_t *counters;      // [0] most PPR sweeps of any column, [1] BFS levels, [2] packed columns, [3], [4] those left to narrower jobs, [5] rows listed, [6] 1: not a closed set, [7] last columns
    int32_t pack_max;       // a job stops once at most this many of its columns iterate (0: never)
    BPend *pend;            // [3][ngraphs * K] the columns left iterating, in job order: for jobs of 32, 8 and 4
    float *XP0, *XP1;       // [max n][32] iterates of a packed job (rows as wide as the job)
    unsigned long long *mcount;  // MS-BFS [2][ngraphs][4]: frontier vertices, their out-edges, open in-edges, new bits
    GridSync *sync;
};

// ------------------------------------------------------------------ batched PPR

// Pairs of FP32 values, added (and so on) by one instruction, rounded as the scalar operations are.
__device__ __forceinline__ uint64_t pk(float x, float y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpk(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {  // a - b as b * -1 + a, rounded once
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(0xbf800000bf800000ull), "l"(a));
    return r;
}

// Compensated (Kahan) accumulation of f * r: a column sums up to thousands of
// terms one after another, so the running rounding error is carried in `lo`,
// negated: the sum is hi + lo.
__device__ __forceinline__ void kahan_add2(uint64_t &hi, uint64_t &lo, uint64_t f, uint64_t r) {
    uint64_t y;  // f * r + lo, rounded once
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(y) : "l"(f), "l"(r), "l"(lo));
    const uint64_t t = add2(hi, y);
    lo = sub2(y, sub2(t, hi));
    hi = t;
}

// A job of KS columns maps a warp onto NG = 32 / (KS / 4) edge groups of
// KS / 4 lanes; lane c4 of a group holds columns 4*c4 .. 4*c4+3 of a row (one
// float4), so one warp-wide load fetches NG row segments.  Light vertices take
// one group each; the edges of a chunk or of a big vertex are split over the
// groups, whose sums are then added with shuffles.
template <int KS>
struct Lanes {
    static constexpr int LPR = KS / 4;   // lanes per row segment
    static constexpr int NG = 32 / LPR;  // edge groups per warp
};

#ifndef GP_BT_INFLIGHT
#define GP_BT_INFLIGHT 6
#endif
// Row segments in flight per lane: 6 of 4 registers each fit the 64 registers a
// thread has at two blocks per SM with few spills (R-MAT 2^17, 128 columns: 219
// us a sweep; 8 in flight 237, 4 in flight 247, 4 at three blocks per SM 254).
constexpr int BT_INFLIGHT = GP_BT_INFLIGHT;

// Row segments are read through L2 (ld.global.cg): the iterates are rewritten
// by the kernel itself between sweeps, so the non-coherent read-only path may
// not be used for them.
__device__ __forceinline__ float4 ld_seg(const float *X, int K, int32_t u, int c4) {
    return __ldcg(reinterpret_cast<const float4 *>(X + (int64_t)u * K) + c4);
}

// Compensated partial sums of a lane's four columns, in pairs: the value is hi + lo.
struct Sum4 {
    uint64_t hi[2] = {0, 0}, lo[2] = {0, 0};
    __device__ __forceinline__ void add(uint64_t f, const float4 &r) {
        kahan_add2(hi[0], lo[0], f, pk(r.x, r.y));
        kahan_add2(hi[1], lo[1], f, pk(r.z, r.w));
    }
};

// BT_INFLIGHT edges from e on, every `step`; those from `end` on add zero (FULL_W: there are none).
template <bool FULL_W>
__device__ __forceinline__ void gather_window(const BGraph &G, const float *X, int K, int64_t e, int64_t end, int step,
                                              int c4, Sum4 &a) {
    int32_t u[BT_INFLIGHT];
    float f[BT_INFLIGHT];
    float4 r[BT_INFLIGHT];
#pragma unroll
    for (int q = 0; q < BT_INFLIGHT; ++q) u[q] = FULL_W || e + q * step < end ? __ldg(G.csc_idx + e + q * step) : -1;
#pragma unroll
    for (int q = 0; q < BT_INFLIGHT; ++q) {
        if (!FULL_W) r[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (FULL_W || u[q] >= 0) r[q] = ld_seg(X, K, u[q], c4);
    }
#pragma unroll
    for (int q = 0; q < BT_INFLIGHT; ++q) {
        f[q] = FULL_W || u[q] >= 0 ? __ldg(G.inv_deg + u[q]) : 0.f;
        if (G.csc_w && (FULL_W || u[q] >= 0)) f[q] *= __ldg(G.csc_w + e + q * step);
    }
#pragma unroll
    for (int q = 0; q < BT_INFLIGHT; ++q) a.add(pk(f[q], f[q]), r[q]);
}

// Sum over in-edges beg, beg + step, beg + 2 step, ... < end of the rows' four
// columns at c4 (X points at column c0 of row 0; rows are K floats apart), each
// product folded into a compensated (Kahan) sum: a column sums up to
// thousands of terms, and a hub's FP32 rounding feeds back into every sweep.
// The last window is predicated, not walked edge by edge: most lists are shorter
// than one window, and their edges' loads would wait for one another.
__device__ __forceinline__ Sum4 gather_seg(const BGraph &G, const float *X, int K, int64_t beg, int64_t end, int step,
                                           int c4) {
    Sum4 a;
    int64_t e = beg;
    for (; e + (BT_INFLIGHT - 1) * step < end; e += BT_INFLIGHT * step) gather_window<true>(G, X, K, e, end, step, c4, a);
    if (e < end) gather_window<false>(G, X, K, e, end, step, c4, a);
    return a;
}

__device__ __forceinline__ float4 value4(const Sum4 &a) {
    const float2 x = unpk(add2(a.hi[0], a.lo[0])), y = unpk(add2(a.hi[1], a.lo[1]));
    return make_float4(x.x, x.y, y.x, y.y);
}

// Adds the groups' compensated sums of a warp (every group then holds the
// total): error-free two-sums of the leading parts, corrections added.
template <int KS>
__device__ __forceinline__ Sum4 groups_sum(Sum4 a) {
#pragma unroll
    for (int o = Lanes<KS>::LPR; o < 32; o <<= 1) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint64_t ohi = __shfl_xor_sync(FULL, a.hi[i], o), olo = __shfl_xor_sync(FULL, a.lo[i], o);
            const uint64_t t = add2(a.hi[i], ohi);
            const uint64_t bp = sub2(t, a.hi[i]);
            const uint64_t err = add2(sub2(a.hi[i], sub2(t, bp)), sub2(ohi, bp));
            a.hi[i] = t;
            a.lo[i] = add2(add2(a.lo[i], olo), err);
        }
    }
    return a;
}
template <int KS>
__device__ __forceinline__ float4 groups_total(const Sum4 &a) {
    return value4(groups_sum<KS>(a));
}

// The columns one PageRank job iterates: a slice of a graph's own iterates
// (pend == nullptr: columns c0 .. c0 + KS - 1 of X0/X1, rows K apart), or a
// packed job over the batch's packed iterates (rows KS apart), whose column j
// continues the graph's column pend[j].col after pend[j].kdone sweeps.
struct PView {
    int graph;
    float *X0, *X1;     // the start and the result are in X0
    int ld;             // row stride of X0 and X1 (floats)
    int c0;
    const BPend *pend;  // packed job, or nullptr
    int cnt;            // packed job: columns in use (the rest idle)
    // columns still iterating when at most `leave` are left go to `list`, whose length is *count
    int leave;
    BPend *list;
    int32_t *count;
};

// A job's columns in shared memory: the graph's column and the seed of each,
// the sweeps it has had before, and whether it still iterates.
struct PCols {
    __align__(16) int col[BT_MAX_KS], seed[BT_MAX_KS], kbase[BT_MAX_KS], active[BT_MAX_KS];
    int next[2];                              // by sweep parity: the block's next unit
    // per lane: |y - x| of its four columns in the present unit, and in those before as hi + lo (see
    // res_unit), pairs as packed values
    __align__(16) float res[BT_THREADS / 32][32][4];
    uint64_t hi[BT_THREADS / 32][32][2], lo[BT_THREADS / 32][32][2];
};

// The lane's sums of one unit into its hi + lo, error-free but for the roundings
// of lo (2^-48 of the sum each).  Warps draw their units in no fixed order, so a
// column's change is summed in another order in every run; that precisely, and
// the sweep in which it falls below the tolerance is the same one.  (A unit's
// rows have their order, so plain sums do there.)
__device__ __forceinline__ void res_unit(PCols &C, int wib, int lane) {
    float4 &r = *reinterpret_cast<float4 *>(C.res[wib][lane]);
    const uint64_t x[2] = {pk(r.x, r.y), pk(r.z, r.w)};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        uint64_t &hi = C.hi[wib][lane][q], &lo = C.lo[wib][lane][q];
        const uint64_t h = hi, t = add2(h, x[q]);
        const uint64_t bp = sub2(t, h);
        lo = add2(lo, add2(sub2(h, sub2(t, bp)), sub2(x[q], bp)));
        hi = t;
    }
    r = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Writes the lane's four columns of row v of the slice of Y from the gathered
// sum and the row x of the current iterate, carrying stopped columns forward;
// adds |y - x| of the columns still iterating to the lane's residual slots
// (shared memory, one owner each).
__device__ __forceinline__ void finish_seg(const BatchDev &B, float *Y, int64_t o, int64_t v, int c4, const float4 &x,
                                           const float4 &sum, float *my_res, const PCols &C) {
    const float xs[4] = {x.x, x.y, x.z, x.w}, ss[4] = {sum.x, sum.y, sum.z, sum.w};
    const int4 a4 = *reinterpret_cast<const int4 *>(C.active + 4 * c4), s4 = *reinterpret_cast<const int4 *>(C.seed + 4 * c4);
    const int act[4] = {a4.x, a4.y, a4.z, a4.w}, seed[4] = {s4.x, s4.y, s4.z, s4.w};
    float ys[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        ys[q] = xs[q];
        if (act[q]) {
            const float base = seed[q] == (int32_t)v ? B.one_minus_d : 0.f;
            ys[q] = base + B.d * ss[q];
            my_res[q] += fabsf(ys[q] - xs[q]);
        }
    }
    *reinterpret_cast<float4 *>(Y + o) = make_float4(ys[0], ys[1], ys[2], ys[3]);
}

// Sum of partial rows first, first + NG, ... < end (the row's columns at `part`), over the warp's groups.
template <int KS>
__device__ __forceinline__ float4 sum_parts(const float *part, int64_t first, int64_t end) {
    constexpr int NG = Lanes<KS>::NG;
    Sum4 a;
    const uint64_t one = pk(1.f, 1.f);
    for (int64_t c = first; c < end; c += BT_INFLIGHT * NG) {
        float4 p[BT_INFLIGHT];
#pragma unroll
        for (int q = 0; q < BT_INFLIGHT; ++q) {
            p[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c + q * NG < end) p[q] = __ldcg(reinterpret_cast<const float4 *>(part + (c + q * NG) * KS));
        }
#pragma unroll
        for (int q = 0; q < BT_INFLIGHT; ++q) a.add(one, p[q]);
    }
    return groups_total<KS>(a);
}

// The rows that a graph's last columns reach, where they are few.  The slowest
// columns are those seeded in a component of a few vertices (their alternating
// modes decay as d^k: five times the sweeps of the others), and all their other
// rows are zero and stay so.  A column that has been alone for PPR_ALONE sweeps goes
// to a last job (LAST), up to four of a graph together where several slices leave
// one each.  After two sweeps it lists the rows in which any of its columns is not
// zero in either iterate (or has its seed), in the room behind the iterates;
// R.whole stays true unless no out-edge of theirs leaves them, they are at most an
// eighth of the rows and none has a long in-list (those go by chunks).  The sums of
// the listed rows are the same ones in the same order, and the others need no
// writes.  At 131K vertices a sweep of two rows takes about 35 us less than one of
// all: six R-MAT graphs of up to 2^17 vertices with one such column, of 89 sweeps,
// 27.4 -> 25.1 ms (handed over after 4 sweeps alone 24.6, but more columns pay for it).
constexpr int PPR_ALONE = 10;
struct PRows {
    bool whole = true;
    const int32_t *list = nullptr;
    int64_t count = 0;
};
template <int KS>
__device__ __noinline__ bool ppr_rows(const BatchDev &B, const PView &J, const PCols &C, PRows &R) {
    const BGraph &G = B.graphs[J.graph];
    const int64_t n = G.n;
    const int lane = lane_id();
    const int64_t gthread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nthreads = (int64_t)gridDim.x * blockDim.x;
    int32_t *list = reinterpret_cast<int32_t *>(J.X1 + n * KS);  // of X1's 32 columns the job has KS
    uint32_t *bits = reinterpret_cast<uint32_t *>(list + n);
    int32_t *count = B.counters + 5, *out = B.counters + 6;
    for (int64_t v0 = (gthread >> 5) * 32; v0 < n; v0 += nthreads) {
        const int64_t v = v0 + lane;
        bool in = false;
        for (int c = 0; c < J.cnt && v < n; ++c)
            in |= __ldcg(J.X0 + v * KS + c) != 0.f || __ldcg(J.X1 + v * KS + c) != 0.f || v == C.seed[c];
        const unsigned m = __ballot_sync(FULL, in);
        const bool longest = __any_sync(FULL, in && G.csc_off[v + 1] - G.csc_off[v] > B.big_min);
        int at = 0;
        if (lane == 0) {
            bits[v0 >> 5] = m;
            if (m) at = atomicAdd(count, __popc(m));
            if (longest) atomicOr(out, 1);
        }
        at = __shfl_sync(FULL, at, 0);
        if (in) list[at + __popc(m & ((1u << lane) - 1u))] = (int32_t)v;
    }
    if (!grid_sync(B.sync, gridDim.x)) return false;
    R.count = __ldcg(count);
    const bool few = R.count <= n / 8;
    if (few) {
        bool leaves = false;
        for (int64_t i = gthread; i < R.count; i += nthreads) {
            const int32_t u = __ldcg(list + i);
            for (int64_t e = G.csr_off[u]; e < G.csr_off[u + 1] && !leaves; ++e) {
                const int32_t w = __ldg(G.csr_idx + e);
                leaves = !((__ldcg(bits + (w >> 5)) >> (w & 31)) & 1u);
            }
        }
        if (leaves) atomicOr(out, 1);
    }
    if (!grid_sync(B.sync, gridDim.x)) return false;
    R.whole = !few || __ldcg(out) != 0;
    R.list = list;
    return true;
}

// One job: the slice's sweeps from the start vector to convergence, or until at
// most J.leave of its columns still iterate (those are then left, at their
// latest iterate, to a packed job).  Returns false when a grid barrier gave up.
// Bound by the L2 row gathers on large graphs (R-MAT 2^17, 128 columns: 305 ->
// 219 us a sweep, 8.7 TB/s of gathered rows), by the chains of loads per vertex
// and the barrier on small ones (8,155 vertices: 39 -> 29 us).  What the warps
// waited for before was one another: equal shares of unequal units, and a
// second phase with a barrier of its own for the big vertices' partial rows.
// Not inlined: the widths' loops share no registers.
template <int KS, bool LAST = false>
__device__ __noinline__ bool ppr_job(const BatchDev &B, const PView &J, PCols &C) {
    constexpr int LPR = Lanes<KS>::LPR, NG = Lanes<KS>::NG;
    const int K = B.K;
    const int ld = J.ld;
    const BGraph &G = B.graphs[J.graph];
    const int64_t n = G.n;
    const int lane = lane_id(), grp = lane / LPR, c4 = lane % LPR;
    const int wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int64_t gthread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int64_t nwarps = nthreads >> 5;
    if (threadIdx.x < 2) C.next[threadIdx.x] = 0;
    for (int c = threadIdx.x; c < KS; c += blockDim.x) {
        const bool used = !J.pend || c < J.cnt;
        C.col[c] = !used ? 0 : J.pend ? J.pend[c].col : J.c0 + c;
        C.kbase[c] = J.pend && used ? J.pend[c].kdone : 0;
        C.seed[c] = B.seeds[J.graph * K + C.col[c]];
        C.active[c] = used && C.kbase[c] < B.iters;
    }
    __syncthreads();
    if (!J.pend) {
        // start: every column at 1/n, or at its seed's one-hot vector
        const float x0 = 1.0f / (float)n;
        for (int64_t i = gthread; i < n * KS; i += nthreads) {
            const int64_t v = i / KS;
            const int c = (int)(i % KS);
            J.X0[v * ld + J.c0 + c] = B.one_hot_start ? (C.seed[c] == (int32_t)v ? 1.0f : 0.0f) : x0;
        }
    } else {
        // start: the packed columns' latest iterates (idle columns at zero)
        for (int64_t i = gthread; i < n * KS; i += nthreads) {
            const int64_t v = i / KS;
            const int c = (int)(i % KS);
            J.X0[v * ld + c] = c < J.cnt ? __ldcg(G.X0 + v * K + C.col[c]) : 0.f;
        }
    }
    if (gthread < 3 * KS) B.res_acc[(gthread / KS) * K + (gthread % KS)] = 0.0;
    if (LAST && gthread == 0) B.counters[5] = B.counters[6] = 0;
    if (!grid_sync(B.sync, gridDim.x)) return false;
    PRows R;
    int alone = 0;  // sweeps with one column left
    // vertices per warp unit: few where the graph has few, so that every warp gets some
    int seg = BT_SEG;
    while (seg > NG && (n + seg - 1) / seg < nwarps) seg /= 2;
    seg = max(seg, NG);
    const int64_t nseg = (n + seg - 1) / seg;
    int k = 1, last = 0;
    for (; k <= B.iters; ++k) {
        const float *Xc = (k & 1) ? J.X0 : J.X1;
        const float *Xs = Xc + J.c0;  // column c0 of the current iterate
        float *Y = (k & 1) ? J.X1 : J.X0;
        double *racc = B.res_acc + (k % 3) * K;
        if (blockIdx.x == 0)  // the ring slot of sweep k + 1 (last read two sweeps ago)
            for (int c = threadIdx.x; c < KS; c += blockDim.x) B.res_acc[((k + 1) % 3) * K + c] = 0.0;
        float *my_res = C.res[wib][lane];
#pragma unroll
        for (int q = 0; q < 4; ++q) my_res[q] = 0.f;
#pragma unroll
        for (int q = 0; q < 2; ++q) C.hi[wib][lane][q] = C.lo[wib][lane][q] = 0;
        if (threadIdx.x == 0) C.next[(k + 1) & 1] = 0;
        // The block's units, each to the warp that is free (equal shares of them left the warps
        // waiting for one another most of the time on small graphs): chunks of big vertices,
        // split over the groups, then light rows, a vertex per group.
        while (true) {
            int i = 0;
            if (lane == 0) i = atomicAdd(&C.next[k & 1], 1);
            i = __shfl_sync(FULL, i, 0);
            const int64_t u = (int64_t)i * gridDim.x + blockIdx.x;
            const bool few = LAST && !R.whole;  // the listed rows
            if (u >= (few ? (R.count + seg - 1) / seg : G.nchunk + nseg)) break;
            if (!few && u < G.nchunk) {
                const BChunk ch = B.chunks[G.chunk0 + u];
                const int64_t v = ch.v;
                const int64_t o = v * ld + J.c0 + 4 * c4;
                float4 sum = groups_total<KS>(gather_seg(G, Xs, ld, ch.beg + grp, ch.beg + ch.len, NG, c4));
                if (ch.nch > 1) {
                    // the last of the vertex's chunks to finish adds the partial rows, in their order
                    if (grp == 0) *reinterpret_cast<float4 *>(B.part + u * KS + 4 * c4) = sum;
                    __syncwarp();
                    unsigned done = 0;
                    if (lane == 0) {
                        __threadfence();
                        done = atomicInc(B.bdone + ch.r, (unsigned)ch.nch - 1u);  // back at 0 after the last
                        __threadfence();
                    }
                    if (__shfl_sync(FULL, done, 0) != (unsigned)ch.nch - 1u) continue;
                    __syncwarp();  // what lane 0's fence has ordered is ordered for the warp (a shuffle orders no memory)
                    const int64_t cb = B.bcstart[ch.r] - G.chunk0;
                    sum = sum_parts<KS>(B.part + 4 * c4, cb + grp, cb + ch.nch);
                }
                if (grp == 0) {
                    const float4 x = __ldcg(reinterpret_cast<const float4 *>(Xc + o));
                    finish_seg(B, Y, o, v, c4, x, sum, my_res, C);
                    res_unit(C, wib, lane);
                }
            } else {
                const int64_t v0 = (few ? u : u - G.nchunk) * seg;
                int64_t ob = 0;  // the unit's lists, a vertex per lane
                int len = 0;
                int32_t lv = 0;
                if (lane < seg && v0 + lane < (few ? R.count : n)) {
                    if (few) lv = __ldcg(R.list + v0 + lane);
                    ob = G.csc_off[few ? lv : v0 + lane];
                    const int64_t d = G.csc_off[(few ? lv : v0 + lane) + 1] - ob;
                    // big vertices are done above; without in-edges a row is its base in every
                    // sweep, so both iterates hold it after two
                    len = d > B.big_min || (d == 0 && k > 2) ? -1 : (int)d;
                } else {
                    len = -1;
                }
                for (int i2 = 0; i2 < seg; i2 += NG) {
                    const int64_t b = __shfl_sync(FULL, ob, i2 + grp);
                    const int dl = __shfl_sync(FULL, len, i2 + grp);
                    const int32_t l = LAST ? __shfl_sync(FULL, lv, i2 + grp) : 0;
                    if (dl < 0) continue;
                    const int64_t v = few ? l : v0 + i2 + grp, o = v * ld + J.c0 + 4 * c4;
                    const float4 sum = value4(gather_seg(G, Xs, ld, b, b + dl, 1, c4));
                    const float4 x = __ldcg(reinterpret_cast<const float4 *>(Xc + o));
                    finish_seg(B, Y, o, v, c4, x, sum, my_res, C);
                }
                res_unit(C, wib, lane);
            }
        }
        // the block's column residuals: the slots of every warp and group added
        // in a fixed order, then one FP64 atomic per column into the sweep's ring slot
        constexpr int SLOTS = KS < 32 ? 1 : NG;
        if (KS < 32) {  // many groups per column: a warp's are added first, by the same sums
            // (in FP64 six R-MAT graphs of up to 2^17 vertices, 256 columns, took 24.7 ms instead of 24.4)
            Sum4 a;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                a.hi[q] = C.hi[wib][lane][q];
                a.lo[q] = C.lo[wib][lane][q];
            }
            a = groups_sum<KS>(a);
            __syncwarp();
            if (grp == 0)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    C.hi[wib][lane][q] = a.hi[q];
                    C.lo[wib][lane][q] = a.lo[q];
                }
        }
        __syncthreads();
        for (int c = threadIdx.x; c < KS; c += blockDim.x) {
            if (!C.active[c]) continue;
            float t = 0.f, e = 0.f;  // as res_unit
            for (int i = 0; i < wpb; ++i)
                for (int g = 0; g < SLOTS; ++g) {
                    const float hi = reinterpret_cast<const float *>(C.hi[i][g * LPR + c / 4])[c % 4];
                    const float lo = reinterpret_cast<const float *>(C.lo[i][g * LPR + c / 4])[c % 4];
                    const float s = t + hi;
                    const float bp = s - t;
                    e += (t - (s - bp)) + (hi - bp) + lo;
                    t = s;
                }
            const double r = (double)t + (double)e;
            if (r != 0.0) atomicAdd(racc + c, r);
        }
        if (!grid_sync(B.sync, gridDim.x)) return false;
        // every block takes the same decision from the same totals
        int any = 0;
        for (int c = threadIdx.x; c < KS; c += blockDim.x) {
            if (!C.active[c]) continue;
            const double r = __ldcg(racc + c);
            const int kc = C.kbase[c] + k;  // the column's sweeps
            if (blockIdx.x == 0) B.iters_done[J.graph * K + C.col[c]] = kc;
            if (r < B.tol || kc >= B.iters)
                C.active[c] = 0;
            else
                any = 1;
        }
        const int nact = __syncthreads_count(any);  // one column per thread (KS <= blockDim)
        last = k;
        if (!nact) break;
        if constexpr (KS == 4) alone += nact == 1;
        if (nact <= J.leave && (KS != 4 || alone >= PPR_ALONE)) {
            // the few columns left go to a narrower job; block 0 lists them in column order
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                int at = atomicAdd(J.count, nact);
                for (int c = 0; c < KS; ++c)
                    if (C.active[c]) J.list[at++] = BPend{J.graph, C.col[c], C.kbase[c] + k, 0};
            }
            break;
        }
        if constexpr (LAST)  // both iterates are whole
            if (k == 2 && !ppr_rows<KS>(B, J, C, R)) return false;
    }
    // the slice's last iterate was written by sweep `last`: into X1 when odd
    if (last & 1)
        for (int64_t i = gthread; i < n * KS; i += nthreads) {
            const int64_t o = (i / KS) * ld + J.c0 + (i % KS);
            J.X0[o] = __ldcg(J.X1 + o);
        }
    if (J.pend) {
        if (!grid_sync(B.sync, gridDim.x)) return false;
        // the packed columns' results back into the graph's iterates
        for (int64_t i = gthread; i < n * KS; i += nthreads) {
            const int64_t v = i / KS;
            const int c = (int)(i % KS);
            if (c < J.cnt) G.X0[v * K + C.col[c]] = __ldcg(J.X0 + v * ld + c);
        }
    }
    if (gthread == 0) {
        // packed columns: their own counts (written by this block's threads before the last block barrier)
        int most = J.pend ? 0 : last;
        for (int c = 0; J.pend && c < J.cnt; ++c) most = max(most, B.iters_done[J.graph * K + C.col[c]]);
        B.counters[0] = max(B.counters[0], most);
    }
    return grid_sync(B.sync, gridDim.x);  // the next job reuses part and res_acc
}

// Packed jobs over a list of columns, up to 32 of one graph at a time (the list
// is in job order, so a graph's columns are adjacent).  Few columns take a
// narrow job, whose sweeps gather 16 or 32 bytes per edge instead of 128 (R-MAT
// 2^17: 97 us a sweep of 32 columns): one slow column can need five times the
// sweeps of the others.
template <int KS, bool LAST = false>
__device__ bool ppr_packed(const BatchDev &B, const BPend *list, int count, int leave, BPend *next, int32_t *next_count,
                           PCols &C) {
    for (int i = 0; i < count;) {
        const int g = list[i].graph;
        int j = i + 1;
        while (j < count && j - i < KS && list[j].graph == g) ++j;
        const PView J = {g, B.XP0, B.XP1, KS, 0, list + i, j - i, leave, next, next_count};
        if (!ppr_job<KS, LAST>(B, J, C)) return false;
        i = j;
    }
    return true;
}

__global__ void __launch_bounds__(BT_THREADS, GP_BT_MINB) k_ppr_persistent(const __grid_constant__ BatchDev B) {
    __shared__ PCols C;
    for (int ji = 0; ji < B.njobs; ++ji) {
        const BJob Jb = B.jobs[ji];
        const BGraph &G = B.graphs[Jb.graph];
        const PView J = {Jb.graph, G.X0, G.X1, B.K, Jb.c0, nullptr, 0, B.pack_max, B.pend, B.counters + 2};
        bool ok;
        switch (Jb.kpl) {
            case 1: ok = ppr_job<32>(B, J, C); break;
            case 2: ok = ppr_job<64>(B, J, C); break;
            default: ok = ppr_job<128>(B, J, C); break;
        }
        if (!ok) return;
    }
    // the columns the jobs left, 32 to a job; what those leave 8 to a job, then 4, and the
    // slow last one of each of these on the rows that they reach
    const int64_t most = (int64_t)B.ngraphs * B.K;
    volatile int32_t *count = B.counters;
    if (!ppr_packed<32>(B, B.pend, count[2], 8, B.pend + most, B.counters + 3, C)) return;
    if (!ppr_packed<8>(B, B.pend + most, count[3], 4, B.pend + 2 * most, B.counters + 4, C)) return;
    if (!ppr_packed<4>(B, B.pend + 2 * most, count[4], 1, B.pend, B.counters + 7, C)) return;
    ppr_packed<4, true>(B, B.pend, count[7], 0, nullptr, nullptr, C);
}

// ------------------------------------------------------------------ batched multi-source BFS

// Latency-bound: few bytes per level, so what counts is the longest chain of
// dependent loads.  Lists above big_min edges are cut in chunks that warps over
// the whole grid take (one warp walking a hub's 25K edges, 32 at a time, set the
// time of a level), and every list is read BF_U edges at a time.
constexpr int BF_U = 4;

// Top-down over the edges [b, e), from `first`, every `step`: f into the out-neighbours' N.
__device__ __forceinline__ void msbfs_scatter(const BGraph &G, uint64_t f, int64_t first, int64_t e, int step) {
    for (int64_t j = first; j < e; j += BF_U * step) {
        int32_t w[BF_U];
        uint64_t nb[BF_U];
#pragma unroll
        for (int q = 0; q < BF_U; ++q) w[q] = j + q * step < e ? __ldg(G.csr_idx + j + q * step) : -1;
#pragma unroll
        for (int q = 0; q < BF_U; ++q) nb[q] = w[q] >= 0 ? f & ~G.V[w[q]] : 0ull;
#pragma unroll
        for (int q = 0; q < BF_U; ++q)
            if (nb[q]) atomicOr((unsigned long long *)G.N + w[q], (unsigned long long)nb[q]);
    }
}

// All graphs' work of a phase is one range of units (32 vertices, or a chunk)
// that the warps share, so that a batch of small graphs does not line up behind
// its first warps; a unit's graph is found in the prefix sums of their counts.
constexpr int BF_MAX_GRAPHS = 256;

__device__ __forceinline__ int msbfs_graph(const int64_t *prefix, int ng, int64_t unit) {
    int lo = 0, hi = ng;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= unit)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(BT_THREADS) k_msbfs_persistent(BatchDev B) {
    __shared__ int s_dir[BF_MAX_GRAPHS];  // per graph: 0 top-down, 1 bottom-up for the current level
    __shared__ int64_t s_tile[BF_MAX_GRAPHS + 1], s_out[BF_MAX_GRAPHS + 1], s_in[BF_MAX_GRAPHS + 1];
    __shared__ unsigned long long s_count[BF_MAX_GRAPHS][4];
    const int64_t gthread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const int64_t gwarp = gthread >> 5, nwarps = nthreads >> 5;
    const int lane = lane_id();
    const int nsrc = B.nsrc;
    const uint64_t full = nsrc == 64 ? ~0ull : ((1ull << nsrc) - 1ull);
    const int ng = B.ngraphs;
    for (int gi = threadIdx.x; gi < ng; gi += blockDim.x) {
        s_tile[gi + 1] = (B.graphs[gi].n + 31) >> 5;
        s_out[gi + 1] = B.graphs[gi].nochunk;
        s_in[gi + 1] = B.graphs[gi].nchunk;
        s_dir[gi] = 0;  // a few sources: top-down
        for (int q = 0; q < 4; ++q) s_count[gi][q] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        s_tile[0] = s_out[0] = s_in[0] = 0;
        for (int gi = 0; gi < ng; ++gi) {
            s_tile[gi + 1] += s_tile[gi];
            s_out[gi + 1] += s_out[gi];
            s_in[gi + 1] += s_in[gi];
        }
    }
    __syncthreads();
    const int64_t ntiles = s_tile[ng];
    for (int64_t u = gwarp; u < ntiles; u += nwarps) {
        const int gi = msbfs_graph(s_tile, ng, u);
        const BGraph &G = B.graphs[gi];
        const int64_t v = (u - s_tile[gi]) * 32 + lane;
        if (v >= G.n) continue;
        G.F[v] = 0;
        G.V[v] = 0;
        G.N[v] = 0;
    }
    if (gthread < 8 * (int64_t)ng) B.mcount[gthread] = 0;
    if (!grid_sync(B.sync, gridDim.x)) return;
    for (int64_t i = gthread; i < (int64_t)ng * 64; i += nthreads) {  // a thread per search
        const int j = (int)(i & 63);
        if (j >= nsrc) continue;
        const BGraph &G = B.graphs[i >> 6];
        const int32_t s = B.sources[i];
        atomicOr((unsigned long long *)G.F + s, 1ull << j);
        atomicOr((unsigned long long *)G.V + s, 1ull << j);
        B.lev_out[i >> 6][(int64_t)s * 64 + j] = 0;
    }
    if (!grid_sync(B.sync, gridDim.x)) return;
    int L = 0;
    for (;; ++L) {
        // light vertices, a lane each.  Top-down: a frontier vertex's masks into its
        // out-neighbours' N; bottom-up: the in-neighbours' masks, until covered
        for (int64_t u = gwarp; u < ntiles; u += nwarps) {
            const int gi = msbfs_graph(s_tile, ng, u);
            const BGraph &G = B.graphs[gi];
            const int64_t v = (u - s_tile[gi]) * 32 + lane;
            if (v >= G.n) continue;
            if (s_dir[gi] == 0) {
                const uint64_t f = G.F[v];
                if (!f) continue;
                const int64_t b = G.csr_off[v], e = G.csr_off[v + 1];
                if (e - b <= B.big_min) msbfs_scatter(G, f, b, e, 1);
            } else {
                const uint64_t vis = G.V[v];
                if (vis == full) continue;
                const int64_t b = G.csc_off[v], e = G.csc_off[v + 1];
                if (e - b > B.big_min) continue;
                uint64_t acc = 0;
                for (int64_t j = b; j < e && (acc | vis) != full; j += BF_U) {
                    int32_t w[BF_U];
#pragma unroll
                    for (int q = 0; q < BF_U; ++q) w[q] = j + q < e ? __ldg(G.csc_idx + j + q) : -1;
#pragma unroll
                    for (int q = 0; q < BF_U; ++q) acc |= w[q] >= 0 ? G.F[w[q]] : 0ull;
                }
                G.N[v] = acc & ~vis;
            }
        }
        // top-down chunks: a lane looks at every nwarps-th one, the warp takes those in the frontier
        for (int64_t c0 = gwarp; c0 < s_out[ng]; c0 += 32 * nwarps) {
            const int64_t c = c0 + lane * nwarps;
            BChunk ch = {0, 0, 0};
            uint64_t f = 0;
            int gi = 0;
            if (c < s_out[ng]) {
                gi = msbfs_graph(s_out, ng, c);
                if (s_dir[gi] == 0) {
                    ch = B.chunks[B.graphs[gi].ochunk0 + (c - s_out[gi])];
                    f = B.graphs[gi].F[ch.v];
                }
            }
            for (unsigned hm = __ballot_sync(FULL, f != 0); hm; hm &= hm - 1) {
                const int hl = __ffs(hm) - 1;
                const uint64_t hf = __shfl_sync(FULL, f, hl);
                const int64_t hb = __shfl_sync(FULL, ch.beg, hl);
                const int len = __shfl_sync(FULL, ch.len, hl);
                msbfs_scatter(B.graphs[__shfl_sync(FULL, gi, hl)], hf, hb + lane, hb + len, 32);
            }
        }
        // bottom-up chunks: what a chunk finds is added to its vertex's N
        for (int64_t c0 = gwarp; c0 < s_in[ng]; c0 += 32 * nwarps) {
            const int64_t c = c0 + lane * nwarps;
            BChunk ch = {0, 0, 0};
            uint64_t vis = full;
            int gi = 0;
            if (c < s_in[ng]) {
                gi = msbfs_graph(s_in, ng, c);
                if (s_dir[gi] == 1) {
                    const BGraph &G = B.graphs[gi];
                    ch = B.chunks[G.chunk0 + (c - s_in[gi])];
                    // (other chunks of the vertex may have found some already: less to look for)
                    vis = G.V[ch.v] | *(volatile uint64_t *)(G.N + ch.v);
                }
            }
            for (unsigned hm = __ballot_sync(FULL, vis != full); hm; hm &= hm - 1) {
                const int hl = __ffs(hm) - 1;
                const BGraph &G = B.graphs[__shfl_sync(FULL, gi, hl)];
                const uint64_t hv = __shfl_sync(FULL, vis, hl);
                const int64_t hb = __shfl_sync(FULL, ch.beg, hl);
                const int64_t he = hb + __shfl_sync(FULL, ch.len, hl);
                uint64_t acc = 0;
                for (int64_t j = hb + lane; j < he; j += 32 * BF_U) {
                    int32_t w[BF_U];
#pragma unroll
                    for (int q = 0; q < BF_U; ++q) w[q] = j + 32 * q < he ? __ldg(G.csc_idx + j + 32 * q) : -1;
#pragma unroll
                    for (int q = 0; q < BF_U; ++q) acc |= w[q] >= 0 ? G.F[w[q]] : 0ull;
                }
                const unsigned lo = __reduce_or_sync(FULL, (unsigned)acc);
                const unsigned hi = __reduce_or_sync(FULL, (unsigned)(acc >> 32));
                acc = (((uint64_t)hi << 32) | lo) & ~hv;
                if (lane == hl && acc) atomicOr((unsigned long long *)G.N + ch.v, (unsigned long long)acc);
            }
        }
        if (!grid_sync(B.sync, gridDim.x)) return;
        // update: owner-only writes of V, F and the levels of newly reached
        // searches, and the counters of the next level's direction rule
        unsigned long long *mc = B.mcount + (L & 1) * 4 * ng;
        for (int64_t u = gwarp; u < ntiles; u += nwarps) {
            const int gi = msbfs_graph(s_tile, ng, u);
            const BGraph &G = B.graphs[gi];
            const int64_t v0 = (u - s_tile[gi]) * 32, v = v0 + lane;
            uint64_t nw = 0;
            unsigned nf = 0, bits = 0;
            unsigned long long mf = 0, mu = 0;
            if (v < G.n) {
                const uint64_t vis = G.V[v], found = G.N[v];
                nw = found & ~vis;
                G.F[v] = nw;
                if (found) G.N[v] = 0;
                if (nw) {
                    G.V[v] = vis | nw;
                    bits = __popcll(nw);
                    nf = 1;
                    mf = (unsigned long long)(G.csr_off[v + 1] - G.csr_off[v]);
                }
                if ((vis | nw) != full) mu = (unsigned long long)(G.csc_off[v + 1] - G.csc_off[v]);
            }
            // a vertex's 64 levels are one row: written by the warp, two searches to a lane
            int32_t *lev = B.lev_out[gi];
            const unsigned rows = __ballot_sync(FULL, nw != 0);
            for (unsigned m = rows; m; m &= m - 1) {
                const int l = __ffs(m) - 1;
                const uint64_t row = __shfl_sync(FULL, nw, l);
                int32_t *at = lev + (v0 + l) * 64 + lane;
                if ((row >> lane) & 1ull) at[0] = L + 1;
                if ((row >> (lane + 32)) & 1ull) at[32] = L + 1;
            }
            if (rows) {
                nf = __reduce_add_sync(FULL, nf);
                bits = __reduce_add_sync(FULL, bits);
                mf = warp_sum(mf);
            }
            mu = warp_sum(mu);
            if (lane == 0) {
                if (rows) {
                    atomicAdd(&s_count[gi][0], (unsigned long long)nf);
                    atomicAdd(&s_count[gi][1], mf);
                    atomicAdd(&s_count[gi][3], (unsigned long long)bits);
                }
                if (mu) atomicAdd(&s_count[gi][2], mu);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 4 * ng; i += blockDim.x) {
            const unsigned long long c = s_count[i >> 2][i & 3];
            if (c) {
                atomicAdd(mc + i, c);
                s_count[i >> 2][i & 3] = 0;
            }
        }
        if (!grid_sync(B.sync, gridDim.x)) return;
        // every block reads the same counters: next directions, and whether any search moved
        unsigned long long moved = 0;
        const volatile unsigned long long *vmc = mc;
        for (int gi = threadIdx.x; gi < ng; gi += blockDim.x) {
            const unsigned long long nf = vmc[4 * gi], mf = vmc[4 * gi + 1], mu = vmc[4 * gi + 2];
            moved |= vmc[4 * gi + 3];
            const int64_t n = B.graphs[gi].n;
            if (s_dir[gi] == 0)
                s_dir[gi] = ((float)mf * B.alpha > (float)mu) ? 1 : 0;
            else
                s_dir[gi] = ((float)nf * B.beta < (float)n) ? 0 : 1;
        }
        // the other parity's record, last read two barriers ago, is cleared for the next level
        if (gthread < 4 * (int64_t)ng) B.mcount[((L + 1) & 1) * 4 * ng + gthread] = 0;
        if (!__syncthreads_or(moved != 0)) break;
    }
    // what no search reached (with the levels above, every entry is written once)
    for (int64_t u = gwarp; u < ntiles; u += nwarps) {
        const int gi = msbfs_graph(s_tile, ng, u);
        const BGraph &G = B.graphs[gi];
        const int64_t v0 = (u - s_tile[gi]) * 32, v = v0 + lane;
        int32_t *lev = B.lev_out[gi];
        const uint64_t vis = v < G.n ? G.V[v] : ~0ull;
        for (unsigned m = __ballot_sync(FULL, vis != ~0ull); m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const uint64_t row = __shfl_sync(FULL, vis, l);
            int32_t *at = lev + (v0 + l) * 64 + lane;
            if (!((row >> lane) & 1ull)) at[0] = -1;
            if (!((row >> (lane + 32)) & 1ull)) at[32] = -1;
        }
    }
    if (gthread == 0) B.counters[1] = L + 1;
}

}  // namespace gp

// ================================================================== host side

struct gp_batch {
    int device = 0, num_sms = 0;
    int64_t l2_bytes = 0;
    int ngraphs = 0, K = 0;
    gp_batch_options opt;
    std::vector<gp_graph *> graphs;
    std::vector<gp::BGraph> hg;
    std::vector<gp::BJob> jobs;
    gp::BatchDev dev;
    gp::Arena mem;     // iterates, masks, levels and per-batch records
    gp::Arena layout;  // work lists that depend on the options
    gp::BGraph *dgraphs = nullptr;
    int64_t nbig = 0;  // big vertices of all graphs
    int32_t *seeds = nullptr, *sources = nullptr;
    int32_t *counters = nullptr;
    int32_t *hcounters = nullptr;  // pinned
    int32_t **lev_out = nullptr;   // device table of the levels' destinations
    int32_t **hlev_out = nullptr;  // pinned: the call's, before they are copied there
    cudaStream_t home = nullptr;
    cudaGraphExec_t ppr_exec = nullptr, bfs_exec = nullptr;
    bool ppr_stale = true, bfs_stale = true;
    int ppr_iters = -1, bfs_nsrc = -1;
    double ppr_tol = -1.0;
    float ppr_d = -1.f;
    int grid = 0;
};

namespace gp {

static int batch_grid(gp_batch *b, const void *kernel, int &grid) {
    int per_sm = 0;
    GP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, BT_THREADS, 0));
    if (per_sm < 1) return set_error(GP_ERR_UNSUPPORTED, "batched kernel does not fit on an SM");
    grid = per_sm * b->num_sms;
    return GP_OK;
}

// Launch (or capture into a CUDA graph and replay) the cooperative kernel.
static int coop_launch(gp_batch *b, const void *kernel, cudaGraphExec_t &exec, bool rebuild, cudaStream_t s) {
    if (rebuild && exec) {
        cudaGraphExecDestroy(exec);
        exec = nullptr;
    }
    if (!exec) {
        cudaStream_t cap;
        GP_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) e = cudaMemsetAsync(b->dev.sync, 0, sizeof(GridSync), cap);
        if (e == cudaSuccess) e = cudaMemsetAsync(b->counters, 0, 8 * sizeof(int32_t), cap);
        if (e == cudaSuccess && b->nbig) e = cudaMemsetAsync(b->dev.bdone, 0, b->nbig * sizeof(unsigned), cap);
        if (e == cudaSuccess) {
            cudaLaunchConfig_t cfg;
            memset(&cfg, 0, sizeof(cfg));
            cfg.gridDim = dim3((unsigned)b->grid);
            cfg.blockDim = dim3(BT_THREADS);
            cfg.stream = cap;
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeCooperative;
            attr.val.cooperative = 1;
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            void *args[] = {&b->dev};
            e = cudaLaunchKernelExC(&cfg, kernel, args);
        }
        cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
        if (e == cudaSuccess) e = e2;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        cudaStreamDestroy(cap);
        if (e != cudaSuccess) {
            cudaGetLastError();
            exec = nullptr;
            return set_error(GP_ERR_CUDA, "capturing the batched launch: %s", cudaGetErrorString(e));
        }
    }
    GP_CUDA(cudaGraphLaunch(exec, s));
    return GP_OK;
}

// Edges per chunk of a graph of m edges: the option's, halved while that leaves
// a warp of the grid without a chunk's worth of edges (a chunk's windows of loads
// follow one another: at 128 edges they are a small graph's whole sweep).
static int64_t chunk_size(const gp_batch *b, int64_t m) {
    const int64_t warps = (int64_t)b->num_sms * GP_BT_MINB * (BT_THREADS / 32);
    int64_t c = b->opt.chunk_edges;
    while (c >= 64 && c * warps > m) c /= 2;
    return c;
}

// Work lists for the current options: big in-degree vertices and their chunks,
// big out-degree vertices, and the PPR jobs (column slices sized to the L2
// budget).  Reads the offsets once; synchronises the stream.  Where something
// fails the batch keeps the lists it had.
static int batch_layout(gp_batch *b, cudaStream_t s) {
    const int K = b->K;
    const int64_t big_min = b->opt.big_in_degree;
    int32_t nbig = 0;
    std::vector<int64_t> bcstart(1, 0);
    std::vector<BChunk> chunks;
    int64_t max_chunks = 1;
    std::vector<BJob> jobs;
    std::vector<BGraph> hg = b->hg;
    const int64_t budget = (int64_t)b->opt.l2_budget_mb << 20;
    for (int gi = 0; gi < b->ngraphs; ++gi) {
        gp_graph *g = b->graphs[gi];
        std::vector<int64_t> off((size_t)g->n + 1);
        cudaError_t e = cudaMemcpyAsync(off.data(), g->csc_off, off.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return set_error(GP_ERR_CUDA, "batch layout: %s", cudaGetErrorString(e));
        const int64_t C = chunk_size(b, g->m);
        BGraph &G = hg[gi];
        G.chunk0 = (int64_t)chunks.size();
        for (int64_t v = 0; v < g->n; ++v) {
            const int64_t d = off[v + 1] - off[v];
            if (d <= big_min) continue;
            const int32_t r = nbig++, nch = (int32_t)((d + C - 1) / C);
            for (int64_t p = off[v]; p < off[v + 1]; p += C)
                chunks.push_back(BChunk{p, (int32_t)std::min<int64_t>(C, off[v + 1] - p), (int32_t)v, r, nch});
            bcstart.push_back((int64_t)chunks.size());
        }
        G.nchunk = (int64_t)chunks.size() - G.chunk0;
        max_chunks = std::max(max_chunks, G.nchunk);
        G.ochunk0 = G.chunk0;
        G.nochunk = G.nchunk;
        // the widest slice whose two iterates fit the budget (at least 32 columns)
        int ks = std::min(K, BT_MAX_KS);
        while (ks > 32 && 2 * g->n * (int64_t)ks * 4 > budget) ks /= 2;
        for (int c0 = 0; c0 < K; c0 += ks) jobs.push_back(BJob{gi, c0, ks / 32, 0});
    }
    // after every graph's in-edge chunks (bcstart numbers those): the out-edge ones where the orders differ
    for (int gi = 0; gi < b->ngraphs; ++gi) {
        gp_graph *g = b->graphs[gi];
        if (g->csr_off == g->csc_off) continue;
        std::vector<int64_t> off((size_t)g->n + 1);
        cudaError_t e = cudaMemcpyAsync(off.data(), g->csr_off, off.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return set_error(GP_ERR_CUDA, "batch layout: %s", cudaGetErrorString(e));
        const int64_t C = chunk_size(b, g->m);
        BGraph &G = hg[gi];
        G.ochunk0 = (int64_t)chunks.size();
        for (int64_t v = 0; v < g->n; ++v)
            if (off[v + 1] - off[v] > big_min)
                for (int64_t p = off[v]; p < off[v + 1]; p += C)
                    chunks.push_back(BChunk{p, (int32_t)std::min<int64_t>(C, off[v + 1] - p), (int32_t)v, 0, 0});
        G.nochunk = (int64_t)chunks.size() - G.ochunk0;
    }
    Arena layout;
    BatchDev D = b->dev;
    int64_t *dbc = nullptr;
    BChunk *dch = nullptr;
    BJob *djobs = nullptr;
    int st = GP_OK;
    if (st == GP_OK) st = layout.alloc(dbc, bcstart.size(), s);
    if (st == GP_OK) st = layout.alloc(dch, std::max<size_t>(chunks.size(), 1), s);
    if (st == GP_OK) st = layout.alloc(djobs, jobs.size(), s);
    if (st == GP_OK) st = layout.alloc(D.part, (size_t)max_chunks * K, s);
    if (st == GP_OK) st = layout.alloc(D.bdone, (size_t)std::max(nbig, 1), s);
    if (st != GP_OK) {
        layout.release(s);
        return st;
    }
    cudaError_t e = cudaMemcpyAsync(dbc, bcstart.data(), bcstart.size() * sizeof(int64_t), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && !chunks.empty()) e = cudaMemcpyAsync(dch, chunks.data(), chunks.size() * sizeof(BChunk), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(djobs, jobs.data(), jobs.size() * sizeof(BJob), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b->dgraphs, hg.data(), b->ngraphs * sizeof(BGraph), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        layout.release(s);
        return set_error(GP_ERR_CUDA, "batch layout copy: %s", cudaGetErrorString(e));
    }
    D.big_min = big_min;
    D.bcstart = dbc;
    D.chunks = dch;
    D.jobs = djobs;
    D.njobs = (int)jobs.size();
    D.alpha = b->opt.msbfs_alpha;
    D.beta = b->opt.msbfs_beta;
    D.one_hot_start = b->opt.ppr_start;
    D.pack_max = b->opt.ppr_pack;
    b->dev = D;
    b->nbig = nbig;
    b->hg = std::move(hg);
    b->jobs = std::move(jobs);
    b->layout.release(s);
    b->layout = std::move(layout);
    b->ppr_stale = b->bfs_stale = true;  // captured launches hold the old arguments
    return GP_OK;
}

}  // namespace gp

using namespace gp;

extern "C" int gp_batch_options_default(gp_batch_options *opt) {
    clear_error();
    if (!opt) return set_error(GP_ERR_INVALID, "gp_batch_options_default: NULL");
    memset(opt, 0, sizeof(*opt));
    opt->big_in_degree = 32;
    opt->chunk_edges = 128;
    opt->l2_budget_mb = 128;
    opt->msbfs_alpha = 16.0f;
    opt->msbfs_beta = 24.0f;
    opt->ppr_start = 1;
    opt->ppr_pack = 16;
    return GP_OK;
}

extern "C" int gp_batch_create(gp_batch **out, gp_graph *const *graphs, int ngraphs, int k_ppr, void *stream) {
    clear_error();
    if (!out) return set_error(GP_ERR_INVALID, "gp_batch_create: out is NULL");
    *out = nullptr;
    if (!graphs || ngraphs < 1) return set_error(GP_ERR_INVALID, "gp_batch_create: need at least one graph");
    if (ngraphs > 256) return set_error(GP_ERR_INVALID, "gp_batch_create: at most 256 graphs");
    if (k_ppr != 32 && k_ppr != 64 && k_ppr != 128 && k_ppr != 256)
        return set_error(GP_ERR_INVALID, "gp_batch_create: k_ppr must be 32, 64, 128 or 256");
    for (int i = 0; i < ngraphs; ++i)
        if (!graphs[i] || graphs[i]->n < 1) return set_error(GP_ERR_INVALID, "gp_batch_create: graph %d empty or NULL", i);
    cudaStream_t s = (cudaStream_t)stream;
    gp_batch *b = new gp_batch();
    b->home = s;
    b->ngraphs = ngraphs;
    b->K = k_ppr;
    b->graphs.assign(graphs, graphs + ngraphs);
    gp_batch_options_default(&b->opt);
    auto fail = [&](int st) {
        b->layout.release(s);
        b->mem.release(s);
        pinned_free(b->hcounters, 8 * sizeof(int32_t));
        pinned_free(b->hlev_out, ngraphs * sizeof(int32_t *));
        delete b;
        return st;
    };
    {
        cudaError_t e = cudaGetDevice(&b->device);
        int l2 = 0;
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->num_sms, cudaDevAttrMultiProcessorCount, b->device);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, b->device);
        if (e != cudaSuccess) return fail(set_error(GP_ERR_CUDA, "gp_batch_create: %s", cudaGetErrorString(e)));
        b->l2_bytes = l2;
    }
    b->hg.resize(ngraphs);
    const int K = k_ppr;
    BatchDev &D = b->dev;
    memset(&D, 0, sizeof(D));
    D.ngraphs = ngraphs;
    D.K = K;
    int st = GP_OK;
    int64_t nmax = 1;
    for (int gi = 0; gi < ngraphs && st == GP_OK; ++gi) {
        gp_graph *g = graphs[gi];
        nmax = std::max(nmax, g->n);
        BGraph &G = b->hg[gi];
        memset(&G, 0, sizeof(G));
        G.n = g->n;
        G.csc_off = g->csc_off;
        G.csc_idx = g->csc_idx;
        G.csc_w = g->csc_w;
        G.csr_off = g->csr_off;
        G.csr_idx = g->csr_idx;
        G.inv_deg = g->inv_deg;
        const size_t n = (size_t)G.n;
        if (st == GP_OK) st = b->mem.alloc(G.X0, n * K, s);
        if (st == GP_OK) st = b->mem.alloc(G.X1, n * K, s);
        if (st == GP_OK) st = b->mem.alloc(G.F, n, s);
        if (st == GP_OK) st = b->mem.alloc(G.V, n, s);
        if (st == GP_OK) st = b->mem.alloc(G.N, n, s);
        if (st == GP_OK) st = b->mem.alloc(G.levels, n * 64, s);
    }
    if (st == GP_OK) st = b->mem.alloc(b->dgraphs, (size_t)ngraphs, s);
    if (st == GP_OK) st = b->mem.alloc(D.res_acc, (size_t)3 * K, s);
    if (st == GP_OK) st = b->mem.alloc(b->seeds, (size_t)ngraphs * K, s);
    if (st == GP_OK) st = b->mem.alloc(b->sources, (size_t)ngraphs * 64, s);
    if (st == GP_OK) st = b->mem.alloc(D.iters_done, (size_t)ngraphs * K, s);
    if (st == GP_OK) st = b->mem.alloc(b->counters, 8, s);
    if (st == GP_OK) st = b->mem.alloc(D.mcount, (size_t)ngraphs * 8, s);
    if (st == GP_OK) st = b->mem.alloc(D.pend, (size_t)3 * ngraphs * K, s);
    if (st == GP_OK) st = b->mem.alloc(D.XP0, (size_t)nmax * 32, s);
    if (st == GP_OK) st = b->mem.alloc(D.XP1, (size_t)nmax * 32, s);
    if (st == GP_OK) st = b->mem.alloc(b->lev_out, (size_t)ngraphs, s);
    GridSync *sync = nullptr;
    if (st == GP_OK) st = b->mem.alloc(sync, 1, s);
    if (st != GP_OK) return fail(st);
    {
        void *h = nullptr;
        st = pinned_alloc(&h, 8 * sizeof(int32_t));
        if (st != GP_OK) return fail(st);
        b->hcounters = (int32_t *)h;
        st = pinned_alloc(&h, ngraphs * sizeof(int32_t *));
        if (st != GP_OK) return fail(st);
        b->hlev_out = (int32_t **)h;
    }
    D.graphs = b->dgraphs;
    D.seeds = b->seeds;
    D.sources = b->sources;
    D.counters = b->counters;
    D.lev_out = b->lev_out;
    D.sync = sync;
    st = batch_layout(b, s);
    if (st != GP_OK) return fail(st);
    *out = b;
    return GP_OK;
}

extern "C" int gp_batch_set_options(gp_batch *b, const gp_batch_options *opt, void *stream) {
    clear_error();
    if (!b || !opt) return set_error(GP_ERR_INVALID, "gp_batch_set_options: NULL argument");
    if (opt->big_in_degree < 0 || opt->chunk_edges < 32 || opt->chunk_edges > (1 << 20) || opt->l2_budget_mb < 1 ||
        opt->l2_budget_mb > (1 << 20) || !(opt->msbfs_alpha > 0.f) || !(opt->msbfs_beta > 0.f) ||
        (opt->ppr_start != 0 && opt->ppr_start != 1) || opt->ppr_pack < 0 || opt->ppr_pack > BT_MAX_KS)
        return set_error(GP_ERR_INVALID, "gp_batch_set_options: option out of range");
    const gp_batch_options old = b->opt;
    b->opt = *opt;
    if (old.big_in_degree != opt->big_in_degree || old.chunk_edges != opt->chunk_edges ||
        old.l2_budget_mb != opt->l2_budget_mb) {
        const int st = batch_layout(b, (cudaStream_t)stream);
        if (st != GP_OK) b->opt = old;
        return st;
    }
    b->dev.alpha = opt->msbfs_alpha;
    b->dev.beta = opt->msbfs_beta;
    b->dev.one_hot_start = opt->ppr_start;
    b->dev.pack_max = opt->ppr_pack;
    b->bfs_stale = b->ppr_stale = true;
    return GP_OK;
}

extern "C" int gp_batch_get_options(const gp_batch *b, gp_batch_options *opt) {
    clear_error();
    if (!b || !opt) return set_error(GP_ERR_INVALID, "gp_batch_get_options: NULL argument");
    *opt = b->opt;
    return GP_OK;
}

extern "C" int gp_batch_free(gp_batch *b) {
    clear_error();
    if (!b) return GP_OK;
    cudaDeviceSynchronize();
    if (b->ppr_exec) cudaGraphExecDestroy(b->ppr_exec);
    if (b->bfs_exec) cudaGraphExecDestroy(b->bfs_exec);
    b->layout.release(b->home);
    b->mem.release(b->home);
    pinned_free(b->hcounters, 8 * sizeof(int32_t));
    pinned_free(b->hlev_out, b->ngraphs * sizeof(int32_t *));
    cudaError_t e = cudaStreamSynchronize(b->home);
    delete b;
    if (e != cudaSuccess) return set_error(GP_ERR_CUDA, "gp_batch_free: %s", cudaGetErrorString(e));
    return GP_OK;
}

extern "C" int gp_ppr_batched(gp_batch *b, const int32_t *seeds, float damping, int iters, double tol, float *const *out,
                              int32_t *iters_done, gp_batch_stats *stats, void *stream) {
    clear_error();
    if (!b || !seeds) return set_error(GP_ERR_INVALID, "gp_ppr_batched: NULL argument");
    if (!(damping > 0.f && damping < 1.f)) return set_error(GP_ERR_INVALID, "damping %g outside (0, 1)", (double)damping);
    if (iters < 1 || !(tol >= 0.0)) return set_error(GP_ERR_INVALID, "gp_ppr_batched: iters >= 1 and tol >= 0 required");
    cudaStream_t s = (cudaStream_t)stream;
    const int K = b->K;
    for (int gi = 0; gi < b->ngraphs; ++gi)
        for (int j = 0; j < K; ++j) {
            const int32_t v = seeds[(size_t)gi * K + j];
            if (v < 0 || (int64_t)v >= b->hg[gi].n)
                return set_error(GP_ERR_INVALID, "seed %d of graph %d outside [0, n)", v, gi);
        }
    if (stats) memset(stats, 0, sizeof(*stats));
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (stats) {
        GP_CUDA(cudaEventCreate(&ev0));
        GP_CUDA(cudaEventCreate(&ev1));
    }
    GP_CUDA(cudaMemcpyAsync(b->seeds, seeds, (size_t)b->ngraphs * K * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    bool other_weights = false;  // since the batch was made, or the last call
    for (int gi = 0; gi < b->ngraphs; ++gi) {
        other_weights |= b->hg[gi].csc_w != b->graphs[gi]->csc_w;
        b->hg[gi].csc_w = b->graphs[gi]->csc_w;
    }
    if (other_weights)
        GP_CUDA(cudaMemcpyAsync(b->dgraphs, b->hg.data(), b->ngraphs * sizeof(BGraph), cudaMemcpyHostToDevice, s));
    const void *kernel = (const void *)k_ppr_persistent;
    const bool rebuild = b->ppr_stale || b->ppr_iters != iters || b->ppr_tol != tol || b->ppr_d != damping;
    if (rebuild) {
        GP_TRY(batch_grid(b, kernel, b->grid));
        b->dev.d = damping;
        b->dev.one_minus_d = 1.0f - damping;
        b->dev.tol = tol;
        b->dev.iters = iters;
        b->ppr_iters = iters;
        b->ppr_tol = tol;
        b->ppr_d = damping;
        b->ppr_stale = false;
    }
    if (stats) GP_CUDA(cudaEventRecord(ev0, s));
    GP_TRY(coop_launch(b, kernel, b->ppr_exec, rebuild, s));
    if (stats) GP_CUDA(cudaEventRecord(ev1, s));
    for (int gi = 0; gi < b->ngraphs; ++gi)
        if (out && out[gi])
            GP_CUDA(cudaMemcpyAsync(out[gi], b->hg[gi].X0, (size_t)b->hg[gi].n * K * sizeof(float), cudaMemcpyDefault, s));
    if (iters_done)
        GP_CUDA(cudaMemcpyAsync(iters_done, b->dev.iters_done, (size_t)b->ngraphs * K * sizeof(int32_t), cudaMemcpyDefault, s));
    GP_CUDA(cudaMemcpyAsync(b->hcounters, b->counters, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    GridSync hs;
    GP_CUDA(cudaMemcpyAsync(&hs, b->dev.sync, sizeof(hs), cudaMemcpyDeviceToHost, s));
    GP_CUDA(cudaStreamSynchronize(s));
    if (stats) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev0, ev1);
        cudaEventDestroy(ev0);
        cudaEventDestroy(ev1);
        stats->sweeps = b->hcounters[0];
        stats->ms = ms;
        stats->blocks = b->grid;
        stats->jobs = (int32_t)b->jobs.size();
        stats->packed = b->hcounters[2];
    }
    if (hs.err) return set_error(GP_ERR_TIMEOUT, "batched PageRank: a grid barrier wait ran out");
    return GP_OK;
}

extern "C" int gp_msbfs_batched(gp_batch *b, const int32_t *sources, int nsrc, int32_t *const *levels_out,
                                gp_batch_stats *stats, void *stream) {
    clear_error();
    if (!b || !sources) return set_error(GP_ERR_INVALID, "gp_msbfs_batched: NULL argument");
    if (nsrc < 1 || nsrc > 64) return set_error(GP_ERR_INVALID, "gp_msbfs_batched: nsrc %d outside [1, 64]", nsrc);
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<int32_t> src((size_t)b->ngraphs * 64, 0);
    for (int gi = 0; gi < b->ngraphs; ++gi)
        for (int j = 0; j < nsrc; ++j) {
            const int32_t v = sources[(size_t)gi * nsrc + j];
            if (v < 0 || (int64_t)v >= b->hg[gi].n)
                return set_error(GP_ERR_INVALID, "source %d of graph %d outside [0, n)", v, gi);
            src[(size_t)gi * 64 + j] = v;
        }
    if (stats) memset(stats, 0, sizeof(*stats));
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (stats) {
        GP_CUDA(cudaEventCreate(&ev0));
        GP_CUDA(cudaEventCreate(&ev1));
    }
    GP_CUDA(cudaMemcpyAsync(b->sources, src.data(), src.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    // device outputs are written by the kernel, the others copied from the batch's own buffers
    for (int gi = 0; gi < b->ngraphs; ++gi)
        b->hlev_out[gi] = levels_out && levels_out[gi] && is_device_ptr(levels_out[gi]) ? levels_out[gi] : b->hg[gi].levels;
    GP_CUDA(cudaMemcpyAsync(b->lev_out, b->hlev_out, b->ngraphs * sizeof(int32_t *), cudaMemcpyHostToDevice, s));
    const bool rebuild = b->bfs_stale || b->bfs_nsrc != nsrc;
    int grid = 0;
    GP_TRY(batch_grid(b, (const void *)k_msbfs_persistent, grid));
    const int saved = b->grid;
    b->grid = grid;
    b->dev.nsrc = nsrc;
    b->bfs_nsrc = nsrc;
    b->bfs_stale = false;
    if (stats) GP_CUDA(cudaEventRecord(ev0, s));
    int st = coop_launch(b, (const void *)k_msbfs_persistent, b->bfs_exec, rebuild, s);
    b->grid = saved;
    GP_TRY(st);
    if (stats) GP_CUDA(cudaEventRecord(ev1, s));
    for (int gi = 0; gi < b->ngraphs; ++gi)
        if (levels_out && levels_out[gi] && b->hlev_out[gi] == b->hg[gi].levels)
            GP_CUDA(cudaMemcpyAsync(levels_out[gi], b->hg[gi].levels, (size_t)b->hg[gi].n * 64 * sizeof(int32_t),
                                    cudaMemcpyDefault, s));
    GP_CUDA(cudaMemcpyAsync(b->hcounters, b->counters, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    GridSync hs;
    GP_CUDA(cudaMemcpyAsync(&hs, b->dev.sync, sizeof(hs), cudaMemcpyDeviceToHost, s));
    GP_CUDA(cudaStreamSynchronize(s));
    if (stats) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev0, ev1);
        cudaEventDestroy(ev0);
        cudaEventDestroy(ev1);
        stats->levels = b->hcounters[1];
        stats->ms = ms;
        stats->blocks = grid;
        stats->jobs = (int32_t)b->jobs.size();
    }
    if (hs.err) return set_error(GP_ERR_TIMEOUT, "batched BFS: a grid barrier wait ran out");
    return GP_OK;
}

// ------------------------------------------------------------------ tuning

namespace gp {

// Device time of one batched call (a warm-up call first: a changed option
// re-captures the launch).
static int time_ppr(gp_batch *b, const int32_t *seeds, int sweeps, cudaStream_t s, float &ms) {
    gp_batch_stats st;
    GP_TRY(gp_ppr_batched(b, seeds, 0.85f, sweeps, 0.0, nullptr, nullptr, &st, s));
    GP_TRY(gp_ppr_batched(b, seeds, 0.85f, sweeps, 0.0, nullptr, nullptr, &st, s));
    ms = st.ms;
    return GP_OK;
}

static int time_msbfs(gp_batch *b, const int32_t *sources, int nsrc, cudaStream_t s, float &ms) {
    gp_batch_stats st;
    GP_TRY(gp_msbfs_batched(b, sources, nsrc, nullptr, &st, s));
    GP_TRY(gp_msbfs_batched(b, sources, nsrc, nullptr, &st, s));
    ms = st.ms;
    return GP_OK;
}

}  // namespace gp

extern "C" int gp_batch_autotune(gp_batch *b, const int32_t *seeds, const int32_t *sources, int nsrc, int ppr_sweeps,
                                 gp_batch_tune_result *res, void *stream) {
    clear_error();
    if (!b || !res) return set_error(GP_ERR_INVALID, "gp_batch_autotune: NULL argument");
    if (ppr_sweeps < 1) return set_error(GP_ERR_INVALID, "gp_batch_autotune: ppr_sweeps must be >= 1");
    if (sources && (nsrc < 1 || nsrc > 64)) return set_error(GP_ERR_INVALID, "gp_batch_autotune: nsrc outside [1, 64]");
    cudaStream_t s = (cudaStream_t)stream;
    memset(res, 0, sizeof(*res));
    gp_batch_options best = b->opt;
    int trials = 0;
    // coordinate descent, each axis over its candidates with the others fixed
    auto axis_i32 = [&](int32_t gp_batch_options::*field, std::initializer_list<int32_t> cands, bool ppr,
                        float &best_ms) -> int {
        for (int32_t c : cands) {
            gp_batch_options o = best;
            o.*field = c;
            GP_TRY(gp_batch_set_options(b, &o, stream));
            float ms = 0.f;
            if (ppr)
                GP_TRY(time_ppr(b, seeds, ppr_sweeps, s, ms));
            else
                GP_TRY(time_msbfs(b, sources, nsrc, s, ms));
            ++trials;
            if (best_ms <= 0.f || ms < best_ms) {
                best_ms = ms;
                best = o;
            }
        }
        return gp_batch_set_options(b, &best, stream);
    };
    auto axis_f32 = [&](float gp_batch_options::*field, std::initializer_list<float> cands, float &best_ms) -> int {
        for (float c : cands) {
            gp_batch_options o = best;
            o.*field = c;
            GP_TRY(gp_batch_set_options(b, &o, stream));
            float ms = 0.f;
            GP_TRY(time_msbfs(b, sources, nsrc, s, ms));
            ++trials;
            if (best_ms <= 0.f || ms < best_ms) {
                best_ms = ms;
                best = o;
            }
        }
        return gp_batch_set_options(b, &best, stream);
    };
    float ppr_ms = 0.f, bfs_ms = 0.f;
    if (seeds) {
        GP_TRY(axis_i32(&gp_batch_options::big_in_degree, {8, 16, 32, 64, 128}, true, ppr_ms));
        GP_TRY(axis_i32(&gp_batch_options::chunk_edges, {64, 128, 256}, true, ppr_ms));
        GP_TRY(axis_i32(&gp_batch_options::l2_budget_mb, {48, 64, 96, 128, 192}, true, ppr_ms));
    }
    if (sources) {
        GP_TRY(axis_f32(&gp_batch_options::msbfs_alpha, {2.f, 4.f, 8.f, 16.f, 32.f, 64.f}, bfs_ms));
        GP_TRY(axis_f32(&gp_batch_options::msbfs_beta, {8.f, 24.f, 64.f}, bfs_ms));
    }
    res->options = best;
    res->ppr_ms = ppr_ms;
    res->msbfs_ms = bfs_ms;
    res->trials = trials;
    return GP_OK;
}
