// pagerank.cu -- push and pull PageRank sweeps and the gp_pagerank driver.
//
// One sweep computes (Section 3.1 formula; Algorithm 1, push- and pull-based PR)
//     y[v] = (1-d) s[v] + d * sum_{(u->v)} P_vu x[u]
// from the contribution vector c[u] = x[u] * inv_deg[u] (so the gather never
// fetches a neighbour's degree, the extra cost of pulling named in Section 7.3)
// and edge factor w_uv (1 when unweighted).
//
// Pull (owner-only writes, no atomics; Section 4.1 "Atomics/Locks"):
//   k_pull_tiles  -- the edge list in tiles of 256 consecutive edges, one warp
//                    each, whatever the vertices' degrees; a segmented warp sum
//                    (Section 4's CREW binary merge-tree) gives one partial per
//                    row and tile.
//   k_pull_finish -- one thread per row adds its tiles' partials (a warp where
//                    the row spans many) and writes the vertex's y,
//                    c' = y*inv_deg and |y - x|; every vertex has one writer.
// Push (scatter with atomics; Section 4.1: O(Lm) write conflicts):
//   k_push_tiles     -- each source adds d*c[u]*w_uv into y[v] for its
//                       out-edges with atomics (RED), over tiles of the
//                       out-edge list like the pull's.
//   k_push_epilogue  -- per vertex: residual, c' and the (1-d)s reset of the
//                       buffer the next sweep accumulates into.
// Convergence (not in the paper, which runs a fixed L): the L1 residual is
// reduced in FP64 per block; the first kernel of the next sweep reduces the
// block partials (every block, same order, so all agree) and stops the
// iteration on the device, so the host only polls every few sweeps.
#include <algorithm>
#include <cmath>

#include "gp_internal.cuh"

namespace gp {

struct PrStatus {
    int32_t done;
    int32_t iters_done;
    double residual;
    int32_t converged;
    int32_t pad;
    // push scatter, summed over the sweeps of a call: updates sent to L2 as
    // atomics, added into a block's shared-memory accumulators, and folded into
    // another lane's update inside a warp; plus the flushes of the shared ones
    unsigned long long upd_l2, upd_shared, upd_merged, flush_l2;
};

struct PrArgs {
    int64_t n;
    const int64_t *off;  // CSC (pull) or CSR (push) offsets
    const int32_t *idx;
    const float *w;      // edge factors in the same order, or nullptr
    const float *inv_deg;
    // big-vertex chunks
    const int32_t *big;
    const int64_t *cstart;
    const Chunk *chunks;
    int64_t nbig, nchunks;
    int32_t light_max;
    // vectors
    const float *x;  // previous iterate
    float *y;        // new iterate
    const float *c;  // contributions of x
    float *c_next;   // contributions of y (pull)
    const float *s;  // teleport vector (forward) or dL/dx (adjoint), or nullptr
    float s_scale;       // factor of s in the base term: 1-d (forward), 1 (adjoint)
    float base_uniform;  // base term when s is nullptr: (1-d)/n
    const float *post_scale;  // factor of the gathered sum per owner (adjoint: inv_deg), or nullptr
    const float *cmul;        // c_next = y * cmul (forward: inv_deg), or nullptr (c_next = y)
    float d;
    double tol;
    int32_t k;  // sweep number, 1-based
    int32_t nprev;
    double *partials;
    double *acc64;  // FP64 push accumulator (or nullptr)
    float *c_hot;   // hot contributions (pull, HOT kernels)
    const int32_t *hot_id;  // hot vertices (push HOT kernels)
    const uint32_t *hot_bits;    // pull: which vertices are hot, and
    const int32_t *hot_prefix;   // the slot of the first hot vertex of each word
    int64_t nhot;
    // pull: the edge tiles (see EdgeTiles)
    const uint8_t *heads;
    const int32_t *tile_row, *rows, *long_rows;
    float *acc, *carry;
    float *chunk_part;     // adjoint pull: the long rows' chunk sums
    int32_t split_blocks;  // adjoint pull: blocks of short rows (the others add the long rows' chunks)
    int64_t m, ntiles, nrows, nlong;
    int32_t vec_tiles;  // the leading tiles that may be read 32 bytes at a time: full, arrays on 32-byte boundaries
    PrStatus *status;
};

__device__ __forceinline__ float base_term(const PrArgs &a, int64_t v) {
    return a.s ? a.s_scale * a.s[v] : a.base_uniform;
}
__device__ __forceinline__ float post_factor(const PrArgs &a, int64_t v) { return a.post_scale ? a.post_scale[v] : 1.f; }
__device__ __forceinline__ float c_factor(const PrArgs &a, int64_t v) { return a.cmul ? a.cmul[v] : 1.f; }

// Whether the iteration has stopped, read by one thread per block: every warp
// loading the flag itself would queue thousands of requests on the one L2 line
// that holds it at each launch.  Called by all threads of the block.
__device__ __forceinline__ bool pr_stopped(const PrStatus *status) {
    __shared__ int stop;
    if (threadIdx.x == 0) stop = ((volatile const PrStatus *)status)->done;
    __syncthreads();
    return stop != 0;
}

// Convergence gate at the start of sweep k: every block reduces the residual
// partials of sweep k-1 in the same order, so all blocks take the same
// decision; block 0 records it.  Returns true when the iteration has stopped.
// With tol = 0 there is nothing to decide: only the record after the last sweep
// (`record`) reduces them, and the sweeps start 2 us earlier.
__device__ bool pr_gate(const PrArgs &a, int k, bool record = false) {
    __shared__ double sm[32];
    __shared__ int stop;
    volatile PrStatus *st = a.status;
    if (threadIdx.x == 0) stop = st->done;
    __syncthreads();
    if (stop) return true;
    if (k > 1 && (a.tol > 0.0 || record)) {
        double r = 0.0;
        for (int i = threadIdx.x; i < a.nprev; i += blockDim.x) r += a.partials[i];
        r = block_sum(r, sm);
        if (threadIdx.x == 0) {
            const int conv = r < a.tol;
            if (blockIdx.x == 0) {
                st->residual = r;
                st->iters_done = k - 1;
                if (conv) {
                    st->converged = 1;
                    st->done = 1;
                }
            }
            stop = conv;
        }
        __syncthreads();
    }
    return stop != 0;
}

// c_hot[slot of v] = c where v is hot (see HotSet).
__device__ __forceinline__ void store_hot(const uint32_t *bits, const int32_t *prefix, float *c_hot, int64_t v, float c) {
    const uint32_t word = bits[v >> 5], bit = 1u << (v & 31);
    if (word & bit) c_hot[prefix[v >> 5] + __popc(word & (bit - 1u))] = c;
}

// x = x0 (or 1/n), c = x * cmul, and the push accumulators zeroed.
__global__ void k_pr_init(int64_t n, const float *x0, const float *cmul, float *r0, float *c, float *r_push,
                          double *acc64, const uint32_t *hot_bits, const int32_t *hot_prefix, float *c_hot,
                          PrStatus *status, GridSync *sync) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const float x_uniform = 1.0f / (float)n;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const float x = x0 ? x0[v] : x_uniform;
        const float cv = cmul ? x * cmul[v] : x;
        r0[v] = x;
        c[v] = cv;
        if (hot_bits) store_hot(hot_bits, hot_prefix, c_hot, v, cv);
        if (r_push) r_push[v] = 0.f;
        if (acc64) acc64[v] = 0.0;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        status->done = 0;
        status->iters_done = 0;
        status->residual = 0.0;
        status->converged = 0;
        status->upd_l2 = status->upd_shared = status->upd_merged = status->flush_l2 = 0;
        *sync = GridSync();
    }
}

// Records the decision for the last sweep enqueued (sweep k-1) without doing a
// sweep, and writes the status into the host's mapped mirror slot: the host
// polls it with no copy, so polling never waits behind other transfers.
__global__ void k_pr_finish(PrArgs a, PrStatus *mirror) {
    pr_gate(a, a.k, true);
    if (threadIdx.x == 0) {
        *mirror = *a.status;  // the gate ended with a block barrier
        __threadfence_system();
    }
}

// dst = src over n floats (the result's move into the caller's buffer, kept
// off the copy engines for the same reason).
__global__ void k_copy_f32(int64_t n, const float *__restrict__ src, float *__restrict__ dst) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) dst[i] = src[i];
}

// ------------------------------------------------------------------ pull

// Shared-memory copy of the hot contributions (see HotSet): loaded once per
// block, then every gather of a hot vertex is a shared-memory read.
template <bool HOT>
__device__ __forceinline__ void load_hot(const PrArgs &a, float *sh) {
    if (!HOT) return;
    const int64_t nh = a.nhot;
    const float4 *src = reinterpret_cast<const float4 *>(a.c_hot);
    float4 *dst = reinterpret_cast<float4 *>(sh);
    for (int64_t i = threadIdx.x; i < nh / 4; i += blockDim.x) dst[i] = __ldg(src + i);
    for (int64_t i = (nh & ~int64_t(3)) + threadIdx.x; i < nh; i += blockDim.x) sh[i] = __ldg(a.c_hot + i);
    __syncthreads();
}

// LOOP: the contributions are rewritten by the same launch, so they may be kept
// in L1 between barriers but not taken through the read-only path.
template <bool HOT, bool LOOP>
__device__ __forceinline__ float gather_c(const float *c, const float *sh, int32_t u) {
    if (HOT && u < 0) return sh[u & 0x7fffffff];
    if (!LOOP) return __ldg(c + u);
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(c + u));
    return v;
}

#ifndef GP_TILE_THREADS
#define GP_TILE_THREADS 768
#endif
constexpr int TILE_THREADS = GP_TILE_THREADS;  // threads per block of the tile kernel, two blocks per SM
constexpr int LANE_EDGES = TILE_EDGES / 32;  // consecutive edges of a tile that one lane sums
static_assert(LANE_EDGES == 8, "one head byte and one 32-byte index load per lane");

// Eight consecutive 32-bit words.  The index and weight arrays are streamed
// once per sweep: evict-first in L2 and not kept in L1, so that they do not
// push the gathered contributions out.
__device__ __forceinline__ void ld_stream8(const void *p, uint32_t (&v)[8]) {
    asm volatile("ld.global.nc.L1::no_allocate.L2::evict_first.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(p));
}

// A tile's sums by row, from its lanes' products f (eight consecutive edges
// each), row-start bits h and the row open at its start.  A row that starts in
// the tile leaves its sum there in acc[row]; edges of a row started in an
// earlier tile leave theirs in carry[t].  Called by the whole warp.
__device__ __forceinline__ void tile_sums(const PrArgs &a, int64_t t, unsigned h, int32_t row0, const float (&f)[8]) {
    const int lane = lane_id();
    const unsigned below = (1u << lane) - 1u;
    const unsigned starts = __ballot_sync(FULL, h != 0);  // lanes where a row starts
    if (starts == 0) {  // the inside of one long row
        float s = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7]));
        s = warp_sum(s);
        if (lane == 0) a.carry[t] = s;
        return;
    }
    // rows started in the lanes below: prefix sum of popc(h) <= 8, by its binary digits
    const unsigned cnt = __popc(h);
    int before = 0, all = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const unsigned digit = __ballot_sync(FULL, (cnt >> b) & 1u);
        before += __popc(digit & below) << b;
        all += __popc(digit) << b;
    }
    const int32_t row = row0 + before;  // the row open at the lane's first edge
    float open = 0.f, s = 0.f;
    int32_t r = row;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if ((h >> q) & 1u) {
            if (r == row)
                open = s;  // what the lane adds to the row open at its start
            else
                a.acc[r] = s;  // a row that starts and ends in the lane
            ++r;
            s = 0.f;
        }
        s += f[q];
    }
    // segmented inclusive scan over the lanes: s becomes the sum of the row
    // open at the lane's end, back to the lane where it starts
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float up = __shfl_up_sync(FULL, s, o);
        // lanes lane-o+1 .. lane start no row
        if (lane >= o && (starts & (below + below + 1u) & ~((1u << (lane - o + 1)) - 1u)) == 0) s += up;
    }
    float in = __shfl_up_sync(FULL, s, 1);
    if (lane == 0) in = 0.f;
    if (h) {
        if ((starts & below) == 0)
            a.carry[t] = in + open;
        else
            a.acc[row] = in + open;
    }
    if (lane == 31) a.acc[row0 + all] = s;
}

// One sweep's sums: tiles warp, warp + nwarps, ...
template <bool W, bool HOT, bool LOOP>
__device__ __forceinline__ void pull_tiles_step(const PrArgs &a, const float *sh, int warp, int nwarps) {
    const int lane = lane_id();
    const int32_t *__restrict__ idx = a.idx;
    const float *c = a.c;
    const int ntiles = (int)a.ntiles;
    for (int t = warp; t < ntiles; t += nwarps) {
        const int64_t e0 = (int64_t)t * TILE_EDGES + lane * LANE_EDGES;
        const unsigned h = a.heads[(int64_t)t * 32 + lane];  // bit q: edge e0 + q is the first of its row
        const int32_t row0 = a.tile_row[t];
        float f[8];
        if (t < a.vec_tiles) {
            uint32_t u[8];
            ld_stream8(idx + e0, u);
#pragma unroll
            for (int q = 0; q < 8; ++q) f[q] = gather_c<HOT, LOOP>(c, sh, (int32_t)u[q]);
            if (W) {
                ld_stream8(a.w + e0, u);
#pragma unroll
                for (int q = 0; q < 8; ++q) f[q] *= __uint_as_float(u[q]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                f[q] = 0.f;
                if (e0 + q < a.m) {
                    f[q] = gather_c<HOT, LOOP>(c, sh, __ldg(idx + e0 + q));
                    if (W) f[q] *= __ldg(a.w + e0 + q);
                }
            }
        }
        tile_sums(a, t, h, row0, f);
    }
}

// Bound by the random 4-byte gathers (one per edge; L1 tags and L2 sectors:
// ~300 G/s from L2).  Equal tiles keep every lane's eight gathers in use at any
// degree, where a warp per long list and a lane per short one left most of them
// idle at degrees near 16: a sweep of a uniform graph (n = 8.0M, m = 128M) took
// 555 + 335 us split that way and takes 462 + 55 us; R-MAT 22 (m = 128M) 295 +
// 84 + 4 us, now 286 + 26 us (40 or 32 registers, 768 or 1024 threads a block:
// within 1% there; 768 is 10% faster on a graph of 16K vertices).
template <bool W, bool HOT>
__global__ void __launch_bounds__(TILE_THREADS, 2) k_pull_tiles(PrArgs a) {
    extern __shared__ float sh_hot[];
    if (pr_gate(a, a.k)) return;
    load_hot<HOT>(a, sh_hot);
    pull_tiles_step<W, HOT, false>(a, sh_hot, (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                            (int)(gridDim.x * blockDim.x) >> 5);
}

// What a vertex's new iterate takes beside its gathered sum.
struct PullRow {
    float x, base, post, c;
    __device__ __forceinline__ PullRow(const PrArgs &a, int64_t v)
        : x(a.x[v]), base(base_term(a, v)), post(post_factor(a, v)), c(c_factor(a, v)) {}
};

template <bool HOT>
__device__ __forceinline__ void pull_write(const PrArgs &a, int64_t v, const PullRow &row, float sum, ResSum &res) {
    const float y = row.base + a.d * (row.post * sum);
    const float cn = y * row.c;
    res.add(y, row.x);
    a.y[v] = y;
    a.c_next[v] = cn;
    if (HOT) store_hot(a.hot_bits, a.hot_prefix, a.c_hot, v, cn);
}

// Rows, then, in the first two sweeps, the vertices without in-edges: theirs is
// the base term in every sweep, so both iterate buffers hold it from then on.
// Bound by memory, and short of it by latency: the next row's number and a row's
// operands are fetched before they are needed (n = 8.0M, 36 bytes a row: 68 -> 55
// us; R-MAT 22: 26; four rows a thread were slower than one).
// long_warp: this warp's place among those that deal out the long rows.  A launch
// of its own deals them over the blocks, the sweeps in one launch over few blocks
// (R-MAT 2^18, directed, 40 sweeps and 40 of the adjoint: 2.45 ms, 2.48 the other way).
template <bool HOT>
__device__ __forceinline__ void pull_finish_step(const PrArgs &a, int64_t thread, int64_t nthreads, int64_t long_warp,
                                                 ResSum &res) {
    const int64_t count = a.k <= 2 ? a.n : a.nrows;
    uint32_t next = thread < count ? (uint32_t)a.rows[thread] : 0u;
    for (int64_t r = thread; r < count; r += nthreads) {
        const uint32_t code = next;
        if (r + nthreads < count) next = (uint32_t)a.rows[r + nthreads];
        const int64_t v = code & ~HOT_BIT;
        float sum = r < a.nrows ? a.acc[r] : 0.f;
        const PullRow row(a, v);
        if (code & HOT_BIT) {  // the row spans tiles
            const int64_t t0 = a.off[v] / TILE_EDGES, t1 = (a.off[v + 1] - 1) / TILE_EDGES;
            if (t1 - t0 > TILE_LONG) continue;  // below
            for (int64_t t = t0 + 1; t <= t1; ++t) sum += a.carry[t];
        }
        pull_write<HOT>(a, v, row, sum, res);
    }
    const int lane = lane_id();
    for (int64_t i = long_warp; i < a.nlong; i += nthreads >> 5) {
        const int32_t r = a.long_rows[i];
        const int64_t v = (uint32_t)a.rows[r] & ~HOT_BIT;
        const int64_t t0 = a.off[v] / TILE_EDGES, t1 = (a.off[v + 1] - 1) / TILE_EDGES;
        float sum = 0.f;
        for (int64_t t = t0 + 1 + lane; t <= t1; t += 32) sum += a.carry[t];
        sum = warp_sum(sum);
        if (lane == 0) pull_write<HOT>(a, v, PullRow(a, v), a.acc[r] + sum, res);
    }
}

template <bool HOT>
__global__ void __launch_bounds__(256) k_pull_finish(PrArgs a) {
    __shared__ double sm[32];
    if (pr_stopped(a.status)) return;
    ResSum res;
    // (neighbouring long rows to different blocks: in a power-law graph the longest are neighbours)
    pull_finish_step<HOT>(a, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x,
                          (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x, res);
    const double r = block_residual(res, sm);
    if (threadIdx.x == 0) a.partials[blockIdx.x] = r;
}

// All sweeps of a small graph in one cooperative launch: two barriers a sweep
// instead of two launches, and the convergence test on the device.  Without a
// hot set: on such graphs most of the contribution vector stays in L1.
struct PrLoop {
    PrArgs a;  // sweep k from R[(k-1)&1], C[(k-1)&1] to R[k&1], C[k&1]
    float *R[2], *C[2];
    int32_t iters;
    PrStatus *mirror;
    GridSync *sync;
};

// The end of sweep k, called by every block: true when it was the last one.
__device__ __forceinline__ bool loop_end(const PrLoop &P, int k, double *sm, double &residual) {
    __shared__ double s_res;
    if (P.a.tol <= 0.0 && k < P.iters) return false;
    double t = 0.0;  // the same sum in the same order in every block
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) t += P.a.partials[i];
    t = block_sum(t, sm);
    if (threadIdx.x == 0) s_res = t;
    __syncthreads();
    residual = s_res;
    return residual < P.a.tol || k == P.iters;
}

__device__ __forceinline__ void loop_status(const PrLoop &P, int k, double residual) {
    PrStatus *st = P.a.status;
    st->done = st->converged = residual < P.a.tol;
    st->iters_done = k;
    st->residual = residual;
    *P.mirror = *st;
    __threadfence_system();
}

template <bool W>
__global__ void __launch_bounds__(TILE_THREADS, 2) k_pull_loop(const __grid_constant__ PrLoop P) {
    __shared__ double sm[32];
    PrArgs a = P.a;
    const int64_t thread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nthreads = (int64_t)gridDim.x * blockDim.x;
    double residual = 0.0;
    int k = 1;
    for (;; ++k) {
        a.k = k;
        a.x = P.R[(k - 1) & 1];
        a.y = P.R[k & 1];
        a.c = P.C[(k - 1) & 1];
        a.c_next = P.C[k & 1];
        pull_tiles_step<W, false, true>(a, nullptr, (int)(thread >> 5), (int)(nthreads >> 5));
        if (!grid_sync(P.sync, gridDim.x)) return;
        ResSum res;
        pull_finish_step<false>(a, thread, nthreads, thread >> 5, res);
        const double r = block_residual(res, sm);
        if (threadIdx.x == 0) a.partials[blockIdx.x] = r;
        if (!grid_sync(P.sync, gridDim.x)) return;
        if (loop_end(P, k, sm, residual)) break;
    }
    if (k & 1)  // the caller's buffer is R[0]
        for (int64_t v = thread; v < a.n; v += nthreads) P.R[0][v] = P.R[1][v];
    if (thread == 0) loop_status(P, k, residual);
}

// The same with a tile to a warp and a row to a thread, for graphs that the grid
// holds that way: what does not change between sweeps (indices, weights, row
// numbers and places, the vertex's factors) and the iterate itself stay in
// registers, and a sweep is two chains of one load each between its barriers:
// 5 us a sweep at R-MAT 2^14, where the loop above takes 9 and launches 17.
template <bool W>
__global__ void __launch_bounds__(TILE_THREADS, 1) k_pull_loop_regs(const __grid_constant__ PrLoop P) {
    __shared__ double sm[32];
    const PrArgs &a = P.a;
    const int lane = lane_id();
    const int64_t thread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // the warp's tile
    const int64_t t = thread >> 5;
    const bool tile = t < a.ntiles;
    const int64_t e0 = t * TILE_EDGES + lane * LANE_EDGES;
    const unsigned h = tile ? a.heads[t * 32 + lane] : 0u;
    const int32_t row0 = tile ? a.tile_row[t] : 0;
    int32_t u[8];
    float w[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const bool edge = tile && e0 + q < a.m;
        u[q] = edge ? __ldg(a.idx + e0 + q) : -1;
        w[q] = W && edge ? __ldg(a.w + e0 + q) : 0.f;
    }
    // the thread's row, or vertex without in-edges (acc: its sum's place; long rows are a warp's)
    const bool has = thread < a.n, filled = thread < a.nrows;
    int64_t v = 0, c0 = 0, c1 = 0;  // the carries to add: [c0, c1)
    bool mine = has;
    if (has) {
        const uint32_t code = (uint32_t)a.rows[thread];
        v = code & ~HOT_BIT;
        if (code & HOT_BIT) {
            c0 = a.off[v] / TILE_EDGES + 1;
            c1 = (a.off[v + 1] - 1) / TILE_EDGES + 1;
            mine = c1 - c0 <= TILE_LONG;
        }
    }
    // the warp's long row
    const bool longrow = t < a.nlong;
    int32_t lr = 0;
    int64_t lv = 0, l0 = 0, l1 = 0;
    if (longrow) {
        lr = a.long_rows[t];
        lv = (uint32_t)a.rows[lr] & ~HOT_BIT;
        l0 = a.off[lv] / TILE_EDGES + 1;
        l1 = (a.off[lv + 1] - 1) / TILE_EDGES + 1;
    }
    const bool leader = longrow && lane == 0;
    const float base = has ? base_term(a, v) : 0.f, cm = has ? c_factor(a, v) : 0.f;
    const float lbase = leader ? base_term(a, lv) : 0.f, lcm = leader ? c_factor(a, lv) : 0.f;
    float x = has ? P.R[0][v] : 0.f, lx = leader ? P.R[0][lv] : 0.f;
    double residual = 0.0;
    int k = 1;
    for (;; ++k) {
        const float *c = P.C[(k - 1) & 1];
        float *c_next = P.C[k & 1];
        if (tile) {
            float f[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                f[q] = u[q] >= 0 ? gather_c<false, true>(c, nullptr, u[q]) : 0.f;
                if (W) f[q] *= w[q];
            }
            tile_sums(a, t, h, row0, f);
        }
        if (!grid_sync(P.sync, gridDim.x)) return;
        ResSum res;
        if (mine) {
            float sum = filled ? a.acc[thread] : 0.f;
            for (int64_t i = c0; i < c1; ++i) sum += a.carry[i];
            const float y = base + a.d * sum;
            res.add(y, x);
            x = y;
            c_next[v] = y * cm;
        }
        if (longrow) {
            float sum = 0.f;
            for (int64_t i = l0 + lane; i < l1; i += 32) sum += a.carry[i];
            sum = warp_sum(sum);
            if (lane == 0) {
                const float y = lbase + a.d * (a.acc[lr] + sum);
                res.add(y, lx);
                lx = y;
                c_next[lv] = y * lcm;
            }
        }
        if (a.tol > 0.0 || k == P.iters) {
            const double r = block_residual(res, sm);
            if (threadIdx.x == 0) a.partials[blockIdx.x] = r;
        }
        if (!grid_sync(P.sync, gridDim.x)) return;
        if (loop_end(P, k, sm, residual)) break;
    }
    if (mine) P.R[0][v] = x;
    if (leader) P.R[0][lv] = lx;
    if (thread == 0) loop_status(P, k, residual);
}

// The adjoint's pull sweep sums a row in a fixed order of its own, whatever the
// rows around it: a short row's edges one after another in its lane, a long
// row's in warp chunks and the chunks one after another.  The gradient of a
// normalised weight is (x_u / S_u)(d lambda_v - lambda_u + g_u), and where u's
// edges are few and light the bracket cancels while the factor is large: there
// the order of summation, not only its error, shows in the result (two orders
// differ by up to 1e-3 of the gradients' RMS on R-MAT 18 with weights in (0, 1]),
// so gradients keep the order that they have always had.
constexpr int BIG_UNROLL = 8;

// Index arrays are streamed once per sweep: loaded with the evict-first hint so
// they do not push the gathered contribution vector out of L2.
__device__ __forceinline__ int32_t ld_idx(const int32_t *p) { return __ldcs(p); }

// The row's new value.  Rounded as written here, whatever is around it: left to
// the compiler, the base's product and this one compete for the fused addition,
// and short and long rows were rounded unlike (fused, and not), which stays.
__device__ __forceinline__ float adj_value(const PrArgs &a, float base, float ps, float sum, bool long_row) {
    const float g = __fmul_rn(ps, sum);
    return long_row ? __fadd_rn(base, __fmul_rn(a.d, g)) : __fmaf_rn(a.d, g, base);
}

// The long rows' chunks, chunk j by warp j mod nwarps.
template <bool W, bool LOOP>
__device__ __forceinline__ void adj_big_step(const PrArgs &a, int64_t warp, int64_t nwarps) {
    const int lane = lane_id();
    const int32_t *__restrict__ idx = a.idx;
    const float *c = a.c;
    const float *__restrict__ w = a.w;
    for (int64_t j = warp; j < a.nchunks; j += nwarps) {
        const Chunk ch = a.chunks[j];
        const int32_t *ip = idx + ch.beg;
        const float *wp = W ? w + ch.beg : nullptr;
        float acc = 0.f;
        for (int i0 = 0; i0 < ch.len; i0 += 32 * BIG_UNROLL) {
            // all index loads of the window first, then all gathers: BIG_UNROLL in flight per lane
            int32_t u[BIG_UNROLL];
#pragma unroll
            for (int q = 0; q < BIG_UNROLL; ++q) {
                const int i = i0 + q * 32 + lane;
                u[q] = i < ch.len ? ld_idx(ip + i) : 0;
            }
            float f[BIG_UNROLL];
#pragma unroll
            for (int q = 0; q < BIG_UNROLL; ++q) {
                const int i = i0 + q * 32 + lane;
                f[q] = 0.f;
                if (i < ch.len) {
                    f[q] = gather_c<false, LOOP>(c, nullptr, u[q]);
                    if (W) f[q] = __fmul_rn(f[q], __ldg(wp + i));
                }
            }
#pragma unroll
            for (int q = 0; q < BIG_UNROLL; ++q) acc = __fadd_rn(acc, f[q]);
        }
        acc = warp_sum(acc);
        if (lane == 0) a.chunk_part[j] = acc;
    }
}

constexpr int LIGHT_UNROLL = 8;  // in-edges of a light vertex in flight per lane

// The short rows, 32 vertices to a warp.
template <bool W, bool LOOP>
__device__ __forceinline__ void adj_light_step(const PrArgs &a, int64_t warp, int64_t nwarps, ResSum &res) {
    const int lane = lane_id();
    const int64_t n = a.n;
    const int64_t ntiles = (n + 31) >> 5;
    const int32_t *__restrict__ idx = a.idx;
    const float *c = a.c;
    const float *__restrict__ wv = a.w;
    // offsets of the first tile; inside the loop the next tile's are fetched early
    int64_t t = warp;
    int64_t nb = 0, ne = 0;
    if (t < ntiles && t * 32 + lane < n) {
        nb = a.off[t * 32 + lane];
        ne = a.off[t * 32 + lane + 1];
    }
    for (; t < ntiles; t += nwarps) {
        const int64_t v = t * 32 + lane;
        const int64_t b = nb, e = ne;
        // per-vertex operands, independent of the edges: issued now
        float xv = 0.f, cm = 0.f, ps = 0.f, base_v = 0.f;
        if (v < n) {
            xv = a.x[v];
            cm = c_factor(a, v);
            ps = post_factor(a, v);
            base_v = base_term(a, v);
        }
        const int64_t tn = t + nwarps, vn = tn * 32 + lane;
        nb = ne = 0;
        if (tn < ntiles && vn < n) {
            nb = a.off[vn];
            ne = a.off[vn + 1];
        }
        const int64_t dd = e - b;
        const bool big = dd > a.light_max;
        // a light vertex's own lane sums its in-list, LIGHT_UNROLL loads in flight
        const int64_t e1 = big ? b : e;
        float acc = 0.f;
        for (int64_t p0 = b; p0 < e1; p0 += LIGHT_UNROLL) {
            int32_t u[LIGHT_UNROLL];
            float f[LIGHT_UNROLL];
#pragma unroll
            for (int q = 0; q < LIGHT_UNROLL; ++q) u[q] = p0 + q < e1 ? ld_idx(idx + p0 + q) : 0;
#pragma unroll
            for (int q = 0; q < LIGHT_UNROLL; ++q) {
                f[q] = 0.f;
                if (p0 + q < e1) {
                    f[q] = gather_c<false, LOOP>(c, nullptr, u[q]);
                    if (W) f[q] = __fmul_rn(f[q], __ldg(wv + p0 + q));
                }
            }
#pragma unroll
            for (int q = 0; q < LIGHT_UNROLL; ++q) acc = __fadd_rn(acc, f[q]);
        }
        if (v < n && !big) {
            const float y = adj_value(a, base_v, ps, acc, false);
            if (!LOOP) res.add(y, xv);  // (the loop draws its rows in no fixed order)
            a.y[v] = y;
            a.c_next[v] = y * cm;
        }
    }
}

// The long rows' chunk sums, one after another: a warp loads 32 at a time and
// every lane adds them in their order (a thread that walked a hub's 200 took
// most of the kernel's time).
__device__ __forceinline__ void adj_combine_step(const PrArgs &a, int64_t warp, int64_t nwarps, ResSum &res) {
    const int lane = lane_id();
    for (int64_t r0 = warp * 32; r0 < a.nbig; r0 += nwarps * 32) {
        const int64_t r = r0 + lane;
        int64_t c0 = 0, c1 = 0;
        int32_t v = 0;
        if (r < a.nbig) {
            v = a.big[r];
            c0 = a.cstart[r];
            c1 = a.cstart[r + 1];
        }
        float acc = 0.f;
        const bool wide = c1 - c0 > 16;
        if (!wide) {
#pragma unroll 4
            for (int64_t j = c0; j < c1; ++j) acc += a.chunk_part[j];
        }
        for (unsigned m = __ballot_sync(FULL, wide); m; m &= m - 1) {
            const int l = __ffs(m) - 1;
            const int64_t b = __shfl_sync(FULL, c0, l), e = __shfl_sync(FULL, c1, l);
            float sum = 0.f;
            for (int64_t j = b; j < e; j += 32) {
                const float part = j + lane < e ? a.chunk_part[j + lane] : 0.f;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float p = __shfl_sync(FULL, part, i);
                    if (j + i < e) sum += p;
                }
            }
            if (lane == l) acc = sum;
        }
        if (r < a.nbig) {
            const float y = adj_value(a, base_term(a, v), post_factor(a, v), acc, true);
            res.add(y, a.x[v]);
            a.y[v] = y;
            a.c_next[v] = y * c_factor(a, v);
        }
    }
}

template <bool W>
__global__ void __launch_bounds__(1024) k_adj_big(PrArgs a) {
    if (pr_gate(a, a.k)) return;
    adj_big_step<W, false>(a, ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, ((int64_t)gridDim.x * blockDim.x) >> 5);
}

template <bool W>
__global__ void __launch_bounds__(512, 3) k_adj_light(PrArgs a) {
    __shared__ double sm[32];
    if (pr_stopped(a.status)) return;
    ResSum res;
    if ((int)blockIdx.x < a.split_blocks)
        adj_light_step<W, false>(a, ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                                 ((int64_t)a.split_blocks * blockDim.x) >> 5, res);
    else
        adj_combine_step(a, ((int64_t)(blockIdx.x - a.split_blocks) * blockDim.x + threadIdx.x) >> 5,
                         ((int64_t)(gridDim.x - a.split_blocks) * blockDim.x) >> 5, res);
    const double r = block_residual(res, sm);
    if (threadIdx.x == 0) a.partials[blockIdx.x] = r;
}

// All sweeps of a small graph's adjoint in one cooperative launch, as k_pull_loop.
// A block's warps draw its units -- 32 short rows, or a long row's chunk, short rows
// first as they take longest -- from a counter in shared memory: units differ
// severalfold in time, and with a fixed share for every warp (5.4 chunks and 1.1
// groups of rows at R-MAT 2^18) half of the sweep was waiting for the last ones.
// 34 -> 26 us a sweep there; the chunks first measured 30, a draw ahead of the work 27.
// Rows' values don't depend on who computes them; the residual's FP64 sum would, so
// a sweep that needs it takes the short rows' part in a pass of its own.
template <bool W>
__global__ void __launch_bounds__(512, 3) k_adj_loop(const __grid_constant__ PrLoop P) {
    __shared__ double sm[32];
    PrArgs a = P.a;
    __shared__ int drawn[2];
    const int64_t thread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nthreads = (int64_t)gridDim.x * blockDim.x;
    const int wib = threadIdx.x >> 5;
    // the block's groups of rows and chunks: those congruent to its number
    const int64_t B = gridDim.x, b = blockIdx.x;
    const int rows = (int)((((a.n + 31) >> 5) - b + B - 1) / B);
    const int units = rows + (int)((a.nchunks - b + B - 1) / B);
    if (threadIdx.x < 2) drawn[threadIdx.x] = 0;
    __syncthreads();
    double residual = 0.0;
    int k = 1;
    for (;; ++k) {
        a.x = P.R[(k - 1) & 1];
        a.y = P.R[k & 1];
        a.c = P.C[(k - 1) & 1];
        a.c_next = P.C[k & 1];
        if (threadIdx.x == 0) drawn[(k + 1) & 1] = 0;  // the next sweep's, behind two barriers
        ResSum res;
        for (;;) {
            int u = 0;
            if (lane_id() == 0) u = atomicAdd(&drawn[k & 1], 1);
            u = __shfl_sync(FULL, u, 0);
            if (u >= units) break;
            if (u < rows)
                adj_light_step<W, true>(a, b + (int64_t)u * B, 1 << 30, res);
            else
                adj_big_step<W, true>(a, b + (int64_t)(u - rows) * B, 1 << 30);
        }
        if (!grid_sync(P.sync, gridDim.x)) return;
        if (a.tol > 0.0 || k == P.iters)
            for (int64_t v = thread; v < a.n; v += nthreads)
                if (a.off[v + 1] - a.off[v] <= a.light_max) res.add(a.y[v], a.x[v]);
        adj_combine_step(a, wib * B + b, nthreads >> 5, res);
        const double r = block_residual(res, sm);
        if (threadIdx.x == 0) a.partials[blockIdx.x] = r;
        if (!grid_sync(P.sync, gridDim.x)) return;
        if (loop_end(P, k, sm, residual)) break;
    }
    if (k & 1)  // the caller's buffer is R[0]
        for (int64_t v = thread; v < a.n; v += nthreads) P.R[0][v] = P.R[1][v];
    if (thread == 0) loop_status(P, k, residual);
}

// Owner lane of virtual edge `eid` in a tile: the last lane k with excl[k] <= eid
// (zero-degree lanes share their successor's excl, so the last one is non-empty).
__device__ __forceinline__ int tile_owner(int excl, int eid) {
    int k = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const int ex = __shfl_sync(FULL, excl, k + s);
        if (ex <= eid) k += s;
    }
    return k;
}

// ------------------------------------------------------------------ push

// Accumulator of the scattered updates: FP32 (the paper's float atomics) or
// FP64 (same atomic count; the order-dependent rounding of FP32 atomics at hubs
// otherwise leaves an L1 residual floor above 1e-7 on graphs with 4M vertices).
// HOT: the partition-awareness of the paper's Section 5 recast for a GPU block --
// updates to the H most updated vertices (encoded in the index array) are
// summed in the block's shared memory with shared-memory atomics and flushed
// once per block; only the other updates use global atomics.
struct PushCount {
    unsigned l2 = 0, shared = 0, merged = 0, flush = 0;
};

template <class T, bool HOT>
__device__ __forceinline__ void scatter_add(T *y, float *sh, int32_t dst, float val, PushCount &cnt) {
    if (HOT && dst < 0) {
        atomicAdd(sh + (dst & 0x7fffffff), val);
        ++cnt.shared;
    } else {
        atomicAdd(y + dst, (T)val);
        ++cnt.l2;
    }
}

// Bound by the latency of its chains (indices, row, contribution) and the
// shared-memory atomics, not by the reductions in L2: without those it is 4%
// faster.  So what pays is equal work per lane and full occupancy: tiles and two
// blocks per SM take R-MAT n = 1.0M (30M edges) from 150 to 110 us a sweep, where a
// warp walked each 256-edge piece of a long list, a merged stream of the short
// ones found every edge's source by a search over the warp, and one block of
// 32768 accumulators filled the SM's shared memory.
template <bool W, class T, bool HOT>
__global__ void __launch_bounds__(TILE_THREADS, 2) k_push_tiles(PrArgs a) {
    extern __shared__ float sh_acc[];
    __shared__ float agg[TILE_THREADS];
    if (pr_gate(a, a.k)) return;
    if (HOT) {
        for (int64_t i = threadIdx.x; i < a.nhot; i += blockDim.x) sh_acc[i] = 0.f;
        __syncthreads();
    }
    const int lane = lane_id();
    const unsigned below = (1u << lane) - 1u;
    T *y = sizeof(T) == 8 ? (T *)a.acc64 : (T *)a.y;
    const int warp = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (int)(gridDim.x * blockDim.x) >> 5;
    const int ntiles = (int)a.ntiles;
    PushCount cnt;
    for (int t = warp; t < ntiles; t += nwarps) {
        const int64_t e0 = (int64_t)t * TILE_EDGES + lane * LANE_EDGES;
        const unsigned h = a.heads[(int64_t)t * 32 + lane];  // bit q: edge e0 + q is the first of its source
        const int32_t row0 = a.tile_row[t];
        int32_t dst[8];
        float val[8];
        if (t < a.vec_tiles) {
            uint32_t u[8];
            ld_stream8(a.idx + e0, u);
#pragma unroll
            for (int q = 0; q < 8; ++q) dst[q] = (int32_t)u[q];
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) dst[q] = e0 + q < a.m ? __ldg(a.idx + e0 + q) : 0;
        }
        // the sources' contributions: sources started in the lanes below (as in tile_sums), then in the lane
        const unsigned nh = __popc(h);
        int row = row0, sources = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const unsigned digit = __ballot_sync(FULL, (nh >> b) & 1u);
            row += __popc(digit & below) << b;
            sources += __popc(digit) << b;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            int32_t v = -1;
            if (((h >> q) & 1u) || (q == 0 && e0 < a.m)) v = a.rows[row + __popc(h & ((2u << q) - 1u))] & 0x7fffffff;
            val[q] = __int_as_float(v);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int32_t v = __float_as_int(val[q]);
            val[q] = v >= 0 ? a.d * __ldg(a.c + v) : 0.f;
        }
#pragma unroll
        for (int q = 1; q < 8; ++q)
            if (!((h >> q) & 1u)) val[q] = val[q - 1];
        if (W) {
            if (t < a.vec_tiles) {
                uint32_t w[8];
                ld_stream8(a.w + e0, w);
#pragma unroll
                for (int q = 0; q < 8; ++q) val[q] *= __uint_as_float(w[q]);
            } else {
#pragma unroll
                for (int q = 0; q < 8; ++q) val[q] *= e0 + q < a.m ? __ldg(a.w + e0 + q) : 0.f;
            }
        }
        // Updates of one vertex by different sources (a hub by its leaves) are summed
        // first: a lane's neighbouring ones, then, where the tile has many sources,
        // the warp's.  A hub's FP32 accumulator then takes few terms.
        bool crowd = sources >= 8;
        if (crowd)  // (most such tiles share no vertex: their first edges tell)
            crowd = !__all_sync(FULL, __match_any_sync(FULL, e0 < a.m ? dst[0] : (int32_t)(0x7fffffff - lane)) == (1u << lane));
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            bool mine = e0 + q < a.m;
            if (q < 7 && e0 + q + 1 < a.m && dst[q] == dst[q + 1]) {
                val[q + 1] += val[q];
                ++cnt.merged;
                mine = false;
            }
            if (!crowd) {
                if (mine) scatter_add<T, HOT>(y, sh_acc, dst[q], val[q], cnt);
                continue;
            }
            // idle lanes get keys no update has: positive and >= n is impossible for
            // plain vertices, and HOT keys are negative
            const unsigned peers = __match_any_sync(FULL, mine ? dst[q] : (int32_t)(0x7fffffff - lane));
            if (__all_sync(FULL, peers == (1u << lane))) {
                if (mine) scatter_add<T, HOT>(y, sh_acc, dst[q], val[q], cnt);
            } else {
                agg[threadIdx.x] = val[q];
                __syncwarp();
                if (mine && (peers & below) == 0) {  // lowest lane of its group
                    float sum = val[q];
                    for (unsigned rest = peers & ~(1u << lane); rest; rest &= rest - 1)
                        sum += agg[(threadIdx.x & ~31u) + (__ffs(rest) - 1)];
                    scatter_add<T, HOT>(y, sh_acc, dst[q], sum, cnt);
                    cnt.merged += __popc(peers) - 1;
                }
                __syncwarp();
            }
        }
    }
    if (HOT) {  // flush: one global atomic per touched hot vertex per block
        __syncthreads();
        for (int64_t i = threadIdx.x; i < a.nhot; i += blockDim.x) {
            const float v = sh_acc[i];
            if (v != 0.f) {
                atomicAdd(y + a.hot_id[i], (T)v);
                ++cnt.flush;
            }
        }
    }
    // the block's update counts, one reduction and four atomics per block
    __shared__ unsigned long long csum[4][32];
    unsigned long long c4[4] = {cnt.l2, cnt.shared, cnt.merged, cnt.flush};
#pragma unroll
    for (int i = 0; i < 4; ++i) c4[i] = warp_sum(c4[i]);
    __syncthreads();
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) csum[i][threadIdx.x >> 5] = c4[i];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int i = 0; i < 4; ++i) c4[i] = warp_sum(threadIdx.x < (blockDim.x >> 5) ? csum[i][threadIdx.x] : 0ull);
        if (threadIdx.x == 0) {
            if (c4[0]) atomicAdd(&a.status->upd_l2, c4[0]);
            if (c4[1]) atomicAdd(&a.status->upd_shared, c4[1]);
            if (c4[2]) atomicAdd(&a.status->upd_merged, c4[2]);
            if (c4[3]) atomicAdd(&a.status->flush_l2, c4[3]);
        }
    }
}

// Per vertex: y = base + post_scale * (scattered sum), rounded to the FP32 rank;
// the residual, the next contribution, and the zeroing of the buffer the next
// sweep accumulates into.
template <class T>
__global__ void __launch_bounds__(256) k_push_epilogue(PrArgs a) {
    __shared__ double sm[32];
    if (pr_stopped(a.status)) return;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    ResSum res;
    float *x_reset = const_cast<float *>(a.x);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += stride) {
        const float base = base_term(a, v), ps = post_factor(a, v);
        float y;
        if (sizeof(T) == 8) {
            // the FP64 sum rounded once to FP32, then the FP32 epilogue
            y = fmaf(ps, f64_to_f32_rn(a.acc64[v]), base);
            a.acc64[v] = 0.0;
        } else {
            y = base + ps * a.y[v];
        }
        res.add(y, a.x[v]);
        a.y[v] = y;
        a.c_next[v] = y * c_factor(a, v);
        if (sizeof(T) != 8) x_reset[v] = 0.f;  // the next sweep accumulates into this buffer
    }
    const double r = block_residual(res, sm);
    if (threadIdx.x == 0) a.partials[blockIdx.x] = r;
}

// ------------------------------------------------------------------ adjoint gradients

// grad_s[v] = (1-d) lambda_v
__global__ void k_grad_s(int64_t n, float one_minus_d, const float *lam, float *grad_s) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) grad_s[v] = one_minus_d * lam[v];
}

struct GradArgs {
    int64_t n;
    const int64_t *off;  // CSR
    const int32_t *idx;
    const float *x, *lam, *g, *inv_deg;
    const Chunk *chunks;
    int64_t nchunks;
    int32_t light_max;
    float d;
    int normalized;
    float *grad_w;
    int32_t split_blocks;
};

// dL/dP_vu = d lambda_v x_u for the CSR edge e = (u -> v); with per-source
// normalisation P_vu = w_uv / S_u the raw-weight gradient is
// (x_u / S_u) (d lambda_v - lambda_u + g_u), using lambda_u = g_u + d (P^T lambda)_u.
__device__ __forceinline__ float edge_grad(const GradArgs &a, int32_t u, int32_t v, float xu_or_coef, float lam_u_term) {
    return a.normalized ? xu_or_coef * (a.d * a.lam[v] - lam_u_term) : a.d * a.lam[v] * xu_or_coef;
}

__global__ void __launch_bounds__(256) k_grad_w(GradArgs a) {
    const int lane = lane_id();
    if ((int)blockIdx.x < a.split_blocks) {
        const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        const int64_t nwarps = ((int64_t)a.split_blocks * blockDim.x) >> 5;
        for (int64_t j = warp; j < a.nchunks; j += nwarps) {
            const Chunk ch = a.chunks[j];
            const int32_t u = ch.v;
            const float coef = a.normalized ? a.x[u] * a.inv_deg[u] : a.x[u];
            const float lt = a.normalized ? a.lam[u] - a.g[u] : 0.f;
            for (int i = lane; i < ch.len; i += 32) {
                const int64_t pos = ch.beg + i;
                a.grad_w[pos] = edge_grad(a, u, a.idx[pos], coef, lt);
            }
        }
    } else {
        const int64_t warp = ((int64_t)(blockIdx.x - a.split_blocks) * blockDim.x + threadIdx.x) >> 5;
        const int64_t nwarps = ((int64_t)(gridDim.x - a.split_blocks) * blockDim.x) >> 5;
        const int64_t ntiles = (a.n + 31) >> 5;
        for (int64_t t = warp; t < ntiles; t += nwarps) {
            const int64_t u = t * 32 + lane;
            int64_t b = 0, e = 0;
            float coef = 0.f, lt = 0.f;
            if (u < a.n) {
                b = a.off[u];
                e = a.off[u + 1];
                coef = a.normalized ? a.x[u] * a.inv_deg[u] : a.x[u];
                lt = a.normalized ? a.lam[u] - a.g[u] : 0.f;
            }
            const int64_t dd = e - b;
            const int deg = dd > a.light_max ? 0 : (int)dd;
            const int incl = warp_incl_scan(deg);
            const int excl = incl - deg;
            const int E = __shfl_sync(FULL, incl, 31);
            for (int base = 0; base < E; base += 32) {
                const int eid = base + lane;
                const int k = tile_owner(excl, eid);
                const int64_t kb = __shfl_sync(FULL, b, k);
                const int kex = __shfl_sync(FULL, excl, k);
                const float kc = __shfl_sync(FULL, coef, k);
                const float kl = __shfl_sync(FULL, lt, k);
                const int32_t ku = (int32_t)(t * 32 + k);
                if (eid < E) {
                    const int64_t pos = kb + (eid - kex);
                    a.grad_w[pos] = edge_grad(a, ku, a.idx[pos], kc, kl);
                }
            }
        }
    }
}

// ------------------------------------------------------------------ driver

void release_pr_work(gp_graph *g, cudaStream_t s) {
    for (cudaEvent_t e : g->pr.ev)
        if (e) cudaEventDestroy(e);
    pinned_free(g->pr.status_host, 4 * sizeof(PrStatus));
    g->pr.status_host = nullptr;
    g->pr.mem.release(s);
    g->pr = PrWork();
}

// Resident blocks per SM of `kernel` (raising its dynamic shared-memory limit
// first), asked once per graph and shape: the two queries cost a call 5 us.
static int occupancy(PrWork &w, const void *kernel, int threads, size_t smem, int &blocks) {
    for (const PrWork::Fit &f : w.fits)
        if (f.kernel == kernel && f.threads == threads && f.smem == smem) {
            blocks = f.blocks;
            return GP_OK;
        }
    // the opt-in is needed whenever dynamic + static shared memory exceeds 48 KiB; set it for any size
    if (smem > 0) GP_TRY(allow_smem(kernel));
    GP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, threads, smem));
    if (blocks < 1) return set_error(GP_ERR_UNSUPPORTED, "kernel does not fit on an SM (%zu B shared memory)", smem);
    w.fits.push_back({kernel, threads, smem, blocks});
    return GP_OK;
}

static int ensure_pr_work(gp_graph *g, cudaStream_t s) {
    PrWork &w = g->pr;
    if (w.ready) return GP_OK;
    const size_t n = (size_t)std::max<int64_t>(g->n, 1);
    const int64_t nbig = std::max(g->pull_bins.nbig, g->push_bins.nbig);
    // covers any grid: at most 32 resident blocks per SM, plus the blocks that add the adjoint's chunks
    w.max_blocks = (int)(std::max(g->num_sms * 32, grid_blocks(g, 256)) + (nbig + 511) / 512 + 64);
    GP_TRY(w.mem.alloc(w.r1, n, s));
    GP_TRY(w.mem.alloc(w.c0, n, s));
    GP_TRY(w.mem.alloc(w.c1, n, s));
    GP_TRY(w.mem.alloc(w.partials, (size_t)w.max_blocks, s));
    PrStatus *st = nullptr;
    GP_TRY(w.mem.alloc(st, 1, s));
    w.status = st;
    GP_TRY(w.mem.alloc(w.sync, 1, s));
    GP_TRY(pinned_alloc(&w.status_host, 4 * sizeof(PrStatus)));
    GP_TRY(pinned_device_ptr(w.status_host, &w.status_mirror));
    for (cudaEvent_t &e : w.ev) GP_CUDA(cudaEventCreate(&e));
    w.ready = true;
    return GP_OK;
}

static int ensure_vec(gp_graph *g, float *&slot, cudaStream_t s) {
    if (slot) return GP_OK;
    return g->pr.mem.alloc(slot, (size_t)std::max<int64_t>(g->n, 1), s);
}

static const void *push_kernel(bool W, bool fp64, bool hot) {
    if (fp64) {
        if (W) return hot ? (const void *)k_push_tiles<true, double, true> : (const void *)k_push_tiles<true, double, false>;
        return hot ? (const void *)k_push_tiles<false, double, true> : (const void *)k_push_tiles<false, double, false>;
    }
    if (W) return hot ? (const void *)k_push_tiles<true, float, true> : (const void *)k_push_tiles<true, float, false>;
    return hot ? (const void *)k_push_tiles<false, float, true> : (const void *)k_push_tiles<false, float, false>;
}

// Width of the push accumulator.  FP64 sums make the scattered result independent
// of the atomic order up to one final rounding, and cost no throughput while the
// 8n-byte accumulator stays in L2; above half the L2 its reductions reach DRAM
// (Erdos-Renyi 2^24: 4.7 ms per scatter against 2.5 ms in FP32), so the default
// (-1) switches to FP32 there unless some vertex takes more than
// PUSH_FP32_MAX_UPDATES updates per sweep (FP32 order noise at such hubs sets a
// residual floor near 1e-7).
constexpr int64_t PUSH_FP32_MAX_UPDATES = 4096;

// Pull graphs of at most this many edge tiles run all sweeps in one launch.
// Measured per call of 20 sweeps, a launch per step and one launch: R-MAT 2^14
// (1.7K tiles) 360 and 168 us, 2^16 (7.1K) 460 and 288, 2^18 (30K) 624 and 574,
// uniform 2^18 (16K) 732 and 606; above, the hot set that the launches keep in
// shared memory wins on skewed graphs (R-MAT 2^20, 123K tiles: 1480 and 1810).
constexpr int64_t LOOP_TILES = 32768;
static bool push_fp64(const gp_graph *g, int64_t max_updates) {
    if (g->opt.push_fp64_accum >= 0) return g->opt.push_fp64_accum != 0;
    const bool fits = 8 * g->n <= g->l2_bytes / 2;
    return fits || max_updates > PUSH_FP32_MAX_UPDATES;
}

// Whether the out- and in-edges are one array pair.
static bool one_order(const gp_graph *g) { return g->csr_off == g->csc_off; }

// One power iteration y = base + d * post_scale * (gather or scatter over the
// given adjacency) of a PageRank-type linear system, with on-device
// convergence; used for the forward pass and for the adjoint.
struct IterSpec {
    bool push;        // scatter with atomics (else gather, owner-only writes)
    bool hot;         // use the pull hot-contribution cache (forward pull only)
    const int64_t *off;
    const int32_t *idx;
    const float *w;
    EdgeTiles *tiles;     // the adjacency's tiles (built on first use); nullptr: adjoint pull,
    const BigBins *bins;  // which takes the chunks of its long lists
    const float *s;   // base vector (nullable: uniform base_uniform)
    float s_scale, base_uniform, d;
    const float *x0;  // start vector (nullable: 1/n)
    const float *post_scale, *cmul;
    int iters;
    double tol;
    int64_t max_updates;  // push: most updates any vertex takes per sweep (its max in-degree)
};

static int pr_iterate(gp_graph *g, const IterSpec &sp, float *out, PrStatus &fin, cudaStream_t s) {
    const int64_t n = g->n;
    PrWork &w = g->pr;
    float *R[2] = {out, w.r1};
    float *C[2] = {w.c0, w.c1};
    PrStatus *status = (PrStatus *)w.status;
    const bool push = sp.push;
    const bool W = sp.w != nullptr;

    PrArgs a;
    memset(&a, 0, sizeof(a));
    a.n = n;
    a.off = sp.off;
    a.idx = sp.idx;
    a.w = sp.w;
    if (sp.bins) {
        a.big = sp.bins->big;
        a.cstart = sp.bins->cstart;
        a.chunks = sp.bins->chunks;
        a.nbig = sp.bins->nbig;
        a.nchunks = sp.bins->nchunks;
        a.light_max = sp.bins->light_max;
    }
    a.s = sp.s;
    a.s_scale = sp.s_scale;
    a.base_uniform = sp.base_uniform;
    a.post_scale = sp.post_scale;
    a.cmul = sp.cmul;
    a.d = sp.d;
    a.tol = sp.tol;
    a.partials = w.partials;
    a.status = status;

    const int gb = grid_blocks(g, 256);
    const int64_t ntiles = (n + 31) / 32;
    bool hot = false;
    size_t smem = 0;
    const bool tiled = !push && sp.tiles;
    bool loop = false;  // all sweeps in one launch
    if (!push && !tiled) {
        loop = g->m <= LOOP_TILES * TILE_EDGES;
        if (!w.chunk_part) GP_TRY(w.mem.alloc(w.chunk_part, (size_t)std::max<int64_t>(a.nchunks, 1), s));
        a.chunk_part = w.chunk_part;
    }
    if (sp.tiles) {
        GP_TRY(build_tiles(g, *sp.tiles, sp.off, s));
        const EdgeTiles &t = *sp.tiles;
        a.m = g->m;
        a.heads = t.heads;
        a.tile_row = t.tile_row;
        a.rows = t.rows;
        a.long_rows = t.long_rows;
        a.acc = t.acc;
        a.carry = t.carry;
        a.ntiles = t.ntiles;
        a.nrows = t.nrows;
        a.nlong = t.nlong;
        loop = !push && t.ntiles <= LOOP_TILES;
    }
    if (tiled) {
        if (sp.hot && !loop) {
            if (g->pull_hot.slots != g->opt.pull_hot_slots) GP_TRY(build_pull_hot(g, g->opt.pull_hot_slots, s));
            hot = g->pull_hot.nhot > 0;
        }
        if (hot) {
            smem = (size_t)((g->pull_hot.nhot + 3) & ~int64_t(3)) * sizeof(float);
            a.c_hot = g->pull_hot.c_hot;
            a.hot_bits = g->pull_hot.bits;
            a.hot_prefix = g->pull_hot.prefix;
            a.nhot = g->pull_hot.nhot;
            a.idx = g->pull_hot.enc_idx;
        }
    }
    if (push && sp.hot) {
        if (g->push_hot.slots != g->opt.push_hot_slots) GP_TRY(build_push_hot(g, g->opt.push_hot_slots, s));
        hot = g->push_hot.nhot > 0;
        if (hot) {
            smem = (size_t)g->push_hot.nhot * sizeof(float);
            a.hot_id = g->push_hot.hot_id;
            a.nhot = g->push_hot.nhot;
            a.idx = g->push_hot.enc_idx;
        }
    }
    a.vec_tiles = ((uintptr_t)a.idx | (uintptr_t)a.w) % 32 == 0 ? (int32_t)(a.m / TILE_EDGES) : 0;
    int g1, g2;
    int tpt = TILE_THREADS;    // its threads per block
    const void *kl = nullptr;  // the kernel of all sweeps
    if (!push && !tiled && loop) {
        int ob = 0;
        kl = W ? (const void *)k_adj_loop<true> : (const void *)k_adj_loop<false>;
        tpt = 512;
        GP_TRY(occupancy(w, kl, tpt, 0, ob));
        g1 = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)ob * g->num_sms, (std::max(a.nchunks, ntiles) + 15) / 16));
        g2 = g1;
    } else if (!push && !tiled) {
        int ob = 0, ol = 0;
        GP_TRY(occupancy(w, W ? (const void *)k_adj_big<true> : (const void *)k_adj_big<false>, 1024, 0, ob));
        GP_TRY(occupancy(w, W ? (const void *)k_adj_light<true> : (const void *)k_adj_light<false>, 512, 0, ol));
        g1 = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)ob * g->num_sms, (a.nchunks + 31) / 32));
        a.split_blocks = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)ol * g->num_sms, (ntiles + 15) / 16));
        g2 = a.split_blocks + (int)std::min<int64_t>((a.nbig + 511) / 512, (int64_t)ol * g->num_sms);
    } else if (loop) {
        // a warp per tile and a thread per row where the grid holds that many, and no
        // more blocks than that to wait for
        constexpr int wpb = TILE_THREADS / 32;
        const int64_t regs = std::max((a.ntiles + wpb - 1) / wpb, (n + TILE_THREADS - 1) / TILE_THREADS);
        int ob = 0;
        kl = W ? (const void *)k_pull_loop_regs<true> : (const void *)k_pull_loop_regs<false>;
        GP_TRY(occupancy(w, kl, TILE_THREADS, 0, ob));
        if (regs > (int64_t)ob * g->num_sms || a.nlong > regs * wpb) {
            kl = W ? (const void *)k_pull_loop<true> : (const void *)k_pull_loop<false>;
            GP_TRY(occupancy(w, kl, TILE_THREADS, 0, ob));
        }
        g1 = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)ob * g->num_sms, regs));
        g2 = g1;
    } else if (!push) {
        int ob = 0, of = 0;
        const void *kb_ = W ? (hot ? (const void *)k_pull_tiles<true, true> : (const void *)k_pull_tiles<true, false>)
                            : (hot ? (const void *)k_pull_tiles<false, true> : (const void *)k_pull_tiles<false, false>);
        GP_TRY(occupancy(w, kb_, tpt, smem, ob));
        GP_TRY(occupancy(w, hot ? (const void *)k_pull_finish<true> : (const void *)k_pull_finish<false>, 256, 0, of));
        const int wpb = tpt / 32;
        g1 = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)ob * g->num_sms, (a.ntiles + wpb - 1) / wpb));
        g2 = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)of * g->num_sms, (n + 255) / 256));
    } else {
        const void *ks = push_kernel(W, push_fp64(g, sp.max_updates), hot);
        int os = 0;
        GP_TRY(occupancy(w, ks, TILE_THREADS, smem, os));
        const int wpb = TILE_THREADS / 32;
        g1 = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)os * g->num_sms, (a.ntiles + wpb - 1) / wpb));
        g2 = (int)std::max<int64_t>(1, std::min<int64_t>(gb, (n + 255) / 256));
    }
    if (g2 > w.max_blocks) return set_error(GP_ERR_INVALID, "internal: partials too small");
    a.nprev = g2;

    const int ib = (int)std::max<int64_t>(1, std::min<int64_t>(gb, (n + 255) / 256));
    const bool fp64 = push && push_fp64(g, sp.max_updates);
    if (fp64 && !w.acc64) GP_TRY(w.mem.alloc(w.acc64, (size_t)n, s));
    a.acc64 = fp64 ? w.acc64 : nullptr;
    GP_LAUNCH("pr_init", s, (k_pr_init<<<ib, 256, 0, s>>>(n, sp.x0, sp.cmul, R[0], C[0], (push && !fp64) ? R[1] : nullptr,
                                                          a.acc64, a.hot_bits, a.hot_prefix, a.c_hot, status, w.sync)));
    GP_TRY(check_launch("pr_init"));
    auto enqueue_sweep = [&](int k) -> int {
        PrArgs b = a;
        b.k = k;
        b.x = R[(k - 1) & 1];
        b.y = R[k & 1];
        if (!push) {
            b.c = C[(k - 1) & 1];
            b.c_next = C[k & 1];
            if (!tiled && W) {
                GP_LAUNCH("adj_big", s, (k_adj_big<true><<<g1, 1024, 0, s>>>(b)));
                GP_LAUNCH("adj_light", s, (k_adj_light<true><<<g2, 512, 0, s>>>(b)));
                return check_launch("adjoint sweep");
            }
            if (!tiled) {
                GP_LAUNCH("adj_big", s, (k_adj_big<false><<<g1, 1024, 0, s>>>(b)));
                GP_LAUNCH("adj_light", s, (k_adj_light<false><<<g2, 512, 0, s>>>(b)));
                return check_launch("adjoint sweep");
            }
            if (W && hot)
                GP_LAUNCH("pull_tiles", s, (k_pull_tiles<true, true><<<g1, tpt, smem, s>>>(b)));
            else if (W)
                GP_LAUNCH("pull_tiles", s, (k_pull_tiles<true, false><<<g1, tpt, 0, s>>>(b)));
            else if (hot)
                GP_LAUNCH("pull_tiles", s, (k_pull_tiles<false, true><<<g1, tpt, smem, s>>>(b)));
            else
                GP_LAUNCH("pull_tiles", s, (k_pull_tiles<false, false><<<g1, tpt, 0, s>>>(b)));
            if (hot)
                GP_LAUNCH("pull_finish", s, (k_pull_finish<true><<<g2, 256, 0, s>>>(b)));
            else
                GP_LAUNCH("pull_finish", s, (k_pull_finish<false><<<g2, 256, 0, s>>>(b)));
        } else {
            b.c = C[0];
            b.c_next = C[0];
            const void *ks = push_kernel(W, fp64, hot);
            {
                ProfScope ps("push_tiles", s);
                void *args[] = {&b};
                GP_CUDA(cudaLaunchKernel(ks, dim3((unsigned)g1), dim3(TILE_THREADS), args, smem, s));
            }
            if (fp64)
                GP_LAUNCH("push_epilogue", s, (k_push_epilogue<double><<<g2, 256, 0, s>>>(b)));
            else
                GP_LAUNCH("push_epilogue", s, (k_push_epilogue<float><<<g2, 256, 0, s>>>(b)));
        }
        return check_launch("pagerank sweep");
    };
    auto enqueue_finish = [&](int k_next, int slot) -> int {
        PrArgs b = a;
        b.k = k_next;
        GP_LAUNCH("pr_finish", s, (k_pr_finish<<<1, 256, 0, s>>>(b, (PrStatus *)w.status_mirror + slot)));
        return check_launch("pr_finish");
    };

    if (loop) {
        PrLoop P;
        P.a = a;
        P.R[0] = R[0];
        P.R[1] = R[1];
        P.C[0] = C[0];
        P.C[1] = C[1];
        P.iters = sp.iters;
        P.mirror = (PrStatus *)w.status_mirror + 2;
        P.sync = w.sync;
        volatile PrStatus *host = (PrStatus *)w.status_host + 2;
        host->iters_done = -1;  // the launch's last block of work replaces it
        {
            ProfScope ps(tiled ? "pull_loop" : "adj_loop", s);
            void *args[] = {&P};
            GP_CUDA(cudaLaunchCooperativeKernel(kl, dim3((unsigned)g1), dim3((unsigned)tpt), args, 0, s));
        }
        GP_CUDA(cudaStreamSynchronize(s));
        if (host->iters_done < 0) return set_error(GP_ERR_TIMEOUT, "PageRank: a grid barrier wait ran out");
        memcpy(&fin, (const PrStatus *)w.status_host + 2, sizeof(fin));
        return GP_OK;
    }
    const int poll = std::max(1, g->opt.poll_interval);
    const int iters = sp.iters;
    int issued = 0;
    cudaEvent_t evs[2] = {nullptr, nullptr};
    GP_CUDA(cudaEventCreateWithFlags(&evs[0], cudaEventDisableTiming));
    GP_CUDA(cudaEventCreateWithFlags(&evs[1], cudaEventDisableTiming));
    int pending[2] = {-1, -1};  // batch ids waiting on each slot
    int batch = 0, oldest = 0;
    bool stop = false;
    int st = GP_OK;
    if (sp.tol <= 0.0) {
        for (int k = 1; k <= iters && st == GP_OK; ++k) st = enqueue_sweep(k);
        if (st == GP_OK) st = enqueue_finish(iters + 1, 0);
        issued = iters;
    } else {
        // Sweeps worth enqueuing: the cap, lowered once two polls give the
        // residual's rate of decrease to the predicted stopping sweep plus one
        // (sweeps enqueued past the stop only return at once, but each still costs
        // a few microseconds of launches per kernel); raised again a batch at a
        // time if the iteration outlives the prediction.
        int limit = iters;
        int k_last = 0;
        double r_last = 0.0;
        while (st == GP_OK) {
            const int slot = batch & 1;
            if (!stop && issued < limit && pending[slot] < 0) {
                const int kb = std::min(poll, limit - issued);
                for (int i = 0; i < kb && st == GP_OK; ++i) st = enqueue_sweep(++issued);
                if (st == GP_OK) st = enqueue_finish(issued + 1, slot);
                if (st == GP_OK) {
                    cudaError_t e = cudaEventRecord(evs[slot], s);
                    if (e != cudaSuccess) st = set_error(GP_ERR_CUDA, "event: %s", cudaGetErrorString(e));
                }
                pending[slot] = batch++;
                continue;
            }
            const int os = oldest & 1;
            if (pending[os] < 0) {  // nothing outstanding
                if (!stop && issued < iters) {
                    limit = std::min(iters, issued + poll);
                    continue;
                }
                break;
            }
            cudaError_t e = cudaEventSynchronize(evs[os]);
            if (e != cudaSuccess) {
                st = set_error(GP_ERR_CUDA, "pagerank poll: %s", cudaGetErrorString(e));
                break;
            }
            pending[os] = -1;
            ++oldest;
            const PrStatus ps = ((const PrStatus *)w.status_host)[os];
            if (ps.done) {
                stop = true;
            } else {
                if (k_last > 0 && ps.iters_done > k_last && ps.residual > 0.0 && ps.residual < r_last) {
                    const double rate = std::pow(ps.residual / r_last, 1.0 / (ps.iters_done - k_last));
                    const double more = std::ceil(std::log(sp.tol / ps.residual) / std::log(rate));
                    if (more >= 0.0 && more < (double)iters)
                        limit = std::max<int64_t>(issued, std::min<int64_t>(iters, (int64_t)ps.iters_done + (int64_t)more + 1));
                }
                k_last = ps.iters_done;
                r_last = ps.residual;
            }
            if (stop && pending[oldest & 1] < 0) break;
            if (!stop && issued >= iters && pending[oldest & 1] < 0) break;
        }
    }
    cudaError_t e = cudaStreamSynchronize(s);
    cudaEventDestroy(evs[0]);
    cudaEventDestroy(evs[1]);
    if (st != GP_OK) return st;
    if (e != cudaSuccess) return set_error(GP_ERR_CUDA, "pagerank iteration: %s", cudaGetErrorString(e));
    // the final status: one more gate-only launch (the iteration has stopped,
    // so it changes nothing) writes it into mirror slot 2
    {
        PrArgs b = a;
        b.k = issued + 1;
        GP_LAUNCH("pr_finish", s, (k_pr_finish<<<1, 256, 0, s>>>(b, (PrStatus *)w.status_mirror + 2)));
        GP_TRY(check_launch("pr_finish"));
    }
    GP_CUDA(cudaStreamSynchronize(s));
    memcpy(&fin, (const PrStatus *)w.status_host + 2, sizeof(fin));  // written by the kernel, complete after the sync
    if ((fin.iters_done & 1) && fin.iters_done > 0) {
        const int cb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 4 * (int64_t)g->num_sms));
        GP_LAUNCH("copy_result", s, (k_copy_f32<<<cb, 256, 0, s>>>(n, R[1], out)));
        GP_TRY(check_launch("copy_result"));
    }
    return GP_OK;
}

// Device pointer for a caller array of n floats that may live in host memory.
static int device_input(gp_graph *g, const float *p, float *&slot, const float *&dev, cudaStream_t s) {
    dev = p;
    if (p && !is_device_ptr(p)) {
        GP_TRY(ensure_vec(g, slot, s));
        GP_CUDA(cudaMemcpyAsync(slot, p, g->n * sizeof(float), cudaMemcpyHostToDevice, s));
        dev = slot;
    }
    return GP_OK;
}

static int pr_validate(const gp_graph *g, int mode, float damping, int iters, double tol) {
    if (!g) return set_error(GP_ERR_INVALID, "graph is NULL");
    if (!(damping > 0.f && damping < 1.f)) return set_error(GP_ERR_INVALID, "damping %g outside (0, 1)", (double)damping);
    if (iters < 1) return set_error(GP_ERR_INVALID, "iters = %d < 1", iters);
    if (!(tol >= 0.0)) return set_error(GP_ERR_INVALID, "tol must be >= 0");
    if (mode != GP_PUSH && mode != GP_PULL && mode != GP_AUTO) return set_error(GP_ERR_INVALID, "bad mode %d", mode);
    return GP_OK;
}

}  // namespace gp

using namespace gp;

extern "C" int gp_pagerank(const gp_graph *gc, int mode, float damping, int iters, double tol,
                           const float *personalization, const float *x0, float *ranks_out, gp_pr_stats *stats,
                           void *stream) {
    clear_error();
    gp_graph *g = const_cast<gp_graph *>(gc);
    GP_TRY(pr_validate(g, mode, damping, iters, tol));
    if (!ranks_out) return set_error(GP_ERR_INVALID, "gp_pagerank: ranks_out is NULL");
    cudaStream_t s = (cudaStream_t)stream;
    if (mode == GP_AUTO) mode = g->opt.pr_auto_mode >= 0 ? g->opt.pr_auto_mode : GP_PULL;
    const int64_t n = g->n;
    if (stats) memset(stats, 0, sizeof(*stats));
    if (n == 0) {
        if (stats) {
            stats->mode_used = mode;
            stats->converged = 1;
        }
        return GP_OK;
    }
    GP_TRY(ensure_pr_work(g, s));
    PrWork &w = g->pr;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (stats) {
        ev0 = w.ev[0];
        ev1 = w.ev[1];
        GP_CUDA(cudaEventRecord(ev0, s));
    }
    const bool out_dev = is_device_ptr(ranks_out);
    float *R0 = ranks_out;
    if (!out_dev) {
        GP_TRY(ensure_vec(g, w.out_dev, s));
        R0 = w.out_dev;
    }
    const float *S = nullptr, *X0 = nullptr;
    GP_TRY(device_input(g, personalization, w.s_dev, S, s));
    GP_TRY(device_input(g, x0, w.x0_dev, X0, s));
    const bool push = mode == GP_PUSH;
    IterSpec sp;
    sp.push = push;
    sp.hot = true;
    sp.off = push ? g->csr_off : g->csc_off;
    sp.idx = push ? g->csr_idx : g->csc_idx;
    sp.w = g->weighted ? (push ? g->csr_w : g->csc_w) : nullptr;
    sp.tiles = push && !one_order(g) ? &g->out_tiles : &g->tiles;
    sp.bins = nullptr;
    sp.s = S;
    sp.s_scale = 1.0f - damping;
    sp.base_uniform = (float)((1.0 - (double)damping) / (double)n);
    sp.d = damping;
    sp.x0 = X0;
    sp.post_scale = nullptr;
    sp.cmul = g->inv_deg;
    sp.iters = iters;
    sp.tol = tol;
    sp.max_updates = g->max_in;
    PrStatus fin;
    GP_TRY(pr_iterate(g, sp, R0, fin, s));
    if (!out_dev) GP_CUDA(cudaMemcpyAsync(ranks_out, R0, n * sizeof(float), cudaMemcpyDeviceToHost, s));
    if (stats) {
        GP_CUDA(cudaEventRecord(ev1, s));
        GP_CUDA(cudaEventSynchronize(ev1));
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev0, ev1);
        stats->iters_done = fin.iters_done;
        stats->mode_used = mode;
        stats->residual = fin.residual;
        stats->ms = ms;
        stats->converged = (tol <= 0.0) ? 1 : fin.converged;
        stats->push_updates_l2 = (int64_t)fin.upd_l2;
        stats->push_updates_shared = (int64_t)fin.upd_shared;
        stats->push_updates_merged = (int64_t)fin.upd_merged;
        stats->push_flush_l2 = (int64_t)fin.flush_l2;
    } else if (!out_dev) {
        GP_CUDA(cudaStreamSynchronize(s));
    }
    if (tol > 0.0 && !fin.converged)
        return set_error(GP_ERR_NOT_CONVERGED, "residual %.3e >= tol %.3e after %d sweeps", fin.residual, tol,
                         fin.iters_done);
    return GP_OK;
}

extern "C" int gp_pagerank_backward(const gp_graph *gc, int mode, float damping, const float *ranks,
                                    const float *grad_ranks, float *grad_weights, float *grad_personalization,
                                    int iters, double tol, gp_pr_stats *stats, void *stream) {
    clear_error();
    gp_graph *g = const_cast<gp_graph *>(gc);
    GP_TRY(pr_validate(g, mode, damping, iters, tol));
    if (!ranks || !grad_ranks) return set_error(GP_ERR_INVALID, "gp_pagerank_backward: ranks and grad_ranks are required");
    cudaStream_t s = (cudaStream_t)stream;
    if (mode == GP_AUTO) mode = GP_PULL;
    const int64_t n = g->n, m = g->m;
    if (stats) memset(stats, 0, sizeof(*stats));
    if (n == 0) return GP_OK;
    GP_TRY(ensure_pr_work(g, s));
    PrWork &w = g->pr;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (stats) {
        ev0 = w.ev[0];
        ev1 = w.ev[1];
        GP_CUDA(cudaEventRecord(ev0, s));
    }
    const float *X = nullptr, *G = nullptr;
    GP_TRY(device_input(g, ranks, w.x0_dev, X, s));
    GP_TRY(device_input(g, grad_ranks, w.s_dev, G, s));
    GP_TRY(ensure_vec(g, w.lam, s));
    // (I - d P^T) lambda = g: the transposed sweep.  Pull gathers lambda over the
    // out-edges (CSR) of every vertex; push scatters lambda_v over the in-edges (CSC).
    const bool push = mode == GP_PUSH;
    IterSpec sp;
    sp.push = push;
    sp.hot = false;
    sp.off = push ? g->csc_off : g->csr_off;
    sp.idx = push ? g->csc_idx : g->csr_idx;
    sp.w = g->weighted ? (push ? g->csc_w : g->csr_w) : nullptr;
    sp.tiles = push ? &g->tiles : nullptr;
    sp.bins = &g->push_bins;
    sp.s = G;
    sp.s_scale = 1.0f;
    sp.base_uniform = 0.f;
    sp.d = damping;
    sp.x0 = G;
    sp.post_scale = g->inv_deg;
    sp.cmul = nullptr;
    sp.iters = iters;
    sp.tol = tol;
    sp.max_updates = g->max_out;  // the transposed scatter lands on sources
    PrStatus fin;
    GP_TRY(pr_iterate(g, sp, w.lam, fin, s));
    const int gb = grid_blocks(g, 256);
    if (grad_personalization) {
        const bool dev = is_device_ptr(grad_personalization);
        float *dst = grad_personalization;
        if (!dev) {
            GP_TRY(ensure_vec(g, w.out_dev, s));
            dst = w.out_dev;
        }
        const int b = (int)std::max<int64_t>(1, std::min<int64_t>(gb, (n + 255) / 256));
        GP_LAUNCH("grad_s", s, (k_grad_s<<<b, 256, 0, s>>>(n, 1.0f - damping, w.lam, dst)));
        GP_TRY(check_launch("grad_s"));
        if (!dev) GP_CUDA(cudaMemcpyAsync(grad_personalization, dst, n * sizeof(float), cudaMemcpyDeviceToHost, s));
    }
    if (grad_weights && m > 0) {
        const bool dev = is_device_ptr(grad_weights);
        float *dst = grad_weights;
        if (!dev) {
            if (!w.gw_dev) GP_TRY(w.mem.alloc(w.gw_dev, (size_t)m, s));
            dst = w.gw_dev;
        }
        GradArgs ga;
        ga.n = n;
        ga.off = g->csr_off;
        ga.idx = g->csr_idx;
        ga.x = X;
        ga.lam = w.lam;
        ga.g = G;
        ga.inv_deg = g->inv_deg;
        ga.chunks = g->push_bins.chunks;
        ga.nchunks = g->push_bins.nchunks;
        ga.light_max = g->push_bins.light_max;
        ga.d = damping;
        ga.normalized = g->normalized ? 1 : 0;
        ga.grad_w = dst;
        const int64_t ntiles = (n + 31) / 32;
        ga.split_blocks = (int)std::min<int64_t>(gb, (ga.nchunks + 7) / 8);
        const int b = ga.split_blocks + (int)std::max<int64_t>(1, std::min<int64_t>(gb, (ntiles + 7) / 8));
        GP_LAUNCH("grad_w", s, (k_grad_w<<<b, 256, 0, s>>>(ga)));
        GP_TRY(check_launch("grad_w"));
        if (!dev) GP_CUDA(cudaMemcpyAsync(grad_weights, dst, m * sizeof(float), cudaMemcpyDeviceToHost, s));
    }
    if (stats) {
        GP_CUDA(cudaEventRecord(ev1, s));
        GP_CUDA(cudaEventSynchronize(ev1));
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev0, ev1);
        stats->iters_done = fin.iters_done;
        stats->mode_used = mode;
        stats->residual = fin.residual;
        stats->ms = ms;
        stats->converged = (tol <= 0.0) ? 1 : fin.converged;
    }
    GP_CUDA(cudaStreamSynchronize(s));
    if (tol > 0.0 && !fin.converged)
        return set_error(GP_ERR_NOT_CONVERGED, "adjoint residual %.3e >= tol %.3e after %d sweeps", fin.residual, tol,
                         fin.iters_done);
    return GP_OK;
}

extern "C" int gp_graph_set_weights(gp_graph *g, const float *csr_w, const float *csc_w, void *stream) {
    clear_error();
    if (!g) return set_error(GP_ERR_INVALID, "gp_graph_set_weights: graph is NULL");
    if (!g->weighted) return set_error(GP_ERR_UNSUPPORTED, "gp_graph_set_weights: the graph was uploaded without weights");
    if (!csr_w || !is_device_ptr(csr_w)) return set_error(GP_ERR_INVALID, "gp_graph_set_weights: csr_w must be device memory");
    const bool shared = g->csc_idx == g->csr_idx;
    if (!shared && (!csc_w || !is_device_ptr(csc_w)))
        return set_error(GP_ERR_INVALID, "gp_graph_set_weights: csc_w must be device memory");
    cudaStream_t s = (cudaStream_t)stream;
    g->csr_w = csr_w;
    g->csc_w = shared ? csr_w : csc_w;
    sssp_new_weights(g);
    // weights as given: the scale is 1 (0 where there are no edges) whatever they are
    return g->normalized ? weight_scale(g, s) : GP_OK;
}
