// tc.cu -- per-vertex triangle counts by the push- and pull-based
// NodeIterator of the paper's Section 3 listing.
//
// Every edge is directed from its end of lower degree to the other (ties by
// id), so that a triangle has one lowest vertex u, whose other two corners v
// and x are both out-neighbours of u and joined by v -> x.  u's warp or block
// keeps N+(u) in shared memory (a hash table or a bitmap), streams N+(v) for every v in
// N+(u), and counts the hits for each member of N+(u) beside its entry.
//   pull: the counts go into u's slots of its out-neighbours' in-lists, each
//         written by u alone; then every vertex adds its own slots (only v's
//         owner writes tc[v]);
//   push: u adds them to its out-neighbours' tc with fetch-and-adds (the
//         listing's FAA atomics).
// The listing meets every triangle six times (each corner, each order of the
// other two) and halves; here it is met once.  The directed lists are laid out
// once per graph.  Graphs outside the contract that the layout detects
// (unsorted or duplicate edges, an edge without its reverse), lists of more than
// TC_MAX_OUT out-neighbours and a layout that finds no memory take the listing
// itself (k_tc): one warp per edge (v, w1), the shorter list's elements
// binary-searched in the longer one.
#include <algorithm>
#include <cstring>

#include "gp_internal.cuh"

namespace gp {

struct TcArgs {
    int64_t n;
    const int64_t *off;
    const int32_t *idx;
    const int32_t *rank;    // [n] rank among heavy vertices, -1 light
    const int64_t *cstart;  // heavy vertex r's chunks: [cstart[r], cstart[r+1])
    const Chunk *chunks;
    const int32_t *big;     // heavy vertex of rank r
    int64_t nchunks, nbig;
    int push;
    unsigned long long *tc;       // [n] counts (push: atomics; pull: owner writes)
    unsigned long long *chunk_part;  // pull: [nchunks] sums of heavy vertices' chunks
    unsigned long long *probes;   // elements searched (statistic)
};

// |a n b| \ {x0, x1} for sorted a[0..na), b[0..nb); every lane gets the count.
__device__ __forceinline__ unsigned long long warp_intersect(const int32_t *__restrict__ a, int na,
                                                             const int32_t *__restrict__ b, int nb, int32_t x0,
                                                             int32_t x1) {
    unsigned long long cnt = 0;
    for (int i = lane_id(); i < na; i += 32) {
        const int32_t x = __ldg(a + i);
        if (x == x0 || x == x1) continue;
        int lo = 0, hi = nb;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(b + mid) < x)
                lo = mid + 1;
            else
                hi = mid;
        }
        cnt += lo < nb && __ldg(b + lo) == x;
    }
    return warp_sum(cnt);
}

// Triangle-closing count of the edge slots [e0, e1) of v, summed; push also
// credits each w1 with its own count.
__device__ unsigned long long tc_edges(const TcArgs &a, int32_t v, int64_t e0, int64_t e1, unsigned long long &probes) {
    const int64_t bv = a.off[v];
    const int dv = (int)(a.off[v + 1] - bv);
    unsigned long long sum = 0;
    for (int64_t e = e0; e < e1; ++e) {
        const int32_t w1 = __ldg(a.idx + e);
        if (w1 == v) continue;  // self-loop
        const int64_t bw = a.off[w1];
        const int dw = (int)(a.off[w1 + 1] - bw);
        const bool vshort = dv <= dw;
        const unsigned long long k = vshort ? warp_intersect(a.idx + bv, dv, a.idx + bw, dw, v, w1)
                                            : warp_intersect(a.idx + bw, dw, a.idx + bv, dv, v, w1);
        if (lane_id() == 0) probes += (unsigned long long)(vshort ? dv : dw);
        if (a.push) {
            if (k && lane_id() == 0) atomicAdd(a.tc + w1, k);
        } else {
            sum += k;
        }
    }
    return sum;
}

__global__ void __launch_bounds__(256) k_tc(TcArgs a) {
    const int lane = lane_id();
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long probes = 0;
    // heavy vertices: one chunk of the list per unit
    for (int64_t j = warp; j < a.nchunks; j += nwarps) {
        const Chunk ch = a.chunks[j];
        const unsigned long long s = tc_edges(a, ch.v, ch.beg, ch.beg + ch.len, probes);
        if (!a.push && lane == 0) a.chunk_part[j] = s;
    }
    // light vertices: the whole list per unit
    for (int64_t v = warp; v < a.n; v += nwarps) {
        if (a.rank[v] >= 0) continue;
        const int64_t b = a.off[v], e = a.off[v + 1];
        if (b == e) {
            if (!a.push && lane == 0) a.tc[v] = 0;
            continue;
        }
        const unsigned long long s = tc_edges(a, (int32_t)v, b, e, probes);
        if (!a.push && lane == 0) a.tc[v] = s / 2;
    }
    probes = warp_sum(probes);
    if (lane == 0 && probes) atomicAdd(a.probes, probes);
}

// pull: heavy vertices add their chunk sums (one writer per count).
__global__ void k_tc_combine(TcArgs a) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < a.nbig; r += stride) {
        unsigned long long s = 0;
        for (int64_t j = a.cstart[r]; j < a.cstart[r + 1]; ++j) s += a.chunk_part[j];
        a.tc[a.big[r]] = s / 2;
    }
}

// push: every count was met twice; halve, and sum for the total.
__global__ void k_tc_finish(int64_t n, int push, unsigned long long *tc, unsigned long long *total) {
    __shared__ unsigned long long sm[32];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long s = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        unsigned long long c = tc[v];
        if (push) {
            c /= 2;
            tc[v] = c;
        }
        s += c;
    }
    s = block_sum(s, sm);
    if (threadIdx.x == 0 && s) atomicAdd(total, s);
}

// ------------------------------------------------------------------ directed lists

// Out-neighbours up to which a warp counts for a vertex.  Kernel times at 16, 32
// and 64: R-MAT 2^18 1070, 1041 and 1188 us, n = 50K 180, 197 and 302, n = 400K 2406,
// 2143 and 2165; uniform 260K (lists of about 16) 810, 200 and 200.
constexpr int TC_WARP_OUT = 32;
constexpr int TC_MAX_OUT = 8192;    // and a block (table of at most 16384 entries)
constexpr int TC_WARP_TABLE = 256;  // entries of a warp's table
constexpr int TC_WARPS = 8;         // warps per block of the counting kernels
constexpr int32_t TC_FREE = -1;     // key of a free entry

struct TcPlanStat {
    unsigned long long general;  // the graph is outside the contract
    unsigned long long max_out;
    unsigned long long probes;   // sum over ordered edges of the shorter list's length
    unsigned long long out, in;  // lengths of the two kinds of list, all vertices
    unsigned long long light, heavy, mid, wide;  // vertices by out-neighbours and by in-list (see TcRun, k_tc_gather)
};

// v before w: lower degree, or equal and lower id.
__device__ __forceinline__ bool tc_before(int64_t dv, int32_t v, int64_t dw, int32_t w) {
    return dv < dw || (dv == dw && v < w);
}

// In-lists of over TC_WIDE entries take a block each in the pull's gather, of over 32 a warp.
constexpr int TC_WIDE = 1024;

// Per vertex, the neighbours after it (out) and before it (in), a warp per vertex.
__global__ void __launch_bounds__(256) k_tc_count(int64_t n, const int64_t *off, const int32_t *idx, int64_t *nout,
                                                  int64_t *nin, TcPlanStat *st) {
    const int lane = lane_id();
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long probes = 0, most = 0, outs = 0, ins = 0;
    unsigned kind[4] = {0, 0, 0, 0};
    bool bad = false;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += nwarps) {
        const int64_t b = off[v], e = off[v + 1];
        int out = 0, in = 0;
        constexpr int U = 4;
        for (int64_t e0 = b + lane; e0 < e; e0 += 32 * U) {
            int32_t w[U];
            int64_t dw[U];
#pragma unroll
            for (int q = 0; q < U; ++q) w[q] = e0 + 32 * q < e ? __ldg(idx + e0 + 32 * q) : (int32_t)v;
#pragma unroll
            for (int q = 0; q < U; ++q) dw[q] = off[w[q] + 1] - off[w[q]];
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const int64_t p = e0 + 32 * q;
                if (p >= e) continue;
                bad |= p > b && __ldg(idx + p - 1) >= w[q];
                if (w[q] == (int32_t)v) continue;  // self-loop
                probes += (unsigned long long)(dw[q] < e - b ? dw[q] : e - b);
                if (tc_before(e - b, (int32_t)v, dw[q], w[q]))
                    ++out;
                else
                    ++in;
            }
        }
        out = warp_sum(out);
        in = warp_sum(in);
        most = max(most, (unsigned long long)out);
        outs += (unsigned)out;
        ins += (unsigned)in;
        kind[0] += out >= 2 && out <= TC_WARP_OUT;
        kind[1] += out > TC_WARP_OUT;
        kind[2] += in > 32 && in <= TC_WIDE;
        kind[3] += in > TC_WIDE;
        if (lane == 0) {
            nout[v] = out;
            nin[v] = in;
        }
    }
    probes = warp_sum(probes);
    bad = __any_sync(FULL, bad);
    if (lane == 0) {
        if (probes) atomicAdd(&st->probes, probes);
        if (most) atomicMax(&st->max_out, most);
        if (bad) atomicOr(&st->general, 1ull);
        if (outs) atomicAdd(&st->out, outs);
        if (ins) atomicAdd(&st->in, ins);
        if (kind[0]) atomicAdd(&st->light, (unsigned long long)kind[0]);
        if (kind[1]) atomicAdd(&st->heavy, (unsigned long long)kind[1]);
        if (kind[2]) atomicAdd(&st->mid, (unsigned long long)kind[2]);
        if (kind[3]) atomicAdd(&st->wide, (unsigned long long)kind[3]);
    }
}

// The lists of vertices by kind, in any order (at[] counts them).
__global__ void k_tc_kinds(int64_t n, const int64_t *out_off, const int64_t *in_off, int32_t *light, int32_t *heavy,
                           int32_t *mid, int32_t *wide, unsigned long long *at) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~int64_t(31); v0 < n; v0 += stride) {
        const int64_t v = v0 + lane_id();
        const int64_t out = v < n ? out_off[v + 1] - out_off[v] : 0, in = v < n ? in_off[v + 1] - in_off[v] : 0;
        const bool is[4] = {out >= 2 && out <= TC_WARP_OUT, out > TC_WARP_OUT, in > 32 && in <= TC_WIDE, in > TC_WIDE};
        int32_t *list[4] = {light, heavy, mid, wide};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned m = __ballot_sync(FULL, is[k]);
            if (!m) continue;
            unsigned long long p = 0;
            if (lane_id() == __ffs(m) - 1) p = atomicAdd(at + k, (unsigned long long)__popc(m));
            p = __shfl_sync(FULL, p, __ffs(m) - 1);
            if (is[k]) list[k][p + __popc(m & ((1u << lane_id()) - 1u))] = (int32_t)v;
        }
    }
}

// The two lists of every vertex, in the order of its neighbours.
__global__ void __launch_bounds__(256) k_tc_lists(int64_t n, const int64_t *off, const int32_t *idx, const int64_t *out_off,
                                                  const int64_t *in_off, int32_t *out, int32_t *in) {
    const int lane = lane_id();
    const unsigned below = (1u << lane) - 1u;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += nwarps) {
        const int64_t b = off[v], e = off[v + 1];
        int64_t po = out_off[v], pi = in_off[v];
        constexpr int U = 4;
        for (int64_t e0 = b; e0 < e; e0 += 32 * U) {
            int32_t w[U];
            int64_t dw[U];
#pragma unroll
            for (int q = 0; q < U; ++q) w[q] = e0 + 32 * q + lane < e ? __ldg(idx + e0 + 32 * q + lane) : (int32_t)v;
#pragma unroll
            for (int q = 0; q < U; ++q) dw[q] = off[w[q] + 1] - off[w[q]];
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const bool other = w[q] != (int32_t)v;
                const bool after = other && tc_before(e - b, (int32_t)v, dw[q], w[q]);
                const unsigned mo = __ballot_sync(FULL, after), mi = __ballot_sync(FULL, other && !after);
                if (after)
                    out[po + __popc(mo & below)] = w[q];
                else if (other)
                    in[pi + __popc(mi & below)] = w[q];
                po += __popc(mo);
                pi += __popc(mi);
            }
        }
    }
}

// rev[e]: the place of u in the in-list of x, for every directed edge e = (u -> x)
// (-1: not there; the counts made so are dropped, but stay in bounds).
__global__ void __launch_bounds__(256) k_tc_reverse(int64_t n, const int64_t *out_off, const int64_t *in_off,
                                                    const int32_t *out, const int32_t *in, int32_t *rev, TcPlanStat *st) {
    const int lane = lane_id();
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    bool bad = false;
    for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += nwarps) {
        for (int64_t e = out_off[u] + lane; e < out_off[u + 1]; e += 32) {
            const int32_t x = out[e];
            const int32_t *list = in + in_off[x];
            const int len = (int)(in_off[x + 1] - in_off[x]);
            int lo = 0, hi = len;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (__ldg(list + mid) < (int32_t)u)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            if (lo == len || __ldg(list + lo) != (int32_t)u) {
                bad = true;  // no edge back, so no slot
                lo = -1;
            }
            rev[e] = lo;
        }
    }
    if (__any_sync(FULL, bad) && lane == 0) atomicOr(&st->general, 2ull);
}

// ------------------------------------------------------------------ counting

struct TcRun {
    const int64_t *out_off, *in_off;
    const int32_t *out, *rev;
    const int32_t *list;         // the vertices this launch counts for
    int64_t count;
    int table;                   // entries of a block's table (a power of two)
    int push;
    int32_t *slots;              // pull: per in-list entry, the triangles counted by that neighbour
    unsigned long long *own;     // pull: [n] triangles whose lowest vertex this is
    unsigned long long *tc;      // push: [n] counts
    unsigned long long *total;
    unsigned long long *ticket;  // the next entry of `list` to hand out
};

// u's out-neighbours: a filter of TC_FILTER bits per table entry, which tells
// most of the other vertices off with one load, then an open-addressed table
// with a count per entry.  Both are indexed by one hash, the entry by its high
// bits.  (Without the filter a warp walks the longest of its 32 probe runs for
// every 32 elements: 64 issued instructions, against about half of that.)
constexpr int TC_FILTER = 16;
struct TcTable {
    int32_t *key;
    int *cnt;
    uint32_t *filter;
    unsigned bits;  // TC_FILTER * entries - 1
    __device__ __forceinline__ unsigned hash(int32_t x) const { return ((unsigned)x * 0x9E3779B1u >> 9) & bits; }
    __device__ __forceinline__ unsigned next(unsigned e) const { return (e + 1) & (bits / TC_FILTER); }
    // entry of x, or -1
    __device__ __forceinline__ int find(int32_t x) const {
        const unsigned h = hash(x);
        if (!((filter[h >> 5] >> (h & 31)) & 1u)) return -1;
        for (unsigned e = h / TC_FILTER;; e = next(e)) {
            const int32_t k = key[e];
            if (k == x) return (int)e;
            if (k == TC_FREE) return -1;
        }
    }
    __device__ __forceinline__ void insert(int32_t x) const {
        const unsigned h = hash(x);
        atomicOr(filter + (h >> 5), 1u << (h & 31));
        unsigned e = h / TC_FILTER;
        while (atomicCAS(key + e, TC_FREE, x) != TC_FREE) e = next(e);
    }
};

// Hits of the list elements [b, e) in the table, counted beside their entries, by the whole warp.
__device__ __forceinline__ int tc_stream(const TcRun &R, int64_t b, int64_t e, const TcTable &T) {
    constexpr int U = 4;
    int hits = 0;
    for (int64_t p = b + lane_id(); p < e; p += 32 * U) {
        int32_t x[U];
#pragma unroll
        for (int q = 0; q < U; ++q) x[q] = p + 32 * q < e ? __ldg(R.out + p + 32 * q) : TC_FREE;
#pragma unroll
        for (int q = 0; q < U; ++q) {
            if (x[q] < 0) continue;
            const int at = T.find(x[q]);
            if (at >= 0) {
                atomicAdd(T.cnt + at, 1);
                ++hits;
            }
        }
    }
    return hits;
}

// What u counted for its out-neighbour of edge e: into that one's in-list slot, or onto its count.
__device__ __forceinline__ void tc_give(const TcRun &R, int64_t e, int c) {
    const int32_t x = R.out[e];
    if (!R.push) {
        if (R.rev[e] >= 0) R.slots[R.in_off[x] + R.rev[e]] = c;
    } else if (c) {
        atomicAdd(R.tc + x, (unsigned long long)c);
    }
}

__device__ __forceinline__ void tc_own(const TcRun &R, int32_t u, unsigned long long t) {
    if (!R.push)
        R.own[u] = t;
    else if (t)
        atomicAdd(R.tc + u, t);
}

// Measured on R-MAT 2^18 (3.8M undirected edges, 6.6e8 list elements streamed):
// k_tc 47.9 ms; this kernel and the next but one 290 + 752 us, the gather 16 us.
// A warp per vertex u of few out-neighbours.  Its out-neighbours' lists, 32 at a
// time, are one stream of edges over the lanes (whatever their lengths), four
// windows of 32 in flight (a list each where they average 32 elements and more).
__global__ void __launch_bounds__(TC_WARPS * 32) k_tc_warp(TcRun R) {
    __shared__ int32_t s_key[TC_WARPS][TC_WARP_TABLE];
    __shared__ int s_cnt[TC_WARPS][TC_WARP_TABLE];
    __shared__ uint32_t s_filter[TC_WARPS][TC_WARP_TABLE * TC_FILTER / 32];
    constexpr int U = 4;
    const int lane = lane_id(), wib = threadIdx.x >> 5;
    const TcTable T = {s_key[wib], s_cnt[wib], s_filter[wib], TC_WARP_TABLE * TC_FILTER - 1};
    for (int i = lane; i < TC_WARP_TABLE; i += 32) {
        T.key[i] = TC_FREE;
        T.cnt[i] = 0;
    }
    for (int i = lane; i < TC_WARP_TABLE * TC_FILTER / 32; i += 32) T.filter[i] = 0u;
    unsigned long long total = 0;
    constexpr int TAKE = 4;  // vertices per ticket
    while (true) {
        unsigned long long t0 = 0;
        if (lane == 0) t0 = atomicAdd(R.ticket, (unsigned long long)TAKE);
        t0 = __shfl_sync(FULL, t0, 0);
        if ((int64_t)t0 >= R.count) break;
        const int64_t t1 = min((int64_t)t0 + TAKE, R.count);
        for (int64_t t = (int64_t)t0; t < t1; ++t) {
            const int32_t u = R.list[t];
            const int64_t b = R.out_off[u], e = R.out_off[u + 1];
            __syncwarp();
            for (int64_t p = b + lane; p < e; p += 32) T.insert(R.out[p]);
            __syncwarp();
            unsigned long long sum = 0;
            for (int64_t p = b; p < e; p += 32) {
                int64_t lb = 0;
                int len = 0, at_v = 0;
                if (p + lane < e) {
                    const int32_t v = R.out[p + lane];
                    lb = R.out_off[v];
                    len = (int)(R.out_off[v + 1] - lb);
                    at_v = T.find(v);
                }
                const int incl = warp_incl_scan(len), excl = incl - len;
                const int E = __shfl_sync(FULL, incl, 31);
                int hits = 0;
                // long lists one after another: finding each element's list costs more than their ends waste
                const bool each = E >= 32 * 32;
                for (int i = 0; each && i < 32 && p + i < e; ++i) {
                    const int64_t vb = __shfl_sync(FULL, lb, i);
                    const int vl = __shfl_sync(FULL, len, i);
                    const int mine = tc_stream(R, vb, vb + vl, T);
                    const int all = warp_sum(mine);
                    hits += mine;
                    if (lane == i && all) atomicAdd(T.cnt + at_v, all);
                }
                for (int e0 = 0; !each && e0 < E; e0 += 32 * U) {
                    int32_t x[U];
                    int from[U];
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        const int id = e0 + 32 * q + lane;
                        int k = 0;  // the list that holds element id
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) {
                            const int ek = __shfl_sync(FULL, excl, k + o);
                            if (ek <= id) k += o;
                        }
                        const int64_t kb = __shfl_sync(FULL, lb, k);
                        const int ke = __shfl_sync(FULL, excl, k);
                        from[q] = __shfl_sync(FULL, at_v, k);
                        x[q] = id < E ? __ldg(R.out + kb + (id - ke)) : TC_FREE;
                    }
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        if (x[q] < 0) continue;
                        const int at = T.find(x[q]);
                        if (at >= 0) {
                            atomicAdd(T.cnt + at, 1);
                            atomicAdd(T.cnt + from[q], 1);
                            ++hits;
                        }
                    }
                }
                sum += (unsigned long long)hits;
            }
            sum = warp_sum(sum);
            __syncwarp();
            // counts read by every lane before any entry is freed
            int c[(TC_WARP_OUT + 31) / 32], at[(TC_WARP_OUT + 31) / 32];
            unsigned h[(TC_WARP_OUT + 31) / 32];
#pragma unroll
            for (int q = 0; q < (TC_WARP_OUT + 31) / 32; ++q) {
                const int64_t p = b + 32 * q + lane;
                const int32_t x = p < e ? R.out[p] : 0;
                at[q] = p < e ? T.find(x) : -1;
                c[q] = at[q] >= 0 ? T.cnt[at[q]] : 0;
                h[q] = T.hash(x);
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < (TC_WARP_OUT + 31) / 32; ++q) {
                if (at[q] < 0) continue;
                T.key[at[q]] = TC_FREE;
                T.cnt[at[q]] = 0;
                T.filter[h[q] >> 5] = 0u;
                tc_give(R, b + 32 * q + lane, c[q]);
            }
            if (lane == 0) tc_own(R, u, sum);
            total += sum;
        }
    }
    if (lane == 0 && total) atomicAdd(R.total, total);
}

// A block per vertex u of many out-neighbours, a warp per list N+(v).
__global__ void __launch_bounds__(TC_WARPS * 32) k_tc_block(TcRun R) {
    extern __shared__ int32_t s_table[];
    __shared__ long long s_ticket;
    __shared__ unsigned long long s_sum[32];
    const int lane = lane_id(), wib = threadIdx.x >> 5;
    unsigned long long total = 0;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s_ticket = (long long)atomicAdd(R.ticket, 1ull);
        __syncthreads();
        const int64_t t = s_ticket;
        if (t >= R.count) break;
        const int32_t u = R.list[t];
        const int64_t b = R.out_off[u], e = R.out_off[u + 1];
        int size = 4 * TC_WARP_OUT;  // four times the list, where the table has the room
        while (size < R.table && size < 4 * (e - b)) size *= 2;
        const TcTable T = {s_table, s_table + size, (uint32_t *)s_table + 2 * size, (unsigned)size * TC_FILTER - 1u};
        for (int i = threadIdx.x; i < size; i += blockDim.x) {
            T.key[i] = TC_FREE;
            T.cnt[i] = 0;
        }
        for (int i = threadIdx.x; i < size * TC_FILTER / 32; i += blockDim.x) T.filter[i] = 0u;
        __syncthreads();
        for (int64_t p = b + threadIdx.x; p < e; p += blockDim.x) T.insert(R.out[p]);
        __syncthreads();
        unsigned long long sum = 0;
        for (int64_t p0 = b + wib; p0 < e; p0 += 32 * TC_WARPS) {
            // the warp's next 32 lists located at once
            const int64_t p = p0 + (int64_t)lane * TC_WARPS;
            int64_t lb = 0, le = 0;
            int at_v = -1;
            if (p < e) {
                const int32_t v = R.out[p];
                lb = R.out_off[v];
                le = R.out_off[v + 1];
                at_v = T.find(v);
            }
            const int lists = __popc(__ballot_sync(FULL, at_v >= 0));
            for (int i = 0; i < lists; ++i) {
                const int64_t vb = __shfl_sync(FULL, lb, i), ve = __shfl_sync(FULL, le, i);
                const int hits = warp_sum(tc_stream(R, vb, ve, T));
                if (lane == i && hits) {
                    atomicAdd(T.cnt + at_v, hits);
                    sum += (unsigned long long)hits;
                }
            }
        }
        sum = block_sum(sum, s_sum);  // (a block barrier: every count is in)
        for (int64_t p = b + threadIdx.x; p < e; p += blockDim.x) tc_give(R, p, T.cnt[T.find(R.out[p])]);
        if (threadIdx.x == 0) {
            tc_own(R, u, sum);
            total += sum;
        }
    }
    if (threadIdx.x == 0 && total) atomicAdd(R.total, total);
}

// The same with u's out-neighbours as a bitmap over all vertices, for graphs
// whose bitmap fits in shared memory: a search is one load and a test, and a
// hit's place in the list is the word's first place and a bit count, with no
// probing.  Bound by the bank conflicts of those loads and of the counts (13
// cycles of an SM per 32 elements): 629 -> 529 us on R-MAT 2^18 with the lists of
// more than 64, 755 with those of more than 32.
constexpr int TC_BITS_WARPS = 16;
constexpr int64_t TC_BITS_MAX = int64_t(1) << 19;  // vertices: two blocks of 96 KB per SM

__global__ void __launch_bounds__(TC_BITS_WARPS * 32) k_tc_bits(TcRun R, int64_t n) {
    extern __shared__ int32_t s_table[];
    __shared__ long long s_ticket;
    __shared__ unsigned long long s_sum[32];
    const int lane = lane_id(), wib = threadIdx.x >> 5;
    const int nwords = (int)((n + 31) >> 5);
    uint32_t *bits = (uint32_t *)s_table;
    int *cnt = s_table + nwords;                       // [the longest list]
    uint16_t *first = (uint16_t *)(cnt + R.table);     // place in the list of a word's first vertex
    for (int i = threadIdx.x; i < nwords; i += blockDim.x) bits[i] = 0u;
    unsigned long long total = 0;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s_ticket = (long long)atomicAdd(R.ticket, 1ull);
        __syncthreads();
        const int64_t t = s_ticket;
        if (t >= R.count) break;
        const int32_t u = R.list[t];
        const int64_t b = R.out_off[u], e = R.out_off[u + 1];
        for (int64_t p = b + threadIdx.x; p < e; p += blockDim.x) {
            const int32_t x = R.out[p];
            if (p == b || R.out[p - 1] >> 5 != x >> 5) first[x >> 5] = (uint16_t)(p - b);
            atomicOr(bits + (x >> 5), 1u << (x & 31));
            cnt[p - b] = 0;
        }
        __syncthreads();
        unsigned long long sum = 0;
        for (int64_t p0 = b + wib; p0 < e; p0 += 32 * TC_BITS_WARPS) {
            // the warp's next 32 lists located at once
            const int64_t p = p0 + (int64_t)lane * TC_BITS_WARPS;
            int64_t lb = 0;
            int len = 0;
            if (p < e) {
                const int32_t v = R.out[p];
                lb = R.out_off[v];
                len = (int)(R.out_off[v + 1] - lb);
            }
            const int lists = __popc(__ballot_sync(FULL, p < e));
            for (int i = 0; i < lists; ++i) {
                const int32_t *list = R.out + __shfl_sync(FULL, lb, i);
                const int l = __shfl_sync(FULL, len, i);
                int hits = 0;
                constexpr int U = 4;
                for (int j = lane; j < l; j += 32 * U) {
                    int32_t x[U];
#pragma unroll
                    for (int q = 0; q < U; ++q) x[q] = j + 32 * q < l ? __ldg(list + j + 32 * q) : -1;
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        if (x[q] < 0) continue;
                        const uint32_t word = bits[x[q] >> 5], bit = 1u << (x[q] & 31);
                        if (word & bit) {
                            atomicAdd(cnt + first[x[q] >> 5] + __popc(word & (bit - 1u)), 1);
                            ++hits;
                        }
                    }
                }
                hits = __reduce_add_sync(FULL, hits);
                if (lane == i && hits) {
                    atomicAdd(cnt + (p - b), hits);
                    sum += (unsigned)hits;
                }
            }
        }
        sum = block_sum(sum, s_sum);  // (a block barrier: every count is in)
        for (int64_t p = b + threadIdx.x; p < e; p += blockDim.x) {
            tc_give(R, p, cnt[p - b]);
            bits[R.out[p] >> 5] = 0u;
        }
        if (threadIdx.x == 0) {
            tc_own(R, u, sum);
            total += sum;
        }
    }
    if (threadIdx.x == 0 && total) atomicAdd(R.total, total);
}

// pull: a vertex's count is its own triangles and those its in-neighbours
// counted for it.  Long in-lists take a block each (a warp over 25K entries took
// 0.5 ms), shorter ones a warp, the others a thread.
__global__ void __launch_bounds__(256) k_tc_gather(int64_t n, const int64_t *in_off, const int32_t *slots,
                                                   const unsigned long long *own, const int32_t *mid, int64_t nmid,
                                                   const int32_t *wide, int64_t nwide, unsigned long long *tc) {
    __shared__ unsigned long long sm[32];
    for (int64_t i = blockIdx.x; i < nwide; i += gridDim.x) {
        const int32_t v = wide[i];
        const int64_t e = in_off[v + 1];
        unsigned long long s = 0;
#pragma unroll 4
        for (int64_t p = in_off[v] + threadIdx.x; p < e; p += 256) s += (unsigned long long)slots[p];
        s = block_sum(s, sm);
        if (threadIdx.x == 0) tc[v] = own[v] + s;
    }
    const int64_t thread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nthreads = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = thread >> 5; i < nmid; i += nthreads >> 5) {
        const int32_t v = mid[i];
        const int64_t e = in_off[v + 1];
        unsigned long long s = 0;
#pragma unroll 4
        for (int64_t p = in_off[v] + lane_id(); p < e; p += 32) s += (unsigned long long)slots[p];
        s = warp_sum(s);
        if (lane_id() == 0) tc[v] = own[v] + s;
    }
    for (int64_t v = thread; v < n; v += nthreads) {
        const int64_t b = in_off[v], e = in_off[v + 1];
        if (e - b > 32) continue;
        unsigned long long s = own[v];
#pragma unroll 4
        for (int64_t p = b; p < e; ++p) s += (unsigned long long)slots[p];
        tc[v] = s;
    }
}

}  // namespace gp

using namespace gp;

struct gp_tc_work {
    bool ready = false, general = false;
    TcPlanStat *fresh = nullptr;  // after the layout, until the first call has read it
    int64_t *out_off = nullptr, *in_off = nullptr;
    int32_t *out = nullptr, *rev = nullptr, *slots = nullptr;
    unsigned long long *own = nullptr;
    int32_t *light = nullptr, *heavy = nullptr;  // vertices by out-neighbours (counting)
    int64_t nlight = 0, nheavy = 0;
    int32_t *mid = nullptr, *wide = nullptr;     // vertices by in-list (gather)
    int64_t nmid = 0, nwide = 0;
    int table = 0, max_out = 0;
    unsigned long long probes = 0;
    Arena mem;
};

namespace gp {

void release_tc_work(gp_graph *g, cudaStream_t s) {
    if (!g->tc) return;
    g->tc->mem.release(s);
    delete g->tc;
    g->tc = nullptr;
}

size_t tc_work_bytes(const gp_graph *g) { return g->tc ? g->tc->mem.total : 0; }

// The directed lists; general = true where the listing has to be run instead.
static int build_tc(gp_graph *g, gp_tc_work &w, cudaStream_t s) {
    if (w.ready) return GP_OK;
    const int64_t n = g->n;
    Arena tmp;
    TcPlanStat *st = nullptr, hs;
    memset(&hs, 0, sizeof(hs));
    int32_t *in = nullptr;
    unsigned long long *at = nullptr;
    const int wb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 7) / 8, (int64_t)g->num_sms * 8));
    // (few allocations: a dozen of them were a third of a small graph's first call)
    int64_t *offs = nullptr;
    int r = w.mem.alloc(offs, 2 * ((size_t)n + 1) + sizeof(TcPlanStat) / sizeof(int64_t), s);
    if (r == GP_OK) {
        w.out_off = offs;
        w.in_off = offs + n + 1;
        st = (TcPlanStat *)(offs + 2 * (n + 1));
    }
    if (r == GP_OK) {
        cudaError_t e = cudaMemsetAsync(st, 0, sizeof(*st), s);
        if (e == cudaSuccess) {
            GP_LAUNCH("tc_count", s, (k_tc_count<<<wb, 256, 0, s>>>(n, g->csr_off, g->csr_idx, w.out_off, w.in_off, st)));
            e = read_mapped(&hs, st, sizeof(hs), s);
        }
        if (e != cudaSuccess) r = set_error(GP_ERR_CUDA, "triangle lists: %s", cudaGetErrorString(e));
    }
    w.probes = hs.probes;
    w.general = hs.general || hs.max_out > (unsigned long long)TC_MAX_OUT || hs.out != hs.in;
    if (r == GP_OK && !w.general) {
        w.nlight = (int64_t)hs.light;
        w.nheavy = (int64_t)hs.heavy;
        w.nmid = (int64_t)hs.mid;
        w.nwide = (int64_t)hs.wide;
        r = exclusive_scan(w.out_off, w.out_off, n, tmp, s);
        if (r == GP_OK) r = exclusive_scan(w.in_off, w.in_off, n, tmp, s);
        const size_t edges = (size_t)hs.out, kinds = (size_t)(hs.light + hs.heavy + hs.mid + hs.wide);
        unsigned long long *wide = nullptr;  // own, the counters of the kinds, then the 32-bit arrays
        if (r == GP_OK) r = w.mem.alloc(wide, (size_t)n + 4 + (3 * edges + kinds) / 2 + 1, s);
        if (r == GP_OK) r = tmp.alloc(in, (size_t)hs.in, s);
        if (r == GP_OK) {
            w.own = wide;
            at = wide + n;
            w.slots = (int32_t *)(wide + n + 4);
            w.out = w.slots + edges;
            w.rev = w.out + edges;
            w.light = w.rev + edges;
            w.heavy = w.light + hs.light;
            w.mid = w.heavy + hs.heavy;
            w.wide = w.mid + hs.mid;
            // entries that no list writes (vertices of fewer than two out-neighbours) stay zero
            cudaError_t e = cudaMemsetAsync(wide, 0, ((size_t)n + 4) * sizeof(*wide) + edges * sizeof(int32_t), s);
            if (e == cudaSuccess) {
                const int vb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)g->num_sms * 8));
                GP_LAUNCH("tc_kinds", s, (k_tc_kinds<<<vb, 256, 0, s>>>(n, w.out_off, w.in_off, w.light, w.heavy, w.mid, w.wide, at)));
                GP_LAUNCH("tc_lists", s, (k_tc_lists<<<wb, 256, 0, s>>>(n, g->csr_off, g->csr_idx, w.out_off, w.in_off, w.out, in)));
                GP_LAUNCH("tc_reverse", s, (k_tc_reverse<<<wb, 256, 0, s>>>(n, w.out_off, w.in_off, w.out, in, w.rev, st)));
                e = cudaGetLastError();
            }
            if (e != cudaSuccess) r = set_error(GP_ERR_CUDA, "triangle lists: %s", cudaGetErrorString(e));
        }
        w.fresh = st;  // whether every edge has its reverse is read with the first counts
        w.max_out = (int)hs.max_out;
        w.table = 4 * TC_WARP_OUT;
        while (w.table < 2 * TC_MAX_OUT && w.table < 4 * (int64_t)hs.max_out) w.table *= 2;
    }
    tmp.release(s);
    w.ready = r == GP_OK;
    if (r == GP_ERR_OOM) {  // no room for the lists: the listing needs none, and the next call tries again
        clear_error();
        r = GP_OK;
        w.general = true;
    }
    if (w.general || r != GP_OK) w.mem.release(s);
    return r;
}

// Counts by the directed lists into tc, the number of triangles into scal[0].
static int run_tc(gp_graph *g, const gp_tc_work &w, bool push, unsigned long long *tc, unsigned long long *scal,
                  cudaStream_t s) {
    TcRun R;
    memset(&R, 0, sizeof(R));
    R.out_off = w.out_off;
    R.in_off = w.in_off;
    R.out = w.out;
    R.rev = w.rev;
    R.table = w.table;
    R.push = push;
    R.slots = w.slots;
    R.own = w.own;
    R.tc = tc;
    R.total = scal;
    if (w.nheavy > 0) {
        const bool bits = g->n <= TC_BITS_MAX;
        const size_t words = (size_t)((g->n + 31) >> 5);
        const size_t smem = bits ? words * (sizeof(uint32_t) + sizeof(uint16_t)) + (size_t)w.max_out * sizeof(int32_t) + 4
                                 : (size_t)w.table * (2 * sizeof(int32_t) + TC_FILTER / 8);
        const void *kernel = bits ? (const void *)k_tc_bits : (const void *)k_tc_block;
        const int threads = (bits ? TC_BITS_WARPS : TC_WARPS) * 32;
        int per_sm = 0;
        GP_TRY(allow_smem(kernel));
        GP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
        R.list = w.heavy;
        R.count = w.nheavy;
        R.ticket = scal + 1;
        const int b = (int)std::max<int64_t>(1, std::min<int64_t>(w.nheavy, (int64_t)std::max(per_sm, 1) * g->num_sms));
        if (bits) {
            R.table = w.max_out;
            GP_LAUNCH("tc_bits", s, (k_tc_bits<<<b, threads, smem, s>>>(R, g->n)));
        } else {
            GP_LAUNCH("tc_block", s, (k_tc_block<<<b, threads, smem, s>>>(R)));
        }
        GP_TRY(check_launch("tc_block"));
    }
    if (w.nlight > 0) {
        R.list = w.light;
        R.count = w.nlight;
        R.ticket = scal + 2;
        const int b = (int)std::max<int64_t>(1, std::min<int64_t>((w.nlight + 4 * TC_WARPS - 1) / (4 * TC_WARPS), (int64_t)g->num_sms * 8));
        GP_LAUNCH("tc_warp", s, (k_tc_warp<<<b, TC_WARPS * 32, 0, s>>>(R)));
        GP_TRY(check_launch("tc_warp"));
    }
    if (!push) {
        const int b = (int)std::max<int64_t>(1, std::min<int64_t>(std::max((g->n + 255) / 256, w.nwide), (int64_t)g->num_sms * 8));
        GP_LAUNCH("tc_gather", s, (k_tc_gather<<<b, 256, 0, s>>>(g->n, w.in_off, w.slots, w.own, w.mid, w.nmid, w.wide,
                                                               w.nwide, tc)));
        GP_TRY(check_launch("tc_gather"));
    }
    return GP_OK;
}

}  // namespace gp

extern "C" int gp_triangles(const gp_graph *gc, int mode, int64_t *tc_out, int64_t *total_out, gp_tc_stats *stats,
                            void *stream) {
    clear_error();
    if (!gc) return set_error(GP_ERR_INVALID, "gp_triangles: graph is NULL");
    gp_graph *g = const_cast<gp_graph *>(gc);
    if (mode != GP_PUSH && mode != GP_PULL && mode != GP_AUTO) return set_error(GP_ERR_INVALID, "gp_triangles: bad mode %d", mode);
    if (!g->symmetric) return set_error(GP_ERR_INVALID, "gp_triangles: the graph must be undirected (uploaded as symmetric)");
    if (!tc_out && !total_out) return set_error(GP_ERR_INVALID, "gp_triangles: no output");
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t n = g->n;
    if (stats) memset(stats, 0, sizeof(*stats));
    const bool push = mode == GP_PUSH;
    if (!g->tc) g->tc = new gp_tc_work();
    gp_tc_work &w = *g->tc;
    if (n > 0) GP_TRY(build_tc(g, w, s));
    const bool lists = n > 0 && !w.general;
    Arena tmp;
    unsigned long long *tc = nullptr, *cp = nullptr, *scal = nullptr;
    const bool dev_out = tc_out && is_device_ptr(tc_out);
    if (dev_out) {
        tc = (unsigned long long *)tc_out;
    } else {
        GP_TRY(tmp.alloc(tc, (size_t)std::max<int64_t>(n, 1), s));
    }
    int st = tmp.alloc(scal, 3, s);  // [0] total, [1] probes; by the lists: [0] triangles, [1], [2] tickets
    if (st == GP_OK && !push && !lists) st = tmp.alloc(cp, (size_t)std::max<int64_t>(g->push_bins.nchunks, 1), s);
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (st == GP_OK && stats) {
        cudaEventCreate(&ev0);
        cudaEventCreate(&ev1);
        cudaEventRecord(ev0, s);
    }
    unsigned long long host[2] = {0, 0};
    TcPlanStat plan;
    memset(&plan, 0, sizeof(plan));
    cudaError_t e = cudaSuccess;
    if (st == GP_OK) {
        e = cudaMemsetAsync(scal, 0, 3 * sizeof(unsigned long long), s);
        if (e == cudaSuccess && push && n > 0) e = cudaMemsetAsync(tc, 0, (size_t)n * sizeof(unsigned long long), s);
    }
    if (st == GP_OK && e == cudaSuccess && lists) st = run_tc(g, w, push, tc, scal, s);
    if (st == GP_OK && e == cudaSuccess && n > 0 && !lists) {
        TcArgs a;
        memset(&a, 0, sizeof(a));
        a.n = n;
        a.off = g->csr_off;
        a.idx = g->csr_idx;
        a.rank = g->push_bins.rank;
        a.cstart = g->push_bins.cstart;
        a.chunks = g->push_bins.chunks;
        a.big = g->push_bins.big;
        a.nchunks = g->push_bins.nchunks;
        a.nbig = g->push_bins.nbig;
        a.push = push;
        a.tc = tc;
        a.chunk_part = cp;
        a.probes = scal + 1;
        const int grid = grid_blocks(g, 256);
        GP_LAUNCH("tc", s, (k_tc<<<grid, 256, 0, s>>>(a)));
        e = cudaGetLastError();
        if (e == cudaSuccess && !push && a.nbig > 0) {
            const int gb = (int)std::max<int64_t>(1, std::min<int64_t>((a.nbig + 255) / 256, grid));
            GP_LAUNCH("tc_combine", s, (k_tc_combine<<<gb, 256, 0, s>>>(a)));
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) {
            const int gf = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, grid));
            GP_LAUNCH("tc_finish", s, (k_tc_finish<<<gf, 256, 0, s>>>(n, push, tc, scal)));
            e = cudaGetLastError();
        }
    }
    if (st == GP_OK && e == cudaSuccess && tc_out && !dev_out && n > 0)
        e = cudaMemcpyAsync(tc_out, tc, (size_t)n * sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    if (st == GP_OK && e == cudaSuccess) e = cudaMemcpyAsync(host, scal, sizeof(host), cudaMemcpyDeviceToHost, s);
    const bool fresh = lists && w.fresh;
    if (st == GP_OK && e == cudaSuccess && fresh) e = cudaMemcpyAsync(&plan, w.fresh, sizeof(plan), cudaMemcpyDeviceToHost, s);
    if (st == GP_OK && e == cudaSuccess && stats) e = cudaEventRecord(ev1, s);
    if (st == GP_OK && e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (st == GP_OK && e == cudaSuccess && fresh) {
        w.fresh = nullptr;
        if (plan.general) {  // an edge without its reverse: the listing's counts instead
            w.general = true;
            w.mem.release(s);
            tmp.release(s);
            if (ev0) cudaEventDestroy(ev0);
            if (ev1) cudaEventDestroy(ev1);
            return gp_triangles(gc, mode, tc_out, total_out, stats, stream);
        }
    }
    if (lists) {
        host[0] *= 3;  // as the sum of the counts
        host[1] = w.probes;
    }
    if (stats && ev0) {
        float ms = 0.f;
        if (e == cudaSuccess) cudaEventElapsedTime(&ms, ev0, ev1);
        cudaEventDestroy(ev0);
        cudaEventDestroy(ev1);
        stats->ms = ms;
        stats->probes = (int64_t)host[1];
        stats->triangles = (int64_t)(host[0] / 3);
        stats->mode_used = push ? GP_PUSH : GP_PULL;
    }
    tmp.release(s);
    if (st != GP_OK) return st;
    if (e != cudaSuccess) return set_error(GP_ERR_CUDA, "gp_triangles: %s", cudaGetErrorString(e));
    if (total_out) *total_out = (int64_t)(host[0] / 3);
    return GP_OK;
}
