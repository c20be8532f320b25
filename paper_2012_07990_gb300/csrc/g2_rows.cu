// g2_rows.cu — multi-source SSSP over distance rows: the tuned batch on
// graphs that are not of bounded degree.
//
// The distances of a vertex from all sources lie in one row of K = 8, 16 or
// 32 values (the smallest that holds the batch), so that a relaxation of one
// arc for every source is one coalesced access, a lane per source, where
// stacked arrays of n take a scattered access per (arc, source).  Rounds relax
// the arcs of every vertex whose row changed in the round before until none
// does (distances only fall and every change is flagged, so the result is the
// shortest distance whatever the order).  On power-law graphs the frontiers
// of a batch cover most vertices for a few rounds, and there the union of the
// sources' delta-stepping buckets visits each arc many times for a few
// sources each: counted on RMAT-18 with 32 sources, buckets of 64 visit
// every arc 17.0 times (3.9 sources a visit), rounds without buckets 5.5
// times (16.2 sources a visit).  So the near/far threshold is not used here.
//
// A round with at least 1/32 of the vertices flagged sweeps all arcs in order,
// 32 to a warp at a time (a hub's arcs spread over the grid; larger shares
// left some CTAs with the hubs: 256 arcs a share 10.2 ms for the whole call,
// 128 arcs 9.7, 32 arcs 8.3), tests the source's flag in a bitmap that stays
// in L1, and relaxes kRowFlight arcs at once.  A round with fewer takes the
// flagged vertices as a list, their arcs divided evenly by a prefix sum.
//
// Bound: the row reads through L1 (57% of its peak, a quarter of the sectors
// hit; issue 48%, L2 26%, DRAM 13%; 36 warps per SM with 8 rows each in flight).
// RMAT-21, 32 sources, weights 1-255: a sweep with every vertex flagged 1.4 ms,
// the whole call 8.1-8.4 ms, against 40-43 ms for STRICT delta-stepping over
// stacked arrays when the rows replaced it (33.8 ms since).  Measured
// and rejected: the arcs held a lane each and handed out by shuffles (36
// instructions an arc, 2.5 ms a sweep), fewer registers for more warps (6 CTAs
// per SM 13.0 ms, 8 CTAs 19.7 ms: spills).
#include <cuda_runtime.h>

#include <algorithm>

#include "g2_host.h"
#include "g2_lb.cuh"

namespace g2 {

constexpr int kRowTile = 128;   // arcs of a list that a warp takes at a time
constexpr int kRowFlight = 8;   // rows in flight per lane
// Rounds without buckets repeat work where paths are long (a road network with
// a hub): power-law graphs take 12-15 rounds.  A batch that has not ended after
// this many goes on with the near/far queue, from the distances found so far
// and the vertices that are flagged.  It does so after kRowLook rounds already
// if the frontier has not begun to fall by then: power-law and random graphs of
// 2^10 to 2^21 vertices are below half of their largest frontier there, with 1
// to 32 sources and weights to 20,000; a band of the same degree (60 hops
// across) is at 0.82 to 1.0 of it.  On that band 1 / 5 / 32 sources
// take 3.5 / 7.5 / 12.4 ms so, 3.5 / 8.4 / 12.7 without the look.
constexpr int kRowRounds = 32, kRowLook = 16;

__global__ void k_rows_fill(int32_t *D, int64_t count4) {
    const int4 inf = make_int4(G2_INF32, G2_INF32, G2_INF32, G2_INF32);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count4;
         i += (int64_t)gridDim.x * blockDim.x)
        reinterpret_cast<int4 *>(D)[i] = inf;
}

__global__ void k_rows_seed(const int32_t *srcs, int32_t k, int32_t K, int32_t *D,
                            uint32_t *flags) {
    const int i = threadIdx.x;
    if (i < k) {
        const int32_t s = srcs[i];
        D[(int64_t)s * K + i] = 0;
        atomicOr(&flags[s >> 5], 1u << (s & 31));
    }
}

// The flagged vertices to list (the first cap of them) and their number to
// *cnt; `clear` zeroed for the next round's flags.
__global__ void k_rows_list(const uint32_t *flags, int32_t words, uint32_t *clear, int32_t *list,
                            int32_t cap, int32_t *cnt) {
    const int lane = threadIdx.x & 31;
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; base < words;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + lane;
        uint32_t x = 0;
        if (i < words) {
            x = flags[i];
            clear[i] = 0;
        }
        const int c = __popc(x);
        const int incl = warp_incl_scan(c);
        const int tot = __shfl_sync(G2_FULL, incl, 31);
        if (tot == 0) continue;
        int b = 0;
        if (lane == 31) b = atomicAdd(cnt, tot);
        int pos = __shfl_sync(G2_FULL, b, 31) + incl - c;
        while (x && pos < cap) {
            list[pos++] = (int32_t)(i * 32 + __ffs(x) - 1);
            x &= x - 1;
        }
    }
}

__global__ void k_rows_degrees(const int32_t *rowptr, const int32_t *list, int32_t size,
                               int32_t *deg) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < size;
         i += (int64_t)gridDim.x * blockDim.x)
        deg[i] = rowptr[list[i] + 1] - rowptr[list[i]];
}

// The lanes of a group of K hold one vertex, a lane per source; control flow
// is uniform within a group.  Sums are unsigned: INT32_MAX + w does not wrap
// and is never less than a distance.

// Where nd < old in any lane: lower v's row and flag v.
__device__ __forceinline__ void rows_lower(int32_t *Dl, int K, uint32_t *next, int32_t v,
                                           unsigned nd, unsigned old, unsigned group, int sl) {
    const bool fell = nd < old;
    if (fell) atomicMin(Dl + (int64_t)v * K, (int32_t)nd);
    if (__any_sync(group, fell) && sl == 0) atomicOr(&next[v >> 5], 1u << (v & 31));
}

// The kRowFlight arcs u -> v[t] of one vertex whose row is du.  The rows of
// all are loaded before any is looked at; most fall in no lane, which one
// vote finds for all of them.
template <int K>
__device__ __forceinline__ void rows_same_source(int32_t *Dl, uint32_t *next, unsigned du,
                                                 const int32_t (&v)[kRowFlight],
                                                 const int32_t (&w)[kRowFlight], unsigned group,
                                                 int sl) {
    unsigned old[kRowFlight];
#pragma unroll
    for (int t = 0; t < kRowFlight; ++t) old[t] = (unsigned)Dl[(int64_t)v[t] * K];
    bool any = false;
#pragma unroll
    for (int t = 0; t < kRowFlight; ++t) any |= du + (unsigned)w[t] < old[t];
    if (!__any_sync(group, any)) return;
#pragma unroll
    for (int t = 0; t < kRowFlight; ++t)
        rows_lower(Dl, K, next, v[t], du + (unsigned)w[t], old[t], group, sl);
}

// One round over every arc row[e] -> col[e] whose source is flagged.  A group
// takes kRowFlight consecutive arcs at a time; the ids and weights are read
// with 16-byte loads at the same address in every lane of the group, so that
// an arc costs no shuffle.  (With the arcs held a lane each and handed out by
// shuffles the sweep was bound by its 36 instructions an arc: 2.5 ms on
// RMAT-21 with every vertex flagged, 70% of the issue slots.)
template <int K>
__global__ void __launch_bounds__(kCta) k_rows_sweep(const int32_t *__restrict__ row,
                                                     const int32_t *__restrict__ col,
                                                     const int32_t *__restrict__ w, int32_t m,
                                                     int32_t *D, const uint32_t *__restrict__ cur,
                                                     uint32_t *next, unsigned long long *ctr) {
    constexpr int F = kRowFlight, G = 32 / K;
    static_assert(F == 8, "two 16-byte loads");
    const int lane = threadIdx.x & 31, sl = lane % K, gi = lane / K;
    const unsigned group = K == 32 ? G2_FULL : ((1u << K % 32) - 1u) << (gi * K);
    int32_t *Dl = D + sl;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int32_t us = -1;  // the vertex whose row is in du
    unsigned du = 0;
    int32_t nu = gw * 32 + lane < m ? row[gw * 32 + lane] : -1;  // a step ahead
    for (int64_t c0 = gw * 32; c0 < m; c0 += nw * 32) {
        const int32_t ul = nu;
        const int64_t e1 = c0 + nw * 32 + lane;
        nu = e1 < m ? row[e1] : -1;
        const unsigned act =
            __ballot_sync(G2_FULL, ul >= 0 && ((cur[ul >> 5] >> (ul & 31)) & 1u));
        if (act == 0) continue;
        count_arcs(ctr, (act >> lane) & 1u);
#pragma unroll 1
        for (int s = gi * F; s < 32; s += G * F) {
            const unsigned on = (act >> s) & 255u;
            if (on == 0) continue;
            const int64_t e = c0 + s;
            if (on == 255u && row[e] == row[e + F - 1]) {
                const int32_t u = row[e];
                if (u != us) {
                    us = u;
                    du = (unsigned)Dl[(int64_t)u * K];
                }
                const int4 c0v = *reinterpret_cast<const int4 *>(col + e);
                const int4 c1v = *reinterpret_cast<const int4 *>(col + e + 4);
                const int4 w0v = *reinterpret_cast<const int4 *>(w + e);
                const int4 w1v = *reinterpret_cast<const int4 *>(w + e + 4);
                const int32_t v[F] = {c0v.x, c0v.y, c0v.z, c0v.w, c1v.x, c1v.y, c1v.z, c1v.w};
                const int32_t x[F] = {w0v.x, w0v.y, w0v.z, w0v.w, w1v.x, w1v.y, w1v.z, w1v.w};
                rows_same_source<K>(Dl, next, du, v, x, group, sl);
                continue;
            }
            // several sources, or some not flagged
            int32_t v[F];
            unsigned nd[F], old[F];
            bool any = false;
#pragma unroll
            for (int t = 0; t < F; ++t) {
                v[t] = 0;
                nd[t] = old[t] = 0;
                if ((on >> t) & 1u) {
                    v[t] = col[e + t];
                    nd[t] = (unsigned)Dl[(int64_t)row[e + t] * K] + (unsigned)w[e + t];
                    old[t] = (unsigned)Dl[(int64_t)v[t] * K];
                }
            }
#pragma unroll
            for (int t = 0; t < F; ++t) any |= nd[t] < old[t];
            if (!__any_sync(group, any)) continue;
#pragma unroll
            for (int t = 0; t < F; ++t)
                rows_lower(Dl, K, next, v[t], nd[t], old[t], group, sl);
        }
        __syncwarp();
    }
}

// One round over the arcs of list[0, size): arc k of their sequence belongs to
// the entry i with scan[i] <= k < scan[i + 1].
template <int K>
__global__ void __launch_bounds__(kCta) k_rows_push(DevGraph g, const int32_t *list, int32_t size,
                                                    const int32_t *scan, int32_t *D, uint32_t *next,
                                                    unsigned long long *ctr) {
    constexpr int F = kRowFlight, G = 32 / K;
    const int lane = threadIdx.x & 31, sl = lane % K, gi = lane / K;
    const unsigned group = K == 32 ? G2_FULL : ((1u << K % 32) - 1u) << (gi * K);
    int32_t *Dl = D + sl;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int32_t total = scan[size];
    for (int64_t t0 = gw * kRowTile; t0 < total; t0 += nw * kRowTile) {
        const int32_t len = (int32_t)(total - t0 < kRowTile ? total - t0 : kRowTile);
        count_arcs(ctr, lane == 0 ? len : 0);
        const int32_t own = scan_owner(scan, size, (int32_t)t0);
        if (len == kRowTile && scan[own + 1] >= t0 + kRowTile) {
            // the whole tile belongs to one vertex
            const int32_t u = list[own];
            const int64_t e0 = g.rowptr[u] + (t0 - scan[own]);
            const unsigned du = (unsigned)Dl[(int64_t)u * K];
#pragma unroll 1
            for (int s = gi * F; s < kRowTile; s += G * F) {
                int32_t v[F], x[F];
#pragma unroll
                for (int t = 0; t < F; ++t) {
                    v[t] = g.col[e0 + s + t];
                    x[t] = g.w[e0 + s + t];
                }
                rows_same_source<K>(Dl, next, du, v, x, group, sl);
            }
            __syncwarp();
            continue;
        }
#pragma unroll 1
        for (int b = 0; b < len; b += 32) {
            const int32_t k = (int32_t)(t0 + b) + lane;
            int32_t u = -1, v = 0, wt = 0;
            if (b + lane < len) {
                // the last entry from own on with scan <= k
                int32_t lo = own, hi = own;
                for (int32_t d = 1; hi < size - 1 && scan[hi + 1] <= k; d <<= 1) {
                    lo = hi + 1;
                    hi = hi + 1 + d < size - 1 ? hi + 1 + d : size - 1;
                    if (scan[hi] > k) break;
                }
                while (lo < hi) {
                    const int32_t mid = lo + (hi - lo + 1) / 2;
                    if (scan[mid] <= k) lo = mid;
                    else hi = mid - 1;
                }
                u = list[lo];
                const int32_t e = g.rowptr[u] + (k - scan[lo]);
                v = g.col[e];
                wt = g.w[e];
            }
            const unsigned act = __ballot_sync(G2_FULL, u >= 0);
#pragma unroll 1
            for (int s = 0; s < K; s += F / 2) {
                int32_t vj[F / 2];
                unsigned nd[F / 2], old[F / 2];
#pragma unroll
                for (int t = 0; t < F / 2; ++t) {
                    const int j = gi * K + s + t;  // this group's arcs are its own lanes'
                    const int32_t uj = __shfl_sync(G2_FULL, u, j);
                    vj[t] = __shfl_sync(G2_FULL, v, j);
                    nd[t] = (unsigned)__shfl_sync(G2_FULL, wt, j);
                    old[t] = 0;
                    if ((act >> j) & 1u) {
                        nd[t] += (unsigned)Dl[(int64_t)uj * K];
                        old[t] = (unsigned)Dl[(int64_t)vj[t] * K];
                    }
                }
#pragma unroll
                for (int t = 0; t < F / 2; ++t)
                    rows_lower(Dl, K, next, vj[t], nd[t], old[t], group, sl);
            }
        }
    }
}

// rows -> dist[k][n] (a warp turns 32 vertices at a time in shared memory,
// both sides coalesced) and the largest finite distance to *dmax
template <int K>
__global__ void __launch_bounds__(kCta) k_rows_out(const int32_t *__restrict__ D, int32_t n,
                                                   int32_t k, int32_t *dist, int32_t *dmax) {
    __shared__ int32_t s_all[kWarps][32][K + 1];
    const int lane = threadIdx.x & 31;
    auto s = s_all[threadIdx.x >> 5];
    int32_t best = 0;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v0 = gw * 32; v0 < n; v0 += nw * 32) {
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const int x = i * 32 + lane;
            s[x / K][x % K] = v0 + x / K < n ? D[v0 * K + x] : G2_INF32;
        }
        __syncwarp();
        if (v0 + lane < n) {
#pragma unroll 8
            for (int i = 0; i < k; ++i) {
                const int32_t d = s[lane][i];
                dist[(int64_t)i * n + v0 + lane] = d;
                if (d != G2_INF32) best = max(best, d);
            }
        }
        __syncwarp();
    }
    best = __reduce_max_sync(G2_FULL, best);
    if (lane == 0 && best > 0) atomicMax(dmax, best);
}

// error G2_EOVERFLOW if an arc out of a reached vertex leads to INT32_MAX or beyond
__global__ void k_rows_check(const int32_t *row, const int32_t *w, int32_t m, const int32_t *dist,
                             int32_t n, int32_t k, int32_t *err) {
    for (int32_t i = 0; i < k; ++i)
        for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
             e += (int64_t)gridDim.x * blockDim.x) {
            const int32_t d = dist[(int64_t)i * n + row[e]];
            if (d != G2_INF32 && (int64_t)d + w[e] >= G2_INF32) set_error(err, G2_EOVERFLOW);
        }
}

// the largest of a[0, n) that is not `skip`
__global__ void k_max_i32(const int32_t *a, int64_t n, int32_t skip, int32_t *out) {
    int32_t best = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t x = a[i];
        if (x != skip) best = max(best, x);
    }
    best = __reduce_max_sync(G2_FULL, best);
    if ((threadIdx.x & 31) == 0 && best > 0) atomicMax(out, best);
}

// Largest arc weight (weights are >= 0), computed on the device once per graph.
static g2_status max_weight(g2_graph *g, int32_t *d_tmp, cudaStream_t st, int32_t *d_err,
                            int32_t *out) {
    Topology *t = g->topo;
    std::lock_guard<std::recursive_mutex> lk(t->layout_mu);
    if (t->max_w < 0) {
        G2_CK(cudaMemsetAsync(d_tmp, 0, 4, st));
        k_max_i32<<<grid_for(g, t->m, kCta * 4), kCta, 0, st>>>(t->w, t->m, -1, d_tmp);
        stats().launches += 1;
        G2_TRY(read_counters(g, d_tmp, 1, st, d_err));
        t->max_w = g->h_ctr[0];
    }
    *out = t->max_w;
    return G2_OK;
}

// The overflow rule on final distances, the largest finite of which is dmax.
static g2_status check_overflow(g2_graph *g, const int32_t *dist, int32_t k, int32_t dmax,
                                int32_t wmax, cudaStream_t st, int32_t *d_err) {
    Topology *t = g->topo;
    if ((int64_t)dmax + wmax < G2_INF32) return G2_OK;
    k_rows_check<<<grid_for(g, t->m, kCta), kCta, 0, st>>>(t->coo_src, t->w, t->m, dist, t->n, k, d_err);
    G2_CK(cudaGetLastError());
    stats().launches += 1;
    return G2_OK;
}

// For a batch that went on from rows: they drop a distance of INT32_MAX or
// beyond without a word, so the rule is applied to what the batch ended with.
g2_status sssp_batch_check(g2_graph *g, const int32_t *dist, int32_t k, cudaStream_t st,
                           int32_t *d_err) {
    const int64_t count = (int64_t)k * g->topo->n;
    int32_t *ctrs = d_err - 62, wmax = 0;
    G2_TRY(max_weight(g, ctrs + 1, st, d_err, &wmax));
    G2_CK(cudaMemsetAsync(ctrs + 1, 0, 4, st));
    k_max_i32<<<grid_for(g, count, kCta * 4), kCta, 0, st>>>(dist, count, G2_INF32, ctrs + 1);
    stats().launches += 1;
    G2_TRY(read_counters(g, ctrs + 1, 1, st, d_err));
    return check_overflow(g, dist, k, g->h_ctr[0], wmax, st, d_err);
}

// *left: null where the batch ended, else the flags of the vertices whose arcs
// are still to be relaxed from the distances in dist.
template <int K>
static g2_status run_rows(g2_graph *g, const int32_t *srcs, int32_t k, int32_t *dist,
                          cudaStream_t st, int32_t *d_err, const uint32_t **left) {
    Topology *t = g->topo;
    const int32_t n = t->n, m = t->m;
    const int32_t words = (n + 31) / 32, cap = std::max(n / 32, 1);
    int32_t *ctrs = d_err - 62;
    uint32_t *flags[2];
    int32_t *D, *list, *deg, *scan, *dsrc;
    G2_TRY(ws(g, B_ROWS, (size_t)n * K, &D));
    G2_TRY(ensure_coo(g, st));
    G2_TRY(ws(g, B_BM0, (size_t)words + 1, &flags[0]));
    G2_TRY(ws(g, B_BM1, (size_t)words + 1, &flags[1]));
    G2_TRY(ws(g, B_Q0, (size_t)n, &list));
    G2_TRY(ws(g, B_I1, (size_t)std::max(n, 64) + 1, &deg));
    G2_TRY(ws(g, B_SCAN, (size_t)n + 1, &scan));
    dsrc = deg;  // read by the seed kernel, before the first degrees
    G2_TRY(put_array(dsrc, srcs, k, st));
    k_rows_fill<<<grid_for(g, (int64_t)n * K / 4, kCta), kCta, 0, st>>>(D, (int64_t)n * K / 4);
    G2_CK(cudaMemsetAsync(flags[0], 0, (size_t)words * 4, st));
    k_rows_seed<<<1, 32, 0, st>>>(dsrc, k, K, D, flags[0]);
    stats().launches += 2;
    const int sweep = grid_for(g, m, kCta);
    unsigned long long *ctr = nullptr;
    if (count_arcs_enabled()) G2_TRY(ws(g, B_ARCS, 2, &ctr));
    int p = 0;
    int32_t peak = 0;  // the largest frontier so far
    for (;; p ^= 1) {
        // (all counters are zero at the start of the call)
        if (stats().iterations) G2_CK(cudaMemsetAsync(ctrs, 0, 4, st));
        k_rows_list<<<grid_for(g, words, kCta), kCta, 0, st>>>(flags[p], words, flags[p ^ 1], list,
                                                             cap, ctrs);
        stats().launches += 1;
        G2_TRY(read_counters(g, ctrs, 1, st, d_err));
        const int32_t size = g->h_ctr[0];
        if (size == 0) break;
        peak = std::max(peak, size);
        if (stats().iterations == kRowRounds ||
            (stats().iterations == kRowLook && size > peak / 4 * 3)) {
            *left = flags[p];
            break;
        }
        // the line: a sweep reads the source id of every arc (RMAT-21: 0.36 ms
        // with 8% of the vertices flagged), a list of fewer than 1/32 of the
        // vertices takes 0.05 ms, 0.25 ms where it holds the hubs
        if (size <= cap && size < n / 32) {
            k_rows_degrees<<<grid_for(g, size, kCta), kCta, 0, st>>>(t->rowptr, list, size, deg);
            G2_TRY(exclusive_scan_i32(g, deg, scan, size, st));
            k_rows_push<K><<<t->sm_count * 8, kCta, 0, st>>>(t->view(), list, size, scan, D,
                                                           flags[p ^ 1], ctr);
            stats().launches += 2;
        } else {
            k_rows_sweep<K><<<sweep, kCta, 0, st>>>(t->coo_src, t->col, t->w, m, D, flags[p],
                                                 flags[p ^ 1], ctr);
            stats().launches += 1;
        }
        stats().push_rounds++;
        stats().iterations++;
    }
    int32_t wmax = 0;
    if (!*left) G2_TRY(max_weight(g, ctrs + 1, st, d_err, &wmax));
    G2_CK(cudaMemsetAsync(ctrs + 1, 0, 4, st));
    k_rows_out<K><<<grid_for(g, n, kCta), kCta, 0, st>>>(D, n, k, dist, ctrs + 1);
    stats().launches += 1;
    G2_TRY(read_counters(g, ctrs + 1, 1, st, d_err));
    return *left ? G2_OK : check_overflow(g, dist, k, g->h_ctr[0], wmax, st, d_err);
}

// Shortest distances of k sources over rows.  *how says what is left to do:
// nothing (ROWS_DONE); everything, where the form does not apply (ROWS_NONE: no
// arcs, or no memory for the rows, the arcs' source ids or the lists beside
// what the device already holds); or the rest, after kRowRounds rounds
// (ROWS_LEFT: dist holds distances, and the arcs of the vertices flagged in
// *left are still to be relaxed).  The rows' memory is given back unless the
// batch is done: what runs next needs its own.
g2_status sssp_batch_rows(g2_graph *g, const int32_t *srcs, int32_t k, int32_t *dist,
                          cudaStream_t st, int32_t *d_err, int *how, const uint32_t **left) {
    *how = ROWS_NONE;
    *left = nullptr;
    if (g->topo->m == 0) return G2_OK;
    const g2_status r = k <= 8    ? run_rows<8>(g, srcs, k, dist, st, d_err, left)
                        : k <= 16 ? run_rows<16>(g, srcs, k, dist, st, d_err, left)
                                  : run_rows<32>(g, srcs, k, dist, st, d_err, left);
    if (r == G2_OK && !*left) {
        *how = ROWS_DONE;
        return G2_OK;
    }
    if (r != G2_OK && r != G2_ENOMEM) return r;
    ws_release(g, B_ROWS);
    G2_CK(cudaMemsetAsync(d_err - 62, 0, 8, st));  // the counters that run_rows used
    if (r == G2_OK) {
        *how = ROWS_LEFT;
    } else {
        *left = nullptr;
        stats().iterations = stats().push_rounds = 0;
    }
    return G2_OK;
}

}  // namespace g2
