// g2_bc.cu — betweenness centrality (Sec. VII; Brandes, "A faster algorithm
// for betweenness centrality", 2001) summed over a list of sources.
//
// Per source: a level-synchronous BFS whose levels are appended to one list,
// path counts sigma for each new level (pull over in-neighbours one level up),
// then dependencies delta level by level from the deepest (pull over
// out-neighbours one level down), bc[v] += delta[v] for v != source.
//
// Path counts grow like binomials on grids (C(2k, k) after 2k levels) and two
// vertices of one level can differ by more than the fp64 range, so sigma is an
// extended-range number: a 64-bit integer mantissa and an int32 exponent per
// vertex.  The dependency sum delta_v = sum_w sigma_v / sigma_w (1 + delta_w)
// is formed as sigma_v * sum_w C_w with C_w = (1 + delta_w) / sigma_w kept per
// vertex in the same form, so both passes add integers per arc: GB300's fp64
// units take 16 cycles for a warp's add (delta's pass over RMAT-21: 618 us a
// source with an fp64 scaling and add per arc and the fp64 finish in one lane
// of a warp, 583 us so, before the rest below).  fp64 is left to one finish
// per vertex, 32 vertices at a time.
//
// A vertex's mantissa, exponent and level lie in one 16-byte record, so that a
// neighbour costs one aligned load (one 32-byte sector) whether it counts or
// not.  The backward pass replaces sigma by C.
//
// Schedules: each level's discovery is one edgeset.apply round (PUSH or PULL
// per the hybrid schedule; the tuned schedule finds all depths of a source in
// one launch of the fused hybrid when there are several sources), then the
// reached vertices are grouped by level and degree, and sigma and delta are
// pulled level by level over the groups: a thread, eight lanes, a warp or a
// CTA per piece of a vertex by its degree (on a symmetric bounded-degree graph a
// thread per vertex over the levels as found).  With kernel fusion the whole
// source runs in one persistent cooperative kernel with one grid barrier per
// level and pass; there the pulls give a thread to the vertices below
// kThreadDeg arcs, a warp to those below kBigDeg and a whole CTA to the rest,
// or a thread to every vertex on a symmetric bounded-degree graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "g2_cluster.cuh"
#include "g2_host.h"
#include "g2_lb.cuh"

namespace g2 {

g2_status bfs_fused_do(g2_graph *g, int32_t src, int32_t *depth, int32_t *parent,
                       const g2_hybrid &h, bool by_arcs, cudaStream_t st, int32_t *d_err);

constexpr int32_t kBigDeg = 4096;    // a CTA per vertex from this many arcs
constexpr int32_t kThreadDeg = 32;   // a thread per vertex below this many arcs

// Extended-range path count: an integer mantissa m, 0 or in [2^62, 2^63),
// and an exponent e; the value is m * 2^(e - 63).  Sums take integer shifts
// and adds only (no fp64 on the per-arc path; fp64 is slow on this GPU), with
// 63 mantissa bits.
struct BigF {
    unsigned long long m;
    int e;
};

// m * 2^-63 in [0.5, 1) as fp64 (once per vertex)
__device__ __forceinline__ double bf_mant(unsigned long long m) {
    return (double)m * 0x1p-63;
}

// The value x * 2^e (x > 0 normal) as an extended-range number.
__device__ __forceinline__ BigF bf_from(double x, int e) {
    const long long b = __double_as_longlong(x);
    const int ex = (int)(b >> 52) - 1023;
    const unsigned long long f = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
    return BigF{f << 10, ex + 1 + e};
}

// a * 2^k as fp64; 0 below 2^-1022 (below the rounding of what it is added to)
__device__ __forceinline__ double bf_value(BigF a, int k) {
    const int e = a.e + k;
    if (a.m == 0 || e < -1021) return 0.0;
    return bf_mant(a.m) * __hiloint2double((e + 1023) << 20, 0);
}

// a + b: the smaller mantissa shifted to the larger one's exponent (the
// bits shifted out are dropped: below 2^-62 of the sum), the sum brought back
// under 2^63.
__device__ __forceinline__ BigF bf_add(BigF a, BigF b) {
    if (a.m == 0) return b;
    if (b.m == 0) return a;
    if (a.e < b.e) {
        BigF t = a;
        a = b;
        b = t;
    }
    const int d = a.e - b.e;
    unsigned long long sum = d > 63 ? a.m : a.m + (b.m >> d);
    int e = a.e;
    if (sum >> 63) {
        sum >>= 1;
        ++e;
    }
    return BigF{sum, e};
}

__device__ __forceinline__ BigF bf_shfl_xor(BigF a, int d) {
    return BigF{__shfl_xor_sync(G2_FULL, a.m, d), __shfl_xor_sync(G2_FULL, a.e, d)};
}

// What the pulls need of a vertex.
struct __align__(16) BcRec {
    unsigned long long m;  // sigma (BigF); C once delta is known
    int e;
    int d;                 // level, -1 before sigma is known
};

struct BcState {
    DevGraph g;
    int32_t *depth;
    BcRec *rec;
    double *bc;
    int32_t *lvl;  // all levels, in order
    int32_t src;
    // granularity: one thread per vertex on a symmetric bounded-degree graph
    // (every list short), else by degree (fused kernels: threads, warps and,
    // when some vertex may have kBigDeg or more arcs (`big`), CTAs for those)
    int32_t per_thread;
    int32_t big;
};

// One 16-byte load, written out: left to the compiler it became two of 8
// bytes, and the pulls are bound by the L1 tag look-ups of their loads.
__device__ __forceinline__ BcRec bc_load(const BcState &s, int32_t v) {
    unsigned m0, m1;
    BcRec r;
    asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(m0), "=r"(m1), "=r"(r.e), "=r"(r.d)
                 : "l"(s.rec + v)
                 : "memory");
    r.m = (unsigned long long)m0 | (unsigned long long)m1 << 32;
    return r;
}

__device__ __forceinline__ void bc_store(const BcState &s, int32_t v, BigF a, int32_t d) {
    *reinterpret_cast<int4 *>(s.rec + v) =
        make_int4((int)(unsigned)a.m, (int)(unsigned)(a.m >> 32), a.e, d);
}

// A thread's part of a vertex's sum: every step-th arc of list[b, e) from
// b + off, N records in flight, those of level `want` added in arc order.
// sigma: the in-neighbours one level up; delta: the out-neighbours one level
// down.
template <int N>
__device__ __forceinline__ BigF bc_part(const BcState &s, const int32_t *list, int32_t want, int32_t b,
                                        int32_t e, int step, int off) {
    BigF acc{0, 0};
    for (int64_t k0 = (int64_t)b + off; k0 < e; k0 += (int64_t)N * step) {
        int32_t u[N];
        BcRec r[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int64_t x = k0 + (int64_t)j * step;
            u[j] = x < e ? list[x] : -1;
        }
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (u[j] >= 0) r[j] = bc_load(s, u[j]);
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (u[j] >= 0 && r[j].d == want) acc = bf_add(acc, BigF{r[j].m, r[j].e});
    }
    return acc;
}

// sigma_v, v at level d
__device__ __forceinline__ void bc_finish_sigma(const BcState &s, int32_t v, BigF a, int32_t d) {
    bc_store(s, v, a, d);
}

// delta_v from the sum of its successors' C: added to bc (but for the source)
// and kept as the C that the level above uses
__device__ __forceinline__ void bc_finish_delta(const BcState &s, int32_t v, BigF sum) {
    const BcRec r = bc_load(s, v);
    const double m = bf_mant(r.m), dl = m * bf_value(sum, r.e);
    if (v != s.src) s.bc[v] += dl;
    bc_store(s, v, bf_from((1.0 + dl) / m, -r.e), r.d);
}

template <bool SIGMA>
__device__ __forceinline__ void bc_finish(const BcState &s, int32_t v, BigF a, int32_t d) {
    if (SIGMA) bc_finish_sigma(s, v, a, d + 1);
    else bc_finish_delta(s, v, a);
}

// The sums for one thread over a whole (short) list.
__device__ __forceinline__ BigF bc_sigma_thread(const BcState &s, int32_t w, int32_t d) {
    return bc_part<4>(s, s.g.ccol, d, s.g.crowptr[w], s.g.crowptr[w + 1], 1, 0);
}

__device__ __forceinline__ BigF bc_delta_thread(const BcState &s, int32_t v, int32_t d) {
    return bc_part<4>(s, s.g.col, d + 1, s.g.rowptr[v], s.g.rowptr[v + 1], 1, 0);
}

// Sum of a group's parts (the lanes of a group of G, G a power of two).
template <int G>
__device__ __forceinline__ BigF bc_group_sum(BigF a) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) a = bf_add(a, bf_shfl_xor(a, o));
    return a;
}

// The sum of the CTA's parts, in thread 0.
__device__ __forceinline__ BigF bc_cta_sum(BigF a) {
    __shared__ unsigned long long s_m[kWarps];
    __shared__ int s_e[kWarps];
    a = bc_group_sum<32>(a);
    if ((threadIdx.x & 31) == 0) {
        s_m[threadIdx.x >> 5] = a.m;
        s_e[threadIdx.x >> 5] = a.e;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int k = 1; k < kWarps; ++k) a = bf_add(a, BigF{s_m[k], s_e[k]});
    __syncthreads();
    return a;
}

// The whole CTA on vertex v.
template <bool SIGMA>
__device__ void bc_cta_vertex(const BcState &s, int32_t v, int32_t d) {
    const int32_t *rp = SIGMA ? s.g.crowptr : s.g.rowptr;
    const BigF a = bc_cta_sum(bc_part<4>(s, SIGMA ? s.g.ccol : s.g.col, SIGMA ? d : d + 1, rp[v],
                                         rp[v + 1], kCta, (int)threadIdx.x));
    if (threadIdx.x == 0) bc_finish<SIGMA>(s, v, a, d);
}

// Groups of G lanes, a vertex each, over list[0, cnt) (PICK: those with
// lo <= degree < hi only).  The sums of delta's pass wait in shared memory
// until 32 can be finished at once (its fp64 takes a warp's time however few
// lanes it has).
template <bool SIGMA, int G, int N, bool PICK>
__device__ __forceinline__ void bc_groups(const BcState &s, const int32_t *list, int32_t cnt,
                                          int32_t d, int32_t lo, int32_t hi, int bid, int nb) {
    constexpr bool kWait = !SIGMA && G > 1;
    __shared__ int32_t s_v[kWait ? kWarps : 1][32];
    __shared__ int s_e[kWait ? kWarps : 1][32];
    __shared__ unsigned long long s_m[kWait ? kWarps : 1][32];
    const int32_t *rp = SIGMA ? s.g.crowptr : s.g.rowptr;
    const int32_t *arcs = SIGMA ? s.g.ccol : s.g.col;
    const int lane = threadIdx.x & 31, sub = lane % G, wid = kWait ? threadIdx.x >> 5 : 0;
    const int64_t gw = (int64_t)bid * kWarps + (threadIdx.x >> 5), nw = (int64_t)nb * kWarps;
    int waiting = 0;
    auto flush = [&]() {
        __syncwarp();
        if (lane < waiting) bc_finish<SIGMA>(s, s_v[wid][lane], BigF{s_m[wid][lane], s_e[wid][lane]}, d);
        __syncwarp();
        waiting = 0;
    };
    for (int64_t base = gw * (32 / G); base < cnt; base += nw * (32 / G)) {
        const int64_t i = base + lane / G;
        int32_t v = 0, b = 0, e = 0;
        bool on = i < cnt;
        if (on) {
            v = list[i];
            b = rp[v];
            e = rp[v + 1];
            if (PICK) on = e - b >= lo && e - b < hi;
        }
        if (!on) b = e = 0;
        BigF a = bc_part<N>(s, arcs, SIGMA ? d : d + 1, b, e, G, sub);
        if (G > 1) __syncwarp();
        a = bc_group_sum<G>(a);
        const bool lead = on && sub == 0;
        if (!kWait) {
            if (lead) bc_finish<SIGMA>(s, v, a, d);
        } else {
            const unsigned mask = __ballot_sync(G2_FULL, lead);
            if (waiting + 32 / G > 32) flush();
            if (lead) {
                const int p = waiting + __popc(mask & lanemask_lt());
                s_v[wid][p] = v;
                s_m[wid][p] = a.m;
                s_e[wid][p] = a.e;
            }
            waiting += __popc(mask);
        }
    }
    if (kWait) flush();
}

// Level pass of the fused kernels over list[0, cnt): small vertices one per
// thread or warp, big ones one per CTA.  The backward pass of the deepest
// level has no successors to look for (`deepest`).  SHORT: every list is short.
template <bool SIGMA, bool SHORT>
__device__ void bc_level_pass(const BcState &s, const int32_t *list, int32_t cnt, int32_t d,
                              int bid, int nb, bool deepest = false) {
    if (SHORT || deepest) {  // uniform over the grid
        const int64_t nt = (int64_t)nb * blockDim.x;
        for (int64_t i = (int64_t)bid * blockDim.x + threadIdx.x; i < cnt; i += nt) {
            const int32_t v = list[i];
            if (SIGMA) bc_finish_sigma(s, v, bc_sigma_thread(s, v, d), d + 1);
            else bc_finish_delta(s, v, deepest ? BigF{0, 0} : bc_delta_thread(s, v, d));
        }
        return;
    }
    bc_groups<SIGMA, 1, 4, true>(s, list, cnt, d, 0, kThreadDeg, bid, nb);
    bc_groups<SIGMA, 32, 4, true>(s, list, cnt, d, kThreadDeg, kBigDeg, bid, nb);
    if (!s.big) return;  // uniform: no vertex has that many arcs
    const int32_t *rp = SIGMA ? s.g.crowptr : s.g.rowptr;
    for (int32_t i = bid; i < cnt; i += nb) {
        const int32_t v = list[i];
        if (rp[v + 1] - rp[v] >= kBigDeg) bc_cta_vertex<SIGMA>(s, v, d);
    }
}

// --------------------------------------------------- levels grouped by degree
// The reached vertices sorted by (class, level) into one list: class 0 below
// 9 arcs (a thread per vertex), 1 below 129 (eight lanes), 2 below kBcPiece (a
// warp), 3 the rest (a CTA per piece of kBcPiece arcs), so that no pass reads
// a vertex it does not work on and no CTA walks a hub alone (RMAT-21: a level
// of three hubs took one CTA 149 us).  Counting sort: k_bc_sort twice, with a
// scan of the counts between.  The first kBcKeys keys are counted in shared
// memory (a power-law graph has a dozen levels), one global atomic per key
// and CTA.
constexpr int kBcKeys = 256;
constexpr int kBcPiece = 2048;

__device__ __forceinline__ int bc_class(int32_t deg) {
    return deg < 9 ? 0 : deg < 129 ? 1 : deg < kBcPiece ? 2 : 3;
}

template <bool PLACE>
__global__ void __launch_bounds__(kCta) k_bc_sort(const int32_t *depth, const int32_t *rowptr,
                                                  int32_t n, int32_t levels, int32_t *cnt,
                                                  const int32_t *off, int32_t *order) {
    __shared__ int32_t s_cnt[kBcKeys], s_base[kBcKeys];
    constexpr int kPer = 8;
    const int64_t tile = (int64_t)kCta * kPer;
    for (int64_t t0 = (int64_t)blockIdx.x * tile; t0 < n; t0 += (int64_t)gridDim.x * tile) {
        for (int i = threadIdx.x; i < kBcKeys; i += kCta) s_cnt[i] = 0;
        __syncthreads();
        int key[kPer], pos[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int64_t v = t0 + j * kCta + threadIdx.x;
            const int32_t dv = v < n ? depth[v] : -1;
            key[j] = dv < 0 ? -1 : bc_class(rowptr[v + 1] - rowptr[v]) * levels + dv;
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            // one atomic per key of a warp
            const unsigned same = __match_any_sync(G2_FULL, key[j]);
            const int lead = __ffs(same) - 1;
            int p = 0;
            if (key[j] >= 0 && (int)(threadIdx.x & 31) == lead)
                p = atomicAdd(key[j] < kBcKeys ? &s_cnt[key[j]] : &cnt[key[j]], __popc(same));
            pos[j] = __shfl_sync(G2_FULL, p, lead) + __popc(same & lanemask_lt());
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kBcKeys; i += kCta)
            if (s_cnt[i]) s_base[i] = atomicAdd(&cnt[i], s_cnt[i]);
        __syncthreads();
        if (PLACE) {
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (key[j] >= 0)
                    order[off[key[j]] + (key[j] < kBcKeys ? s_base[key[j]] : 0) + pos[j]] =
                        (int32_t)(t0 + j * kCta + threadIdx.x);
        }
        __syncthreads();
    }
}

// pieces of the class 3 vertices, and nothing of them done yet
__global__ void k_bc_pieces(const int32_t *rowptr, const int32_t *hubs, int32_t cnt, int32_t *np,
                            int32_t *done) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = hubs[i];
        np[i] = (rowptr[v + 1] - rowptr[v] + kBcPiece - 1) / kBcPiece;
        done[i] = 0;
    }
}

// One level's vertices: `list` and the length of each class' part of it.
struct BcLevel {
    const int32_t *list[4];
    int32_t cnt[4];
    // class 3: first piece of each vertex (cnt[3] + 1 entries; numbers of the
    // whole graph's pieces), pieces done of each vertex, results of the pieces
    const int32_t *piece;
    int32_t *done;
    int4 *part;
};

// sigma of the vertices at level d + 1 (SIGMA), or delta of those at level d.
// The largest first, each class by the whole grid.  Bound: the gathered records
// through L1 (66% of its peak on RMAT-20's largest levels) and L2 (45%).  Six
// CTAs per SM, though delta's pass spills 104 bytes at its 40 registers: it
// needs 70 unbounded (17.4 ms for 16 sources of RMAT-21 against 19.4, 17.7 with
// five, 18.9 with eight); two records in flight per lane instead of four 18.9 ms.
template <bool SIGMA>
__global__ void __launch_bounds__(kCta, 6) k_bc_level(BcState s, BcLevel l, int32_t d,
                                                   int32_t deepest) {
    if (deepest) {
        for (int c = 0; c < 4; ++c)
            for (int64_t i = (int64_t)blockIdx.x * kCta + threadIdx.x; i < l.cnt[c];
                 i += (int64_t)gridDim.x * kCta)
                bc_finish_delta(s, l.list[c][i], BigF{0, 0});
        return;
    }
    if (l.cnt[3] > 0) {
        __shared__ int s_last;
        const int32_t *rp = SIGMA ? s.g.crowptr : s.g.rowptr;
        const int32_t p1 = l.piece[l.cnt[3]];
        for (int32_t p = l.piece[0] + (int32_t)blockIdx.x; p < p1; p += gridDim.x) {
            const int32_t h = scan_owner(l.piece, l.cnt[3], p);
            const int32_t v = l.list[3][h], first = l.piece[h], np = l.piece[h + 1] - first;
            const int32_t e = rp[v + 1], b = rp[v] + (p - first) * kBcPiece;
            BigF a = bc_cta_sum(bc_part<4>(s, SIGMA ? s.g.ccol : s.g.col, SIGMA ? d : d + 1, b,
                                           e - b < kBcPiece ? e : b + kBcPiece, kCta,
                                           (int)threadIdx.x));
            if (threadIdx.x == 0) {
                __stcg(l.part + p, make_int4((int)(unsigned)a.m, (int)(unsigned)(a.m >> 32), a.e, 0));
                __threadfence();
                s_last = atomicAdd(l.done + h, 1) == np - 1;
            }
            __syncthreads();
            if (s_last) {
                // the last piece to end sums the results, always in one order
                __threadfence();
                a = BigF{0, 0};
                for (int32_t j = threadIdx.x; j < np; j += kCta) {
                    const int4 r = __ldcg(l.part + first + j);
                    a = bf_add(a, BigF{(unsigned long long)(unsigned)r.x |
                                           (unsigned long long)(unsigned)r.y << 32,
                                       r.z});
                }
                a = bc_cta_sum(a);
                if (threadIdx.x == 0) {
                    l.done[h] = 0;  // for the backward pass
                    bc_finish<SIGMA>(s, v, a, d);
                }
            }
            __syncthreads();
        }
    }
    bc_groups<SIGMA, 32, 4, false>(s, l.list[2], l.cnt[2], d, 0, 0, blockIdx.x, gridDim.x);
    bc_groups<SIGMA, 8, 4, false>(s, l.list[1], l.cnt[1], d, 0, 0, blockIdx.x, gridDim.x);
    bc_groups<SIGMA, 1, 4, false>(s, l.list[0], l.cnt[0], d, 0, 0, blockIdx.x, gridDim.x);
}

// depths and records before the source's search (its own set)
__global__ void k_bc_init(BcState s, int32_t n, int32_t *cnt3) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const bool is_src = v == s.src;
        s.depth[v] = is_src ? 0 : -1;
        // sigma(src) = 1 = 2^62 * 2^(1 - 63)
        bc_finish_sigma(s, (int32_t)v, BigF{is_src ? 1ull << 62 : 0ull, is_src ? 1 : 0},
                        is_src ? 0 : -1);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        s.lvl[0] = s.src;
        if (cnt3) {
            cnt3[0] = cnt3[1] = cnt3[2] = 0;
        }
    }
}

// the records alone
__global__ void k_bc_init_rec(BcState s, int32_t n) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const bool is_src = v == s.src;
        bc_finish_sigma(s, (int32_t)v, BigF{is_src ? 1ull << 62 : 0ull, is_src ? 1 : 0},
                        is_src ? 0 : -1);
    }
}

// ------------------------------------------------------------ fused source
struct BcFusedArgs {
    BcState s;
    int32_t *off;    // level offsets into lvl (off[d] = start of level d)
    int32_t *cnt3;   // rotating append counters (zero at launch)
    GridBarrier bar;
    int32_t *err;
    uint64_t limit_ns;
    int32_t fwd;     // 1: forward phases from level d0, whose list is lvl[b0, e0)
    int32_t d0, b0, e0;
    int32_t lo;      // > 0: after a phase, stop before a level of fewer vertices
    int32_t bwd;     // 1: backward pass after the forward pass (levels D-1 .. 0)
    int32_t Lhi, Llo;  // without the forward pass: backward over levels Lhi down to Llo
    int32_t deepest;   // ... of which this one is the deepest (no successors)
    int32_t *result; // out: [0] 1 if stopped for the cluster loop, [1] levels found (or
                     // the next level), [2] its start in lvl, [3] its size
};

// SHORT (a symmetric bounded-degree graph): a kernel without the passes by degree,
// in 64 registers, so that queries run side by side on a graph (a launch of one CTA per
// SM each) run four at a time: eight streams, one source each on the 4096^2 grid,
// 97 ms; 130 with the 128 registers of one kernel for both, 128 with 96, 86 with 48
// (but 39.9 ms against 38.9 alone).
constexpr int kBcBeside = 4;
template <int LB, bool SHORT>
__global__ void __launch_bounds__(kCta, SHORT ? kBcBeside : 2) k_bc_fused(BcFusedArgs a) {
    const BcState &s = a.s;
    int32_t Lhi = a.Lhi, deepest = a.deepest;
    const int32_t Llo = a.Llo;
    if (a.fwd) {
        OpBFS op{s.depth, nullptr};
        OutCtx out;
        memset(&out, 0, sizeof(out));
        out.mode = OUT_SPARSE;
        out.dedup = DD_NONE;
        out.err = a.err;
        int32_t b = a.b0, e = a.e0, d = a.d0;
        // one barrier per level: the discovery of level d+1 from level d and
        // the sigma of level d (pulled from level d-1) share a phase.  The
        // discovery reads no sigma, and the sigma pass only looks for depth
        // d-1, which no vertex discovered in the same phase (-1 -> d+1) has.
        for (;; ++d) {
            FrontierIn fin{s.lvl + b, e - b, nullptr};
            out.q = s.lvl + e;
            out.cnt = a.cnt3 + d % 3;
            out.cap = s.g.n - e;
            if (blockIdx.x == 0 && threadIdx.x == 0) a.cnt3[(d + 1) % 3] = 0;
            if (LB == G2_LB_WM) lb_warp(s.g, fin, e - b, op, out, blockIdx.x, gridDim.x, nullptr);
            else if (LB == G2_LB_CM) lb_cta(s.g, fin, e - b, op, out, blockIdx.x, gridDim.x, nullptr);
            else if (LB == G2_LB_ETWC) lb_etwc(s.g, fin, e - b, op, out, blockIdx.x, gridDim.x, nullptr);
            else lb_vertex(s.g, fin, e - b, op, out, blockIdx.x, gridDim.x, nullptr);
            if (d > 0) bc_level_pass<true, SHORT>(s, s.lvl + b, e - b, d - 1, blockIdx.x, gridDim.x);
            if (!grid_sync(a.bar, a.err, a.limit_ns)) return;
            const int32_t nn = ld_relaxed_i32(a.cnt3 + d % 3);
            if (nn == 0) break;
            if (blockIdx.x == 0 && threadIdx.x == 0) a.off[d + 2] = e + nn;
            b = e;
            e += nn;
            if (nn < a.lo) {  // the same length in every CTA
                if (blockIdx.x == 0 && threadIdx.x == 0) {
                    a.result[0] = 1;
                    a.result[1] = d + 1;
                    a.result[2] = b;
                    a.result[3] = nn;
                }
                return;
            }
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            a.result[0] = 0;
            a.result[1] = d + 1;
        }
        if (!a.bwd) return;
        Lhi = deepest = d;  // levels 0..d
    }
    for (int32_t L = Lhi; L >= Llo; --L) {
        const int32_t lb0 = ld_relaxed_i32(a.off + L), lb1 = ld_relaxed_i32(a.off + L + 1);
        bc_level_pass<false, SHORT>(s, s.lvl + lb0, lb1 - lb0, L, blockIdx.x, gridDim.x, L == deepest);
        if (!grid_sync(a.bar, a.err, a.limit_ns)) return;
    }
}

// --------------------------------------------------- fused source in one cluster
// On a symmetric bounded-degree graph (the thread-per-vertex passes) the
// small levels of a fused WM source run inside one thread-block cluster, as
// the fused BFS does: the CTAs keep the vertices they discover in shared
// memory, a level ends at the cluster barrier, and every CTA takes an equal
// slice of the concatenated level, read through distributed shared memory.
// In the phase of level d a CTA copies its part of level d to the global
// level list (for the backward pass), discovers level d+1 from its slice
// (the slice's arcs spread over the warp's lanes, four deep) and computes the
// slice's sigma from level d-1.  A level of more than `hi` vertices goes to
// the grid-wide kernel (k_bc_fused), which hands the forward pass back below
// `lo`; the backward pass runs level ranges on one or the other by level
// size.  A level that outgrows a CTA's buffer (appends past the capacity are
// counted, not stored) ends the launch; its vertices all carry their depth,
// so the host rebuilds the level's list from the depths.
constexpr int kBcQcap = 28672;  // level entries per CTA and buffer (2 buffers: 224 KiB)
constexpr size_t kBcSmem = 2 * (size_t)kBcQcap * 4;

struct ClusterBcArgs {
    BcState s;
    int32_t *off;     // level offsets into s.lvl (off[d] = start of level d)
    int32_t fwd;      // 1: forward phases from level d0 (list lvl[start0, start0 + n0))
    int32_t d0, start0, n0;
    int32_t hi;       // stop before a level with more vertices
    int32_t Lhi, Llo; // without the forward pass: backward over levels Lhi down to Llo
    int32_t deepest;  // ... of which this one is the deepest (no successors)
    int32_t *result;  // out: [0] CL_DONE / CL_TO_GRID / CL_OVERFLOW, [1] levels found (or
                      // the level handed over), [2] its start in lvl, [3] its size
};

template <int CL>
__global__ void __launch_bounds__(kClCta, 1) k_bc_cluster(ClusterBcArgs a) {
    const BcState &s = a.s;
    extern __shared__ int32_t s_q[];  // [2][kBcQcap]
    __shared__ int32_t s_cnt[2];
    __shared__ int32_t s_off[CL + 1];
    __shared__ int32_t s_over;
    const uint32_t rank = cl_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t *__restrict__ rowptr = s.g.rowptr;
    const int32_t *__restrict__ col = s.g.col;
    if (!a.fwd) {
        for (int32_t L = a.Lhi; L >= a.Llo; --L) {
            const int32_t b0 = a.off[L], cnt = a.off[L + 1] - b0;
            const int32_t lo = (int32_t)((int64_t)cnt * rank / CL);
            const int32_t hi = (int32_t)((int64_t)cnt * (rank + 1) / CL);
            for (int32_t i = lo + threadIdx.x; i < hi; i += kClCta) {
                const int32_t v = s.lvl[b0 + i];
                bc_finish_delta(s, v, L == a.deepest ? BigF{0, 0} : bc_delta_thread(s, v, L));
            }
            cl_barrier();  // level L's dependencies visible to level L-1
        }
        return;
    }
    if (threadIdx.x == 0) {
        s_cnt[0] = 0;
        s_cnt[1] = 0;
    }
    int32_t start = a.start0, total = a.n0;  // level d: lvl[start, start + total)
    int reason = CL_DONE;
    cl_barrier();
    int d = a.d0;
    for (;; ++d) {
        const int cb = d & 1, nb = cb ^ 1;
        const bool first = d == a.d0;
        if (!first) {
            if (warp == 0) {
                int32_t c = lane < CL ? cl_read(&s_cnt[cb], lane) : 0;
                const bool ov = __any_sync(G2_FULL, c > kBcQcap);
#pragma unroll
                for (int o = 1; o < CL; o <<= 1) {
                    const int32_t t = __shfl_up_sync(G2_FULL, c, o);
                    if (lane >= o) c += t;
                }
                if (lane < CL) s_off[lane + 1] = c;
                if (lane == 0) {
                    s_off[0] = 0;
                    s_over = ov;
                    s_cnt[nb] = 0;
                }
            }
            __syncthreads();
            total = s_off[CL];
            if (total == 0) break;
            if (s_over) {
                reason = CL_OVERFLOW;
                break;
            }
            // level d to the global list
            const int32_t mine = s_off[rank + 1] - s_off[rank];
            int32_t *dst = s.lvl + start + s_off[rank];
            for (int32_t j = threadIdx.x; j < mine; j += kClCta) dst[j] = s_q[cb * kBcQcap + j];
            if (total > a.hi) {
                reason = CL_TO_GRID;
                break;
            }
        }
        if (rank == 0 && threadIdx.x == 0) a.off[d] = start;
        const int32_t *cur = s_q + cb * kBcQcap;
        int32_t *nxt = s_q + nb * kBcQcap;
        const int32_t lo = (int32_t)((int64_t)total * rank / CL);
        const int32_t hi = (int32_t)((int64_t)total * (rank + 1) / CL);
        for (int32_t base = lo + warp * 32; base < hi; base += kClCta) {
            const int32_t i = base + lane;
            int32_t u = 0, beg = 0, deg = 0;
            if (i < hi) {
                if (first) {
                    u = s.lvl[start + i];
                } else {
                    const int r = cl_owner<CL>(s_off, i);
                    u = cl_read(cur + (i - s_off[r]), (uint32_t)r);
                }
                beg = __ldg(rowptr + u);
                deg = __ldg(rowptr + u + 1) - beg;
                if (d > 0) bc_finish_sigma(s, u, bc_sigma_thread(s, u, d - 1), d);
            }
            int32_t incl = deg;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t t = __shfl_up_sync(G2_FULL, incl, o);
                if (lane >= o) incl += t;
            }
            const int32_t tot = __shfl_sync(G2_FULL, incl, 31);
            const int32_t excl = incl - deg;
            for (int32_t k0 = 0; k0 < tot; k0 += 32 * 4) {
                int32_t v[4], dv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int32_t k = k0 + 32 * j + lane;
                    int own = 0;
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) {
                        const int32_t ex = __shfl_sync(G2_FULL, excl, own + step);
                        if (ex <= k) own += step;
                    }
                    const int32_t ob = __shfl_sync(G2_FULL, beg, own);
                    const int32_t oe = __shfl_sync(G2_FULL, excl, own);
                    v[j] = k < tot ? __ldg(col + ob + (k - oe)) : -1;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) dv[j] = v[j] >= 0 ? atomicCAS(s.depth + v[j], -1, d + 1) : 0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    cta_append(nxt, &s_cnt[nb], kBcQcap, v[j], v[j] >= 0 && dv[j] == -1, lane);
            }
        }
        start += total;
        cl_barrier();  // level d+1 found, sigma of level d and the list of level d written
    }
    cl_barrier();  // no CTA leaves while a peer may still read its counts
    if (rank == 0 && threadIdx.x == 0) {
        a.result[0] = reason;
        a.result[1] = d;
        a.result[2] = start;
        a.result[3] = total;
        a.off[d] = start;
        if (reason == CL_TO_GRID) a.off[d + 1] = start + total;
    }
}

// ------------------------------------------------------------------- host
// The source's depths by one edgeset.apply round per level.  Level L's vertices
// are s.lvl[starts[L], starts[L + 1]).
static g2_status bc_depths(g2_graph *g, const BcState &s, const g2_hybrid &h,
                           std::vector<int32_t> &starts, cudaStream_t st, int32_t *d_err) {
    Topology *t = g->topo;
    const int32_t n = t->n;
    int32_t *ctrs = d_err - 62;
    uint32_t *bm;
    uint8_t *bo;
    G2_TRY(ws(g, B_BM0, (size_t)(n + 31) / 32 + 1, &bm));
    G2_TRY(ws(g, B_BOOL0, (size_t)std::max(n, 1), &bo));
    int32_t b = 0, e = 1;
    starts.assign(1, 0);
    for (;;) {
        starts.push_back(e);
        const int32_t size = e - b;
        const g2_schedule &sc = pick_schedule(h, size, n);
        G2_TRY(check_schedule(g, sc, K_BFS, false));
        if (sc.load_balance == G2_LB_EDGE_ONLY)
            return fail(G2_EUNSUPPORTED, "BC's BFS is frontier-driven; EDGE_ONLY is for full sweeps");
        VSet in{OUT_SPARSE, s.lvl + b, size, nullptr, nullptr, nullptr, size};
        if (sc.direction == G2_PULL) {
            int want = sc.pull_frontier == G2_BITMAP ? OUT_BITMAP : OUT_BOOLMAP;
            VSet tt{want, nullptr, 0, nullptr, bm, bo, size};
            G2_TRY(vset_convert(g, in, want, tt, st));
            in = tt;
        }
        OpArgs a;
        memset(&a, 0, sizeof(a));
        a.kind = K_BFS;
        a.i0 = s.depth;
        a.err = d_err;
        a.threshold = G2_INF32;
        OutArgs o;
        memset(&o, 0, sizeof(o));
        o.rep = OUT_SPARSE;
        o.q = s.lvl + e;
        o.qcap = n - e;
        o.cnt = ctrs + 3;
        o.dedup = DD_NONE;
        G2_CK(cudaMemsetAsync(o.cnt, 0, 4, st));
        G2_TRY(apply_round(g, sc, a, in, o, st));
        sc.direction == G2_PUSH ? stats().push_rounds++ : stats().pull_rounds++;
        G2_TRY(read_counters(g, ctrs, 4, st, d_err));
        const int32_t nn = g->h_ctr[3];
        if (nn == 0) return G2_OK;
        stats().iterations++;
        b = e;
        e += nn;
    }
}

// A source's levels grouped by class (bc_group): bounds on the host.
struct BcGroups {
    std::vector<int32_t> off;  // class c of level L: order[off[c * levels + L], off[c * levels + L + 1])
    int32_t levels;
    const int32_t *piece;
    int32_t *done;
    int4 *part;
};

// The vertices of every level grouped by class of their degree in `rowptr`
// into s.lvl.
static g2_status bc_group(g2_graph *g, const BcState &s, const int32_t *rowptr, int32_t levels,
                          BcGroups &gr, cudaStream_t st, int32_t *d_err) {
    const int32_t n = g->topo->n, keys = std::max(4 * levels, kBcKeys);
    int32_t *cnt, *doff;
    G2_TRY(ws(g, B_I1, (size_t)keys, &cnt));
    G2_TRY(ws(g, B_SCAN, (size_t)keys + 1, &doff));
    const int grid = grid_for(g, n, kCta * 8);
    G2_CK(cudaMemsetAsync(cnt, 0, (size_t)keys * 4, st));
    k_bc_sort<false><<<grid, kCta, 0, st>>>(s.depth, rowptr, n, levels, cnt, nullptr, nullptr);
    G2_TRY(exclusive_scan_i32(g, cnt, doff, keys, st));
    G2_CK(cudaMemsetAsync(cnt, 0, (size_t)keys * 4, st));
    k_bc_sort<true><<<grid, kCta, 0, st>>>(s.depth, rowptr, n, levels, cnt, doff, s.lvl);
    stats().launches += 2;
    gr.levels = levels;
    gr.off.resize((size_t)4 * levels + 1);
    G2_CK(cudaMemcpyAsync(gr.off.data(), doff, gr.off.size() * 4, cudaMemcpyDeviceToHost, st));
    G2_TRY(sync_and_check(g, st, d_err));
    const int32_t h0 = gr.off[(size_t)3 * levels], hubs = gr.off[(size_t)4 * levels] - h0;
    gr.piece = nullptr;
    gr.done = nullptr;
    gr.part = nullptr;
    if (hubs > 0) {
        int32_t *np, *piece;
        G2_TRY(ws(g, B_TWC_S, (size_t)hubs, &np));
        G2_TRY(ws(g, B_TWC_M, (size_t)hubs + 1, &piece));
        G2_TRY(ws(g, B_TWC_L, (size_t)hubs, &gr.done));
        // every piece but a vertex's last is full
        G2_TRY(ws(g, B_D1, (size_t)g->topo->m / kBcPiece + (size_t)hubs, &gr.part));
        k_bc_pieces<<<grid_for(g, hubs, kCta), kCta, 0, st>>>(rowptr, s.lvl + h0, hubs, np, gr.done);
        G2_TRY(exclusive_scan_i32(g, np, piece, hubs, st));
        stats().launches += 1;
        gr.piece = piece;
    }
    return G2_OK;
}

// One level's pass over the groups.
template <bool SIGMA>
static void launch_level(g2_graph *g, const BcState &s, const BcGroups &gr, int32_t level, int32_t d,
                         bool deepest, cudaStream_t st) {
    BcLevel l;
    for (int c = 0; c < 4; ++c) {
        const int32_t *o = gr.off.data() + (size_t)c * gr.levels + level;
        l.list[c] = s.lvl + o[0];
        l.cnt[c] = o[1] - o[0];
    }
    const int32_t h = gr.off[(size_t)3 * gr.levels + level] - gr.off[(size_t)3 * gr.levels];
    l.piece = gr.piece ? gr.piece + h : nullptr;
    l.done = gr.done ? gr.done + h : nullptr;
    l.part = gr.part;
    // enough CTAs for every class at once, of hubs with a few dozen pieces
    const int64_t want = (int64_t)l.cnt[3] * 32 + (l.cnt[2] + kWarps - 1) / kWarps +
                         (l.cnt[1] + kCta / 8 - 1) / (kCta / 8) + (l.cnt[0] + kCta - 1) / kCta;
    k_bc_level<SIGMA><<<grid_for(g, want, 1), kCta, 0, st>>>(s, l, d, deepest);
    stats().launches += 1;
}

// One source: depths (one fused launch with `fused_depths`, else a round per
// level), the levels grouped, sigma level by level, delta from the deepest.
static g2_status bc_one_plain(g2_graph *g, const BcState &s, const g2_hybrid &h, bool fused_depths,
                              BcGroups &gr, cudaStream_t st, int32_t *d_err) {
    Topology *t = g->topo;
    const int32_t n = t->n;
    int32_t levels = 0;
    if (fused_depths) {
        const int32_t it = stats().iterations, push = stats().push_rounds, pull = stats().pull_rounds;
        // the hybrid's counters, zero at the start of a call, lie in ctrs[20, 56)
        G2_CK(cudaMemsetAsync(d_err - 62 + 20, 0, 36 * 4, st));
        G2_TRY(bfs_fused_do(g, s.src, s.depth, nullptr, h, true, st, d_err));
        levels = stats().iterations;
        stats().iterations += it - 1;
        stats().push_rounds += push;
        stats().pull_rounds += pull;
        k_bc_init_rec<<<grid_for(g, n, kCta), kCta, 0, st>>>(s, n);
    } else {
        k_bc_init<<<grid_for(g, n, kCta), kCta, 0, st>>>(s, n, nullptr);
        G2_TRY(bc_depths(g, s, h, gr.off, st, d_err));
        levels = (int32_t)gr.off.size() - 1;
    }
    stats().launches += 1;
    if (!fused_depths && s.per_thread) {
        // short lists: the levels as they were found, a thread per vertex (all
        // of class 0; sorting each source's vertices by degree costs a 64 x 64
        // grid 4% of the call)
        gr.levels = levels;
        gr.off.resize((size_t)4 * levels + 1, gr.off.back());
        gr.piece = nullptr;
        gr.done = nullptr;
        gr.part = nullptr;
    } else {
        G2_TRY(bc_group(g, s, s.g.crowptr, levels, gr, st, d_err));
    }
    for (int32_t L = 1; L < levels; ++L) launch_level<true>(g, s, gr, L, L - 1, false, st);
    if (!t->symmetric) G2_TRY(bc_group(g, s, s.g.rowptr, levels, gr, st, d_err));
    for (int32_t L = levels - 1; L >= 0; --L)
        launch_level<false>(g, s, gr, L, L, L == levels - 1, st);
    G2_CK(cudaGetLastError());
    return G2_OK;
}

template <class A>
static g2_status launch_bc_grid(g2_graph *g, const g2_schedule &sc, A &a, cudaStream_t st) {
    auto launch = [&](auto kern) -> g2_status {
        int per_sm = 0;
        G2_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kCta, 0));
        if (per_sm < 1) return fail(G2_EUNSUPPORTED, "fused BC kernel does not fit on an SM");
        void *params[] = {&a};
        G2_CK(cudaLaunchCooperativeKernel((const void *)kern, dim3(g->topo->sm_count), dim3(kCta),
                                          params, 0, st));
        stats().launches += 1;
        return G2_OK;
    };
    const bool brief = a.s.per_thread;
    switch (sc.load_balance) {
        case G2_LB_WM:
            return brief ? launch(k_bc_fused<G2_LB_WM, true>) : launch(k_bc_fused<G2_LB_WM, false>);
        case G2_LB_CM:
            return brief ? launch(k_bc_fused<G2_LB_CM, true>) : launch(k_bc_fused<G2_LB_CM, false>);
        case G2_LB_ETWC:
            return brief ? launch(k_bc_fused<G2_LB_ETWC, true>) : launch(k_bc_fused<G2_LB_ETWC, false>);
        default:
            return brief ? launch(k_bc_fused<G2_LB_VERTEX_BASED, true>)
                         : launch(k_bc_fused<G2_LB_VERTEX_BASED, false>);
    }
}

static g2_status check_fused_bc(const g2_schedule &sc) {
    switch (sc.load_balance) {
        case G2_LB_VERTEX_BASED: case G2_LB_WM: case G2_LB_CM: case G2_LB_ETWC: break;
        default:
            return fail(G2_EUNSUPPORTED, "fused BC supports VERTEX_BASED, WM, CM and ETWC");
    }
    if (sc.direction != G2_PUSH) return fail(G2_EUNSUPPORTED, "fused BC runs PUSH discovery");
    return G2_OK;
}

// One source in one grid-wide cooperative launch (forward and backward).
static g2_status bc_one_fused(g2_graph *g, const BcState &s, const g2_schedule &sc, cudaStream_t st,
                              int32_t *d_err) {
    G2_TRY(check_fused_bc(sc));
    Topology *t = g->topo;
    const int32_t n = t->n;
    int32_t *ctrs = d_err - 62;
    BcFusedArgs a;
    memset(&a, 0, sizeof(a));
    a.s = s;
    G2_TRY(ws(g, B_I1, (size_t)n + 2, &a.off));
    a.cnt3 = ctrs + 20;
    a.bar = GridBarrier{reinterpret_cast<unsigned long long *>(ctrs + 28)};
    a.err = d_err;
    a.limit_ns = barrier_limit_ns();
    a.fwd = 1;
    a.d0 = 0;
    a.b0 = 0;
    a.e0 = 1;
    a.lo = 0;
    a.bwd = 1;
    a.Llo = 0;
    a.result = ctrs + 24;
    k_bc_init<<<grid_for(g, n, kCta), kCta, 0, st>>>(s, n, ctrs + 20);
    stats().launches += 1;
    G2_TRY(put_i32(st, {{a.off, 0}, {a.off + 1, 1}}));
    G2_CK(cudaMemsetAsync(ctrs + 28, 0, 8, st));  // barrier words
    G2_TRY(launch_bc_grid(g, sc, a, st));
    G2_TRY(read_counters(g, ctrs + 24, 2, st, d_err));
    stats().iterations += g->h_ctr[1];
    stats().barriers += 2 * g->h_ctr[1];
    return G2_OK;
}

// One fused WM source whose small levels run in one cluster of `cl` CTAs and
// large ones in the grid-wide kernel: the forward pass moves between the two
// at level boundaries (to the grid above `hi` vertices, back below `lo`), the
// backward pass runs each maximal range of small or large levels on one or
// the other.
static g2_status bc_one_cluster(g2_graph *g, const BcState &s, const g2_schedule &sc, int cl,
                                cudaStream_t st, int32_t *d_err) {
    G2_TRY(check_fused_bc(sc));
    Topology *t = g->topo;
    const int32_t n = t->n;
    int32_t *ctrs = d_err - 62;
    int32_t *off;
    G2_TRY(ws(g, B_I1, (size_t)n + 2, &off));
    ClusterBcArgs c;
    memset(&c, 0, sizeof(c));
    c.s = s;
    c.off = off;
    c.hi = env_i32("G2_CLUSTER_BC_HI", 256 * cl);
    c.result = ctrs + 32;
    BcFusedArgs a;
    memset(&a, 0, sizeof(a));
    a.s = s;
    a.off = off;
    a.cnt3 = ctrs + 20;
    a.bar = GridBarrier{reinterpret_cast<unsigned long long *>(ctrs + 28)};
    a.err = d_err;
    a.limit_ns = barrier_limit_ns();
    a.lo = std::max(1, env_i32("G2_CLUSTER_BC_LO", 128 * cl));
    a.result = ctrs + 24;
    const size_t smem = kBcSmem;
    auto cluster = [&]() -> g2_status {
        return cl == 16 ? launch_cluster(k_bc_cluster<16>, 16, smem, c, st)
                        : launch_cluster(k_bc_cluster<8>, 8, smem, c, st);
    };
    k_bc_init<<<grid_for(g, n, kCta), kCta, 0, st>>>(s, n, nullptr);
    stats().launches += 1;
    G2_CK(cudaGetLastError());
    G2_CK(cudaMemsetAsync(ctrs + 28, 0, 8, st));  // barrier words
    // forward
    int32_t level = 0, start = 0, count = 1, D = 0;
    bool in_cluster = true;
    for (;;) {
        if (in_cluster) {
            c.fwd = 1;
            c.d0 = level;
            c.start0 = start;
            c.n0 = count;
            G2_TRY(cluster());
            G2_TRY(read_counters(g, ctrs + 32, 4, st, d_err));
            const int32_t why = g->h_ctr[0], d = g->h_ctr[1];
            if (d <= level) return fail(G2_ECUDA, "cluster BC made no progress");
            level = d;
            start = g->h_ctr[2];
            count = g->h_ctr[3];
            if (why == CL_DONE) {
                D = d;
                break;
            }
            if (why == CL_OVERFLOW) {  // the level's list from the depths
                G2_CK(cudaMemsetAsync(ctrs + 36, 0, 4, st));
                k_level_list<<<grid_for(g, n, kCta), kCta, 0, st>>>(s.depth, n, level, s.lvl + start,
                                                                    ctrs + 36, d_err);
                stats().launches += 1;
                G2_TRY(read_counters(g, ctrs + 36, 1, st, d_err));
                count = g->h_ctr[0];
            }
        } else {
            G2_TRY(put_i32(st, {{off + level, start}, {off + level + 1, start + count}}));
            G2_CK(cudaMemsetAsync(a.cnt3, 0, 12, st));
            a.fwd = 1;
            a.bwd = 0;
            a.d0 = level;
            a.b0 = start;
            a.e0 = start + count;
            G2_TRY(launch_bc_grid(g, sc, a, st));
            G2_TRY(read_counters(g, ctrs + 24, 4, st, d_err));
            const int32_t back = g->h_ctr[0], d = g->h_ctr[1];
            if (d <= level) return fail(G2_ECUDA, "fused BC made no progress");
            if (!back) {
                D = d;
                break;
            }
            level = d;
            start = g->h_ctr[2];
            count = g->h_ctr[3];
        }
        in_cluster = !in_cluster;
    }
    stats().iterations += D;
    stats().barriers += 2 * D;
    // backward over levels D-1 .. 0, by ranges of small / large levels
    if (D < 2) return G2_OK;  // (the source alone)
    c.deepest = a.deepest = D - 1;
    std::vector<int32_t> offs((size_t)D + 1);
    G2_CK(cudaMemcpyAsync(offs.data(), off, ((size_t)D + 1) * 4, cudaMemcpyDeviceToHost, st));
    G2_TRY(sync_and_check(g, st, d_err));
    for (int32_t L = D - 1; L >= 0;) {
        const bool small = offs[L + 1] - offs[L] <= c.hi;
        int32_t Llo = L;
        while (Llo > 0 && (offs[Llo] - offs[Llo - 1] <= c.hi) == small) --Llo;
        if (small) {
            c.fwd = 0;
            c.Lhi = L;
            c.Llo = Llo;
            G2_TRY(cluster());
        } else {
            a.fwd = 0;
            a.Lhi = L;
            a.Llo = Llo;
            G2_TRY(launch_bc_grid(g, sc, a, st));
        }
        L = Llo - 1;
    }
    return G2_OK;
}

g2_status bc_run(g2_graph *g, const int32_t *srcs, int32_t k, double *bc, const g2_hybrid &h,
                 bool fused_depths, cudaStream_t st, int32_t *d_err) {
    Topology *t = g->topo;
    const int32_t n = t->n;
    BcState s;
    s.g = t->view();
    s.bc = bc;
    int32_t dmax = 0;
    G2_TRY(max_out_degree(g, st, &dmax));
    s.per_thread = t->symmetric && dmax <= kBoundedDegree;
    s.big = !(t->symmetric && dmax < kBigDeg);
    G2_TRY(ws(g, B_I0, (size_t)std::max(n, 1), &s.depth));
    G2_TRY(ws(g, B_LVL, (size_t)std::max(n, 1), &s.lvl));
    G2_TRY(ws(g, B_D0, (size_t)std::max(n, 1), &s.rec));
    G2_CK(cudaMemsetAsync(bc, 0, (size_t)n * 8, st));
    BcGroups groups;
    // fused WM sources on a symmetric bounded-degree graph use the cluster
    const int cl = h.s1.kernel_fusion && h.s1.load_balance == G2_LB_WM && s.per_thread
                       ? cluster_size(2, k_bc_cluster<16>, k_bc_cluster<8>, kBcSmem)
                       : 0;
    for (int32_t i = 0; i < k; ++i) {
        s.src = srcs[i];
        if (cl) G2_TRY(bc_one_cluster(g, s, h.s1, cl, st, d_err));
        else if (h.s1.kernel_fusion) G2_TRY(bc_one_fused(g, s, h.s1, st, d_err));
        else G2_TRY(bc_one_plain(g, s, h, fused_depths, groups, st, d_err));
        G2_TRY(sync_and_check(g, st, d_err));
    }
    return G2_OK;
}

}  // namespace g2

using namespace g2;

// Tuned schedule when the caller passes none: the direction-optimising
// hybrid of BFS (STRICT PUSH below 2% of n, VERTEX_BASED PULL over a bitmap);
// on a bounded-degree graph each source runs fused (WM PUSH).
static g2_hybrid tuned_bc_hybrid(g2_graph *g, cudaStream_t st) {
    int32_t dmax = 0;
    if (max_out_degree(g, st, &dmax) == G2_OK && dmax <= kBoundedDegree) {
        g2_hybrid h = default_hybrid();
        h.s1.load_balance = G2_LB_WM;
        h.s1.kernel_fusion = 1;
        h.s2 = h.s1;
        return h;
    }
    g2_hybrid h = default_hybrid();
    h.criteria = G2_INPUT_VERTEXSET_SIZE;
    h.threshold = 0.02f;
    h.s1.load_balance = G2_LB_STRICT;
    h.s2.load_balance = G2_LB_VERTEX_BASED;
    h.s2.direction = G2_PULL;
    h.s2.pull_frontier = G2_BITMAP;
    h.s2.dedup = G2_DEDUP_DISABLED;
    return h;
}

extern "C" g2_status g2_bc(g2_graph *g, const int32_t *srcs, int32_t k, double *bc,
                           const g2_hybrid *sched, void *stream) {
    if (!g || !bc || (k > 0 && !srcs) || k < 0) return fail(G2_EINVAL, "bad BC arguments");
    for (int32_t i = 0; i < k; ++i)
        if (srcs[i] < 0 || srcs[i] >= g->topo->n) return fail(G2_EINVAL, "source vertex out of range");
    cudaStream_t st = as_stream(stream);
    g2_hybrid h = sched ? *sched : tuned_bc_hybrid(g, st);
    if (h.s1.kernel_fusion && h.criteria != G2_CRITERIA_NONE && !h.s2.kernel_fusion)
        return fail(G2_EUNSUPPORTED, "kernel fusion must be set on both hybrid schedules");
    int32_t *d_err;
    G2_TRY(begin_call(g, st, &d_err));
    // Tuned, several sources on a power-law graph: each source's depths in one
    // launch of the fused direction-optimising hybrid.  (A single source keeps
    // the rounds: that cooperative launch needs every SM at once, and a server
    // runs single sources beside other streams.)
    const bool fused_depths = !sched && !h.s1.kernel_fusion && k > 1;
    G2_TRY(bc_run(g, srcs, k, bc, h, fused_depths, st, d_err));
    return end_call(g, st, d_err);
}
