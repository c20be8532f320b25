// g2_batch.cu — multi-source traversals: up to 64 BFS sources share one
// frontier loop with one bit per source in per-vertex 64-bit masks, and up to
// 32 SSSP sources relax stacked distance arrays together, so the topology is
// read once per round for all of them.  PUSH rounds reuse the load-balancing
// library with mask-valued update functions; the BFS's PULL rounds have kernels
// of their own.
#include <cuda_runtime.h>

#include <string>
#include <thread>
#include <vector>

#include <algorithm>
#include <cstring>
#include <vector>

#include "g2_host.h"
#include "g2_lb.cuh"
#include "g2_push.cuh"

namespace g2 {

typedef unsigned long long u64;

// ------------------------------------------------------- multi-source BFS
// PUSH: the bits of u's frontier mask not yet visited at v are ORed into v's
// next mask; the first arc to touch v lists it.
struct OpMsBfs {
    const u64 *visit;
    const u64 *fcur;
    u64 *fnext;
    typedef u64 S;
    struct Pre {
        u64 seen, next;
    };
    typedef u64 Old;
    static constexpr int kFlight = 4;
    __device__ __forceinline__ S load(int32_t u) const { return fcur[u]; }
    __device__ __forceinline__ bool skip(S m) const { return m == 0; }
    __device__ __forceinline__ Pre pre(int32_t v, int32_t) const {
        return Pre{visit[v], fnext[v]};
    }
    __device__ __forceinline__ Old act(int32_t, S fm, int32_t v, int32_t, Pre p) const {
        const u64 m = fm & ~p.seen;
        return (p.next & m) == m ? ~0ull : atomicOr(&fnext[v], m);
    }
    __device__ __forceinline__ int fin(int32_t, S, int32_t, Pre, Old old) const {
        return old == 0;
    }
};

// Where the levels of a search go.  Up to kMsPlanes levels' bits are kept as
// bit planes: bit b of plane[j][v] is bit j of the depth of v from source b, so
// that a round writes 8 bytes a plane and vertex, and k_ms_out writes every
// depth once, in order.  (Written to depth[b][v] round by round, the 64 arrays
// took 446 us of RMAT-21's rounds in part lines, beside 80 us to clear them.)
// A search of more levels goes on writing its depths directly, and so does one
// without room for the planes or of few sources (12 sources: 0.36 against 0.37 ms
// on RMAT-14, 0.40 against 0.43 on 300,001 vertices, 0.63 against 0.67 on RMAT-20).
constexpr int kMsPlanes = 5;   // depths up to 31
constexpr int kMsDirect = 16;  // sources whose depths are written directly
struct MsLevels {
    u64 *plane[kMsPlanes];
    int32_t *depth;  // null while the planes are used
    int32_t n;
};

// The lanes' vertices v (nm: new bits) at `level`.  Called by all 32 lanes.
__device__ __forceinline__ void ms_set_level(const MsLevels &l, int32_t v, u64 nm, int32_t level) {
    if (!l.depth) {
#pragma unroll
        for (int j = 0; j < kMsPlanes; ++j)
            if (nm && ((level >> j) & 1)) l.plane[j][v] |= nm;
        return;
    }
    u64 any = (u64)__reduce_or_sync(G2_FULL, (unsigned)nm) |
              (u64)__reduce_or_sync(G2_FULL, (unsigned)(nm >> 32)) << 32;
    while (any) {
        const int b = __ffsll((long long)any) - 1;
        any &= any - 1;
        if ((nm >> b) & 1u) l.depth[(int64_t)b * l.n + v] = level;
    }
}

// depth[b][v] of every source b < k from the first `planes` planes (-1 where
// visit has not the bit).
__global__ void __launch_bounds__(kCta) k_ms_out(MsLevels l, const u64 *visit, int32_t planes,
                                                 int32_t k, int32_t *depth) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < l.n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const u64 seen = visit[v];
        u64 p[kMsPlanes];
#pragma unroll
        for (int j = 0; j < kMsPlanes; ++j) p[j] = j < planes ? l.plane[j][v] : 0;
#pragma unroll 8
        for (int b = 0; b < k; ++b) {
            int32_t d = 0;
#pragma unroll
            for (int j = 0; j < kMsPlanes; ++j) d |= (int32_t)((p[j] >> b) & 1u) << j;
            depth[(int64_t)b * l.n + v] = (seen >> b) & 1u ? d : -1;
        }
    }
}

// the bits of the warp's new masks into *active.  Called by all 32 lanes.
__device__ __forceinline__ void ms_note_active(u64 *active, u64 nm) {
    const u64 any = (u64)__reduce_or_sync(G2_FULL, (unsigned)nm) |
                    (u64)__reduce_or_sync(G2_FULL, (unsigned)(nm >> 32)) << 32;
    if ((threadIdx.x & 31) == 0 && (any & ~*active)) atomicOr(active, any);
}

// PULL: every vertex ORs the frontier masks of its in-neighbours and stops
// once it has every bit it can still get: those not yet visited of the sources
// whose frontier is not empty (`active`; a source in a small component ends
// after a level or two, and waiting for its bit made every vertex read its
// whole list).  Three kernels by the length of the list: k_ms_pull_pieces for
// kMsPiece arcs and more (where the graph has such a vertex), k_ms_pull for the
// first kMsThread arcs of the rest, a thread each, k_ms_pull_rest for what those
// threads leave, a warp each from a list (left to the warp that found them, the
// low ids of a power-law graph held it for half a millisecond; not launched where
// no list is longer).  A vertex's new bits become visited, its level noted and
// the vertex listed in k_ms_pull, for the pieces' vertices too, and those of
// the rest in k_ms_pull_end, a lane each (by the warps of k_ms_pull_rest, a
// vertex each: RMAT-20 5% slower; 32 vertices a warp there: 26%).  64 sources:
// RMAT-21, the whole tuned search 1.10 ms (with a thread per vertex waiting for
// every source 3.7, 6 where one source lay in a small component).
struct MsPullArgs {
    DevGraph g;
    u64 *visit;
    const u64 *fcur;
    u64 *fnext;
    const u64 *active;  // sources with a frontier
    u64 *active_next;
    MsLevels l;
    int32_t level;
    int32_t *q, *q_cnt;  // the vertices with new bits
    int32_t *rest, *rest_cnt;
    int32_t alone;       // arcs a thread walks before it leaves the rest
    int32_t *err;
    unsigned long long *ctr;
};

constexpr int32_t kMsThread = 32;   // arcs a thread walks alone ...
constexpr int32_t kMsAlone = 128;   // ... or the whole list where none is longer than this
constexpr int32_t kMsPiece = 2048;  // arcs of a big vertex a CTA takes

// the OR of up to four masks, in flight together, at arcs e, e + step, ...
__device__ __forceinline__ u64 ms_gather(const MsPullArgs &a, int64_t e, int step, int64_t end) {
    int32_t u[4];
    u64 m = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) u[j] = e + (int64_t)j * step < end ? a.g.ccol[e + (int64_t)j * step] : -1;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (u[j] >= 0) m |= a.fcur[u[j]];
    return m;
}

__device__ __forceinline__ OutCtx ms_out(const MsPullArgs &a) {
    OutCtx out;
    memset(&out, 0, sizeof(out));
    out.mode = OUT_SPARSE;
    out.q = a.q;
    out.cnt = a.q_cnt;
    out.cap = out.cap2 = a.g.n;
    out.q2 = a.rest;
    out.cnt2 = a.rest_cnt;
    out.err = a.err;
    return out;
}

__global__ void __launch_bounds__(kCta) k_ms_pull(MsPullArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const u64 active = *a.active;
    const int32_t n = a.g.n;
    const OutCtx out = ms_out(a);
    Stage st = stage_begin();
    for (int64_t base = gw * 32; base < n; base += nw * 32) {
        const int64_t v = base + lane;
        const u64 seen = v < n ? a.visit[v] : ~0ull;
        const u64 need = active & ~seen;
        u64 nm = 0;
        int32_t b = 0, e = 0;
        int cnt = 0;
        bool more = false;
        if (need) {
            b = a.g.crowptr[v];
            e = a.g.crowptr[v + 1];
            if (e - b < kMsPiece) {
                const int32_t e1 = e - b > a.alone ? b + a.alone : e;
                for (; b < e1 && (nm & need) != need; b += 4) {
                    nm |= ms_gather(a, b, 1, e1);
                    cnt += e1 - b < 4 ? e1 - b : 4;
                }
                nm &= need;
                more = b < e && nm != need;
                if (nm) a.fnext[v] = nm;
            } else {
                nm = a.fnext[v];  // the pieces' result
            }
        }
        count_arcs(a.ctr, cnt);
        if (more) nm = 0;  // k_ms_pull_rest goes on from fnext
        const bool found = nm != 0;
        if (__any_sync(G2_FULL, found)) {
            if (found) a.visit[v] = seen | nm;
            ms_set_level(a.l, (int32_t)v, nm, a.level);
            ms_note_active(a.active_next, nm);
        }
        const int32_t vs[1] = {(int32_t)v};
        const int code[1] = {found ? 1 : more ? 2 : 0};
        emit_n<1>(out, st, vs, code);
    }
    stage_end(out, st);
}

__global__ void __launch_bounds__(kCta) k_ms_pull_rest(MsPullArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const u64 active = *a.active;
    const int32_t cnt = *a.rest_cnt;
    for (int64_t i = gw; i < cnt; i += nw) {
        const int32_t v = a.rest[i];
        const u64 need = active & ~a.visit[v], have = a.fnext[v];
        const int64_t e = a.g.crowptr[v + 1];
        u64 got = have;
        int64_t k = (int64_t)a.g.crowptr[v] + kMsThread;
        for (; k < e && (got & need) != need; k += 128) {
            const u64 m = ms_gather(a, k + lane, 32, e);
            got |= (u64)__reduce_or_sync(G2_FULL, (unsigned)m) |
                   (u64)__reduce_or_sync(G2_FULL, (unsigned)(m >> 32)) << 32;
        }
        if (lane == 0) {
            got &= need;
            if (got != have) a.fnext[v] = got;
            if (a.ctr) atomicAdd(a.ctr, (u64)((k < e ? k : e) - a.g.crowptr[v] - kMsThread));
        }
    }
}

// Piece p belongs to the vertex big[i] with piece[i] <= p < piece[i + 1].
__global__ void __launch_bounds__(kCta) k_ms_pull_pieces(MsPullArgs a, const int32_t *big,
                                                         int32_t nbig, const int32_t *piece) {
    __shared__ u64 s_m[kWarps];
    const u64 active = *a.active;
    const int32_t total = piece[nbig];
    for (int32_t p = blockIdx.x; p < total; p += gridDim.x) {
        const int32_t i = scan_owner(piece, nbig, p), v = big[i];
        const u64 need = active & ~a.visit[v];
        const int64_t b = (int64_t)a.g.crowptr[v] + (int64_t)(p - piece[i]) * kMsPiece;
        const int64_t e1 = a.g.crowptr[v + 1], e = e1 - b < kMsPiece ? e1 : b + kMsPiece;
        u64 m = 0;
        if (need && (*(volatile u64 *)&a.fnext[v] & need) != need) {
            for (int64_t k = b + threadIdx.x; k < e; k += 4 * kCta) m |= ms_gather(a, k, kCta, e);
            if (a.ctr && threadIdx.x == 0) atomicAdd(a.ctr, (u64)(e - b));
        }
        m = (u64)__reduce_or_sync(G2_FULL, (unsigned)m) |
            (u64)__reduce_or_sync(G2_FULL, (unsigned)(m >> 32)) << 32;
        if ((threadIdx.x & 31) == 0) s_m[threadIdx.x >> 5] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < kWarps; ++w) m |= s_m[w];
            if (m & need) atomicOr(&a.fnext[v], m & need);
        }
        __syncthreads();
    }
}

// the vertices of at least `big` in-arcs, and their numbers of pieces
__global__ void k_ms_big(const int32_t *crowptr, int32_t n, int32_t big, int32_t *list, int32_t *np,
                         int32_t *cnt) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t d = crowptr[v + 1] - crowptr[v];
        if (d >= big) {
            const int32_t i = atomicAdd(cnt, 1);
            list[i] = (int32_t)v;
            np[i] = (d + kMsPiece - 1) / kMsPiece;
        }
    }
}

// after a PUSH round: the new masks of the listed vertices (their number on
// the device) become visited, their levels noted
__global__ void k_ms_commit(const int32_t *touched, const int32_t *cnt_ptr, u64 *visit,
                            const u64 *fnext, MsLevels l, int32_t level, u64 *active_next) {
    const int lane = threadIdx.x & 31;
    const int32_t cnt = *cnt_ptr;
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; base < cnt;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + lane;
        int32_t v = 0;
        u64 nm = 0;
        if (i < cnt) {
            v = touched[i];
            nm = fnext[v];
            visit[v] |= nm;
        }
        ms_set_level(l, v, nm, level);
        ms_note_active(active_next, nm);
    }
}

// The end of a level: the masks of the spent frontier back to zero, and with
// them what the next levels count in.
struct MsEnd {
    const int32_t *list;  // the spent frontier
    int32_t cnt;
    u64 *f;
    int32_t *next_cnt, *next_rest;
    u64 *active;
};

__device__ __forceinline__ void ms_end(const MsEnd &z) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *z.next_cnt = 0;
        *z.next_rest = 0;
        *z.active = 0;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < z.cnt;
         i += (int64_t)gridDim.x * blockDim.x)
        z.f[z.list[i]] = 0ull;
}

__global__ void k_ms_end(MsEnd z) { ms_end(z); }

// ... and what k_ms_pull_rest found becomes visited.
__global__ void __launch_bounds__(kCta) k_ms_pull_end(MsPullArgs a, MsEnd z) {
    const int lane = threadIdx.x & 31;
    const int32_t cnt = *a.rest_cnt;
    OutCtx out = ms_out(a);
    out.q2 = nullptr;
    Stage st = stage_begin();
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; base < cnt;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + lane;
        const int32_t v = i < cnt ? a.rest[i] : 0;
        const u64 nm = i < cnt ? a.fnext[v] : 0;
        if (nm) a.visit[v] |= nm;
        ms_set_level(a.l, v, nm, a.level);
        ms_note_active(a.active_next, nm);
        const int32_t vs[1] = {v};
        const int code[1] = {nm != 0};
        emit_n<1>(out, st, vs, code);
    }
    stage_end(out, st);
    ms_end(z);
}

__global__ void k_ms_seed(const int32_t *srcs, int32_t k, u64 *visit, u64 *fcur, int32_t *depth,
                          int32_t n, int32_t *list, int32_t *cnt) {
    int i = threadIdx.x;
    if (i < k) {
        int32_t s = srcs[i];
        atomicOr(&visit[s], 1ull << i);
        u64 old = atomicOr(&fcur[s], 1ull << i);
        if (depth) depth[(int64_t)i * n + s] = 0;
        if (old == 0) list[atomicAdd(cnt, 1)] = s;
    }
}

// ------------------------------------------- multi-source BFS, fused
// The whole multi-source loop in one cooperative kernel (kernel fusion for
// the batch): per level a WM PUSH over the list of vertices whose frontier
// mask is non-zero, a grid barrier, the commit of the newly reached bits
// (visit masks, depths) together with clearing the spent frontier masks, and
// a second barrier.  Counters rotate over three words so that a level's
// count is read after the barrier that completed it and reset two levels
// ahead.
struct MsBfsFusedArgs {
    DevGraph g;
    u64 *visit;
    u64 *F[2];
    int32_t *list[2];
    int32_t *cnt;     // [3] rotating list lengths; cnt[0] = seeded sources
    int32_t *depth;   // [k][n]
    int32_t *levels;  // out
    GridBarrier bar;
    int32_t *err;
    uint64_t limit_ns;
};

__global__ void __launch_bounds__(kCta) k_ms_bfs_fused(MsBfsFusedArgs a) {
    const int32_t n = a.g.n;
    OutCtx out;
    memset(&out, 0, sizeof(out));
    out.mode = OUT_SPARSE;
    out.dedup = DD_NONE;  // the first arc that turns a mask non-zero lists the vertex
    out.cap = n;
    out.err = a.err;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nt = (int64_t)gridDim.x * blockDim.x;
    int level = 1;
    for (;; ++level) {
        const int p = (level - 1) & 1, q = level & 1;
        const int32_t size = ld_relaxed_i32(a.cnt + (level - 1) % 3);
        if (size == 0) break;
        FrontierIn fin{a.list[p], size, nullptr};
        out.q = a.list[q];
        out.cnt = a.cnt + level % 3;
        if (blockIdx.x == 0 && threadIdx.x == 0) a.cnt[(level + 1) % 3] = 0;
        lb_warp(a.g, fin, size, OpMsBfs{a.visit, a.F[p], a.F[q]}, out, blockIdx.x, gridDim.x,
                nullptr);
        if (!grid_sync(a.bar, a.err, a.limit_ns)) return;
        const int32_t nt_new = ld_relaxed_i32(a.cnt + level % 3);
        for (int64_t i = tid; i < nt_new; i += nt) {
            const int32_t v = a.list[q][i];
            u64 nm = a.F[q][v];
            a.visit[v] |= nm;
            while (nm) {
                const int b = __ffsll((long long)nm) - 1;
                nm &= nm - 1;
                a.depth[(int64_t)b * n + v] = level;
            }
        }
        for (int64_t i = tid; i < size; i += nt) a.F[p][a.list[p][i]] = 0ull;
        if (!grid_sync(a.bar, a.err, a.limit_ns)) return;
    }
    if (tid == 0) *a.levels = level - 1;
}

static g2_status batch_lb(const g2_schedule &s) {
    if (s.load_balance < G2_LB_VERTEX_BASED || s.load_balance > G2_LB_TWC)
        return fail(G2_EINVAL, "bad load_balance");
    if (s.load_balance == G2_LB_EDGE_ONLY)
        return fail(G2_EUNSUPPORTED, "multi-source traversals are frontier-driven (no EDGE_ONLY)");
    if (s.direction == G2_PULL && s.load_balance != G2_LB_VERTEX_BASED &&
        s.load_balance != G2_LB_WM)
        return fail(G2_EUNSUPPORTED, "multi-source PULL supports VERTEX_BASED and WM");
    return G2_OK;
}

static g2_status bfs_batch_fused(g2_graph *g, const int32_t *srcs, int32_t k, int32_t *depth,
                                 const g2_schedule &sc, cudaStream_t st, int32_t *d_err) {
    if (sc.direction != G2_PUSH || sc.load_balance != G2_LB_WM)
        return fail(G2_EUNSUPPORTED, "the fused multi-source BFS runs WM PUSH rounds");
    Topology *t = g->topo;
    const int32_t n = t->n;
    int32_t *ctrs = d_err - 62;
    MsBfsFusedArgs a;
    a.g = t->view();
    int32_t *dsrc;
    G2_TRY(ws(g, B_MS0, (size_t)std::max(n, 1), &a.visit));
    G2_TRY(ws(g, B_MS1, (size_t)std::max(n, 1), &a.F[0]));
    G2_TRY(ws(g, B_MS2, (size_t)std::max(n, 1), &a.F[1]));
    G2_TRY(ws(g, B_Q0, (size_t)std::max(n, 1), &a.list[0]));
    G2_TRY(ws(g, B_Q1, (size_t)std::max(n, 1), &a.list[1]));
    G2_TRY(ws(g, B_I1, 64, &dsrc));
    G2_CK(cudaMemsetAsync(a.visit, 0, (size_t)n * 8, st));
    G2_CK(cudaMemsetAsync(a.F[0], 0, (size_t)n * 8, st));
    G2_CK(cudaMemsetAsync(a.F[1], 0, (size_t)n * 8, st));
    G2_CK(cudaMemsetAsync(depth, 0xFF, (size_t)k * n * 4, st));
    G2_TRY(put_array(dsrc, srcs, k, st));
    a.cnt = ctrs + 20;  // [20..22]; zero from begin_call
    a.levels = ctrs + 24;
    k_ms_seed<<<1, 64, 0, st>>>(dsrc, k, a.visit, a.F[0], depth, n, a.list[0], a.cnt);
    a.depth = depth;
    a.bar = GridBarrier{reinterpret_cast<unsigned long long *>(ctrs + 28)};
    a.err = d_err;
    a.limit_ns = barrier_limit_ns();
    stats().launches += 1;
    G2_TRY(launch_coop(g, k_ms_bfs_fused, a, st));
    G2_TRY(read_counters(g, ctrs + 24, 1, st, d_err));
    stats().iterations = g->h_ctr[0];
    stats().push_rounds = g->h_ctr[0];
    stats().barriers = 2 * g->h_ctr[0];
    return G2_OK;
}

g2_status bfs_batch_run(g2_graph *g, const int32_t *srcs, int32_t k, int32_t *depth,
                        const g2_hybrid &h, cudaStream_t st, int32_t *d_err) {
    if (h.s1.kernel_fusion) {
        if (h.criteria != G2_CRITERIA_NONE && !h.s2.kernel_fusion)
            return fail(G2_EUNSUPPORTED, "kernel fusion must be set on both hybrid schedules");
        return bfs_batch_fused(g, srcs, k, depth, h.s1, st, d_err);
    }
    Topology *t = g->topo;
    const int32_t n = t->n;
    int32_t *ctrs = d_err - 62;
    u64 *visit, *F[2];
    int32_t *list[2], *dsrc;
    G2_TRY(ws(g, B_MS0, (size_t)std::max(n, 1), &visit));
    G2_TRY(ws(g, B_MS1, (size_t)std::max(n, 1), &F[0]));
    G2_TRY(ws(g, B_MS2, (size_t)std::max(n, 1), &F[1]));
    G2_TRY(ws(g, B_Q0, (size_t)std::max(n, 1), &list[0]));
    G2_TRY(ws(g, B_Q1, (size_t)std::max(n, 1), &list[1]));
    G2_TRY(ws(g, B_I1, 64, &dsrc));
    G2_CK(cudaMemsetAsync(visit, 0, (size_t)n * 8, st));
    G2_CK(cudaMemsetAsync(F[0], 0, (size_t)n * 8, st));
    G2_CK(cudaMemsetAsync(F[1], 0, (size_t)n * 8, st));
    MsLevels lv;
    u64 *planes = nullptr;
    if (k > kMsDirect) {
        const g2_status room = ws(g, B_ROWS, (size_t)kMsPlanes * std::max(n, 1), &planes);
        if (room != G2_ENOMEM) G2_TRY(room);
    }
    for (int j = 0; j < kMsPlanes; ++j) lv.plane[j] = planes + (size_t)j * n;
    lv.depth = planes ? nullptr : depth;
    if (lv.depth) G2_CK(cudaMemsetAsync(depth, 0xFF, (size_t)k * n * 4, st));
    lv.n = n;
    int nplanes = 0;  // cleared so far
    G2_TRY(put_array(dsrc, srcs, k, st));
    // ctrs: [0..1] list lengths, [2] big vertices, [3..4] a pull's rest by level parity, [8..11]
    // active masks of the even and odd levels (all zero at the start of the call)
    u64 *active[2] = {reinterpret_cast<u64 *>(ctrs + 8), reinterpret_cast<u64 *>(ctrs + 10)};
    k_ms_seed<<<1, 64, 0, st>>>(dsrc, k, visit, F[0], lv.depth, n, list[0], ctrs + 0);
    const u64 full = k == 64 ? ~0ull : ((1ull << k) - 1);
    G2_TRY(put_i32(st, {{ctrs + 8, (int32_t)(uint32_t)full}, {ctrs + 9, (int32_t)(uint32_t)(full >> 32)}}));
    stats().launches += 1;
    // PULL: the vertices whose lists go to the grid in pieces
    int32_t *big = nullptr, *piece = nullptr, *rest = nullptr;
    int32_t nbig = 0;
    const bool pulls = h.s1.direction == G2_PULL ||
                       (h.criteria == G2_INPUT_VERTEXSET_SIZE && h.s2.direction == G2_PULL);
    bool long_lists = true;  // in-lists that a thread leaves to a warp
    if (pulls) {
        if (t->symmetric) {
            int32_t dmax = 0;
            G2_TRY(max_out_degree(g, st, &dmax));
            long_lists = dmax > kMsAlone;
        }
        int32_t *np;
        const size_t room = (size_t)t->m / kMsPiece + 1;  // vertices of kMsPiece arcs or more
        G2_TRY(ws(g, B_F0, room, &big));
        G2_TRY(ws(g, B_F1, room, &np));
        k_ms_big<<<grid_for(g, n, kCta), kCta, 0, st>>>(t->crowptr, n, kMsPiece, big, np, ctrs + 2);
        stats().launches += 1;
        G2_TRY(read_counters(g, ctrs, 4, st, d_err));
        nbig = g->h_ctr[2];
        G2_TRY(ws(g, B_F2, (size_t)std::max(n, 1), &rest));
        if (nbig > 0) {
            G2_TRY(ws(g, B_LVL, (size_t)nbig + 1, &piece));
            G2_TRY(exclusive_scan_i32(g, np, piece, nbig, st));
        }
    } else {
        G2_TRY(read_counters(g, ctrs, 4, st, d_err));
    }
    int32_t size = g->h_ctr[0];
    unsigned long long *ctr = nullptr;
    if (count_arcs_enabled()) G2_TRY(ws(g, B_ARCS, 2, &ctr));
    int p = 0;
    for (int level = 1; size > 0; ++level) {
        const g2_schedule &s = pick_schedule(h, size, n);
        G2_TRY(batch_lb(s));
        int q = 1 - p;
        u64 *act = active[(level - 1) & 1], *act_next = active[level & 1];
        int32_t *rest_cnt = ctrs + 3 + (level & 1);
        // (the masks of the level's frontier become the all-zero array of the
        // level after the next)
        const MsEnd end{list[p], size, F[p], ctrs + p, ctrs + 3 + (1 - (level & 1)), act};
        if (!lv.depth && level == 1 << nplanes) {
            if (nplanes < kMsPlanes) {
                G2_CK(cudaMemsetAsync(lv.plane[nplanes++], 0, (size_t)n * 8, st));
            } else {
                k_ms_out<<<grid_for(g, n, kCta), kCta, 0, st>>>(lv, visit, nplanes, k, depth);
                stats().launches += 1;
                lv.depth = depth;
            }
        }
        if (s.direction == G2_PUSH) {
            OutCtx out;
            memset(&out, 0, sizeof(out));
            out.mode = OUT_SPARSE;
            out.q = list[q];
            out.cnt = ctrs + q;
            out.cap = n;
            out.err = d_err;
            VSet in{OUT_SPARSE, list[p], n, ctrs + p, nullptr, nullptr, size};
            G2_TRY(push_round(g, s, OpMsBfs{visit, F[p], F[q]}, in, out, ctr, st));
            k_ms_commit<<<t->sm_count * 8, kCta, 0, st>>>(list[q], ctrs + q, visit, F[q], lv, level,
                                                        act_next);
            k_ms_end<<<grid_for(g, size, kCta), kCta, 0, st>>>(end);
            stats().push_rounds++;
            stats().launches += 2;
        } else {
            // (the schedule's VERTEX_BASED and WM run the same kernels)
            MsPullArgs a{t->view(), visit, F[p], F[q], act, act_next, lv, level, list[q], ctrs + q, rest,
                         rest_cnt, long_lists ? kMsThread : kMsAlone, d_err, ctr};
            if (nbig > 0) {
                k_ms_pull_pieces<<<grid_for(g, (int64_t)t->m / kMsPiece + nbig, 1), kCta, 0, st>>>(
                    a, big, nbig, piece);
                stats().launches += 1;
            }
            k_ms_pull<<<grid_for(g, n, kCta), kCta, 0, st>>>(a);
            if (long_lists) {
                k_ms_pull_rest<<<t->sm_count * 16, kCta, 0, st>>>(a);
                k_ms_pull_end<<<std::max(t->sm_count * 8, grid_for(g, size, kCta)), kCta, 0, st>>>(a, end);
                stats().launches += 1;
            } else {
                k_ms_end<<<grid_for(g, size, kCta), kCta, 0, st>>>(end);
            }
            G2_CK(cudaGetLastError());
            stats().pull_rounds++;
            stats().launches += 2;
        }
        G2_TRY(read_counters(g, ctrs, 4, st, d_err));
        size = g->h_ctr[q];
        p = q;
        stats().iterations++;
    }
    if (!lv.depth) {
        k_ms_out<<<grid_for(g, n, kCta), kCta, 0, st>>>(lv, visit, nplanes, k, depth);
        stats().launches += 1;
        G2_CK(cudaGetLastError());
    }
    return G2_OK;
}

// ------------------------------------------------------ multi-source SSSP
// Masks: M[p][v] = sources whose dist at v improved below the bucket
// threshold and wait to be relaxed; Far[v] = sources improved to a value at
// or above it.  Lists hold each vertex once (the first arc that turns its
// mask non-zero lists it).
struct OpMsRelax {
    int32_t *dist;  // [k][n]
    const int32_t *w;
    const unsigned *mcur;
    unsigned *mnext;
    unsigned *far;
    int32_t n;
    int32_t T;
    int32_t *err;
    typedef unsigned S;
    typedef int32_t Pre;
    typedef int Old;
    static constexpr int kFlight = 1;  // a loop over the mask's bits per arc
    __device__ __forceinline__ S load(int32_t u) const { return mcur[u]; }
    __device__ __forceinline__ bool skip(S m) const { return m == 0; }
    __device__ __forceinline__ Pre pre(int32_t, int32_t) const { return 0; }
    __device__ __forceinline__ int fin(int32_t, S, int32_t, Pre, Old code) const { return code; }
    __device__ __forceinline__ Old act(int32_t u, S mu, int32_t v, int32_t e, Pre) const {
        const int32_t wt = w[e];
        unsigned nb = 0, fb = 0;
        while (mu) {
            int i = __ffs(mu) - 1;
            mu &= mu - 1;
            int32_t du = dist[(int64_t)i * n + u];
            int64_t nd = (int64_t)du + wt;
            if (nd >= G2_INF32) {
                set_error(err, G2_EOVERFLOW);
                continue;
            }
            int32_t *dv = dist + (int64_t)i * n + v;
            if ((int32_t)nd < *dv) {
                int32_t old = atomicMin(dv, (int32_t)nd);
                if ((int32_t)nd < old) {
                    if ((int32_t)nd < T) nb |= 1u << i;
                    else fb |= 1u << i;
                }
            }
        }
        int code = 0;
        if (nb && atomicOr(&mnext[v], nb) == 0) code |= 1;
        if (fb && atomicOr(&far[v], fb) == 0) code |= 2;
        return code;
    }
};

__global__ void k_msr_far_min(const int32_t *flist, int32_t cnt, const unsigned *far,
                              const int32_t *dist, int32_t n, int32_t Told, int32_t *out) {
    int32_t best = G2_INF32;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t v = flist[i];
        unsigned m = far[v];
        while (m) {
            int b = __ffs(m) - 1;
            m &= m - 1;
            int32_t d = dist[(int64_t)b * n + v];
            if (d >= Told && d < best) best = d;
        }
    }
    best = (int32_t)__reduce_min_sync(G2_FULL, (unsigned)best);
    if ((threadIdx.x & 31) == 0 && best != G2_INF32) atomicMin(out, best);
}

__global__ void k_msr_far_split(const int32_t *flist, int32_t cnt, unsigned *far,
                                const int32_t *dist, int32_t n, int32_t Told, int32_t Tnew,
                                unsigned *mnear, int32_t *nlist, int32_t *ncnt, int32_t *flist2,
                                int32_t *fcnt2, int32_t *err) {
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; base < cnt;
         base += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = base + (threadIdx.x & 31);
        int32_t v = 0;
        unsigned nb = 0, fb = 0;
        if (i < cnt) {
            v = flist[i];
            unsigned m = far[v];
            while (m) {
                int b = __ffs(m) - 1;
                m &= m - 1;
                int32_t d = dist[(int64_t)b * n + v];
                if (d < Told) continue;  // settled in an earlier bucket
                if (d < Tnew) nb |= 1u << b;
                else fb |= 1u << b;
            }
            far[v] = fb;
            if (nb) mnear[v] = nb;
        }
        warp_append(nlist, ncnt, n, err, v, nb != 0);
        warp_append(flist2, fcnt2, n, err, v, fb != 0);
    }
}

// ------------------------------------------ multi-source SSSP, fused
// The near/far loop of the multi-source relaxation in one cooperative kernel.
// Near round r pushes from list NL[r % 3] with masks M[r % 3] into
// NL[(r + 1) % 3] / M[(r + 1) % 3] (and the far pile), while the masks of
// round r - 1's input (M[(r + 2) % 3], listed in NL[(r + 2) % 3]) are
// cleared: three rotating buffers make one grid barrier per round enough.
// When a round produces nothing, the smallest far distance at or above the
// threshold picks the next bucket and the far pile is split as in the plain
// loop (two barriers per bucket).
struct MsSsspFusedArgs {
    DevGraph g;
    int32_t *dist;  // [k][n]
    unsigned *M[3];
    unsigned *far;
    int32_t *NL[3];
    int32_t *FL[2];
    int32_t *ncnt;    // [3]; ncnt[0] = seeded sources
    int32_t *fcnt;    // [2]
    int32_t *dmin;    // [2]; dmin[0] = G2_INF32 at launch
    int32_t *result;  // [0] near rounds, [1] buckets
    int32_t delta;    // 0: one bucket
    GridBarrier bar;
    int32_t *err;
    uint64_t limit_ns;
};

__global__ void __launch_bounds__(kCta) k_msr_fused(MsSsspFusedArgs a) {
    const int32_t n = a.g.n;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nt = (int64_t)gridDim.x * blockDim.x;
    const bool bucketed = a.delta > 0;
    int64_t T = bucketed ? a.delta : (int64_t)G2_INF32;
    int r = 0, fp = 0, epoch = 0;
    int32_t prev_size = 0;
    OutCtx out;
    memset(&out, 0, sizeof(out));
    out.mode = OUT_SPARSE;
    out.dedup = DD_NONE;  // a vertex is listed when its mask turns non-zero
    out.cap = n;
    out.cap2 = n;
    out.err = a.err;
    for (;;) {
        for (;;) {
            const int ia = r % 3, ib = (r + 1) % 3, ic = (r + 2) % 3;
            const int32_t size = ld_relaxed_i32(a.ncnt + ia);
            if (size == 0) break;
            out.q = a.NL[ib];
            out.cnt = a.ncnt + ib;
            out.q2 = a.FL[fp];
            out.cnt2 = a.fcnt + fp;
            if (tid == 0) a.ncnt[ic] = 0;  // round r + 1's output count
            for (int64_t i = tid; i < prev_size; i += nt) a.M[ic][a.NL[ic][i]] = 0u;
            FrontierIn fin{a.NL[ia], size, nullptr};
            OpMsRelax op{a.dist, a.g.w, a.M[ia], a.M[ib], a.far, n,
                         (int32_t)(T < G2_INF32 ? T : G2_INF32), a.err};
            lb_warp(a.g, fin, size, op, out, blockIdx.x, gridDim.x, nullptr);
            if (!grid_sync(a.bar, a.err, a.limit_ns)) return;
            prev_size = size;
            ++r;
        }
        const int32_t nfar = ld_relaxed_i32(a.fcnt + fp);
        if (!bucketed || nfar == 0) break;
        const int32_t Told = (int32_t)(T < G2_INF32 ? T : G2_INF32);
        // phase A: the smallest live far distance
        {
            int32_t best = G2_INF32;
            for (int64_t i = tid; i < nfar; i += nt) {
                const int32_t v = a.FL[fp][i];
                unsigned m = a.far[v];
                while (m) {
                    const int b = __ffs(m) - 1;
                    m &= m - 1;
                    const int32_t d = a.dist[(int64_t)b * n + v];
                    if (d >= Told && d < best) best = d;
                }
            }
            best = (int32_t)__reduce_min_sync(G2_FULL, (unsigned)best);
            if ((threadIdx.x & 31) == 0 && best != G2_INF32) atomicMin(a.dmin + (epoch & 1), best);
            if (tid == 0) {
                a.fcnt[1 - fp] = 0;                 // the far pile of the next epoch
                a.dmin[(epoch + 1) & 1] = G2_INF32;  // its minimum
            }
        }
        if (!grid_sync(a.bar, a.err, a.limit_ns)) return;
        const int32_t dmin = ld_relaxed_i32(a.dmin + (epoch & 1));
        if (dmin == G2_INF32) break;
        const int64_t Tnew = ((int64_t)dmin / a.delta + 1) * (int64_t)a.delta;
        const int32_t Tn = (int32_t)(Tnew < G2_INF32 ? Tnew : G2_INF32);
        // phase B: split the far pile into round r's near list and the next pile
        {
            const int ia = r % 3;
            for (int64_t base = tid & ~31LL; base < nfar; base += nt) {
                const int64_t i = base + (threadIdx.x & 31);
                int32_t v = 0;
                unsigned nb = 0, fb = 0;
                if (i < nfar) {
                    v = a.FL[fp][i];
                    unsigned m = a.far[v];
                    while (m) {
                        const int b = __ffs(m) - 1;
                        m &= m - 1;
                        const int32_t d = a.dist[(int64_t)b * n + v];
                        if (d < Told) continue;  // settled in an earlier bucket
                        if (d < Tn) nb |= 1u << b;
                        else fb |= 1u << b;
                    }
                    a.far[v] = fb;
                    if (nb) a.M[ia][v] = nb;
                }
                warp_append(a.NL[ia], a.ncnt + ia, n, a.err, v, nb != 0);
                warp_append(a.FL[1 - fp], a.fcnt + 1 - fp, n, a.err, v, fb != 0);
            }
        }
        if (!grid_sync(a.bar, a.err, a.limit_ns)) return;
        fp = 1 - fp;
        T = Tnew;
        ++epoch;
    }
    if (tid == 0) {
        a.result[0] = r;
        a.result[1] = epoch;
    }
}

__global__ void k_msr_seed(const int32_t *srcs, int32_t k, int32_t *dist, int32_t n, unsigned *m,
                           int32_t *list, int32_t *cnt) {
    int i = threadIdx.x;
    if (i < k) {
        int32_t s = srcs[i];
        dist[(int64_t)i * n + s] = 0;
        if (atomicOr(&m[s], 1u << i) == 0) list[atomicAdd(cnt, 1)] = s;
    }
}

// Going on from distance rows: every flagged vertex waits with each source that
// has reached it (which of them changed last is not known).
__global__ void k_msr_resume(const uint32_t *flags, int32_t words, const int32_t *dist, int32_t n,
                             int32_t k, unsigned *mask, int32_t *list, int32_t *cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = gw; i < words; i += nw) {
        const uint32_t x = flags[i];
        if (x == 0) continue;
        const int64_t v = i * 32 + lane;
        const bool on = (x >> lane) & 1u;
        unsigned m = 0;
        if (on)
            for (int32_t b = 0; b < k; ++b)
                if (dist[(int64_t)b * n + v] != G2_INF32) m |= 1u << b;
        int base = 0;
        if (lane == 0) base = atomicAdd(cnt, __popc(x));
        base = __shfl_sync(G2_FULL, base, 0);
        if (on) {
            mask[v] = m;
            list[base + __popc(x & lanemask_lt())] = (int32_t)v;
        }
    }
}

__global__ void k_msr_clear(const int32_t *list, int32_t cnt, unsigned *m) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (int64_t)gridDim.x * blockDim.x)
        m[list[i]] = 0u;
}

__global__ void k_fill_i32_b(int32_t *a, int64_t n, int32_t val) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        a[v] = val;
}

static g2_status sssp_batch_fused(g2_graph *g, const int32_t *srcs, int32_t k, int32_t delta,
                                  int32_t *dist, const g2_schedule &sc, cudaStream_t st,
                                  int32_t *d_err) {
    if (sc.direction != G2_PUSH || sc.load_balance != G2_LB_WM)
        return fail(G2_EUNSUPPORTED, "the fused multi-source SSSP runs WM PUSH rounds");
    Topology *t = g->topo;
    const int32_t n = t->n;
    int32_t *ctrs = d_err - 62;
    MsSsspFusedArgs a;
    a.g = t->view();
    a.dist = dist;
    int32_t *dsrc;
    int32_t *m2;
    G2_TRY(ws(g, B_F0, (size_t)std::max(n, 1), &a.M[0]));
    G2_TRY(ws(g, B_F1, (size_t)std::max(n, 1), &a.M[1]));
    G2_TRY(ws(g, B_STAMP, (size_t)std::max(n, 1), &m2));
    a.M[2] = reinterpret_cast<unsigned *>(m2);
    G2_TRY(ws(g, B_F2, (size_t)std::max(n, 1), &a.far));
    G2_TRY(ws(g, B_Q0, (size_t)std::max(n, 1), &a.NL[0]));
    G2_TRY(ws(g, B_Q1, (size_t)std::max(n, 1), &a.NL[1]));
    G2_TRY(ws(g, B_Q2, (size_t)std::max(n, 1), &a.NL[2]));
    G2_TRY(ws(g, B_Q3, (size_t)std::max(n, 1), &a.FL[0]));
    G2_TRY(ws(g, B_STAMP2, (size_t)std::max(n, 1), &a.FL[1]));
    G2_TRY(ws(g, B_I1, 64, &dsrc));
    for (int i = 0; i < 3; ++i) G2_CK(cudaMemsetAsync(a.M[i], 0, (size_t)n * 4, st));
    G2_CK(cudaMemsetAsync(a.far, 0, (size_t)n * 4, st));
    k_fill_i32_b<<<grid_for(g, (int64_t)k * n, kCta), kCta, 0, st>>>(dist, (int64_t)k * n, G2_INF32);
    G2_TRY(put_array(dsrc, srcs, k, st));
    a.ncnt = ctrs + 36;   // [36..38], zero from begin_call
    a.fcnt = ctrs + 39;   // [39..40]
    a.dmin = ctrs + 41;   // [41..42]
    a.result = ctrs + 43; // [43..44]
    const int32_t inf = G2_INF32;
    G2_TRY(put_i32(st, {{a.dmin, inf}}));
    k_msr_seed<<<1, 32, 0, st>>>(dsrc, k, dist, n, a.M[0], a.NL[0], a.ncnt);
    a.delta = delta;
    a.bar = GridBarrier{reinterpret_cast<unsigned long long *>(ctrs + 28)};
    a.err = d_err;
    a.limit_ns = barrier_limit_ns();
    stats().launches += 2;
    G2_TRY(launch_coop(g, k_msr_fused, a, st));
    G2_TRY(read_counters(g, ctrs + 43, 2, st, d_err));
    stats().iterations = g->h_ctr[0];
    stats().push_rounds = g->h_ctr[0];
    stats().barriers = g->h_ctr[0] + 2 * g->h_ctr[1];
    return G2_OK;
}

// `left` (may be null): dist holds distances already, and the arcs of the
// vertices flagged there are still to be relaxed.
g2_status sssp_batch_run(g2_graph *g, const int32_t *srcs, int32_t k, int32_t delta, int32_t *dist,
                         const g2_hybrid &h, const uint32_t *left, cudaStream_t st,
                         int32_t *d_err) {
    if (h.s1.kernel_fusion) {
        if (h.criteria != G2_CRITERIA_NONE && !h.s2.kernel_fusion)
            return fail(G2_EUNSUPPORTED, "kernel fusion must be set on both hybrid schedules");
        return sssp_batch_fused(g, srcs, k, delta, dist, h.s1, st, d_err);
    }
    Topology *t = g->topo;
    const int32_t n = t->n;
    int32_t *ctrs = d_err - 62;
    unsigned *M[2], *far;
    int32_t *nl[2], *fl[2], *dsrc;
    G2_TRY(ws(g, B_F0, (size_t)std::max(n, 1), &M[0]));
    G2_TRY(ws(g, B_F1, (size_t)std::max(n, 1), &M[1]));
    G2_TRY(ws(g, B_F2, (size_t)std::max(n, 1), &far));
    G2_TRY(ws(g, B_Q0, (size_t)std::max(n, 1), &nl[0]));
    G2_TRY(ws(g, B_Q1, (size_t)std::max(n, 1), &nl[1]));
    G2_TRY(ws(g, B_Q2, (size_t)std::max(n, 1), &fl[0]));
    G2_TRY(ws(g, B_Q3, (size_t)std::max(n, 1), &fl[1]));
    G2_TRY(ws(g, B_I1, 64, &dsrc));
    G2_CK(cudaMemsetAsync(M[0], 0, (size_t)n * 4, st));
    G2_CK(cudaMemsetAsync(M[1], 0, (size_t)n * 4, st));
    G2_CK(cudaMemsetAsync(far, 0, (size_t)n * 4, st));
    const bool bucketed = delta > 0;
    int64_t T = bucketed ? delta : (int64_t)G2_INF32;
    // (all counters are zero here)
    if (left) {
        // no bucket is settled yet: what waits is the far pile, to be split at
        // the first threshold
        const int32_t words = (n + 31) / 32;
        if (bucketed) T = 0;
        k_msr_resume<<<grid_for(g, words, kWarps), kCta, 0, st>>>(
            left, words, dist, n, k, bucketed ? far : M[0], bucketed ? fl[0] : nl[0],
            bucketed ? ctrs + 4 : ctrs);
        stats().launches += 1;
    } else {
        k_fill_i32_b<<<grid_for(g, (int64_t)k * n, kCta), kCta, 0, st>>>(dist, (int64_t)k * n,
                                                                       G2_INF32);
        G2_TRY(put_array(dsrc, srcs, k, st));
        k_msr_seed<<<1, 32, 0, st>>>(dsrc, k, dist, n, M[0], nl[0], ctrs + 0);
        stats().launches += 2;
    }
    G2_TRY(read_counters(g, ctrs, 8, st, d_err));
    int32_t size = g->h_ctr[0];
    unsigned long long *ctr = nullptr;
    if (count_arcs_enabled()) G2_TRY(ws(g, B_ARCS, 2, &ctr));
    int p = 0, fp = 0;
    for (;;) {
        while (size > 0) {
            const g2_schedule &s = pick_schedule(h, size, n);
            G2_TRY(batch_lb(s));
            if (s.direction != G2_PUSH)
                return fail(G2_EUNSUPPORTED, "multi-source SSSP relaxes in the PUSH direction");
            int q = 1 - p;
            OutCtx out;
            memset(&out, 0, sizeof(out));
            out.mode = OUT_SPARSE;
            out.q = nl[q];
            out.cnt = ctrs + q;
            out.cap = n;
            out.q2 = fl[fp];
            out.cnt2 = ctrs + 4 + fp;
            out.cap2 = n;
            out.err = d_err;
            G2_CK(cudaMemsetAsync(ctrs + q, 0, 4, st));
            VSet in{OUT_SPARSE, nl[p], n, ctrs + p, nullptr, nullptr, size};
            // distances that rows left may still fall: the overflow rule is
            // applied to the final ones (sssp_batch_check)
            OpMsRelax op{dist, t->w, M[p], M[q], far, n, (int32_t)std::min<int64_t>(T, G2_INF32),
                         left ? nullptr : d_err};
            G2_TRY(push_round(g, s, op, in, out, ctr, st));
            k_msr_clear<<<grid_for(g, size, kCta), kCta, 0, st>>>(nl[p], size, M[p]);
            stats().launches += 2;
            stats().push_rounds++;
            stats().iterations++;
            G2_TRY(read_counters(g, ctrs, 8, st, d_err));
            size = g->h_ctr[q];
            p = q;
        }
        int32_t nfar = g->h_ctr[4 + fp];
        if (!bucketed || nfar == 0) break;
        int32_t Told = (int32_t)std::min<int64_t>(T, G2_INF32);
        int32_t inf = G2_INF32;
        G2_TRY(put_i32(st, {{ctrs + 6, inf}}));
        k_msr_far_min<<<grid_for(g, nfar, kCta), kCta, 0, st>>>(fl[fp], nfar, far, dist, n, Told,
                                                               ctrs + 6);
        G2_TRY(read_counters(g, ctrs, 8, st, d_err));
        int32_t dmin = g->h_ctr[6];
        if (dmin == G2_INF32) break;
        int64_t Tnew = ((int64_t)dmin / delta + 1) * (int64_t)delta;
        int nf = 1 - fp;
        G2_CK(cudaMemsetAsync(ctrs + p, 0, 4, st));
        G2_CK(cudaMemsetAsync(ctrs + 4 + nf, 0, 4, st));
        k_msr_far_split<<<grid_for(g, nfar, kCta), kCta, 0, st>>>(
            fl[fp], nfar, far, dist, n, Told, (int32_t)std::min<int64_t>(Tnew, G2_INF32), M[p],
            nl[p], ctrs + p, fl[nf], ctrs + 4 + nf, d_err);
        stats().launches += 2;
        G2_TRY(read_counters(g, ctrs, 8, st, d_err));
        size = g->h_ctr[p];
        fp = nf;
        T = Tnew;
        stats().barriers++;
    }
    return G2_OK;
}

}  // namespace g2

using namespace g2;

// Tuned schedules when the caller passes none: multi-source BFS switches from
// STRICT PUSH to VERTEX_BASED PULL once the union frontier holds 2% of the
// vertices; multi-source SSSP relaxes distance rows.
// Tuned multi-source BFS: the direction-optimising hybrid (STRICT PUSH below
// 2% of n, VERTEX_BASED PULL); on a bounded-degree graph the fused WM PUSH
// loop (thousands of small levels: launches and host round trips dominate).
static g2_hybrid tuned_batch_bfs(g2_graph *g, cudaStream_t st) {
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
    return h;
}

// Tuned multi-source SSSP: distance rows (g2_rows.cu; the STRICT PUSH below is
// its stand-in where the rows do not apply); the fused WM PUSH loop
// on a bounded-degree graph.
static g2_hybrid tuned_batch_sssp(g2_graph *g, cudaStream_t st) {
    int32_t dmax = 0;
    if (max_out_degree(g, st, &dmax) == G2_OK && dmax <= kBoundedDegree) {
        g2_hybrid h = default_hybrid();
        h.s1.load_balance = G2_LB_WM;
        h.s1.kernel_fusion = 1;
        h.s2 = h.s1;
        return h;
    }
    g2_hybrid h = default_hybrid();
    h.s1.load_balance = G2_LB_STRICT;
    return h;
}

extern "C" {

g2_status g2_bfs_batch(g2_graph *g, const int32_t *srcs, int32_t k, int32_t *depth,
                       const g2_hybrid *sched, void *stream);
g2_status g2_sssp_batch(g2_graph *g, const int32_t *srcs, int32_t k, int32_t delta, int32_t *dist,
                        const g2_hybrid *sched, void *stream);

}  // extern "C"

namespace g2 {

// Split mode for the NULL schedule on a bounded-degree graph: the sources run
// as single-source fused queries, `workers` at a time, each on a view of the
// graph (its own workspace) and a stream of its own, driven by a host thread.
// A single-source fused loop keeps most levels of a road graph inside one
// 16-CTA thread-block cluster, so about nine of them fit on the GPU at once;
// on the 4096^2 road grid 64 BFS sources take 156-166 ms this way against 286
// ms in one multi-source traversal (whose 64 wavefronts rarely meet, so it does
// the same vertex work with wider masks), and 32 SSSP sources 291 ms against
// 376 ms.  Outputs are row i of the caller's k x n array, as in the batched
// traversal.
static int split_workers(g2_graph *g, int32_t k, int per_sm_default) {
    int w = std::max(1, g->topo->sm_count / per_sm_default);
    if (const char *e = getenv("G2_BATCH_SPLIT_WORKERS")) w = atoi(e);
    return std::min(w, (int)k);
}

static g2_status split_run(g2_graph *g, const int32_t *srcs, int32_t k, int32_t delta, int32_t *out,
                           int workers, cudaStream_t st) {
    Topology *t = g->topo;
    const int64_t n = t->n;
    G2_CK(cudaStreamSynchronize(st));  // the caller's earlier work on its stream comes first
    std::vector<g2_graph *> views(workers, nullptr);
    std::vector<cudaStream_t> streams(workers, nullptr);
    g2_status made = G2_OK;
    for (int i = 0; i < workers && made == G2_OK; ++i) {
        made = g2_graph_view(g, &views[i]);
        if (made == G2_OK && cudaStreamCreateWithFlags(&streams[i], cudaStreamNonBlocking) != cudaSuccess)
            made = fail(G2_ECUDA, "stream for a split batch");
    }
    struct Res {
        g2_status s = G2_OK;
        std::string msg;
        int64_t launches = 0, iterations = 0, barriers = 0;
    };
    std::vector<Res> res(workers);
    if (made == G2_OK) {
        const int dev = t->device;
        std::vector<std::thread> th;
        for (int w = 0; w < workers; ++w)
            th.emplace_back([&, w]() {
                cudaSetDevice(dev);
                for (int32_t i = w; i < k && res[w].s == G2_OK; i += workers) {
                    g2_status r = delta > 0
                                      ? g2_sssp_delta(views[w], srcs[i], delta, out + i * n, nullptr,
                                                      streams[w])
                                      : g2_bfs(views[w], srcs[i], out + i * n, nullptr, nullptr,
                                               streams[w]);
                    g2_stats st_w;
                    g2_last_stats(&st_w);
                    res[w].launches += st_w.launches;
                    res[w].iterations += st_w.iterations;
                    res[w].barriers += st_w.barriers;
                    if (r != G2_OK) {
                        res[w].s = r;
                        res[w].msg = g2_last_error();
                    }
                }
            });
        for (auto &x : th) x.join();
    }
    for (int i = 0; i < workers; ++i) {
        if (streams[i]) cudaStreamDestroy(streams[i]);
        if (views[i]) g2_free_graph(views[i]);
    }
    G2_TRY(made);
    for (const Res &r : res) {
        stats().launches += (int32_t)r.launches;
        stats().iterations += (int32_t)r.iterations;
        stats().barriers += (int32_t)r.barriers;
    }
    for (const Res &r : res)
        if (r.s != G2_OK) return fail(r.s, "split batch: " + r.msg);
    return G2_OK;
}

}  // namespace g2

extern "C" {

g2_status g2_bfs_batch(g2_graph *g, const int32_t *srcs, int32_t k, int32_t *depth,
                       const g2_hybrid *sched, void *stream) {
    if (!g || !depth || !srcs || k < 1 || k > 64) return fail(G2_EINVAL, "need 1 <= k <= 64 sources");
    for (int32_t i = 0; i < k; ++i)
        if (srcs[i] < 0 || srcs[i] >= g->topo->n) return fail(G2_EINVAL, "source out of range");
    if ((int64_t)k * g->topo->n >= (int64_t)1 << 40) return fail(G2_EINVAL, "output too large");
    cudaStream_t st = as_stream(stream);
    g2_hybrid h = sched ? *sched : tuned_batch_bfs(g, st);
    int32_t *d_err;
    G2_TRY(begin_call(g, st, &d_err));
    if (!sched && h.s1.kernel_fusion && k >= 2) {
        const int workers = split_workers(g, k, 12);
        if (workers >= 2) {
            G2_TRY(split_run(g, srcs, k, 0, depth, workers, st));
            return end_call(g, st, d_err);
        }
    }
    G2_TRY(bfs_batch_run(g, srcs, k, depth, h, st, d_err));
    return end_call(g, st, d_err);
}

g2_status g2_sssp_batch(g2_graph *g, const int32_t *srcs, int32_t k, int32_t delta, int32_t *dist,
                        const g2_hybrid *sched, void *stream) {
    if (!g || !dist || !srcs || k < 1 || k > 32) return fail(G2_EINVAL, "need 1 <= k <= 32 sources");
    if (!g->topo->w) return fail(G2_EINVAL, "SSSP needs arc weights");
    for (int32_t i = 0; i < k; ++i)
        if (srcs[i] < 0 || srcs[i] >= g->topo->n) return fail(G2_EINVAL, "source out of range");
    cudaStream_t st = as_stream(stream);
    g2_hybrid h = sched ? *sched : tuned_batch_sssp(g, st);
    if (delta <= 0 && h.s1.delta > 0) delta = h.s1.delta;
    int32_t *d_err;
    G2_TRY(begin_call(g, st, &d_err));
    if (!sched && h.s1.kernel_fusion && k >= 2) {
        const int workers = split_workers(g, k, 19);
        if (workers >= 2) {
            G2_TRY(split_run(g, srcs, k, delta > 0 ? delta : 1, dist, workers, st));
            return end_call(g, st, d_err);
        }
    }
    if (!sched && !h.s1.kernel_fusion) {
        // rows of distances (RMAT-21, 32 sources: 8.3 ms against 33.8 ms for
        // STRICT delta-stepping over stacked arrays)
        int how;
        const uint32_t *left;
        G2_TRY(sssp_batch_rows(g, srcs, k, dist, st, d_err, &how, &left));
        if (how == ROWS_LEFT) {
            G2_TRY(sssp_batch_run(g, srcs, k, delta, dist, h, left, st, d_err));
            G2_TRY(sssp_batch_check(g, dist, k, st, d_err));
        }
        if (how != ROWS_NONE) return end_call(g, st, d_err);
    }
    G2_TRY(sssp_batch_run(g, srcs, k, delta, dist, h, nullptr, st, d_err));
    return end_call(g, st, d_err);
}

}  // extern "C"
