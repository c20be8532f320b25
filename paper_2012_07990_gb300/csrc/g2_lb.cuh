// g2_lb.cuh — the load-balancing library (Sec. III and VI-C): how the arcs of
// the input vertexset are divided among threads in the PUSH direction, and
// how destinations are divided in the PULL direction.
//
// Every routine takes a virtual CTA index `bid` and CTA count `nb` so it can
// run from a per-round __global__ wrapper (bid = blockIdx.x) or inside the
// fused persistent kernel (Sec. VI-C, kernel fusion), where a few resident
// CTAs do the work of many.  All inner loops are warp-uniform so that the
// warp-aggregated enqueue (emit) sees all 32 lanes.
#pragma once
#include "g2_device.cuh"

namespace g2 {

template <class T>
__device__ __forceinline__ T shfl_xor_acc(T x, int d) {
    return __shfl_xor_sync(G2_FULL, x, d);
}

// --------------------------------------------------------------- VERTEX_BASED
// Every lane walks every stride-th of the len arcs from beg, kFlight a step
// (len may be negative: none).
template <class Op>
__device__ __forceinline__ void walk_lists(const DevGraph &g, const Op &op, const OutCtx &out,
                                           Stage &st, int32_t u, typename Op::S s, int32_t beg,
                                           int32_t len, int stride = 1) {
    constexpr int N = Op::kFlight;
    const int maxlen = (int)__reduce_max_sync(G2_FULL, (unsigned)max(len, 0));
    for (int k = 0; k < maxlen; k += N * stride) {
        int32_t us[N], e[N];
        typename Op::S ss[N];
        bool on[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            us[j] = u;
            ss[j] = s;
            e[j] = beg + k + j * stride;
            on[j] = k + j * stride < len;
        }
        apply_arcs<N>(op, out, st, us, ss, g.col, e, on);
    }
}

// A group of `width` threads (this one is number `t` of it) walks the arcs
// [beg, end) of one vertex, kFlight steps of `width` arcs at a time.
template <class Op>
__device__ __forceinline__ void walk_group(const DevGraph &g, const Op &op, const OutCtx &out,
                                           Stage &st, int32_t u, typename Op::S s, int32_t beg, int32_t end,
                                           int t, int width) {
    constexpr int N = Op::kFlight;
    for (int64_t e0 = beg; e0 < end; e0 += N * width) {
        int32_t us[N], e[N];
        typename Op::S ss[N];
        bool on[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int64_t k = e0 + j * width + t;
            us[j] = u;
            ss[j] = s;
            on[j] = k < end;
            e[j] = on[j] ? (int32_t)k : 0;
        }
        apply_arcs<N>(op, out, st, us, ss, g.col, e, on);
    }
}

// One thread per active vertex, serial walk of its arcs.
template <class Op>
__device__ void lb_vertex(const DevGraph &g, const FrontierIn &fin, int32_t fsize, const Op &op,
                          const OutCtx &out, int bid, int nb, unsigned long long *ctr) {
    Stage st = stage_begin();
    const int lane = threadIdx.x & 31;
    const int gw = bid * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int nw = nb * (blockDim.x >> 5);
    for (int64_t base = (int64_t)gw * 32; base < fsize; base += (int64_t)nw * 32) {
        int32_t i = (int32_t)base + lane;
        int32_t u = 0, beg = 0, len = 0;
        typename Op::S s{};
        if (i < fsize) {
            u = fin.vertex(i);
            s = op.load(u);
            if (!op.skip(s)) {
                beg = g.rowptr[u];
                len = g.rowptr[u + 1] - beg;
            }
        }
        count_arcs(ctr, len);
        walk_lists(g, op, out, st, u, s, beg, len);
    }
    stage_end(out, st);
}

// ------------------------------------------------------------------------ WM
// A warp takes up to 32 active vertices (fewer where the list is short: an
// equal share for every warp), prefix-sums their degrees with shuffles and
// walks the combined arc range 32 arcs at a time, kFlight such steps in
// flight; each lane finds the owner of its arc by a 5-step binary search over
// the lanes' prefix sums.
template <class Op>
__device__ void lb_warp(const DevGraph &g, const FrontierIn &fin, int32_t fsize, const Op &op,
                        const OutCtx &out, int bid, int nb, unsigned long long *ctr) {
    Stage st = stage_begin();
    constexpr int N = Op::kFlight;
    const int lane = threadIdx.x & 31;
    const int gw = bid * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int nw = nb * (blockDim.x >> 5);
    const int per = fsize < nw * 32 ? (fsize + nw - 1) / nw : 32;
    for (int64_t base = (int64_t)gw * per; base < fsize; base += (int64_t)nw * per) {
        int32_t i = (int32_t)base + lane;
        int32_t u = 0, beg = 0, len = 0;
        typename Op::S s{};
        if (lane < per && i < fsize) {
            u = fin.vertex(i);
            s = op.load(u);
            if (!op.skip(s)) {
                beg = g.rowptr[u];
                len = g.rowptr[u + 1] - beg;
            }
        }
        count_arcs(ctr, len);
        int incl = warp_incl_scan(len);
        int total = __shfl_sync(G2_FULL, incl, 31);
        int off = beg - (incl - len);  // arc k of the range sits at off + k
        for (int k0 = 0; k0 < total; k0 += 32 * N) {
            int32_t us[N], e[N];
            typename Op::S ss[N];
            bool on[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                int k = k0 + 32 * j + lane;
                int lo = 0, hi = 31;
#pragma unroll
                for (int b = 0; b < 5; ++b) {
                    int mid = (lo + hi) >> 1;
                    int im = __shfl_sync(G2_FULL, incl, mid);
                    if (im > k) hi = mid;
                    else lo = mid + 1;
                }
                lo &= 31;  // past the range: any lane
                us[j] = __shfl_sync(G2_FULL, u, lo);
                ss[j] = shfl(s, lo);
                e[j] = __shfl_sync(G2_FULL, off, lo) + k;
                on[j] = k < total;
            }
            apply_arcs<N>(op, out, st, us, ss, g.col, e, on);
        }
    }
    stage_end(out, st);
}

// ------------------------------------------------------------------------ CM
// A CTA takes kCta active vertices, block-scans their degrees in shared memory
// and walks the combined arc range kCta arcs at a time, kFlight such steps in
// flight.
template <class Op>
__device__ void lb_cta(const DevGraph &g, const FrontierIn &fin, int32_t fsize, const Op &op,
                       const OutCtx &out, int bid, int nb, unsigned long long *ctr) {
    Stage st = stage_begin();
    constexpr int N = Op::kFlight;
    __shared__ int s_incl[kCta];
    __shared__ int32_t s_u[kCta];
    __shared__ int32_t s_beg[kCta];
    __shared__ typename Op::S s_s[kCta];
    __shared__ int s_warp[kWarps];
    const int tid = threadIdx.x;
    for (int64_t base = (int64_t)bid * kCta; base < fsize; base += (int64_t)nb * kCta) {
        int32_t i = (int32_t)base + tid;
        int32_t u = 0, beg = 0, len = 0;
        typename Op::S s{};
        if (i < fsize) {
            u = fin.vertex(i);
            s = op.load(u);
            if (!op.skip(s)) {
                beg = g.rowptr[u];
                len = g.rowptr[u + 1] - beg;
            }
        }
        count_arcs(ctr, len);
        int total;
        int incl = block_incl_scan(len, s_warp, &total);
        s_incl[tid] = incl;
        s_u[tid] = u;
        s_beg[tid] = beg - (incl - len);  // arc index = s_beg[owner] + k
        s_s[tid] = s;
        __syncthreads();
        for (int k0 = 0; k0 < total; k0 += kCta * N) {
            int32_t us[N], e[N];
            typename Op::S ss[N];
            bool on[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const int k = k0 + kCta * j + tid;
                on[j] = k < total;
                int lo = 0, hi = on[j] ? kCta - 1 : 0;
                while (lo < hi) {
                    int mid = (lo + hi) >> 1;
                    if (s_incl[mid] > k) hi = mid;
                    else lo = mid + 1;
                }
                us[j] = s_u[lo];
                ss[j] = s_s[lo];
                e[j] = s_beg[lo] + k;
            }
            apply_arcs<N>(op, out, st, us, ss, g.col, e, on);
        }
        __syncthreads();
    }
    stage_end(out, st);
}

// -------------------------------------------------------------------- STRICT
// Every thread gets the same number of arcs: arc k of the frontier-wide arc
// sequence belongs to the active vertex i with scan[i] <= k < scan[i+1]
// (scan = exclusive prefix sum of the active vertices' degrees, computed by a
// separate pass).  A CTA takes runs of up to kStrictRun consecutive tiles of
// kTile arcs: a run's first owner by a 32-way search of every warp, the
// owners of a tile read into shared memory in one pass (each with its source
// value and arc base, so that an arc reads nothing of its owner from global
// memory) and found there by binary search, kFlight arcs per thread at
// once; the next tile starts at the last owner.  A tile with more owners than
// fit (vertices without arcs in the list) searches the scan itself.
constexpr int kStrictRun = 8;

// The owners of a tile, in shared memory (one copy for both forms below: what
// it takes comes out of L1).
template <class Op>
struct StrictOwners {
    static constexpr int kTile = kCta * Op::kFlight;
    static constexpr int kOwn = kTile + kCta;  // a tile of one-arc owners and the last one's
    int32_t at[kOwn];    // first arc of the owner, from the tile's start
    int32_t base[kOwn];  // arc k of the tile sits at base[owner] + k
    int32_t u[kOwn];
    typename Op::S s[kOwn];
};
template <class Op>
__device__ __forceinline__ StrictOwners<Op> &strict_owners() {
    __shared__ StrictOwners<Op> x;
    return x;
}

// STRICT for an update of one arc in flight (it loops over sources for every
// arc, and lives on what L1 keeps of their distances): the tiles' owners would
// be shared memory taken from L1, and tiles of kCta arcs.  A warp takes
// kStrictWarp arcs (32 where there are not as many for every warp), and a lane
// searches the scan itself, between the owners of the first and the last.  32
// sources of RMAT-20, weights 1-255: 16.9 ms, 27.7 with owners in shared memory
// in tiles of kCta arcs, 23.9 in tiles of 4 kCta, 19.8 with 512 arcs a warp.
// RMAT-14: 3.7 ms, 4.4 with 128 arcs for every warp; 400 x 400 grid 26.9 and 32.2.
constexpr int kStrictWarp = 128;

template <class Op>
__device__ void lb_strict_single(const DevGraph &g, const FrontierIn &fin, int32_t fsize,
                                 const int32_t *scan, const Op &op, const OutCtx &out, int bid,
                                 int nb, unsigned long long *ctr) {
    Stage st = stage_begin();
    const int lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)bid * kWarps + (threadIdx.x >> 5), nw = (int64_t)nb * kWarps;
    const int32_t total = scan[fsize];
    const int share = total < nw * kStrictWarp ? 32 : kStrictWarp;
    for (int64_t t0 = gw * share; t0 < total; t0 += nw * share) {
        const int64_t t1 = t0 + share < total ? t0 + share : total;
        const int32_t own0 = scan_owner(scan, fsize, (int32_t)t0);
        const int32_t own1 = scan_owner(scan, fsize, (int32_t)(t1 - 1));
        count_arcs(ctr, lane == 0 ? (int)(t1 - t0) : 0);
#pragma unroll 1
        for (int64_t b = t0; b < t1; b += 32) {
            const int64_t k = b + lane;
            int32_t us[1] = {0}, e[1] = {0};
            typename Op::S ss[1] = {};
            bool on[1] = {k < t1};
            if (on[0]) {
                int32_t lo = own0, hi = own1;
                while (lo < hi) {
                    const int32_t mid = lo + (hi - lo + 1) / 2;
                    if (scan[mid] <= k) lo = mid;
                    else hi = mid - 1;
                }
                us[0] = fin.vertex(lo);
                ss[0] = op.load(us[0]);
                e[0] = g.rowptr[us[0]] + (int32_t)(k - scan[lo]);
            }
            apply_arcs<1>(op, out, st, us, ss, g.col, e, on);
        }
    }
    stage_end(out, st);
}

template <class Op>
__device__ void lb_strict(const DevGraph &g, const FrontierIn &fin, int32_t fsize,
                          const int32_t *scan, const Op &op, const OutCtx &out, int bid, int nb,
                          unsigned long long *ctr) {
    Stage st = stage_begin();
    constexpr int N = Op::kFlight;
    constexpr int kTile = StrictOwners<Op>::kTile, kOwn = StrictOwners<Op>::kOwn;
    StrictOwners<Op> &own = strict_owners<Op>();
    int32_t *s_at = own.at, *s_base = own.base, *s_u = own.u;
    typename Op::S *s_s = own.s;
    const int tid = threadIdx.x;
    const int32_t total = scan[fsize];
    // (tile numbers fit: total < 2^31)
    const int32_t tiles = (int32_t)(((int64_t)total + kTile - 1) / kTile);
    // runs of one to kStrictRun tiles, four or more per CTA where there are
    // as many: neighbouring arcs (a hub's) go to several CTAs
    int32_t run = tiles / (nb * 4);
    run = run < 1 ? 1 : run > kStrictRun ? kStrictRun : run;
    int32_t own0 = 0;
    int left = 0;  // tiles of the current run
    for (int32_t it = run * bid; it < tiles; ++it) {
        const int64_t t0 = (int64_t)it * kTile;
        if (left == 0) {
            own0 = scan_owner(scan, fsize, (int32_t)t0);
            left = run;
        }
        const int len = (int)(total - t0 < kTile ? total - t0 : kTile);
        // owners of the tile: the entries from own0 on that start before its end
        int no = 0;
        bool more = true;
        while (more && no < kOwn) {
            const int64_t i = (int64_t)own0 + no + tid;
            int32_t at = 0;
            bool in = i < fsize;
            if (in) {
                at = (int32_t)((int64_t)scan[i] - t0);
                in = at < len;
            }
            if (in) {
                const int32_t u = fin.vertex((int32_t)i);
                s_at[no + tid] = at;
                s_u[no + tid] = u;
                s_s[no + tid] = op.load(u);
                s_base[no + tid] = g.rowptr[u] - at;
            }
            const int c = __syncthreads_count(in);
            more = c == kCta;
            no += c;
        }
        if (!more) {
            // shared search, the thread's arcs side by side
            int top = 1;
            while (top < no) top <<= 1;
            int lo[N];
#pragma unroll
            for (int j = 0; j < N; ++j) lo[j] = 0;
            for (int d = top >> 1; d > 0; d >>= 1) {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const int m = lo[j] + d;
                    if (m < no && s_at[m] <= j * kCta + tid) lo[j] = m;
                }
            }
            int cnt = 0;
            int32_t us[N], e[N];
            typename Op::S ss[N];
            bool on[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const int k = j * kCta + tid;
                on[j] = k < len;
                us[j] = s_u[lo[j]];
                ss[j] = s_s[lo[j]];
                e[j] = s_base[lo[j]] + k;
                cnt += on[j];
            }
            apply_arcs<N>(op, out, st, us, ss, g.col, e, on);
            count_arcs(ctr, cnt);
            // the last owner of this tile may reach into the next one
            own0 += no - 1;
        } else {
            int cnt = 0;
#pragma unroll 1
            for (int j = 0; j < N; ++j) {
                const int64_t k = t0 + j * kCta + tid;
                int32_t us[1] = {0}, e[1] = {0};
                typename Op::S ss[1] = {};
                bool on[1] = {k < t0 + len};
                if (on[0]) {
                    int32_t lo = own0, hi = fsize - 1;
                    while (lo < hi) {
                        const int32_t mid = lo + (hi - lo + 1) / 2;
                        if (scan[mid] <= k) lo = mid;
                        else hi = mid - 1;
                    }
                    us[0] = fin.vertex(lo);
                    ss[0] = op.load(us[0]);
                    e[0] = g.rowptr[us[0]] + (int32_t)(k - scan[lo]);
                    ++cnt;
                }
                apply_arcs<1>(op, out, st, us, ss, g.col, e, on);
            }
            count_arcs(ctr, cnt);
            own0 = scan_owner(scan, fsize, (int32_t)(t0 + len - 1));
        }
        if (--left == 0) it += run * (nb - 1);
        __syncthreads();
    }
    stage_end(out, st);
}

// STRICT for a list of up to kStrictSmall entries in a fused loop, without a
// scan of the whole grid before it: every CTA scans the list's degrees itself
// (1 us, against two grid barriers and a pass over the list) and takes every
// nb-th tile of its arcs.  False, in every CTA, and nothing done if there are
// more than `most` arcs.
constexpr int kStrictSmall = 4 * kCta;

template <class Op>
__device__ bool lb_strict_small(const DevGraph &g, const FrontierIn &fin, int32_t fsize, const Op &op,
                                const OutCtx &out, int bid, int nb, unsigned long long *ctr,
                                int32_t most = 0x7fffffff) {
    typedef typename Op::S S;
    constexpr int N = Op::kFlight, kTile = kCta * N, kPer = kStrictSmall / kCta;
    Stage st = stage_begin();
    static_assert(kStrictSmall <= StrictOwners<Op>::kOwn, "the list fits");
    StrictOwners<Op> &own = strict_owners<Op>();
    int32_t *s_at = own.at, *s_base = own.base, *s_u = own.u;
    S *s_s = own.s;
    __shared__ int s_warp[kWarps];
    const int tid = threadIdx.x;
    int32_t u[kPer], b[kPer], deg[kPer];
    int sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int i = tid * kPer + j;
        u[j] = i < fsize ? fin.vertex(i) : -1;
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        b[j] = deg[j] = 0;
        if (u[j] >= 0) {
            b[j] = g.rowptr[u[j]];
            deg[j] = g.rowptr[u[j] + 1] - b[j];
            s_s[tid * kPer + j] = op.load(u[j]);
        }
        sum += deg[j];
    }
    int total;
    int at = block_incl_scan(sum, s_warp, &total) - sum;
    if (total > most) return false;  // the same in every CTA
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int i = tid * kPer + j;
        s_at[i] = at;
        s_u[i] = u[j];
        s_base[i] = b[j] - at;
        at += deg[j];
    }
    __syncthreads();
    int top = 1;
    while (top < fsize) top <<= 1;
    for (int64_t t0 = (int64_t)bid * kTile; t0 < total; t0 += (int64_t)nb * kTile) {
        int lo[N];
#pragma unroll
        for (int j = 0; j < N; ++j) lo[j] = 0;
        for (int d = top >> 1; d > 0; d >>= 1) {
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const int m = lo[j] + d;
                if (m < fsize && s_at[m] <= t0 + j * kCta + tid) lo[j] = m;
            }
        }
        int32_t us[N], e[N];
        S ss[N];
        bool on[N];
        int cnt = 0;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int64_t k = t0 + j * kCta + tid;
            on[j] = k < total;
            us[j] = s_u[lo[j]];
            ss[j] = s_s[lo[j]];
            e[j] = s_base[lo[j]] + (int32_t)k;
            cnt += on[j];
        }
        apply_arcs<N>(op, out, st, us, ss, g.col, e, on);
        count_arcs(ctr, cnt);
    }
    stage_end(out, st);
    __syncthreads();  // the next call writes the arrays
    return true;
}

// ---------------------------------------------------------------------- ETWC
// Algorithm 3.  Inside each CTA every thread takes one active vertex and
// splits its arc range into a multiple of the CTA size, a multiple of the warp
// size and a remainder, pushed to three shared-memory queues; then the
// remainder entries are walked by single threads, the warp entries by whole
// warps and the CTA entries by the whole CTA (cyclic distribution).
template <class S>
struct EtwcEntry {
    int32_t beg, end, u;
    S s;
};

// Frontier-wide hand-off of the CTA-stage entries: on a power-law graph a few
// CTAs hold most of them (RMAT-22's first BFS round is one 163K-arc vertex; a
// frontier in vertex order puts the hubs into its first CTAs), and the rest
// of the grid waits.  Such entries go, in pieces of kEtwcPiece arcs, to a
// list that a second pass spreads over every CTA (k_push_etwc_spill).  q ==
// null: no hand-off, every entry stays with its CTA, as in Algorithm 3.  An
// entry that no longer fits the list stays with its CTA too.
constexpr int32_t kEtwcPiece = 4 * kCta;
template <class S>
struct EtwcSpill {
    EtwcEntry<S> *q;
    int32_t *cnt;
    int32_t cap;
};

// Room for the hand-off of a frontier without repeats: every entry has at
// least kCta arcs and one piece that is not full.
__host__ __device__ inline int64_t etwc_spill_cap(int64_t fsize, int64_t m) {
    const int64_t big = m / kCta;
    return (fsize < big ? fsize : big) + m / kEtwcPiece + 1;
}

template <class Op>
__device__ void lb_etwc(const DevGraph &g, const FrontierIn &fin, int32_t fsize, const Op &op,
                        const OutCtx &out, int bid, int nb, unsigned long long *ctr,
                        EtwcSpill<typename Op::S> spill = {nullptr, nullptr, 0}) {
    Stage st = stage_begin();
    typedef typename Op::S S;
    __shared__ EtwcEntry<S> q0[kCta], q1[kCta], q2[kCta];
    __shared__ int n0, n1, n2;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    // the list in groups of 32, group x to CTA x mod nb: neighbours in the
    // list (hubs, where it is in vertex order) go to different CTAs
    const int64_t groups = ((int64_t)fsize + 31) / 32;
    for (int64_t base = 0; base + bid < groups; base += (int64_t)nb * kWarps) {
        if (tid == 0) n0 = n1 = n2 = 0;
        __syncthreads();
        const int64_t i = (base + (int64_t)wid * nb + bid) * 32 + lane;
        int len0 = 0;
        if (i < fsize) {
            int32_t u = fin.vertex((int32_t)i);
            S s = op.load(u);
            if (!op.skip(s)) {
                int32_t beg = g.rowptr[u], end = g.rowptr[u + 1];
                int32_t size = end - beg;
                len0 = size;
                int32_t c = (size / kCta) * kCta;  // CTA-granularity part
                if (c > 0) {
                    bool keep = true;
                    if (spill.q) {
                        const int32_t np = (c + kEtwcPiece - 1) / kEtwcPiece;
                        const int32_t p = atomicAdd(spill.cnt, np);
                        keep = p > spill.cap - np;
                        for (int32_t x = 0; x < np && p + x < spill.cap && p >= 0; ++x) {
                            const int32_t b = keep ? beg + c : beg + x * kEtwcPiece;
                            const int32_t e = beg + c - b < kEtwcPiece ? beg + c : b + kEtwcPiece;
                            spill.q[p + x] = EtwcEntry<S>{b, e, u, s};
                        }
                    }
                    if (keep) {
                        int p = atomicAdd(&n2, 1);
                        q2[p] = EtwcEntry<S>{beg, beg + c, u, s};
                    }
                    beg += c;
                    size -= c;
                }
                int32_t wpart = (size / 32) * 32;  // warp-granularity part
                if (wpart > 0) {
                    int p = atomicAdd(&n1, 1);
                    q1[p] = EtwcEntry<S>{beg, beg + wpart, u, s};
                    beg += wpart;
                    size -= wpart;
                }
                if (size > 0) {  // remainder, < 32 arcs
                    int p = atomicAdd(&n0, 1);
                    q0[p] = EtwcEntry<S>{beg, end, u, s};
                }
            }
        }
        count_arcs(ctr, len0);
        __syncthreads();
        // stage 0: four neighbouring threads per entry (one thread per entry
        // leaves most of a CTA idle behind its longest remainder, and its
        // reads of the arcs uncoalesced)
        {
            const int sub = lane & 3;
            for (int j0 = wid * 8; j0 < n0; j0 += kWarps * 8) {
                const int j = j0 + (lane >> 2);
                int32_t beg = 0, len = 0, u = 0;
                S s{};
                if (j < n0) {
                    beg = q0[j].beg;
                    len = q0[j].end - beg;
                    u = q0[j].u;
                    s = q0[j].s;
                }
                walk_lists(g, op, out, st, u, s, beg + sub, len - sub, 4);
            }
        }
        // stage 1: one warp per entry, lanes cyclic
        for (int j = wid; j < n1; j += kWarps) {
            EtwcEntry<S> en = q1[j];
            walk_group(g, op, out, st, en.u, en.s, en.beg, en.end, lane, 32);
        }
        // stage 2: the whole CTA per entry
        for (int j = 0; j < n2; ++j) {
            EtwcEntry<S> en = q2[j];
            walk_group(g, op, out, st, en.u, en.s, en.beg, en.end, tid, kCta);
        }
        __syncthreads();
    }
    stage_end(out, st);
}

// The handed-off pieces, one CTA each in turn.
template <class Op>
__device__ void lb_etwc_spill(const DevGraph &g, const EtwcSpill<typename Op::S> &spill,
                              const Op &op, const OutCtx &out, int bid, int nb) {
    Stage st = stage_begin();
    int32_t k = *spill.cnt;
    if (k > spill.cap || k < 0) k = spill.cap;
    for (int32_t j = bid; j < k; j += nb) {
        const EtwcEntry<typename Op::S> en = spill.q[j];
        walk_group(g, op, out, st, en.u, en.s, en.beg, en.end, (int)threadIdx.x, kCta);
    }
    stage_end(out, st);
}

// ----------------------------------------------------------------------- TWC
// Frontier-wide degree buckets (Merrill et al.): a classification pass puts
// each active vertex into the small (< 32 arcs), medium (< kCta) or large
// queue; then small vertices are walked by one thread, medium by a warp and
// large by a whole CTA.
template <class Op>
__device__ void lb_twc_classify(const DevGraph &g, const FrontierIn &fin, int32_t fsize,
                                const Op &op, int32_t *qs, int32_t *qm, int32_t *ql,
                                int32_t *counts, int bid, int nb) {
    const int lane = threadIdx.x & 31;
    const int gw = bid * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int nw = nb * (blockDim.x >> 5);
    for (int64_t base = (int64_t)gw * 32; base < fsize; base += (int64_t)nw * 32) {
        int32_t i = (int32_t)base + lane;
        int32_t u = 0, deg = 0;
        if (i < fsize) {
            u = fin.vertex(i);
            if (!op.skip(op.load(u))) deg = g.rowptr[u + 1] - g.rowptr[u];
        }
        warp_append(qs, counts + 0, fsize, nullptr, u, deg > 0 && deg < 32);
        warp_append(qm, counts + 1, fsize, nullptr, u, deg >= 32 && deg < kCta);
        warp_append(ql, counts + 2, fsize, nullptr, u, deg >= kCta);
    }
}

template <class Op>
__device__ void lb_twc_process(const DevGraph &g, const int32_t *qs, const int32_t *qm,
                               const int32_t *ql, const int32_t *counts, const Op &op,
                               const OutCtx &out, int bid, int nb, unsigned long long *ctr) {
    Stage st = stage_begin();
    typedef typename Op::S S;
    const int tid = threadIdx.x, lane = tid & 31;
    const int gw = bid * kWarps + (tid >> 5);
    const int nw = nb * kWarps;
    const int32_t ns = counts[0], nm = counts[1], nl = counts[2];
    // small: thread per vertex
    for (int64_t base = (int64_t)gw * 32; base < ns; base += (int64_t)nw * 32) {
        int32_t i = (int32_t)base + lane;
        int32_t u = 0, beg = 0, len = 0;
        S s{};
        if (i < ns) {
            u = qs[i];
            s = op.load(u);
            beg = g.rowptr[u];
            len = g.rowptr[u + 1] - beg;
        }
        count_arcs(ctr, len);
        walk_lists(g, op, out, st, u, s, beg, len);
    }
    // medium: warp per vertex
    for (int32_t j = gw; j < nm; j += nw) {
        int32_t u = qm[j];
        int32_t beg = g.rowptr[u], end = g.rowptr[u + 1];
        if (ctr && lane == 0) atomicAdd(ctr, (unsigned long long)(end - beg));
        walk_group(g, op, out, st, u, op.load(u), beg, end, lane, 32);
    }
    // large: CTA per vertex
    for (int32_t j = bid; j < nl; j += nb) {
        int32_t u = ql[j];
        int32_t beg = g.rowptr[u], end = g.rowptr[u + 1];
        if (ctr && tid == 0) atomicAdd(ctr, (unsigned long long)(end - beg));
        walk_group(g, op, out, st, u, op.load(u), beg, end, tid, kCta);
    }
    stage_end(out, st);
}

// ----------------------------------------------------------------- EDGE_ONLY
// Arc-parallel over arcs [e0, e1) of a COO (src[], dst[]) array: the whole
// edge set, or one EdgeBlocking segment (Algorithm 2's cooperative for).
template <class Op>
__device__ void lb_edges(const int32_t *src, const int32_t *dst, int64_t e0, int64_t e1,
                         const Op &op, const OutCtx &out, int bid, int nb,
                         unsigned long long *ctr) {
    Stage st = stage_begin();
    constexpr int N = Op::kFlight;
    const int lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)bid * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nw = (int64_t)nb * (blockDim.x >> 5);
    int cnt = 0;
    for (int64_t base = e0 + gw * 32 * N; base < e1; base += nw * 32 * N) {
        int32_t us[N], e[N];
        typename Op::S ss[N];
        bool on[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int64_t k = base + 32 * j + lane;
            on[j] = k < e1;
            e[j] = on[j] ? (int32_t)k : 0;
            us[j] = on[j] ? src[e[j]] : 0;
            cnt += on[j];
        }
#pragma unroll
        for (int j = 0; j < N; ++j) {
            ss[j] = typename Op::S{};
            if (on[j]) {
                ss[j] = op.load(us[j]);
                on[j] = !op.skip(ss[j]);
            }
        }
        apply_arcs<N>(op, out, st, us, ss, dst, e, on);
    }
    count_arcs(ctr, cnt);
    stage_end(out, st);
}

// ---------------------------------------------------------------- PULL side
// Destinations v in [0, n) (or the items of a candidate list) that pass the
// filter scan their in-neighbours u (CSC, ascending) that are in the input
// frontier.  Group size 1 (VERTEX_BASED), 32 (WM) or kCta (CM) threads per
// destination; the group combines its partial results and may stop early.
template <class P, int G>
__device__ void lb_pull(const DevGraph &g, const int32_t *cand, int32_t ncand, const Member &mem,
                        const P &op, const OutCtx &out, int bid, int nb, unsigned long long *ctr) {
    typedef typename P::Acc Acc;
    typedef typename P::Ctx Ctx;
    const int tid = threadIdx.x, lane = tid & 31;
    if (G == 1) {
        const int gw = bid * kWarps + (tid >> 5);
        const int nw = nb * kWarps;
        for (int64_t base = (int64_t)gw * 32; base < ncand; base += (int64_t)nw * 32) {
            int32_t i = (int32_t)base + lane;
            int code = 0;
            int32_t v = 0;
            int cnt = 0;
            if (i < ncand) {
                v = cand ? cand[i] : i;
                Ctx c = op.ctx(v);
                if (op.filter(c)) {
                    Acc acc = op.identity();
                    int32_t e1 = g.crowptr[v + 1];
                    for (int32_t e = g.crowptr[v]; e < e1; ++e) {
                        int32_t u = g.ccol[e];
                        ++cnt;
                        if (mem.has(u)) {
                            acc = op.combine(acc, op.edge(c, u, e));
                            if (op.stop(acc)) break;
                        }
                    }
                    code = op.finish(v, c, acc);
                }
            }
            count_arcs(ctr, cnt);
            if (out.mode == OUT_BITMAP && !cand) {
                // the warp's 32 destinations are one aligned bitmap word
                unsigned mask = __ballot_sync(G2_FULL, code & 1);
                if (lane == 0 && mask) atomicOr(&out.bitmap[base >> 5], mask);
            } else {
                emit(out, v, code);
            }
        }
    } else if (G == 32) {
        const int gw = bid * kWarps + (tid >> 5);
        const int nw = nb * kWarps;
        for (int32_t i = gw; i < ncand; i += nw) {
            int32_t v = cand ? cand[i] : i;
            Ctx c = op.ctx(v);
            int code = 0;
            int cnt = 0;
            if (op.filter(c)) {
                Acc acc = op.identity();
                int32_t e1 = g.crowptr[v + 1];
                for (int32_t e0 = g.crowptr[v]; e0 < e1; e0 += 32) {
                    int32_t e = e0 + lane;
                    Acc a = op.identity();
                    if (e < e1) {
                        int32_t u = g.ccol[e];
                        ++cnt;
                        if (mem.has(u)) a = op.edge(c, u, e);
                    }
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) a = op.combine(a, shfl_xor_acc(a, d));
                    acc = op.combine(acc, a);
                    if (op.stop(acc)) break;
                }
                if (lane == 0) code = op.finish(v, c, acc);
            }
            count_arcs(ctr, cnt);
            // one destination per warp: only lane 0 may emit
            emit(out, v, code);
        }
    } else {
        __shared__ Acc s_red[kWarps];
        __shared__ int s_stop;
        for (int32_t i = bid; i < ncand; i += nb) {
            int32_t v = cand ? cand[i] : i;
            Ctx c = op.ctx(v);
            int code = 0;
            int cnt = 0;
            if (op.filter(c)) {
                Acc acc = op.identity();
                int32_t e1 = g.crowptr[v + 1];
                for (int32_t e0 = g.crowptr[v]; e0 < e1; e0 += kCta) {
                    int32_t e = e0 + tid;
                    Acc a = op.identity();
                    if (e < e1) {
                        int32_t u = g.ccol[e];
                        ++cnt;
                        if (mem.has(u)) a = op.edge(c, u, e);
                    }
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) a = op.combine(a, shfl_xor_acc(a, d));
                    if (lane == 0) s_red[tid >> 5] = a;
                    __syncthreads();
                    if (tid == 0) {
                        Acc t = s_red[0];
                        for (int k = 1; k < kWarps; ++k) t = op.combine(t, s_red[k]);
                        acc = op.combine(acc, t);
                        s_stop = op.stop(acc);
                    }
                    __syncthreads();
                    if (s_stop) break;
                }
                if (tid == 0) code = op.finish(v, c, acc);
            }
            count_arcs(ctr, cnt);
            emit(out, v, code);
            __syncthreads();
        }
    }
}

}  // namespace g2
