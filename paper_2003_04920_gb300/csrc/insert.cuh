// Batched-Extension insertion (Alg. 3) as one cooperative launch.
//
// Four passes over the block, separated by grid barriers: validate the edges
// and count what each row gains; give the rows that overflow room at the end of
// the pool; move them and set the new lengths (and seed the new vertices);
// write the entries and offer the next Improve its candidates.  As launches of
// their own they took seven, with a copy and a host wait in the middle for the
// room needed.  Here the kernel itself stops after the second pass when
// the edges are bad or the pool is used up (the host then repacks it and runs
// the last two passes as launches), and leaves what the host needs in
// page-locked memory right then, so the host goes on while the entries are
// still being written.
//
// What bounds it: for a small block the launches and barriers; for a large one
// scattered 32-byte sectors of deg, rows, g and the pool (about five per new
// entry) and atomics.  Lists are appended to once per CTA and pass -- one atomic
// per warp on the list's counter had cost more than the counting itself -- and
// edges that follow one another with the same endpoint, as a block's usually
// do, count and take their slots with one atomic.
//
// Measured, a call of the block schedules, as seven launches and now: 100
// vertices of 10,000 in 2-D 55 -> 32 us; 10,000 of 200,000 103 -> 67; 50,000 in 6-D
// of 500,000 152 -> 112, of 10^6 145 -> 106, of 4 10^6 205 -> 145.  One edge at a
// time and three CTAs of 512 threads per SM; two edges with two CTAs: 34 / 67 / 109
// / 107 / 150; with three: 38 / 67 / 119 / 108 / 149; four edges with one CTA: 45 /
// 74 / 133 / 134 / 184; one edge with four CTAs: 33 / 70 / 119 / 110 / 153.
#pragma once

#include <cfloat>

#include "graph_kernels.cuh"

namespace pirrt {

constexpr int kInsertThreads = 512;
constexpr int kInsertUnroll = 1;  // edges a thread handles at once

// What the host waits for, in page-locked memory; seq is written last.
struct InsertReport {
    unsigned long long need;  // pool room the block takes
    unsigned status;          // kStatus* bits
    unsigned seq;             // number of the insertion
};

template <typename CT>
struct InsertArgs {
    int64_t n_edges, n_old, n_after;
    const int32_t *src, *dst;
    const CT *cost;
    int32_t root;
    unsigned seq;
    RowExt *rows;
    int32_t *deg, *touched, *alloc;
    int64_t *off;
    Entry<CT> *pool;
    long long pool_used, pool_cap;
    double *g;
    float *g32;
    int32_t *p;
    CT *pc;
    unsigned long long *cand;
    unsigned *stamp;
    int32_t *list[2];
    DevCounters *ctr;
    InsertReport *report;
};

// A run of lanes (from the lowest) that share a key: its first lane, its length
// and this lane's place.
struct Run {
    int first, length, place;
};
__device__ __forceinline__ Run warp_run(int32_t key) {
    const int lane = threadIdx.x & 31;
    const int32_t before = __shfl_up_sync(0xffffffffu, key, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || before != key);
    const unsigned upto = heads & (0xffffffffu >> (31 - lane));
    const int first = 31 - __clz(upto);
    const unsigned after = lane == 31 ? 0u : heads & (0xfffffffeu << lane);
    const int end = after ? __ffs(after) - 1 : 32;
    return Run{first, end - first, lane - first};
}

// Extent of row v, written earlier in this launch by other CTAs.
__device__ __forceinline__ RowExt row_now(const RowExt *rows, int64_t v) {
    static_assert(sizeof(RowExt) == 16, "one 16-byte load");
    const int4 q = __ldcg(reinterpret_cast<const int4 *>(rows + v));
    RowExt r;
    memcpy(&r, &q, sizeof(r));
    return r;
}

// Pass 1: validate the undirected edges and count, per endpoint, the CSR entries
// the block adds (deg is all zero between insertions).  Invalid input raises
// kStatusBadInput and is not counted (the host then discards the block).  An old
// row gaining its first entry joins the touched list; the new rows
// [n_old, n_after) are handled as a range.
template <typename CT>
__device__ __forceinline__ void insert_count(const InsertArgs<CT> &a, unsigned long long *s_scan) {
    constexpr int U = kInsertUnroll;
    const int lane = threadIdx.x & 31;
    for (int64_t base = (int64_t)blockIdx.x * (kInsertThreads * U); base < a.n_edges;
         base += (int64_t)gridDim.x * (kInsertThreads * U)) {
        int32_t x[2 * U];
        bool bad = false;
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t e = base + k * kInsertThreads + threadIdx.x;
            x[2 * k] = x[2 * k + 1] = -1;
            if (e < a.n_edges) {
                const int32_t u = a.src[e], v = a.dst[e];
                const double c = (double)a.cost[e];
                const bool ok = u >= 0 && v >= 0 && u < a.n_after && v < a.n_after && u != v &&
                                c > 0.0 && c <= DBL_MAX;  // rejects NaN, +inf, <= 0
                if (ok) {
                    x[2 * k] = u;
                    x[2 * k + 1] = v;
                } else {
                    bad = true;
                }
            }
        }
        if (bad) atomicOr(&a.ctr->insert_status, kStatusBadInput);
        unsigned first = 0;  // rows whose count this lane raised from 0
#pragma unroll
        for (int k = 0; k < 2 * U; ++k) {
            const Run r = warp_run(x[k]);
            if (lane == r.first && x[k] >= 0 && atomicAdd(&a.deg[x[k]], r.length) == 0 &&
                x[k] < a.n_old)
                first |= 1u << k;
        }
        unsigned at, none;
        block_reserve2<kInsertThreads>(__popc(first), 0u, &a.ctr->n_touched, &a.ctr->n_touched,
                                       s_scan, at, none);
#pragma unroll
        for (int k = 0; k < 2 * U; ++k)
            if ((first >> k) & 1u) a.touched[at++] = x[k];
    }
}

// Item k of the rows an insertion changes: the touched old rows, then the new
// rows [n_old, n_after).
__device__ __forceinline__ int64_t changed_row(int64_t k, int64_t nt, const int32_t *touched,
                                               int64_t n_old) {
    return k < nt ? (int64_t)__ldcg(&touched[k]) : n_old + (k - nt);
}

// Pass 2: a changed row that would overflow (every new row with entries) takes
// room at the end of the pool from a cursor, one atomic per CTA; pool offsets
// (relative to the cursor's base) go to off[v].  Rows keep their relative order
// within a CTA only, which nothing relies on.
template <typename CT>
__device__ __forceinline__ void insert_room(const InsertArgs<CT> &a, int64_t nt,
                                            unsigned long long *s_scan) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = kInsertThreads / 32;
    const int64_t total = nt + (a.n_after - a.n_old);
    for (int64_t base = (int64_t)blockIdx.x * kInsertThreads; base < total;
         base += (int64_t)gridDim.x * kInsertThreads) {
        const int64_t k = base + threadIdx.x;
        int32_t room = 0;
        int64_t v = -1;
        if (k < total) {
            v = changed_row(k, nt, a.touched, a.n_old);
            int32_t len = 0, cap = 0;
            if (v < a.n_old) {
                const RowExt r = a.rows[v];
                len = r.len;
                cap = r.cap;
            }
            const int32_t need = len + __ldcg(&a.deg[v]);
            if (need > cap) room = row_room(need, false);
            a.alloc[v] = room;
        }
        unsigned long long incl = (unsigned long long)room;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_scan[warp] = incl;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long run = 0;
            for (int w = 0; w < NW; ++w) {
                const unsigned long long t = s_scan[w];
                s_scan[w] = run;
                run += t;
            }
            s_scan[NW] = run ? atomicAdd(&a.ctr->pool_cursor, run) : 0ull;
        }
        __syncthreads();
        if (room > 0) a.off[v] = (int64_t)(s_scan[NW] + s_scan[warp] + incl - (unsigned)room);
        __syncthreads();
    }
}

// Pass 3: move the changed rows that took room (their old entries first) and set
// every changed row's extent to its length after the block.  One warp per 32 rows.
template <typename CT>
__device__ __forceinline__ void insert_move(const InsertArgs<CT> &a, int64_t nt) {
    const int lane = threadIdx.x & 31;
    const int64_t total = nt + (a.n_after - a.n_old);
    const int64_t warps = (int64_t)gridDim.x * (kInsertThreads / 32);
    unsigned long long copied = 0;
    for (int64_t w0 = ((int64_t)blockIdx.x * (kInsertThreads / 32) + (threadIdx.x >> 5)) * 32;
         w0 < total; w0 += warps * 32) {
        const int64_t k = w0 + lane;
        long long ob = 0, nb = 0;
        int32_t len = 0;
        bool move = false;
        if (k < total) {
            const int64_t v = changed_row(k, nt, a.touched, a.n_old);
            RowExt r{0, 0, 0};
            if (v < a.n_old) r = a.rows[v];
            const int32_t room = __ldcg(&a.alloc[v]);
            len = r.len;
            ob = r.beg;
            RowExt nr = r;
            nr.len = r.len + __ldcg(&a.deg[v]);
            if (room > 0) {
                nb = a.pool_used + __ldcg(&a.off[v]);
                nr.beg = nb;
                nr.cap = room;
                move = len > 0;
            }
            a.rows[v] = nr;
        }
        unsigned todo = __ballot_sync(0xffffffffu, move);
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1u;
            const long long sb = __shfl_sync(0xffffffffu, ob, l);
            const long long db = __shfl_sync(0xffffffffu, nb, l);
            const int32_t n = __shfl_sync(0xffffffffu, len, l);
            for (int32_t q = lane; q < n; q += 32) a.pool[db + q] = ld_stream(&a.pool[sb + q]);
            copied += (unsigned long long)n;
        }
    }
    if (lane == 0 && copied) atomicAdd(&a.ctr->insert_copied, copied);
}

// Seed the new vertices: g = +inf (0 for the root), no parent, no offer.  They
// join the next Improve frontier through the offers of their new edges.
template <typename CT>
__device__ __forceinline__ void insert_init(const InsertArgs<CT> &a) {
    for (int64_t v = a.n_old + (int64_t)blockIdx.x * kInsertThreads + threadIdx.x; v < a.n_after;
         v += (int64_t)gridDim.x * kInsertThreads) {
        a.g[v] = (v == a.root) ? 0.0 : CUDART_INF;
        a.g32[v] = (v == a.root) ? 0.0f : __int_as_float(0x7f800000);
        a.p[v] = (v == a.root) ? kRootMark : -1;
        a.pc[v] = CT(0);
        a.cand[v] = kCandNone;
    }
}

// Pass 4: both directions of every new edge at the tail of its rows (filled from
// the row end, taking every count back to zero; order within a row is
// irrelevant), and the next Improve frontier.  The new edge offers each endpoint
// the other's candidate; an endpoint joins the list only if that candidate beats
// its g (g >= cur, so a candidate not below g can never win; a new vertex has g =
// +inf and joins with its first finite neighbour).
template <typename CT>
__device__ __forceinline__ void insert_entries(const InsertArgs<CT> &a,
                                               unsigned long long *s_scan) {
    constexpr int U = kInsertUnroll;
    const int lane = threadIdx.x & 31;
    const unsigned epoch = a.ctr->epoch;
    int32_t *active = (a.ctr->la & 1u) ? a.list[1] : a.list[0];
    for (int64_t base = (int64_t)blockIdx.x * (kInsertThreads * U); base < a.n_edges;
         base += (int64_t)gridDim.x * (kInsertThreads * U)) {
        int32_t x[2 * U];
        CT w[U];
        bool better[2 * U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int64_t e = base + k * kInsertThreads + threadIdx.x;
            x[2 * k] = x[2 * k + 1] = -1;
            w[k] = CT(0);
            if (e < a.n_edges) {
                x[2 * k] = a.src[e];
                x[2 * k + 1] = a.dst[e];
                w[k] = a.cost[e];
            }
        }
        Run run[2 * U];
        int32_t left[2 * U];
#pragma unroll
        for (int k = 0; k < 2 * U; ++k) {
            run[k] = warp_run(x[k]);
            left[k] = 0;
            if (lane == run[k].first && x[k] >= 0) left[k] = atomicSub(&a.deg[x[k]], run[k].length);
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int32_t u = x[2 * k], v = x[2 * k + 1];
            bool bu = false, bv = false;
            const int32_t lu = __shfl_sync(0xffffffffu, left[2 * k], run[2 * k].first);
            const int32_t lv = __shfl_sync(0xffffffffu, left[2 * k + 1], run[2 * k + 1].first);
            if (u >= 0) {
                const RowExt ru = row_now(a.rows, u), rv = row_now(a.rows, v);
                const double gu = __ldcg(&a.g[u]), gv = __ldcg(&a.g[v]);
                Entry<CT> eu{}, ev{};
                eu.col = v;
                eu.w = w[k];
                ev.col = u;
                ev.w = w[k];
                a.pool[ru.beg + ru.len - lu + run[2 * k].place] = eu;
                a.pool[rv.beg + rv.len - lv + run[2 * k + 1].place] = ev;
                const double cu = gv + widen(w[k]), cv = gu + widen(w[k]);
                bu = u != a.root && gv < CUDART_INF && cu < gu;
                bv = v != a.root && gu < CUDART_INF && cv < gv;
                if (bu) offer(a.cand, u, cu);
                if (bv) offer(a.cand, v, cv);
            }
            better[2 * k] = bu;
            better[2 * k + 1] = bv;
        }
        // one stamp per run of the same endpoint
        unsigned join = 0;
#pragma unroll
        for (int k = 0; k < 2 * U; ++k) {
            const unsigned any = __ballot_sync(0xffffffffu, better[k]);
            const unsigned mine = (0xffffffffu >> (32 - run[k].length)) << run[k].first;
            if (lane == run[k].first && (any & mine) != 0u &&
                atomicExch(&a.stamp[x[k]], epoch) != epoch)
                join |= 1u << k;
        }
        unsigned at, none;
        block_reserve2<kInsertThreads>(__popc(join), 0u, &a.ctr->n_active, &a.ctr->n_active, s_scan,
                                       at, none);
#pragma unroll
        for (int k = 0; k < 2 * U; ++k)
            if ((join >> k) & 1u) active[at++] = x[k];
    }
}

template <typename CT>
__device__ __forceinline__ void insert_report(const InsertArgs<CT> &a, unsigned status) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    volatile InsertReport *r = a.report;
    r->need = __ldcg(&a.ctr->pool_cursor);
    r->status = status;
    __threadfence_system();
    r->seq = a.seq;
}

// A barrier timed out here: later launches see it whatever this one reports.
__device__ __forceinline__ unsigned insert_gave_up(DevCounters *c) {
    if (threadIdx.x == 0) atomicExch(&c->insert_late, 1u);
    return kStatusTimeout;
}

template <typename CT>
__global__ void __launch_bounds__(kInsertThreads, 3)
insert_kernel(const __grid_constant__ InsertArgs<CT> a) {
    __shared__ unsigned long long s_scan[kInsertThreads / 32 + 2];
    DevCounters *c = a.ctr;
    // (set by an earlier launch, or past this one's first barrier)
    if (__ldcg(&c->insert_late) != 0u) return insert_report<CT>(a, kStatusTimeout);
    // what an earlier exploit reported does not stop the next one
    if (blockIdx.x == 0 && threadIdx.x == 0) c->status = 0u;
    insert_count<CT>(a, s_scan);
    if (!grid_barrier(c, gridDim.x)) return insert_report<CT>(a, insert_gave_up(c));
    const unsigned status = __ldcg(&c->insert_status);
    if (status != 0u) return insert_report<CT>(a, status);
    const int64_t nt = (int64_t)__ldcg(&c->n_touched);
    insert_room<CT>(a, nt, s_scan);
    if (!grid_barrier(c, gridDim.x)) return insert_report<CT>(a, insert_gave_up(c));
    insert_report<CT>(a, 0u);
    if (a.pool_used + (long long)__ldcg(&c->pool_cursor) > a.pool_cap) return;
    insert_move<CT>(a, nt);
    insert_init<CT>(a);
    if (!grid_barrier(c, gridDim.x)) {
        insert_gave_up(c);
        return;
    }
    insert_entries<CT>(a, s_scan);
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // as the next insertion expects them
        c->n_touched = 0u;
        c->pool_cursor = 0ull;
    }
}

// The last two passes as a launch of their own, once the host has repacked the
// pool (rows and lengths are set): seed, then entries.
template <typename CT>
__global__ void __launch_bounds__(kInsertThreads, 3)
insert_init_kernel(const __grid_constant__ InsertArgs<CT> a) {
    insert_init<CT>(a);
}

template <typename CT>
__global__ void __launch_bounds__(kInsertThreads, 3)
insert_entries_kernel(const __grid_constant__ InsertArgs<CT> a) {
    __shared__ unsigned long long s_scan[kInsertThreads / 32 + 2];
    insert_entries<CT>(a, s_scan);
}

// After an insertion that did not run to its end: as the next one expects them.
static __global__ void insert_clear_kernel(DevCounters *c) {
    c->n_touched = 0u;
    c->insert_status = 0u;
    c->pool_cursor = 0ull;
    c->bar_count = 0u;
}

}  // namespace pirrt
