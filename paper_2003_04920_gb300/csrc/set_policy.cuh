// set_policy in one cooperative launch: look up every parent edge's cost, commit
// the policy, evaluate it (walk_rounds).
//
// Looking up was one thread per vertex going through its row alone, and the steps
// took seven launches and three waits of the host.  Here eight lanes share a row,
// the costs found are the evaluation's first records, nothing is written to the
// graph before every vertex's parent edge has passed the check (a cycle shows in the
// evaluation only: it is reported, and again by an exploit), and the host polls one
// word.
// What bounds it is the row reads for large graphs, the barriers and the host's
// part of the call for small ones.  2,000 vertices with FP64 costs: a call 102 us
// before, 31 now.  Above 500,000 vertices two CTAs of 64 registers per SM, which spill
// in the evaluation but keep more row reads in flight: with one / with two, rows of
// 32 entries, FP32: 30,000 vertices 45 / 56 us, 300,000 152 / 124, 10^6 434 / 294, 3 10^6
// 1214 / 781 (as separate launches 114, 181, 350, 818); rows of 8: 300,000 86 / 98,
// 10^6 297 / 227.
#pragma once

#include "evaluate_walk.cuh"
#include "graph_kernels.cuh"

namespace pirrt {

template <typename CT>
struct PolicyArgs {
    int64_t n;
    int32_t root;
    const int32_t *parent;  // the caller's
    const RowExt *rows;
    const Entry<CT> *adj;
    int32_t *p;
    CT *pc;
    double *g;
    float *g32;
    WalkRec *rec[2];
    WalkBar bar;
    DevCounters *ctr;
    HostSignal *host;
    unsigned seq;
};

template <typename CT, int OCC>  // CTAs per SM
__global__ void __launch_bounds__(kWalkThreads, OCC)
set_policy_kernel(const __grid_constant__ PolicyArgs<CT> a) {
    constexpr int L = 8;  // lanes per row
    const int lane = threadIdx.x & 31, gl = lane & (L - 1);
    unsigned n_open = 0, n_bad = 0;
    bool bad = false;
    if (__ldcg(&a.ctr->insert_late) != 0u) {  // an insertion did not end: its rows are not followed
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            volatile HostSignal *h = a.host;
            h->status = kStatusTimeout;
            __threadfence_system();
            h->seq = a.seq;
        }
        return;
    }

    // the cheapest edge to the parent, for parallel edges
    const int64_t warps = (int64_t)gridDim.x * (kWalkThreads / 32);
    for (int64_t v0 = ((int64_t)blockIdx.x * (kWalkThreads / 32) + (threadIdx.x >> 5)) * (32 / L);
         v0 < a.n; v0 += warps * (32 / L)) {
        const int64_t v = v0 + lane / L;
        int32_t q = -1;
        double best = CUDART_INF;
        if (v < a.n) {
            q = a.parent[v];
            if (v == a.root) {
                if (q != -1) bad = true;
            } else if (q != -1) {
                if (q < 0 || (int64_t)q >= a.n) {
                    bad = true;
                } else {
                    int64_t b, e;
                    row_range(a.rows, v, b, e);
                    for (int64_t i = b + gl; i < e; i += L) {
                        const Entry<CT> en = a.adj[i];
                        if (en.col == q && widen(en.w) < best) best = widen(en.w);
                    }
                }
            }
        }
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1)
            best = fmin(best, __shfl_xor_sync(0xffffffffu, best, o));
        if (gl == 0 && v < a.n) {
            const bool top = v == a.root || q == -1;
            if (!top && best == CUDART_INF) bad = true;
            WalkRec r;
            r.pad = 0;
            r.acc = v == a.root ? 0.0 : best;  // +inf without a parent
            r.anc = top ? -2 : q;
            a.rec[0][v] = r;
            if (top) a.rec[1][v] = r;
        }
    }
    bool ok = walk_sync(a.bar, 0, false, bad, n_open, n_bad);
    if (ok && n_bad == 0u) {
        for (int64_t v = (int64_t)blockIdx.x * kWalkThreads + threadIdx.x; v < a.n;
             v += (int64_t)gridDim.x * kWalkThreads) {
            const int4 r = __ldcg(reinterpret_cast<const int4 *>(a.rec[0] + v));
            const bool linked = r.z >= 0;
            a.p[v] = v == a.root ? kRootMark : linked ? r.z : -1;
            a.pc[v] = linked ? (CT)__hiloint2double(r.y, r.x) : CT(0);
            a.g[v] = v == a.root ? 0.0 : CUDART_INF;
            a.g32[v] = v == a.root ? 0.0f : __int_as_float(0x7f800000);
        }
        ok = walk_rounds(a.rec, a.n, a.bar, n_open, [&](int64_t v, double g) {
            a.g[v] = g;
            a.g32[v] = g32_of(g);
        });
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned status = !ok ? kStatusTimeout : n_bad ? kStatusBadInput
                                : n_open ? kStatusBadTree : 0u;
        // what an earlier exploit found wrong is replaced; a policy that was committed
        // and could not be evaluated stops the next one
        a.ctr->status = status & (kStatusBadTree | kStatusTimeout);
        if (status == 0u) {
            a.ctr->dense = 1u;  // the next Improve sweeps every vertex; the seeded list is moot
            a.ctr->g32_stale = 0u;
        }
        volatile HostSignal *h = a.host;
        h->status = status;
        __threadfence_system();
        h->seq = a.seq;
    }
}

}  // namespace pirrt
