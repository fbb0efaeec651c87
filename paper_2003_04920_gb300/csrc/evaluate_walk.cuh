// Evaluate of a whole policy in one cooperative launch: g(v) = the FP64 sum of
// policy-edge costs up to the root, from a parent array and edge costs alone.
//
// What bounds it is not bandwidth (28 B in and out per vertex) but the chain
// of dependent round trips from the deepest vertex to the root, the grid
// barriers between rounds (2,350 cycles against 302 for a link that hits L2)
// and, from some 10^5 vertices, the rate of scattered loads (one sector per
// cycle and SM).  A round follows three links of the last round's records
// before it meets a barrier, so records span 4^r links after round r.  A link
// is one 16-byte record {cost sum, ancestor}: one load instead of an ancestor,
// a sum and a finishing round from three arrays.  Finished vertices leave
// their g in the record, so no work list is kept: a thread goes over its own
// vertices again, and one that is done costs it one coalesced load.  One CTA
// per SM (152 arrivals at a barrier instead of 1,216), fewer when the policy
// is smaller than that.
//
// Measured, whole calls: 200,003 vertices 236 edges deep 128 -> 44 us, of
// which the kernel 92 -> 27.  Links per round (in one run), at 3,000 / 200,003 / 262,144
// vertices (the last some 800 deep): two 39.8 / 48.2 / 56.6 us, four 38.3 /
// 43.0 / 50.9, eight 42.1 / 49.4 / 62.1.  Three take 35.1 / 39.7 / 46.2, but
// need two additions per factor of three in depth: with four links added in
// pairs (two additions per factor of four) the rounding error is bounded as
// it is for doubling, one addition per factor of two, plus the last one.
// 1,024 threads with two vertices each: 38.7 / 44.0 / 49.2; with four 53.2 /
// 64.5 / 74.4 (64 registers do not hold them).
#pragma once

#include <cfloat>
#include <cstdint>
#include <math_constants.h>

#include "device_common.cuh"

namespace pirrt {

constexpr int kWalkThreads = 512;
constexpr int kWalkLinks = 4;   // links a round sums: its own and three more
constexpr int kWalkSlots = 4;   // vertices a thread follows at once
// After round r every vertex less than 4^r edges deep is done: 16 rounds pass
// any 32-bit vertex count, so vertices open after them lie below a cycle.
constexpr int kWalkRounds = 16;
constexpr int kWalkBarStride = 16;    // 64-bit words between barrier words
constexpr size_t kWalkBarBytes = sizeof(unsigned long long) * kWalkBarStride * (kWalkRounds + 1);
constexpr int kWalkMaxBlocks = 512;   // barrier words count to 1,023

struct __align__(16) WalkRec {
    double acc;   // cost up to anc; g once anc < 0
    int32_t anc;  // ancestor, -1: finished in the last round, -2: before it
    int32_t pad;
};

struct WalkBar {
    unsigned long long *word;  // kWalkRounds + 1 barrier words, kWalkBarStride apart
    unsigned long long call;   // number of this call: larger than any before it on these words
};

struct WalkArgs {
    const int32_t *parent;
    const double *cost;
    double *g;
    WalkRec *rec[2];
    WalkBar bar;
    unsigned *status;         // [0] outcome, [1] raised by a barrier that timed out
    int64_t n;
    int32_t root;
};

// Grid barrier `k` of the call; every CTA brings two flags, and the poll that
// sees the last arrival holds how many CTAs raised each.  The word carries the
// call's number above the counts (10 bits each, grids of at most kWalkMaxBlocks), so
// it needs no clearing between calls: the first arrival of a call replaces
// whatever an older one left.  Bounded: false after kBarrierSpinLimit polls.
__device__ __forceinline__ bool walk_sync(const WalkBar &a, int k, bool open, bool bad,
                                          unsigned &n_open, unsigned &n_bad) {
    __shared__ unsigned s_open, s_bad, s_ok;
    const int o = __syncthreads_or(open), b = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        unsigned long long *word = a.word + kWalkBarStride * k;
        const unsigned long long base = a.call << 30;
        atomicMax(word, base);
        const unsigned long long add = 1ull | (o ? 1ull << 10 : 0ull) | (b ? 1ull << 20 : 0ull);
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"(add) : "memory");
        unsigned long long v, spins = 0;
        s_ok = 1u;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(word) : "memory");
            if (((unsigned)v & 1023u) == gridDim.x && (v >> 30) == a.call) break;
            if (++spins > kBarrierSpinLimit) {
                s_ok = 0u;
                break;
            }
            __nanosleep(20);
        }
        s_open = ((unsigned)v >> 10) & 1023u;
        s_bad = ((unsigned)v >> 20) & 1023u;
    }
    __syncthreads();
    n_open = s_open;
    n_bad = s_bad;
    return s_ok != 0u;
}

// The rounds of a walk over the records rec[0] (and rec[1] for the vertices
// finished at the start), written before the barrier in front.  done(v, g) takes
// each vertex's g; a thread gets the vertices of a grid-stride loop.  False when a
// barrier timed out; n_open > 0 afterwards: vertices below a cycle.
template <typename Done>
__device__ __forceinline__ bool walk_rounds(WalkRec *const (&rec)[2], int64_t n, const WalkBar &bar,
                                            unsigned &n_open, const Done &done_with) {
    constexpr int K = kWalkSlots;
    const int64_t stride = (int64_t)gridDim.x * kWalkThreads;
    const int64_t t0 = (int64_t)blockIdx.x * kWalkThreads + threadIdx.x;
    unsigned none = 0;
    for (int r = 1;; ++r) {
        const WalkRec *rd = rec[(r - 1) & 1];
        WalkRec *wr = rec[r & 1];
        bool open = false;
        for (int64_t base = t0; base < n; base += K * stride) {
            double s[K], low[K], end[K];
            int32_t x[K];
            unsigned work = 0, done = 0;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int64_t v = base + k * stride;
                x[k] = -2;
                s[k] = low[k] = end[k] = 0.0;
                if (v < n) {
                    const int4 q = __ldcg(reinterpret_cast<const int4 *>(rd + v));
                    x[k] = q.z;
                    s[k] = __hiloint2double(q.y, q.x);
                }
                if (x[k] >= 0) work |= 1u << k;
            }
            const unsigned mine = work;
#pragma unroll
            for (int hop = 1; hop < kWalkLinks; ++hop) {
                int4 t[K];
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if ((work >> k) & 1u) t[k] = *reinterpret_cast<const int4 *>(rd + x[k]);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    double add = 0.0;
                    if ((work >> k) & 1u) {
                        const double val = __hiloint2double(t[k].y, t[k].x);
                        if (t[k].z < 0) {
                            end[k] = val;
                            done |= 1u << k;
                            work &= ~(1u << k);
                        } else {
                            add = val;
                            x[k] = t[k].z;
                        }
                    }
                    // links in pairs: (0 + 1) + (2 + 3)
                    if (hop == 1) s[k] += add;
                    if (hop == 2) low[k] = add;
                    if (hop == 3) s[k] += low[k] + add;
                }
            }
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int64_t v = base + k * stride;
                WalkRec o;
                o.pad = 0;
                o.acc = s[k];
                o.anc = x[k];
                if ((done >> k) & 1u) {
                    o.acc = s[k] + end[k];
                    o.anc = -1;
                    done_with(v, o.acc);
                } else if ((mine >> k) & 1u) {
                    open = true;
                } else if (x[k] == -1) {
                    o.anc = -2;  // finished last round: its g goes into the other record too
                } else {
                    continue;
                }
                wr[v] = o;
            }
        }
        if (!walk_sync(bar, r, open, false, n_open, none)) return false;
        if (n_open == 0u || r == kWalkRounds) return true;
    }
}

static __global__ void __launch_bounds__(kWalkThreads, 1)
walk_policy_kernel(const __grid_constant__ WalkArgs a) {
    const int64_t stride = (int64_t)gridDim.x * kWalkThreads;
    const int64_t t0 = (int64_t)blockIdx.x * kWalkThreads + threadIdx.x;
    unsigned n_open = 0, n_bad = 0;

    // Initial values, and the check of the policy before anything follows it:
    // every parent is -1 or an id in [0, n), every used cost finite and >= 0.
    bool bad = false;
    for (int64_t v = t0; v < a.n; v += stride) {
        const int32_t pv = a.parent[v];
        const double c = a.cost[v];
        const bool top = v == a.root || pv == -1;
        WalkRec o;
        o.pad = 0;
        o.acc = v == a.root ? 0.0 : top ? CUDART_INF : c;
        o.anc = top ? -2 : pv;
        a.g[v] = v == a.root ? 0.0 : CUDART_INF;
        a.rec[0][v] = o;
        if (top) a.rec[1][v] = o;
        else if (pv < 0 || (int64_t)pv >= a.n || !(c >= 0.0 && c <= DBL_MAX)) bad = true;
    }
    bool ok = walk_sync(a.bar, 0, false, bad, n_open, n_bad);
    if (ok && n_bad != 0u) {
        if (blockIdx.x == 0 && threadIdx.x == 0) a.status[0] = kStatusBadInput;
        return;
    }

    ok = ok && walk_rounds(a.rec, a.n, a.bar, n_open, [&](int64_t v, double g) { a.g[v] = g; });
    if (threadIdx.x != 0) return;
    if (!ok) *reinterpret_cast<volatile unsigned *>(a.status + 1) = kStatusTimeout;
    else if (blockIdx.x == 0) a.status[0] = n_open ? kStatusBadTree : 0u;
}

}  // namespace pirrt
