// The whole Replan loop (Alg. 2: Improve, test Delta J, Evaluate, repeat) as
// one cooperative launch: every CTA keeps the loop state in shared memory and
// the phases are separated by the grid barrier alone, so an iteration costs no
// kernel launch, no counter reset kernel and no read-back.
//
// The loop is bound by latency, not by bytes: an Evaluate follows tree edges,
// and a tree level is a chain of dependent round trips (row entries, then the
// neighbours' parent and g, then the atomic that lowers g; about 300 cycles each
// from L2, 870 from DRAM, 500 for an atomic) and of one warp's instructions,
// which cost as much again.  So:
//   * a grid barrier carries a count, so the size of the next list needs no
//     further round trip (2,100 cycles with 16 CTAs, 2,350 with 152);
//   * one CTA of 512 threads per SM, 128 registers a thread: two CTAs of 64
//     registers spill in every phase (2-D queries of 10^4 vertices 18.5 against
//     16.5 ms), so they are taken only where an exploit goes over much of a large
//     graph and the loads in flight count; small graphs get as many CTAs as they
//     have work for;
//   * a switched vertex enters the Evaluate with the value Improve computed for
//     it and its row extent, so Evaluate's first level starts at the row;
//   * rows are classified first and their atomics issued by class; few vertices
//     take a warp each, many 8 lanes each (4*10^6 vertices: 73 ms of waves a
//     schedule against 87 with a warp each);
//   * pointer jumping follows several links between two barriers.
// Whole schedules with one launch per iteration in a CUDA-graph WHILE node and seven
// per insertion, and now (insert.cuh included; same GPU): 2-D query of 10^4 vertices
// toward a goal, 100 blocks, 45.8 -> 18.0 ms; 2-D, 2*10^5 vertices, 20 blocks, 50.4 ->
// 24.4 ms; 6-D toward a goal, 10^6 vertices, 14.6 -> 8.0 ms; 6-D, 4*10^6 vertices, 80
// blocks, 163 -> 126 ms.
#pragma once

#include "graph_kernels.cuh"
#include "improve_screen.cuh"

namespace pirrt {

constexpr int kLoopThreads = 512;
constexpr int kLoopWarps = kLoopThreads / 32;
constexpr unsigned kChunk = kLoopThreads;  // vertices a CTA takes from a list at a time
constexpr unsigned kStage = 768;     // lowered children staged per CTA
constexpr unsigned kMarkCap = 2048;  // Improve-list appends staged per CTA

// A vertex to expand: its row [beg, beg + len), the lowered g it carries and its
// depth below the switched vertex it came from.
struct __align__(16) WaveItem {
    long long beg;
    double gu;
    int32_t u, len, depth, pad;
};

// Pointer jumping: the sum of policy-edge costs up to the ancestor anc, or
// (anc < 0) the final g.
struct __align__(16) JumpRec {
    double acc;
    int32_t anc, pad;
};

// What an exploit reports (page-locked host memory, written by the last CTA).
struct LoopResult {
    unsigned long long relax, improved, evaluated, offers, switches;
    unsigned iter, converged, status, wave_epoch;
    unsigned wave_levels, dense_sweeps, jump_rounds, jump_evals, deep;
};

template <typename CT>
struct LoopArgs {
    const RowExt *rows;
    const Entry<CT> *adj;
    double *g;
    float *g32;
    int32_t *p;
    CT *pc;
    unsigned long long *cand;
    unsigned *stamp, *wstamp;
    int32_t *list[2];
    WaveItem *items[2];   // step t reads items[(t & 1) ^ 1], writes items[t & 1]
    JumpRec *rec[2];
    int32_t *dg;          // vertices changed by pointer jumping
    DevCounters *ctr;
    LoopResult *res;
    const float *h;       // goal-directed: heuristic; null = goal-free
    const double *goal_g;
    double eps;
    int64_t n;
    int64_t list_cap;
    int32_t root;
    int32_t jump;         // every Evaluate by pointer jumping
    unsigned jump_above;  // ... or those after more switches than this
    int32_t hops;         // links followed per pointer-jumping round
    int32_t top_rounds;   // FP64 costs: rounds summed from the root down before it
    int32_t walk;         // the policy fits shared memory: each vertex walks up to the root
    unsigned max_iters;
    unsigned dense_limit, max_levels;
    unsigned tail_max, local_levels, local_max, local_step;
};

// What a grid step's warps share.
constexpr unsigned kStepOffersOnly = 1u;  // the list overflowed: no children
constexpr unsigned kStepTraced = 2u;      // this CTA's tiles are traced
struct StepView {
    int32_t *next;
    WaveItem *out;
    unsigned *out_cnt;
    unsigned tag, epoch;
    unsigned flags;
};

struct LoopTrace {
    long long t, tile;
    unsigned long long ns0;
    int state;  // -1 off, -2 between steps, b >= 0 the running step's bucket
};

template <typename CT>
struct LoopShared {
    LoopTrace tr;
    StepView step;
    WaveItem item[2][kStage];  // vertices to expand, and their children; Improve stages
                               // its switches in item[0]
    int32_t mark[kMarkCap];
    int32_t order[kLoopWarps][32];
    unsigned nitem[2];
    unsigned nmark, nfirst, nstage, incomplete, over;
    unsigned base[4];
    unsigned long long dj;
    unsigned long long tot[4];  // relax, improved, evaluated, offers
    unsigned long long scan[kLoopWarps + 2];
    // read by thread 0 after a grid barrier
    unsigned v_ndg, v_next, v_jump, v_flags, v_status, v_ok;
    unsigned rounds, bad;              // of the last pointer jumping
    unsigned barriers, total, direct;  // barriers passed, count of the last one
    unsigned long long seen[2];
    double bound;
};

// The CTA's shared state.
template <typename CT>
__device__ __forceinline__ LoopShared<CT> &loop_shared() {
    extern __shared__ __align__(16) unsigned char loop_smem[];
    return *reinterpret_cast<LoopShared<CT> *>(loop_smem);
}

__device__ __forceinline__ unsigned vld(const unsigned *p) {
    return *reinterpret_cast<const volatile unsigned *>(p);
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release(unsigned long long *p, unsigned long long v) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Grid barrier that also sums one count over the CTAs: a CTA arrives by adding
// 2^40 + its count to a word, so the poll that sees the last arrival holds the
// total as well, with no further round trip.  Two words take turns -- a word is
// added to again only once every CTA has left the barrier before, hence has
// read this one -- and both are 0 at the start of a launch (the CTA that
// reports clears them).  The wait is bounded: on a timeout kStatusTimeout is
// raised and the caller returns.  s.total gets the sum.
template <typename CT>
__device__ __forceinline__ bool loop_sync(DevCounters *c, LoopShared<CT> &sh, unsigned count) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned k = sh.barriers & 1u;
        unsigned long long *word = &c->loop_bar[16u * k];
        const unsigned target = (sh.barriers / 2u + 1u) * gridDim.x;
        red_release(word, (1ull << 40) | (unsigned long long)count);
        unsigned ok = 1u;
        unsigned long long spins = 0, v;
        for (;;) {
            v = ld_acquire(word);
            // arrivals, modulo 2^24
            if ((((unsigned)(v >> 40) - target) & 0x800000u) == 0u) break;
            if (++spins > kBarrierSpinLimit) {
                atomicOr(&c->status, kStatusTimeout);
                ok = 0u;
                break;
            }
            __nanosleep(20);
        }
        const unsigned long long sum = v & ((1ull << 40) - 1ull);
        sh.total = (unsigned)(sum - sh.seen[k]);
        sh.seen[k] = sum;
        ++sh.barriers;
        sh.v_ok = ok;
    }
    __syncthreads();
    return sh.v_ok != 0u;
}

// After a barrier: the iteration's counters, fetched together.  Ends with a
// CTA barrier.
template <typename CT>
__device__ __forceinline__ void loop_fetch(DevCounters *c, LoopCounters *ic, LoopShared<CT> &sh) {
    if (threadIdx.x == 0) {
        const unsigned vd = vld(&ic->n_dg), vn = vld(&ic->n_next), vj = vld(&ic->n_jump);
        const unsigned vf = vld(&ic->flags), vs = vld(&c->status);
        sh.v_ndg = vd;
        sh.v_next = vn;
        sh.v_jump = vj;
        sh.v_flags = vf;
        sh.v_status = vs;
    }
    __syncthreads();
}

// Append the values v[q] of the set bits of mk to the staged Improve list,
// beyond its room straight to the global list.  One lane.
template <typename CT, int U>
__device__ __forceinline__ void stage_marks(LoopShared<CT> &sh, unsigned mk, const int32_t (&v)[U],
                                            int32_t *next, unsigned *n_next) {
    const unsigned n = __popc(mk);
    unsigned k = atomicAdd(&sh.nmark, n), o = 0;
    if (k + n > kMarkCap) o = atomicAdd(n_next, k >= kMarkCap ? n : k + n - kMarkCap);
#pragma unroll
    for (int q = 0; q < U; ++q)
        if ((mk >> q) & 1u) {
            if (k < kMarkCap) sh.mark[k] = v[q];
            else next[o++] = v[q];
            ++k;
        }
}

// Staged appends to the Improve list: one atomic per CTA.  Ends with a CTA
// barrier only if something was staged; call between CTA barriers.
template <typename CT>
__device__ __forceinline__ void flush_marks(LoopShared<CT> &sh, int32_t *next, unsigned *n_next) {
    const unsigned nm = sh.nmark < kMarkCap ? sh.nmark : kMarkCap;
    if (nm == 0u) return;  // uniform
    if (threadIdx.x == 0) sh.base[1] = atomicAdd(n_next, nm);
    __syncthreads();
    for (unsigned i = threadIdx.x; i < nm; i += kLoopThreads) next[sh.base[1] + i] = sh.mark[i];
    __syncthreads();
    if (threadIdx.x == 0) sh.nmark = 0u;
}

__device__ __forceinline__ void add_total(unsigned long long x, unsigned long long *t) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(t, x);
}

// atomicAdd(p, 1), one atomic for the lanes that are here together.
__device__ __forceinline__ unsigned add_one(unsigned *p) {
    const unsigned m = __activemask(), lane = threadIdx.x & 31u;
    const int leader = __ffs(m) - 1;
    unsigned base = 0;
    if ((int)lane == leader) base = atomicAdd(p, (unsigned)__popc(m));
    return __shfl_sync(m, base, leader) + __popc(m & ((1u << lane) - 1u));
}

// A switched vertex, ready for the Evaluate's first step (one lane).  In a sweep that
// switches most of a large graph every vertex gets here, and the CTA's counters set
// its time: 3,000,000 vertices, 24 million entries, eight such sweeps of 1.5 ms with an
// atomic of its own for each switch, 0.7 this way.
template <typename CT>
__device__ __forceinline__ void stage_switch(const LoopArgs<CT> &a, LoopShared<CT> &sh,
                                             LoopCounters *ic, int32_t v, double best,
                                             long long beg, int len, double cur) {
    WaveItem it;
    it.beg = beg;
    it.gu = best;
    it.u = v;
    it.len = len;
    it.depth = 0;
    it.pad = 0;
    const unsigned k = add_one(&sh.nstage);
    if (k < kStage) sh.item[0][k] = it;
    else a.items[1][add_one(&ic->n_switched)] = it;
    // (most lose: the shared maximum is read before its slow atomic)
    const unsigned long long d = (unsigned long long)__double_as_longlong(cur - best);
    if (d > *reinterpret_cast<volatile unsigned long long *>(&sh.dj)) atomicMax(&sh.dj, d);
}

// Improve over a list (from offers, see improve_push.cuh: a vertex whose best
// offer is not below its current value keeps its parent unread) or, with
// dense, over every vertex.  A warp takes up to 32 vertices: one lane each
// decides, then 8 lanes scan each deciding row exactly, four rows at a time.
// Short lists are cut so that every warp has a row; the row extent is loaded
// beside the offer, so a deciding row starts one round trip earlier.
template <typename CT>
__device__ __forceinline__ void loop_improve(const LoopArgs<CT> &a, LoopCounters *ic, const int32_t *list, int64_t count,
                                          bool dense) {
    LoopShared<CT> &sh = loop_shared<CT>();
    constexpr int G = 8, U = 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gl = lane & (G - 1), grp = lane / G;
    const unsigned gmask = ((1u << G) - 1u) << (lane & ~(G - 1));
    const double bound = sh.bound;
    unsigned long long relax = 0;
    unsigned improved = 0;
    const int64_t per = (count + gridDim.x - 1) / gridDim.x;
    const int64_t lo = (int64_t)blockIdx.x * per;
    const int64_t hi = lo + per < count ? lo + per : count;
    int B = 32;
    if (per < (int64_t)kLoopWarps * 32) {
        B = (int)((per + kLoopWarps - 1) / kLoopWarps);
        B = (B + 3) & ~3;
        if (B < 4) B = 4;
    }
    for (int64_t base = lo + (int64_t)warp * B; base < hi; base += (int64_t)kLoopWarps * B) {
        const int64_t i = base + lane;
        bool dec = false;
        int32_t v = -1;
        double cur = CUDART_INF;
        long long beg = 0;
        int len = 0;
        if (lane < B && i < hi) {
            v = dense ? (int32_t)i : __ldcg(&list[i]);
            if (v != a.root) {
                const int32_t pv = __ldcg(&a.p[v]);
                const unsigned long long cb = __ldcg(&a.cand[v]);
                const CT pcv = __ldcg(&a.pc[v]);
                const longlong2 e = __ldg(reinterpret_cast<const longlong2 *>(a.rows) + v);
                if (cb != kCandNone) a.cand[v] = kCandNone;
                if (pv != kRootMark) {
                    if (pv >= 0) cur = a.g[pv] + widen(pcv);
                    const double cv = __longlong_as_double((long long)cb);
                    // goal-directed: an offer that cannot make v promising is
                    // dropped (the row's best is no larger than any offer)
                    dec = dense || (cb < kCandNone && cv < cur && promising(a.h, v, cv, bound));
                    beg = e.x;
                    len = (int)(unsigned)((unsigned long long)e.y & 0xffffffffull);
                    ++improved;
                }
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, dec);
        const int nd = __popc(mask);
        if (nd == 0) continue;
        __syncwarp();
        if (dec) sh.order[warp][__popc(mask & ((1u << lane) - 1u))] = lane;
        __syncwarp();
        for (int r0 = 0; r0 < nd; r0 += 32 / G) {
            const int k = r0 + grp;
            const bool mine = k < nd;
            const int src = mine ? sh.order[warp][k] : 0;
            const int32_t sv = __shfl_sync(0xffffffffu, v, src);
            const double scur = __shfl_sync(0xffffffffu, cur, src);
            const long long b = __shfl_sync(0xffffffffu, beg, src);
            const int n = __shfl_sync(0xffffffffu, len, src);
            unsigned long long bv = kCandNone + 1ull;
            int32_t bid = INT_MAX;
            CT bw = CT(0);
            if (mine) {
                const Entry<CT> *row = a.adj + b;
                for (int i0 = gl; i0 < n; i0 += G * U) {
                    Entry<CT> en[U];
                    double gv[U];
#pragma unroll
                    for (int q = 0; q < U; ++q)
                        if (i0 + q * G < n) en[q] = ld_stream(&row[i0 + q * G]);
#pragma unroll
                    for (int q = 0; q < U; ++q)
                        gv[q] = (i0 + q * G < n) ? a.g[en[q].col] : CUDART_INF;
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        if (i0 + q * G < n) {
                            const unsigned long long vb =
                                (unsigned long long)__double_as_longlong(gv[q] + widen(en[q].w));
                            if (vb < bv || (vb == bv && (en[q].col < bid ||
                                                         (en[q].col == bid && en[q].w < bw)))) {
                                bv = vb;
                                bid = en[q].col;
                                bw = en[q].w;
                            }
                        }
                    }
                }
            }
#pragma unroll
            for (int off = G / 2; off > 0; off >>= 1) {
                const unsigned long long ov = __shfl_xor_sync(gmask, bv, off, G);
                const int32_t oi = __shfl_xor_sync(gmask, bid, off, G);
                const CT ow = __shfl_xor_sync(gmask, bw, off, G);
                if (ov < bv || (ov == bv && (oi < bid || (oi == bid && ow < bw)))) {
                    bv = ov;
                    bid = oi;
                    bw = ow;
                }
            }
            if (mine && gl == 0) {
                relax += (unsigned long long)n;
                if (bv < kCandNone) {
                    const double best = __longlong_as_double((long long)bv);
                    if (best < scur && promising(a.h, sv, best, bound)) {
                        a.p[sv] = bid;
                        a.pc[sv] = bw;
                        stage_switch<CT>(a, sh, ic, sv, best, b, n, scur);
                    }
                }
            }
        }
    }
    add_total(relax, &sh.tot[0]);
    add_total(improved, &sh.tot[1]);
}

// Dense sweep for FP32 costs: 4 lanes per vertex, candidates screened in FP32
// and decided exactly (improve_screen.cuh gives the margin), next vertex's row
// extent and next batch of entries requested ahead.  Offers start afresh.
__device__ __forceinline__ void loop_dense_screen(const LoopArgs<float> &a, LoopCounters *ic) {
    LoopShared<float> &sh = loop_shared<float>();
    constexpr int G = 4, kU = 4;
    constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;
    const int lane = threadIdx.x & 31, gl = threadIdx.x & (G - 1);
    const unsigned gmask = ((1u << G) - 1u) << (lane & ~(G - 1));
    const int64_t gstride = (int64_t)gridDim.x * (kLoopThreads / G);
    const float kInf = __int_as_float(0x7f800000);
    const double bound = sh.bound;
    unsigned long long relax = 0;
    unsigned improved = 0;
    const int64_t t0 = (int64_t)blockIdx.x * kLoopThreads + threadIdx.x;
    for (int64_t v = t0; v < a.n; v += (int64_t)gridDim.x * kLoopThreads) a.cand[v] = kCandNone;
    int64_t nb = 0, ne = 0;
    int64_t item = t0 / G;
    if (item < a.n) row_range(a.rows, item, nb, ne);
    for (; item < a.n; item += gstride) {
        const int32_t v = (int32_t)item;
        const int64_t b = nb, e = ne;
        if (item + gstride < a.n) row_range(a.rows, item + gstride, nb, ne);
        if (v == a.root) continue;  // uniform within the group
        int32_t pv = -1;
        float pcv = 0.f;
        double gp = CUDART_INF;
        if (gl == 0) {
            pv = __ldcg(&a.p[v]);
            pcv = __ldcg(&a.pc[v]);
            if (pv >= 0) gp = a.g[pv];
        }
        float m1 = kInf, m2 = kInf;
        int64_t i1 = -1;
        int exact_row = 0;
        Entry<float> en[kU];
        int64_t i0 = b + gl;
#pragma unroll
        for (int q = 0; q < kU; ++q)
            if (i0 + q * G < e) en[q] = ld_stream(&a.adj[i0 + q * G]);
        for (; i0 < e; i0 += (int64_t)G * kU) {
            float gu[kU];
#pragma unroll
            for (int q = 0; q < kU; ++q)
                if (i0 + q * G < e) gu[q] = a.g32[en[q].col];
            Entry<float> nx[kU];
            const int64_t i1n = i0 + (int64_t)G * kU;
#pragma unroll
            for (int q = 0; q < kU; ++q)
                if (i1n + q * G < e) nx[q] = ld_stream(&a.adj[i1n + q * G]);
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                if (i0 + q * G < e) {
                    const float av = gu[q] + en[q].w;
                    exact_row |= (gu[q] < 0.f) | (isinf(av) & !isinf(gu[q]));
                    if (av < m1) {
                        m2 = m1;
                        m1 = av;
                        i1 = i0 + q * G;
                    } else if (av < m2) {
                        m2 = av;
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < kU; ++q) en[q] = nx[q];
        }
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) {
            const float om1 = __shfl_xor_sync(gmask, m1, off, G);
            const float om2 = __shfl_xor_sync(gmask, m2, off, G);
            const int64_t oi1 = __shfl_xor_sync(gmask, i1, off, G);
            exact_row |= __shfl_xor_sync(gmask, exact_row, off, G);
            const float lo = fminf(m1, om1), hi = fmaxf(m1, om1);
            if (om1 < m1 || (om1 == m1 && oi1 >= 0 && (i1 < 0 || oi1 < i1))) i1 = oi1;
            m2 = fminf(hi, fminf(m2, om2));
            m1 = lo;
        }
        // exact FP64 lexicographic minimum over the candidates in play
        unsigned long long bv = kInfBits + 1ull;
        int32_t bid = INT_MAX;
        unsigned bw = 0xffffffffu;
        const float tau = m1 * (1.0f + 0x1p-20f) + 0x1p-125f;
        const bool rescan = exact_row || (m2 <= tau && !isinf(m1));
        if (rescan) {
            for (int64_t i = b + gl; i < e; i += G) {
                const Entry<float> x = a.adj[i];
                if (exact_row || a.g32[x.col] + x.w <= tau) {
                    const unsigned long long vb = (unsigned long long)__double_as_longlong(
                        a.g[x.col] + widen(x.w));
                    const unsigned wb = __float_as_uint(x.w);
                    if (vb < bv || (vb == bv && (x.col < bid || (x.col == bid && wb < bw)))) {
                        bv = vb;
                        bid = x.col;
                        bw = wb;
                    }
                }
            }
#pragma unroll
            for (int off = G / 2; off > 0; off >>= 1) {
                const unsigned long long ov = __shfl_xor_sync(gmask, bv, off, G);
                const int32_t oi = __shfl_xor_sync(gmask, bid, off, G);
                const unsigned ow = __shfl_xor_sync(gmask, bw, off, G);
                if (ov < bv || (ov == bv && (oi < bid || (oi == bid && ow < bw)))) {
                    bv = ov;
                    bid = oi;
                    bw = ow;
                }
            }
        } else if (gl == 0 && i1 >= 0 && !isinf(m1)) {
            const Entry<float> x = a.adj[i1];
            bv = (unsigned long long)__double_as_longlong(a.g[x.col] + widen(x.w));
            bid = x.col;
            bw = __float_as_uint(x.w);
        }
        if (gl == 0 && pv != kRootMark) {
            const double cur = pv >= 0 ? gp + widen(pcv) : CUDART_INF;
            if (bv <= kInfBits) {
                const double best = __longlong_as_double((long long)bv);
                if (best < cur && promising(a.h, v, best, bound)) {
                    a.p[v] = bid;
                    a.pc[v] = __uint_as_float(bw);
                    stage_switch<float>(a, sh, ic, v, best, b, (int)(e - b), cur);
                }
            }
            relax += (unsigned long long)(e - b);
            ++improved;
        }
    }
    __syncwarp();
    add_total(relax, &sh.tot[0]);
    add_total(improved, &sh.tot[1]);
}

// Expand the vertices it (one per L lanes; len 0: none): scan the row, lower
// the children by an atomic minimum, offer the other neighbours their candidate
// where it beats their g, and list them for the next Improve (the reasoning
// stands at wave_tile).  Lowered children that are to be expanded go to the
// CTA's stage `nx`.  The row entries are classified first and the atomics issued
// by class, so that a row costs few instructions: one warp's instruction chain,
// not the memory, sets the time of a thin level.
template <typename CT, int L, int U>
__device__ __forceinline__ void expand(const LoopArgs<CT> &a, LoopShared<CT> &sh, LoopCounters *ic,
                                       const StepView &s, const WaveItem &it, unsigned nx,
                                       bool offering, unsigned &recomputed, unsigned &first) {
    const unsigned lane = threadIdx.x & 31u;
    const int gl = (int)(lane & (unsigned)(L - 1));
    const bool nochild =
        (s.flags & kStepOffersOnly) != 0u || (unsigned)it.depth >= a.max_levels;
    const int32_t u = nochild ? INT_MIN : it.u;  // no parent: every neighbour is offered to
    const int depth = it.depth + 1, len = it.len;
    const Entry<CT> *row = a.adj + it.beg;
    for (int e0 = gl; __any_sync(0xffffffffu, e0 - gl < len); e0 += L * U) {
        int32_t col[U];
        unsigned long long val[U];
        Entry<CT> en[U];
#pragma unroll
        for (int q = 0; q < U; ++q)
            if (e0 + L * q < len) en[q] = ld_stream(&row[e0 + L * q]);
        int32_t px[U];
        unsigned long long gold[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            gold[q] = 0ull;  // no value is below it
            px[q] = -2;
            col[q] = 0;
            if (e0 + L * q < len) {
                col[q] = en[q].col;
                px[q] = __ldcg(&a.p[col[q]]);
                gold[q] = __ldcg(reinterpret_cast<const unsigned long long *>(a.g) + col[q]);
            }
        }
        unsigned cm = 0, om = 0;
#pragma unroll
        for (int q = 0; q < U; ++q) {
            // non-negative doubles order like their bit patterns
            val[q] = 0ull;
            if (e0 + L * q < len)
                val[q] = (unsigned long long)__double_as_longlong(it.gu + widen(en[q].w));
            const bool less = val[q] < gold[q];
            const bool child = px[q] == u;
            if (less && child) cm |= 1u << q;
            if (less && !child) om |= 1u << q;
        }
        if (!offering) om = 0u;
        unsigned mk = 0;
#pragma unroll
        for (int q = 0; q < U; ++q)
            if ((om >> q) & 1u) {
                atomicMin(a.cand + col[q], val[q]);
                if (atomicExch(&a.stamp[col[q]], s.epoch) != s.epoch) mk |= 1u << q;
            }
        // one child per lane and turn (a row seldom holds more)
        while (__any_sync(0xffffffffu, cm != 0u)) {
            if (cm) {
                int32_t cc = 0;
                unsigned long long cv = 0ull;
                const unsigned bit = cm & (0u - cm);
                cm ^= bit;
#pragma unroll
                for (int q = 0; q < U; ++q)
                    if (bit == (1u << q)) {
                        cc = col[q];
                        cv = val[q];
                    }
                const longlong2 ext = __ldg(reinterpret_cast<const longlong2 *>(a.rows) + cc);
                const bool prom =
                    promising(a.h, cc, __longlong_as_double((long long)cv), sh.bound);
                const unsigned long long old =
                    atomicMin(reinterpret_cast<unsigned long long *>(&a.g[cc]), cv);
                // counted once; a vertex another expansion lowered further in
                // between has changed as well
                if (atomicExch(&a.wstamp[cc], s.tag) != s.tag) ++first;
                if (old > cv) {
                    ++recomputed;
                    if ((unsigned)depth >= a.max_levels) sh.incomplete = 1u;
                    if (prom) {
                        WaveItem c;
                        c.beg = ext.x;
                        c.gu = __longlong_as_double((long long)cv);
                        c.u = cc;
                        c.len = (int)(unsigned)((unsigned long long)ext.y & 0xffffffffull);
                        c.depth = depth;
                        c.pad = 0;
                        const unsigned k = atomicAdd(&sh.nitem[nx], 1u);
                        if (k < kStage) {
                            sh.item[nx][k] = c;
                        } else {
                            atomicAdd(&sh.direct, 1u);
                            const unsigned o = atomicAdd(s.out_cnt, 1u);
                            if ((int64_t)o < a.list_cap) s.out[o] = c;
                        }
                    }
                }
            }
        }
        if (mk) stage_marks<CT, U>(sh, mk, col, s.next, &ic->n_next);
    }
}

// Expand the n vertices of stage `cur` (their children go to the other stage):
// few of them, a warp each and the whole row at once, the shortest chain; more,
// 8 lanes each and 40 entries at a time, the fewest instructions per entry.
template <typename CT>
__device__ __forceinline__ void expand_stage(const LoopArgs<CT> &a, LoopShared<CT> &sh,
                                             LoopCounters *ic, const StepView &s, unsigned cur,
                                             unsigned n) {
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    unsigned recomputed = 0, first = 0;
    unsigned long long offers = 0;
    // past the dense limit the offers are not needed: the warp with the least to
    // do publishes the CTA's first changes and looks at the count
    if (threadIdx.x == kLoopThreads - 32) {
        const unsigned f = atomicExch(&sh.nfirst, 0u);
        if ((f ? atomicAdd(&ic->n_dg, f) + f : vld(&ic->n_dg)) > a.dense_limit) sh.over = 1u;
    }
    if (n <= 2u * kLoopWarps) {
        for (unsigned i = warp; i < n; i += kLoopWarps) {
            const WaveItem it = sh.item[cur][i];
            const bool offering = vld(&sh.over) == 0u;
            expand<CT, 32, 2>(a, sh, ic, s, it, cur ^ 1u, offering, recomputed, first);
            if (lane == 0 && offering) offers += (unsigned)it.len;
        }
    } else {
        for (unsigned i0 = 4u * warp; i0 < n; i0 += 4u * kLoopWarps) {
            WaveItem it;
            it.len = it.depth = it.u = 0;
            it.beg = 0;
            it.gu = 0.0;
            const unsigned i = i0 + (lane >> 3);
            if (i < n) it = sh.item[cur][i];
            const bool offering = vld(&sh.over) == 0u;
            expand<CT, 8, 5>(a, sh, ic, s, it, cur ^ 1u, offering, recomputed, first);
            if ((lane & 7u) == 0u && offering) offers += (unsigned)it.len;
            if (warp == 0u) {  // in a wide step, more often
                const unsigned f = __reduce_add_sync(0xffffffffu, first);
                first = 0u;
                if (lane == 0 && f && atomicAdd(&ic->n_dg, f) + f > a.dense_limit) sh.over = 1u;
            }
        }
    }
    first = __reduce_add_sync(0xffffffffu, first);
    if (lane == 0 && first) atomicAdd(&sh.nfirst, first);
    add_total(recomputed, &sh.tot[2]);
    add_total(offers, &sh.tot[3]);
}

// Hand the n staged vertices of stage k to the next step's list, the staged
// Improve-list entries to theirs and the first changes to their counter, one
// atomic each, together.  Whole CTA, after a CTA barrier; ends with one.
template <typename CT>
__device__ __forceinline__ void step_flush(const LoopArgs<CT> &a, LoopShared<CT> &sh,
                                           LoopCounters *ic, const StepView &s, unsigned k,
                                           unsigned n) {
    const unsigned nm = sh.nmark < kMarkCap ? sh.nmark : kMarkCap;
    if (threadIdx.x == 0 && n) sh.base[0] = atomicAdd(s.out_cnt, n);
    if (threadIdx.x == 32 && nm) sh.base[1] = atomicAdd(&ic->n_next, nm);
    if (threadIdx.x == 64 && sh.nfirst) {
        if (atomicAdd(&ic->n_dg, sh.nfirst) + sh.nfirst > a.dense_limit) sh.over = 1u;
    }
    if (threadIdx.x == 96 && sh.incomplete) atomicOr(&ic->flags, kLoopIncomplete);
    __syncthreads();
    if (n) {
        const uint4 *from = reinterpret_cast<const uint4 *>(sh.item[k]);
        uint4 *to = reinterpret_cast<uint4 *>(s.out + sh.base[0]);
        const int64_t room = 2 * (a.list_cap - (int64_t)sh.base[0]);
        for (unsigned i = threadIdx.x; i < 2u * n && (int64_t)i < room; i += kLoopThreads)
            to[i] = from[i];
    }
    for (unsigned i = threadIdx.x; i < nm; i += kLoopThreads) s.next[sh.base[1] + i] = sh.mark[i];
    if (threadIdx.x == 0) {
        sh.direct += n;
        sh.nitem[k] = 0u;
        sh.nmark = 0u;
        sh.nfirst = 0u;
        sh.incomplete = 0u;
    }
    __syncthreads();
}

// Level trace of CTA 0's thread 0 while tracing (profile fields level_*,
// share_*, local_*, wave_*): a grid step's cycles run from its start to the next
// one's, a tile's from its start to the barrier that ends it.
__device__ __forceinline__ unsigned long long loop_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void trace_iteration(DevCounters *c, LoopTrace &tr, unsigned iter) {
    if (tr.state == -1) return;
    tr.state = -2;
    tr.t = clock64();
    const unsigned long long now = loop_ns();
    if (iter > 0u) {
        c->gap_ns += now - tr.ns0;  // tr.ns0: end of the iteration before
        c->gaps += 1ull;
    }
    tr.ns0 = now;
}

__device__ __forceinline__ void trace_step(DevCounters *c, LoopTrace &tr, long long count) {
    if (tr.state == -1) return;
    const long long now = clock64();
    const unsigned long long d = (unsigned long long)(now - tr.t);
    if (tr.state == -2) c->ph_pre_cyc += d;
    else {
        c->lvl_cyc[tr.state] += d;
    }
    tr.t = now;
    tr.state = -2;
    if (count > 0) {
        int b = 64 - __clzll((unsigned long long)count);
        if (b >= kLevelBuckets) b = kLevelBuckets - 1;
        c->lvl_n[b] += 1ull;
        c->lvl_items[b] += (unsigned long long)count;
        tr.state = b;
    }
}

// A tile of nv vertices (its start in shared memory: a register held across the
// expansion spills).
__device__ __forceinline__ void trace_tile_start(LoopTrace &tr) {
    if (threadIdx.x == 0) tr.tile = clock64();
}
__device__ __forceinline__ void trace_tile(LoopTrace &tr, unsigned long long *n,
                                           unsigned long long *items, unsigned long long *cyc,
                                           unsigned nv) {
    if (threadIdx.x != 0) return;
    int b = 32 - __clz(nv);
    if (b >= kLevelBuckets) b = kLevelBuckets - 1;
    n[b] += 1ull;
    items[b] += (unsigned long long)nv;
    cyc[b] += (unsigned long long)(clock64() - tr.tile);
}

__device__ __forceinline__ void trace_end(DevCounters *c, LoopTrace &tr) {
    if (tr.state == -1) return;
    c->ph_post_cyc += (unsigned long long)(clock64() - tr.t);
    const unsigned long long now = loop_ns();
    c->span_ns += now - tr.ns0;
    c->spans += 1ull;
    c->ph_calls += 1ull;
    tr.ns0 = now;
}

// One CTA's part of a grid step: its share [lo, hi) of the step's list, a chunk
// at a time, then, where `levels` allows, the lowered children on its own, tree
// level by tree level, while there are at most `limit` of them.  What is left
// joins the next step's list.  Returns what the CTA added to that list.
template <typename CT>
__device__ __forceinline__ unsigned loop_step(const LoopArgs<CT> &a, LoopCounters *ic, const WaveItem *in, bool switched,
                                           int64_t lo, int64_t hi, unsigned levels,
                                           unsigned limit) {
    LoopShared<CT> &sh = loop_shared<CT>();
    const StepView s = sh.step;
    unsigned cur = 0;
    for (int64_t c0 = lo; c0 < hi; c0 += kChunk) {
        if (s.flags & kStepTraced) trace_tile_start(sh.tr);
        const unsigned n = hi - c0 < (int64_t)kChunk ? (unsigned)(hi - c0) : kChunk;
        unsigned gone = 0;
        if (threadIdx.x < n) {
            const longlong2 *q = reinterpret_cast<const longlong2 *>(in + c0 + threadIdx.x);
            const longlong2 x = __ldcg(q), y = __ldcg(q + 1);
            WaveItem it;
            it.beg = x.x;
            it.gu = __longlong_as_double(x.y);
            it.u = (int)(unsigned)((unsigned long long)y.x & 0xffffffffull);
            it.len = (int)(unsigned)((unsigned long long)y.x >> 32);
            it.depth = (int)(unsigned)((unsigned long long)y.y & 0xffffffffull);
            it.pad = 0;
            if (switched) {
                // every switched vertex takes the value Improve found for it
                gone = 1u;
                const unsigned long long b = (unsigned long long)__double_as_longlong(it.gu);
                const unsigned long long old =
                    atomicMin(reinterpret_cast<unsigned long long *>(&a.g[it.u]), b);
                if (old > b) {
                    if (atomicExch(&a.wstamp[it.u], s.tag) != s.tag) atomicAdd(&sh.nfirst, 1u);
                    if (promising(a.h, it.u, it.gu, sh.bound)) gone = 0u;
                }
                if (gone) it.len = 0;
            }
            sh.item[cur][threadIdx.x] = it;
        }
        if ((s.flags & kStepOffersOnly) && threadIdx.x == 0) sh.incomplete = 1u;
        if (switched && threadIdx.x == 0) sh.tot[2] += n;
        __syncthreads();
        expand_stage<CT>(a, sh, ic, s, cur, n);
        __syncthreads();
        if (s.flags & kStepTraced)
            trace_tile(sh.tr, a.ctr->shr_n, a.ctr->shr_items, a.ctr->shr_cyc, n);
        if (c0 + kChunk < hi && (sh.nitem[cur ^ 1u] > kStage / 2 || sh.nmark > kMarkCap / 2))
            step_flush<CT>(a, sh, ic, s, cur ^ 1u,
                           sh.nitem[cur ^ 1u] < kStage ? sh.nitem[cur ^ 1u] : kStage);
    }
    for (unsigned l = 0;; ++l) {
        const unsigned m = sh.nitem[cur ^ 1u], n = m < kStage ? m : kStage;
        if (n == 0u || l >= levels || m > limit) break;
        if (s.flags & kStepTraced) trace_tile_start(sh.tr);
        cur ^= 1u;
        __syncthreads();  // every thread has read the count
        expand_stage<CT>(a, sh, ic, s, cur, n);
        __syncthreads();
        if (s.flags & kStepTraced)
            trace_tile(sh.tr, a.ctr->loc_n, a.ctr->loc_items, a.ctr->loc_cyc, n);
        if (threadIdx.x == 0) sh.nitem[cur] = 0u;
    }
    const unsigned k = cur ^ 1u, m = sh.nitem[k];
    step_flush<CT>(a, sh, ic, s, k, m < kStage ? m : kStage);
    const unsigned made = sh.direct;
    __syncthreads();
    if (threadIdx.x == 0) sh.direct = 0u;
    return made;
}

// One round over every vertex that follows at most kTopLinks links and finishes
// the vertices it finds a finished ancestor (or the root) for, adding the links'
// costs from that ancestor down -- Alg. 2's sums bit for bit, which pointer
// jumping reassociates.  Each such round finishes kTopLinks more tree levels, so
// it serves shallow trees: FP64 costs, whose sums round.  An unfinished
// vertex's record stays its own link, from which pointer jumping can go on.
constexpr int kTopLinks = 12;

template <typename CT>
__device__ __forceinline__ bool top_round(const LoopArgs<CT> &a, LoopCounters *ic, unsigned r,
                                          bool stale, unsigned &finished) {
    LoopShared<CT> &sh = loop_shared<CT>();
    JumpRec *wr = a.rec[r & 1u];
    const JumpRec *rd = a.rec[(r & 1u) ^ 1u];
    bool open = false;
    for (int64_t base = (int64_t)blockIdx.x * kLoopThreads; base < a.n;
         base += (int64_t)gridDim.x * kLoopThreads) {
        const int64_t v = base + threadIdx.x;
        bool changed = false;
        if (v < a.n) {
            JumpRec o;
            o.pad = 0;
            double link;
            int32_t x;
            if (r == 1u) {
                x = __ldcg(&a.p[v]);
                link = widen(__ldcg(&a.pc[v]));
                if (x < 0) x = -3;
            } else {
                const int4 q = __ldcg(reinterpret_cast<const int4 *>(rd + v));
                x = q.z;
                link = __hiloint2double(q.y, q.x);
            }
            if (x >= 0) {
                double cost[kTopLinks];
                const int32_t parent = x;
                double end = 0.0;
                int found = -1;  // links below the finished ancestor, less one
#pragma unroll
                for (int k = 1; k < kTopLinks; ++k) cost[k] = 0.0;
                cost[0] = link;
#pragma unroll
                for (int k = 0; k < kTopLinks; ++k) {
                    if (found < 0) {
                        int32_t nx;
                        double add;
                        if (r == 1u) {
                            nx = a.p[x];
                            add = widen(a.pc[x]);
                        } else {
                            const int4 t = *reinterpret_cast<const int4 *>(rd + x);
                            nx = t.z;
                            add = __hiloint2double(t.y, t.x);
                        }
                        if (nx < 0) {
                            end = r == 1u ? a.g[x] : add;
                            found = k;
                        } else if (k + 1 < kTopLinks) {
                            cost[k + 1] = add;
                            x = nx;
                        }
                    }
                }
                if (found >= 0) {
                    double gw = end;
#pragma unroll
                    for (int k = kTopLinks - 1; k >= 0; --k)
                        if (k <= found) gw = gw + cost[k];
                    const double old = __ldcg(&a.g[v]);
                    changed = __double_as_longlong(gw) != __double_as_longlong(old);
                    if (changed) a.g[v] = gw;
                    if (changed || stale) a.g32[v] = g32_of(gw);
                    ++finished;
                    o.acc = gw;
                    o.anc = -1;
                } else {
                    open = true;
                    o.acc = link;
                    o.anc = parent;
                }
                wr[v] = o;
            } else if (x == -1) {
                o.acc = link;
                o.anc = -2;
                wr[v] = o;
            } else if (x == -3) {
                o.acc = 0.0;
                o.anc = -2;  // no parent: nothing to do in any round
                a.rec[0][v] = o;
                a.rec[1][v] = o;
            }
        }
        if (changed) sh.mark[atomicAdd(&sh.nmark, 1u)] = (int32_t)v;
        __syncthreads();
        flush_marks<CT>(sh, a.dg, &ic->n_jump);
        __syncthreads();
    }
    return open;
}

// Pointer jumping over every vertex (any grid): g(v) = the sum of policy-edge
// costs up to the root.  Between two grid barriers a vertex follows up to
// `hops` + 1 links of the last round's records (a barrier costs several links'
// round trips), so a chain of length L takes about log_(hops + 1) L rounds;
// the first round follows p and pc themselves.  Every record read in a round
// was written before it, so the sums do not depend on scheduling.  Changed
// vertices are listed in a.dg.  Returns false when a barrier timed out;
// *rounds gets the rounds run.
template <typename CT>
__device__ __forceinline__ bool loop_jump(const LoopArgs<CT> &a, LoopCounters *ic, bool stale) {
    LoopShared<CT> &sh = loop_shared<CT>();
    DevCounters *c = a.ctr;
    constexpr int K = 2;  // vertices a thread follows at once: their links' round trips overlap
    const int64_t stride = (int64_t)gridDim.x * kLoopThreads;
    const int64_t t0 = (int64_t)blockIdx.x * kLoopThreads + threadIdx.x;
    unsigned finished = 0;
    unsigned r = 1;
    for (;; ++r) {
        JumpRec *wr = a.rec[r & 1u];
        const JumpRec *rd = a.rec[(r & 1u) ^ 1u];
        bool open = false;
        bool top = false;
        if constexpr (sizeof(CT) == 8) {
            top = r <= (unsigned)a.top_rounds;
            if (top) open = top_round<CT>(a, ic, r, stale, finished);
        }
        for (int64_t base = top ? a.n + threadIdx.x : t0; base - threadIdx.x < a.n; base += K * stride) {
            double s[K], end[K];
            int32_t x[K];
            unsigned work = 0, done = 0;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int64_t v = base + k * stride;
                s[k] = end[k] = 0.0;
                x[k] = -2;
                if (v < a.n) {
                    if (r == 1u) {
                        x[k] = __ldcg(&a.p[v]);
                        s[k] = widen(__ldcg(&a.pc[v]));
                        if (x[k] < 0) x[k] = -3;
                    } else {
                        const int4 q = __ldcg(reinterpret_cast<const int4 *>(rd + v));
                        x[k] = q.z;
                        s[k] = __hiloint2double(q.y, q.x);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (x[k] >= 0) work |= 1u << k;
            const unsigned mine = work;
            for (int hop = 0; hop <= a.hops && work; ++hop) {
                // every open vertex follows one link
                int32_t nx[K];
                double add[K];
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    nx[k] = 0;
                    add[k] = 0.0;
                    if ((work >> k) & 1u) {
                        if (r == 1u) {
                            nx[k] = a.p[x[k]];
                            add[k] = widen(a.pc[x[k]]);
                        } else {
                            const int4 t = *reinterpret_cast<const int4 *>(rd + x[k]);
                            nx[k] = t.z;
                            add[k] = __hiloint2double(t.y, t.x);
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if ((work >> k) & 1u) {
                        if (nx[k] < 0) {
                            end[k] = r == 1u ? a.g[x[k]] : add[k];
                            done |= 1u << k;
                            work &= ~(1u << k);
                        } else if (hop < a.hops) {
                            s[k] += add[k];
                            x[k] = nx[k];
                        }
                    }
            }
            unsigned changed = 0;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int64_t v = base + k * stride;
                JumpRec o;
                o.pad = 0;
                if ((done >> k) & 1u) {
                    const double gw = s[k] + end[k];
                    const double old = __ldcg(&a.g[v]);
                    const bool diff = __double_as_longlong(gw) != __double_as_longlong(old);
                    if (diff) {
                        a.g[v] = gw;
                        changed |= 1u << k;
                    }
                    // a wave leaves the FP32 shadow behind: every one is rewritten then
                    if (diff || stale) a.g32[v] = g32_of(gw);
                    ++finished;
                    o.acc = gw;
                    o.anc = -1;
                    wr[v] = o;
                } else if ((mine >> k) & 1u) {
                    open = true;
                    o.acc = s[k];
                    o.anc = x[k];
                    wr[v] = o;
                } else if (x[k] == -1) {
                    // finished last round: leave the value in both records
                    o.acc = s[k];
                    o.anc = -2;
                    wr[v] = o;
                } else if (x[k] == -3) {
                    o.acc = 0.0;
                    o.anc = -2;  // no parent: nothing to do in any round
                    a.rec[0][v] = o;
                    a.rec[1][v] = o;
                }
            }
            // list the changed vertices, staged in the mark buffer
            if (changed) {
                const unsigned n = __popc(changed);
                unsigned at = atomicAdd(&sh.nmark, n);
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if ((changed >> k) & 1u) sh.mark[at++] = (int32_t)(base + k * stride);
            }
            if (base - threadIdx.x + K * stride < a.n) {  // another pass: make room
                __syncthreads();
                flush_marks<CT>(sh, a.dg, &ic->n_jump);
                __syncthreads();
            }
        }
        const unsigned left = __syncthreads_or(open) ? 1u : 0u;
        flush_marks<CT>(sh, a.dg, &ic->n_jump);
        if (!loop_sync<CT>(c, sh, left)) return false;
        if (sh.total == 0u || r >= (unsigned)kMaxJumpRounds) break;
    }
    // every CTA knows of vertices left over: their parents form a cycle
    if (threadIdx.x == 0) {
        sh.rounds = r;
        sh.bad = sh.total;
        if (sh.total != 0u && blockIdx.x == 0) atomicOr(&c->status, kStatusBadTree);
    }
    add_total(finished, &sh.tot[2]);
    return true;
}

// The same for a policy that fits shared memory: every CTA loads all of it
// (coalesced, out of L2) and walks up from its own vertices, a link being a
// shared-memory round trip (some 30 cycles) instead of an L2 one (302), to the
// root in one go: no records, no rounds, one barrier.  With FP32 costs a vertex's
// sum runs from itself upwards, as in loop_jump; with FP64 costs, whose sums
// round, the links are kept on a stack and added from the root down, as Alg. 2
// adds them, up to the depth that top_round covers.  A vertex deeper than that, or
// below a cycle, sends the whole Evaluate to loop_jump (and the rest of the exploit
// goes there at once): every CTA first puts back what it wrote and the list of
// changed vertices starts empty, because pointer jumping may round the same sums
// differently, and a vertex listed by both would not fit the list, which has room
// for each vertex once.
// At most 128 vertices a CTA (64 with stacks): with one warp per scheduler the
// slow FP64 additions hide behind the loads.
//
// Measured, ms of exploit by loop_jump and by loop_walk: 10,000 vertices in 2-D in
// 100 goal-directed blocks 16.7 and 15.2, 3,000 in 20 blocks 3.52 and 2.81, 10,000
// in 6-D in 10 blocks 1.48 and 1.22; a policy of 2,000 with FP64 costs 0.241 and
// 0.145, of 9,500 0.65 and 0.32; FP64 blocks up to 9,700 in 2-D 6.9 and 3.6.  The
// limits are what shared memory holds beside the loop's own; at 16,000 vertices
// 0.434 and 0.408, at 19,000 (where the L1 cache left over shrinks further) 0.416
// and 0.445.
constexpr int64_t kWalkVertices = 16384, kWalkVerticesF64 = 9728;
constexpr int kWalkPer = 128;    // vertices of a CTA: one warp per scheduler
constexpr int kWalkPerF64 = 64;  // ... FP64 costs, whose stacks take room
constexpr int kWalkDepth = 96;   // FP64 costs: links kept to be added from the root down

// Shared memory beyond LoopShared.
template <typename CT>
constexpr size_t walk_bytes(int64_t n) {
    return sizeof(CT) == 4 ? 8 * (size_t)((n + 3) & ~3ll)
                           : 12 * (size_t)((n + 3) & ~3ll) + 8 * (size_t)(kWalkDepth * kWalkPerF64);
}

template <typename CT>
__device__ __forceinline__ bool loop_walk(const LoopArgs<CT> &a, LoopCounters *ic, bool stale,
                                          bool &walk) {
    LoopShared<CT> &sh = loop_shared<CT>();
    constexpr size_t kAt = (sizeof(LoopShared<CT>) + 15) & ~size_t(15);
    unsigned char *mem = reinterpret_cast<unsigned char *>(&sh) + kAt;
    const int n = (int)a.n, n4 = n & ~3;
    const int per = (n + (int)gridDim.x - 1) / (int)gridDim.x;
    const int v = (int)blockIdx.x * per + (int)threadIdx.x;
    bool open = false, changed = false;
    unsigned finished = 0;
    // the whole policy, 16 bytes a load
    int2 *link = reinterpret_cast<int2 *>(mem);                 // FP32: {parent, cost}
    double *cost = reinterpret_cast<double *>(mem);             // FP64: costs, parents, stack
    int32_t *par = reinterpret_cast<int32_t *>(mem + 8 * (size_t)((n + 3) & ~3));
    double *stack = reinterpret_cast<double *>(mem + 12 * (size_t)((n + 3) & ~3));
    for (int i = 4 * (int)threadIdx.x; i < n4; i += 4 * kLoopThreads) {
        const int4 q = __ldcg(reinterpret_cast<const int4 *>(a.p + i));
        if constexpr (sizeof(CT) == 4) {
            const int4 w = __ldcg(reinterpret_cast<const int4 *>(a.pc + i));
            *reinterpret_cast<int4 *>(link + i) = make_int4(q.x, w.x, q.y, w.y);
            *reinterpret_cast<int4 *>(link + i + 2) = make_int4(q.z, w.z, q.w, w.w);
        } else {
            *reinterpret_cast<int4 *>(par + i) = q;
            const int4 *w = reinterpret_cast<const int4 *>(a.pc + i);
            reinterpret_cast<int4 *>(cost + i)[0] = __ldcg(w);
            reinterpret_cast<int4 *>(cost + i)[1] = __ldcg(w + 1);
        }
    }
    for (int i = n4 + (int)threadIdx.x; i < n; i += kLoopThreads) {
        if constexpr (sizeof(CT) == 4) {
            link[i] = make_int2(__ldcg(a.p + i), __float_as_int(__ldcg(a.pc + i)));
        } else {
            par[i] = __ldcg(a.p + i);
            cost[i] = __ldcg(a.pc + i);
        }
    }
    double old = 0.0;
    const bool mine = (int)threadIdx.x < per && v < n;
    if (mine) old = __ldcg(&a.g[v]);
    __syncthreads();
    if (mine) {
        double gw = 0.0;
        bool has = false;
        if constexpr (sizeof(CT) == 4) {
            int2 t = link[v];
            if (t.x >= 0) {
                has = true;
                double s = (double)__int_as_float(t.y);
                int x = t.x, hops = 0;
                for (t = link[x]; t.x >= 0; t = link[x]) {
                    s += (double)__int_as_float(t.y);
                    x = t.x;
                    if (++hops > n) {  // a cycle: left to pointer jumping, which reports it
                        open = true;
                        break;
                    }
                }
                gw = s + __ldcg(&a.g[x]);
            }
        } else {
            int x = par[v];
            if (x >= 0) {
                has = true;
                stack[threadIdx.x] = cost[v];
                int d = 1;
                for (int up = par[x]; up >= 0; up = par[x]) {
                    if (d == kWalkDepth) {
                        open = true;
                        break;
                    }
                    stack[d++ * kWalkPerF64 + threadIdx.x] = cost[x];
                    x = up;
                }
                gw = __ldcg(&a.g[x]);
                while (--d >= 0) gw = gw + stack[d * kWalkPerF64 + threadIdx.x];
            }
        }
        if (has && !open) {
            const bool diff = __double_as_longlong(gw) != __double_as_longlong(old);
            if (diff) a.g[v] = gw;
            // a wave leaves the FP32 shadow behind: every one is rewritten then
            if (diff || stale) a.g32[v] = g32_of(gw);
            changed = diff;
            finished = 1u;
        }
    }
    if (changed) sh.mark[atomicAdd(&sh.nmark, 1u)] = v;
    const unsigned left = __syncthreads_or(open) ? 1u : 0u;
    flush_marks<CT>(sh, a.dg, &ic->n_jump);
    if (!loop_sync<CT>(a.ctr, sh, left)) return false;
    if (sh.total != 0u) {
        walk = false;
        if (changed) {
            a.g[v] = old;
            a.g32[v] = g32_of(old);
        }
        // (every append came before the barrier above, loop_jump's come after the next)
        if (blockIdx.x == 0 && threadIdx.x == 0) ic->n_jump = 0u;
        if (!loop_sync<CT>(a.ctr, sh, 0u)) return false;
        return loop_jump<CT>(a, ic, stale);
    }
    if (threadIdx.x == 0) {
        sh.rounds = 1u;
        sh.bad = 0u;
    }
    add_total(finished, &sh.tot[2]);
    __syncthreads();
    return true;
}


// After pointer jumping: every changed vertex offers its neighbours their
// candidate through it where it beats their g, and lists them.  L lanes per
// changed vertex.
template <typename CT, int L, int U>
__device__ __forceinline__ void loop_mark(const LoopArgs<CT> &a, LoopCounters *ic, unsigned n_dg, int32_t *next,
                                       unsigned epoch) {
    LoopShared<CT> &sh = loop_shared<CT>();
    const int gl = (int)(threadIdx.x & (unsigned)(L - 1));
    const int64_t groups = (int64_t)gridDim.x * (kLoopThreads / L);
    unsigned long long offers = 0;
    for (int64_t j = ((int64_t)blockIdx.x * kLoopThreads + threadIdx.x) / L; j < (int64_t)n_dg;
         j += groups) {
        const int32_t x = __ldcg(&a.dg[j]);
        const longlong2 e = __ldg(reinterpret_cast<const longlong2 *>(a.rows) + x);
        const int len = (int)(unsigned)((unsigned long long)e.y & 0xffffffffull);
        const Entry<CT> *row = a.adj + e.x;
        const double gx = __ldcg(&a.g[x]);
        if (gl == 0) offers += (unsigned)len;
        for (int e0 = gl; e0 < len; e0 += L * U) {
            Entry<CT> en[U];
            unsigned long long gold[U];
#pragma unroll
            for (int q = 0; q < U; ++q)
                if (e0 + L * q < len) en[q] = ld_stream(&row[e0 + L * q]);
#pragma unroll
            for (int q = 0; q < U; ++q)
                gold[q] = e0 + L * q < len
                              ? __ldcg(reinterpret_cast<const unsigned long long *>(a.g) + en[q].col)
                              : 0ull;
            unsigned mk = 0;
#pragma unroll
            for (int q = 0; q < U; ++q)
                if (e0 + L * q < len) {
                    const unsigned long long val =
                        (unsigned long long)__double_as_longlong(gx + widen(en[q].w));
                    if (val < gold[q]) {
                        atomicMin(a.cand + en[q].col, val);
                        if (atomicExch(&a.stamp[en[q].col], epoch) != epoch) mk |= 1u << q;
                    }
                }
            if (mk) {
                int32_t col[U];
#pragma unroll
                for (int q = 0; q < U; ++q) col[q] = en[q].col;
                stage_marks<CT, U>(sh, mk, col, next, &ic->n_next);
            }
        }
    }
    add_total(offers, &sh.tot[3]);
    __syncthreads();
    flush_marks<CT>(sh, next, &ic->n_next);
}

template <typename CT, int OCC>  // CTAs per SM
__global__ void __launch_bounds__(kLoopThreads, OCC)
replan_loop_kernel(const __grid_constant__ LoopArgs<CT> a) {
    LoopShared<CT> &sh = loop_shared<CT>();
    DevCounters *c = a.ctr;
    const int tid = threadIdx.x;
    if (tid == 0) {
        sh.nitem[0] = sh.nitem[1] = 0u;
        sh.nmark = sh.nfirst = sh.nstage = sh.incomplete = sh.over = 0u;
        sh.dj = 0ull;
        for (int k = 0; k < 4; ++k) sh.tot[k] = 0ull;
        sh.barriers = sh.direct = sh.bad = sh.rounds = 0u;
        sh.seen[0] = sh.seen[1] = 0ull;
        sh.bound = a.goal_g != nullptr ? __ldcg(a.goal_g) : CUDART_INF;
    }
    if (tid == 0) {
        sh.tr.state = (blockIdx.x == 0 && c->lvl_trace != 0u) ? -2 : -1;
        sh.tr.t = sh.tr.tile = 0;
        sh.tr.ns0 = 0ull;
    }
    // loop state, the same in every CTA; CTA 0 writes it back at the end
    unsigned la = c->la & 1u, epoch = c->epoch, tag = c->wave_epoch, par = c->loop_par & 1u;
    unsigned n_active = c->n_active;
    bool dense = c->dense != 0u, stale = c->g32_stale != 0u;
    unsigned iter = 0, levels_sum = 0, dense_sum = 0, rounds_sum = 0, jump_sum = 0, deep_sum = 0;
    unsigned long long switches = 0;  // thread 0
    bool converged = false, ok = true;
    bool walk = a.walk != 0;  // ... until a policy is too deep for it
    LoopCounters *ic = &c->loop[par];
    if (blockIdx.x == 0 && tid == 0) {
        // the other loop forms leave their totals behind (this one's are added
        // after its barriers)
        c->relax = 0ull;
        c->improved = 0ull;
        c->evaluated = 0ull;
        c->offers = 0ull;
    }
    __syncthreads();
    if (vld(&c->insert_late) != 0u) {  // an insertion did not end: its rows are not followed
        ok = false;
        if (tid == 0) atomicOr(&c->status, kStatusTimeout);
    }
    if (sizeof(CT) == 4 && ok && dense && stale) {
        for (int64_t v = (int64_t)blockIdx.x * kLoopThreads + tid; v < a.n;
             v += (int64_t)gridDim.x * kLoopThreads)
            a.g32[v] = g32_of(__ldcg(&a.g[v]));
        stale = false;
        ok = loop_sync<CT>(c, sh, 0u);
    }
    while (ok) {
        if (tid == 0) trace_iteration(c, sh.tr, iter);
        ic = &c->loop[par];
        // ---- Improve
        if constexpr (sizeof(CT) == 4) {
            if (dense) loop_dense_screen(a, ic);
            else loop_improve<CT>(a, ic, la ? a.list[1] : a.list[0], (int64_t)n_active, false);
        } else {
            loop_improve<CT>(a, ic, la ? a.list[1] : a.list[0], dense ? a.n : (int64_t)n_active,
                             dense);
        }
        __syncthreads();
        const unsigned mine = sh.nstage;
        const unsigned staged = mine < kStage ? mine : kStage;
        if (staged) {
            if (tid == 0) sh.base[0] = atomicAdd(&ic->n_switched, staged);
            if (tid == 32) atomicMax(&ic->dj_bits, sh.dj);
            __syncthreads();
            const uint4 *from = reinterpret_cast<const uint4 *>(sh.item[0]);
            uint4 *to = reinterpret_cast<uint4 *>(a.items[1] + sh.base[0]);
            for (unsigned i = tid; i < 2u * staged; i += kLoopThreads) to[i] = from[i];
        }
        ok = loop_sync<CT>(c, sh, mine);
        if (!ok) break;
        const unsigned n_sw = sh.total;
        const double dj = __longlong_as_double((long long)__ldcg(&ic->dj_bits));
        if (tid == 0) {
            sh.over = 0u;
            sh.nstage = 0u;
            sh.dj = 0ull;
            switches += n_sw;
        }
        // every CTA is past its last read of the other counter set
        if (blockIdx.x == 0 && tid < (int)(sizeof(LoopCounters) / 4))
            reinterpret_cast<unsigned *>(&c->loop[par ^ 1u])[tid] = 0u;
        const bool was_dense = dense;
        if (was_dense) ++dense_sum;
        ++iter;
        unsigned next_count = 0;
        bool next_dense = false;
        unsigned levels = 0;
        int32_t *next = la ? a.list[0] : a.list[1];
        bool jump = a.jump != 0 || n_sw > a.jump_above;
        if (tid == 0 && (n_sw == 0u || jump)) trace_step(c, sh.tr, 0);
        if (n_sw != 0u) {
            if (!jump) {
                // ---- Evaluate, top-down in grid steps
                int64_t count = (int64_t)n_sw;
                bool lost = false;
                for (unsigned t = 0;; ++t) {
                    // a vertex lowered several times in a step (parallel edges)
                    // takes as many entries: those past the end of the list are
                    // lost, and with them the offers of their vertices.  Pointer
                    // jumping finishes every value; the next sweep is dense.
                    const bool stop = count > a.list_cap;
                    if (stop) count = a.list_cap;
                    if (tid == 0) {
                        sh.step.next = next;
                        sh.step.out = a.items[t & 1u];
                        sh.step.out_cnt = &ic->wave_cnt[(t + 1u) % 3u];
                        sh.step.tag = tag;
                        sh.step.epoch = epoch + 1u;
                        sh.step.flags = (stop ? kStepOffersOnly : 0u) |
                                        (sh.tr.state != -1 ? kStepTraced : 0u);
                    }
                    __syncthreads();
                    const bool tail = count <= (int64_t)a.tail_max;
                    const bool alone = !stop && (tail || count <= (int64_t)a.local_step);
                    const int64_t per = tail ? count : (count + gridDim.x - 1) / gridDim.x;
                    const int64_t lo = (int64_t)blockIdx.x * per < count
                                           ? (int64_t)blockIdx.x * per : count;
                    const int64_t hi = lo + per < count ? lo + per : count;
                    if (blockIdx.x == 0 && tid == 0) ic->wave_cnt[(t + 2u) % 3u] = 0u;
                    if (tid == 0) trace_step(c, sh.tr, count);
                    ++levels;
                    unsigned made = 0;
                    if (lo < hi)
                        made = loop_step<CT>(a, ic, a.items[(t & 1u) ^ 1u], t == 0u, lo, hi,
                                             !alone ? 0u : tail ? 0xffffffffu : a.local_levels,
                                             tail ? kStage : a.local_max);
                    ok = loop_sync<CT>(c, sh, made);
                    lost = stop;
                    if (!ok || stop) break;
                    count = (int64_t)sh.total;
                    if (count == 0) break;
                }
                if (!ok) break;
                loop_fetch<CT>(c, ic, sh);
                if (tid == 0) trace_step(c, sh.tr, 0);
                next_dense = lost || sh.v_ndg > a.dense_limit;
                next_count = sh.v_next;
                jump = (sh.v_flags & kLoopIncomplete) != 0u;
                stale = true;
                if (jump) ++deep_sum;
                if (jump && next_dense) next_count = 0u;
            }
            if (jump) {
                // ---- Evaluate, or the rest of a wave too deep, by pointer jumping
                const long long tj = clock64();
                ok = walk ? loop_walk<CT>(a, ic, stale, walk) : loop_jump<CT>(a, ic, stale);
                if (tid == 0 && sh.tr.state != -1)
                    c->ph_jump_cyc += (unsigned long long)(clock64() - tj);
                if (!ok) break;
                rounds_sum += sh.rounds;
                jump_sum += 1u;
                stale = false;
                loop_fetch<CT>(c, ic, sh);
                const unsigned n_jump = sh.v_jump;
                if (n_jump > a.dense_limit) next_dense = true;
                if (!next_dense && n_jump != 0u) {
                    if (n_jump <= gridDim.x * kLoopWarps)
                        loop_mark<CT, 32, 3>(a, ic, n_jump, next, epoch + 1u);
                    else
                        loop_mark<CT, 8, 5>(a, ic, n_jump, next, epoch + 1u);
                    ok = loop_sync<CT>(c, sh, 0u);
                    if (!ok) break;
                    loop_fetch<CT>(c, ic, sh);
                    next_count = sh.v_next;
                }
            }
            if (sizeof(CT) == 4 && next_dense && stale) {
                for (int64_t v = (int64_t)blockIdx.x * kLoopThreads + tid; v < a.n;
                     v += (int64_t)gridDim.x * kLoopThreads)
                    a.g32[v] = g32_of(__ldcg(&a.g[v]));
                stale = false;
                ok = loop_sync<CT>(c, sh, 0u);
                if (!ok) break;
            }
        }
        // ---- end of the iteration
        levels_sum += levels;
        la ^= 1u;
        epoch += 1u;
        tag += 1u;
        par ^= 1u;
        dense = next_dense;
        n_active = next_dense ? 0u : next_count;
        if (tid == 0) trace_end(c, sh.tr);
        if (n_sw == 0u) loop_fetch<CT>(c, ic, sh);
        const bool stable = n_sw == 0u || dj <= a.eps;
        const bool failed = sh.bad != 0u || sh.v_status != 0u;
        converged = stable && !failed;
        if (stable || failed || iter >= a.max_iters) break;
        if (tid == 0 && a.goal_g != nullptr) sh.bound = __ldcg(a.goal_g);
        __syncthreads();
    }
    // ---- totals; the last CTA reports
    __syncthreads();
    if (tid == 0) {
        unsigned long long *tot[4] = {&c->relax, &c->improved, &c->evaluated, &c->offers};
        for (int k = 0; k < 4; ++k)
            if (sh.tot[k]) atomicAdd(tot[k], sh.tot[k]);
        if (blockIdx.x == 0) {
            c->loop_state.iter = iter;
            c->loop_state.converged = converged ? 1u : 0u;
            c->loop_state.switches = switches;
            c->loop_state.wave_levels = levels_sum;
            c->loop_state.dense_sweeps = dense_sum;
            c->loop_state.jump_rounds = rounds_sum;
            c->loop_state.jump_evals = jump_sum;
            c->loop_state.deep = deep_sum;
            c->la = la;
            c->epoch = epoch;
            c->wave_epoch = tag;
            c->dense = dense ? 1u : 0u;
            c->n_active = n_active;
            c->g32_stale = stale ? 1u : 0u;
            c->loop_par = par;
        }
        __threadfence();
        if (atomicAdd(&c->wave_ticket, 1u) == gridDim.x - 1u) {
            __threadfence();
            c->wave_ticket = 0u;
            // both counter sets start clean (the last iteration's is not
            // cleared by a following one)
            c->loop_bar[0] = 0ull;
            c->loop_bar[16] = 0ull;
            unsigned *w = reinterpret_cast<unsigned *>(&c->loop[par ^ 1u]);
            for (int k = 0; k < (int)(sizeof(LoopCounters) / 4); ++k) w[k] = 0u;
            LoopResult r;
            r.relax = __ldcg(&c->relax);
            r.improved = __ldcg(&c->improved);
            r.evaluated = __ldcg(&c->evaluated);
            r.offers = __ldcg(&c->offers);
            r.switches = __ldcg(&c->loop_state.switches);
            r.iter = __ldcg(&c->loop_state.iter);
            r.converged = __ldcg(&c->loop_state.converged);
            r.status = __ldcg(&c->status);
            r.wave_epoch = tag;
            r.wave_levels = __ldcg(&c->loop_state.wave_levels);
            r.dense_sweeps = __ldcg(&c->loop_state.dense_sweeps);
            r.jump_rounds = __ldcg(&c->loop_state.jump_rounds);
            r.jump_evals = __ldcg(&c->loop_state.jump_evals);
            r.deep = __ldcg(&c->loop_state.deep);
            *a.res = r;
        }
    }
}

}  // namespace pirrt
