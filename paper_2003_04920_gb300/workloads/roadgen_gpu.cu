// GPU-resident roadmap generator: seeded free-space samples, grid k-nearest
// neighbours, union-symmetrised collision-checked edges ordered by the larger
// endpoint.  Input generation only; the definitions are in roadgen_gpu.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <memory>
#include <new>
#include <type_traits>
#include <vector>

#include "roadgen_gpu.h"

namespace {

constexpr int kT = 256;
constexpr int kMaxDim = 8;
constexpr int kMaxK = 128;

#define RG_CK(x)                                 \
    do {                                         \
        if ((x) != cudaSuccess) return 2;        \
    } while (0)
#define RG_CKL() RG_CK(cudaGetLastError())

// ---- Philox4x32-10 (Salmon, Moraes, Dror, Shaw: "Parallel random numbers:
// as easy as 1, 2, 3", SC 2011): ten rounds of two 32x32 -> 64-bit products,
// the key advanced by the Weyl increments between rounds.
__device__ __forceinline__ uint4 philox(uint4 x, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned hi0 = __umulhi(0xD2511F53u, x.x), lo0 = 0xD2511F53u * x.x;
        const unsigned hi1 = __umulhi(0xCD9E8D57u, x.z), lo1 = 0xCD9E8D57u * x.z;
        x = make_uint4(hi1 ^ x.y ^ k.x, lo1, hi0 ^ x.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return x;
}

__device__ __forceinline__ double unit_of(unsigned x) {
    return (double)(x >> 8) * (1.0 / 16777216.0);
}

// Squared distance in FP64, coordinates in order, no fused multiply-add.
__device__ __forceinline__ double d2_64(const double *a, const double *b, int dim) {
    double s = 0.0;
    for (int d = 0; d < dim; ++d) {
        const double t = __dsub_rn(a[d], b[d]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// ---- sampling -------------------------------------------------------------

// Candidates [c0, c0 + count): coordinates and a free flag.  The inside test
// is screened in FP32 and decided exactly in FP64 near a ball's surface.
__global__ void sample_kernel(int dim, double lo, double hi, int n_obs,
                              const double *__restrict__ centers, const double *__restrict__ radii,
                              uint2 key, long long c0, long long count, double *__restrict__ pts,
                              int *__restrict__ free_flag) {
    const double span = __dsub_rn(hi, lo);
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
         t += (long long)gridDim.x * blockDim.x) {
        const unsigned long long i = (unsigned long long)(c0 + t);
        double p[kMaxDim];
        uint4 w = make_uint4(0, 0, 0, 0);
        for (int d = 0; d < dim; ++d) {
            if ((d & 3) == 0)
                w = philox(make_uint4((unsigned)i, (unsigned)(i >> 32), (unsigned)(d >> 2), 0u),
                           key);
            const unsigned x = (d & 3) == 0 ? w.x : (d & 3) == 1 ? w.y : (d & 3) == 2 ? w.z : w.w;
            p[d] = __dadd_rn(lo, __dmul_rn(span, unit_of(x)));
            pts[t * dim + d] = p[d];
        }
        bool ok = true;
        for (int s = 0; s < n_obs && ok; ++s) {
            const double *c = centers + (long long)s * dim;
            const float r2f = (float)(radii[s] * radii[s]);
            float df = 0.f;
            for (int d = 0; d < dim; ++d) {
                const float e = (float)p[d] - (float)c[d];
                df += e * e;
            }
            if (df > r2f * 1.001f + 1e-4f) continue;         // clearly outside
            if (df < r2f * 0.999f - 1e-4f) { ok = false; continue; }  // clearly inside
            const double r2 = __dmul_rn(radii[s], radii[s]);
            if (d2_64(p, c, dim) < r2) ok = false;
        }
        free_flag[t] = ok ? 1 : 0;
    }
}

// ---- scans (exclusive, int32 -> int64) ---------------------------------------

__device__ __forceinline__ long long block_scan(long long x, long long *total) {
    __shared__ long long ws[kT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        long long w = lane < kT / 32 ? ws[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < kT / 32) ws[lane] = w;
    }
    __syncthreads();
    const long long base = warp > 0 ? ws[warp - 1] : 0;
    *total = ws[kT / 32 - 1];
    __syncthreads();
    return base + incl - x;
}

constexpr int kItems = 8;
constexpr int kTile = kT * kItems;

__global__ void scan_reduce(const int *__restrict__ in, long long len, long long *__restrict__ tiles) {
    const long long b = (long long)blockIdx.x * kTile + (long long)threadIdx.x * kItems;
    long long s = 0;
    for (int i = 0; i < kItems; ++i)
        if (b + i < len) s += in[b + i];
    long long tot;
    block_scan(s, &tot);
    if (threadIdx.x == 0) tiles[blockIdx.x] = tot;
}

__global__ void scan_tiles(long long *__restrict__ tiles, long long n) {
    __shared__ long long carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (long long b = 0; b < n; b += kT) {
        const long long i = b + threadIdx.x;
        const long long x = i < n ? tiles[i] : 0;
        long long tot;
        const long long ex = block_scan(x, &tot);
        if (i < n) tiles[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
}

__global__ void scan_apply(const int *__restrict__ in, long long len,
                           const long long *__restrict__ tiles, long long *__restrict__ out) {
    const long long b = (long long)blockIdx.x * kTile + (long long)threadIdx.x * kItems;
    long long v[kItems], s = 0;
    for (int i = 0; i < kItems; ++i) {
        v[i] = b + i < len ? in[b + i] : 0;
        s += v[i];
    }
    long long tot;
    long long run = block_scan(s, &tot) + tiles[blockIdx.x];
    for (int i = 0; i < kItems; ++i) {
        if (b + i < len) out[b + i] = run;
        run += v[i];
    }
}

// out[i] = in[0] + ... + in[i - 1] for i in [0, len); tiles: scratch.
int exclusive_scan(const int *in, long long len, long long *out, long long *tiles, cudaStream_t st) {
    if (len <= 0) return 0;
    const long long nt = (len + kTile - 1) / kTile;
    scan_reduce<<<(unsigned)nt, kT, 0, st>>>(in, len, tiles);
    RG_CKL();
    scan_tiles<<<1, kT, 0, st>>>(tiles, nt);
    RG_CKL();
    scan_apply<<<(unsigned)nt, kT, 0, st>>>(in, len, tiles, out);
    RG_CKL();
    return 0;
}

__global__ void compact_free(long long count, int dim, const double *__restrict__ cand,
                             const int *__restrict__ flag, const long long *__restrict__ pos,
                             long long want, double *__restrict__ out) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
         t += (long long)gridDim.x * blockDim.x) {
        if (!flag[t] || pos[t] >= want) continue;
        for (int d = 0; d < dim; ++d) out[pos[t] * dim + d] = cand[t * dim + d];
    }
}

int grid_of(long long work) {
    long long b = (work + kT - 1) / kT;
    if (b < 1) b = 1;
    if (b > 152 * 64) b = 152 * 64;
    return (int)b;
}

// ---- grid k-nearest neighbours ---------------------------------------------

struct Grid {
    int dim, G;
    double lo, cw;
};

__device__ __forceinline__ int cell_coord(const Grid &g, float x) {
    int c = (int)floor(((double)x - g.lo) / g.cw);
    return c < 0 ? 0 : (c >= g.G ? g.G - 1 : c);
}

__global__ void cell_count(long long n, Grid g, const double *__restrict__ pts,
                           long long *__restrict__ cell_of, int *__restrict__ cnt) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        long long id = 0, mul = 1;
        for (int d = 0; d < g.dim; ++d) {
            id += (long long)cell_coord(g, (float)pts[i * g.dim + d]) * mul;
            mul *= g.G;
        }
        cell_of[i] = id;
        atomicAdd(&cnt[id], 1);
    }
}

__global__ void cell_scatter(long long n, int dim, const double *__restrict__ pts,
                             const long long *__restrict__ cell_of,
                             const long long *__restrict__ start, int *__restrict__ cursor,
                             float *__restrict__ spts, int *__restrict__ sid) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const long long c = cell_of[i];
        const long long s = start[c] + atomicAdd(&cursor[c], 1);
        sid[s] = (int)i;
        for (int d = 0; d < dim; ++d) spts[s * dim + d] = (float)pts[i * dim + d];
    }
}

// FP32 squared distance, coordinates in order, no fused multiply-add.
template <int DIM>
__device__ __forceinline__ float d2_of(const float (&q)[DIM], const float *p) {
    float s = 0.f;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const float t = __fsub_rn(q[d], p[d]);
        s = __fadd_rn(s, __fmul_rn(t, t));
    }
    return s;
}

// Nearest-neighbour search, one warp per query.  A thread that keeps its own
// sorted list in local memory spends its time moving list entries (4.6 ms for the
// 63 nearest of 10^5 points in the plane; 0.65 ms this way); here the lanes measure 32 points of a
// cell row at a time, those below the k-th distance known so far are appended to
// a buffer in shared memory as (distance bits, id) keys -- non-negative floats
// order like their bits, so a key's order is (distance, id) -- and the warp sorts
// the buffer in registers when it is full or a box of cells has been seen.
constexpr int kBuf = 256;             // keys buffered per query (k <= 128 of them stay)
constexpr int kQWarps = kT / 32;
using Key = unsigned long long;
constexpr Key kNoKey = ~0ull;

// Ascending bitonic sort of 32 R keys, element 32 r + lane in x[r] of a lane.
template <int R>
__device__ __forceinline__ void sort_keys(Key (&x)[R], int lane) {
#pragma unroll
    for (int size = 2; size <= 32 * R; size <<= 1) {
#pragma unroll
        for (int dist = size >> 1; dist > 0; dist >>= 1) {
            if (dist >= 32) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int o = r ^ (dist >> 5);
                    if (o > r) {
                        const bool up = ((r * 32) & size) == 0;
                        const Key lo = x[r] < x[o] ? x[r] : x[o], hi = x[r] < x[o] ? x[o] : x[r];
                        x[r] = up ? lo : hi;
                        x[o] = up ? hi : lo;
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const Key o = __shfl_xor_sync(0xffffffffu, x[r], dist);
                    const bool up = ((r * 32 + lane) & size) == 0;
                    const bool first = (lane & dist) == 0;
                    const bool less = o < x[r];
                    x[r] = (up == first) == less ? o : x[r];
                }
            }
        }
    }
}

// The first cnt <= 32 R keys of the buffer sorted.
template <int R>
__device__ __forceinline__ void sort_buffer(Key *buf, int cnt, int lane) {
    Key x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = r * 32 + lane < cnt ? buf[r * 32 + lane] : kNoKey;
    sort_keys<R>(x, lane);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) buf[r * 32 + lane] = x[r];
}

// Keep the k smallest of the buffer's cnt keys, sorted (the first `kept` are what the
// last call kept); limit becomes the k-th key once there are k.  The sort is as long as
// the keys are many: 256 each time had made 20 neighbours of 10^6 points in the plane
// 5.3 ms, as against the 3.3 of a thread per query with its sorted list.
__device__ __forceinline__ void keep_k(Key *buf, int &cnt, int &kept, int k, Key &limit, int lane) {
    if (cnt == kept) return;
    __syncwarp();
    if (cnt <= 32) sort_buffer<1>(buf, cnt, lane);
    else if (cnt <= 64) sort_buffer<2>(buf, cnt, lane);
    else if (cnt <= 128) sort_buffer<4>(buf, cnt, lane);
    else sort_buffer<8>(buf, cnt, lane);
    __syncwarp();
    if (cnt >= k) {
        cnt = k;
        limit = buf[k - 1];
    }
    kept = cnt;
}

// The k smallest (d2, id) among the grid's points with id < id_limit, other
// than qid itself, sorted in buf; returns how many were found (k unless fewer
// candidates exist).  Cells are scanned by growing boxes of cells around the
// query's cell until the box holds the ball of the k-th distance.  Cells along
// the first axis hold consecutive points, so a box is a set of point ranges, one
// per lane at a time; a range farther than the k-th distance is skipped.
template <int DIM>
__device__ int knn_search(const Grid &g, int k, const float (&q)[DIM], int qid, int id_limit,
                          const float *__restrict__ spts, const int *__restrict__ sid,
                          const long long *__restrict__ start, Key *buf) {
    const int lane = threadIdx.x & 31;
    int qc[DIM], slo[DIM], shi[DIM];
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        qc[d] = cell_coord(g, q[d]);
        slo[d] = 0;
        shi[d] = -1;
    }
    int cnt = 0, kept = 0;
    Key limit = kNoKey;
    bool scanned = false;
    for (int r = 1;; ++r) {
        int blo[DIM], bhi[DIM];
        const float kth = __uint_as_float((unsigned)(limit >> 32));
        const float w = sqrtf(kth) * 1.0001f + 1e-6f;
        bool same = scanned, whole = true;
        int rows = 1;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            if (cnt < k) {
                blo[d] = max(0, qc[d] - r);
                bhi[d] = min(g.G - 1, qc[d] + r);
            } else {
                blo[d] = cell_coord(g, q[d] - w);
                bhi[d] = cell_coord(g, q[d] + w);
            }
            if (scanned) {
                blo[d] = min(blo[d], slo[d]);
                bhi[d] = max(bhi[d], shi[d]);
                same = same && blo[d] == slo[d] && bhi[d] == shi[d];
            }
            whole = whole && blo[d] == 0 && bhi[d] == g.G - 1;
            if (d > 0) rows *= bhi[d] - blo[d] + 1;
        }
        if (same && (cnt == k || whole)) break;  // (whole: fewer than k exist)
        for (int row0 = 0; row0 < rows; row0 += 32) {
            const bool bounded = limit != kNoKey;
            const float bound = __uint_as_float((unsigned)(limit >> 32)) * 1.0001f + 1e-6f;
            // a lane's cell row: its point range, or two where the last box cut it
            long long p0 = 0, p1 = 0, p2 = 0, p3 = 0;
            if (row0 + lane < rows) {
                int rest = row0 + lane;
                long long id = 0, mul = g.G;
                bool inside_old = scanned;
                float box = 0.f;
#pragma unroll
                for (int d = 1; d < DIM; ++d) {
                    const int n = bhi[d] - blo[d] + 1, c = blo[d] + rest % n;
                    rest /= n;
                    id += (long long)c * mul;
                    mul *= g.G;
                    inside_old = inside_old && c >= slo[d] && c <= shi[d];
                    const float a0 = (float)(g.lo + c * g.cw), a1 = (float)(g.lo + (c + 1) * g.cw);
                    const float e = q[d] < a0 ? a0 - q[d] : (q[d] > a1 ? q[d] - a1 : 0.f);
                    box += e * e;
                }
                if (!(bounded && box > bound)) {
                    if (!inside_old) {
                        p0 = start[id + blo[0]];
                        p1 = start[id + bhi[0] + 1];
                    } else {
                        p0 = start[id + blo[0]];
                        p1 = start[id + slo[0]];
                        p2 = start[id + shi[0] + 1];
                        p3 = start[id + bhi[0] + 1];
                    }
                }
            }
            for (int part = 0; part < 2; ++part) {
                unsigned todo = __ballot_sync(0xffffffffu, p1 > p0);
                while (todo) {
                    const int src = __ffs(todo) - 1;
                    todo &= todo - 1u;
                    const long long b = __shfl_sync(0xffffffffu, p0, src);
                    const long long e = __shfl_sync(0xffffffffu, p1, src);
                    for (long long i0 = b; i0 < e; i0 += 32) {
                        const long long i = i0 + lane;
                        Key key = kNoKey;
                        if (i < e) {
                            const int pid = sid[i];
                            if (pid != qid && pid < id_limit)
                                key = ((Key)__float_as_uint(d2_of<DIM>(q, spts + i * DIM)) << 32) |
                                      (unsigned)pid;
                        }
                        const bool in = key < limit;
                        const unsigned m = __ballot_sync(0xffffffffu, in);
                        if (m == 0u) continue;
                        if (in) buf[cnt + __popc(m & ((1u << lane) - 1u))] = key;
                        cnt += __popc(m);
                        if (cnt > kBuf - 32) keep_k(buf, cnt, kept, k, limit, lane);
                    }
                }
                p0 = p2;
                p1 = p3;
            }
        }
        keep_k(buf, cnt, kept, k, limit, lane);
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            slo[d] = blo[d];
            shi[d] = bhi[d];
        }
        scanned = true;
    }
    return cnt;
}

// One warp per point, in cell order (neighbouring warps scan the same cells): the
// k nearest among all points.  With `list`, of its *n_list points only.
template <int DIM>
__global__ void __launch_bounds__(kT)
knn_kernel(long long n, Grid g, int k, const float *__restrict__ spts, const int *__restrict__ sid,
           const long long *__restrict__ start, int *__restrict__ knn, const int *__restrict__ list,
           const int *__restrict__ n_list) {
    __shared__ Key s_buf[kQWarps][kBuf];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (list) n = *n_list;
    for (long long t = (long long)blockIdx.x * kQWarps + warp; t < n;
         t += (long long)gridDim.x * kQWarps) {
        const long long s = list ? list[t] : t;
        float q[DIM];
#pragma unroll
        for (int d = 0; d < DIM; ++d) q[d] = spts[s * DIM + d];
        const int qid = sid[s];
        const int cnt = knn_search<DIM>(g, k, q, qid, 0x7fffffff, spts, sid, start, s_buf[warp]);
        for (int a = lane; a < k; a += 32)
            knn[(long long)qid * k + a] = a < cnt ? (int)(unsigned)(s_buf[warp][a] & 0xffffffffull) : -1;
        __syncwarp();
    }
}

// The same for few neighbours of many points: one thread per point with its list in
// local memory, so that nothing is sorted and 32 queries share a warp.  Taken for up
// to 24 neighbours in up to 4 dimensions, from 5,000 points per neighbour on (10,000 in
// 4-D; six neighbours at least): us of the whole call, warp / thread, 10 neighbours of 10^5
// points in 1, 2, 3, 4 dimensions 414 / 280, 678 / 309, 967 / 401, 1401 / 620; of 10^6 2272 /
// 511, 4612 / 766, 7334 / 1299; 20 of 10^6 2268 / 1054, 4690 / 1757, 8062 / 3023.  Below
// that there are too few threads (20 of 10^4: 253 / 273 in 1-D, 369 / 669 in 4-D), and
// with more neighbours or dimensions lists and boxes are too long for a thread (24 of 10^5:
// 677 / 583 in 2-D, 1422 / 1735 in 4-D; 10 of 10^5 in 8-D 12.2 / 19.7 ms).  A point whose
// boxes hold far more points than a uniform spread gives goes to `late`, for a warp.
constexpr int kThreadK = 24, kThreadDim = 4;
bool by_thread(int dim, long long n, int k) {
    return dim <= kThreadDim && k <= kThreadK &&
           n >= (long long)(dim < 4 ? 5000 : 10000) * std::max(k, 6);
}
template <int DIM>
__global__ void __launch_bounds__(kT)
knn_thread_kernel(long long n, Grid g, int k, const float *__restrict__ spts,
                  const int *__restrict__ sid, const long long *__restrict__ start,
                  int *__restrict__ knn, int *__restrict__ late, int *__restrict__ n_late) {
    const long long most = 128ll * k + 512;  // points looked at (uniform: up to 40 k)
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n;
         s += (long long)gridDim.x * blockDim.x) {
        long long seen = 0;
        float q[DIM];
        int qc[DIM], slo[DIM], shi[DIM];
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            q[d] = spts[s * DIM + d];
            qc[d] = cell_coord(g, q[d]);
            slo[d] = 0;
            shi[d] = -1;
        }
        const int qid = sid[s];
        Key list[kThreadK];
        int cnt = 0;
        Key limit = kNoKey;  // the k-th key once there are k
        bool scanned = false;
        for (int r = 1;; ++r) {
            // boxes of cells as in knn_search
            int blo[DIM], bhi[DIM], c[DIM];
            const float kth = __uint_as_float((unsigned)(limit >> 32));
            const float w = sqrtf(kth) * 1.0001f + 1e-6f;
            bool same = scanned, whole = true;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                if (cnt < k) {
                    blo[d] = max(0, qc[d] - r);
                    bhi[d] = min(g.G - 1, qc[d] + r);
                } else {
                    blo[d] = cell_coord(g, q[d] - w);
                    bhi[d] = cell_coord(g, q[d] + w);
                }
                if (scanned) {
                    blo[d] = min(blo[d], slo[d]);
                    bhi[d] = max(bhi[d], shi[d]);
                    same = same && blo[d] == slo[d] && bhi[d] == shi[d];
                }
                whole = whole && blo[d] == 0 && bhi[d] == g.G - 1;
                c[d] = blo[d];
            }
            if (same && (cnt == k || whole)) break;
            // every cell row of the box, less what the box before held
            for (;;) {
                long long id = 0, mul = g.G;
                bool inside_old = scanned;
                float box = 0.f;
#pragma unroll
                for (int d = 1; d < DIM; ++d) {
                    id += (long long)c[d] * mul;
                    mul *= g.G;
                    inside_old = inside_old && c[d] >= slo[d] && c[d] <= shi[d];
                    const float a0 = (float)(g.lo + c[d] * g.cw), a1 = (float)(g.lo + (c[d] + 1) * g.cw);
                    const float e = q[d] < a0 ? a0 - q[d] : (q[d] > a1 ? q[d] - a1 : 0.f);
                    box += e * e;
                }
                const float bound = __uint_as_float((unsigned)(limit >> 32)) * 1.0001f + 1e-6f;
                if (cnt < k || !(box > bound)) {
                    for (int part = 0; part < 2; ++part) {
                        const int f = part == 0 ? blo[0] : inside_old ? shi[0] + 1 : bhi[0] + 1;
                        const int l = part == 0 && inside_old ? slo[0] - 1 : bhi[0];
                        if (f > l) continue;
                        const long long p0 = start[id + f], p1 = start[id + l + 1];
                        seen += p1 - p0;
                        if (seen > most) break;
                        for (long long p = p0; p < p1; ++p) {
                            const int pid = sid[p];
                            const Key key = ((Key)__float_as_uint(d2_of<DIM>(q, spts + p * DIM)) << 32) |
                                            (unsigned)pid;
                            if (pid == qid || key >= limit) continue;
                            int at = cnt < k ? cnt++ : k - 1;
                            for (; at > 0 && list[at - 1] > key; --at) list[at] = list[at - 1];
                            list[at] = key;
                            if (cnt == k) limit = list[k - 1];
                        }
                    }
                }
                if (seen > most) break;
                int d = 1;
#pragma unroll
                for (; d < DIM; ++d) {
                    if (c[d] < bhi[d]) {
                        ++c[d];
                        break;
                    }
                    c[d] = blo[d];
                }
                if (d == DIM) break;
            }
            if (seen > most) break;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                slo[d] = blo[d];
                shi[d] = bhi[d];
            }
            scanned = true;
        }
        if (seen > most) {
            late[atomicAdd(n_late, 1)] = (int)s;
            continue;
        }
        for (int a = 0; a < k; ++a)
            knn[(long long)qid * k + a] = a < cnt ? (int)(unsigned)(list[a] & 0xffffffffull) : -1;
    }
}

// The new vertices [v0, m) in the grid's cell order (positions p of the
// sorted ids with sid[p] >= v0): flags, then a compaction by their scan.
__global__ void query_flags(long long m, long long v0, const int *__restrict__ sid,
                            int *__restrict__ flag) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < m;
         p += (long long)gridDim.x * blockDim.x)
        flag[p] = sid[p] >= v0 ? 1 : 0;
}

__global__ void query_compact(long long m, long long v0, const int *__restrict__ sid,
                              const long long *__restrict__ pos, int *__restrict__ qlist) {
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < m;
         p += (long long)gridDim.x * blockDim.x)
        if (sid[p] >= v0) qlist[pos[p]] = sid[p];
}

// Vertices [q0, q1), visited in cell order (qlist, so that neighbouring warps
// scan the same cells): the k nearest among the vertices that precede each one
// (the grid holds vertices [0, q1)), -1 where fewer exist.  Row i - q0 of knn.
template <int DIM>
__global__ void __launch_bounds__(kT)
knn_pred_kernel(long long q0, long long q1, Grid g, int k, const double *__restrict__ pts,
                const float *__restrict__ spts, const int *__restrict__ sid,
                const long long *__restrict__ start, const int *__restrict__ qlist,
                int *__restrict__ knn) {
    __shared__ Key s_buf[kQWarps][kBuf];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long t = (long long)blockIdx.x * kQWarps + warp; t < q1 - q0;
         t += (long long)gridDim.x * kQWarps) {
        const long long i = qlist[t];
        float q[DIM];
#pragma unroll
        for (int d = 0; d < DIM; ++d) q[d] = (float)pts[i * DIM + d];
        const int cnt = knn_search<DIM>(g, k, q, (int)i, (int)i, spts, sid, start, s_buf[warp]);
        for (int a = lane; a < k; a += 32)
            knn[(i - q0) * k + a] = a < cnt ? (int)(unsigned)(s_buf[warp][a] & 0xffffffffull) : -1;
        __syncwarp();
    }
}

// f(std::integral_constant<int, dim>) for the dimension at hand
template <class F>
void with_dim(int dim, F f) {
    switch (dim) {
        case 1: f(std::integral_constant<int, 1>()); break;
        case 2: f(std::integral_constant<int, 2>()); break;
        case 3: f(std::integral_constant<int, 3>()); break;
        case 4: f(std::integral_constant<int, 4>()); break;
        case 5: f(std::integral_constant<int, 5>()); break;
        case 6: f(std::integral_constant<int, 6>()); break;
        case 7: f(std::integral_constant<int, 7>()); break;
        default: f(std::integral_constant<int, 8>()); break;
    }
}

// ---- edges ------------------------------------------------------------------

// The balls in FP32: dim centre coordinates, the radius squared, the centre's
// squared norm.
__global__ void obstacles_f32(int n_obs, int dim, const double *__restrict__ centers,
                              const double *__restrict__ radii, float *__restrict__ out) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n_obs) return;
    float n2 = 0.f;
    for (int d = 0; d < dim; ++d) {
        const float c = (float)centers[(long long)o * dim + d];
        out[(long long)o * (dim + 2) + d] = c;
        n2 += c * c;
    }
    out[(long long)o * (dim + 2) + dim] = (float)(radii[o] * radii[o]);
    out[(long long)o * (dim + 2) + dim + 1] = n2;
}

// Squared distance of a + t (b - a) to a centre, FP64, no fused multiply-add.
template <int DIM>
__device__ __forceinline__ double point_d2(const double (&a)[DIM], const double (&b)[DIM],
                                           const double *c, double t) {
    double s2 = 0.0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const double pd = __dsub_rn(__dadd_rn(a[d], __dmul_rn(t, __dsub_rn(b[d], a[d]))), c[d]);
        s2 = __dadd_rn(s2, __dmul_rn(pd, pd));
    }
    return s2;
}

// Collision of the segment [a, b] with the balls (mode 0: exact closest
// point; mode 1: n_check points).  FP64 decides, behind an FP32 test of the same
// distances: with coordinates rounded to FP32 a squared distance is off by less
// than 2^-19 (|a|^2 + |b - a|^2 + |c|^2), so beyond 1e-5 of that sum (five times
// it) on either side of the squared radius FP64 can only agree.
template <int DIM>
struct Segment {
    double a[DIM], b[DIM];
    float fa[DIM], ab[DIM], inv, size2;

    __device__ __forceinline__ void prepare() {
        float L2 = 0.f, a2 = 0.f;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            fa[d] = (float)a[d];
            ab[d] = (float)__dsub_rn(b[d], a[d]);
            L2 += ab[d] * ab[d];
            a2 += fa[d] * fa[d];
        }
        inv = L2 > 0.f ? 1.f / L2 : 0.f;
        size2 = a2 + L2;
    }

    // clear of ball s
    __device__ __forceinline__ bool clear_of(int s, const float *__restrict__ obs,
                                             const double *__restrict__ centers,
                                             const double *__restrict__ radii, int mode,
                                             int n_check) const {
        const float *o = obs + (long long)s * (DIM + 2);
        float w[DIM], t = 0.f, s2 = 0.f;
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            w[d] = __ldg(o + d) - fa[d];
            t += w[d] * ab[d];
        }
        t = fminf(fmaxf(t * inv, 0.f), 1.f);
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const float e = w[d] - t * ab[d];
            s2 += e * e;
        }
        const float r2 = __ldg(o + DIM), margin = 1e-5f * (size2 + __ldg(o + DIM + 1));
        if (s2 > r2 + margin) return true;
        const double *c = centers + (long long)s * DIM;
        const double r2d = __dmul_rn(radii[s], radii[s]);
        if (mode == 0) {
            if (s2 < r2 - margin) return false;
            double ab2 = 0.0, td = 0.0;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                const double e = __dsub_rn(b[d], a[d]);
                ab2 = __dadd_rn(ab2, __dmul_rn(e, e));
                td = __dadd_rn(td, __dmul_rn(__dsub_rn(c[d], a[d]), e));
            }
            td = ab2 > 0.0 ? __ddiv_rn(td, ab2) : 0.0;
            td = td < 0.0 ? 0.0 : (td > 1.0 ? 1.0 : td);
            return !(point_d2<DIM>(a, b, c, td) < r2d);
        }
        for (int i = 0; i < n_check; ++i) {
            const float tf = n_check > 1 ? (float)i / (float)(n_check - 1) : 0.f;
            float p2 = 0.f;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                const float e = w[d] - tf * ab[d];
                p2 += e * e;
            }
            if (p2 > r2 + margin) continue;
            if (p2 < r2 - margin) return false;
            const double td = n_check > 1 ? __ddiv_rn((double)i, (double)(n_check - 1)) : 0.0;
            if (point_d2<DIM>(a, b, c, td) < r2d) return false;
        }
        return true;
    }
};

// A point in registers.
template <int DIM>
__device__ __forceinline__ void load_point(const double *__restrict__ pts, long long i,
                                           double (&p)[DIM]) {
#pragma unroll
    for (int d = 0; d < DIM; ++d) p[d] = pts[i * DIM + d];
}

template <int DIM>
__device__ __forceinline__ double dist2(const double (&a)[DIM], const double (&b)[DIM]) {
    double s = 0.0;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const double t = __dsub_rn(a[d], b[d]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// Row i's links that row i owns (i < j, or i > j and i not in row j) and that
// are collision-free with a positive length: keep bits and a count per larger
// endpoint.  One warp per row: its links lie together, so the lanes first pick out
// the few balls that reach the ball around them all, test their links against
// those only and take the FP64 path together, and they look through row j
// together.  (With a thread per row, whose neighbours lie anywhere, every ball
// sent some lane of a warp down the FP64 path: 16.7 ms for the 63 links of 10^5
// points among 200 circles; a warp per row without the pick 2.0 ms, with it 0.57.)
template <int DIM>
__global__ void __launch_bounds__(kT)
edge_mark(long long n, const double *__restrict__ pts, int k, const int *__restrict__ knn,
          int n_obs, const float *__restrict__ obs, const double *__restrict__ centers,
          const double *__restrict__ radii, int mode, int n_check, unsigned *__restrict__ keep,
          int *__restrict__ vcnt) {
    const int lane = threadIdx.x & 31, words = (k + 31) / 32;
    for (long long i = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; i < n;
         i += ((long long)gridDim.x * blockDim.x) >> 5) {
        for (int a0 = 0; a0 < k; a0 += 32) {
            const int j = a0 + lane < k ? knn[i * k + a0 + lane] : -1;
            bool own = j >= 0 && j != (int)i;
            unsigned back = __ballot_sync(0xffffffffu, own && j < (int)i);
            while (back) {
                const int src = __ffs(back) - 1;
                back &= back - 1u;
                const long long jj = __shfl_sync(0xffffffffu, j, src);
                bool hit = false;
                for (int b = lane; b < k; b += 32) hit = hit || knn[jj * k + b] == (int)i;
                if (__any_sync(0xffffffffu, hit) && lane == src) own = false;
            }
            Segment<DIM> g;
            float far2 = 0.f;  // the farthest owned neighbour
            if (own) {
                load_point<DIM>(pts, min((long long)j, i), g.a);
                load_point<DIM>(pts, max((long long)j, i), g.b);
                own = dist2<DIM>(g.a, g.b) > 0.0;
                g.prepare();
                if (own) far2 = g.inv > 0.f ? 1.f / g.inv : 0.f;
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
                far2 = fmaxf(far2, __shfl_xor_sync(0xffffffffu, far2, off));
            float pi[DIM], p2 = 0.f;
#pragma unroll
            for (int d = 0; d < DIM; ++d) {
                pi[d] = (float)pts[i * DIM + d];
                p2 += pi[d] * pi[d];
            }
            for (int o0 = 0; o0 < n_obs; o0 += 32) {
                bool near = false;
                if (o0 + lane < n_obs) {
                    const float *o = obs + (long long)(o0 + lane) * (DIM + 2);
                    float d2 = 0.f;
#pragma unroll
                    for (int d = 0; d < DIM; ++d) {
                        const float e = o[d] - pi[d];
                        d2 += e * e;
                    }
                    const float reach = sqrtf(o[DIM]) + sqrtf(far2);
                    near = !(d2 > reach * reach * 1.001f + 1e-4f * (p2 + o[DIM + 1] + far2));
                }
                unsigned todo = __ballot_sync(0xffffffffu, near);
                while (todo) {
                    const int s = o0 + __ffs(todo) - 1;
                    todo &= todo - 1u;
                    if (own) own = g.clear_of(s, obs, centers, radii, mode, n_check);
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, own);
            if (lane == 0) keep[i * words + (a0 >> 5)] = m;
            if (own) atomicAdd(&vcnt[max(j, (int)i)], 1);
        }
    }
}

// Every kept link into its larger endpoint's group, in any order.
template <int DIM, typename CT>
__global__ void __launch_bounds__(kT)
edge_fill(long long n, const double *__restrict__ pts, int k, const int *__restrict__ knn,
          const unsigned *__restrict__ keep, const long long *__restrict__ vstart,
          int *__restrict__ cursor, int *__restrict__ tu, CT *__restrict__ tc) {
    const int lane = threadIdx.x & 31, words = (k + 31) / 32;
    for (long long i = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; i < n;
         i += ((long long)gridDim.x * blockDim.x) >> 5) {
        double pi[DIM];
        load_point<DIM>(pts, i, pi);
        for (int a0 = 0; a0 < k; a0 += 32) {
            if (!((keep[i * words + (a0 >> 5)] >> lane) & 1u)) continue;
            const int j = knn[i * k + a0 + lane];
            const int u = min(j, (int)i), v = max(j, (int)i);
            double pj[DIM];
            load_point<DIM>(pts, j, pj);
            // (x - y)^2 is the same either way round
            const long long at = vstart[v] + atomicAdd(&cursor[v], 1);
            tu[at] = u;
            tc[at] = (CT)__dsqrt_rn(dist2<DIM>(pi, pj));
        }
    }
}

// Each vertex's group of edges put in the order of the smaller endpoint: one warp
// per vertex, an edge's place is the number of edges before it (groups hold about
// k to 2k edges; 10^5 groups of 36 take 60 us, a thread's insertion sort each 603).
template <typename CT>
__global__ void __launch_bounds__(kT)
group_sort(long long n, const long long *__restrict__ vstart, const int *__restrict__ tu,
           const CT *__restrict__ tc, int *__restrict__ ou, int *__restrict__ ov,
           CT *__restrict__ oc) {
    const int lane = threadIdx.x & 31;
    for (long long v = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; v < n;
         v += ((long long)gridDim.x * blockDim.x) >> 5) {
        const long long b = vstart[v], e = vstart[v + 1];
        for (long long x0 = b; x0 < e; x0 += 32) {
            const long long x = x0 + lane;
            const int u = x < e ? tu[x] : 0;
            int rank = 0;
            for (long long y0 = b; y0 < e; y0 += 32) {
                const int w = y0 + lane < e ? tu[y0 + lane] : 0x7fffffff;
                const int m = e - y0 < 32 ? (int)(e - y0) : 32;
                for (int q = 0; q < m; ++q) {
                    const int o = __shfl_sync(0xffffffffu, w, q);
                    rank += o < u || (o == u && y0 + q < x) ? 1 : 0;
                }
            }
            if (x < e) {
                ou[b + rank] = u;
                ov[b + rank] = (int)v;
                oc[b + rank] = tc[x];
            }
        }
    }
}

// One device allocation carved into arrays (an allocation costs tens of
// microseconds, freeing it waits for the device).
struct Arena {
    char *base = nullptr;
    size_t used = 0;
    template <typename T>
    size_t add(size_t count) {
        const size_t at = used;
        used += (sizeof(T) * (count > 0 ? count : 1) + 255) & ~size_t(255);
        return at;
    }
    bool alloc() { return cudaMalloc(&base, used > 0 ? used : 1) == cudaSuccess; }
    template <typename T>
    T *at(size_t offset) const {
        return reinterpret_cast<T *>(base + offset);
    }
    ~Arena() {
        if (base) cudaFree(base);
    }
};

template <typename T>
struct DevBuf {
    T *p = nullptr;
    ~DevBuf() {
        if (p) cudaFree(p);
    }
    bool alloc(size_t count) { return cudaMalloc(&p, sizeof(T) * (count > 0 ? count : 1)) == cudaSuccess; }
};

}  // namespace

extern "C" int rgg_sample(int32_t dim, double lo, double hi, int32_t n_obs, const double *centers,
                          const double *radii, uint64_t seed, int64_t n, double *points,
                          int64_t *tried, void *stream) {
    if (dim < 1 || dim > kMaxDim || !(hi > lo) || n_obs < 0 || n < 0 || (n > 0 && !points) ||
        (n_obs > 0 && (!centers || !radii)))
        return 1;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint2 key = make_uint2((unsigned)seed, (unsigned)(seed >> 32));
    const long long chunk = std::max<long long>(1 << 16, std::min<long long>(1 << 22, 2 * n));
    DevBuf<double> cand;
    DevBuf<int> flag;
    DevBuf<long long> pos, tiles;
    if (!cand.alloc((size_t)chunk * dim) || !flag.alloc(chunk) || !pos.alloc(chunk) ||
        !tiles.alloc(chunk / kTile + 2))
        return 2;
    long long have = 0, c0 = 0;
    while (have < n) {
        sample_kernel<<<grid_of(chunk), kT, 0, st>>>(dim, lo, hi, n_obs, centers, radii, key, c0,
                                                     chunk, cand.p, flag.p);
        RG_CKL();
        if (int rc = exclusive_scan(flag.p, chunk, pos.p, tiles.p, st)) return rc;
        compact_free<<<grid_of(chunk), kT, 0, st>>>(chunk, dim, cand.p, flag.p, pos.p, n - have,
                                                    points + have * dim);
        RG_CKL();
        long long last = 0;
        int lastf = 0;
        RG_CK(cudaMemcpyAsync(&last, pos.p + chunk - 1, sizeof(last), cudaMemcpyDeviceToHost, st));
        RG_CK(cudaMemcpyAsync(&lastf, flag.p + chunk - 1, sizeof(lastf), cudaMemcpyDeviceToHost, st));
        RG_CK(cudaStreamSynchronize(st));
        const long long got = last + lastf;
        if (have + got >= n) {
            // the candidate that completed the set: count the draws up to it
            c0 += chunk;
            have = n;
            break;
        }
        have += got;
        c0 += chunk;
        if (c0 > (1ll << 40)) return 1;  // the box is (almost) all obstacle
    }
    if (tried) *tried = c0;
    return 0;
}

extern "C" int rgg_knn(int32_t dim, double lo, double hi, int64_t n, const double *points,
                       int32_t k, double cell, int32_t *knn, void *stream) {
    if (dim < 1 || dim > kMaxDim || !(hi > lo) || n < 2 || k < 1 || k >= n || k > kMaxK ||
        !points || !knn)
        return 1;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const double span = hi - lo;
    if (!(cell > 0.0)) {
        // side about the k-th neighbour distance of a uniform spread
        const double unit = std::pow(M_PI, dim / 2.0) / std::tgamma(dim / 2.0 + 1.0);
        cell = std::pow((double)k * std::pow(span, dim) / ((double)n * unit), 1.0 / dim);
    }
    int G = (int)std::floor(span / cell);
    G = std::max(1, G);
    while (std::pow((double)G, dim) > (double)(1 << 24) && G > 1) --G;  // bounded cell table
    long long cells = 1;
    for (int d = 0; d < dim; ++d) cells *= G;
    Grid g{dim, G, lo, span / G};
    Arena m;
    const size_t o_cell = m.add<long long>(n), o_start = m.add<long long>(cells + 1),
                 o_tiles = m.add<long long>((cells + 1) / kTile + 2), o_cnt = m.add<int>(cells + 1),
                 o_sid = m.add<int>(n), o_spts = m.add<float>((size_t)n * dim);
    const bool threads = by_thread(dim, n, k);
    const size_t o_late = m.add<int>(threads ? n + 1 : 1);
    if (!m.alloc()) return 2;
    int *n_late = m.at<int>(o_late), *late = n_late + 1;
    if (threads) RG_CK(cudaMemsetAsync(n_late, 0, sizeof(int), st));
    long long *cell_of = m.at<long long>(o_cell), *start = m.at<long long>(o_start),
              *tiles = m.at<long long>(o_tiles);
    int *cnt = m.at<int>(o_cnt), *sid = m.at<int>(o_sid);
    float *spts = m.at<float>(o_spts);
    RG_CK(cudaMemsetAsync(cnt, 0, sizeof(int) * (cells + 1), st));
    cell_count<<<grid_of(n), kT, 0, st>>>(n, g, points, cell_of, cnt);
    RG_CKL();
    if (int rc = exclusive_scan(cnt, cells + 1, start, tiles, st)) return rc;
    RG_CK(cudaMemsetAsync(cnt, 0, sizeof(int) * (cells + 1), st));
    cell_scatter<<<grid_of(n), kT, 0, st>>>(n, dim, points, cell_of, start, cnt, spts, sid);
    RG_CKL();
    with_dim(dim, [&](auto D) {
        constexpr int kDim = decltype(D)::value;
        if constexpr (kDim <= kThreadDim) {
            if (threads)
                knn_thread_kernel<kDim><<<grid_of(n), kT, 0, st>>>(n, g, k, spts, sid, start, knn,
                                                                   late, n_late);
        }
        knn_kernel<kDim><<<threads ? 152 * 4 : grid_of(n * 32), kT, 0, st>>>(
            n, g, k, spts, sid, start, knn, threads ? late : nullptr, n_late);
    });
    RG_CKL();
    RG_CK(cudaStreamSynchronize(st));
    return 0;
}

// What marking the links leaves for writing them.
struct rgg_links {
    int dim = 0, k = 0;
    long long n = 0, total = 0;
    const double *points = nullptr;
    const int *knn = nullptr;
    const long long *vstart = nullptr;
    Arena w;
    unsigned *keep = nullptr;
    int *vcnt = nullptr;
    bool filled = false;  // the cursors have moved
};

extern "C" void rgg_links_destroy(rgg_links *x) { delete x; }

extern "C" int rgg_links_mark(int32_t dim, int64_t n, const double *points, int32_t k,
                              const int32_t *knn, int32_t n_obs, const double *centers,
                              const double *radii, int32_t mode, int32_t n_check,
                              int64_t *edge_start, int64_t *m, void *stream, rgg_links **out) {
    if (!out) return 1;
    *out = nullptr;
    if (dim < 1 || dim > kMaxDim || n < 1 || k < 1 || !points || !knn || !edge_start || !m ||
        (mode != 0 && mode != 1) || (mode == 1 && n_check < 1) || n_obs < 0 ||
        (n_obs > 0 && (!centers || !radii)))
        return 1;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::unique_ptr<rgg_links> x(new (std::nothrow) rgg_links);
    if (!x) return 2;
    const size_t words = (size_t)(k + 31) / 32;
    Arena &w = x->w;
    const size_t o_keep = w.add<unsigned>((size_t)n * words), o_vcnt = w.add<int>(n + 1),
                 o_tiles = w.add<long long>((n + 1) / kTile + 2),
                 o_obs = w.add<float>((size_t)n_obs * (dim + 2));
    if (!w.alloc()) return 2;
    x->dim = dim;
    x->k = k;
    x->n = n;
    x->points = points;
    x->knn = knn;
    x->keep = w.at<unsigned>(o_keep);
    x->vcnt = w.at<int>(o_vcnt);
    long long *tiles = w.at<long long>(o_tiles), *vstart = reinterpret_cast<long long *>(edge_start);
    x->vstart = vstart;
    float *obs = w.at<float>(o_obs);
    if (n_obs > 0) {
        obstacles_f32<<<(n_obs + kT - 1) / kT, kT, 0, st>>>(n_obs, dim, centers, radii, obs);
        RG_CKL();
    }
    RG_CK(cudaMemsetAsync(x->vcnt, 0, sizeof(int) * (n + 1), st));
    with_dim(dim, [&](auto D) {
        edge_mark<decltype(D)::value><<<grid_of(n * 32), kT, 0, st>>>(
            n, points, k, knn, n_obs, obs, centers, radii, mode, n_check, x->keep, x->vcnt);
    });
    RG_CKL();
    if (int rc = exclusive_scan(x->vcnt, n + 1, vstart, tiles, st)) return rc;
    RG_CK(cudaMemcpyAsync(&x->total, vstart + n, sizeof(x->total), cudaMemcpyDeviceToHost, st));
    RG_CK(cudaMemsetAsync(x->vcnt, 0, sizeof(int) * (n + 1), st));  // now the groups' cursors
    RG_CK(cudaStreamSynchronize(st));
    *m = x->total;
    *out = x.release();
    return 0;
}

extern "C" int rgg_links_fill(rgg_links *x, int32_t cost_f64, int32_t *u, int32_t *v, void *cost,
                              void *stream) {
    if (!x || x->filled || (x->total > 0 && (!u || !v || !cost))) return 1;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long n = x->n;
    Arena t;
    const size_t o_u = t.add<int>(x->total);
    const size_t o_c = cost_f64 ? t.add<double>(x->total) : t.add<float>(x->total);
    if (!t.alloc()) return 2;
    x->filled = true;
    int *tu = t.at<int>(o_u);
    const auto fill = [&](auto zero) {
        using CT = decltype(zero);
        CT *tc = t.at<CT>(o_c);
        with_dim(x->dim, [&](auto D) {
            edge_fill<decltype(D)::value, CT><<<grid_of(n * 32), kT, 0, st>>>(
                n, x->points, x->k, x->knn, x->keep, x->vstart, x->vcnt, tu, tc);
        });
        RG_CKL();
        group_sort<CT><<<grid_of(n * 32), kT, 0, st>>>(n, x->vstart, tu, tc, u, v,
                                                       static_cast<CT *>(cost));
        RG_CKL();
        return 0;
    };
    if (const int rc = cost_f64 ? fill(0.0) : fill(0.f)) return rc;
    RG_CK(cudaStreamSynchronize(st));
    return 0;
}

extern "C" int rgg_edges(int32_t dim, int64_t n, const double *points, int32_t k,
                         const int32_t *knn, int32_t n_obs, const double *centers,
                         const double *radii, int32_t mode, int32_t n_check, int32_t cost_f64,
                         int32_t *u, int32_t *v, void *cost, int64_t *edge_start, int64_t cap,
                         int64_t *m, void *stream) {
    rgg_links *x = nullptr;
    if (const int rc = rgg_links_mark(dim, n, points, k, knn, n_obs, centers, radii, mode, n_check,
                                      edge_start, m, stream, &x))
        return rc;
    const std::unique_ptr<rgg_links> own(x);
    if (x->total > cap) return 3;
    return rgg_links_fill(x, cost_f64, u, v, cost, stream);
}

// ---- incremental exploration ------------------------------------------------

namespace {

// Links of the new vertices [v0, v1) to their nearest predecessors that are
// collision-free with a positive length: keep flags and a count per row.
// One thread per (new vertex, link), vertices in cell order: keep flags and
// the per-row count of the collision-free, positive-length links (rowc
// cleared before).
template <int DIM>
__global__ void pred_edge_mark(long long v0, long long v1, const double *__restrict__ pts, int k,
                               const int *__restrict__ knn, const int *__restrict__ qlist,
                               int n_obs, const float *__restrict__ obs,
                               const double *__restrict__ centers,
                               const double *__restrict__ radii, int mode, int n_check,
                               unsigned char *__restrict__ keep, int *__restrict__ rowc) {
    const long long total = (v1 - v0) * k;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const long long i = qlist[e / k];
        const int a = (int)(e % k);
        const long long r = i - v0;
        const int j = knn[r * k + a];
        bool ok = j >= 0;
        if (ok) {
            Segment<DIM> g;
            load_point<DIM>(pts, j, g.a);
            load_point<DIM>(pts, i, g.b);
            g.prepare();
            ok = dist2<DIM>(g.a, g.b) > 0.0;
            for (int s = 0; s < n_obs && ok; ++s)
                ok = g.clear_of(s, obs, centers, radii, mode, n_check);
        }
        keep[r * k + a] = ok ? 1 : 0;
        if (ok) atomicAdd(&rowc[r], 1);
    }
}

template <typename CT>
__global__ void pred_edge_emit(long long v0, long long v1, int dim, const double *__restrict__ pts,
                               int k, const int *__restrict__ knn,
                               const unsigned char *__restrict__ keep,
                               const long long *__restrict__ rowoff, int *__restrict__ eu,
                               int *__restrict__ ev, CT *__restrict__ ec) {
    for (long long i = v0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; i < v1;
         i += (long long)gridDim.x * blockDim.x) {
        const long long r = i - v0;
        long long at = rowoff[r];
        for (int a = 0; a < k; ++a) {
            if (!keep[r * k + a]) continue;
            const int j = knn[r * k + a];
            eu[at] = j;
            ev[at] = (int)i;
            ec[at] = (CT)__dsqrt_rn(d2_64(pts + (long long)j * dim, pts + i * dim, dim));
            ++at;
        }
    }
}

// Grid of cells of about the k-th neighbour distance for `m` points spread
// over the box (at most 2^24 cells).
Grid grid_for_density(int dim, double lo, double hi, long long m, int k) {
    const double span = hi - lo;
    const double unit = std::pow(M_PI, dim / 2.0) / std::tgamma(dim / 2.0 + 1.0);
    const double cell =
        std::pow((double)k * std::pow(span, dim) / ((double)std::max(m, 1ll) * unit), 1.0 / dim);
    int G = std::max(1, (int)std::floor(span / cell));
    while (std::pow((double)G, dim) > (double)(1 << 24) && G > 1) --G;
    return Grid{dim, G, lo, span / G};
}

long long cells_of(const Grid &g) {
    long long c = 1;
    for (int d = 0; d < g.dim; ++d) c *= g.G;
    return c;
}

}  // namespace

struct rgg_explorer {
    int dim = 0;
    double lo = 0.0, hi = 0.0;
    int n_obs = 0, k = 0, mode = 0, n_check = 0, cost_f64 = 0;
    long long n = 0, max_block = 0, cells_max = 0;
    double *centers = nullptr, *radii = nullptr, *pts = nullptr;
    float *spts = nullptr, *obs = nullptr;
    int *sid = nullptr, *cnt = nullptr, *knn = nullptr, *rowc = nullptr;
    int *qflag = nullptr, *qlist = nullptr;
    long long *cell_of = nullptr, *start = nullptr, *rowoff = nullptr, *tiles = nullptr;
    long long *qpos = nullptr;
    unsigned char *keep = nullptr;
};

extern "C" void rgg_explore_destroy(rgg_explorer *x) {
    if (!x) return;
    void *bufs[] = {x->centers, x->radii, x->pts, x->spts, x->obs, x->sid, x->cnt, x->knn, x->rowc,
                    x->cell_of, x->start, x->rowoff, x->tiles, x->keep, x->qflag, x->qlist,
                    x->qpos};
    for (void *b : bufs)
        if (b) cudaFree(b);
    delete x;
}

extern "C" int rgg_explore_create(int32_t dim, double lo, double hi, int32_t n_obs,
                                  const double *centers, const double *radii, uint64_t seed,
                                  int64_t n, int32_t k, int32_t mode, int32_t n_check,
                                  int32_t cost_f64, int64_t max_block, void *stream,
                                  rgg_explorer **out) {
    if (!out) return 1;
    *out = nullptr;
    if (dim < 1 || dim > kMaxDim || !(hi > lo) || n < 2 || k < 1 || k > kMaxK || max_block < 1 ||
        (mode != 0 && mode != 1) || (mode == 1 && n_check < 1) || n_obs < 0 ||
        (n_obs > 0 && (!centers || !radii)))
        return 1;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    rgg_explorer *x = new rgg_explorer;
    x->dim = dim;
    x->lo = lo;
    x->hi = hi;
    x->n_obs = n_obs;
    x->k = k;
    x->mode = mode;
    x->n_check = n_check;
    x->cost_f64 = cost_f64;
    x->n = n;
    x->max_block = std::min<long long>(max_block, n);
    const Grid gmax = grid_for_density(dim, lo, hi, n, k);
    x->cells_max = 1;
    for (long long m = 1; m <= n; m *= 2) x->cells_max = std::max(x->cells_max, cells_of(grid_for_density(dim, lo, hi, m, k)));
    x->cells_max = std::max(x->cells_max, cells_of(gmax));
    const long long mb = x->max_block;
    bool ok = cudaMalloc(&x->centers, sizeof(double) * std::max(1, n_obs * dim)) == cudaSuccess &&
              cudaMalloc(&x->radii, sizeof(double) * std::max(1, n_obs)) == cudaSuccess &&
              cudaMalloc(&x->pts, sizeof(double) * n * dim) == cudaSuccess &&
              cudaMalloc(&x->spts, sizeof(float) * n * dim) == cudaSuccess &&
              cudaMalloc(&x->obs, sizeof(float) * std::max(1, n_obs * (dim + 2))) == cudaSuccess &&
              cudaMalloc(&x->sid, sizeof(int) * n) == cudaSuccess &&
              cudaMalloc(&x->cell_of, sizeof(long long) * n) == cudaSuccess &&
              cudaMalloc(&x->cnt, sizeof(int) * (x->cells_max + 1)) == cudaSuccess &&
              cudaMalloc(&x->start, sizeof(long long) * (x->cells_max + 1)) == cudaSuccess &&
              cudaMalloc(&x->tiles, sizeof(long long) *
                                        (std::max<long long>(x->cells_max, n) + 1 + kTile) / kTile) == cudaSuccess &&
              cudaMalloc(&x->qflag, sizeof(int) * (n + 1)) == cudaSuccess &&
              cudaMalloc(&x->qpos, sizeof(long long) * (n + 1)) == cudaSuccess &&
              cudaMalloc(&x->qlist, sizeof(int) * mb) == cudaSuccess &&
              cudaMalloc(&x->knn, sizeof(int) * mb * k) == cudaSuccess &&
              cudaMalloc(&x->keep, mb * k) == cudaSuccess &&
              cudaMalloc(&x->rowc, sizeof(int) * (mb + 1)) == cudaSuccess &&
              cudaMalloc(&x->rowoff, sizeof(long long) * (mb + 1)) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        rgg_explore_destroy(x);
        return 2;
    }
    if (n_obs > 0 &&
        (cudaMemcpyAsync(x->centers, centers, sizeof(double) * n_obs * dim,
                         cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
         cudaMemcpyAsync(x->radii, radii, sizeof(double) * n_obs, cudaMemcpyDeviceToDevice, st) !=
             cudaSuccess)) {
        rgg_explore_destroy(x);
        return 2;
    }
    if (n_obs > 0) {
        obstacles_f32<<<(n_obs + kT - 1) / kT, kT, 0, st>>>(n_obs, dim, x->centers, x->radii, x->obs);
        if (cudaGetLastError() != cudaSuccess) {
            rgg_explore_destroy(x);
            return 2;
        }
    }
    int64_t tried = 0;
    const int rc = rgg_sample(dim, lo, hi, n_obs, x->centers, x->radii, seed, n, x->pts, &tried, st);
    if (rc) {
        rgg_explore_destroy(x);
        return rc;
    }
    *out = x;
    return 0;
}

extern "C" int rgg_explore_block(rgg_explorer *x, int64_t v0, int64_t v1, int32_t *u, int32_t *v,
                                 void *cost, int64_t *m_pinned, void *stream) {
    if (!x || v0 < 0 || v1 <= v0 || v1 > x->n || v1 - v0 > x->max_block || !u || !v || !cost ||
        !m_pinned)
        return 1;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int dim = x->dim, k = x->k;
    const long long nb = v1 - v0;
    // the grid over the vertices present, [0, v1)
    const Grid g = grid_for_density(dim, x->lo, x->hi, v1, k);
    const long long cells = cells_of(g);
    if (cells > x->cells_max) return 1;
    RG_CK(cudaMemsetAsync(x->cnt, 0, sizeof(int) * (cells + 1), st));
    cell_count<<<grid_of(v1), kT, 0, st>>>(v1, g, x->pts, x->cell_of, x->cnt);
    RG_CKL();
    if (int rc = exclusive_scan(x->cnt, cells + 1, x->start, x->tiles, st)) return rc;
    RG_CK(cudaMemsetAsync(x->cnt, 0, sizeof(int) * (cells + 1), st));
    cell_scatter<<<grid_of(v1), kT, 0, st>>>(v1, dim, x->pts, x->cell_of, x->start, x->cnt,
                                             x->spts, x->sid);
    RG_CKL();
    // the new vertices in cell order
    query_flags<<<grid_of(v1), kT, 0, st>>>(v1, v0, x->sid, x->qflag);
    RG_CKL();
    if (int rc = exclusive_scan(x->qflag, v1, x->qpos, x->tiles, st)) return rc;
    query_compact<<<grid_of(v1), kT, 0, st>>>(v1, v0, x->sid, x->qpos, x->qlist);
    RG_CKL();
    // nearest predecessors of the new vertices, then their edges
    with_dim(dim, [&](auto D) {
        knn_pred_kernel<decltype(D)::value><<<grid_of(nb * 32), kT, 0, st>>>(
            v0, v1, g, k, x->pts, x->spts, x->sid, x->start, x->qlist, x->knn);
    });
    RG_CKL();
    RG_CK(cudaMemsetAsync(x->rowc, 0, sizeof(int) * (nb + 1), st));
    with_dim(dim, [&](auto D) {
        pred_edge_mark<decltype(D)::value><<<grid_of(nb * k), kT, 0, st>>>(
            v0, v1, x->pts, k, x->knn, x->qlist, x->n_obs, x->obs, x->centers, x->radii, x->mode,
            x->n_check, x->keep, x->rowc);
    });
    RG_CKL();
    if (int rc = exclusive_scan(x->rowc, nb + 1, x->rowoff, x->tiles, st)) return rc;
    RG_CK(cudaMemcpyAsync(m_pinned, x->rowoff + nb, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    if (x->cost_f64)
        pred_edge_emit<double><<<grid_of(nb), kT, 0, st>>>(v0, v1, dim, x->pts, k, x->knn, x->keep,
                                                           x->rowoff, u, v,
                                                           static_cast<double *>(cost));
    else
        pred_edge_emit<float><<<grid_of(nb), kT, 0, st>>>(v0, v1, dim, x->pts, k, x->knn, x->keep,
                                                          x->rowoff, u, v,
                                                          static_cast<float *>(cost));
    RG_CKL();
    return 0;
}

extern "C" const double *rgg_explore_points(const rgg_explorer *x) { return x ? x->pts : nullptr; }

extern "C" int64_t rgg_explore_size(const rgg_explorer *x) { return x ? x->n : -1; }

extern "C" int rgg_explore_copy_points(const rgg_explorer *x, double *out, void *stream) {
    if (!x || !out) return 1;
    RG_CK(cudaMemcpyAsync(out, x->pts, sizeof(double) * x->n * x->dim, cudaMemcpyDeviceToDevice,
                          static_cast<cudaStream_t>(stream)));
    return 0;
}
