// Backward pass of the learned sampling proposal (mlp_kernels.cuh): from the
// selected draws, one per target, to the gradient of every parameter.
//
// Two thousand rows of 256 units are little work; spread over one kernel per
// step, with column sums taken by one thread per unit over all rows, it was all
// waiting (layer 1's sums 1014 us, the output layer's 84, a column sum 72, the
// GEMMs 180, at 2,048 rows).  So one kernel takes 32 rows at a time through the
// whole network and back with the activations in shared memory, every sum over
// rows is taken per CTA and finished in a second kernel in CTA order (the
// gradient is the same from run to run), and the two products over the rows
// are split so that they fill the GPU.  At 2,048 rows of 32 scenes: the row kernel
// 20 us, the parts of dW2 4, the finished sums 5, dW1g 5, Adam (one launch instead
// of seven) 12; a training step of 32,768 draws 1682 -> 151 us.
//
// The rounding points are those of the layer-by-layer path: BF16 weights, noise,
// h1, h2, da2 and per-scene sums D, FP32 sums; layer 1, both 256 x 256 products,
// the output layer and every elementwise step keep its order of operations, only
// the sums over rows are grouped differently.
#pragma once

#include "mlp_kernels.cuh"

namespace pirrt {
namespace mlp {

constexpr int kBwRows = 32;            // rows per tile
constexpr int kBwThreads = 256;        // one per hidden unit
constexpr int kBwPad = kHidden + 8;    // padded BF16 row
constexpr int kBwFPad = kHidden + 4;   // padded FP32 row
constexpr int kBwSplit = 16;           // at most: parts of the dW2 product

struct BwShared {
    __nv_bfloat16 W[kHidden][kBwPad];     // W2, then W2 transposed
    __nv_bfloat16 h1[kBwRows][kBwPad];
    __nv_bfloat16 h2[kBwRows][kBwPad];    // then da2
    float f[kBwRows][kBwFPad];            // da2, then da1
    float z[kBwRows][kNoise];             // noise, BF16-rounded
    uint32_t m1[kBwRows][kHidden / 32];   // a1 > 0
    float d[kBwRows][kOut];               // dL/da3
    float e[kBwRows];                     // squared error
    int scene[kBwRows];
};

// Per-CTA partial sums (over the CTA's rows, in row order).
struct BwPartials {
    float *w3;      // [ctas][2][256]
    float *b2;      // [ctas][256]
    float *w1n;     // [ctas][256][8]
    float *b1;      // [ctas][256]
    float *tail;    // [ctas][4]: loss, db3[0], db3[1]
    float *run;     // [rows][256]: da1 summed over a run of rows of one scene;
                    // CTA c's runs start at its first row
    int *run_scene; // [rows]: the run's scene, -1 past the CTA's last run
};

struct BwArgs {
    int rows, tiles, tiles_per_cta, n_scenes;
    const float *hg, *b1, *b2, *b3, *W1n;
    const __nv_bfloat16 *W2b, *W2Tb, *W3b;
    const int32_t *scene;
    const float *z, *target;
    __nv_bfloat16 *h1, *h2, *da2;  // [tiles * 32 x 256]
    float *y;                      // [rows x 2]
    BwPartials part;
    int *status;                   // error bits
};

constexpr int kBwErrScene = 2;

__device__ __forceinline__ void bw_load_matrix(BwShared &sh, const __nv_bfloat16 *W) {
    for (int i = threadIdx.x; i < kHidden * (kHidden / 8); i += kBwThreads) {
        const int r = i >> 5, k = (i & 31) * 8;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&sh.W[r][k])),
                     "l"(W + (size_t)r * kHidden + k)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// acc += A[32 x 256] * W[256 x 256]^T for this warp's 32 output columns, in steps
// of 16 along K in ascending order.
__device__ __forceinline__ void bw_product(const __nv_bfloat16 (*A)[kBwPad],
                                           const __nv_bfloat16 (*W)[kBwPad], int wn,
                                           float (&acc)[2][4][4]) {
    const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
#pragma unroll 4
    for (int kk = 0; kk < kHidden; kk += 16) {
        uint32_t af[2][4], bf[4][2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = i * 16 + gid;
            af[i][0] = *reinterpret_cast<const uint32_t *>(&A[r][kk + tig * 2]);
            af[i][1] = *reinterpret_cast<const uint32_t *>(&A[r + 8][kk + tig * 2]);
            af[i][2] = *reinterpret_cast<const uint32_t *>(&A[r][kk + tig * 2 + 8]);
            af[i][3] = *reinterpret_cast<const uint32_t *>(&A[r + 8][kk + tig * 2 + 8]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = wn + j * 8 + gid;
            bf[j][0] = *reinterpret_cast<const uint32_t *>(&W[c][kk + tig * 2]);
            bf[j][1] = *reinterpret_cast<const uint32_t *>(&W[c][kk + tig * 2 + 8]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j]);
    }
}

// A warp owns 32 columns of the two products; thread j owns column j of the sums
// over rows.
static __global__ void __launch_bounds__(kBwThreads, 1) backward_rows_kernel(const BwArgs A) {
    extern __shared__ __align__(16) unsigned char bw_smem[];
    BwShared &sh = *reinterpret_cast<BwShared *>(bw_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, j = tid;
    const int gid = lane >> 2, tig = lane & 3, wn = warp * 32;
    const int t0 = blockIdx.x * A.tiles_per_cta;
    const int t1 = t0 + A.tiles_per_cta < A.tiles ? t0 + A.tiles_per_cta : A.tiles;
    float w1n[kNoise], gw[kNoise] = {};
#pragma unroll
    for (int k = 0; k < kNoise; ++k)
        w1n[k] = __bfloat162float(__float2bfloat16_rn(A.W1n[j * kNoise + k]));
    const float b1 = A.b1[j], b30 = A.b3[0], b31 = A.b3[1];
    float g30 = 0.f, g31 = 0.f, gb2 = 0.f, gb1 = 0.f;  // dW3[:, j], db2[j], db1[j]
    float loss = 0.f, t30 = 0.f, t31 = 0.f;            // thread 0: loss, db3
    float run = 0.f;
    int run_scene = -1, runs = 0;
    const int run0 = t0 * kBwRows;
    const float scale = 2.f / (float)A.rows;
    for (int t = t0; t < t1; ++t) {
        const int r0 = t * kBwRows;
        bw_load_matrix(sh, A.W2b);
        if (tid < kBwRows) {
            const int r = r0 + tid;
            int s = 0;
            if (r < A.rows) {
                s = A.scene[r];
                if (s < 0 || s >= A.n_scenes) {
                    atomicOr(A.status, kBwErrScene);
                    s = 0;
                }
            }
            sh.scene[tid] = s;
        }
        {
            const int r = tid >> 3, k = tid & 7;
            sh.z[r][k] = r0 + r < A.rows
                             ? __bfloat162float(__float2bfloat16_rn(A.z[(size_t)(r0 + r) * kNoise + k]))
                             : 0.f;
        }
        __syncthreads();
        // ---- layer 1
#pragma unroll 8
        for (int r = 0; r < kBwRows; ++r) {
            float a = 0.f;
            if (r0 + r < A.rows) {
                a = A.hg[(size_t)sh.scene[r] * kHidden + j] + b1;
#pragma unroll
                for (int k = 0; k < kNoise; ++k) a += w1n[k] * sh.z[r][k];
            }
            const __nv_bfloat16 h = __float2bfloat16_rn(a > 0.f ? a : 0.f);
            sh.h1[r][j] = h;
            A.h1[(size_t)(r0 + r) * kHidden + j] = h;
            const uint32_t m = __ballot_sync(0xffffffffu, a > 0.f);
            if (lane == 0) sh.m1[r][warp] = m;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        // ---- layer 2; m2: which of this thread's 32 elements are positive
        uint32_t m2 = 0;
        {
            float acc[2][4][4] = {};
            bw_product(sh.h1, sh.W, wn, acc);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int r = i * 16 + gid + (x >> 1) * 8, c = wn + q * 8 + tig * 2 + (x & 1);
                        const float v = r0 + r < A.rows ? acc[i][q][x] + A.b2[c] : 0.f;
                        if (v > 0.f) m2 |= 1u << (i * 16 + q * 4 + x);
                        sh.h2[r][c] = __float2bfloat16_rn(v > 0.f ? v : 0.f);
                    }
        }
        __syncthreads();
        bw_load_matrix(sh, A.W2Tb);  // every warp is done with W2
        // ---- output layer: one warp per row
        for (int r = warp; r < kBwRows; r += kBwThreads / 32) {
            float s0 = 0.f, s1 = 0.f;
            for (int c = lane; c < kHidden; c += 32) {
                const float h = __bfloat162float(sh.h2[r][c]);
                s0 += h * __bfloat162float(A.W3b[c]);
                s1 += h * __bfloat162float(A.W3b[kHidden + c]);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                s0 += __shfl_xor_sync(0xffffffffu, s0, off);
                s1 += __shfl_xor_sync(0xffffffffu, s1, off);
            }
            if (lane == 0) {
                float d0 = 0.f, d1 = 0.f, e = 0.f;
                if (r0 + r < A.rows) {
                    const float y0 = 1.f / (1.f + __expf(-(s0 + b30)));
                    const float y1 = 1.f / (1.f + __expf(-(s1 + b31)));
                    A.y[2 * (size_t)(r0 + r)] = y0;
                    A.y[2 * (size_t)(r0 + r) + 1] = y1;
                    const float e0 = y0 - A.target[2 * (size_t)(r0 + r)];
                    const float e1 = y1 - A.target[2 * (size_t)(r0 + r) + 1];
                    d0 = scale * e0 * y0 * (1.f - y0);
                    d1 = scale * e1 * y1 * (1.f - y1);
                    e = e0 * e0 + e1 * e1;
                }
                sh.d[r][0] = d0;
                sh.d[r][1] = d1;
                sh.e[r] = e;
            }
        }
        __syncthreads();
        // ---- back through the output layer
        if (tid == 0)
            for (int r = 0; r < kBwRows; ++r) {
                loss += sh.e[r];
                t30 += sh.d[r][0];
                t31 += sh.d[r][1];
            }
#pragma unroll 8
        for (int r = 0; r < kBwRows; ++r) {
            const __nv_bfloat16 hb = sh.h2[r][j];
            A.h2[(size_t)(r0 + r) * kHidden + j] = hb;
            const float h = __bfloat162float(hb);
            g30 += sh.d[r][0] * h;
            g31 += sh.d[r][1] * h;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int r = i * 16 + gid + (x >> 1) * 8, c = wn + q * 8 + tig * 2 + (x & 1);
                    const float dh = sh.d[r][0] * __bfloat162float(A.W3b[c]) +
                                     sh.d[r][1] * __bfloat162float(A.W3b[kHidden + c]);
                    sh.f[r][c] = (m2 >> (i * 16 + q * 4 + x)) & 1u ? dh : 0.f;
                }
        __syncthreads();
#pragma unroll 8
        for (int r = 0; r < kBwRows; ++r) {
            const float da = sh.f[r][j];
            gb2 += da;
            const __nv_bfloat16 q = __float2bfloat16_rn(da);
            sh.h2[r][j] = q;
            A.da2[(size_t)(r0 + r) * kHidden + j] = q;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        // ---- back through layer 2
        {
            float acc[2][4][4] = {};
            bw_product(sh.h2, sh.W, wn, acc);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int r = i * 16 + gid + (x >> 1) * 8, c = wn + q * 8 + tig * 2 + (x & 1);
                        sh.f[r][c] = (sh.m1[r][c >> 5] >> (c & 31)) & 1u ? acc[i][q][x] : 0.f;
                    }
        }
        __syncthreads();
        // ---- layer 1's sums over rows; a run ends where the scene changes
        for (int r = 0; r < kBwRows && r0 + r < A.rows; ++r) {
            const float d = sh.f[r][j];
            const int s = sh.scene[r];
            if (s != run_scene) {
                if (run_scene >= 0) {
                    A.part.run[(size_t)(run0 + runs) * kHidden + j] = run;
                    if (tid == 0) A.part.run_scene[run0 + runs] = run_scene;
                    ++runs;
                }
                run_scene = s;
                run = 0.f;
            }
            run += d;
            gb1 += d;
#pragma unroll
            for (int k = 0; k < kNoise; ++k) gw[k] += d * sh.z[r][k];
        }
        __syncthreads();
    }
    if (run_scene >= 0) {
        A.part.run[(size_t)(run0 + runs) * kHidden + j] = run;
        if (tid == 0) A.part.run_scene[run0 + runs] = run_scene;
        ++runs;
    }
    for (int q = runs + tid; q < (t1 - t0) * kBwRows; q += kBwThreads)
        A.part.run_scene[run0 + q] = -1;
    const size_t c = blockIdx.x;
    A.part.w3[c * 512 + j] = g30;
    A.part.w3[c * 512 + kHidden + j] = g31;
    A.part.b2[c * kHidden + j] = gb2;
    A.part.b1[c * kHidden + j] = gb1;
#pragma unroll
    for (int k = 0; k < kNoise; ++k) A.part.w1n[(c * kHidden + j) * kNoise + k] = gw[k];
    if (tid == 0) {
        A.part.tail[c * 4] = loss;
        A.part.tail[c * 4 + 1] = t30;
        A.part.tail[c * 4 + 2] = t31;
    }
}

// dW2's parts: part[s] = sum over the rows of part s of da2[r]^T h1[r], a 64 x 64
// tile per CTA; both operands lie with the rows along K, so the fragments are
// read transposed.
static __global__ void __launch_bounds__(128)
dw2_parts_kernel(int rows_pad, int rows_per_part, const __nv_bfloat16 *__restrict__ da2,
                 const __nv_bfloat16 *__restrict__ h1, float *__restrict__ part) {
    constexpr int KT = 32, LD = 64 + 8;
    __shared__ __align__(16) __nv_bfloat16 sA[2][KT][LD], sB[2][KT][LD];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * 64, n0 = blockIdx.y * 64;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int k0 = blockIdx.z * rows_per_part;
    const int k1 = k0 + rows_per_part < rows_pad ? k0 + rows_per_part : rows_pad;
    auto load = [&](int b, int k) {
        if (k < k1) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int i = tid + q * 128, r = i >> 3, c = (i & 7) * 8;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(&sA[b][r][c])),
                             "l"(da2 + (size_t)(k + r) * kHidden + m0 + c)
                             : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(&sB[b][r][c])),
                             "l"(h1 + (size_t)(k + r) * kHidden + n0 + c)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[2][4][4] = {};
    load(0, k0);
    int b = 0;
    for (int k = k0; k < k1; k += KT, b ^= 1) {
        load(b ^ 1, k + KT);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < KT; kk += 16) {
            uint32_t af[2][4], bf[4][2];
            const int sub = lane >> 3, row = lane & 7;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                // 8 x 8 blocks (k, m): (0,0) (0,8) (8,0) (8,8), each transposed
                const uint32_t p = (uint32_t)__cvta_generic_to_shared(
                    &sA[b][kk + (sub >> 1) * 8 + row][wm + i * 16 + (sub & 1) * 8]);
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(af[i][0]), "=r"(af[i][1]), "=r"(af[i][2]), "=r"(af[i][3])
                             : "r"(p)
                             : "memory");
            }
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                // (k, n): (0,0) (8,0) (0,8) (8,8)
                const uint32_t p = (uint32_t)__cvta_generic_to_shared(
                    &sB[b][kk + (sub & 1) * 8 + row][wn + q * 8 + (sub >> 1) * 8]);
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(bf[q][0]), "=r"(bf[q][1]), "=r"(bf[q + 1][0]),
                               "=r"(bf[q + 1][1])
                             : "r"(p)
                             : "memory");
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) mma_bf16(acc[i][q], af[i], bf[q]);
        }
        __syncthreads();
    }
    float *out = part + (size_t)blockIdx.z * kHidden * kHidden;
    const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = m0 + wm + i * 16 + gid, c = n0 + wn + q * 8 + tig * 2;
            *reinterpret_cast<float2 *>(&out[(size_t)r * kHidden + c]) =
                make_float2(acc[i][q][0], acc[i][q][1]);
            *reinterpret_cast<float2 *>(&out[(size_t)(r + 8) * kHidden + c]) =
                make_float2(acc[i][q][2], acc[i][q][3]);
        }
}

// The sums finished, in part and CTA order: blocks [0, 256) a row of dW2 each,
// [256, 266) the small gradients and the loss, from 266 on the per-scene sums D
// (BF16), one scene each.
constexpr int kFinishRow = 256, kFinishSmall = 10;
static __global__ void __launch_bounds__(256)
finish_backward_kernel(int ctas, int splits, int slots, int rows, BwPartials part,
                       const float *__restrict__ w2part, float *__restrict__ gW2,
                       float *__restrict__ gW3, float *__restrict__ gb2, float *__restrict__ gb3,
                       float *__restrict__ gW1n, float *__restrict__ gb1,
                       float *__restrict__ loss, __nv_bfloat16 *__restrict__ D) {
    const int tid = threadIdx.x;
    if (blockIdx.x < kFinishRow) {
        const size_t i = (size_t)blockIdx.x * kHidden + tid;
        float s = 0.f;
        for (int p = 0; p < splits; ++p) s += w2part[(size_t)p * kHidden * kHidden + i];
        gW2[i] += s;
        return;
    }
    const int k = (int)blockIdx.x - kFinishRow;
    if (k < kFinishSmall) {
        // 8 blocks of dW1n, one of dW3, one of db1, db2, db3 and the loss
        if (k < 8) {
            const int i = k * 256 + tid;
            float s = 0.f;
            for (int c = 0; c < ctas; ++c) s += part.w1n[(size_t)c * kHidden * kNoise + i];
            gW1n[i] += s;
        } else if (k == 8) {
            float s0 = 0.f, s1 = 0.f;
            for (int c = 0; c < ctas; ++c) {
                s0 += part.w3[(size_t)c * 512 + tid];
                s1 += part.w3[(size_t)c * 512 + kHidden + tid];
            }
            gW3[tid] += s0;
            gW3[kHidden + tid] += s1;
        } else {
            float s1 = 0.f, s2 = 0.f;
            for (int c = 0; c < ctas; ++c) {
                s1 += part.b1[(size_t)c * kHidden + tid];
                s2 += part.b2[(size_t)c * kHidden + tid];
            }
            gb1[tid] += s1;
            gb2[tid] += s2;
            if (tid < 3) {
                float s = 0.f;
                for (int c = 0; c < ctas; ++c) s += part.tail[(size_t)c * 4 + tid];
                if (tid == 0) loss[0] = s / (float)rows;
                else gb3[tid - 1] += s;
            }
        }
        return;
    }
    // the scene's runs, 256 slots at a time, in order
    const int scene = k - kFinishSmall, lane = tid & 31, warp = tid >> 5;
    __shared__ int list[256], count[8];
    float s = 0.f;
    for (int q0 = 0; q0 < slots; q0 += 256) {
        const bool mine = q0 + tid < slots && part.run_scene[q0 + tid] == scene;
        const uint32_t b = __ballot_sync(0xffffffffu, mine);
        if (lane == 0) count[warp] = __popc(b);
        __syncthreads();
        int at = 0, n = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) at += count[w];
            n += count[w];
        }
        if (mine) list[at + __popc(b & ((1u << lane) - 1u))] = q0 + tid;
        __syncthreads();
        for (int q = 0; q < n; q += 8) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = q + u < n ? part.run[(size_t)list[q + u] * kHidden + tid] : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u];
        }
        __syncthreads();
    }
    D[(size_t)scene * kHidden + tid] = __float2bfloat16_rn(s);
}

// dW1g += D^T grid: C[j][c] += sum_s D[s][j] bf16(grid[s][c]), a 64 x 64 tile per
// CTA, scenes along K in ascending order, read transposed.
static __global__ void __launch_bounds__(128)
dw1g_kernel(int n_scenes, const __nv_bfloat16 *__restrict__ D, const float *__restrict__ grids,
            float *__restrict__ grad) {
    constexpr int KT = 32, LD = 64 + 8;
    __shared__ __align__(16) __nv_bfloat16 sA[KT][LD], sB[KT][LD];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * 64, n0 = blockIdx.y * 64;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    float acc[2][4][4] = {};
    for (int k = 0; k < n_scenes; k += KT) {
        for (int i = tid; i < KT * 64; i += 128) {
            const int r = i >> 6, c = i & 63;
            const bool in = k + r < n_scenes;
            sA[r][c] = in ? D[(size_t)(k + r) * kHidden + m0 + c] : __float2bfloat16_rn(0.f);
            sB[r][c] = __float2bfloat16_rn(in ? grids[(size_t)(k + r) * kGrid + n0 + c] : 0.f);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < KT; kk += 16) {
            uint32_t af[2][4], bf[4][2];
            const int sub = lane >> 3, row = lane & 7;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint32_t p = (uint32_t)__cvta_generic_to_shared(
                    &sA[kk + (sub >> 1) * 8 + row][wm + i * 16 + (sub & 1) * 8]);
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(af[i][0]), "=r"(af[i][1]), "=r"(af[i][2]), "=r"(af[i][3])
                             : "r"(p)
                             : "memory");
            }
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                const uint32_t p = (uint32_t)__cvta_generic_to_shared(
                    &sB[kk + (sub & 1) * 8 + row][wn + q * 8 + (sub >> 1) * 8]);
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(bf[q][0]), "=r"(bf[q][1]), "=r"(bf[q + 1][0]),
                               "=r"(bf[q + 1][1])
                             : "r"(p)
                             : "memory");
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) mma_bf16(acc[i][q], af[i], bf[q]);
        }
        __syncthreads();
    }
    const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = m0 + wm + i * 16 + gid, c = n0 + wn + q * 8 + tig * 2;
            float2 *p0 = reinterpret_cast<float2 *>(&grad[(size_t)r * kGrid + c]);
            float2 *p1 = reinterpret_cast<float2 *>(&grad[(size_t)(r + 8) * kGrid + c]);
            float2 v0 = *p0, v1 = *p1;
            v0.x += acc[i][q][0];
            v0.y += acc[i][q][1];
            v1.x += acc[i][q][2];
            v1.y += acc[i][q][3];
            *p0 = v0;
            *p1 = v1;
        }
}

// IMLE selection for training: the draw of target t (rows t*K .. t*K+K-1 of y)
// nearest the target, lowest index on ties, and its noise.  8 lanes per target.
static __global__ void __launch_bounds__(256)
select_noise_kernel(int n_targets, int K, const float *__restrict__ y,
                    const float *__restrict__ target, const float *__restrict__ z_all,
                    float *__restrict__ z_sel) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 3, l = threadIdx.x & 7;
    const int tt = t < n_targets ? t : n_targets - 1;
    const float tx = target[2 * (size_t)tt], ty = target[2 * (size_t)tt + 1];
    float best = 3.4e38f;
    int bi = 0x7fffffff;
    for (int k = l; k < K; k += 8) {
        const size_t r = (size_t)tt * K + k;
        const float dx = y[2 * r] - tx, dy = y[2 * r + 1] - ty;
        const float d = dx * dx + dy * dy;
        if (d < best) {
            best = d;
            bi = k;
        }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
        if (ob < best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
        }
    }
    if (bi == 0x7fffffff) bi = 0;  // no finite distance: the first draw
    if (t < n_targets) z_sel[(size_t)t * kNoise + l] = z_all[((size_t)t * K + bi) * kNoise + l];
}

// Adam over the packed parameters in one launch (the order W1g, W1n, b1, W2, b2,
// W3, b3), with the BF16 working copies of W1g, W2 (and transposed) and W3.
// Skipped when an earlier kernel of the call reported an error.
struct AdamArgs {
    float *w, *m, *v, *grad;
    __nv_bfloat16 *W1gb, *W2b, *W2Tb, *W3b;
    int64_t n, oW2, ob2, oW3, ob3, nW1g;
    float lr, beta1, beta2, eps, bc1, bc2;
    const int *status;
};

static __global__ void __launch_bounds__(256) adam_all_kernel(const AdamArgs A) {
    if (A.status != nullptr && __ldcg(A.status) != 0) return;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    const float gr = A.grad[i];
    const float mi = A.beta1 * A.m[i] + (1.f - A.beta1) * gr;
    const float vi = A.beta2 * A.v[i] + (1.f - A.beta2) * gr * gr;
    A.m[i] = mi;
    A.v[i] = vi;
    const float wi = A.w[i] - A.lr * (mi / A.bc1) / (sqrtf(vi / A.bc2) + A.eps);
    A.w[i] = wi;
    A.grad[i] = 0.f;
    const __nv_bfloat16 q = __float2bfloat16_rn(wi);
    if (i < A.nW1g) {
        A.W1gb[i] = q;
    } else if (i >= A.oW2 && i < A.ob2) {
        const int64_t k = i - A.oW2;
        A.W2b[k] = q;
        A.W2Tb[(k % kHidden) * kHidden + k / kHidden] = q;
    } else if (i >= A.oW3 && i < A.ob3) {
        A.W3b[i - A.oW3] = q;
    }
}

}  // namespace mlp
}  // namespace pirrt
