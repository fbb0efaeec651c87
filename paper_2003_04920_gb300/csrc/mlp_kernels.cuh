// Kernels of the learned sampling proposal: a 3-layer MLP mapping a scene's
// 64x64 occupancy grid plus 8-D Gaussian noise to a sample position,
//   a1 = W1g grid + W1n z + b1,  h1 = relu(a1)
//   a2 = W2 h1 + b2,             h2 = relu(a2)
//   y  = sigmoid(W3 h2 + b3)     in [0, 1]^2
// BF16 weights and layer inputs on the tensor cores (mma m16n8k16, FP32
// accumulate), FP32 master weights updated by Adam.  Trained by implicit
// maximum-likelihood estimation: for each target sample, K noise draws are
// pushed through the network and only the output nearest the target is
// pulled towards it (squared error).
#pragma once

#include <cuda_bf16.h>
#include <cstdint>

namespace pirrt {
namespace mlp {

constexpr int kGrid = 4096;   // 64 x 64 occupancy
constexpr int kNoise = 8;
constexpr int kHidden = 256;
constexpr int kOut = 2;

// ---------------------------------------------------------------------------
// C[M x N] (FP32, row-major, leading dim ldc) = A[M x K] * B[N x K]^T, A and
// B BF16 row-major with K contiguous ("NT").  M and N multiples of 64, K a
// multiple of 32, all leading dimensions multiples of 8 elements.  A 64 x 64
// CTA tile (M tiles along grid x, N tiles along grid y), four warps of
// 32 x 32, K in steps of 32 staged in shared memory; fragments are read with
// 32-bit shared loads in the m16n8k16 register layout.  beta = 0 overwrites
// C, 1 accumulates into it.
// ---------------------------------------------------------------------------
constexpr int kGT = 64, kGK = 32;

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4],
                                         const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__global__ void __launch_bounds__(128)
gemm_nt_bf16(int M, int N, int K, const __nv_bfloat16 *__restrict__ A, int lda,
             const __nv_bfloat16 *__restrict__ B, int ldb, float *__restrict__ C, int ldc,
             int beta) {
    __shared__ __align__(16) __nv_bfloat16 sA[kGT][kGK + 8];  // +8: fewer bank conflicts
    __shared__ __align__(16) __nv_bfloat16 sB[kGT][kGK + 8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * kGT, n0 = blockIdx.y * kGT;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int gid = lane >> 2, tig = lane & 3;
    float acc[2][4][4] = {};
    for (int k0 = 0; k0 < K; k0 += kGK) {
        // 64 x 32 BF16 per operand = 256 16-byte vectors; 2 per thread each
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int idx = tid + r * 128;
            const int row = idx >> 2, col = (idx & 3) * 8;
            *reinterpret_cast<uint4 *>(&sA[row][col]) =
                *reinterpret_cast<const uint4 *>(&A[(size_t)(m0 + row) * lda + k0 + col]);
            *reinterpret_cast<uint4 *>(&sB[row][col]) =
                *reinterpret_cast<const uint4 *>(&B[(size_t)(n0 + row) * ldb + k0 + col]);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kGK; kk += 16) {
            uint32_t af[2][4], bf[4][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = wm + i * 16 + gid;
                af[i][0] = *reinterpret_cast<const uint32_t *>(&sA[r][kk + tig * 2]);
                af[i][1] = *reinterpret_cast<const uint32_t *>(&sA[r + 8][kk + tig * 2]);
                af[i][2] = *reinterpret_cast<const uint32_t *>(&sA[r][kk + tig * 2 + 8]);
                af[i][3] = *reinterpret_cast<const uint32_t *>(&sA[r + 8][kk + tig * 2 + 8]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = wn + j * 8 + gid;
                bf[j][0] = *reinterpret_cast<const uint32_t *>(&sB[c][kk + tig * 2]);
                bf[j][1] = *reinterpret_cast<const uint32_t *>(&sB[c][kk + tig * 2 + 8]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = m0 + wm + i * 16 + gid, c = n0 + wn + j * 8 + tig * 2;
            float *c0 = &C[(size_t)r * ldc + c];
            float *c1 = &C[(size_t)(r + 8) * ldc + c];
            if (beta) {
                c0[0] += acc[i][j][0];
                c0[1] += acc[i][j][1];
                c1[0] += acc[i][j][2];
                c1[1] += acc[i][j][3];
            } else {
                c0[0] = acc[i][j][0];
                c0[1] = acc[i][j][1];
                c1[0] = acc[i][j][2];
                c1[1] = acc[i][j][3];
            }
        }
}

// ---------------------------------------------------------------------------
// The grid part of layer 1, once per scene: hg[s][j] = sum_k grid[s][k] W1g[j][k]
// (the grid rounded to BF16, FP32 accumulation) and hgb = hg + b1.
//
// 32 hidden-unit groups of 8 and a handful of scenes give few tiles, and each
// output is one accumulation over K = 4096: the time is the chain of 256
// dependent m16n8k16 steps (21 cycles each, 2.8 us) plus what it waits for its
// operands.  So a warp owns one 16 x 8 tile and takes the steps in order (the
// sums are those of gemm_nt_bf16, bit for bit), two warps of a CTA serve 32
// scenes, and all four keep a four-stage ring of asynchronous copies ahead of
// them: 256 values of K of W1g and of the caller's FP32 grids, which are
// converted on their way into the fragments.  Measured, 1 to 32 scenes:
// 99 us with 64 x 64 tiles, no prefetch, and conversion and transposition passes
// before it; 12 us for 32 now.
// ---------------------------------------------------------------------------
constexpr int kSceneN = 8;                 // hidden units per CTA
constexpr int kSceneM = 32;                // scenes per CTA
constexpr int kSceneK = 256, kSceneStages = 4;
constexpr int kSceneGRow = kSceneK + 8;    // padded rows (FP32 grids, BF16 weights)
struct SceneStage {
    float grid[kSceneM][kSceneGRow];
    __nv_bfloat16 w[kSceneN][kSceneGRow];
};
constexpr int kSceneSmem = kSceneStages * (int)sizeof(SceneStage);

__device__ __forceinline__ uint32_t pack2(float2 v) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(v.x, v.y);
    return *reinterpret_cast<const uint32_t *>(&p);
}

static __global__ void __launch_bounds__(128)
scene_features_kernel(int n_scenes, const float *__restrict__ grids,
                      const __nv_bfloat16 *__restrict__ W1gb, const float *__restrict__ b1,
                      float *__restrict__ hg, float *__restrict__ hgb) {
    extern __shared__ __align__(16) unsigned char scene_smem[];
    SceneStage *st = reinterpret_cast<SceneStage *>(scene_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n0 = blockIdx.x * kSceneN, c0 = blockIdx.y * kSceneM, s0 = c0 + warp * 16;
    const int rows = n_scenes - c0 < kSceneM ? n_scenes - c0 : kSceneM;
    const int gid = lane >> 2, tig = lane & 3;
    const bool vec = (reinterpret_cast<uintptr_t>(grids) & 15u) == 0u;
    auto load = [&](int chunk) {
        if (chunk < kGrid / kSceneK) {
            SceneStage &d = st[chunk % kSceneStages];
            const int k0 = chunk * kSceneK;
            if (vec) {
                for (int i = tid; i < rows * (kSceneK / 4); i += 128) {
                    const int r = i / (kSceneK / 4), k = i % (kSceneK / 4) * 4;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(&d.grid[r][k])),
                                 "l"(grids + (size_t)(c0 + r) * kGrid + k0 + k)
                                 : "memory");
                }
            } else {
                for (int i = tid; i < rows * kSceneK; i += 128) {
                    const int r = i / kSceneK, k = i % kSceneK;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(&d.grid[r][k])),
                                 "l"(grids + (size_t)(c0 + r) * kGrid + k0 + k)
                                 : "memory");
                }
            }
#pragma unroll
            for (int q = 0; q < kSceneN * kSceneK / 8 / 128; ++q) {
                const int i = tid + q * 128, r = i / (kSceneK / 8), k = i % (kSceneK / 8) * 8;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(&d.w[r][k])),
                             "l"(W1gb + (size_t)(n0 + r) * kGrid + k0 + k)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // rows past the last scene stay zero (their results are not stored)
    for (int b = 0; b < kSceneStages; ++b)
        for (int i = tid; i < (kSceneM - rows) * kSceneGRow; i += 128)
            st[b].grid[rows + i / kSceneGRow][i % kSceneGRow] = 0.f;
#pragma unroll
    for (int c = 0; c < kSceneStages - 1; ++c) load(c);
    const bool live = warp < 2 && s0 < n_scenes;  // warp-uniform
    float acc[4] = {};
#pragma unroll 1
    for (int c = 0; c < kGrid / kSceneK; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kSceneStages - 2) : "memory");
        __syncthreads();
        load(c + kSceneStages - 1);  // into the stage read last turn
        if (!live) continue;
        const SceneStage &d = st[c % kSceneStages];
        const float *ga = &d.grid[warp * 16 + gid][tig * 2], *gb = ga + 8 * kSceneGRow;
        const __nv_bfloat16 *wr = &d.w[gid][tig * 2];
#pragma unroll
        for (int k = 0; k < kSceneK; k += 16) {
            const uint32_t af[4] = {pack2(*reinterpret_cast<const float2 *>(ga + k)),
                                    pack2(*reinterpret_cast<const float2 *>(gb + k)),
                                    pack2(*reinterpret_cast<const float2 *>(ga + k + 8)),
                                    pack2(*reinterpret_cast<const float2 *>(gb + k + 8))};
            const uint32_t bf[2] = {*reinterpret_cast<const uint32_t *>(wr + k),
                                    *reinterpret_cast<const uint32_t *>(wr + k + 8)};
            mma_bf16(acc, af, bf);
        }
    }
    if (!live) return;
    const int c = n0 + tig * 2;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int s = s0 + gid + 8 * h;
        if (s >= n_scenes) continue;
        const size_t o = (size_t)s * kHidden + c;
        hg[o] = acc[2 * h];
        hg[o + 1] = acc[2 * h + 1];
        hgb[o] = acc[2 * h] + b1[c];
        hgb[o + 1] = acc[2 * h + 1] + b1[c + 1];
    }
}

// ---------------------------------------------------------------------------
// Elementwise and small kernels.  Rows are padded to multiples of 64; padded
// rows carry zeros and are excluded by `rows` where it matters.
// ---------------------------------------------------------------------------

// FP32 -> BF16 (round to nearest even), out[r][c] for r < rows, c < cols, with
// an optional transposed copy outT[c][r] (leading dim ldt).
__global__ void to_bf16(int rows, int cols, const float *__restrict__ in, int ldi,
                        __nv_bfloat16 *__restrict__ out, int ldo, __nv_bfloat16 *__restrict__ outT,
                        int ldt) {
    const int64_t total = (int64_t)rows * cols;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(i / cols), c = (int)(i % cols);
        const __nv_bfloat16 v = __float2bfloat16_rn(in[(size_t)r * ldi + c]);
        if (out) out[(size_t)r * ldo + c] = v;
        if (outT) outT[(size_t)c * ldt + r] = v;
    }
}

// Layer 1 for sample rows: a1[r][j] = hg[scene[r]][j] + sum_k W1n[j][k] z[r][k]
// + b1[j] (FP32; z and W1n used in their BF16-rounded values), h1 = relu(a1) as
// BF16; row r's scene is scene[r / rows_per_scene].
__global__ void layer1_rows(int rows, int rows_pad, const float *__restrict__ hg,
                            const int32_t *__restrict__ scene, int rows_per_scene,
                            const float *__restrict__ z, const float *__restrict__ W1n,
                            const float *__restrict__ b1,
                            float *__restrict__ a1, __nv_bfloat16 *__restrict__ h1) {
    const int64_t total = (int64_t)rows_pad * kHidden;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(i / kHidden), j = (int)(i % kHidden);
        float a = 0.f;
        if (r < rows) {
            a = hg[(size_t)scene[r / rows_per_scene] * kHidden + j] + b1[j];
#pragma unroll
            for (int k = 0; k < kNoise; ++k)
                a += __bfloat162float(__float2bfloat16_rn(W1n[j * kNoise + k])) *
                     __bfloat162float(__float2bfloat16_rn(z[r * kNoise + k]));
        }
        a1[i] = a;
        const __nv_bfloat16 h = __float2bfloat16_rn(r < rows && a > 0.f ? a : 0.f);
        h1[i] = h;
    }
}

// a2 += b2 (rows), h2 = relu(a2) as BF16.
__global__ void bias_relu(int rows, int rows_pad, float *__restrict__ a, const float *__restrict__ b,
                          __nv_bfloat16 *__restrict__ h) {
    const int64_t total = (int64_t)rows_pad * kHidden;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(i / kHidden), j = (int)(i % kHidden);
        const float v = r < rows ? a[i] + b[j] : 0.f;
        a[i] = v;
        const __nv_bfloat16 q = __float2bfloat16_rn(v > 0.f ? v : 0.f);
        h[i] = q;
    }
}

// Output layer (N = 2, plain dot products): y = sigmoid(W3 h2 + b3), one warp
// per row.
__global__ void layer3_rows(int rows, const __nv_bfloat16 *__restrict__ h2,
                            const __nv_bfloat16 *__restrict__ W3b, const float *__restrict__ b3,
                            float *__restrict__ y) {
    const int lane = threadIdx.x & 31;
    for (int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows;
         r += gridDim.x * (blockDim.x >> 5)) {
        float s0 = 0.f, s1 = 0.f;
        for (int j = lane; j < kHidden; j += 32) {
            const float h = __bfloat162float(h2[(size_t)r * kHidden + j]);
            s0 += h * __bfloat162float(W3b[j]);
            s1 += h * __bfloat162float(W3b[kHidden + j]);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, off);
            s1 += __shfl_xor_sync(0xffffffffu, s1, off);
        }
        if (lane == 0) {
            y[2 * r] = 1.f / (1.f + __expf(-(s0 + b3[0])));
            y[2 * r + 1] = 1.f / (1.f + __expf(-(s1 + b3[1])));
        }
    }
}

// IMLE selection: for target t (rows t*K .. t*K+K-1 of y) the draw whose
// output is nearest the target (lowest index on ties).
__global__ void imle_select(int n_targets, int K, const float *__restrict__ y,
                            const float *__restrict__ target, int32_t *__restrict__ pick) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_targets; t += gridDim.x * blockDim.x) {
        float best = 3.4e38f;
        int bi = 0;
        for (int k = 0; k < K; ++k) {
            const float dx = y[2 * (t * K + k)] - target[2 * t];
            const float dy = y[2 * (t * K + k) + 1] - target[2 * t + 1];
            const float d = dx * dx + dy * dy;
            if (d < best) {
                best = d;
                bi = k;
            }
        }
        pick[t] = bi;
    }
}

// 50/50 (or any fraction) mixture with uniform samples: row r keeps the
// network's output when coin[r] < learned_fraction, else the caller's uniform
// sample.  The random numbers are inputs, so the mixture is reproducible.
__global__ void mix_samples(int rows, const float *__restrict__ y, const float *__restrict__ uni,
                            const float *__restrict__ coin, float learned_fraction,
                            float *__restrict__ out) {
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += gridDim.x * blockDim.x) {
        const bool learned = coin[r] < learned_fraction;
        out[2 * r] = learned ? y[2 * r] : uni[2 * r];
        out[2 * r + 1] = learned ? y[2 * r + 1] : uni[2 * r + 1];
    }
}

}  // namespace mlp
}  // namespace pirrt
