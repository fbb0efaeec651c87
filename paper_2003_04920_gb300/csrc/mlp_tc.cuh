// Fused forward pass of the learned sampling proposal on the 5th-generation
// tensor cores (tcgen05): the three layers of the network of mlp_kernels.cuh,
//   a1 = W1g grid + W1n z + b1,  h1 = relu(a1)
//   a2 = W2 h1 + b2,             h2 = relu(a2)
//   y  = sigmoid(W3 h2 + b3)
// for 128 sample rows per tile, with the activations kept on chip: every
// contraction is a tcgen05.mma chain (BF16 operands in shared memory, FP32
// accumulator in tensor memory), every elementwise step runs on CUDA cores
// beside it, and only the noise in and the two outputs per row touch HBM (40
// bytes per row).
//
//   layer 1: D[128 x 256] = Z[128 x 16] * W1n'[256 x 16]^T   (K padded 8 -> 16)
//            h1 = relu(D + (W1g grid + b1)[scene])  -> H (shared, BF16)
//   layer 2: D[128 x 256] = H[128 x 256] * W2[256 x 256]^T
//            h2 = relu(D + b2), rounded to BF16, kept in registers
//   layer 3: y = sigmoid(W3 h2 + b3): two FP32 dot products per row on the
//            CUDA cores (N = 2 is too narrow for an MMA round trip)
//
// The grid part of layer 1 (one 4096 x 256 product per scene) is computed
// once per call outside this kernel; W1g grid + b1 arrives per scene.  The
// rounding points are those of the unfused path: BF16 weights, BF16 noise,
// BF16 h1 and h2, FP32 accumulation, FP32 bias additions and sigmoid.
//
// Persistent: one CTA per SM (about 210 KB of shared memory: W2 stays resident
// across tiles), tiles strided over the grid, and three roles that hand tiles
// to one another through mbarriers:
//   * one thread issues the MMAs.  Layer 2 of a tile follows H block by block
//     (64 columns each) and gives each block back as it is done with it; the
//     next tile's layer 1 goes out in front of the last block;
//   * eight warps turn layer 1's accumulator into H;
//   * eight warps turn layer 2's accumulator into y.
// So the tensor core works on one tile while the CUDA cores finish the one
// before it and prepare the one after it.  With both epilogues on the same
// warps and a CTA barrier between the phases the tensor core waited for each
// of them: 10^6 rows over 32 scenes took 418 us, now 163.
//
// What bounds it is the path that MMA operands, gathers and epilogues share into
// shared memory and L1, and the chain between the roles: the MMAs alone take 1.44 us
// a tile, with either epilogue beside them 2.4, with both 2.9.  The layouts below are
// chosen to move fewer bytes (that path was 100 % busy before the last of these
// steps, 62 % after).  Both accumulators are read as 16 lanes x 32 columns, which
// gives a thread several columns of four rows instead of many columns of one: a
// row's scene terms then arrive as whole 128-byte lines (a thread per row: one
// 16-byte piece of 32 different lines a load, 250 us a call against 225), and b2
// and W3 are read once for four rows.  The accumulators' columns are permuted
// (column_unit: in the weights' rows, at no cost) so that a thread's eight are
// consecutive.  N = 256 instructions read H once instead of twice (225 -> 209 us a
// call together with two-wide FP32 arithmetic).  Tried and slower: a second
// register set for the next block's sums (233 - 267 us, spills), a loading warp
// (213 - 227), layer 2 in two column halves with early release of the accumulator
// (212 - 223).
//
// Every wait is bounded.  A wait that expires ends every other wait of its CTA at
// once, so the roles run to the end without waiting for one another and issue no
// further MMA; the CTA waits a bounded time more for the MMAs in flight, frees
// its tensor memory and returns with an error bit set.
//
// Operand layouts in shared memory (K-major, i.e. each row's K elements
// contiguous, as tcgen05 descriptors describe them):
//   * 128-byte swizzle for H and W2: 8-row groups of 8 x 128 bytes, the
//     16-byte chunk c of row r stored at chunk c ^ (r mod 8); K in blocks of
//     64 elements, one such block of all rows after another;
//   * no swizzle for the K = 16 operands Z and W1n': 8 x 16-byte core
//     matrices, the two K halves 128 bytes apart, 8-row groups 256 bytes
//     apart.
#pragma once

#include <cuda_bf16.h>
#include <cstdint>

#include "mlp_kernels.cuh"

namespace pirrt {
namespace mlp {
namespace tc {

constexpr int kRowsPerTile = 128;
constexpr int kHiddenWarps = 8;   // layer-1 epilogue
constexpr int kOutputWarps = 8;   // layer-2 epilogue, layer 3
constexpr int kThreads = (kHiddenWarps + kOutputWarps + 1) * 32;  // ... and the warp that issues
constexpr int kKBlocks = 4;       // H in blocks of 64 columns, handed over one by one
constexpr uint32_t kTmemCols = 512;  // a layer-1 and a layer-2 accumulator of 256 columns
constexpr int kK1 = 16;   // layer-1 K padded to one MMA step

// shared-memory map, offsets from a 1024-byte-aligned base
constexpr int kW2Bytes = kHidden * kHidden * 2;     // 131072
constexpr int kHBytes = kRowsPerTile * kHidden * 2;  // 65536
constexpr int kZBytes = kRowsPerTile * kK1 * 2;      // 4096
constexpr int kW1Bytes = kHidden * kK1 * 2;          // 8192
constexpr int oW2 = 0;
constexpr int oH = oW2 + kW2Bytes;
constexpr int oZ = oH + kHBytes;
constexpr int oW1 = oZ + kZBytes;
constexpr int oB2 = oW1 + kW1Bytes;          // b2: 256 FP32
constexpr int oW3 = oB2 + kHidden * 4;       // BF16 W3 as FP32 [2][256]
constexpr int oY = oW3 + kHidden * 2 * 4;    // second half's layer-3 sums [tile parity][128 rows][2]
constexpr int oBar = oY + 2 * kRowsPerTile * 2 * 4;  // mbarriers
// one phase of each mbarrier per tile
constexpr int bAcc1Full = 0;                 // layer 1 is in its accumulator (commit)
constexpr int bNextReady = 1;                // ... has been read, and the next noise is staged
constexpr int bHFull = 2;                    // [kKBlocks] block of H written
constexpr int bHFree = bHFull + kKBlocks;    // [kKBlocks] ... and read (commit)
constexpr int bAcc2Full = bHFree + kKBlocks; // layer 2 is in its accumulator (commit)
constexpr int bAcc2Free = bAcc2Full + 1;     // ... and read
constexpr int bDrained = bAcc2Free + 1;      // every MMA of the CTA has ended (commit)
constexpr int kBars = bDrained + 1;
constexpr int oTmem = oBar + kBars * 8;      // TMEM base address written by tcgen05.alloc
constexpr int oBad = oTmem + 4;              // a wait expired
constexpr int oLate = oBad + 4;              // ... the last one
constexpr int kSmemUsed = oLate + 4;
constexpr int kSmemBytes = kSmemUsed + 1024;  // + alignment slack

constexpr unsigned long long kMmaWaitNs = 1000000000ull;  // 1 s per wait

// Error bits the kernel leaves in *status (0 = success).
constexpr int kErrTimeout = 1;
constexpr int kErrScene = 2;

__device__ __forceinline__ uint32_t saddr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// byte offset of the 16-byte chunk holding elements k .. k+7 of row r in a
// 128-byte-swizzled K-major operand of `rows` rows
__device__ __forceinline__ uint32_t sw128(int r, int k, int rows) {
    const int kb = k >> 6, c = (k >> 3) & 7;
    return (uint32_t)(kb * rows * 128 + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4));
}

// byte offset of the 16-byte core-matrix row holding elements 8*kc .. 8*kc+7
// of row r in an unswizzled K-major operand with K = 16
__device__ __forceinline__ uint32_t plain16(int r, int kc) {
    return (uint32_t)((r >> 3) * 256 + kc * 128 + (r & 7) * 16);
}

// shared-memory matrix descriptor: start address, leading-dimension byte
// offset (LBO), stride-dimension byte offset (SBO), descriptor version 1,
// swizzle mode (0 none, 2 = 128-byte)
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo,
                                              uint32_t swizzle) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46) | ((uint64_t)swizzle << 61);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                    uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(saddr(bar))
                 : "memory");
}

__device__ __forceinline__ void fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// generic-proxy shared-memory writes made visible to the tensor core's reads
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ bool bar_try(uint64_t *bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(saddr(bar)), "r"(parity)
        : "memory");
    return done != 0u;
}

// Bounded wait; the first expiry in a CTA ends every other wait at once.
__device__ __forceinline__ bool bar_wait(uint64_t *bar, uint32_t parity, int *s_bad,
                                         unsigned long long ns) {
    if (bar_try(bar, parity)) return true;
    const unsigned long long t0 = now_ns();
    for (;;) {
        if (*reinterpret_cast<volatile int *>(s_bad)) return false;
        if (bar_try(bar, parity)) return true;
        if (now_ns() - t0 > ns) {
            *reinterpret_cast<volatile int *>(s_bad) = 1;
            return false;
        }
    }
}

// Arrival of a whole warp: every lane's work before it, one count.
__device__ __forceinline__ void warp_arrive(uint64_t *bar) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}

// 16 lanes (rows) x 32 FP32 columns: register 4 k + 2 u + j of thread i holds
// row i / 4 + 8 u, column 8 k + 2 (i mod 4) + j.  Not complete before
// tmem_wait32.
__device__ __forceinline__ void tmem_ld16x32(uint32_t taddr, uint32_t *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// 8 FP32 values, 32-byte aligned, read-only, in one load.
__device__ __forceinline__ void ldg8(const float *p, float (&v)[8]) {
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
          "=f"(v[7])
        : "l"(p));
}

// Completes two tmem_ld16x32; tied to their registers so that no use is
// scheduled before it.
__device__ __forceinline__ void tmem_wait32(uint32_t (&r)[32]) {
#define PIRRT_TC_TIE8(o)                                                                          \
    "+r"(r[o]), "+r"(r[o + 1]), "+r"(r[o + 2]), "+r"(r[o + 3]), "+r"(r[o + 4]), "+r"(r[o + 5]),   \
        "+r"(r[o + 6]), "+r"(r[o + 7])
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : PIRRT_TC_TIE8(0), PIRRT_TC_TIE8(8), PIRRT_TC_TIE8(16), PIRRT_TC_TIE8(24)
                 :
                 : "memory");
#undef PIRRT_TC_TIE8
}

// Row of a group of eight that layer 1's accumulator lane p (mod 8) holds, and
// the lane that holds row r.  Lanes 2 j and 2 j + 1 hold rows four apart, so the
// four threads of each store their 16-byte chunks of the 128-byte-swizzled H
// to eight different bank groups.
__device__ __forceinline__ int lane_row(int p) { return (p & ~7) | ((p & 1) << 2) | ((p >> 1) & 3); }
__device__ __forceinline__ int row_lane(int r) { return (r & ~7) | ((r & 3) << 1) | ((r >> 2) & 1); }

// Hidden unit of layer 1's accumulator column n: a thread of tmem_ld16x32 gets
// eight consecutive units of its row (columns 2 (i mod 4) + {0, 1} of four groups
// of eight).
__device__ __forceinline__ int column_unit(int n) {
    return (n & ~31) | (((n >> 1) & 3) << 3) | (((n >> 3) & 3) << 1) | (n & 1);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&p);
}


// Two FP32 values in a register pair, and arithmetic on both at once (each
// rounded as the scalar instruction rounds).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pair(float x, float y) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpair(f32x2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

struct FwdArgs {
    int rows, n_scenes;
    const float *hgb;              // [n_scenes x 256] W1g grid + b1 per scene
    const int32_t *scene;          // [rows / rows_per_scene]: row r's is scene[r / rows_per_scene]
    int rows_per_scene;
    const float *z;                // [rows x 8]
    const float *W1n;              // [256 x 8] FP32 master weights (rounded here)
    const __nv_bfloat16 *W2b;      // [256 x 256], row = output unit
    const float *b2;               // [256]
    const __nv_bfloat16 *W3b;      // [2 x 256]
    const float *b3;               // [2]
    float *y;                      // [rows x 2] or null
    const float *uniform_xy;       // mixture: out[r] = coin[r] < frac ? y[r] : uniform_xy[r]
    const float *coin;
    float frac;
    float *out;                    // [rows x 2] or null
    __nv_bfloat16 *cap_h1, *cap_h2;  // optional copies of h1 / h2 [rows x 256]
    int *status;                   // error bits (kErr*)
};

// noise of row r as BF16 pairs (zeros past the last row)
__device__ __forceinline__ uint4 load_z(const float *z, int r, bool valid) {
    if (!valid) return make_uint4(0u, 0u, 0u, 0u);
    const float4 z0 = *reinterpret_cast<const float4 *>(z + (size_t)r * kNoise);
    const float4 z1 = *reinterpret_cast<const float4 *>(z + (size_t)r * kNoise + 4);
    return make_uint4(pack_bf16(z0.x, z0.y), pack_bf16(z0.z, z0.w), pack_bf16(z1.x, z1.y),
                      pack_bf16(z1.z, z1.w));
}

__global__ void __launch_bounds__(kThreads, 1) mlp_forward_tc(const FwdArgs A) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = saddr(smem_raw);
    uint8_t *sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    const uint32_t sb = saddr(sm);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + oBar);
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(sm + oTmem);
    int *s_bad = reinterpret_cast<int *>(sm + oBad);
    float *s_b2 = reinterpret_cast<float *>(sm + oB2);
    float *s_w3 = reinterpret_cast<float *>(sm + oW3);  // [2][256]
    float2 *s_y = reinterpret_cast<float2 *>(sm + oY);    // [tile parity][row]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int quad = warp & 3, part = (warp >> 2) & 1;  // TMEM lane quadrant, column part

    // resident operands: W2 (swizzled), W1n' (K 8..15 zero), the zero K half
    // of Z, b2, W3 (BF16 values as FP32); rows of W2 and W1n' in the order of
    // the accumulators' columns
    for (int i = tid; i < kHidden * (kHidden / 8); i += kThreads) {
        const int n = i >> 5, c = i & 31;
        const uint4 v = *reinterpret_cast<const uint4 *>(
            A.W2b + (size_t)column_unit(n) * kHidden + c * 8);
        *reinterpret_cast<uint4 *>(sm + oW2 + sw128(n, c * 8, kHidden)) = v;
    }
    for (int n = tid; n < kHidden; n += kThreads) {
        const float *w = A.W1n + column_unit(n) * kNoise;
        *reinterpret_cast<uint4 *>(sm + oW1 + plain16(n, 0)) =
            make_uint4(pack_bf16(w[0], w[1]), pack_bf16(w[2], w[3]), pack_bf16(w[4], w[5]),
                       pack_bf16(w[6], w[7]));
        *reinterpret_cast<uint4 *>(sm + oW1 + plain16(n, 1)) = make_uint4(0u, 0u, 0u, 0u);
        s_b2[n] = A.b2[n];
        s_w3[n] = __bfloat162float(A.W3b[n]);
        s_w3[kHidden + n] = __bfloat162float(A.W3b[kHidden + n]);
    }
    const int ntiles = (A.rows + kRowsPerTile - 1) / kRowsPerTile;
    const int first = blockIdx.x, step = gridDim.x;
    if (tid < kRowsPerTile) {
        *reinterpret_cast<uint4 *>(sm + oZ + plain16(tid, 1)) = make_uint4(0u, 0u, 0u, 0u);
        const int r = first * kRowsPerTile + tid;
        *reinterpret_cast<uint4 *>(sm + oZ + plain16(row_lane(tid), 0)) =
            load_z(A.z, r, r < A.rows);
    }
    if (tid == 0) {
        s_bad[0] = s_bad[1] = 0;
        for (int b = 0; b < kBars; ++b) {
            const uint32_t count = b == bNextReady || (b >= bHFull && b < bHFree) ? kHiddenWarps
                                   : b == bAcc2Free ? kOutputWarps : 1;
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar + b)), "r"(count)
                         : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(saddr(s_tmem)), "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t acc1 = *s_tmem, acc2 = acc1 + 256u;
    const uint32_t lane_off = (uint32_t)(quad * 32) << 16;

    if (warp < kHiddenWarps) {
        // ---- layer-1 epilogue: rows 32 quad .. + 31, half of each 64-column block
        const int q = lane & 3, sub = lane >> 2;
        auto row_scene = [&](int tile, int j) {  // scene of this thread's j-th row
            const int r = tile * kRowsPerTile + quad * 32 + 8 * j + lane_row(sub);
            if (tile >= ntiles || r >= A.rows) return 0;
            return A.scene[A.rows_per_scene == 1 ? r : r / A.rows_per_scene];
        };
        int s[4], sn[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) sn[j] = row_scene(first, j);
        uint32_t it = 0;
        for (int tile = first; tile < ntiles; ++it, tile += step) {
            const int next = tile + step;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                s[j] = sn[j];
                if (s[j] < 0 || s[j] >= A.n_scenes) {
                    if (part == 0 && q == 0) atomicOr(A.status, kErrScene);
                    s[j] = 0;
                }
            }
            // the next tile's scenes and noise, in flight during this one
#pragma unroll
            for (int j = 0; j < 4; ++j) sn[j] = row_scene(next, j);
            uint4 zn = make_uint4(0u, 0u, 0u, 0u);
            if (tid < kRowsPerTile && next < ntiles) {
                const int rn = next * kRowsPerTile + tid;
                zn = load_z(A.z, rn, rn < A.rows);
            }
            bar_wait(bar + bAcc1Full, it & 1u, s_bad, kMmaWaitNs);
            fence_after();
#pragma unroll 1
            for (int b = 0; b < kKBlocks; ++b) {
                const int col = b * 64 + part * 32;
                uint32_t v[32];
                tmem_ld16x32(acc1 + lane_off + col, v);
                tmem_ld16x32(acc1 + lane_off + (16u << 16) + col, v + 16);
                float hb[4][8];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    ldg8(A.hgb + (size_t)s[j] * kHidden + col + 8 * q, hb[j]);
                tmem_wait32(v);
                if (b == kKBlocks - 1) {
                    // layer 1 of this tile has been read: the next one's noise
                    // takes the place of the noise it was computed from
                    if (tid < kRowsPerTile && next < ntiles) {
                        *reinterpret_cast<uint4 *>(sm + oZ + plain16(row_lane(tid), 0)) = zn;
                        fence_async_smem();
                    }
                    fence_before();
                    warp_arrive(bar + bNextReady);
                }
                if (it > 0) bar_wait(bar + bHFree + b, (it - 1) & 1u, s_bad, kMmaWaitNs);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t *w = v + (j >> 1) * 16 + (j & 1) * 2;
                    uint32_t o[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        o[k] = pack_bf16(fmaxf(hb[j][2 * k] + __uint_as_float(w[4 * k]), 0.f),
                                         fmaxf(hb[j][2 * k + 1] + __uint_as_float(w[4 * k + 1]), 0.f));
                    const uint4 o4 = make_uint4(o[0], o[1], o[2], o[3]);
                    const int row = quad * 32 + 8 * j + lane_row(sub), r = tile * kRowsPerTile + row;
                    *reinterpret_cast<uint4 *>(sm + oH + sw128(row, col + 8 * q, kRowsPerTile)) = o4;
                    if (A.cap_h1 && r < A.rows)
                        *reinterpret_cast<uint4 *>(A.cap_h1 + (size_t)r * kHidden + col + 8 * q) = o4;
                }
                fence_async_smem();
                warp_arrive(bar + bHFull + b);
            }
        }
    } else if (warp < kHiddenWarps + kOutputWarps) {
        // ---- layer-2 epilogue and layer 3: rows 32 quad .. + 31, 128 columns a warp
        const int q = lane & 3, sub = lane >> 2, col0 = part * 128;
        const float b30 = A.b3[0], b31 = A.b3[1];
        uint32_t it = 0;
        for (int tile = first; tile < ntiles; ++it, tile += step) {
            bar_wait(bar + bAcc2Full, it & 1u, s_bad, kMmaWaitNs);
            fence_after();
            f32x2 z0[4] = {0, 0, 0, 0}, z1[4] = {0, 0, 0, 0};  // even and odd units apart
#pragma unroll 1
            for (int c = 0; c < 128; c += 32) {
                uint32_t v[32];
                tmem_ld16x32(acc2 + lane_off + col0 + c, v);
                tmem_ld16x32(acc2 + lane_off + (16u << 16) + col0 + c, v + 16);
                const int unit = col0 + c + 8 * q;  // eight units from here, of four rows
                tmem_wait32(v);
                if (c == 96) {
                    fence_before();
                    warp_arrive(bar + bAcc2Free);
                }
                uint32_t p[4][4];
#pragma unroll
                for (int k = 0; k < 4; k += 2) {  // four units
                    const ulonglong2 b2 =
                        *reinterpret_cast<const ulonglong2 *>(s_b2 + unit + 2 * k);
                    const ulonglong2 wa =
                        *reinterpret_cast<const ulonglong2 *>(s_w3 + unit + 2 * k);
                    const ulonglong2 wb =
                        *reinterpret_cast<const ulonglong2 *>(s_w3 + kHidden + unit + 2 * k);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t *w = v + (j >> 1) * 16 + (j & 1) * 2 + 4 * (k + i);
                            const float2 t =
                                unpair(add2(pair(__uint_as_float(w[0]), __uint_as_float(w[1])),
                                            i ? b2.y : b2.x));
                            const uint32_t o = pack_bf16(fmaxf(t.x, 0.f), fmaxf(t.y, 0.f));
                            p[j][k + i] = o;
                            // layer 3 on the BF16 h2 values
                            const f32x2 h = pair(__uint_as_float(o << 16),
                                                 __uint_as_float(o & 0xFFFF0000u));
                            z0[j] = fma2(h, i ? wa.y : wa.x, z0[j]);
                            z1[j] = fma2(h, i ? wb.y : wb.x, z1[j]);
                        }
                    }
                }
                if (A.cap_h2) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int r = tile * kRowsPerTile + quad * 32 + 8 * j + sub;
                        if (r < A.rows)
                            *reinterpret_cast<uint4 *>(A.cap_h2 + (size_t)r * kHidden + unit) =
                                make_uint4(p[j][0], p[j][1], p[j][2], p[j][3]);
                    }
                }
            }
            // the four threads of a row, then (once per tile) the two halves;
            // the buffer alternates, so the first half has read a tile's sums
            // before they are overwritten
            float a0 = 0.f, a1 = 0.f;  // row 8 q + sub
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 e0 = unpair(z0[j]), e1 = unpair(z1[j]);
                float y0 = e0.x + e0.y, y1 = e1.x + e1.y;
                y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
                y1 += __shfl_xor_sync(0xffffffffu, y1, 1);
                y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
                y1 += __shfl_xor_sync(0xffffffffu, y1, 2);
                if (j == q) {
                    a0 = y0;
                    a1 = y1;
                }
            }
            const int row = quad * 32 + 8 * q + sub, r = tile * kRowsPerTile + row;
            if (part == 1) s_y[(it & 1u) * kRowsPerTile + row] = make_float2(a0, a1);
            asm volatile("bar.sync 1, %0;" ::"n"(kOutputWarps * 32) : "memory");
            if (part == 0 && r < A.rows) {
                const float2 pb = s_y[(it & 1u) * kRowsPerTile + row];
                const float o0 = 1.f / (1.f + __expf(-(a0 + pb.x + b30)));
                const float o1 = 1.f / (1.f + __expf(-(a1 + pb.y + b31)));
                if (A.y) *reinterpret_cast<float2 *>(A.y + 2 * (size_t)r) = make_float2(o0, o1);
                if (A.out) {
                    const bool learned = A.coin[r] < A.frac;
                    const float2 u = *reinterpret_cast<const float2 *>(A.uniform_xy + 2 * (size_t)r);
                    *reinterpret_cast<float2 *>(A.out + 2 * (size_t)r) =
                        learned ? make_float2(o0, o1) : u;
                }
            }
        }
    } else if (lane == 0) {
        // ---- the issuing thread (its warp's other lanes wait at the end)
        const uint32_t id256 = idesc_bf16(kRowsPerTile, kHidden);
        auto issue_layer1 = [&]() {
            mma(acc1, smem_desc(sb + oZ, 128, 256, 0), smem_desc(sb + oW1, 128, 256, 0), id256, 0u);
            commit(bar + bAcc1Full);
        };
        bool ok = true;
        if (first < ntiles) issue_layer1();
        uint32_t it = 0;
        for (int tile = first; ok && tile < ntiles; ++it, tile += step) {
            if (it > 0) ok = bar_wait(bar + bAcc2Free, (it - 1) & 1u, s_bad, kMmaWaitNs);
            for (int b = 0; ok && b < kKBlocks; ++b) {
                ok = bar_wait(bar + bHFull + b, it & 1u, s_bad, kMmaWaitNs);
                const bool ahead = b == kKBlocks - 1 && tile + step < ntiles;
                if (ok && ahead) ok = bar_wait(bar + bNextReady, it & 1u, s_bad, kMmaWaitNs);
                if (!ok) break;
                fence_after();
                if (ahead) issue_layer1();
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k)
                    mma(acc2, smem_desc(sb + oH + b * (kRowsPerTile * 128) + k * 32, 16, 1024, 2),
                        smem_desc(sb + oW2 + b * (kHidden * 128) + k * 32, 16, 1024, 2), id256,
                        b > 0 || k > 0 ? 1u : 0u);
                commit(bar + bHFree + b);
            }
            if (ok) commit(bar + bAcc2Full);
        }
        // every MMA issued, also before a wait expired, gets a bounded time to
        // end before the tensor memory is released
        int *late = reinterpret_cast<int *>(sm + oLate);
        commit(bar + bDrained);
        if (!bar_wait(bar + bDrained, 0u, late, kMmaWaitNs))
            *reinterpret_cast<volatile int *>(s_bad) = 1;
    }
    fence_before();
    __syncthreads();
    if (tid == 0 && *s_bad) atomicOr(A.status, kErrTimeout);
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(acc1),
                     "r"(kTmemCols)
                     : "memory");
    }
}

}  // namespace tc
}  // namespace mlp
}  // namespace pirrt
