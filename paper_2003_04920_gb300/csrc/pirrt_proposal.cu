// Host runtime and C ABI of the learned sampling proposal (see
// mlp_kernels.cuh for the network and its training rule).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "mlp_kernels.cuh"
#include "mlp_tc.cuh"
#include "mlp_train.cuh"
#include "pirrt.h"

using namespace pirrt::mlp;

namespace {

// Packed parameter layout (FP32): W1g [256 x 4096], W1n [256 x 8], b1 [256],
// W2 [256 x 256], b2 [256], W3 [2 x 256], b3 [2].
constexpr int64_t oW1g = 0, nW1g = (int64_t)kHidden * kGrid;
constexpr int64_t oW1n = oW1g + nW1g, nW1n = (int64_t)kHidden * kNoise;
constexpr int64_t ob1 = oW1n + nW1n, nb1 = kHidden;
constexpr int64_t oW2 = ob1 + nb1, nW2 = (int64_t)kHidden * kHidden;
constexpr int64_t ob2 = oW2 + nW2, nb2 = kHidden;
constexpr int64_t oW3 = ob2 + nb2, nW3 = (int64_t)kOut * kHidden;
constexpr int64_t ob3 = oW3 + nW3, nb3 = kOut;
constexpr int64_t kParams = ob3 + nb3;  // 1,117,186

int pad64(int x) { return (x + 63) / 64 * 64; }

}  // namespace

struct pirrt_proposal {
    int device = 0;
    cudaStream_t stream = nullptr;
    int max_scenes = 0, max_rows = 0, S = 0, R = 0;  // padded capacities
    float *w = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;
    __nv_bfloat16 *W1gb = nullptr, *W2b = nullptr, *W2Tb = nullptr, *W3b = nullptr;
    float *hg = nullptr;                                // [S x 256]
    float *a1 = nullptr, *a2 = nullptr;                 // [R x 256], the layered forward pass
    __nv_bfloat16 *h1 = nullptr, *h2 = nullptr, *da2 = nullptr;  // [R x 256]
    float *y = nullptr;                                 // [R x 2]
    __nv_bfloat16 *D = nullptr;                         // [S x 256] per-scene sums of da1
    BwPartials part{};                                  // the backward pass's partial sums
    float *w2part = nullptr;                            // [kBwSplit x 256 x 256]
    float *zsel = nullptr;                           // [R x 8]
    float *hgb = nullptr;                            // [S x 256]: W1g grid + b1
    int *status = nullptr;                           // error bits, 0 between calls
    struct Report {                                  // pinned: what a call reads back
        float loss;
        int status;
    } *report = nullptr;
    float *loss = nullptr;
    int64_t adam_t = 0;
    int num_sms = 0;
    int forward_kernel = PIRRT_MLP_FORWARD_TCGEN05;
    int keep_activations = 0;
    int last_rows = 0;       // rows of the last forward pass
    int last_has_acts = 0;   // whether that pass left h1 / h2 in HBM
    cudaEvent_t kev[2] = {nullptr, nullptr};  // around the last fused kernel
    int kev_recorded = 0;
};

namespace {

#define PCK(call)                                    \
    do {                                             \
        cudaError_t e_ = (call);                     \
        if (e_ != cudaSuccess) {                     \
            cudaGetLastError();                      \
            return e_ == cudaErrorMemoryAllocation ? PIRRT_ERR_OOM : PIRRT_ERR_CUDA; \
        }                                            \
    } while (0)

int blocks_for(int64_t n) {
    int64_t b = (n + 255) / 256;
    return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

pirrt_status gemm(pirrt_proposal *P, int M, int N, int K, const __nv_bfloat16 *A, int lda,
                  const __nv_bfloat16 *B, int ldb, float *C, int ldc, int beta) {
    dim3 grid(M / kGT, N / kGT);
    gemm_nt_bf16<<<grid, 128, 0, P->stream>>>(M, N, K, A, lda, B, ldb, C, ldc, beta);
    PCK(cudaGetLastError());
    return PIRRT_OK;
}

// Refresh the BF16 working copies from the FP32 master weights.
pirrt_status refresh_bf16(pirrt_proposal *P) {
    to_bf16<<<blocks_for(nW1g), 256, 0, P->stream>>>(kHidden, kGrid, P->w + oW1g, kGrid, P->W1gb,
                                                     kGrid, nullptr, 0);
    to_bf16<<<blocks_for(nW2), 256, 0, P->stream>>>(kHidden, kHidden, P->w + oW2, kHidden, P->W2b,
                                                    kHidden, P->W2Tb, kHidden);
    to_bf16<<<blocks_for(nW3), 256, 0, P->stream>>>(kOut, kHidden, P->w + oW3, kHidden, P->W3b,
                                                    kHidden, nullptr, 0);
    PCK(cudaGetLastError());
    return PIRRT_OK;
}

// Grid part of layer 1 for the scenes: hg = grid W1g^T and hgb = hg + b1.
pirrt_status scene_features(pirrt_proposal *P, int n_scenes, const float *grids) {
    if (n_scenes < 1 || n_scenes > P->max_scenes) return PIRRT_ERR_CAPACITY;
    scene_features_kernel<<<dim3(kHidden / kSceneN, (n_scenes + kSceneM - 1) / kSceneM), 128, kSceneSmem,
                            P->stream>>>(n_scenes, grids, P->W1gb, P->w + ob1, P->hg, P->hgb);
    PCK(cudaGetLastError());
    return PIRRT_OK;
}

// Rows through the network (after scene_features): y for `rows` samples.
pirrt_status forward_rows(pirrt_proposal *P, int rows, const int32_t *scene, int rows_per_scene,
                          const float *z) {
    if (rows < 1 || rows > P->max_rows) return PIRRT_ERR_CAPACITY;
    const int Rp = pad64(rows);
    layer1_rows<<<blocks_for((int64_t)Rp * kHidden), 256, 0, P->stream>>>(
        rows, Rp, P->hg, scene, rows_per_scene, z, P->w + oW1n, P->w + ob1, P->a1, P->h1);
    PCK(cudaGetLastError());
    pirrt_status rc = gemm(P, Rp, kHidden, kHidden, P->h1, kHidden, P->W2b, kHidden, P->a2, kHidden, 0);
    if (rc) return rc;
    bias_relu<<<blocks_for((int64_t)Rp * kHidden), 256, 0, P->stream>>>(rows, Rp, P->a2, P->w + ob2,
                                                                         P->h2);
    layer3_rows<<<blocks_for((int64_t)rows * 32), 256, 0, P->stream>>>(rows, P->h2, P->W3b,
                                                                        P->w + ob3, P->y);
    PCK(cudaGetLastError());
    return PIRRT_OK;
}

// The fused tcgen05 forward pass over `rows` rows (after scene_features):
// y and / or the mixture `out` (see tc::FwdArgs).  The error bits are read
// after the caller's stream synchronisation (read_status).
pirrt_status forward_fused(pirrt_proposal *P, int n_scenes, int rows, const int32_t *scene,
                           int rows_per_scene, const float *z, float *y, const float *uniform_xy,
                           const float *coin, float frac, float *out) {
    if (rows < 1 || rows > P->max_rows) return PIRRT_ERR_CAPACITY;
    if (reinterpret_cast<uintptr_t>(z) % 16 || reinterpret_cast<uintptr_t>(y) % 8 ||
        reinterpret_cast<uintptr_t>(out) % 8 || reinterpret_cast<uintptr_t>(uniform_xy) % 8)
        return PIRRT_ERR_INVALID_ARG;
    tc::FwdArgs a{};
    a.rows = rows;
    a.n_scenes = n_scenes;
    a.hgb = P->hgb;
    a.scene = scene;
    a.rows_per_scene = rows_per_scene;
    a.z = z;
    a.W1n = P->w + oW1n;
    a.W2b = P->W2b;
    a.b2 = P->w + ob2;
    a.W3b = P->W3b;
    a.b3 = P->w + ob3;
    a.y = y;
    a.uniform_xy = uniform_xy;
    a.coin = coin;
    a.frac = frac;
    a.out = out;
    a.cap_h1 = P->keep_activations ? P->h1 : nullptr;
    a.cap_h2 = P->keep_activations ? P->h2 : nullptr;
    a.status = P->status;
    const int tiles = (rows + tc::kRowsPerTile - 1) / tc::kRowsPerTile;
    const int grid = tiles < P->num_sms ? tiles : P->num_sms;
    PCK(cudaEventRecord(P->kev[0], P->stream));
    tc::mlp_forward_tc<<<grid, tc::kThreads, tc::kSmemBytes, P->stream>>>(a);
    PCK(cudaGetLastError());
    PCK(cudaEventRecord(P->kev[1], P->stream));
    P->kev_recorded = 1;
    P->last_rows = rows;
    P->last_has_acts = P->keep_activations;
    return PIRRT_OK;
}

// The end of a call: the error bits (and, with `loss`, the loss) come back with
// one small copy ordered on the stream, and the call waits for it.
pirrt_status finish_call(pirrt_proposal *P) {
    PCK(cudaMemcpyAsync(P->report, P->loss, sizeof(*P->report), cudaMemcpyDeviceToHost, P->stream));
    PCK(cudaStreamSynchronize(P->stream));
    const int st = P->report->status;
    if (st == 0) return PIRRT_OK;
    PCK(cudaMemsetAsync(P->status, 0, sizeof(int), P->stream));
    return st & tc::kErrTimeout ? PIRRT_ERR_DEVICE_TIMEOUT : PIRRT_ERR_BAD_INPUT;
}

// The forward pass of `rows` rows by the selected kernel into y (P->y if
// null); a mixture into `out` when given.
pirrt_status forward_any(pirrt_proposal *P, int n_scenes, int rows, const int32_t *scene,
                         int rows_per_scene, const float *z, float *y, const float *uniform_xy,
                         const float *coin, float frac, float *out) {
    if (P->forward_kernel == PIRRT_MLP_FORWARD_TCGEN05)
        return forward_fused(P, n_scenes, rows, scene, rows_per_scene, z, y ? y : P->y, uniform_xy,
                             coin, frac, out);
    pirrt_status rc = forward_rows(P, rows, scene, rows_per_scene, z);
    if (rc) return rc;
    P->last_rows = rows;
    P->last_has_acts = 1;
    if (y && y != P->y)
        PCK(cudaMemcpyAsync(y, P->y, sizeof(float) * kOut * (size_t)rows, cudaMemcpyDeviceToDevice,
                            P->stream));
    if (out) {
        mix_samples<<<blocks_for(rows), 256, 0, P->stream>>>(rows, P->y, uniform_xy, coin, frac, out);
        PCK(cudaGetLastError());
    }
    return PIRRT_OK;
}

void free_all(pirrt_proposal *P) {
    void *bufs[] = {P->w, P->m, P->v, P->grad, P->W1gb, P->W2b, P->W2Tb, P->W3b, P->hg, P->a1, P->a2,
                    P->h1, P->h2, P->da2, P->y, P->D, P->loss, P->zsel, P->hgb, P->w2part,
                    P->part.w3, P->part.b2, P->part.w1n, P->part.b1, P->part.tail, P->part.run,
                    P->part.run_scene};
    for (void *b : bufs)
        if (b) cudaFree(b);
    if (P->report) cudaFreeHost(P->report);
    for (cudaEvent_t &e : P->kev)
        if (e) cudaEventDestroy(e);
}

// splitmix64: a counter-based generator for the initial weights
uint64_t splitmix(uint64_t &s) {
    uint64_t z = (s += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

}  // namespace

extern "C" {

int64_t pirrt_proposal_num_params(void) { return kParams; }

pirrt_status pirrt_proposal_create(int32_t max_scenes, int32_t max_rows, uint64_t seed,
                                   int32_t device, void *stream, pirrt_proposal **out) {
    if (!out) return PIRRT_ERR_INVALID_ARG;
    *out = nullptr;
    if (max_scenes < 1 || max_rows < 1) return PIRRT_ERR_INVALID_ARG;
    if (cudaSetDevice(device) != cudaSuccess) return PIRRT_ERR_CUDA;
    pirrt_proposal *P = new (std::nothrow) pirrt_proposal();
    if (!P) return PIRRT_ERR_OOM;
    P->device = device;
    P->stream = static_cast<cudaStream_t>(stream);
    P->max_scenes = max_scenes;
    P->max_rows = max_rows;
    const size_t S = (size_t)pad64(max_scenes), R = (size_t)pad64(max_rows);
    P->S = (int)S;
    P->R = (int)R;
    auto bail = [&](pirrt_status s) {
        free_all(P);
        delete P;
        return s;
    };
#define PA(ptr, bytes)                                                      \
    do {                                                                    \
        if (cudaMalloc((void **)&(ptr), (bytes)) != cudaSuccess) {          \
            cudaGetLastError();                                             \
            return bail(PIRRT_ERR_OOM);                                     \
        }                                                                   \
        if (cudaMemset((ptr), 0, (bytes)) != cudaSuccess) return bail(PIRRT_ERR_CUDA); \
    } while (0)
    const size_t bf = sizeof(__nv_bfloat16), f = sizeof(float);
    PA(P->w, f * kParams);
    PA(P->m, f * kParams);
    PA(P->v, f * kParams);
    PA(P->grad, f * kParams);
    PA(P->W1gb, bf * nW1g);
    PA(P->W2b, bf * nW2);
    PA(P->W2Tb, bf * nW2);
    PA(P->W3b, bf * nW3);
    PA(P->hg, f * S * kHidden);
    PA(P->a1, f * R * kHidden);
    PA(P->a2, f * R * kHidden);
    PA(P->h1, bf * R * kHidden);
    PA(P->h2, bf * R * kHidden);
    PA(P->da2, bf * R * kHidden);
    PA(P->y, f * R * kOut);
    PA(P->D, bf * S * kHidden);
    PA(P->zsel, f * R * kNoise);
    PA(P->hgb, f * S * kHidden);
    PA(P->loss, sizeof(pirrt_proposal::Report));  // the loss, then the error bits
    P->status = reinterpret_cast<int *>(P->loss + 1);
    if (cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
        return bail(PIRRT_ERR_CUDA);
    const size_t C = (size_t)P->num_sms;  // CTAs of the backward pass, at most
    PA(P->part.w3, f * C * kOut * kHidden);
    PA(P->part.b2, f * C * kHidden);
    PA(P->part.w1n, f * C * kHidden * kNoise);
    PA(P->part.b1, f * C * kHidden);
    PA(P->part.tail, f * C * 4);
    PA(P->part.run, f * R * kHidden);
    PA(P->part.run_scene, sizeof(int) * R);
    PA(P->w2part, f * kBwSplit * kHidden * kHidden);
#undef PA
    if (cudaEventCreate(&P->kev[0]) != cudaSuccess || cudaEventCreate(&P->kev[1]) != cudaSuccess ||
        cudaMallocHost((void **)&P->report, sizeof(*P->report)) != cudaSuccess ||
        cudaFuncSetAttribute(backward_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(BwShared)) != cudaSuccess ||
        cudaFuncSetAttribute(tc::mlp_forward_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             tc::kSmemBytes) != cudaSuccess ||
        cudaFuncSetAttribute(scene_features_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kSceneSmem) != cudaSuccess) {
        cudaGetLastError();
        return bail(PIRRT_ERR_CUDA);
    }
    // He-uniform initial weights (fan-in of each layer), zero biases
    std::vector<float> h(kParams, 0.f);
    uint64_t st = seed;
    auto uni = [&](float lim) {
        const double u = (double)(splitmix(st) >> 11) * (1.0 / 9007199254740992.0);
        return (float)((2.0 * u - 1.0) * lim);
    };
    const float l1 = std::sqrt(6.f / (kGrid + kNoise)), l2 = std::sqrt(6.f / kHidden);
    for (int64_t i = 0; i < nW1g; ++i) h[oW1g + i] = uni(l1);
    for (int64_t i = 0; i < nW1n; ++i) h[oW1n + i] = uni(l1);
    for (int64_t i = 0; i < nW2; ++i) h[oW2 + i] = uni(l2);
    for (int64_t i = 0; i < nW3; ++i) h[oW3 + i] = uni(l2);
    if (cudaMemcpy(P->w, h.data(), f * kParams, cudaMemcpyHostToDevice) != cudaSuccess)
        return bail(PIRRT_ERR_CUDA);
    if (refresh_bf16(P) != PIRRT_OK || cudaStreamSynchronize(P->stream) != cudaSuccess)
        return bail(PIRRT_ERR_CUDA);
    *out = P;
    return PIRRT_OK;
}

void pirrt_proposal_destroy(pirrt_proposal *P) {
    if (!P) return;
    cudaSetDevice(P->device);
    cudaStreamSynchronize(P->stream);
    free_all(P);
    delete P;
}

pirrt_status pirrt_proposal_set_weights(pirrt_proposal *P, const float *w, int64_t n) {
    if (!P || !w || n != kParams) return PIRRT_ERR_INVALID_ARG;
    PCK(cudaMemcpyAsync(P->w, w, sizeof(float) * kParams, cudaMemcpyDeviceToDevice, P->stream));
    PCK(cudaMemsetAsync(P->m, 0, sizeof(float) * kParams, P->stream));
    PCK(cudaMemsetAsync(P->v, 0, sizeof(float) * kParams, P->stream));
    PCK(cudaMemsetAsync(P->grad, 0, sizeof(float) * kParams, P->stream));
    P->adam_t = 0;
    pirrt_status rc = refresh_bf16(P);
    if (rc) return rc;
    PCK(cudaStreamSynchronize(P->stream));
    return PIRRT_OK;
}

pirrt_status pirrt_proposal_get_weights(const pirrt_proposal *P, float *w, int64_t n) {
    if (!P || !w || n != kParams) return PIRRT_ERR_INVALID_ARG;
    PCK(cudaMemcpyAsync(w, P->w, sizeof(float) * kParams, cudaMemcpyDeviceToDevice, P->stream));
    PCK(cudaStreamSynchronize(P->stream));
    return PIRRT_OK;
}

pirrt_status pirrt_proposal_get_grads(const pirrt_proposal *P, float *g, int64_t n) {
    if (!P || !g || n != kParams) return PIRRT_ERR_INVALID_ARG;
    PCK(cudaMemcpyAsync(g, P->grad, sizeof(float) * kParams, cudaMemcpyDeviceToDevice, P->stream));
    PCK(cudaStreamSynchronize(P->stream));
    return PIRRT_OK;
}

pirrt_status pirrt_proposal_forward(pirrt_proposal *P, int32_t n_scenes, const float *grids,
                                    int32_t rows, const int32_t *scene, const float *noise,
                                    float *out_xy) {
    if (!P || !grids || !scene || !noise || !out_xy) return PIRRT_ERR_INVALID_ARG;
    PCK(cudaSetDevice(P->device));
    pirrt_status rc = scene_features(P, n_scenes, grids);
    if (rc) return rc;
    if ((rc = forward_any(P, n_scenes, rows, scene, 1, noise, out_xy, nullptr, nullptr, 0.f,
                          nullptr)))
        return rc;
    return finish_call(P);
}

pirrt_status pirrt_proposal_sample(pirrt_proposal *P, int32_t n_scenes, const float *grids,
                                   int32_t rows, const int32_t *scene, const float *noise,
                                   const float *uniform_xy, const float *coin,
                                   float learned_fraction, float *out_xy) {
    if (!P || !grids || !scene || !noise || !uniform_xy || !coin || !out_xy ||
        !(learned_fraction >= 0.f && learned_fraction <= 1.f))
        return PIRRT_ERR_INVALID_ARG;
    PCK(cudaSetDevice(P->device));
    pirrt_status rc = scene_features(P, n_scenes, grids);
    if (rc) return rc;
    if ((rc = forward_any(P, n_scenes, rows, scene, 1, noise, nullptr, uniform_xy, coin,
                          learned_fraction, out_xy)))
        return rc;
    return finish_call(P);
}

pirrt_status pirrt_proposal_imle_select(pirrt_proposal *P, int32_t n_scenes, const float *grids,
                                        int32_t n_targets, const int32_t *draw_scene,
                                        const float *targets, int32_t K, const float *noise,
                                        int32_t *pick) {
    if (!P || !grids || !draw_scene || !targets || !noise || !pick || K < 1 || n_targets < 1)
        return PIRRT_ERR_INVALID_ARG;
    PCK(cudaSetDevice(P->device));
    if ((int64_t)n_targets * K > P->max_rows) return PIRRT_ERR_CAPACITY;
    pirrt_status rc = scene_features(P, n_scenes, grids);
    if (rc) return rc;
    if ((rc = forward_any(P, n_scenes, n_targets * K, draw_scene, 1, noise, nullptr, nullptr, nullptr,
                          0.f, nullptr)))
        return rc;
    imle_select<<<blocks_for(n_targets), 256, 0, P->stream>>>(n_targets, K, P->y, targets, pick);
    PCK(cudaGetLastError());
    return finish_call(P);
}

extern "C++" {
// The backward pass of `rows` rows (after scene_features); the loss stays on the
// device (finish_call reads it).
static pirrt_status backward_rows(pirrt_proposal *P, int n_scenes, const float *grids, int rows,
                                  const int32_t *scene, const float *noise, const float *targets) {
    if (rows < 1 || rows > P->max_rows) return PIRRT_ERR_CAPACITY;
    P->last_rows = rows;
    P->last_has_acts = 1;
    BwArgs a{};
    a.rows = rows;
    a.tiles = pad64(rows) / kBwRows;
    // a CTA's share of the tiles: one each while they last, so that every SM works
    const int most = a.tiles < P->num_sms ? a.tiles : P->num_sms;
    a.tiles_per_cta = (a.tiles + most - 1) / most;
    const int ctas = (a.tiles + a.tiles_per_cta - 1) / a.tiles_per_cta;
    a.n_scenes = n_scenes;
    a.hg = P->hg;
    a.b1 = P->w + ob1;
    a.b2 = P->w + ob2;
    a.b3 = P->w + ob3;
    a.W1n = P->w + oW1n;
    a.W2b = P->W2b;
    a.W2Tb = P->W2Tb;
    a.W3b = P->W3b;
    a.scene = scene;
    a.z = noise;
    a.target = targets;
    a.h1 = P->h1;
    a.h2 = P->h2;
    a.da2 = P->da2;
    a.y = P->y;
    a.part = P->part;
    a.status = P->status;
    backward_rows_kernel<<<ctas, kBwThreads, sizeof(BwShared), P->stream>>>(a);
    PCK(cudaGetLastError());
    // dW2 in parts of at least 128 rows, so that 16 tiles of 64 x 64 become up to
    // 256 CTAs
    const int rows_pad = a.tiles * kBwRows;
    int splits = (rows_pad + 127) / 128;
    if (splits > kBwSplit) splits = kBwSplit;
    const int per = ((rows_pad + splits - 1) / splits + 31) / 32 * 32;
    splits = (rows_pad + per - 1) / per;
    dw2_parts_kernel<<<dim3(4, 4, splits), 128, 0, P->stream>>>(rows_pad, per, P->da2, P->h1,
                                                               P->w2part);
    finish_backward_kernel<<<kFinishRow + kFinishSmall + n_scenes, 256, 0, P->stream>>>(
        ctas, splits, rows_pad, rows, P->part, P->w2part, P->grad + oW2, P->grad + oW3,
        P->grad + ob2, P->grad + ob3, P->grad + oW1n, P->grad + ob1, P->loss, P->D);
    dw1g_kernel<<<dim3(kHidden / 64, kGrid / 64), 128, 0, P->stream>>>(n_scenes, P->D, grids,
                                                                      P->grad + oW1g);
    PCK(cudaGetLastError());
    return PIRRT_OK;
}

// One Adam step for the t-th time; with `status` it is skipped if an earlier
// kernel of the call reported an error.
static pirrt_status adam_all(pirrt_proposal *P, int64_t t, float lr, float beta1, float beta2,
                             float eps, const int *status) {
    AdamArgs a{};
    a.w = P->w;
    a.m = P->m;
    a.v = P->v;
    a.grad = P->grad;
    a.W1gb = P->W1gb;
    a.W2b = P->W2b;
    a.W2Tb = P->W2Tb;
    a.W3b = P->W3b;
    a.n = kParams;
    a.oW2 = oW2;
    a.ob2 = ob2;
    a.oW3 = oW3;
    a.ob3 = ob3;
    a.nW1g = nW1g;
    a.lr = lr;
    a.beta1 = beta1;
    a.beta2 = beta2;
    a.eps = eps;
    a.bc1 = 1.f - std::pow(beta1, (float)t);
    a.bc2 = 1.f - std::pow(beta2, (float)t);
    a.status = status;
    adam_all_kernel<<<(unsigned)((kParams + 255) / 256), 256, 0, P->stream>>>(a);
    PCK(cudaGetLastError());
    return PIRRT_OK;
}
}  // extern "C++"

pirrt_status pirrt_proposal_backward(pirrt_proposal *P, int32_t n_scenes, const float *grids,
                                     int32_t rows, const int32_t *scene, const float *noise,
                                     const float *targets, float *loss_out) {
    if (!P || !grids || !scene || !noise || !targets) return PIRRT_ERR_INVALID_ARG;
    PCK(cudaSetDevice(P->device));
    pirrt_status rc = scene_features(P, n_scenes, grids);
    if (rc) return rc;
    if ((rc = backward_rows(P, n_scenes, grids, rows, scene, noise, targets))) return rc;
    rc = finish_call(P);
    if (loss_out) *loss_out = P->report->loss;
    return rc;
}

pirrt_status pirrt_proposal_adam(pirrt_proposal *P, float lr, float beta1, float beta2, float eps) {
    if (!P || !(lr > 0.f)) return PIRRT_ERR_INVALID_ARG;
    PCK(cudaSetDevice(P->device));
    P->adam_t += 1;
    const pirrt_status rc = adam_all(P, P->adam_t, lr, beta1, beta2, eps, nullptr);
    if (rc) return rc;
    PCK(cudaStreamSynchronize(P->stream));
    return PIRRT_OK;
}

pirrt_status pirrt_proposal_train_step(pirrt_proposal *P, int32_t n_scenes, const float *grids,
                                       int32_t n_targets, const int32_t *target_scene,
                                       const float *targets, int32_t K, const float *noise,
                                       float lr, float *loss_out) {
    if (!P || !grids || !target_scene || !targets || !noise || K < 1 || n_targets < 1)
        return PIRRT_ERR_INVALID_ARG;
    if ((int64_t)n_targets * K > P->max_rows) return PIRRT_ERR_CAPACITY;
    PCK(cudaSetDevice(P->device));
    pirrt_status rc = scene_features(P, n_scenes, grids);
    if (rc) return rc;
    // the draws (row t*K + k in target t's scene), the nearest of each target, its
    // backward pass and Adam, with one wait at the end
    if ((rc = forward_any(P, n_scenes, n_targets * K, target_scene, K, noise, nullptr, nullptr,
                          nullptr, 0.f, nullptr)))
        return rc;
    select_noise_kernel<<<(n_targets * 8 + 255) / 256, 256, 0, P->stream>>>(n_targets, K, P->y, targets,
                                                                          noise, P->zsel);
    PCK(cudaGetLastError());
    if ((rc = backward_rows(P, n_scenes, grids, n_targets, target_scene, P->zsel, targets)))
        return rc;
    const bool step = lr > 0.f;
    if (step && (rc = adam_all(P, P->adam_t + 1, lr, 0.9f, 0.999f, 1e-8f, P->status))) return rc;
    rc = finish_call(P);
    if (loss_out) *loss_out = P->report->loss;
    if (rc) return rc;
    if (!step) return PIRRT_ERR_INVALID_ARG;
    P->adam_t += 1;
    return PIRRT_OK;
}

pirrt_status pirrt_proposal_set_options(pirrt_proposal *P, int32_t forward_kernel,
                                        int32_t keep_activations) {
    if (!P || (forward_kernel != PIRRT_MLP_FORWARD_TCGEN05 &&
               forward_kernel != PIRRT_MLP_FORWARD_LAYERED))
        return PIRRT_ERR_INVALID_ARG;
    P->forward_kernel = forward_kernel;
    P->keep_activations = keep_activations ? 1 : 0;
    return PIRRT_OK;
}

pirrt_status pirrt_proposal_kernel_ms(const pirrt_proposal *P, float *ms) {
    if (!P || !ms || !P->kev_recorded) return PIRRT_ERR_INVALID_ARG;
    PCK(cudaEventSynchronize(P->kev[1]));
    PCK(cudaEventElapsedTime(ms, P->kev[0], P->kev[1]));
    return PIRRT_OK;
}

pirrt_status pirrt_proposal_get_activations(const pirrt_proposal *P, int32_t rows,
                                            uint16_t *h1_out, uint16_t *h2_out) {
    if (!P || rows < 1 || rows > P->last_rows || !P->last_has_acts) return PIRRT_ERR_INVALID_ARG;
    const size_t bytes = sizeof(__nv_bfloat16) * kHidden * (size_t)rows;
    if (h1_out) PCK(cudaMemcpyAsync(h1_out, P->h1, bytes, cudaMemcpyDeviceToDevice, P->stream));
    if (h2_out) PCK(cudaMemcpyAsync(h2_out, P->h2, bytes, cudaMemcpyDeviceToDevice, P->stream));
    PCK(cudaStreamSynchronize(P->stream));
    return PIRRT_OK;
}

pirrt_status pirrt_proposal_zero_grads(pirrt_proposal *P) {
    if (!P) return PIRRT_ERR_INVALID_ARG;
    PCK(cudaMemsetAsync(P->grad, 0, sizeof(float) * kParams, P->stream));
    PCK(cudaStreamSynchronize(P->stream));
    return PIRRT_OK;
}

}  // extern "C"
