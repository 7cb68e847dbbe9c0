// mlp.cu -- learned calibration surrogate of the pseudopotential model.
//
// The paper notes that the pseudopotential model needs preliminary simulations to fix
// its parameters (Secs. 3, 5.1, 5.2: sigma^Li, kappa^P, kappa^Li and the densities,
// width and surface tension they give).  This surrogate maps (Tr, a, b, kappa^P) to the
// calibration observables (rho_l, rho_v, W, sigma) of such runs: an MLP 4 -> 128 -> 128 ->
// 128 -> 4 with GELU, 34,180 weights, trained in FP32 on the GPU by the kernels below
// (one fused forward/backward kernel and one gradient-sum/Adam kernel, mlp_train.cuh), and
// evaluated by fused kernels with BF16 inputs and weights and FP32 accumulation on the
// tensor cores (mlp_infer.cuh).  Inputs and outputs are standardised with the training
// set's statistics; rho_v is learned as ln(rho_v).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <random>
#include <vector>

#include "../../include/lbm.h"

namespace {

thread_local char g_mlp_msg[256] = "";
int mfail(cudaError_t e, const char* what) {
    snprintf(g_mlp_msg, sizeof(g_mlp_msg), "%s: %s", what, cudaGetErrorString(e));
    return LBM_ERR_CUDA;
}
#define MCK(call)                                             \
    do {                                                      \
        cudaError_t e_ = (call);                              \
        if (e_ != cudaSuccess) return mfail(e_, #call);       \
    } while (0)

constexpr int kIn = 4, kHid = 128, kOut = 4, kLayers = 4;
__device__ constexpr int kDims[kLayers + 1] = {kIn, kHid, kHid, kHid, kOut};
// parameter offsets: W_l (out x in, row-major) then b_l
__host__ __device__ constexpr int woff(int l) {
    int o = 0;
    for (int i = 0; i < l; ++i) o += kDims[i + 1] * kDims[i] + kDims[i + 1];
    return o;
}
__host__ __device__ constexpr int boff(int l) { return woff(l) + kDims[l + 1] * kDims[l]; }
constexpr int kNumParams = woff(kLayers);
static_assert(kNumParams == 34180, "4-128-128-128-4 MLP has 34,180 parameters");

}  // namespace

#include "mlp_infer.cuh"
#include "mlp_train.cuh"

namespace {

// (raw inputs, raw targets) -> standardised network inputs / targets (rho_v as ln rho_v)
__global__ void standardise_kernel(const float* __restrict__ X, const float* __restrict__ Yraw, int n,
                                   const float* __restrict__ stats, float* __restrict__ Xn, float* __restrict__ Yn) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        for (int j = 0; j < kIn; ++j) Xn[i * kIn + j] = (X[i * kIn + j] - stats[j]) / stats[4 + j];
        if (Yraw)
            for (int j = 0; j < kOut; ++j) {
                const float y = j == 1 ? logf(Yraw[i * kOut + j]) : Yraw[i * kOut + j];
                Yn[i * kOut + j] = (y - stats[8 + j]) / stats[12 + j];
            }
    }
}

// FP32 reference evaluation (the training forward pass) de-standardised, for comparison.
__global__ void destandardise_kernel(const float* __restrict__ Zn, int n, const float* __restrict__ stats,
                                     float* __restrict__ Y) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n * kOut; i += gridDim.x * blockDim.x) {
        const int c = i % kOut;
        float y = Zn[i] * stats[12 + c] + stats[8 + c];
        Y[i] = c == 1 ? expf(y) : y;
    }
}

}  // namespace

// ---------------------------------------------------------------------------------------
// Host side

namespace {
constexpr int kSMs = 152;                                   // one CTA's worth of samples each
constexpr int kUpdateBlocks = (kNumParams + 1 + 31) / 32;  // parameters and the loss
}  // namespace

struct lbm_surrogate {
    int cap;                  // allocated rows
    float* d_params;          // kNumParams
    float* d_grad;
    float* d_m1;
    float* d_m2;
    float* d_stats;           // in mean[4], in std[4], out mean[4], out std[4]
    float* d_X;               // raw inputs (cap x 4)
    float* d_Yraw;            // raw targets
    float* d_Xn;              // standardised
    float* d_Yn;
    float* d_Z4;              // network outputs (cap x 4)
    float* d_WT;              // the hidden weight matrices transposed
    float* d_part;            // gradient slots (part_slots x kSlot)
    int part_slots;
    float* d_loss;
    float* d_out;
    float h_stats[16];
    int steps_done;
    cudaStream_t stream;
    float last_loss;
};

namespace {

int alloc_rows(lbm_surrogate* m, int n) {
    if (n <= m->cap) return LBM_OK;
    auto drop = [](float** b) {
        if (*b) cudaFree(*b);
        *b = nullptr;
    };
    float** bufs[] = {&m->d_X, &m->d_Yraw, &m->d_Xn, &m->d_Yn, &m->d_Z4, &m->d_out};
    for (float** b : bufs) drop(b);
    m->cap = 0;
    static_assert(kIn == kOut, "one size for every row buffer");
    for (float** b : bufs) MCK(cudaMalloc(b, (size_t)n * kIn * 4));
    m->cap = n;
    return LBM_OK;
}

// Samples per CTA: the batch over all SMs, in whole float4 of samples, at most one tile; below 8 the
// gradient slots would cost more than they spread.
int train_rows(int n) { return std::min(kTrainRows, std::max(8, ((n + kSMs - 1) / kSMs + 3) / 4 * 4)); }
int train_slots(int n) { return std::min(kSMs, (n + train_rows(n) - 1) / train_rows(n)); }

// Prepare a pass over n samples at the current parameters.
int train_setup(lbm_surrogate* m, int n, bool backward) {
    const int slots = train_slots(n);
    if (backward && slots > m->part_slots) {
        if (m->d_part) cudaFree(m->d_part);
        m->d_part = nullptr;
        m->part_slots = 0;
        MCK(cudaMalloc(&m->d_part, sizeof(float) * kSlot * (size_t)slots));
        m->part_slots = slots;
    }
    MCK(cudaFuncSetAttribute(mlp_train_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)));
    MCK(cudaFuncSetAttribute(mlp_train_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)));
    mlp_transpose_kernel<<<64, 256, 0, m->stream>>>(m->d_params, m->d_WT);
    MCK(cudaGetLastError());
    return LBM_OK;
}

// forward pass on d_Xn rows [0, n): fills d_Z4
int forward(lbm_surrogate* m, int n) {
    mlp_train_kernel<false><<<train_slots(n), kTrainThreads, sizeof(TrainSmem), m->stream>>>(
        m->d_Xn, nullptr, n, train_rows(n), m->d_params, m->d_WT, 0.0f, nullptr, m->d_Z4);
    MCK(cudaGetLastError());
    return LBM_OK;
}

// forward and backward pass of the MSE loss against d_Yn (n_valid finite targets) into the slots
int forward_backward(lbm_surrogate* m, int n, float inv_valid) {
    mlp_train_kernel<true><<<train_slots(n), kTrainThreads, sizeof(TrainSmem), m->stream>>>(
        m->d_Xn, m->d_Yn, n, train_rows(n), m->d_params, m->d_WT, inv_valid, m->d_part, nullptr);
    MCK(cudaGetLastError());
    return LBM_OK;
}

// finite target entries (each set needs a finite rho_v > 0; other outputs may be NaN = missing)
long long valid_targets(const float* Y, int n) {
    long long c = 0;
    for (long long i = 0; i < (long long)n * kOut; ++i) {
        if (i % kOut == 1 && !(Y[i] > 0.0f && std::isfinite(Y[i]))) return -1;
        c += std::isfinite(Y[i]) ? 1 : 0;
    }
    return c;
}

int upload_inputs(lbm_surrogate* m, const float* X, const float* Y, int n) {
    int rc = alloc_rows(m, n);
    if (rc) return rc;
    MCK(cudaMemcpyAsync(m->d_X, X, sizeof(float) * n * kIn, cudaMemcpyHostToDevice, m->stream));
    if (Y) MCK(cudaMemcpyAsync(m->d_Yraw, Y, sizeof(float) * n * kOut, cudaMemcpyHostToDevice, m->stream));
    standardise_kernel<<<64, 256, 0, m->stream>>>(m->d_X, Y ? m->d_Yraw : nullptr, n, m->d_stats, m->d_Xn, m->d_Yn);
    MCK(cudaGetLastError());
    return LBM_OK;
}

}  // namespace

extern "C" const char* lbm_surrogate_last_error(void) { return g_mlp_msg; }

extern "C" int lbm_surrogate_num_params(void) { return kNumParams; }

extern "C" void lbm_surrogate_destroy(lbm_surrogate* m) {
    if (!m) return;
    cudaStreamSynchronize(m->stream);
    float* bufs[] = {m->d_params, m->d_grad, m->d_m1, m->d_m2, m->d_stats, m->d_X, m->d_Yraw, m->d_Xn,
                     m->d_Yn, m->d_Z4, m->d_WT, m->d_part, m->d_loss, m->d_out};
    for (float* b : bufs)
        if (b) cudaFree(b);
    if (m->stream) cudaStreamDestroy(m->stream);
    delete m;
}

extern "C" int lbm_surrogate_create(const float* stats16, unsigned seed, lbm_surrogate** out) {
    if (!out || !stats16) return LBM_ERR_ARG;
    *out = nullptr;
    for (int j = 0; j < 4; ++j)
        if (!(stats16[4 + j] > 0) || !(stats16[12 + j] > 0)) return LBM_ERR_ARG;
    lbm_surrogate* m = new (std::nothrow) lbm_surrogate();
    if (!m) return LBM_ERR_ARG;
    auto fail = [&](int rc) {
        lbm_surrogate_destroy(m);
        return rc;
    };
    cudaError_t e;
    if ((e = cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking)) != cudaSuccess) return fail(mfail(e, "stream"));
    float** bufs[] = {&m->d_params, &m->d_grad, &m->d_m1, &m->d_m2};
    for (float** b : bufs)
        if ((e = cudaMalloc(b, sizeof(float) * kNumParams)) != cudaSuccess) return fail(mfail(e, "cudaMalloc(params)"));
    if ((e = cudaMalloc(&m->d_stats, sizeof(float) * 16)) != cudaSuccess ||
        (e = cudaMalloc(&m->d_loss, sizeof(float))) != cudaSuccess ||
        (e = cudaMalloc(&m->d_WT, sizeof(float) * 2 * kHid * kHid)) != cudaSuccess)
        return fail(mfail(e, "cudaMalloc"));
    std::memcpy(m->h_stats, stats16, sizeof(m->h_stats));
    // He-style initialisation (uniform, seeded); zero biases
    std::vector<float> p(kNumParams, 0.0f);
    std::mt19937 rng(seed);
    for (int l = 0; l < kLayers; ++l) {
        const float lim = std::sqrt(6.0f / kDims[l]);
        std::uniform_real_distribution<float> U(-lim, lim);
        for (int i = 0; i < kDims[l + 1] * kDims[l]; ++i) p[woff(l) + i] = U(rng) * (l == kLayers - 1 ? 0.1f : 1.0f);
    }
    if ((e = cudaMemcpy(m->d_params, p.data(), sizeof(float) * kNumParams, cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(m->d_stats, stats16, sizeof(float) * 16, cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemset(m->d_m1, 0, sizeof(float) * kNumParams)) != cudaSuccess ||
        (e = cudaMemset(m->d_m2, 0, sizeof(float) * kNumParams)) != cudaSuccess)
        return fail(mfail(e, "init"));
    *out = m;
    return LBM_OK;
}

extern "C" int lbm_surrogate_set_params(lbm_surrogate* m, const float* params) {
    if (!m || !params) return LBM_ERR_ARG;
    MCK(cudaMemcpy(m->d_params, params, sizeof(float) * kNumParams, cudaMemcpyHostToDevice));
    return LBM_OK;
}

extern "C" int lbm_surrogate_get_params(lbm_surrogate* m, float* params) {
    if (!m || !params) return LBM_ERR_ARG;
    MCK(cudaStreamSynchronize(m->stream));
    MCK(cudaMemcpy(params, m->d_params, sizeof(float) * kNumParams, cudaMemcpyDeviceToHost));
    return LBM_OK;
}

extern "C" int lbm_surrogate_loss_grad(lbm_surrogate* m, const float* X, const float* Y, int n, float* loss,
                                       float* grad) {
    if (!m || !X || !Y || n < 1) return LBM_ERR_ARG;
    const long long nv = valid_targets(Y, n);
    if (nv < 1) return LBM_ERR_ARG;
    int rc = upload_inputs(m, X, Y, n);
    const float inv_valid = (float)(1.0 / (double)nv);
    if (!rc) rc = train_setup(m, n, true);
    if (!rc) rc = forward_backward(m, n, inv_valid);
    if (rc) return rc;
    mlp_update_kernel<false><<<kUpdateBlocks, 32 * kUpdateWarps, 0, m->stream>>>(m->d_part, train_slots(n), inv_valid, m->d_grad,
                                                                  m->d_loss, nullptr, nullptr, nullptr, nullptr, 0, 0, 0,
                                                                  0, 0, 0, 0);
    MCK(cudaGetLastError());
    if (loss) MCK(cudaMemcpyAsync(loss, m->d_loss, sizeof(float), cudaMemcpyDeviceToHost, m->stream));
    if (grad) MCK(cudaMemcpyAsync(grad, m->d_grad, sizeof(float) * kNumParams, cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    return LBM_OK;
}

extern "C" int lbm_surrogate_train(lbm_surrogate* m, const float* X, const float* Y, int n,
                                   const lbm_train_cfg* cfg, float* final_loss) {
    if (!m || !X || !Y || n < 1 || !cfg || cfg->iterations < 0 || !(cfg->lr > 0)) return LBM_ERR_ARG;
    const long long nv = valid_targets(Y, n);
    if (nv < 1) return LBM_ERR_ARG;
    int rc = upload_inputs(m, X, Y, n);
    if (rc) return rc;
    rc = train_setup(m, n, true);
    if (rc) return rc;
    const float inv_valid = (float)(1.0 / (double)nv);
    // one iteration: full-batch forward and backward pass, then the gradient's sum and Adam's update
    for (int it = 0; it < cfg->iterations; ++it) {
        if ((rc = forward_backward(m, n, inv_valid))) return rc;
        const int t = ++m->steps_done;
        // cosine learning-rate decay to lr_min over the run
        const float frac = cfg->iterations > 1 ? (float)it / (float)(cfg->iterations - 1) : 0.0f;
        const float lr = cfg->lr_min + 0.5f * (cfg->lr - cfg->lr_min) * (1.0f + std::cos(3.14159265f * frac));
        const float c1 = 1.0f - std::pow(cfg->beta1, (float)t), c2 = 1.0f - std::pow(cfg->beta2, (float)t);
        mlp_update_kernel<true><<<kUpdateBlocks, 32 * kUpdateWarps, 0, m->stream>>>(
            m->d_part, train_slots(n), inv_valid, m->d_grad, m->d_loss, m->d_params, m->d_WT, m->d_m1, m->d_m2, lr,
            cfg->beta1, cfg->beta2, cfg->eps, c1, c2, cfg->weight_decay);
    }
    MCK(cudaGetLastError());
    MCK(cudaMemcpyAsync(&m->last_loss, m->d_loss, sizeof(float), cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    if (final_loss) *final_loss = m->last_loss;
    return std::isfinite(m->last_loss) ? LBM_OK : LBM_ERR_DIVERGED;
}

extern "C" int lbm_surrogate_predict_fp32(lbm_surrogate* m, const float* X, int n, float* Y) {
    if (!m || !X || !Y || n < 1) return LBM_ERR_ARG;
    int rc = upload_inputs(m, X, nullptr, n);
    if (!rc) rc = train_setup(m, n, false);
    if (!rc) rc = forward(m, n);
    if (rc) return rc;
    destandardise_kernel<<<64, 256, 0, m->stream>>>(m->d_Z4, n, m->d_stats, m->d_out);
    MCK(cudaGetLastError());
    MCK(cudaMemcpyAsync(Y, m->d_out, sizeof(float) * n * kOut, cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    return LBM_OK;
}

// Up to kSmallQueries, three rounds of 32 queries on every SM, the layers are split over a CTA's warps, one
// tile of 16 queries per CTA while there are SMs for that, else two; above it a warp takes its tiles through
// the network alone (split mode, us per call, split over warps and not: 1 query 8.1, 14.6; 4864 10.5, 14.7;
// 9728 14.5, 15.3; 14592 17.6, 18.8; 19456 20.8, 19.6; 65536 56, 46).
constexpr int kSmallQueries = 3 * kSMs * 2 * kInferRows;
template <bool kSplit>
static cudaError_t infer(const lbm_surrogate* m, const float* X, int n, float* Y, cudaStream_t s) {
    const int tiles = n / kInferRows + (n % kInferRows != 0);
    if (n <= kSmallQueries) {
        if (tiles <= kSMs)
            mlp_infer_small_kernel<kSplit, 1><<<tiles, kSmallThreads, 0, s>>>(X, n, m->d_params, m->d_stats, Y);
        else
            mlp_infer_small_kernel<kSplit, 2>
                <<<std::min(kSMs, (tiles + 1) / 2), kSmallThreads, 0, s>>>(X, n, m->d_params, m->d_stats, Y);
        return cudaGetLastError();
    }
    const int smem = (int)sizeof(InferSmem);
    const cudaError_t e =
        cudaFuncSetAttribute(mlp_infer_kernel<kSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    mlp_infer_kernel<kSplit><<<std::min(kSMs, tiles), kInferThreads, smem, s>>>(X, n, m->d_params, m->d_stats, Y);
    return cudaGetLastError();
}

extern "C" int lbm_surrogate_predict_device(lbm_surrogate* m, const float* X_dev, int n, float* Y_dev, int mode,
                                            void* stream) {
    if (!m || !X_dev || !Y_dev || n < 1 || (mode != LBM_INFER_SPLIT_BF16 && mode != LBM_INFER_BF16)) return LBM_ERR_ARG;
    cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : m->stream;
    MCK(mode == LBM_INFER_SPLIT_BF16 ? infer<true>(m, X_dev, n, Y_dev, s) : infer<false>(m, X_dev, n, Y_dev, s));
    return LBM_OK;
}

extern "C" int lbm_surrogate_predict(lbm_surrogate* m, const float* X, int n, float* Y, int mode) {
    if (!m || !X || !Y || n < 1) return LBM_ERR_ARG;
    int rc = alloc_rows(m, n);
    if (rc) return rc;
    MCK(cudaMemcpyAsync(m->d_X, X, sizeof(float) * n * kIn, cudaMemcpyHostToDevice, m->stream));
    rc = lbm_surrogate_predict_device(m, m->d_X, n, m->d_out, mode, m->stream);
    if (rc) return rc;
    MCK(cudaMemcpyAsync(Y, m->d_out, sizeof(float) * n * kOut, cudaMemcpyDeviceToHost, m->stream));
    MCK(cudaStreamSynchronize(m->stream));
    return LBM_OK;
}

extern "C" int lbm_surrogate_stats(const lbm_surrogate* m, float* stats16) {
    if (!m || !stats16) return LBM_ERR_ARG;
    std::memcpy(stats16, m->h_stats, sizeof(m->h_stats));
    return LBM_OK;
}
