// mlp_train.cuh -- FP32 forward and backward pass of the calibration surrogate in one kernel.
//
// A CTA of 512 threads takes up to 56 samples through all four layers and back.  The activations
// A_l and the derivatives gelu'(Z_l) of the three hidden layers stay in shared memory (feature-major,
// 184 KB), the hidden weights stream through three 8 KB stages, dZ_l overwrites
// gelu'(Z_l), and the CTA's share of the parameter gradient goes to its own slot, summed in slot
// order by mlp_update_kernel: no atomics, no activations in global memory, two launches per iteration.
//
// What bounds it: the FMA pipe and, close behind, shared-memory reads (a 16-byte read costs at least
// two wavefronts however few addresses a warp names).  So all six 128 x 128 products of a tile are
// 8 x 4 register tiles in packed FP32: three 16-byte reads per 16 packed multiply-adds (4 x 4 tiles,
// two per 8, were bound by the reads: 77 us per iteration of 7973 samples against 70).  The products
// then run at 55% of the FMA rate (14.8k cycles for 8.2k), the weight gradients at half of it.
// 7973 samples, one iteration with its update: 332 us as separate products, passes and atomics, 66 us now.
#pragma once
#include <cuda_runtime.h>

namespace {

constexpr int kTrainRows = 56;             // most samples per tile
constexpr int kTrainStride = kTrainRows + 4;
constexpr int kTrainStages = 3;
constexpr int kTrainThreads = 512;
constexpr int kSlot = 34184;               // floats per gradient slot: the parameters, then the loss

struct TrainSmem {
    float A[3][kHid][kTrainStride];   // activations of the hidden layers, [feature][sample]
    float G[3][kHid][kTrainStride];   // gelu'(Z), then dZ
    float W[kTrainStages][16][kHid];  // staged weight rows; partial sums of the output layer
    float x[kIn][kTrainStride];
    float y[kOut][kTrainStride];      // targets, then dZ4
    float w1[kHid][kIn];
    float b[4][kHid];
    float w4[kHid][kOut];             // output weights by feature
};
static_assert(sizeof(TrainSmem) <= 232448, "one CTA's shared memory");

__device__ __forceinline__ void stage16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// A thread's place in the 128 features x 56 samples of a layer.  Half the warps (g = 0) sum the first 64
// terms of each product, half (g = 1) the rest; a lane accumulates features c0 .. c0 + 7 of samples
// m0 .. m0 + 3 and, after the halves are exchanged, holds features c .. c + 3 complete.
struct TrainLane {
    int g, c0, m0, c, x;  // x: this lane's place in the exchange between the halves
    bool on;  // this lane's samples are computed (samples M .. of a partly wanted warp are, but not read)
};
__device__ __forceinline__ TrainLane train_lane(int M) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    TrainLane L;
    L.g = warp >> 3;
    L.c0 = (warp & 3) * 32 + (lane & 3) * 8;
    L.m0 = ((warp >> 2) & 1) * 32 + (lane >> 2) * 4;
    L.c = L.c0 + 4 * L.g;
    L.on = ((warp >> 2) & 1) * 32 < M && L.m0 < kTrainRows;
    const int per = (kTrainRows - 32) / 4 * 4;  // lanes of a warp of the second 32 samples
    L.x = (warp & 4 ? 128 + (warp & 3) * per : (warp & 3) * 32) + lane;
    return L;
}

// Stage chunk ch of a product's weights: 8 rows of each half, one float4 per thread.
__device__ __forceinline__ void train_stage(TrainSmem& s, const float* __restrict__ Wg, int ch, int stage) {
    const int r = threadIdx.x >> 5, c = (threadIdx.x & 31) * 4;
    stage16(&s.W[stage][r][c], Wg + ((r >> 3) * 64 + (r & 7) + 8 * ch) * kHid + c);
}
__device__ __forceinline__ void train_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// The first two chunks, in stages 0 and 1: issued as soon as those are free, a phase ahead of the product.
__device__ __forceinline__ void train_prefetch(TrainSmem& s, const float* __restrict__ Wg) {
    for (int ch = 0; ch < 2; ++ch) {
        train_stage(s, Wg, ch, ch);
        train_commit();
    }
}

// out[i][q] = sum_r Wg[r][L.c + i] in[r][L.m0 + q] over the 128 rows r of Wg (row-major, 128 wide), its
// first chunks prefetched; next: the next product's weights, prefetched at the end.  Called by all
// threads; scratch (28 KB) is free for the exchange between the halves, and is still being read when the
// function returns.
__device__ __forceinline__ void train_gemm(TrainSmem& s, const float* __restrict__ Wg,
                                           const float (*in)[kTrainStride], const TrainLane& L, float* scratch,
                                           float out[4][4], const float* __restrict__ next) {
    float2 acc[4][4];  // feature pairs x samples
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = make_float2(0.0f, 0.0f);
    int b = 0, nb = 2;  // stage of chunk ch, and of chunk ch + 2 (the one chunk ch - 1 was read from)
    for (int ch = 0; ch < 8; ++ch) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();  // chunk ch has landed, and every warp is done with chunk ch - 1
        if (ch + 2 < 8) train_stage(s, Wg, ch + 2, nb);
        train_commit();
        if (L.on) {
            const float(*W)[kHid] = s.W[b] + 8 * L.g;
            const float(*a)[kTrainStride] = in + 64 * L.g + 8 * ch;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float4 w0 = *reinterpret_cast<const float4*>(&W[r][L.c0]);
                const float4 w1 = *reinterpret_cast<const float4*>(&W[r][L.c0 + 4]);
                const float4 x = *reinterpret_cast<const float4*>(&a[r][L.m0]);
                const float2 w[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                                     make_float2(w1.z, w1.w)};
                const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float2 xx = make_float2(xv[q], xv[q]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[i][q] = __ffma2_rn(w[i], xx, acc[i][q]);
                }
            }
        }
        b = b == kTrainStages - 1 ? 0 : b + 1;
        nb = nb == kTrainStages - 1 ? 0 : nb + 1;
    }
    // half 0 completes the lower four features, half 1 the upper four
    constexpr int kHalf = 4 * kTrainRows;  // lanes of a half
    float4* x = reinterpret_cast<float4*>(scratch);
    if (L.on) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 u = L.g ? acc[0][q] : acc[2][q], v = L.g ? acc[1][q] : acc[3][q];
            x[(2 * q + L.g) * kHalf + L.x] = make_float4(u.x, u.y, v.x, v.y);
        }
    }
    __syncthreads();
    if (next) train_prefetch(s, next);
    if (L.on) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 u = L.g ? acc[2][q] : acc[0][q], v = L.g ? acc[3][q] : acc[1][q];
            const float4 o = x[(2 * q + 1 - L.g) * kHalf + L.x];
            out[0][q] = u.x + o.x;
            out[1][q] = u.y + o.y;
            out[2][q] = v.x + o.z;
            out[3][q] = v.y + o.w;
        }
    }
}

// out[j][k] (+)= sum_{m < M} dz[j][m] a[k][m], all 128 x 128: a warp 64 j x 16 k, a lane 8 x 4, the even
// and odd samples in the two halves of a packed accumulator.
__device__ __forceinline__ void train_dw(const float (*dz)[kTrainStride], const float (*a)[kTrainStride], int M,
                                         float* __restrict__ out, bool add) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j0 = (warp & 1) * 64 + (lane & 7), k0 = (warp >> 1) * 16 + (lane >> 3) * 4;
    float2 acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = make_float2(0.0f, 0.0f);
#pragma unroll 1
    for (int m = 0; m < M; m += 4) {
        float4 av[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) av[q] = *reinterpret_cast<const float4*>(&a[k0 + q][m]);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 d = *reinterpret_cast<const float4*>(&dz[j0 + 8 * i][m]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                acc[i][q] = __ffma2_rn(make_float2(d.x, d.y), make_float2(av[q].x, av[q].y), acc[i][q]);
                acc[i][q] = __ffma2_rn(make_float2(d.z, d.w), make_float2(av[q].z, av[q].w), acc[i][q]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float4* o = reinterpret_cast<float4*>(out + (j0 + 8 * i) * kHid + k0);
        float4 v = make_float4(acc[i][0].x + acc[i][0].y, acc[i][1].x + acc[i][1].y, acc[i][2].x + acc[i][2].y,
                               acc[i][3].x + acc[i][3].y);
        if (add) {
            const float4 w = *o;
            v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
        }
        *o = v;
    }
}

// sum over m < M of p[m] q[m] (rows of shared memory), four interleaved chains
__device__ __forceinline__ float train_dot(const float* p, const float* q, int M) {
    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int m = 0; m < M; m += 4) {
        const float4 u = *reinterpret_cast<const float4*>(p + m), v = *reinterpret_cast<const float4*>(q + m);
        a = make_float4(fmaf(u.x, v.x, a.x), fmaf(u.y, v.y, a.y), fmaf(u.z, v.z, a.z), fmaf(u.w, v.w, a.w));
    }
    return (a.x + a.y) + (a.z + a.w);
}
__device__ __forceinline__ float train_sum(const float* p, int M) {
    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int m = 0; m < M; m += 4) {
        const float4 u = *reinterpret_cast<const float4*>(p + m);
        a = make_float4(a.x + u.x, a.y + u.y, a.z + u.z, a.w + u.w);
    }
    return (a.x + a.y) + (a.z + a.w);
}

// z -> gelu(z), gelu'(z) with one erff
__device__ __forceinline__ void gelu_both(float z, float& a, float& g) {
    const float e = 1.0f + erff(z * 0.70710678118654752f);
    a = 0.5f * z * e;
    g = 0.5f * e + z * (0.39894228040143268f * expf(-0.5f * z * z));
}

// Xn (n x 4, standardised), Yn (n x 4; NaN: missing) and parameters P, with WT the two hidden weight
// matrices transposed ([k][j]).  CTA b takes tiles b, b + gridDim.x, ... of M samples (a multiple of 4,
// at most 56).  BACKWARD: dLoss/dP and the sum of squared errors of its samples into slot b of part;
// otherwise Z4 (n x 4) into Zout.
template <bool BACKWARD>
__global__ void __launch_bounds__(kTrainThreads, 1)
    mlp_train_kernel(const float* __restrict__ Xn, const float* __restrict__ Yn, int n, int M,
                     const float* __restrict__ P, const float* __restrict__ WT, float inv_valid,
                     float* __restrict__ part, float* __restrict__ Zout) {
    extern __shared__ __align__(16) unsigned char tsm[];
    TrainSmem& s = *reinterpret_cast<TrainSmem*>(tsm);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const TrainLane L = train_lane(M);
    const int c0 = L.c, m0 = L.m0;  // this thread's 4 x 4 of every layer
    const bool on = L.on;
    float* slot = BACKWARD ? part + (size_t)blockIdx.x * kSlot : nullptr;
    s.w4[t >> 2][t & 3] = P[woff(3) + (t & 3) * kHid + (t >> 2)];
    s.w1[t >> 2][t & 3] = P[woff(0) + t];
    s.b[t >> 7][t & 127] = t < 3 * kHid + kOut ? P[boff(t >> 7) + (t & 127)] : 0.0f;
    bool add = false;
    for (int tile = blockIdx.x; (long long)tile * M < n; tile += gridDim.x, add = true) {
        const int q0 = tile * M, cnt = min(M, n - q0);
        __syncthreads();
        if (t < 4 * kTrainRows) {
            const int m = t >> 2, i = t & 3;
            s.x[i][m] = m < cnt ? Xn[(size_t)(q0 + m) * kIn + i] : 0.0f;
            if (BACKWARD) s.y[i][m] = m < cnt ? Yn[(size_t)(q0 + m) * kOut + i] : nanf("");
        }
        train_prefetch(s, WT);
        __syncthreads();
        // layer 1: K = 4
        if (on) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 w = *reinterpret_cast<const float4*>(s.w1[c0 + i]);
                const float b = s.b[0][c0 + i];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int m = m0 + q;
                    const float z = fmaf(w.w, s.x[3][m], fmaf(w.z, s.x[2][m], fmaf(w.y, s.x[1][m], w.x * s.x[0][m]))) + b;
                    gelu_both(z, s.A[0][c0 + i][m], s.G[0][c0 + i][m]);
                }
            }
        }
        __syncthreads();
        // hidden layers 2, 3
        for (int l = 1; l < 3; ++l) {
            float z[4][4];
            train_gemm(s, WT + (l - 1) * kHid * kHid, s.A[l - 1], L, &s.G[l][0][0], z,
                       l == 1 ? WT + kHid * kHid : BACKWARD ? P + woff(2) : nullptr);
            __syncthreads();  // the exchange has been read
            if (on) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float b = s.b[l][c0 + i];
                    float a[4], g[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) gelu_both(z[i][q] + b, a[q], g[q]);
                    *reinterpret_cast<float4*>(&s.A[l][c0 + i][m0]) = make_float4(a[0], a[1], a[2], a[3]);
                    *reinterpret_cast<float4*>(&s.G[l][c0 + i][m0]) = make_float4(g[0], g[1], g[2], g[3]);
                }
            }
            __syncthreads();
        }
        // output layer: thread (m, p) sums 16 features of sample m for all four outputs
        float(*red)[kTrainRows][4] = reinterpret_cast<float(*)[kTrainRows][4]>(&s.W[2][0][0]);  // [8][56][4]
        if ((t & 63) < kTrainRows) {
            const int m = t & 63, p = t >> 6;
            float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
            for (int k = 16 * p; k < 16 * p + 16; ++k) {
                const float a = s.A[2][k][m];
                const float4 w = *reinterpret_cast<const float4*>(s.w4[k]);
                z = make_float4(fmaf(a, w.x, z.x), fmaf(a, w.y, z.y), fmaf(a, w.z, z.z), fmaf(a, w.w, z.w));
            }
            *reinterpret_cast<float4*>(red[p][m]) = z;
        }
        __syncthreads();
        if (t < 4 * kTrainRows) {
            const int m = t >> 2, o = t & 3;
            float z = 0.0f;
#pragma unroll
            for (int p = 0; p < 8; ++p) z += red[p][m][o];
            z += s.b[3][o];
            if (!BACKWARD) {
                if (m < cnt) Zout[(size_t)(q0 + m) * kOut + o] = z;
            } else {
                const float d = isnan(s.y[o][m]) ? 0.0f : z - s.y[o][m];  // NaN: missing, or beyond the batch
                s.y[o][m] = 2.0f * d * inv_valid;
                red[0][m][o] = d;  // (this thread read red[0][m][o] above)
            }
        }
        if (!BACKWARD) continue;
        __syncthreads();
        // squared errors, output bias and weights; dZ3 = (W4^T dZ4) gelu'(Z3)
        if (warp == 0) {
            float e = 0.0f;
            for (int k = lane; k < M * 4; k += 32) {
                const float d = (&red[0][0][0])[k];
                e = fmaf(d, d, e);
            }
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (lane == 0) slot[kNumParams] = (add ? slot[kNumParams] : 0.0f) + e;
        } else if (warp == 1 && lane < 4) {
            const float v = train_sum(s.y[lane], M);
            slot[boff(3) + lane] = (add ? slot[boff(3) + lane] : 0.0f) + v;
        }
        {
            float* o = slot + woff(3) + t;  // output t >> 7, feature t & 127
            *o = (add ? *o : 0.0f) + train_dot(s.y[t >> 7], s.A[2][t & 127], M);
        }
        if (on) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 w = *reinterpret_cast<const float4*>(s.w4[c0 + i]);
                float4* g = reinterpret_cast<float4*>(&s.G[2][c0 + i][m0]);
                const float4 h = *g;
                float v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    v[q] = fmaf(w.w, s.y[3][m0 + q], fmaf(w.z, s.y[2][m0 + q], fmaf(w.y, s.y[1][m0 + q], w.x * s.y[0][m0 + q])));
                *g = make_float4(v[0] * h.x, v[1] * h.y, v[2] * h.z, v[3] * h.w);
            }
        }
        __syncthreads();
        // hidden layers 3, 2: weight gradient, then dZ of the layer below
        for (int l = 2; l > 0; --l) {
            train_dw(s.G[l], s.A[l - 1], M, slot + woff(l), add);
            float d[4][4];
            train_gemm(s, P + woff(l), s.G[l], L, &s.A[l][0][0], d, l == 2 ? P + woff(1) : nullptr);
            if (on) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float4* g = reinterpret_cast<float4*>(&s.G[l - 1][c0 + i][m0]);
                    const float4 h = *g;
                    *g = make_float4(d[i][0] * h.x, d[i][1] * h.y, d[i][2] * h.z, d[i][3] * h.w);
                }
            }
            __syncthreads();
        }
        // first layer's weights, hidden biases
        {
            float* o = slot + woff(0) + t;  // feature t >> 2, input t & 3
            *o = (add ? *o : 0.0f) + train_dot(s.G[0][t >> 2], s.x[t & 3], M);
        }
        if (t < 3 * kHid) {
            const int l = t >> 7, j = t & 127;
            float* o = slot + boff(l) + j;
            *o = (add ? *o : 0.0f) + train_sum(s.G[l][j], M);
        }
    }
}

// WT[l][k][j] = W_{l+2}[j][k] of both hidden matrices
__global__ void mlp_transpose_kernel(const float* __restrict__ P, float* __restrict__ WT) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 2 * kHid * kHid; i += gridDim.x * blockDim.x) {
        const int l = i / (kHid * kHid), k = i / kHid % kHid, j = i % kHid;
        WT[i] = P[woff(l + 1) + j * kHid + k];
    }
}

// The gradient (and the loss) from the slots, summed in a fixed order, and with ADAM the update of the
// parameters and of the transposed copies.  A CTA takes 32 parameters; its eight warps read every
// eighth slot each (a warp per 128-byte run of a slot), which keeps 8 x as many loads in flight as one
// thread per parameter (an iteration of 7973 samples, 143 slots: 69.6 us against 67.5).
constexpr int kUpdateWarps = 8;
template <bool ADAM>
__global__ void __launch_bounds__(32 * kUpdateWarps)
    mlp_update_kernel(const float* __restrict__ part, int slots, float inv_valid, float* __restrict__ grad,
                      float* __restrict__ loss, float* __restrict__ p, float* __restrict__ WT, float* __restrict__ m1,
                      float* __restrict__ m2, float lr, float b1, float b2, float eps, float c1, float c2, float wd) {
    __shared__ float red[kUpdateWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    float s = 0.0f;
    if (i <= kNumParams) {
        float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        int b = warp;
        for (; b + 3 * kUpdateWarps < slots; b += 4 * kUpdateWarps)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] += __ldg(part + (size_t)(b + k * kUpdateWarps) * kSlot + i);
        for (int k = 0; b < slots; b += kUpdateWarps, ++k) v[k] += __ldg(part + (size_t)b * kSlot + i);
        s = (v[0] + v[1]) + (v[2] + v[3]);
    }
    red[warp][lane] = s;
    __syncthreads();
    if (warp != 0 || i > kNumParams) return;
    const float gi = ((red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane])) +
                     ((red[4][lane] + red[5][lane]) + (red[6][lane] + red[7][lane]));
    if (i == kNumParams) {
        *loss = gi * inv_valid;
        return;
    }
    grad[i] = gi;
    if (!ADAM) return;
    const float a = b1 * m1[i] + (1.0f - b1) * gi;
    const float v = b2 * m2[i] + (1.0f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = v;
    const float w = p[i] - lr * ((a / c1) / (sqrtf(v / c2) + eps) + wd * p[i]);
    p[i] = w;
    for (int l = 1; l < 3; ++l) {
        const int k = i - woff(l);
        if (k >= 0 && k < kHid * kHid) WT[(l - 1) * kHid * kHid + k % kHid * kHid + k / kHid] = w;
    }
}

}  // namespace
