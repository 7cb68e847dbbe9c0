// mlp_infer.cuh -- fused tensor-core inference of the calibration surrogate.
//
// A warp takes 16 queries through all four layers without leaving its registers: the accumulators of a
// layer (mma.sync m16n8k16, BF16 x BF16 -> FP32, started at the bias) are, after GELU in FP32, the A
// fragments of the next one.  A CTA of 12 warps stages the whole network once, converting the FP32
// parameters to BF16 on the way, in the order in which a lane's B fragments of two adjacent n-tiles are
// one 16-byte read; then its warps walk over the queries.
//
// Split mode (kSplit): every FP32 operand x is carried as two BF16 numbers, hi = bf16(x) and
// lo = bf16(x - hi), and each tile accumulates hi*hi + lo*hi + hi*lo (the lo*lo term, below
// 2^-16 relative, is dropped): BF16 tensor-core products with FP32 accumulation that keep the
// result within ~2^-16 of the FP32 network.  Single mode rounds every operand to BF16 once
// (relative 2^-8), which costs up to ~1% in rho_v because ln rho_v spans several units.
//
// What bounds it: the tensor pipe, 8.2 cycles per m16n8k16 and sub-partition (measured), 840 of them per
// 16 queries in split mode; below a few thousand queries, staging 137 KB of parameters per CTA.  An
// earlier form kept the activations in shared memory and staged packed weights 2 bytes at a time for
// every 64 queries: 1090 us for 262,144 queries against 147, 53 us for 4096 against 15.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace {

constexpr int kInferWarps = 12;
constexpr int kInferThreads = 32 * kInferWarps;
constexpr int kInferRows = 16;  // queries per warp

// B fragments by part (hi, lo): [k-step][n-tile pair][lane] for the hidden layers, [n-tile pair][lane] for
// the first (K padded to 16), [k-step][lane] for the output layer (N padded to 8).
struct InferSmem {
    uint4 w[2][2][8][8][32];
    uint4 w1[2][8][32];
    uint2 w4[2][8][32];
    float bias[3][kHid];
    float b4[8];
    float stats[16];
};

// (x, y) -> hi = bf16x2(x, y), lo = bf16x2(x - hi.x, y - hi.y)
__device__ __forceinline__ void split_bf16(float2 v, uint32_t& hi, uint32_t& lo) {
    __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
    const float2 hf = __bfloat1622float2(h);
    __nv_bfloat162 l = __floats2bfloat162_rn(v.x - hf.x, v.y - hf.y);
    hi = *reinterpret_cast<uint32_t*>(&h);
    lo = *reinterpret_cast<uint32_t*>(&l);
}

// D (16x8, f32) += A (16x16, bf16, row) * B (16x8, bf16, col)
__device__ __forceinline__ void mma_bf16(float d[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// GELU of two values: gelu(z) = max(z, 0) - |z| Phi(-|z|) with Phi(-a) = 2^-Q(a), Q a polynomial of degree
// 8 fitted to -log2(erfc(a / sqrt 2) / 2) by Lawson's reweighted least squares, weighted by a Phi(-a) over
// 0 <= a <= 6 (beyond, Q keeps growing).  Largest error of the FP32 evaluation against erfc in 64 bits:
// 4e-8 over all z, as FP32 arithmetic on the exact formula has.  16 instructions for two values where erff
// and its branches take 33 issue cycles for one (measured).
__device__ __forceinline__ float2 gelu2(float2 z) {
    const float2 a = make_float2(fabsf(z.x), fabsf(z.y));
    auto c = [](float v) { return make_float2(v, v); };
    float2 q = __ffma2_rn(c(-2.0272058e-6f), a, c(2.9755707e-5f));
    q = __ffma2_rn(q, a, c(-1.4077181e-4f));
    q = __ffma2_rn(q, a, c(-2.4565138e-4f));
    q = __ffma2_rn(q, a, c(7.2036688e-3f));
    q = __ffma2_rn(q, a, c(-5.2591316e-2f));
    q = __ffma2_rn(q, a, c(-0.45917800f));
    q = __ffma2_rn(q, a, c(-1.1511084f));
    q = __ffma2_rn(q, a, c(-1.0f));
    float2 t;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t.x) : "f"(q.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t.y) : "f"(q.y));
    return __ffma2_rn(make_float2(-a.x, -a.y), t, make_float2(fmaxf(z.x, 0.0f), fmaxf(z.y, 0.0f)));
}

// Fill the CTA's network from the FP32 parameters P.
template <bool kSplit>
__device__ __forceinline__ void stage_network(InferSmem& s, const float* __restrict__ P,
                                              const float* __restrict__ stats) {
    const int tid = threadIdx.x;
    auto pair = [&](const float* w) { return *reinterpret_cast<const float2*>(w); };
#pragma unroll 2
    for (int e = tid; e < 2 * 8 * 8 * 32; e += kInferThreads) {
        const int lane = e & 31, np = (e >> 5) & 7, ks = (e >> 8) & 7, l = e >> 11;
        const float* w = P + woff(1 + l) + (np * 16 + (lane >> 2)) * kHid + ks * 16 + (lane & 3) * 2;
        const float2 v[4] = {pair(w), pair(w + 8), pair(w + 8 * kHid), pair(w + 8 * kHid + 8)};
        uint32_t h[4], o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) split_bf16(v[j], h[j], o[j]);
        s.w[l][0][ks][np][lane] = make_uint4(h[0], h[1], h[2], h[3]);
        if (kSplit) s.w[l][1][ks][np][lane] = make_uint4(o[0], o[1], o[2], o[3]);
    }
    for (int e = tid; e < 8 * 32; e += kInferThreads) {
        const int lane = e & 31, j = e >> 5, k = (lane & 3) * 2;
        // first layer: inputs 4 .. 15 are padding
        const float* w = P + woff(0) + (j * 16 + (lane >> 2)) * kIn + k;
        const float2 zero = make_float2(0.0f, 0.0f);
        uint32_t h[2], o[2];
        split_bf16(k < kIn ? pair(w) : zero, h[0], o[0]);
        split_bf16(k < kIn ? pair(w + 8 * kIn) : zero, h[1], o[1]);
        s.w1[0][j][lane] = make_uint4(h[0], 0, h[1], 0);
        if (kSplit) s.w1[1][j][lane] = make_uint4(o[0], 0, o[1], 0);
        // output layer: outputs 4 .. 7 are padding
        const float* u = P + woff(3) + (lane >> 2) * kHid + j * 16 + k;
        split_bf16((lane >> 2) < kOut ? pair(u) : zero, h[0], o[0]);
        split_bf16((lane >> 2) < kOut ? pair(u + 8) : zero, h[1], o[1]);
        s.w4[0][j][lane] = make_uint2(h[0], h[1]);
        if (kSplit) s.w4[1][j][lane] = make_uint2(o[0], o[1]);
    }
    for (int i = tid; i < 3 * kHid; i += kInferThreads) s.bias[i / kHid][i % kHid] = P[boff(i / kHid) + i % kHid];
    if (tid < 8) s.b4[tid] = tid < kOut ? P[boff(3) + tid] : 0.0f;
    if (tid < 16) s.stats[tid] = stats[tid];
}

// X, Y: n x 4, row-major.
template <bool kSplit>
__global__ void __launch_bounds__(kInferThreads, 1)
    mlp_infer_kernel(const float* __restrict__ X, int n, const float* __restrict__ P, const float* __restrict__ stats,
                     float* __restrict__ Y) {
    extern __shared__ __align__(16) unsigned char ism[];
    InferSmem& s = *reinterpret_cast<InferSmem*>(ism);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int tiles = (n + kInferRows - 1) / kInferRows, stride = gridDim.x * kInferWarps;
    int tile = warp * gridDim.x + blockIdx.x;
    // a lane's inputs: columns 2t, 2t + 1 (t < 2) of rows g and g + 8
    auto load = [&](int tl, float2 x[2]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const long long r = (long long)tl * kInferRows + g + 8 * h;
            const float* p = X + r * kIn + 2 * t;  // (aligned to 4 bytes only)
            x[h] = t < 2 && r < n ? make_float2(__ldg(p), __ldg(p + 1)) : make_float2(0.0f, 0.0f);
        }
    };
    float2 x[2];
    load(tile, x);
    stage_network<kSplit>(s, P, stats);
    __syncthreads();
    float acc[16][4];
    uint32_t ah[8][4], al[8][4];
    for (; tile < tiles; tile += stride) {
        // standardised inputs as the A fragment of one k-step (columns 4 .. 15 zero)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 v = t < 2 ? make_float2((x[h].x - s.stats[2 * t]) / s.stats[4 + 2 * t],
                                                 (x[h].y - s.stats[2 * t + 1]) / s.stats[5 + 2 * t])
                                   : make_float2(0.0f, 0.0f);
            split_bf16(v, ah[0][h], al[0][h]);
            ah[0][2 + h] = al[0][2 + h] = 0;
        }
        load(tile + stride, x);
        auto start = [&](int layer) {
#pragma unroll
            for (int nt = 0; nt < 16; ++nt) {
                const float2 b = *reinterpret_cast<const float2*>(&s.bias[layer][nt * 8 + 2 * t]);
                acc[nt][0] = acc[nt][2] = b.x;
                acc[nt][1] = acc[nt][3] = b.y;
            }
        };
        // two n-tiles of one k-step
        auto tile_pair = [&](int np, const uint4& bh, const uint4* lo, const uint32_t a[4], const uint32_t b[4]) {
            mma_bf16(acc[2 * np], a, bh.x, bh.y);
            mma_bf16(acc[2 * np + 1], a, bh.z, bh.w);
            if (kSplit) {
                const uint4 bl = *lo;
                mma_bf16(acc[2 * np], b, bh.x, bh.y);
                mma_bf16(acc[2 * np + 1], b, bh.z, bh.w);
                mma_bf16(acc[2 * np], a, bl.x, bl.y);
                mma_bf16(acc[2 * np + 1], a, bl.z, bl.w);
            }
        };
        // GELU, and the accumulators of n-tiles 2 ks, 2 ks + 1 as the A fragment of k-step ks
        auto activate = [&]() {
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float* c = acc[2 * ks + (j >> 1)];
                    split_bf16(gelu2(make_float2(c[2 * (j & 1)], c[2 * (j & 1) + 1])), ah[ks][j], al[ks][j]);
                }
        };
        start(0);
#pragma unroll
        for (int np = 0; np < 8; ++np) tile_pair(np, s.w1[0][np][lane], &s.w1[1][np][lane], ah[0], al[0]);
        activate();
#pragma unroll 1
        for (int l = 0; l < 2; ++l) {
            start(l + 1);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
#pragma unroll
                for (int np = 0; np < 8; ++np)
                    tile_pair(np, s.w[l][0][ks][np][lane], &s.w[l][1][ks][np][lane], ah[ks], al[ks]);
            activate();
        }
        // output layer: three chains of accumulators, summed
        float o[3][4] = {{s.b4[2 * t], s.b4[2 * t + 1], s.b4[2 * t], s.b4[2 * t + 1]}, {}, {}};
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            const uint2 bh = s.w4[0][ks][lane];
            mma_bf16(o[0], ah[ks], bh.x, bh.y);
            if (kSplit) {
                const uint2 bl = s.w4[1][ks][lane];
                mma_bf16(o[1], al[ks], bh.x, bh.y);
                mma_bf16(o[2], ah[ks], bl.x, bl.y);
            }
        }
        if (t < 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const long long r = (long long)tile * kInferRows + g + 8 * h;
                if (r >= n) continue;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int c = 2 * t + j, k = 2 * h + j;
                    const float y = (o[0][k] + (o[1][k] + o[2][k])) * s.stats[12 + c] + s.stats[8 + c];
                    Y[r * kOut + c] = c == 1 ? expf(y) : y;  // rho_v is learned as ln rho_v
                }
            }
        }
    }
}

}  // namespace
