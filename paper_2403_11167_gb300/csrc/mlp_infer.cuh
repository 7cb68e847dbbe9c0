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
// 16 queries in split mode (262,144 queries: 146 us).  An earlier form kept the activations in shared memory
// and staged packed weights 2 bytes at a time for every 64 queries: 1090 us.
//
// With few queries a warp that takes them through the network alone leaves the other sub-partitions idle and
// staging 137 KB of parameters costs as much again; mlp_infer_small_kernel splits every layer's outputs over
// the warps instead (4096 queries: 10.4 us against 14.7, in a graph 7.6; of these about 2 are the launch, 2
// the parameters' way from L2, 1.6 the products).
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
// 0 <= a <= 6 (beyond, Q keeps growing).  Error of the FP32 evaluation against erfc in 64 bits: below 6.3e-8 plus
// 2^-24 of the value (tests/test_gpu_math.py).  16 instructions for two values where erff
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

// Which neuron of a block of 16 stands at place p of a fragment (of the n-tile pair that computes it, and of
// the k-step that reads it): the four places 2t, 2t + 1, 2t + 8, 2t + 9 of a lane are neurons 4t .. 4t + 3,
// so that its weights are one 16-byte read.  Returned for place g < 8; place g + 8 is the neuron two on.
__device__ __forceinline__ int block_neuron(int g) { return 4 * (g >> 1) + (g & 1); }

// B fragments (hi, lo) of k-step ks for the n-tile pair np of hidden layer l (1, 2), from the FP32 weights.
__device__ __forceinline__ void load_hidden(const float* __restrict__ P, int l, int ks, int np, int lane, float4 w[2]) {
    const float* p = P + woff(l) + (np * 16 + block_neuron(lane >> 2)) * kHid + ks * 16 + 4 * (lane & 3);
    w[0] = __ldg(reinterpret_cast<const float4*>(p));
    w[1] = __ldg(reinterpret_cast<const float4*>(p + 2 * kHid));
}
__device__ __forceinline__ void split_hidden(const float4 w[2], uint4& hi, uint4& lo) {
    split_bf16(make_float2(w[0].x, w[0].y), hi.x, lo.x);
    split_bf16(make_float2(w[0].z, w[0].w), hi.y, lo.y);
    split_bf16(make_float2(w[1].x, w[1].y), hi.z, lo.z);
    split_bf16(make_float2(w[1].z, w[1].w), hi.w, lo.w);
}
// The first layer's (inputs 4 .. 15 of its k-step are padding).
__device__ __forceinline__ void load_first(const float* __restrict__ P, int np, int lane, uint4& hi, uint4& lo) {
    const int k = 2 * (lane & 3);
    const float* p = P + woff(0) + (np * 16 + block_neuron(lane >> 2)) * kIn + k;
    auto pair = [&](const float* w) {
        return k < kIn ? __ldg(reinterpret_cast<const float2*>(w)) : make_float2(0.0f, 0.0f);
    };
    hi = lo = make_uint4(0, 0, 0, 0);
    split_bf16(pair(p), hi.x, lo.x);
    split_bf16(pair(p + 2 * kIn), hi.z, lo.z);
}
// The output layer's (outputs 4 .. 7 are padding).
__device__ __forceinline__ void load_last(const float* __restrict__ P, int ks, int lane, uint2& hi, uint2& lo) {
    const int g = lane >> 2;
    const float4 w = g < kOut ? __ldg(reinterpret_cast<const float4*>(P + woff(3) + g * kHid + ks * 16 + 4 * (lane & 3)))
                              : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    split_bf16(make_float2(w.x, w.y), hi.x, lo.x);
    split_bf16(make_float2(w.z, w.w), hi.y, lo.y);
}

// A lane's inputs of one tile of 16 queries, columns 2t, 2t + 1 (t < 2) of rows g and g + 8 (0 beyond n),
// and the same standardised as the A fragment of one k-step (columns 4 .. 15 zero).
__device__ __forceinline__ void load_queries(const float* __restrict__ X, int n, int tile, int g, int t, float2 x[2]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const long long r = (long long)tile * kInferRows + g + 8 * h;
        const float* p = X + r * kIn + 2 * t;  // (aligned to 4 bytes only)
        x[h] = t < 2 && r < n ? make_float2(__ldg(p), __ldg(p + 1)) : make_float2(0.0f, 0.0f);
    }
}
__device__ __forceinline__ void standardise_queries(const float2 x[2], const float* stats, int t, uint32_t ah[4],
                                                    uint32_t al[4]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 v = t < 2 ? make_float2((x[h].x - stats[2 * t]) / stats[4 + 2 * t],
                                             (x[h].y - stats[2 * t + 1]) / stats[5 + 2 * t])
                               : make_float2(0.0f, 0.0f);
        split_bf16(v, ah[h], al[h]);
        ah[2 + h] = al[2 + h] = 0;
    }
}

// acc (two n-tiles) += A B over one k-step
template <bool kSplit>
__device__ __forceinline__ void mma_pair(float c0[4], float c1[4], const uint32_t ah[4], const uint32_t al[4],
                                         const uint4& bh, const uint4& bl) {
    mma_bf16(c0, ah, bh.x, bh.y);
    mma_bf16(c1, ah, bh.z, bh.w);
    if (kSplit) {
        mma_bf16(c0, al, bh.x, bh.y);
        mma_bf16(c1, al, bh.z, bh.w);
        mma_bf16(c0, ah, bl.x, bl.y);
        mma_bf16(c1, ah, bl.z, bl.w);
    }
}
// GELU of the accumulators of an n-tile pair, as the A fragment of the k-step that reads the block
__device__ __forceinline__ void activate_pair(const float c0[4], const float c1[4], uint32_t ah[4], uint32_t al[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float* c = j < 2 ? c0 : c1;
        split_bf16(gelu2(make_float2(c[2 * (j & 1)], c[2 * (j & 1) + 1])), ah[j], al[j]);
    }
}
// accumulators of an n-tile pair from the block's biases (4 t onwards)
__device__ __forceinline__ void start_pair(float c0[4], float c1[4], const float* bias, int t) {
    const float4 b = *reinterpret_cast<const float4*>(bias + 4 * t);
    c0[0] = c0[2] = b.x;
    c0[1] = c0[3] = b.y;
    c1[0] = c1[2] = b.z;
    c1[1] = c1[3] = b.w;
}
// one k-step of the output layer: three chains of accumulators
template <bool kSplit>
__device__ __forceinline__ void mma_last(float o[3][4], const uint32_t ah[4], const uint32_t al[4], const uint2& bh,
                                         const uint2& bl) {
    mma_bf16(o[0], ah, bh.x, bh.y);
    if (kSplit) {
        mma_bf16(o[1], al, bh.x, bh.y);
        mma_bf16(o[2], ah, bl.x, bl.y);
    }
}
// the chains' sums, de-standardised (columns 2t, 2t + 1, t < 2, of rows g and g + 8)
__device__ __forceinline__ void store_outputs(float* __restrict__ Y, int n, int tile, int g, int t, const float o[3][4],
                                              const float* stats) {
    if (t >= 2) return;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const long long r = (long long)tile * kInferRows + g + 8 * h;
        if (r >= n) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int c = 2 * t + j, k = 2 * h + j;
            const float y = (o[0][k] + (o[1][k] + o[2][k])) * stats[12 + c] + stats[8 + c];
            Y[r * kOut + c] = c == 1 ? expf(y) : y;  // rho_v is learned as ln rho_v
        }
    }
}

// Fill the CTA's network from the FP32 parameters P.
template <bool kSplit>
__device__ __forceinline__ void stage_network(InferSmem& s, const float* __restrict__ P,
                                              const float* __restrict__ stats) {
    const int tid = threadIdx.x;
#pragma unroll 4
    for (int e = tid; e < 2 * 8 * 8 * 32; e += kInferThreads) {
        const int lane = e & 31, np = (e >> 5) & 7, ks = (e >> 8) & 7, l = e >> 11;
        float4 w[2];
        load_hidden(P, 1 + l, ks, np, lane, w);
        uint4 h, o;
        split_hidden(w, h, o);
        s.w[l][0][ks][np][lane] = h;
        if (kSplit) s.w[l][1][ks][np][lane] = o;
    }
    for (int e = tid; e < 8 * 32; e += kInferThreads) {
        const int lane = e & 31, j = e >> 5;
        uint4 h, o;
        load_first(P, j, lane, h, o);
        s.w1[0][j][lane] = h;
        if (kSplit) s.w1[1][j][lane] = o;
        uint2 u, v;
        load_last(P, j, lane, u, v);
        s.w4[0][j][lane] = u;
        if (kSplit) s.w4[1][j][lane] = v;
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
    float2 x[2];
    load_queries(X, n, tile, g, t, x);
    stage_network<kSplit>(s, P, stats);
    __syncthreads();
    float acc[16][4];
    uint32_t ah[8][4], al[8][4];
    for (; tile < tiles; tile += stride) {
        standardise_queries(x, s.stats, t, ah[0], al[0]);
        load_queries(X, n, tile + stride, g, t, x);
        auto start = [&](int layer) {
#pragma unroll
            for (int np = 0; np < 8; ++np) start_pair(acc[2 * np], acc[2 * np + 1], &s.bias[layer][16 * np], t);
        };
        auto activate = [&]() {
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) activate_pair(acc[2 * ks], acc[2 * ks + 1], ah[ks], al[ks]);
        };
        const uint4 none = make_uint4(0, 0, 0, 0);
        start(0);
#pragma unroll
        for (int np = 0; np < 8; ++np)
            mma_pair<kSplit>(acc[2 * np], acc[2 * np + 1], ah[0], al[0], s.w1[0][np][lane],
                             kSplit ? s.w1[1][np][lane] : none);
        activate();
#pragma unroll 1
        for (int l = 0; l < 2; ++l) {
            start(l + 1);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
#pragma unroll
                for (int np = 0; np < 8; ++np)
                    mma_pair<kSplit>(acc[2 * np], acc[2 * np + 1], ah[ks], al[ks], s.w[l][0][ks][np][lane],
                                     kSplit ? s.w[l][1][ks][np][lane] : none);
            activate();
        }
        float o[3][4] = {{s.b4[2 * t], s.b4[2 * t + 1], s.b4[2 * t], s.b4[2 * t + 1]}, {}, {}};
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
            mma_last<kSplit>(o, ah[ks], al[ks], s.w4[0][ks][lane], kSplit ? s.w4[1][ks][lane] : make_uint2(0, 0));
        store_outputs(Y, n, tile, g, t, o, s.stats);
    }
}

// The same network with every layer's outputs split over the eight warps of a CTA: warp w computes the 16
// neurons of block w for one or two tiles of 16 queries (MT at most) and holds its share of the hidden
// weights in registers, read straight from the FP32 parameters; the activations pass from layer to layer
// as A fragments in shared memory, one barrier per layer.  The products, their order and so the results are
// those of mlp_infer_kernel bit for bit.
constexpr int kSmallWarps = 8;
constexpr int kSmallThreads = 32 * kSmallWarps;
template <bool kSplit, int MT>
__global__ void __launch_bounds__(kSmallThreads, 1)
    mlp_infer_small_kernel(const float* __restrict__ X, int n, const float* __restrict__ P,
                           const float* __restrict__ stats, float* __restrict__ Y) {
    __shared__ uint4 s_a[2][MT][kSplit ? 2 : 1][8][32];
    __shared__ uint2 s_w4[kSplit ? 2 : 1][8][32];
    __shared__ float s_stats[16], s_b4[8];
    __shared__ __align__(16) float s_bias[3][kHid];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int tiles = (n + kInferRows - 1) / kInferRows;
    int tile = blockIdx.x * MT;
    float2 x[MT][2];
#pragma unroll
    for (int m = 0; m < MT; ++m) load_queries(X, n, tile + m, g, t, x[m]);
    if (threadIdx.x < 16) s_stats[threadIdx.x] = stats[threadIdx.x];
    if (threadIdx.x < 8) s_b4[threadIdx.x] = threadIdx.x < kOut ? P[boff(3) + threadIdx.x] : 0.0f;
    for (int i = threadIdx.x; i < 3 * kHid; i += kSmallThreads) s_bias[i / kHid][i % kHid] = P[boff(i / kHid) + i % kHid];
    uint4 w1h, w1l, wh[2][8], wl[2][8];
    load_first(P, warp, lane, w1h, w1l);
    {
        float4 raw[2][8][2];
#pragma unroll
        for (int l = 0; l < 2; ++l)
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) load_hidden(P, 1 + l, ks, warp, lane, raw[l][ks]);
#pragma unroll
        for (int l = 0; l < 2; ++l)
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) split_hidden(raw[l][ks], wh[l][ks], wl[l][ks]);
    }
    {
        uint2 h, o;
        load_last(P, warp, lane, h, o);
        s_w4[0][warp][lane] = h;
        if (kSplit) s_w4[kSplit ? 1 : 0][warp][lane] = o;
    }
    __syncthreads();
    int buf = 0;
    float acc[MT][2][4];
    auto start = [&](int layer) {
#pragma unroll
        for (int m = 0; m < MT; ++m) start_pair(acc[m][0], acc[m][1], &s_bias[layer][16 * warp], t);
    };
    auto pass_on = [&]() {
        buf ^= 1;  // its last readers are a barrier behind
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            uint32_t ah[4], al[4];
            activate_pair(acc[m][0], acc[m][1], ah, al);
            s_a[buf][m][0][warp][lane] = make_uint4(ah[0], ah[1], ah[2], ah[3]);
            if (kSplit) s_a[buf][m][kSplit ? 1 : 0][warp][lane] = make_uint4(al[0], al[1], al[2], al[3]);
        }
        __syncthreads();
    };
    auto fragment = [&](int m, int ks, uint32_t ah[4], uint32_t al[4]) {
        const uint4 h = s_a[buf][m][0][ks][lane], o = kSplit ? s_a[buf][m][kSplit ? 1 : 0][ks][lane] : h;
        ah[0] = h.x, ah[1] = h.y, ah[2] = h.z, ah[3] = h.w;
        al[0] = o.x, al[1] = o.y, al[2] = o.z, al[3] = o.w;
    };
    for (; tile < tiles; tile += gridDim.x * MT) {
        start(0);
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            uint32_t ah[4], al[4];
            standardise_queries(x[m], s_stats, t, ah, al);
            mma_pair<kSplit>(acc[m][0], acc[m][1], ah, al, w1h, w1l);
            load_queries(X, n, tile + gridDim.x * MT + m, g, t, x[m]);
        }
        pass_on();
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            start(l + 1);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    uint32_t ah[4], al[4];
                    fragment(m, ks, ah, al);
                    mma_pair<kSplit>(acc[m][0], acc[m][1], ah, al, wh[l][ks], wl[l][ks]);
                }
            pass_on();
        }
        if (warp < MT) {  // a tile's four outputs per query are one warp's
            float o[3][4] = {{s_b4[2 * t], s_b4[2 * t + 1], s_b4[2 * t], s_b4[2 * t + 1]}, {}, {}};
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                uint32_t ah[4], al[4];
                fragment(warp, ks, ah, al);
                mma_last<kSplit>(o, ah, al, s_w4[0][ks][lane], s_w4[kSplit ? 1 : 0][ks][lane]);
            }
            store_outputs(Y, n, tile + warp, g, t, o, s_stats);
        }
    }
}

}  // namespace
