// okr_mlp.cu -- the learned candidate scorer: a three-hidden-layer perceptron
// (128 units, ReLU) that predicts a candidate's normalised score change from
// local feeder features, with hand-written forward, backward and Adam kernels.
//
// Numerics: weights are held in FP32 (the Adam master copy) and used as
// bfloat16 copies in every product; products are accumulated in FP32 in a
// fixed order: a unit's sum runs over its inputs in increasing order (fused
// multiply-adds, from the bias), a weight's gradient over the samples of a
// segment in increasing order, then over the segments.  Every kernel below
// keeps that order whatever its tiling, so a result does not depend on which
// of them computed it, and training is reproducible.
//
// Parameter vector (FP32), in this order: W1 (F x H, row-major), b1 (H),
// W2 (H x H), b2, W3 (H x H), b3, w4 (H), b4 (1).
//
// What bounds it: FP32 multiply-adds (71 TFLOP/s on one GB300).  The weights
// stay in shared memory as FP32 and every thread holds a tile of sums in
// registers, so that one shared load feeds several multiply-adds.  (One sum per
// thread, two shared loads and a bfloat16 conversion per multiply-add, ran at
// 9 TFLOP/s: 300,007 samples forward in 2.28 ms; weight gradients with one
// global-memory chain per output 234 us each, four per training step.)
#include "okr_internal.cuh"
#include "okr_kernels.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace okr {

namespace {

constexpr int kH = kMlpHidden;
constexpr int kTile = 32;                    // samples per tile of a small batch
constexpr int kSeg = 2048;                   // samples per partial sum of a weight gradient

struct Off {
    int w1, b1, w2, b2, w3, b3, w4, b4, total;
};

__host__ __device__ inline Off offsets(int F) {
    Off o;
    o.w1 = 0;
    o.b1 = o.w1 + F * kH;
    o.w2 = o.b1 + kH;
    o.b2 = o.w2 + kH * kH;
    o.w3 = o.b2 + kH;
    o.b3 = o.w3 + kH * kH;
    o.w4 = o.b3 + kH;
    o.b4 = o.w4 + kH;
    o.total = o.b4 + 1;
    return o;
}

}  // namespace

int mlp_param_count(int F) { return offsets(F).total; }

// FP32 master weights -> bfloat16 copies used by the products.
__global__ void k_mlp_to_bf16(const float *theta, int F, __nv_bfloat16 *w1, __nv_bfloat16 *w2, __nv_bfloat16 *w3,
                              __nv_bfloat16 *w4) {
    const Off o = offsets(F);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < kH * kH; e += gridDim.x * blockDim.x) {
        w2[e] = __float2bfloat16_rn(theta[o.w2 + e]);
        w3[e] = __float2bfloat16_rn(theta[o.w3 + e]);
        if (e < F * kH) w1[e] = __float2bfloat16_rn(theta[o.w1 + e]);
        if (e < kH) w4[e] = __float2bfloat16_rn(theta[o.w4 + e]);
    }
}

// ---------------------------------------------------------------- forward, backward
namespace {

constexpr int kPitch = kH + 1;              // of a weight row in shared memory: rows and columns both read without conflicts
constexpr int kTilePitch = kTile + 4;       // of a transposed activation row (16-byte rows)

// A 128 x 128 weight matrix (bfloat16 in device memory) as FP32 in shared
// memory, by 256 threads.  A warp takes 64 consecutive weights, two a lane, so
// that its stores meet in pairs at most, and every load is in flight at once
// (eight at a time took a quarter of a training step's tile kernel).
__device__ __forceinline__ void load_square(float *dst, int pitch, const __nv_bfloat16 *__restrict__ w) {
    constexpr int kPer = kH * kH / 2 / 256;
    unsigned u[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) u[i] = __ldg(reinterpret_cast<const unsigned *>(w) + threadIdx.x + 256 * i);
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int e = threadIdx.x + 256 * i;
        float *d = dst + (e / (kH / 2)) * pitch + (e % (kH / 2)) * 2;
        d[0] = __uint_as_float(u[i] << 16);
        d[1] = __uint_as_float(u[i] & 0xffff0000u);
    }
}
// The first layer's F rows.
__device__ __forceinline__ void load_rows(float *dst, int pitch, const __nv_bfloat16 *__restrict__ w, int rows) {
    for (int e = threadIdx.x; e < rows * kH; e += 256) dst[(e / kH) * pitch + e % kH] = __bfloat162float(w[e]);
}

// One layer on a tile of 32 samples: acc[i][c] += sum over k < K of
// in[k][4 ty + i] * W(k, tx + 32 c), k increasing; T: W is read transposed.  The
// next k's values are loaded before this k's multiply-adds (two warps per
// scheduler hide little); past the last k they are read and not used.
template <bool T>
__device__ __forceinline__ void tile_layer(const float *__restrict__ in, const float *__restrict__ W, int K, int tx,
                                           int ty, float (&acc)[4][4]) {
    float4 a = *reinterpret_cast<const float4 *>(in + 4 * ty);
    float w[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) w[c] = T ? W[(tx + 32 * c) * kPitch] : W[tx + 32 * c];
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float av[4] = {a.x, a.y, a.z, a.w};
        float u[4];
        a = *reinterpret_cast<const float4 *>(in + (k + 1) * kTilePitch + 4 * ty);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            u[c] = w[c];
            w[c] = T ? W[(tx + 32 * c) * kPitch + k + 1] : W[(k + 1) * kPitch + tx + 32 * c];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[i][c] = fmaf(av[i], u[c], acc[i][c]);
    }
}

// The tile's sums as the next layer's input, transposed.
__device__ __forceinline__ void tile_store(float *out, int tx, int ty, const float (&v)[4][4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
        *reinterpret_cast<float4 *>(out + (tx + 32 * c) * kTilePitch + 4 * ty) =
            make_float4(v[0][c], v[1][c], v[2][c], v[3][c]);
}

}  // namespace

// Tiles of 32 samples, 256 threads: warp ty takes samples 4 ty .. 4 ty + 3, lane
// tx units tx, tx + 32, tx + 64, tx + 96 (16 sums a thread; five shared loads,
// 32 bytes a thread, feed 16 multiply-adds: the loads' 128 bytes a cycle and SM
// bound it).  For few samples: 4,096 of a training step are 128 CTAs, 25 us
// forward and back (195 us in two kernels before).  TRAIN: the whole pass forward and back through
// the activations,
//   dy = scale (y - t); d3 = dy w4 [h3 > 0]; d2 = (d3 W3^T) [h2 > 0];
//   d1 = (d2 W2^T) [h1 > 0],
// with h1, h2, h3, d1, d2, d3 [N][H] and dy [N] written for the weight
// gradients; otherwise y alone.
template <bool TRAIN>
__global__ void __launch_bounds__(256, 1) k_mlp_tile(const float *__restrict__ x, const float *__restrict__ t, int N,
                                                     int F, float scale, const float *__restrict__ theta,
                                                     const __nv_bfloat16 *__restrict__ w1,
                                                     const __nv_bfloat16 *__restrict__ w2,
                                                     const __nv_bfloat16 *__restrict__ w3,
                                                     const __nv_bfloat16 *__restrict__ w4, float *h1, float *h2,
                                                     float *h3, float *d1, float *d2, float *d3, float *y, float *dy) {
    extern __shared__ __align__(16) float tile_sm[];
    float *W2 = tile_sm, *W3 = W2 + kH * kPitch, *W1 = W3 + kH * kPitch;
    float *A = W1 + kMlpMaxF * kPitch, *B = A + kH * kTilePitch, *X = B + kH * kTilePitch;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const Off o = offsets(F);
    load_square(W2, kPitch, w2);
    load_square(W3, kPitch, w3);
    load_rows(W1, kPitch, w1, F);
    float b1[4], b2[4], b3[4], u4[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int j = tx + 32 * c;
        b1[c] = theta[o.b1 + j];
        b2[c] = theta[o.b2 + j];
        b3[c] = theta[o.b3 + j];
        u4[c] = __bfloat162float(w4[j]);
    }
    const float b4 = theta[o.b4];
    for (int base = blockIdx.x * kTile; base < N; base += gridDim.x * kTile) {
        const int S = min(kTile, N - base);
        for (int e = threadIdx.x; e < kTile * F; e += 256) {
            const int s = e / F, k = e % F;
            X[k * kTilePitch + s] = s < S ? x[(size_t)(base + s) * F + k] : 0.0f;
        }
        __syncthreads();
        float v1[4][4], v2[4][4], v3[4][4];
        auto set = [&](float (&v)[4][4], const float *b) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) v[i][c] = b ? b[c] : 0.0f;
        };
        auto relu = [&](float (&v)[4][4]) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) v[i][c] = fmaxf(v[i][c], 0.0f);
        };
        auto keep = [&](float *g, const float (&v)[4][4]) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int s = 4 * ty + i;
                if (s >= S) continue;
#pragma unroll
                for (int c = 0; c < 4; ++c) g[(size_t)(base + s) * kH + tx + 32 * c] = v[i][c];
            }
        };
        set(v1, b1);
        tile_layer<false>(X, W1, F, tx, ty, v1);
        relu(v1);
        tile_store(A, tx, ty, v1);
        __syncthreads();
        set(v2, b2);
        tile_layer<false>(A, W2, kH, tx, ty, v2);
        relu(v2);
        tile_store(B, tx, ty, v2);
        __syncthreads();
        set(v3, b3);
        tile_layer<false>(B, W3, kH, tx, ty, v3);
        relu(v3);
        // y = b4 + sum_j h3_j w4_j: lane sums of four, then the warp's tree
        float yv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float acc = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(v3[i][0], u4[0]), __fmul_rn(v3[i][1], u4[1])),
                                            __fmul_rn(v3[i][2], u4[2])),
                                  __fmul_rn(v3[i][3], u4[3]));
            for (int q = 16; q > 0; q >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, q);
            yv[i] = acc + b4;
            const int s = 4 * ty + i;
            if (tx == 0 && s < S) y[base + s] = yv[i];
        }
        if (TRAIN) {
            keep(h1, v1);
            keep(h2, v2);
            keep(h3, v3);
            // (A holds h1, no longer read; B holds h2, read until the barrier below)
            float g[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int s = 4 * ty + i;
                const float dv = s < S ? scale * (yv[i] - t[base + s]) : 0.0f;
                if (tx == 0 && s < S) dy[base + s] = dv;
#pragma unroll
                for (int c = 0; c < 4; ++c) g[i][c] = (s < S && v3[i][c] > 0.0f) ? dv * u4[c] : 0.0f;
            }
            keep(d3, g);
            tile_store(A, tx, ty, g);
            __syncthreads();
            set(g, nullptr);
            tile_layer<true>(A, W3, kH, tx, ty, g);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) g[i][c] = (4 * ty + i < S && v2[i][c] > 0.0f) ? g[i][c] : 0.0f;
            keep(d2, g);
            tile_store(B, tx, ty, g);
            __syncthreads();
            set(g, nullptr);
            tile_layer<true>(B, W2, kH, tx, ty, g);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) g[i][c] = v1[i][c] > 0.0f ? g[i][c] : 0.0f;
            keep(d1, g);
        }
        __syncthreads();                    // (the next tile's features and layer 1 overwrite X and A)
    }
}

// Forward pass of many samples: tiles of 128, 256 threads, 8 x 8 sums a thread
// (samples 8 ty .. 8 ty + 7; units 4 tx .. 4 tx + 3 and 64 more), so that four
// 16-byte shared loads feed 64 multiply-adds; one CTA per SM.  A layer's output
// replaces its input in place.
constexpr int kBig = 128, kBigPitch = kBig + 4;
__global__ void __launch_bounds__(256, 1) k_mlp_forward(const float *__restrict__ x, int N, int F,
                                                        const float *__restrict__ theta,
                                                        const __nv_bfloat16 *__restrict__ w1,
                                                        const __nv_bfloat16 *__restrict__ w2,
                                                        const __nv_bfloat16 *__restrict__ w3,
                                                        const __nv_bfloat16 *__restrict__ w4, float *__restrict__ y) {
    extern __shared__ __align__(16) float big_sm[];
    float *W2 = big_sm, *W3 = W2 + kH * kH, *W1 = W3 + kH * kH;
    float *A = W1 + kMlpMaxF * kH, *X = A + kH * kBigPitch;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Off o = offsets(F);
    load_square(W2, kH, w2);
    load_square(W3, kH, w3);
    load_rows(W1, kH, w1, F);
    const float b4 = theta[o.b4];
    auto unit = [&](int c) { return 4 * tx + (c & 3) + 64 * (c >> 2); };
    float acc[8][8];
    auto layer = [&](const float *in, const float *W, int K, int boff) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float b = __ldg(theta + boff + unit(c));
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i][c] = b;
        }
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            float a[8], w[8];
            *reinterpret_cast<float4 *>(a) = *reinterpret_cast<const float4 *>(in + k * kBigPitch + 8 * ty);
            *reinterpret_cast<float4 *>(a + 4) = *reinterpret_cast<const float4 *>(in + k * kBigPitch + 8 * ty + 4);
            *reinterpret_cast<float4 *>(w) = *reinterpret_cast<const float4 *>(W + k * kH + 4 * tx);
            *reinterpret_cast<float4 *>(w + 4) = *reinterpret_cast<const float4 *>(W + k * kH + 4 * tx + 64);
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[i][c] = fmaf(a[i], w[c], acc[i][c]);
        }
    };
    auto store = [&]() {
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float4 *>(A + unit(c) * kBigPitch + 8 * ty + 4 * h) =
                    make_float4(fmaxf(acc[4 * h][c], 0.0f), fmaxf(acc[4 * h + 1][c], 0.0f),
                                fmaxf(acc[4 * h + 2][c], 0.0f), fmaxf(acc[4 * h + 3][c], 0.0f));
    };
    // the next tile's features are in flight while this tile is computed (x may
    // lie in host memory, read across the chip-to-chip link)
    float xr[kBig * kMlpMaxF / 256];
    auto load_x = [&](long long base) {
#pragma unroll
        for (int i = 0; i < kBig * kMlpMaxF / 256; ++i) {
            const int e = threadIdx.x + 256 * i;
            xr[i] = (e < kBig * F && base * F + e < (long long)N * F) ? __ldg(x + base * F + e) : 0.0f;
        }
    };
    load_x((long long)blockIdx.x * kBig);
    for (long long base = (long long)blockIdx.x * kBig; base < N; base += (long long)gridDim.x * kBig) {
        const int S = (int)min((long long)kBig, N - base);
#pragma unroll
        for (int i = 0; i < kBig * kMlpMaxF / 256; ++i) {
            const int e = threadIdx.x + 256 * i;
            if (e < kBig * F) X[(e % F) * kBigPitch + e / F] = xr[i];
        }
        __syncthreads();
        load_x(base + (long long)gridDim.x * kBig);
        layer(X, W1, F, o.b1);
        store();
        __syncthreads();
        layer(A, W2, kH, o.b2);
        __syncthreads();
        store();
        __syncthreads();
        layer(A, W3, kH, o.b3);
        __syncthreads();
        // the output layer's products, unit by unit (an odd pitch, so that the sums below read without conflicts)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float u = __bfloat162float(w4[unit(c)]);
#pragma unroll
            for (int i = 0; i < 8; ++i) A[unit(c) * (kBig + 1) + 8 * ty + i] = __fmul_rn(fmaxf(acc[i][c], 0.0f), u);
        }
        __syncthreads();
        // y = b4 + sum_j h3_j w4_j: lane sums of four, then the warp's tree
        for (int s = warp; s < S; s += 8) {
            float v = __fadd_rn(__fadd_rn(__fadd_rn(A[lane * (kBig + 1) + s], A[(lane + 32) * (kBig + 1) + s]),
                                          A[(lane + 64) * (kBig + 1) + s]),
                                A[(lane + 96) * (kBig + 1) + s]);
            for (int q = 16; q > 0; q >>= 1) v += __shfl_xor_sync(0xffffffffu, v, q);
            if (lane == 0) y[base + s] = v + b4;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- weight gradients
namespace {

constexpr int kStage = 64, kStages = 3;     // samples per stage of the pipeline, stages in shared memory

__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool in) {      // (not in: zeros)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(in ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// One product of the weight gradients: G[k][c] = sum over n of A[n][k] D[n][c]
// (k < K, c < C) and, as row K, the bias's sum of D[n][c].  A has rows of K
// floats, D of C; K = 128 or the features, C = 128 or 1.
struct WJob {
    const float *A, *D;
    int K, C;
    int off;                    // of G in the parameter vector
    int kt, ct;                 // its tiles along k and c
};

}  // namespace

// Partial gradients over one segment of kSeg samples (blockIdx.y), in parameter
// order: part[seg][P].  The samples are added in increasing order, one chain
// per output, so the parallelism is in the outputs: 64 threads hold a tile of
// 32 x 16 (2 x 4 each: one 8-byte and one 16-byte shared load feed eight
// multiply-adds; 2 x 2 outputs were bound by the shared loads, 77 us against 33
// for 4,096 samples, of which the chains of 2,048 samples at 12 instructions
// each are 12 us and the staging and waits the rest), the segment's rows of A and D
// pass through a three-stage cp.async pipeline.  The last CTA of a segment sums the
// squared errors into loss[seg].
constexpr int kWThreads = 64, kWK = 32, kWC = 16;
__global__ void __launch_bounds__(kWThreads) k_mlp_wgrad(WJob j0, WJob j1, WJob j2, WJob j3, const float *__restrict__ y,
                                                         const float *__restrict__ t, int N, int P, float *part,
                                                         float *loss) {
    __shared__ __align__(16) float sA[kStages][kStage][kWK], sD[kStages][kStage][kWC];
    __shared__ float red[8];
    const int tid = threadIdx.x, seg = blockIdx.y;
    const int n0 = seg * kSeg, n1 = min(N, n0 + kSeg);
    // this CTA's job
    const float *A, *D;
    int K, C, off, ct, tile = blockIdx.x;
    {
        int left = tile;
        auto is = [&](const WJob &j) {
            if (left < 0) return;
            if (left < j.kt * j.ct) {
                A = j.A; D = j.D; K = j.K; C = j.C; off = j.off; ct = j.ct; tile = left;
                left = -1;
            } else {
                left -= j.kt * j.ct;
            }
        };
        A = D = nullptr;
        K = C = off = 0;
        ct = 1;
        is(j0);
        is(j1);
        is(j2);
        is(j3);
    }
    if (!A) {                               // squared errors: the order of eight warps of 32 strided samples
        float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
#pragma unroll
            for (int i = 0; i < kSeg / 256; ++i) {
                const int n = n0 + tid + 64 * h + 256 * i;
                if (n < n1) {
                    const float d = y[n] - t[n];
                    a[h] = fmaf(d, d, a[h]);
                }
            }
        }
        for (int h = 0; h < 4; ++h) {
            for (int q = 16; q > 0; q >>= 1) a[h] += __shfl_xor_sync(0xffffffffu, a[h], q);
            if ((tid & 31) == 0) red[(tid >> 5) + 2 * h] = a[h];
        }
        __syncthreads();
        if (tid == 0) {
            float s = 0.0f;
            for (int w = 0; w < 8; ++w) s += red[w];
            loss[seg] = s;
        }
        return;
    }
    const int k0 = (tile / ct) * kWK, c0 = (tile % ct) * kWC;
    const bool wideA = K == kH, wideD = C == kH;
    // the columns that the narrow operands (the features, dy) leave are zero in every stage
    if (!wideA)
        for (int e = tid; e < kStages * kStage * kWK; e += kWThreads) (&sA[0][0][0])[e] = 0.0f;
    if (!wideD)
        for (int e = tid; e < kStages * kStage * kWC; e += kWThreads) (&sD[0][0][0])[e] = 0.0f;
    __syncthreads();
    // a narrow A is read as consecutive floats: where this thread's go in a stage
    int xo[kMlpMaxF];
#pragma unroll
    for (int i = 0; i < kMlpMaxF; ++i) {
        const int e = tid + kWThreads * i;
        xo[i] = wideA ? 0 : (e / K) * kWK + e % K;
    }
    const float *Aw = A + (size_t)(tid >> 3) * kH + k0 + 4 * (tid & 7), *Dw = D + (size_t)(tid >> 2) * kH + c0 + 4 * (tid & 3);
    auto stage = [&](int st) {
        const int m0 = n0 + st * kStage, b = st % kStages;
        if (m0 < n1) {
            if (wideA) {
#pragma unroll
                for (int i = 0; i < kStage / 8; ++i) {      // 8 samples of 8 x 4 columns
                    const int m = m0 + 8 * i + (tid >> 3);
                    cp_async16(&sA[b][8 * i + (tid >> 3)][4 * (tid & 7)], m < n1 ? Aw + (size_t)(m0 + 8 * i) * kH : A, m < n1);
                }
            } else {
                static_assert(kStage == kWThreads, "K floats a thread and stage");
                const int in = min(kStage, n1 - m0) * K;
#pragma unroll
                for (int i = 0; i < kMlpMaxF; ++i) {
                    const int e = tid + kWThreads * i;
                    if (i < K && e < in) cp_async4(&sA[b][0][0] + xo[i], A + (size_t)m0 * K + e);
                }
            }
            if (wideD) {
#pragma unroll
                for (int i = 0; i < kStage / 16; ++i) {     // 16 samples of 4 x 4 columns
                    const int m = m0 + 16 * i + (tid >> 2);
                    cp_async16(&sD[b][16 * i + (tid >> 2)][4 * (tid & 3)], m < n1 ? Dw + (size_t)(m0 + 16 * i) * kH : D, m < n1);
                }
            } else if (tid < kStage && m0 + tid < n1) {
                cp_async4(&sD[b][tid][0], D + m0 + tid);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int kx = tid & 15, cy = tid >> 4;
    float acc[2][4], bias[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[0][c] = acc[1][c] = bias[c] = 0.0f;
    const int ns = (n1 - n0 + kStage - 1) / kStage;
    for (int st = 0; st < kStages - 1; ++st) stage(st);
    const bool biased = k0 == 0;            // the bias with the first row tile
    auto pass = [&](auto with_bias) {
        for (int st = 0; st < ns; ++st) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
            __syncthreads();
            stage(st + kStages - 1);            // (into the buffer every thread has left: the barrier above)
            const int b = st % kStages, m = min(kStage, n1 - n0 - st * kStage);
            // the next four samples' values are loaded before these four's multiply-adds
            // (with a warp per scheduler nothing else hides the shared loads)
            constexpr int U = 4;
            float2 a[2][U];
            float4 d[2][U];
            auto fetch = [&](int h, int i, int s) {
                a[h][i] = *reinterpret_cast<const float2 *>(&sA[b][s][2 * kx]);
                d[h][i] = *reinterpret_cast<const float4 *>(&sD[b][s][4 * cy]);
            };
            auto add = [&](int h, int j) {
                const float dv[4] = {d[h][j].x, d[h][j].y, d[h][j].z, d[h][j].w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    acc[0][c] = fmaf(a[h][j].x, dv[c], acc[0][c]);
                    acc[1][c] = fmaf(a[h][j].y, dv[c], acc[1][c]);
                }
                if (decltype(with_bias)::value) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) bias[c] += dv[c];
                }
            };
            if (m == kStage) {
#pragma unroll
                for (int j = 0; j < U; ++j) fetch(0, j, j);
#pragma unroll
                for (int s = 0; s < kStage; s += 2 * U) {
#pragma unroll
                    for (int j = 0; j < U; ++j) fetch(1, j, s + U + j);
#pragma unroll
                    for (int j = 0; j < U; ++j) add(0, j);
#pragma unroll
                    for (int j = 0; j < U; ++j)
                        if (s + 2 * U < kStage) fetch(0, j, s + 2 * U + j);
#pragma unroll
                    for (int j = 0; j < U; ++j) add(1, j);
                }
            } else {
                for (int s = 0; s < m; ++s) {
                    fetch(0, 0, s);
                    add(0, 0);
                }
            }
        }
    };
    if (biased) pass(std::true_type());
    else pass(std::false_type());
    float *g = part + (size_t)seg * P + off;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int cc = c0 + 4 * cy + c;
        if (cc >= C) continue;
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (k0 + 2 * kx + i < K) g[(size_t)(k0 + 2 * kx + i) * C + cc] = acc[i][c];
        if (biased && kx == 0) g[(size_t)K * C + cc] = bias[c];
    }
}

// grad[e] = sum over segments (in order) of part[seg][e]; with lr > 0 then Adam
// (bias-corrected) on the FP32 master weights and the bfloat16 copies.
__global__ void __launch_bounds__(256) k_mlp_update(const float *__restrict__ part, int nseg, int P, int F, float *grad,
                                                    float *theta, float *m, float *v, float lr, float beta1, float beta2,
                                                    float eps, float c1, float c2, __nv_bfloat16 *w1, __nv_bfloat16 *w2,
                                                    __nv_bfloat16 *w3, __nv_bfloat16 *w4) {
    const int e = blockIdx.x * 256 + threadIdx.x;
    if (e >= P) return;
    float ge = 0.0f;
#pragma unroll 8
    for (int s = 0; s < nseg; ++s) ge += part[(size_t)s * P + e];
    grad[e] = ge;
    if (!(lr > 0.0f)) return;
    const float me = beta1 * m[e] + (1.0f - beta1) * ge;
    const float ve = beta2 * v[e] + (1.0f - beta2) * ge * ge;
    m[e] = me;
    v[e] = ve;
    const float th = theta[e] - lr * (me / c1) / (sqrtf(ve / c2) + eps);
    theta[e] = th;
    const Off o = offsets(F);
    const __nv_bfloat16 h = __float2bfloat16_rn(th);
    if (e < o.b1) w1[e - o.w1] = h;
    else if (e >= o.w2 && e < o.b2) w2[e - o.w2] = h;
    else if (e >= o.w3 && e < o.b3) w3[e - o.w3] = h;
    else if (e >= o.w4 && e < o.b4) w4[e - o.w4] = h;
}

// ---------------------------------------------------------------- host launches
namespace {

constexpr size_t kTileSmem = sizeof(float) * ((2 * kH + kMlpMaxF) * kPitch + (2 * kH + kMlpMaxF + 1) * kTilePitch);
constexpr size_t kBigSmem = sizeof(float) * ((2 * kH + kMlpMaxF) * kH + (kH + kMlpMaxF) * kBigPitch);

}  // namespace

int mlp_segments(int N) { return (N + kSeg - 1) / kSeg; }

cudaError_t mlp_sync_bf16(const MlpBufs &b, cudaStream_t st) {
    k_mlp_to_bf16<<<64, 256, 0, st>>>(b.theta, b.F, b.w1, b.w2, b.w3, b.w4);
    return cudaGetLastError();
}

// y of N samples.  Tiles of 128 once every SM has one (from num_sms x 128
// samples on; 300,007 samples: 0.48 ms, 43 TFLOP/s, bound by the shared loads'
// 128 bytes a cycle as much as by the multiply-adds), tiles of 32 below.
cudaError_t mlp_forward(const MlpBufs &b, const float *x, int N, float *y, int num_sms, cudaStream_t st) {
    if (N >= num_sms * kBig) {
        const cudaError_t e = cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBigSmem);
        if (e != cudaSuccess) return e;
        k_mlp_forward<<<num_sms, 256, kBigSmem, st>>>(x, N, b.F, b.theta, b.w1, b.w2, b.w3, b.w4, y);
    } else {
        const cudaError_t e = cudaFuncSetAttribute(k_mlp_tile<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmem);
        if (e != cudaSuccess) return e;
        k_mlp_tile<false><<<std::min((N + kTile - 1) / kTile, num_sms), 256, kTileSmem, st>>>(
            x, nullptr, N, b.F, 0.0f, b.theta, b.w1, b.w2, b.w3, b.w4, nullptr, nullptr, nullptr, nullptr, nullptr,
            nullptr, y, nullptr);
    }
    return cudaGetLastError();
}

// Gradient of the mean squared error at the current weights into b.grad (uses
// the work buffers, which must hold N samples) and the squared errors of each
// segment into loss[mlp_segments(N)]; with lr > 0 then the Adam step `step`.
cudaError_t mlp_gradient(const MlpBufs &b, const MlpWork &w, const float *x, const float *t, int N, float *loss, float lr,
                         int step, int num_sms, cudaStream_t st) {
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_tile<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmem);
    if (e != cudaSuccess) return e;
    k_mlp_tile<true><<<std::min((N + kTile - 1) / kTile, num_sms), 256, kTileSmem, st>>>(
        x, t, N, b.F, 2.0f / (float)N, b.theta, b.w1, b.w2, b.w3, b.w4, w.h1, w.h2, w.h3, w.d1, w.d2, w.d3, w.y, w.dy);
    const Off o = offsets(b.F);
    const int nseg = mlp_segments(N), P = o.total;
    auto job = [](const float *A, int K, const float *D, int C, int off) {
        WJob j;
        j.A = A;
        j.D = D;
        j.K = K;
        j.C = C;
        j.off = off;                        // (weights and bias are adjacent in the parameter vector: W then b)
        j.kt = (K + kWK - 1) / kWK;
        j.ct = (C + kWC - 1) / kWC;
        return j;
    };
    const WJob j0 = job(w.h1, kH, w.d2, kH, o.w2), j1 = job(w.h2, kH, w.d3, kH, o.w3), j2 = job(x, b.F, w.d1, kH, o.w1),
               j3 = job(w.h3, kH, w.dy, 1, o.w4);
    const int tiles = j0.kt * j0.ct + j1.kt * j1.ct + j2.kt * j2.ct + j3.kt * j3.ct + 1;
    k_mlp_wgrad<<<dim3((unsigned)tiles, (unsigned)nseg), kWThreads, 0, st>>>(j0, j1, j2, j3, w.y, t, N, P, w.part, loss);
    const float beta1 = 0.9f, beta2 = 0.999f;
    const float c1 = lr > 0.0f ? 1.0f - powf(beta1, (float)step) : 1.0f, c2 = lr > 0.0f ? 1.0f - powf(beta2, (float)step) : 1.0f;
    k_mlp_update<<<(P + 255) / 256, 256, 0, st>>>(w.part, nseg, P, b.F, b.grad, b.theta, b.m, b.v, lr, beta1, beta2, 1e-8f,
                                                  c1, c2, b.w1, b.w2, b.w3, b.w4);
    return cudaGetLastError();
}

}  // namespace okr
