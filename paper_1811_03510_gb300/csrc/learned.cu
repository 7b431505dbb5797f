// Learned sub-domain proposal: parameters (FP32 masters + Adam state + BF16 copy), training kernels
// (per-sample forward and backward, weight-gradient reduction, Adam), and the tensor-core inference
// kernel.  Softmax cross-entropy over the 64 depth-3 cells; mean over the mini-batch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "learned.cuh"

namespace ccs {

// Parameter offsets in the 9920-vector.
constexpr int kOffW1 = 0, kOffB1 = 1536, kOffW2 = 1600, kOffB2 = 5696, kOffW3 = 5760, kOffB3 = 9856;

// ------------------------------------------------------------------------------------------------
// Training.  k_mlp_grad: one launch computes a block's share of the gradient, forward and backward, for tiles of
// kTile samples that stay in shared memory with the weights; k_mlp_reduce adds the blocks' shares and, in a training
// step, applies Adam and publishes the BF16 copy.
//
// Bound: 27.6 k multiply-adds per sample in FP32 (the masters' precision; forward 9,728, backward 8,192, weight gradients
// 9,728), so FP32 issue, 5.6 us at a batch of 8,192, and the shared-memory bandwidth that feeds it.  A thread owns a 4 x 4
// tile of every product (8 x 4 of the weight gradients, which stay in its registers over all of the block's tiles), fed by
// 16-byte loads: 2 loads per 16 multiply-adds.  Rows are padded to 28 or 68 floats, so that 8 threads that read 8 rows hit
// 32 banks.  32 samples per tile give 256 blocks at a batch of 8,192, two per SM; 64 would leave a sixth of the SMs without
// one.
// Measured on GB300, batch 8,192: a gradient call 25 us (this kernel 24 us, 9.4 T FMA/s or 23% of the lanes' rate, and the
// reduction 5 us, under ncu), before 177 us (one thread per sample with its layers in local memory 95 us, one thread per
// parameter and 512 samples with atomics 92 us).  Error against 64 bits 1.7e-7, before 1.4e-6; no atomics, so the sums are
// the same every time.
// ------------------------------------------------------------------------------------------------
constexpr int kTile = 32, kGradThreads = 128;
constexpr int kXs = 28, kHs = 68;                  // row strides in shared memory (24 and 64 columns)
constexpr int kGradStride = 9984;                  // floats of a block's share: kParams, the loss, padding
constexpr int kGradSmem = (64 * kXs + 128 * kHs + 192 + kTile * (kXs + 4 * kHs)) * 4;

// acc[q][c] += sum_k A[r0 + 8 q][k] W[j0 + 16 c][k], in order of k
template <int K, int AS>
__device__ __forceinline__ void tile_fwd(const float *A, const float *W, int r0, int j0, float (&acc)[4][4])
{
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        float4 a[4], w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = *reinterpret_cast<const float4 *>(A + (r0 + 8 * q) * AS + k);
#pragma unroll
        for (int c = 0; c < 4; ++c) w[c] = *reinterpret_cast<const float4 *>(W + (j0 + 16 * c) * AS + k);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                acc[q][c] = fmaf(w[c].w, a[q].w, fmaf(w[c].z, a[q].z, fmaf(w[c].y, a[q].y, fmaf(w[c].x, a[q].x, acc[q][c]))));
    }
}

// D[r][i] = (H[r][i] > 0) sum_j W[j][i] Z[r][j] for rows r0 + 8 q and columns 4 i0 .. 4 i0 + 3
__device__ __forceinline__ void tile_bwd(const float *Z, const float *W, const float *H, float *D, int r0, int i0)
{
    float acc[4][4] = {};
#pragma unroll 4
    for (int j = 0; j < kHid; j += 4) {
        float4 z[4], w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] = *reinterpret_cast<const float4 *>(Z + (r0 + 8 * q) * kHs + j);
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = *reinterpret_cast<const float4 *>(W + (j + e) * kHs + 4 * i0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float zz[4] = {z[q].x, z[q].y, z[q].z, z[q].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                acc[q][0] = fmaf(w[e].x, zz[e], acc[q][0]);
                acc[q][1] = fmaf(w[e].y, zz[e], acc[q][1]);
                acc[q][2] = fmaf(w[e].z, zz[e], acc[q][2]);
                acc[q][3] = fmaf(w[e].w, zz[e], acc[q][3]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int at = (r0 + 8 * q) * kHs + 4 * i0;
        const float4 h = *reinterpret_cast<const float4 *>(H + at);
        *reinterpret_cast<float4 *>(D + at) = make_float4(h.x > 0.0f ? acc[q][0] : 0.0f, h.y > 0.0f ? acc[q][1] : 0.0f,
                                                          h.z > 0.0f ? acc[q][2] : 0.0f, h.w > 0.0f ? acc[q][3] : 0.0f);
    }
}

// gw[jj][ii] += sum over the tile's samples of D[b][4 jg + jj] A[b][i], i = 4 ig + (0..3), + 32 (NI = 8)
template <int NI, int AS>
__device__ __forceinline__ void tile_wgrad(const float *D, const float *A, int jg, int ig, float (&gw)[4][NI])
{
#pragma unroll 4
    for (int b = 0; b < kTile; ++b) {
        const float4 d4 = *reinterpret_cast<const float4 *>(D + b * kHs + 4 * jg);
        const float d[4] = {d4.x, d4.y, d4.z, d4.w};
        float v[NI];
#pragma unroll
        for (int h = 0; h < NI / 4; ++h) {
            const float4 a = *reinterpret_cast<const float4 *>(A + b * AS + 4 * ig + 32 * h);
            v[4 * h + 0] = a.x;
            v[4 * h + 1] = a.y;
            v[4 * h + 2] = a.z;
            v[4 * h + 3] = a.w;
        }
#pragma unroll
        for (int jj = 0; jj < 4; ++jj)
#pragma unroll
            for (int ii = 0; ii < NI; ++ii) gw[jj][ii] = fmaf(d[jj], v[ii], gw[jj][ii]);
    }
}

__global__ void __launch_bounds__(kGradThreads, 2) k_mlp_grad(const float *__restrict__ params, const float *__restrict__ X,
                                                              const uint8_t *__restrict__ labels, uint32_t B,
                                                              float *__restrict__ shares)
{
    extern __shared__ __align__(16) float sg[];
    float *w1 = sg, *w2 = w1 + 64 * kXs, *w3 = w2 + 64 * kHs, *bias = w3 + 64 * kHs;
    float *x = bias + 192, *h1 = x + kTile * kXs, *h2 = h1 + kTile * kHs, *z3 = h2 + kTile * kHs, *dz = z3 + kTile * kHs;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int q = t; q < 64 * 6; q += kGradThreads)
        *reinterpret_cast<float4 *>(w1 + q / 6 * kXs + q % 6 * 4) = __ldg(reinterpret_cast<const float4 *>(params + kOffW1) + q);
    for (int q = t; q < 64 * 16; q += kGradThreads) {
        const int at = q / 16 * kHs + q % 16 * 4;
        *reinterpret_cast<float4 *>(w2 + at) = __ldg(reinterpret_cast<const float4 *>(params + kOffW2) + q);
        *reinterpret_cast<float4 *>(w3 + at) = __ldg(reinterpret_cast<const float4 *>(params + kOffW3) + q);
    }
    if (t < 64) {
        bias[t] = params[kOffB1 + t];
        bias[64 + t] = params[kOffB2 + t];
        bias[128 + t] = params[kOffB3 + t];
    }
    const int r0 = warp * 2 + (lane >> 4), c0 = lane & 15;   // rows and columns of the thread's 4 x 4 tiles
    const int ig = t & 7, jg = t >> 3;                       // of its 4 x 8 tiles of the gradients of W2 and W3
    const int ig1 = t % 6, jg1 = t / 6;                      // of its 4 x 4 tile of W1's (96 threads)
    float g3[4][8] = {}, g2[4][8] = {}, g1[4][4] = {}, gb1 = 0.0f, gb2 = 0.0f, gb3 = 0.0f, loss = 0.0f;
    const float invB = 1.0f / (float)B;
    const uint32_t tiles = (B + kTile - 1) / kTile;
    for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const uint32_t b0 = tile * kTile;
        const int rows = (int)min((uint32_t)kTile, B - b0);
        for (int q = t; q < kTile * 6; q += kGradThreads) {   // rows past the end are zero, and so are their dz3
            const int r = q / 6;
            *reinterpret_cast<float4 *>(x + r * kXs + q % 6 * 4) =
                r < rows ? make_float4(X[(size_t)(b0 + r) * kFeat + q % 6 * 4], X[(size_t)(b0 + r) * kFeat + q % 6 * 4 + 1],
                                       X[(size_t)(b0 + r) * kFeat + q % 6 * 4 + 2], X[(size_t)(b0 + r) * kFeat + q % 6 * 4 + 3])
                         : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        __syncthreads();
        float acc[4][4];
        auto start = [&](const float *b) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[q][c] = b[c0 + 16 * c];
        };
        auto store = [&](float *o, bool relu) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 4; ++c) o[(r0 + 8 * q) * kHs + c0 + 16 * c] = relu ? fmaxf(acc[q][c], 0.0f) : acc[q][c];
        };
        start(bias);
        tile_fwd<kFeat, kXs>(x, w1, r0, c0, acc);
        store(h1, true);
        __syncthreads();
        start(bias + 64);
        tile_fwd<kHid, kHs>(h1, w2, r0, c0, acc);
        store(h2, true);
        __syncthreads();
        start(bias + 128);
        tile_fwd<kHid, kHs>(h2, w3, r0, c0, acc);
        store(z3, false);
        __syncthreads();
        {   // softmax cross-entropy: four threads per sample, 16 classes each
            const int r = t >> 2;
            float *zr = z3 + r * kHs + (t & 3);
            float mx = -INFINITY;
#pragma unroll
            for (int k = 0; k < 16; ++k) mx = fmaxf(mx, zr[4 * k]);
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const int y = r < rows ? labels[b0 + r] : 0;
            float sum = 0.0f, zy = 0.0f, e[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const float z = zr[4 * k];
                e[k] = expf(z - mx);
                sum += e[k];
                if (4 * k + (t & 3) == y) zy = z;
            }
            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
            zy += __shfl_xor_sync(0xffffffffu, zy, 1);
            zy += __shfl_xor_sync(0xffffffffu, zy, 2);
            if (r < rows && (t & 3) == 0) loss += logf(sum) + mx - zy;
#pragma unroll
            for (int k = 0; k < 16; ++k)
                zr[4 * k] = r < rows ? (e[k] / sum - (4 * k + (t & 3) == y ? 1.0f : 0.0f)) * invB : 0.0f;   // dz3
        }
        __syncthreads();
        tile_wgrad<8, kHs>(z3, h2, jg, ig, g3);
        tile_bwd(z3, w3, h2, dz, r0, c0);
        if (t < 64)
            for (int b = 0; b < kTile; ++b) gb3 += z3[b * kHs + t];
        __syncthreads();
        tile_wgrad<8, kHs>(dz, h1, jg, ig, g2);
        tile_bwd(dz, w2, h1, z3, r0, c0);   // dz1 takes the place of dz3
        if (t < 64)
            for (int b = 0; b < kTile; ++b) gb2 += dz[b * kHs + t];
        __syncthreads();
        if (t < 96) tile_wgrad<4, kXs>(z3, x, jg1, ig1, g1);
        if (t < 64)
            for (int b = 0; b < kTile; ++b) gb1 += z3[b * kHs + t];
        __syncthreads();   // x and z3 are overwritten by the next tile
    }
    float *out = shares + (size_t)blockIdx.x * kGradStride;
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int at = (4 * jg + jj) * kHid + 4 * ig + 32 * h;
            *reinterpret_cast<float4 *>(out + kOffW3 + at) =
                make_float4(g3[jj][4 * h], g3[jj][4 * h + 1], g3[jj][4 * h + 2], g3[jj][4 * h + 3]);
            *reinterpret_cast<float4 *>(out + kOffW2 + at) =
                make_float4(g2[jj][4 * h], g2[jj][4 * h + 1], g2[jj][4 * h + 2], g2[jj][4 * h + 3]);
        }
        if (t < 96)
            *reinterpret_cast<float4 *>(out + kOffW1 + (4 * jg1 + jj) * kFeat + 4 * ig1) =
                make_float4(g1[jj][0], g1[jj][1], g1[jj][2], g1[jj][3]);
    }
    if (t < 64) {
        out[kOffB1 + t] = gb1;
        out[kOffB2 + t] = gb2;
        out[kOffB3 + t] = gb3;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) x[warp] = loss;
    __syncthreads();
    if (t == 0) out[kParams] = x[0] + x[1] + x[2] + x[3];
}

// Where parameter p lives in the BF16 copy (biases stay in FP32).
__device__ __forceinline__ void publish_param(MlpWeights *out, int p, float v)
{
    if (p < kOffB1) out->w1[p / kFeat * kW1Stride + p % kFeat] = __float2bfloat16_rn(v);
    else if (p < kOffW2) out->bias[p - kOffB1] = v;
    else if (p < kOffB2) out->w2[(p - kOffW2) / kHid * kW2Stride + (p - kOffW2) % kHid] = __float2bfloat16_rn(v);
    else if (p < kOffW3) out->bias[kHid + p - kOffB2] = v;
    else if (p < kOffB3) out->w3[(p - kOffW3) / kHid * kW2Stride + (p - kOffW3) % kHid] = __float2bfloat16_rn(v);
    else out->bias[2 * kHid + p - kOffB3] = v;
}

// Adds the blocks' shares (8 threads per parameter, then a tree) and writes the gradient and the mean loss, or (STEP)
// applies Adam to the FP32 masters and writes the BF16 copy used by inference.
struct AdamStep {
    float *params, *m, *v;
    MlpWeights *bf16;
    float lr, b1c, b2c;
};
template <bool STEP>
__global__ void __launch_bounds__(256) k_mlp_reduce(const float *__restrict__ shares, int n, float inv_b,
                                                    float *__restrict__ grad, float *__restrict__ loss, AdamStep s)
{
    __shared__ float part[8][32];
    const int c = threadIdx.x & 31, r = threadIdx.x >> 5, p = blockIdx.x * 32 + c;
    float a = 0.0f;
    if (p <= kParams) {
#pragma unroll 8
        for (int k = r; k < n; k += 8) a += __ldg(shares + (size_t)k * kGradStride + p);
    }
    part[r][c] = a;
    __syncthreads();
    if (r != 0 || p > kParams) return;
    const float g = ((part[0][c] + part[1][c]) + (part[2][c] + part[3][c])) +
                    ((part[4][c] + part[5][c]) + (part[6][c] + part[7][c]));
    if (p == kParams) {
        if (loss) *loss = g * inv_b;
    } else if (STEP) {
        const float mm = 0.9f * s.m[p] + 0.1f * g;
        const float vv = 0.999f * s.v[p] + 0.001f * g * g;
        s.m[p] = mm;
        s.v[p] = vv;
        const float w = s.params[p] - s.lr * (mm / s.b1c) / (sqrtf(vv / s.b2c) + 1e-8f);
        s.params[p] = w;
        publish_param(s.bf16, p, w);
    } else {
        grad[p] = g;
    }
}

__global__ void k_publish_bf16(const float *__restrict__ params, MlpWeights *out)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;   // one thread per output row
    if (n >= kHid) return;
    for (int k = 0; k < kW1Stride; ++k)
        out->w1[n * kW1Stride + k] = __float2bfloat16_rn(k < kFeat ? params[kOffW1 + n * kFeat + k] : 0.0f);
    for (int k = 0; k < kW2Stride; ++k) {
        out->w2[n * kW2Stride + k] = __float2bfloat16_rn(k < kHid ? params[kOffW2 + n * kHid + k] : 0.0f);
        out->w3[n * kW2Stride + k] = __float2bfloat16_rn(k < kHid ? params[kOffW3 + n * kHid + k] : 0.0f);
    }
    out->bias[n] = params[kOffB1 + n];
    out->bias[kHid + n] = params[kOffB2 + n];
    out->bias[2 * kHid + n] = params[kOffB3 + n];
}

// ------------------------------------------------------------------------------------------------
// Inference of n feature rows on tensor cores, one warp per 32 rows.  Bound: 96 bytes of features in and 261 of results
// out per row (HBM), with 19 k multiply-adds, few enough for warp-level MMA.  A layer's accumulators are the next
// layer's A fragments as they stand (the m16n8 result of two column tiles is the m16k16 operand), so activations
// never leave the registers; a warp's two row tiles share every B fragment, four of which one ldmatrix fetches; the
// next rows are loaded while the current ones are multiplied.  Loads and stores are 8 bytes per thread (4 lanes: one
// 32-byte sector of a row) where the arrays are aligned for it.
// Measured on GB300, 450,000 rows: 47 us (161 MB: 3.4 TB/s, half of the measured copy bandwidth), before 97 us (each
// activation through shared memory, scalar loads and stores).
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float2 load2(const float *p, bool wide)
{
    return wide ? __ldcs(reinterpret_cast<const float2 *>(p)) : make_float2(__ldcs(p), __ldcs(p + 1));
}

__global__ void __launch_bounds__(128, 3) k_mlp_infer(const MlpWeights *__restrict__ wts, const float *__restrict__ X,
                                                      uint32_t n, float *logits, uint8_t *cells, float *pmax)
{
    __shared__ __align__(16) MlpWeights W;
    load_weights(W, wts);
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const bool wide_in = (reinterpret_cast<uintptr_t>(X) & 7) == 0, wide_out = (reinterpret_cast<uintptr_t>(logits) & 7) == 0;
    const uint32_t tiles = n / 32 + (n % 32 != 0), step = gridDim.x * (blockDim.x >> 5);
    // the features of rows 32 tile + 16 m + g (+ 8): columns 2 t, 2 t + 8, 2 t + 16 (and the next ones)
    float2 x[2][2][3];
    auto load = [&](uint32_t tile) {
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const size_t row = (size_t)tile * 32 + 16 * m + 8 * r + g;
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    x[m][r][k] = row < n ? load2(X + row * kFeat + 8 * k + 2 * t, wide_in) : make_float2(0.0f, 0.0f);
            }
    };
    uint32_t tile = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (tile < tiles) load(tile);
    for (; tile < tiles; tile += step) {
        uint32_t a1[2][2][4];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                a1[m][0][r] = pack_bf16(x[m][r][0].x, x[m][r][0].y);
                a1[m][0][2 + r] = pack_bf16(x[m][r][1].x, x[m][r][1].y);
                a1[m][1][r] = pack_bf16(x[m][r][2].x, x[m][r][2].y);
                a1[m][1][2 + r] = 0u;
            }
        if (tile + step < tiles) load(tile + step);
        float acc[2][8][4];
        uint32_t a[2][4][4];
        mlp_layer<2, 2>(a1, W.w1, kW1Stride, W.bias, acc, lane);
        relu_fragments<2>(acc, a);
        mlp_layer<2, 4>(a, W.w2, kW2Stride, W.bias + kHid, acc, lane);
        relu_fragments<2>(acc, a);
        mlp_layer<2, 4>(a, W.w3, kW2Stride, W.bias + 2 * kHid, acc, lane);
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const size_t row = (size_t)tile * 32 + 16 * m + 8 * h + g;
                if (logits && row < n) {
                    float *o = logits + row * kCells + 2 * t;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        if (wide_out) {
                            __stcs(reinterpret_cast<float2 *>(o + 8 * j), make_float2(acc[m][j][2 * h], acc[m][j][2 * h + 1]));
                        } else {
                            o[8 * j] = acc[m][j][2 * h];
                            o[8 * j + 1] = acc[m][j][2 * h + 1];
                        }
                    }
                }
                if (!cells && !pmax) continue;
                float best, sum;
                int bidx;
                quad_argmax(acc[m], h, t, best, bidx, sum);
                if (t == 0 && row < n) {
                    if (cells) cells[row] = (uint8_t)bidx;
                    if (pmax) pmax[row] = 1.0f / sum;
                }
            }
    }
}


}  // namespace ccs

using namespace ccs;

struct ccs_proposal {
    float *d_params = nullptr, *d_m = nullptr, *d_v = nullptr;
    MlpWeights *d_bf16 = nullptr;
    float *d_scratch = nullptr;   // the blocks' shares of a gradient
    uint32_t scratch_blocks = 0;
    int num_sms = 0;
    uint64_t step = 0;
};

static void prop_free(ccs_proposal *p)
{
    if (!p) return;
    cudaFree(p->d_params);
    cudaFree(p->d_m);
    cudaFree(p->d_v);
    cudaFree(p->d_bf16);
    cudaFree(p->d_scratch);
    delete p;
}

#define PCK(call)                                                                                 \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess) {                                                                  \
            set_error(std::string(#call) + ": " + cudaGetErrorString(e_));                        \
            return e_ == cudaErrorMemoryAllocation ? CCS_ERR_OOM : CCS_ERR_CUDA;                  \
        }                                                                                         \
    } while (0)

static ccs_status publish(ccs_proposal *p, cudaStream_t s)
{
    k_publish_bf16<<<1, kHid, 0, s>>>(p->d_params, p->d_bf16);
    PCK(cudaGetLastError());
    return CCS_OK;
}

namespace ccs {
const MlpWeights *proposal_weights(const ccs_proposal *p) { return p ? p->d_bf16 : nullptr; }
}

extern "C" {

ccs_status ccs_proposal_set_params(ccs_proposal *p, const float *host_params)
{
    if (!p || !host_params) {
        set_error("ccs_proposal_set_params: NULL argument");
        return CCS_ERR_INVALID_ARG;
    }
    PCK(cudaMemcpy(p->d_params, host_params, sizeof(float) * kParams, cudaMemcpyHostToDevice));
    PCK(cudaMemset(p->d_m, 0, sizeof(float) * kParams));
    PCK(cudaMemset(p->d_v, 0, sizeof(float) * kParams));
    p->step = 0;
    ccs_status st = publish(p, nullptr);
    if (st != CCS_OK) return st;
    PCK(cudaDeviceSynchronize());
    return CCS_OK;
}

ccs_status ccs_proposal_create(ccs_proposal **out, uint64_t seed)
{
    if (!out) {
        set_error("ccs_proposal_create: out is NULL");
        return CCS_ERR_INVALID_ARG;
    }
    *out = nullptr;
    ccs_proposal *p = new (std::nothrow) ccs_proposal();
    if (!p) {
        set_error("host allocation failed");
        return CCS_ERR_OOM;
    }
    cudaError_t e = cudaSuccess;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&p->num_sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, kGradSmem)) != cudaSuccess ||
        (e = cudaMalloc(&p->d_params, sizeof(float) * kParams)) != cudaSuccess ||
        (e = cudaMalloc(&p->d_m, sizeof(float) * kParams)) != cudaSuccess ||
        (e = cudaMalloc(&p->d_v, sizeof(float) * kParams)) != cudaSuccess ||
        (e = cudaMalloc(&p->d_bf16, sizeof(MlpWeights))) != cudaSuccess ||
        (e = cudaMemset(p->d_bf16, 0, sizeof(MlpWeights))) != cudaSuccess) {
        set_error(std::string("ccs_proposal_create: ") + cudaGetErrorString(e));
        prop_free(p);
        return e == cudaErrorMemoryAllocation ? CCS_ERR_OOM : CCS_ERR_CUDA;
    }
    // He-normal initialisation from a seeded PCG32 stream (Box-Muller), zero biases
    std::vector<float> h(kParams, 0.0f);
    uint64_t state = 0, inc = (seed << 1) | 1u;
    auto next = [&]() {
        const uint64_t old = state;
        state = old * 6364136223846793005ull + inc;
        const uint32_t xs = (uint32_t)(((old >> 18u) ^ old) >> 27u), rot = (uint32_t)(old >> 59u);
        return (xs >> rot) | (xs << ((32u - rot) & 31u));
    };
    next();
    state += seed;
    next();
    auto normal = [&]() {
        const double u1 = ((next() >> 8) + 1.0) / 16777217.0, u2 = (next() >> 8) / 16777216.0;
        return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
    };
    const int offs[3] = {kOffW1, kOffW2, kOffW3}, fan_in[3] = {kFeat, kHid, kHid};
    for (int l = 0; l < 3; ++l)
        for (int k = 0; k < kHid * fan_in[l]; ++k)
            h[offs[l] + k] = (float)(normal() * std::sqrt(2.0 / fan_in[l]));
    ccs_status st = ccs_proposal_set_params(p, h.data());
    if (st != CCS_OK) {
        prop_free(p);
        return st;
    }
    *out = p;
    return CCS_OK;
}

ccs_status ccs_proposal_destroy(ccs_proposal *p)
{
    prop_free(p);
    return CCS_OK;
}

ccs_status ccs_proposal_get_params(const ccs_proposal *p, float *host_params)
{
    if (!p || !host_params) {
        set_error("ccs_proposal_get_params: NULL argument");
        return CCS_ERR_INVALID_ARG;
    }
    PCK(cudaMemcpy(host_params, p->d_params, sizeof(float) * kParams, cudaMemcpyDeviceToHost));
    return CCS_OK;
}

static const char kMagic[8] = {'C', 'C', 'S', 'P', 'R', 'O', 'P', '1'};

ccs_status ccs_proposal_save(const ccs_proposal *p, const char *path)
{
    if (!p || !path) {
        set_error("ccs_proposal_save: NULL argument");
        return CCS_ERR_INVALID_ARG;
    }
    std::vector<float> h(kParams);
    ccs_status st = ccs_proposal_get_params(p, h.data());
    if (st != CCS_OK) return st;
    FILE *f = std::fopen(path, "wb");
    if (!f) {
        set_error(std::string("ccs_proposal_save: cannot open ") + path);
        return CCS_ERR_INVALID_ARG;
    }
    const uint32_t shape[4] = {kFeat, kHid, kHid, kCells};
    bool ok = std::fwrite(kMagic, 1, 8, f) == 8 && std::fwrite(shape, 4, 4, f) == 4 &&
              std::fwrite(h.data(), 4, kParams, f) == (size_t)kParams;
    ok = (std::fclose(f) == 0) && ok;
    if (!ok) {
        set_error("ccs_proposal_save: write failed");
        return CCS_ERR_INVALID_ARG;
    }
    return CCS_OK;
}

ccs_status ccs_proposal_load(ccs_proposal **out, const char *path)
{
    if (!out || !path) {
        set_error("ccs_proposal_load: NULL argument");
        return CCS_ERR_INVALID_ARG;
    }
    *out = nullptr;
    FILE *f = std::fopen(path, "rb");
    if (!f) {
        set_error(std::string("ccs_proposal_load: cannot open ") + path);
        return CCS_ERR_INVALID_ARG;
    }
    char magic[8];
    uint32_t shape[4];
    std::vector<float> h(kParams);
    bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, kMagic, 8) == 0 &&
              std::fread(shape, 4, 4, f) == 4 && shape[0] == kFeat && shape[1] == kHid && shape[2] == kHid &&
              shape[3] == kCells && std::fread(h.data(), 4, kParams, f) == (size_t)kParams;
    std::fclose(f);
    if (!ok) {
        set_error("ccs_proposal_load: not a proposal file of this network shape");
        return CCS_ERR_INVALID_ARG;
    }
    ccs_status st = ccs_proposal_create(out, 0);
    if (st != CCS_OK) return st;
    return ccs_proposal_set_params(*out, h.data());
}

// The gradient's shares: two blocks per SM, or fewer for a small batch.
static ccs_status run_grad(ccs_proposal *p, const float *X, const uint8_t *y, uint32_t B, cudaStream_t s, uint32_t &blocks)
{
    blocks = std::min((B + kTile - 1) / kTile, 2u * (uint32_t)p->num_sms);
    if (blocks > p->scratch_blocks) {
        PCK(cudaStreamSynchronize(s));
        cudaFree(p->d_scratch);
        p->d_scratch = nullptr;
        p->scratch_blocks = 0;
        PCK(cudaMalloc(&p->d_scratch, sizeof(float) * kGradStride * (size_t)blocks));
        p->scratch_blocks = blocks;
    }
    k_mlp_grad<<<blocks, kGradThreads, kGradSmem, s>>>(p->d_params, X, y, B, p->d_scratch);
    PCK(cudaGetLastError());
    return CCS_OK;
}

ccs_status ccs_proposal_grad(ccs_proposal *p, const float *features, const uint8_t *labels, uint32_t batch,
                             float *grad, float *loss, void *stream)
{
    if (!p || !features || !labels || batch == 0 || !grad) {
        set_error("ccs_proposal_grad: NULL argument or empty batch");
        return CCS_ERR_INVALID_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    uint32_t blocks = 0;
    ccs_status st = run_grad(p, features, labels, batch, s, blocks);
    if (st != CCS_OK) return st;
    k_mlp_reduce<false><<<(kParams + 32) / 32, 256, 0, s>>>(p->d_scratch, (int)blocks, 1.0f / (float)batch, grad, loss,
                                                            AdamStep{});
    PCK(cudaGetLastError());
    return CCS_OK;
}

ccs_status ccs_proposal_train_step(ccs_proposal *p, const float *features, const uint8_t *labels, uint32_t batch,
                                   float lr, float *loss, void *stream)
{
    if (!p || !features || !labels || batch == 0 || !(lr > 0.0f)) {
        set_error("ccs_proposal_train_step: NULL argument, empty batch or lr <= 0");
        return CCS_ERR_INVALID_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    uint32_t blocks = 0;
    ccs_status st = run_grad(p, features, labels, batch, s, blocks);
    if (st != CCS_OK) return st;
    p->step += 1;
    const float b1c = 1.0f - std::pow(0.9f, (float)p->step), b2c = 1.0f - std::pow(0.999f, (float)p->step);
    k_mlp_reduce<true><<<(kParams + 32) / 32, 256, 0, s>>>(p->d_scratch, (int)blocks, 1.0f / (float)batch, nullptr, loss,
                                                           AdamStep{p->d_params, p->d_m, p->d_v, p->d_bf16, lr, b1c, b2c});
    PCK(cudaGetLastError());
    return CCS_OK;
}

ccs_status ccs_proposal_infer(const ccs_proposal *p, const float *features, uint32_t n, float *logits, uint8_t *cells,
                              float *pmax, void *stream)
{
    if (!p || !features) {
        set_error("ccs_proposal_infer: NULL argument");
        return CCS_ERR_INVALID_ARG;
    }
    if (n == 0) return CCS_OK;
    const uint32_t tiles = n / 32 + (n % 32 != 0);
    const uint32_t blocks = std::min((tiles + 3) / 4, 3u * (uint32_t)p->num_sms);
    k_mlp_infer<<<blocks, 128, 0, (cudaStream_t)stream>>>(p->d_bf16, features, n, logits, cells, pmax);
    PCK(cudaGetLastError());
    return CCS_OK;
}

}  // extern "C"
