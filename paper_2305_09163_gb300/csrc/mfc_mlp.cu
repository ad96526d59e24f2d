// Learned WENO weights: training kernels and their C ABI (include/mfc.h).
//
//   mfc_mlp_forward  weights omega for a batch of normalised stencils
//   mfc_mlp_grad_mma loss and gradient of a batch (forward + backpropagation)
//                    on warp-level mma.sync; mfc_mlp_grad (mfc_mlp_tc.cu) is
//                    the same on the fifth-generation tensor cores
//   mfc_mlp_adam     Adam update of the parameter blob
//   mfc_harvest      training samples from a fine primitive field: coarse
//                    (2x restricted) stencils, WENO5 candidates, the fine-grid
//                    face value as target, the WENO5-JS value and a sensor flag
//
// The paper has no learned part; the network replaces the WENO5-JS nonlinear
// weights of Sec. 3.2.  Every matrix product of the forward and backward pass
// (including the batch reductions that form the weight gradients) runs on the
// tensor cores as mma.sync with BF16 operands and FP32 accumulation.
#include <cmath>
#include <cstdint>

#include "../../include/mfc.h"
#include "mfc_launch.cuh"
#include "mfc_mlp.cuh"

using namespace mfc;

namespace {

constexpr int kGradWarps = 4;
constexpr int kGradBlocks = MFC_MLP_GRAD_BLOCKS;
constexpr int kGradStride = kMlpParams + 1;  // parameters + loss
static_assert(kMlpParams == MFC_MLP_PARAMS, "parameter count");
static_assert((long long)kGradBlocks * kGradWarps * kGradStride == MFC_MLP_WORK_FLOATS, "workspace size");

__device__ __constant__ float kIdeal[3] = {0.1f, 0.6f, 0.3f};

// A fragment (m16n8k8) of the inputs of rows row0+g and row0+g+8.
__device__ __forceinline__ void load_inputs(const float* __restrict__ x, long long B, long long row0, int g, int t,
                                            uint32_t* a) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const long long r = row0 + g + 8 * h;
        const int k = 2 * t;
        float v0 = 0.f, v1 = 0.f;
        if (r < B) {
            if (k < kMlpIn) v0 = x[r * kMlpIn + k];
            if (k + 1 < kMlpIn) v1 = x[r * kMlpIn + k + 1];
        }
        a[h] = pack_bf16(v0, v1);
    }
}

__global__ void __launch_bounds__(128) mlp_forward_kernel(const float* __restrict__ P, const float* __restrict__ x,
                                                          long long B, float* __restrict__ omega) {
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    MlpWeights W;
    mlp_load_weights(P, W, lane);
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long tile = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); tile * 16 < B; tile += nw) {
        uint32_t a_in[2];
        load_inputs(x, B, tile * 16, g, t, a_in);
        float c1[4][4], c2[4][4], z[4];
        uint32_t a1[2][4], a2[2][4];
        mlp_tile_forward(W, a_in, c1, a1, c2, a2, z);
        float og[3], og8[3];
        mlp_softmax_rows(z, og, og8);
        if (t == 0) {
            const long long r = tile * 16 + g;
            if (r < B)
                for (int q = 0; q < 3; ++q) omega[r * 3 + q] = og[q];
            if (r + 8 < B)
                for (int q = 0; q < 3; ++q) omega[(r + 8) * 3 + q] = og8[q];
        }
    }
}

// bf16 element (row, col) of a row-major tile stored as 32-bit pairs.
__device__ __forceinline__ uint32_t elem16(const uint32_t* tile, int words_per_row, int row, int col) {
    const uint32_t w = tile[row * words_per_row + (col >> 1)];
    return (col & 1) ? (w >> 16) : (w & 0xFFFFu);
}

__device__ __forceinline__ uint32_t pair16(uint32_t lo, uint32_t hi) { return lo | (hi << 16); }

// A fragment (m16n8k16) of the transpose of a [16 samples][cols] tile:
// A[m][k] = tile[k][col0 + m], rows m >= mmax are zero.
__device__ __forceinline__ void transposed_a(const uint32_t* tile, int wpr, int col0, int mmax, int g, int t,
                                             uint32_t* a) {
    const int m0 = g, m1 = g + 8;
    const int k0 = 2 * t, k1 = 2 * t + 8;
    a[0] = m0 < mmax ? pair16(elem16(tile, wpr, k0, col0 + m0), elem16(tile, wpr, k0 + 1, col0 + m0)) : 0u;
    a[1] = m1 < mmax ? pair16(elem16(tile, wpr, k0, col0 + m1), elem16(tile, wpr, k0 + 1, col0 + m1)) : 0u;
    a[2] = m0 < mmax ? pair16(elem16(tile, wpr, k1, col0 + m0), elem16(tile, wpr, k1 + 1, col0 + m0)) : 0u;
    a[3] = m1 < mmax ? pair16(elem16(tile, wpr, k1, col0 + m1), elem16(tile, wpr, k1 + 1, col0 + m1)) : 0u;
}

// B fragment (m16n8k16) of a [16 samples][cols] tile: B[k][n] = tile[k][col0 + n].
__device__ __forceinline__ void tile_b(const uint32_t* tile, int wpr, int col0, int g, int t, uint32_t* b) {
    const int k0 = 2 * t, k1 = 2 * t + 8;
    b[0] = pair16(elem16(tile, wpr, k0, col0 + g), elem16(tile, wpr, k0 + 1, col0 + g));
    b[1] = pair16(elem16(tile, wpr, k1, col0 + g), elem16(tile, wpr, k1 + 1, col0 + g));
}

__device__ __forceinline__ void to_a(const float* c0, const float* c1, uint32_t* a) {
    a[0] = pack_bf16(c0[0], c0[1]);
    a[1] = pack_bf16(c0[2], c0[3]);
    a[2] = pack_bf16(c1[0], c1[1]);
    a[3] = pack_bf16(c1[2], c1[3]);
}

// Store an A fragment pair (16 x 32 bf16 tile in two k-steps) to a row-major tile.
__device__ __forceinline__ void store_a32(uint32_t* tile, const uint32_t (&a)[2][4], int g, int t) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        tile[g * 16 + 8 * s + t] = a[s][0];
        tile[(g + 8) * 16 + 8 * s + t] = a[s][1];
        tile[g * 16 + 8 * s + 4 + t] = a[s][2];
        tile[(g + 8) * 16 + 8 * s + 4 + t] = a[s][3];
    }
}

struct GradShared {
    uint32_t h1[16 * 16], h2[16 * 16], da2[16 * 16], da1[16 * 16];  // [16 rows][32 bf16]
    uint32_t dz[16 * 4], xin[16 * 4];                                // [16 rows][8 bf16]
};

__global__ void __launch_bounds__(kGradWarps * 32) mlp_grad_kernel(
    const float* __restrict__ P, const float* __restrict__ x, const float* __restrict__ phat,
    const float* __restrict__ target, const float* __restrict__ mask, long long B, float lam,
    float* __restrict__ work) {
    __shared__ GradShared sh[kGradWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    GradShared& S = sh[warp];
    MlpWeights W;
    mlp_load_weights(P, W, lane);
    // backward B fragments: dh2 = dz W3 (B[k][n] = W3[k][n], k < 3) and dh1 = da2 W2 (B[k][n] = W2[k][n])
    uint32_t w3t[4][2], w2t[2][4][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int n = 8 * j + g;
        const int k = 2 * t;
        w3t[j][0] = pack_bf16(k < 3 ? P[kOffW3 + k * kMlpH + n] : 0.f, k + 1 < 3 ? P[kOffW3 + (k + 1) * kMlpH + n] : 0.f);
        w3t[j][1] = 0u;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int k0 = 16 * s + 2 * t;
            w2t[s][j][0] = pack_bf16(P[kOffW2 + k0 * kMlpH + n], P[kOffW2 + (k0 + 1) * kMlpH + n]);
            w2t[s][j][1] = pack_bf16(P[kOffW2 + (k0 + 8) * kMlpH + n], P[kOffW2 + (k0 + 9) * kMlpH + n]);
        }
    }
    float gW3[4][4], gW2[2][4][4], gW1[2][4], gb1[4][2], gb2[4][2], gb3[3] = {0.f, 0.f, 0.f}, lsum = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        gb1[j][0] = gb1[j][1] = gb2[j][0] = gb2[j][1] = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) { gW3[j][e] = 0.f; gW2[0][j][e] = 0.f; gW2[1][j][e] = 0.f; }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) { gW1[0][e] = 0.f; gW1[1][e] = 0.f; }
    const float invB = 1.0f / (float)B;

    const long long nw = (long long)gridDim.x * kGradWarps;
    for (long long tile = (long long)blockIdx.x * kGradWarps + warp; tile * 16 < B; tile += nw) {
        const long long row0 = tile * 16;
        uint32_t a_in[2];
        load_inputs(x, B, row0, g, t, a_in);
        float c1[4][4], c2[4][4], z[4];
        uint32_t a1[2][4], a2[2][4];
        mlp_tile_forward(W, a_in, c1, a1, c2, a2, z);
        float og[3], og8[3];
        mlp_softmax_rows(z, og, og8);
        // loss and dL/dz on the t == 0 lanes for rows g and g+8
        float dzg[3] = {0.f, 0.f, 0.f}, dzg8[3] = {0.f, 0.f, 0.f};
        if (t == 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const long long r = row0 + g + 8 * h;
                if (r < B) {
                    const float* om = h ? og8 : og;
                    float* dz = h ? dzg8 : dzg;
                    const float p0 = phat[r * 3], p1 = phat[r * 3 + 1], p2 = phat[r * 3 + 2];
                    const float tt = target[r], mk = mask[r];
                    const float y = om[0] * p0 + om[1] * p1 + om[2] * p2;
                    const float e = y - tt;
                    float dom[3];
                    const float pp[3] = {p0, p1, p2};
                    float reg = 0.f;
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const float dd = om[q] - kIdeal[q];
                        reg += dd * dd;
                        dom[q] = 2.f * invB * (e * pp[q] + lam * mk * dd);
                    }
                    lsum += invB * (e * e + lam * mk * reg);
                    const float sdot = om[0] * dom[0] + om[1] * dom[1] + om[2] * dom[2];
#pragma unroll
                    for (int q = 0; q < 3; ++q) dz[q] = om[q] * (dom[q] - sdot);
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) gb3[q] += dzg[q] + dzg8[q];
        }
        // dz as an A fragment (columns 0..2): lane t=1 takes column 2 from lane t=0
        const float v2g = __shfl_up_sync(0xffffffffu, dzg[2], 1);
        const float v2g8 = __shfl_up_sync(0xffffffffu, dzg8[2], 1);
        uint32_t a_dz[4];
        a_dz[0] = t == 0 ? pack_bf16(dzg[0], dzg[1]) : (t == 1 ? pack_bf16(v2g, 0.f) : 0u);
        a_dz[1] = t == 0 ? pack_bf16(dzg8[0], dzg8[1]) : (t == 1 ? pack_bf16(v2g8, 0.f) : 0u);
        a_dz[2] = 0u;
        a_dz[3] = 0u;
        // dh2 = dz W3, da2 = dh2 * (a2 > 0)
        float da2[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float d[4] = {0.f, 0.f, 0.f, 0.f};
            mma16816(d, a_dz, w3t[j]);
#pragma unroll
            for (int e = 0; e < 4; ++e) da2[j][e] = c2[j][e] > 0.f ? d[e] : 0.f;
            gb2[j][0] += da2[j][0] + da2[j][2];
            gb2[j][1] += da2[j][1] + da2[j][3];
        }
        uint32_t a_da2[2][4];
        to_a(da2[0], da2[1], a_da2[0]);
        to_a(da2[2], da2[3], a_da2[1]);
        // dh1 = da2 W2, da1 = dh1 * (a1 > 0)
        float da1[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float d[4] = {0.f, 0.f, 0.f, 0.f};
            mma16816(d, a_da2[0], w2t[0][j]);
            mma16816(d, a_da2[1], w2t[1][j]);
#pragma unroll
            for (int e = 0; e < 4; ++e) da1[j][e] = c1[j][e] > 0.f ? d[e] : 0.f;
            gb1[j][0] += da1[j][0] + da1[j][2];
            gb1[j][1] += da1[j][1] + da1[j][3];
        }
        uint32_t a_da1[2][4];
        to_a(da1[0], da1[1], a_da1[0]);
        to_a(da1[2], da1[3], a_da1[1]);
        // stage the tiles whose transposes form the weight gradients
        store_a32(S.h1, a1, g, t);
        store_a32(S.h2, a2, g, t);
        store_a32(S.da2, a_da2, g, t);
        store_a32(S.da1, a_da1, g, t);
        S.dz[g * 4 + t] = a_dz[0];
        S.dz[(g + 8) * 4 + t] = a_dz[1];
        S.xin[g * 4 + t] = a_in[0];
        S.xin[(g + 8) * 4 + t] = a_in[1];
        __syncwarp();
        // dW3 += dz^T h2  (16 x 32, rows 0..2 meaningful)
        {
            uint32_t a[4];
            transposed_a(S.dz, 4, 0, 3, g, t, a);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t b[2];
                tile_b(S.h2, 16, 8 * j, g, t, b);
                mma16816(gW3[j], a, b);
            }
        }
        // dW2 += da2^T h1 (32 x 32) and dW1 += da1^T x (32 x 8)
#pragma unroll
        for (int mi = 0; mi < 2; ++mi) {
            uint32_t a[4];
            transposed_a(S.da2, 16, 16 * mi, 16, g, t, a);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t b[2];
                tile_b(S.h1, 16, 8 * j, g, t, b);
                mma16816(gW2[mi][j], a, b);
            }
            uint32_t a1t[4], bx[2];
            transposed_a(S.da1, 16, 16 * mi, 16, g, t, a1t);
            tile_b(S.xin, 4, 0, g, t, bx);
            mma16816(gW1[mi], a1t, bx);
        }
        __syncwarp();
    }
    // reduce the bias partials and the loss over the eight row groups (lane bits 2..4)
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            gb1[j][0] += __shfl_xor_sync(0xffffffffu, gb1[j][0], o);
            gb1[j][1] += __shfl_xor_sync(0xffffffffu, gb1[j][1], o);
            gb2[j][0] += __shfl_xor_sync(0xffffffffu, gb2[j][0], o);
            gb2[j][1] += __shfl_xor_sync(0xffffffffu, gb2[j][1], o);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) gb3[q] += __shfl_xor_sync(0xffffffffu, gb3[q], o);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    }
    float* out = work + ((long long)blockIdx.x * kGradWarps + warp) * kGradStride;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (g < 3) {
            out[kOffW3 + g * kMlpH + 8 * j + 2 * t] = gW3[j][0];
            out[kOffW3 + g * kMlpH + 8 * j + 2 * t + 1] = gW3[j][1];
        }
#pragma unroll
        for (int mi = 0; mi < 2; ++mi) {
            const int r0 = 16 * mi + g, r1 = r0 + 8, c = 8 * j + 2 * t;
            out[kOffW2 + r0 * kMlpH + c] = gW2[mi][j][0];
            out[kOffW2 + r0 * kMlpH + c + 1] = gW2[mi][j][1];
            out[kOffW2 + r1 * kMlpH + c] = gW2[mi][j][2];
            out[kOffW2 + r1 * kMlpH + c + 1] = gW2[mi][j][3];
        }
        if (g == 0) {
            out[kOffB1 + 8 * j + 2 * t] = gb1[j][0];
            out[kOffB1 + 8 * j + 2 * t + 1] = gb1[j][1];
            out[kOffB2 + 8 * j + 2 * t] = gb2[j][0];
            out[kOffB2 + 8 * j + 2 * t + 1] = gb2[j][1];
        }
    }
#pragma unroll
    for (int mi = 0; mi < 2; ++mi) {
        const int r0 = 16 * mi + g, r1 = r0 + 8;
        const int c = 2 * t;
        if (c < kMlpIn) {
            out[kOffW1 + r0 * kMlpIn + c] = gW1[mi][0];
            out[kOffW1 + r1 * kMlpIn + c] = gW1[mi][2];
        }
        if (c + 1 < kMlpIn) {
            out[kOffW1 + r0 * kMlpIn + c + 1] = gW1[mi][1];
            out[kOffW1 + r1 * kMlpIn + c + 1] = gW1[mi][3];
        }
    }
    if (lane == 0) {
        for (int q = 0; q < 3; ++q) out[kOffB3 + q] = gb3[q];
        out[kMlpParams] = lsum;
    }
}

// Deterministic sum of the partial gradients work[parts][kGradStride]: a CTA of
// kReduceWarps warps takes 32 slots, each warp every kReduceWarps-th partial
// (coalesced 128-byte rows), then the warps' sums in a fixed order.  One thread
// per slot walked all partials alone, on 11 SMs, each load waiting on DRAM or L2
// (304 partials: 14.4 us); 16 chains of 19 loads on 43 SMs take 3 us.
constexpr int kReduceWarps = 16;
__global__ void __launch_bounds__(32 * kReduceWarps) mlp_reduce_kernel(const float* __restrict__ work, int parts,
                                                                       float* __restrict__ grad,
                                                                       float* __restrict__ loss) {
    __shared__ float sh[kReduceWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = blockIdx.x * 32 + lane;
    pdl_wait();
    float s = 0.f;
    if (p <= kMlpParams) {
#pragma unroll 8
        for (int w = warp; w < parts; w += kReduceWarps) s += work[(long long)w * kGradStride + p];
    }
    sh[warp][lane] = s;
    __syncthreads();
    if (warp != 0 || p > kMlpParams) return;
#pragma unroll
    for (int w = 1; w < kReduceWarps; ++w) s += sh[w][lane];
    if (p < kMlpParams) grad[p] = s;
    else if (loss) *loss = s;
}

// Adam (Kingma & Ba 2015): bias corrections c1 = 1/(1-b1^t), c2 = 1/(1-b2^t).
__global__ void mlp_adam_kernel(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ M,
                                float* __restrict__ V, int n, float lr, float b1, float b2, float eps, float c1,
                                float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    pdl_wait();
    const float gi = G[i];
    const float m = b1 * M[i] + (1.f - b1) * gi;
    const float v = b2 * V[i] + (1.f - b2) * gi * gi;
    M[i] = m;
    V[i] = v;
    P[i] -= lr * (m * c1) / (sqrtf(v * c2) + eps);
}

// ---------------------------------------------------------------------------
// Sample harvest.  Sample k picks (by a counter-based hash of seed and k) an
// active direction d, a coarse face I+1/2 of the 2x-restricted grid, the
// transverse coarse cell, a variable and a side: side 0 is the edge of cell I
// (stencil I-2..I+2), side 1 the edge of cell I+1 (stencil I+3..I-1, reversed).
// The coarse value of a cell is the mean of the primitives of its 2^ndim fine
// children.  The target is the fine-grid face value at the coincident fine face,
// 1/2 (left + right WENO5-JS edge values of the fine run), averaged over the
// 2^(ndim-1) fine faces that tile the coarse face.  All in FP64, stored FP32
// and normalised by the stencil scale s.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// Textbook WENO5-JS value at the right edge of the middle cell of v[0..4].
__device__ double weno5_js(const double* v, double eps) {
    const double p0 = (2.0 * v[0] - 7.0 * v[1] + 11.0 * v[2]) / 6.0;
    const double p1 = (-v[1] + 5.0 * v[2] + 2.0 * v[3]) / 6.0;
    const double p2 = (2.0 * v[2] + 5.0 * v[3] - v[4]) / 6.0;
    double q;
    q = v[0] - 2.0 * v[1] + v[2];
    double b0 = 13.0 / 12.0 * q * q;
    q = v[0] - 4.0 * v[1] + 3.0 * v[2];
    b0 += 0.25 * q * q;
    q = v[1] - 2.0 * v[2] + v[3];
    double b1 = 13.0 / 12.0 * q * q;
    q = v[1] - v[3];
    b1 += 0.25 * q * q;
    q = v[2] - 2.0 * v[3] + v[4];
    double b2 = 13.0 / 12.0 * q * q;
    q = 3.0 * v[2] - 4.0 * v[3] + v[4];
    b2 += 0.25 * q * q;
    const double a0 = 0.1 / ((eps + b0) * (eps + b0));
    const double a1 = 0.6 / ((eps + b1) * (eps + b1));
    const double a2 = 0.3 / ((eps + b2) * (eps + b2));
    return (a0 * p0 + a1 * p1 + a2 * p2) / (a0 + a1 + a2);
}

// WENO5-JS increments at the right edge of the middle cell of two stencils side
// by side, X_k the four differences of each (weno5_increments_pair with a stencil
// of its own in every lane), in float-float; optionally the smoothness
// indicators without their 4/3 factor.  e = 3/4 eps.
__device__ __forceinline__ df2 weno5_right_pair(df2 X0, df2 X1, df2 X2, df2 X3, df2 e, df2* beta = nullptr) {
    const df2 S1 = df2_mul(X1, X1), S2 = df2_mul(X2, X2);
    const df2 b0 = df2_add_fast(df2_add_fast(df2_mul(X0, X0), df2_mul_f(df2_mul(X1, X0), f2(-2.75f))),
                                df2_mul_f(S1, f2(2.5f)));
    const df2 b1 = df2_add_fast(df2_add_fast(S1, S2), df2_mul_f(df2_mul(X1, X2), f2(-1.25f)));
    const df2 b2 = df2_add_fast(df2_add_fast(df2_mul(X3, X3), df2_mul_f(df2_mul(X2, X3), f2(-2.75f))),
                                df2_mul_f(S2, f2(2.5f)));
    if (beta) {
        beta[0] = b0;
        beta[1] = b1;
        beta[2] = b2;
    }
    const df2 T0 = df2_add_fast(e, b0), T1 = df2_add_fast(e, b1), T2 = df2_add_fast(e, b2);
    const float2 m = make_float2(fminf(T0.hi.x, fminf(T1.hi.x, T2.hi.x)), fminf(T0.hi.y, fminf(T1.hi.y, T2.hi.y)));
    const df2 g0 = df2_div_f(m, T0), g1 = df2_div_f(m, T1), g2 = df2_div_f(m, T2);
    const df2 w0 = df2_mul(g0, g0), w1 = df2_mul_f(df2_mul(g1, g1), f2(6.f)), w2 = df2_mul_f(df2_mul(g2, g2), f2(3.f));
    const df2 P0 = df2_add_fast(df2_mul_f(X1, f2(5.f)), df2_mul_pow2(X0, f2(-2.f)));
    const df2 P1 = df2_add_fast(X1, df2_mul_pow2(X2, f2(2.f)));
    const df2 P2 = df2_add_fast(df2_mul_pow2(X2, f2(4.f)), df2_neg(X3));
    const df2 num = df2_add_fast(df2_add_fast(df2_mul(w0, P0), df2_mul(w1, P1)), df2_mul(w2, P2));
    return df2_div(num, df2_mul_f(df2_add_fast(df2_add_fast(w0, w1), w2), f2(6.f)));
}

// One sample's outputs in plain FP64, for values outside the range of the
// float-float form below: a centre value or difference of 2^59 (5.8e17) and more or
// not finite, a stencil that spans less than 2^-45 (2.8e-14; the sensor's 1e-6 s^2 would
// fall among the FP32 subnormals, with 9 bits left at 2^-60), eps outside [1e-30, 1],
// tau outside [1e-30, 1e30].  f6: per fine face the six values across it.
__device__ __noinline__ void harvest_sample_f64(const double* st, const double* f6, int ntr, double eps, double tau,
                                                float* x, float* ph, float* to, float* so, float* jo) {
    double tgt = 0.0;
    for (int ch = 0; ch < ntr; ++ch) {
        const double* f = f6 + 6 * ch;
        const double l = weno5_js(f, eps);
        const double rv[5] = {f[5], f[4], f[3], f[2], f[1]};
        tgt += 0.5 * (l + weno5_js(rv, eps));
    }
    tgt /= ntr;
    const double c = st[2];
    double s = 0.0;
    for (int m = 0; m < 5; ++m) s = fmax(s, fabs(st[m] - c));
    const double tn = (tgt - c) / (s + 1e-30);
    for (int m = 0; m < 5; ++m) x[m] = 0.f;
    ph[0] = ph[1] = ph[2] = *to = *jo = *so = 0.f;
    if (!(s > 1e-7 * fabs(c)) || !(s > 1e-300) || !(fabs(tn) <= 8.0)) return;
    s += 1e-30;
    for (int m = 0; m < 5; ++m) x[m] = (float)((st[m] - c) / s);
    const double p0 = (2.0 * st[0] - 7.0 * st[1] + 11.0 * st[2]) / 6.0;
    const double p1 = (-st[1] + 5.0 * st[2] + 2.0 * st[3]) / 6.0;
    const double p2 = (2.0 * st[2] + 5.0 * st[3] - st[4]) / 6.0;
    ph[0] = (float)((p0 - c) / s);
    ph[1] = (float)((p1 - c) / s);
    ph[2] = (float)((p2 - c) / s);
    *to = (float)tn;
    *jo = (float)((weno5_js(st, eps) - c) / s);
    // discontinuity sensor (the same test the learned sweep applies)
    const double D0 = st[1] - st[0], D1 = st[2] - st[1], D2 = st[3] - st[2], D3 = st[4] - st[3];
    const double bb0 = 2.5 * D1 * D1 - 2.75 * D1 * D0 + D0 * D0;
    const double bb1 = D1 * D1 + D2 * D2 - 1.25 * D1 * D2;
    const double bb2 = 2.5 * D2 * D2 - 2.75 * D2 * D3 + D3 * D3;
    const double bmax = fmax(bb0, fmax(bb1, bb2)), bmin = fmin(bb0, fmin(bb1, bb2));
    *so = bmax > tau * (bmin + 1e-6 * s * s) ? 0.f : 1.f;
}

__device__ __forceinline__ unsigned abs_hi(double d) { return (unsigned)__double2hiint(d) & 0x7FFFFFFFu; }

// A stencil flat to FP32 resolution of its centre value carries no shape to
// learn (its normalised target would be round-off); such samples, and any
// whose fine target lies far outside the stencil's range, are stored as
// zeros with smooth = 0 so they add nothing to the loss.
//
// In plain FP64 (nine WENO5-JS values, ~80 divisions) a sample took ~1,400 FP64
// instructions and the kernel was bound by them: 500,000 samples of a 160^3
// field 1.10 ms, now 0.22 ms, bound by the gather (72 values of 8 bytes per
// sample from as many sectors, 0.79 GB from DRAM).  Here FP64 forms the coarse means and all differences; weights,
// increments and normalised values are float-float (mfc_df.cuh, ~2^-46 of the
// differences, far below the FP32 they are stored in), the two sides of a fine
// face in the lanes of packed instructions.  Everything is taken relative to the
// centre value, so nothing cancels where the stencil is small against it.
template <int NDIM>
__global__ void __launch_bounds__(128) harvest_kernel(const double* __restrict__ wf, int nxf, int nyf, int nzf, int ns,
                                                      double eps, double tau, df eps34, df taud, df scale,
                                                      bool eps_in_range,
                                                      long long nsamp, unsigned long long seed,
                                                      float* __restrict__ xo, float* __restrict__ po,
                                                      float* __restrict__ to, float* __restrict__ so,
                                                      float* __restrict__ jo) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nsamp) return;
    const long long nf = (long long)nxf * nyf * nzf;
    const int nc[3] = {nxf / 2, NDIM > 1 ? nyf / 2 : 1, NDIM > 2 ? nzf / 2 : 1};
    const unsigned long long h0 = mix64(seed ^ mix64((unsigned long long)k));
    const unsigned long long h1 = mix64(h0), h2 = mix64(h1), h3 = mix64(h2);
    const int d = (int)(h0 % (unsigned long long)NDIM);
    const int side = (int)((h0 >> 20) & 1ULL);
    const int var = (int)((h0 >> 24) % (unsigned long long)ns);
    const int nd = d == 0 ? nc[0] : d == 1 ? nc[1] : nc[2];
    const int I = 2 + (int)(h1 % (unsigned long long)(nd - 6));
    const int cc[3] = {(int)(h2 % (unsigned long long)nc[0]), (int)((h2 >> 21) % (unsigned long long)nc[1]),
                       (int)(h3 % (unsigned long long)nc[2])};
    const long long sf[3] = {1, (long long)nxf, (long long)nxf * nyf};
    const long long sd = d == 0 ? sf[0] : d == 1 ? sf[1] : sf[2];
    // first fine cell of the coarse column: transverse coordinates 2 cc, 0 along d
    long long base = (long long)var * nf;
#pragma unroll
    for (int a = 0; a < NDIM; ++a) base += a == d ? 0 : 2 * cc[a] * sf[a];
    // strides of the transverse directions, in their order
    const long long t1 = d == 0 ? sf[1] : sf[0], t2 = d == 2 ? sf[1] : sf[2];
    constexpr int NTR = 1 << (NDIM - 1);
    const double* col = wf + base + (long long)(2 * (I - 2)) * sd;   // fine cells 2I-4 .. 2I+7 along d
    // coarse values of cells I-2..I+3 along d: mean of the 2^d children, summed in
    // the children's order (x fastest); the fine values across the face are among them
    double W[6], f6[NTR][6];
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        double v[2][NTR];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int t = 0; t < NTR; ++t) {
                v[h][t] = __ldg(col + (2 * m + h) * sd + (t & 1 ? t1 : 0) + (t & 2 ? t2 : 0));
                const int j = 2 * m + h - 3;   // f6 holds fine cells 2I-1 .. 2I+4
                if (j >= 0 && j < 6) f6[t][j] = v[h][t];
            }
        double s = 0.0;
#pragma unroll
        for (int ch = 0; ch < 2 * NTR; ++ch) {
            // child ch: bit a = fine offset in direction a
            double u0 = v[ch & 1][(ch >> 1) & (NTR - 1)];                                    // d == 0
            if constexpr (NDIM > 1) {
                const double u1 = v[(ch >> 1) & 1][(ch & 1) | ((ch >> 1) & (NTR - 2))];      // d == 1
                u0 = d == 0 ? u0 : u1;
            }
            if constexpr (NDIM > 2) {
                const double u2 = v[(ch >> 2) & 1][ch & 3];                                  // d == 2
                u0 = d == 2 ? u2 : u0;
            }
            s += u0;
        }
        W[m] = s * (1.0 / (2 * NTR));
    }
    double st[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) st[m] = side == 0 ? W[m] : W[5 - m];
    const double c = st[2];
    float x[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, ph[3] = {0.f, 0.f, 0.f}, tv = 0.f, sv = 0.f, jv = 0.f;
    // the stencil about its centre; s its largest distance from it (bit patterns
    // of non-negative doubles order as integers)
    double dm[5];
    unsigned long long sb = 0;
    unsigned big = abs_hi(c);
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        dm[m] = st[m] - c;
        const unsigned long long u = (unsigned long long)__double_as_longlong(dm[m]) & 0x7FFFFFFFFFFFFFFFULL;
        sb = u > sb ? u : sb;
    }
    const double s = __longlong_as_double((long long)sb);
    double e[NTR][5];
#pragma unroll
    for (int t = 0; t < NTR; ++t)
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            e[t][j] = f6[t][j + 1] - f6[t][j];
            big = max(big, abs_hi(e[t][j]));
        }
    big = max(big, (unsigned)(sb >> 32));
    constexpr unsigned kMax = (1023u + 59u) << 20, kMin = (1023u - 45u) << 20;   // 5.8e17, 2.8e-14
    const bool flat = !(s > 1e-7 * fabs(c)) || !(s > 1e-300);
    if (!eps_in_range || big >= kMax || (!flat && (unsigned)(sb >> 32) < kMin)) {
        harvest_sample_f64(st, &f6[0][0], NTR, eps, tau, x, ph, &tv, &sv, &jv);
    } else if (!flat) {
        const df2 ep = df2_make(eps34, eps34);
        // fine target about c: mean over the fine faces of both sides' edge values
        df inc = {0.f, 0.f};
        double mid = 0.0;
#pragma unroll
        for (int t = 0; t < NTR; ++t) {
            df E[5];
#pragma unroll
            for (int j = 0; j < 5; ++j) E[j] = df_from_double(e[t][j]);
            const df2 r = weno5_right_pair(df2_make(E[0], df_neg(E[4])), df2_make(E[1], df_neg(E[3])),
                                           df2_make(E[2], df_neg(E[2])), df2_make(E[3], df_neg(E[1])), ep);
            inc = df_add(inc, df_add(df2_x(r), df2_y(r)));
            mid += (f6[t][2] - c) + (f6[t][3] - c);
        }
        const double tgt = (mid + df_to_double(inc)) * (0.5 / NTR);
        const df S = df_from_double(s + 1e-30);
        const df tn = df_div(df_from_double(tgt), S);
        if (fabsf(tn.hi) <= 8.f && !(fabsf(tn.hi) == 8.f && (tn.hi > 0.f ? tn.lo > 0.f : tn.lo < 0.f))) {
            df dd[5], beta[3];
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                dd[m] = df_from_double(dm[m]);
                x[m] = m == 2 ? 0.f : df_div(dd[m], S).hi;
            }
            df X[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) X[j] = df_from_double(st[j + 1] - st[j]);
            df2 b2[3];
            const df2 r = weno5_right_pair(df2_make(X[0], X[0]), df2_make(X[1], X[1]), df2_make(X[2], X[2]),
                                           df2_make(X[3], X[3]), ep, b2);
            jv = df_div(df2_x(r), S).hi;
            const df S6 = df_mul_f(S, 6.f);
            ph[0] = df_div(df_add(df_mul_pow2(dd[0], 2.f), df_mul_f(dd[1], -7.f)), S6).hi;
            ph[1] = df_div(df_add(df_mul_pow2(dd[3], 2.f), df_neg(dd[1])), S6).hi;
            ph[2] = df_div(df_add(df_mul_f(dd[3], 5.f), df_neg(dd[4])), S6).hi;
            tv = tn.hi;
            // discontinuity sensor (the same test the learned sweep applies)
#pragma unroll
            for (int q = 0; q < 3; ++q) beta[q] = df2_x(b2[q]);
            const df bmax = df_max(beta[0], df_max(beta[1], beta[2])), bmin = df_min(beta[0], df_min(beta[1], beta[2]));
            const df lim = df_mul(taud, df_add(bmin, df_mul(df_mul(S, S), scale)));
            sv = df_lt(lim, bmax) ? 0.f : 1.f;
        }
    }
#pragma unroll
    for (int m = 0; m < 5; ++m) xo[k * 5 + m] = x[m];
#pragma unroll
    for (int m = 0; m < 3; ++m) po[k * 3 + m] = ph[m];
    to[k] = tv;
    so[k] = sv;
    jo[k] = jv;
}

// n / d from the FP64 Newton reciprocal r of d, finished with the exact residual
// (Markstein): the rounding of a division while the residual is representable (|n| from
// 2^-900 on) and the quotient normal.  A zero n is its own sign's quotient; the rest is
// divided (out of line: inlined, the division ran speculatively in every lane, 58
// FP64 instructions per cell instead of 27).
__device__ __noinline__ double div_slow(double n, double d) { return n / d; }
__device__ __forceinline__ double div_by(double n, double d, double r) {
    const double q = n * r;
    const double res = fma(fma(-q, d, n), r, q);
    if (abs_hi(n) >= 0x07B00000u && abs_hi(res) - 0x00100000u < 0x7FE00000u) return res;
    if (((__double_as_longlong(n) | __double_as_longlong(q)) << 1) == 0) return q;
    return div_slow(n, d);
}

// FP64 primitive recovery for output; the six-equation model (SIX) appends the
// phase pressures p_k = (a_k r_k e_k / a_k - P_k)/G_k.  One template per model, so
// that rows are addressed at compile time and a cell's loads go out together, and
// two reciprocals for the d + 1 divisions; the kernel is bound by FP64
// instructions (26 per cell, the FP64 pipe 90% busy).  160^3, two fluids: 312 us
// with run-time loops and divisions, 193 us now.
template <int NF, int NDIM, bool SIX>
__global__ void __launch_bounds__(256) prims_out_kernel(const double* __restrict__ q, double* __restrict__ w,
                                                        long long nc, EosConst e) {
    using Lay = Layout<NF, NDIM, SIX>;
    constexpr int NS = Lay::NS, NQ = Lay::NQ, IM = Lay::IM, IE = Lay::IE, IA = Lay::IA;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc;
         i += (long long)gridDim.x * blockDim.x) {
        double s[NQ];
#pragma unroll
        for (int v = 0; v < NQ; ++v) s[v] = __ldg(q + v * nc + i);
        double rho = s[0], G = e.G_N, P = e.P_N, ke = 0.0;
#pragma unroll
        for (int k = 1; k < NF; ++k) rho += s[k];
#pragma unroll
        for (int k = 0; k < NF - 1; ++k) {
            G = fma(s[IA + k], e.dG[k], G);
            P = fma(s[IA + k], e.dP[k], P);
        }
        const double irho = rcp_nr(rho);
#pragma unroll
        for (int d = 0; d < NDIM; ++d) {
            const double u = div_by(s[IM + d], rho, irho);
            ke = fma(s[IM + d], u, ke);
            s[IM + d] = u;
        }
        s[IE] = div_by(s[IE] - 0.5 * ke - P, G, rcp_nr(G));
        if constexpr (SIX) {
            double aN = 1.0;
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                const double ak = k < NF - 1 ? s[IA + k] : aN;
                if (k < NF - 1) aN -= ak;
                const double Gk = k < NF - 1 ? e.G_N + e.dG[k] : e.G_N;
                const double Pk = k < NF - 1 ? e.P_N + e.dP[k] : e.P_N;
                s[NS + k] = (s[NS + k] / ak - Pk) / Gk;
            }
        }
#pragma unroll
        for (int v = 0; v < NQ; ++v) w[v * nc + i] = s[v];
    }
}

template <int NF, bool SIX>
void launch_prims_out(const double* q, double* w, long long nc, int ndim, const EosConst& e, unsigned blocks,
                      cudaStream_t s) {
    if (ndim == 1) prims_out_kernel<NF, 1, SIX><<<blocks, 256, 0, s>>>(q, w, nc, e);
    else if (ndim == 2) prims_out_kernel<NF, 2, SIX><<<blocks, 256, 0, s>>>(q, w, nc, e);
    else prims_out_kernel<NF, 3, SIX><<<blocks, 256, 0, s>>>(q, w, nc, e);
}

// One warp: the per-lane MMA fragments of a parameter blob, for the sweeps.
__global__ void __launch_bounds__(32) mlp_pack_kernel(const float* __restrict__ P, uint4* __restrict__ frag) {
    MlpWeights W;
    mlp_load_weights(P, W, threadIdx.x);
    mlp_weights_to_frag(W, frag, threadIdx.x);
}

}  // namespace

// Host launcher of the partial-gradient sum, used by both gradient entries.
cudaError_t mfc_launch_mlp_reduce(const float* work, int parts, float* grad, float* loss, cudaStream_t s) {
    return launch_pdl(mlp_reduce_kernel, (kGradStride + 31) / 32, 32 * kReduceWarps, 0, s, work, parts, grad, loss);
}

// Host launcher used by mfc_set_mlp: frag holds kMlpFragBytes.
cudaError_t mfc_launch_mlp_pack(const float* P, void* frag, cudaStream_t s) {
    mlp_pack_kernel<<<1, 32, 0, s>>>(P, static_cast<uint4*>(frag));
    return cudaGetLastError();
}

// Host launcher used by mfc_get_prims in the context code.
cudaError_t mfc_launch_prims_out(const double* q, double* w, long long nc, int nf, int ndim, const EosConst& e,
                                 int six, cudaStream_t s) {
    long long b = (nc + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    const unsigned blocks = (unsigned)b;
    if (six) {
        if (nf == 2) launch_prims_out<2, true>(q, w, nc, ndim, e, blocks, s);
        else launch_prims_out<3, true>(q, w, nc, ndim, e, blocks, s);
    } else if (nf == 1) {
        launch_prims_out<1, false>(q, w, nc, ndim, e, blocks, s);
    } else if (nf == 2) {
        launch_prims_out<2, false>(q, w, nc, ndim, e, blocks, s);
    } else {
        launch_prims_out<3, false>(q, w, nc, ndim, e, blocks, s);
    }
    return cudaGetLastError();
}

extern "C" {

mfc_status mfc_mlp_forward(const float* params, const float* x, long long batch, float* omega, void* stream) {
    if (!params || !x || !omega || batch <= 0) return MFC_ERR_ARG;
    const long long tiles = (batch + 15) / 16;
    long long blocks = (tiles + 3) / 4;
    if (blocks > 152 * 8) blocks = 152 * 8;
    mlp_forward_kernel<<<(unsigned)blocks, 128, 0, static_cast<cudaStream_t>(stream)>>>(params, x, batch, omega);
    return cudaGetLastError() == cudaSuccess ? MFC_OK : MFC_ERR_CUDA;
}

mfc_status mfc_mlp_grad_mma(const float* params, const float* x, const float* phat, const float* target,
                            const float* mask, long long batch, float lam, float* grad, float* loss, float* work,
                            void* stream) {
    if (!params || !x || !phat || !target || !mask || !grad || !work || batch <= 0 || !(lam >= 0.f))
        return MFC_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    mlp_grad_kernel<<<kGradBlocks, kGradWarps * 32, 0, s>>>(params, x, phat, target, mask, batch, lam, work);
    if (cudaGetLastError() != cudaSuccess) return MFC_ERR_CUDA;
    return mfc_launch_mlp_reduce(work, kGradBlocks * kGradWarps, grad, loss, s) == cudaSuccess ? MFC_OK : MFC_ERR_CUDA;
}

mfc_status mfc_mlp_adam(float* params, const float* grad, float* m, float* v, int n, float lr, float beta1,
                        float beta2, float eps, int step, void* stream) {
    if (!params || !grad || !m || !v || n <= 0 || step < 1 || !(lr > 0.f) || !(beta1 >= 0.f && beta1 < 1.f) ||
        !(beta2 >= 0.f && beta2 < 1.f) || !(eps >= 0.f))
        return MFC_ERR_ARG;
    const float c1 = (float)(1.0 / (1.0 - std::pow((double)beta1, step)));
    const float c2 = (float)(1.0 / (1.0 - std::pow((double)beta2, step)));
    return launch_pdl(mlp_adam_kernel, (unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream), params,
                      grad, m, v, n, lr, beta1, beta2, eps, c1, c2) == cudaSuccess
               ? MFC_OK
               : MFC_ERR_CUDA;
}

mfc_status mfc_harvest(const double* w_fine, int nxf, int nyf, int nzf, int num_fluids, double weno_eps, double tau,
                       long long n_samples, unsigned long long seed, float* x, float* phat, float* target,
                       float* smooth, float* js, void* stream) {
    if (!w_fine || !x || !phat || !target || !smooth || !js || n_samples <= 0) return MFC_ERR_ARG;
    if (num_fluids < 1 || num_fluids > 3 || !(weno_eps > 0.0) || !(tau > 0.0)) return MFC_ERR_ARG;
    const int ndim = nzf > 1 ? 3 : (nyf > 1 ? 2 : 1);
    const int nfd[3] = {nxf, nyf, nzf};
    for (int a = 0; a < 3; ++a) {
        if (a < ndim && (nfd[a] % 2 != 0 || nfd[a] / 2 < 8)) return MFC_ERR_ARG;
        if (a >= ndim && nfd[a] != 1) return MFC_ERR_ARG;
    }
    const int ns = 2 * num_fluids + ndim;
    const long long blocks = (n_samples + 127) / 128;
    const df e34 = df_split(0.75 * weno_eps), taud = df_split(tau), scale = df_split(1e-6);
    const bool in_range = weno_eps >= 1e-30 && weno_eps <= 1.0 && tau >= 1e-30 && tau <= 1e30;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    auto go = [&](auto kernel) {
        kernel<<<(unsigned)blocks, 128, 0, st>>>(w_fine, nxf, nyf, nzf, ns, weno_eps, tau, e34, taud, scale, in_range,
                                                 n_samples, seed, x, phat, target, smooth, js);
    };
    if (ndim == 1) go(harvest_kernel<1>);
    else if (ndim == 2) go(harvest_kernel<2>);
    else go(harvest_kernel<3>);
    return cudaGetLastError() == cudaSuccess ? MFC_OK : MFC_ERR_CUDA;
}

}  // extern "C"
