// rb_mlp.cu -- learned far-field correction (not in the paper): a small MLP
// (12 -> 64 -> 64 -> 64 -> 3, GELU tanh form) predicts the residual between
// an accepted cell's exact force (Eq. 1 over its particles) and its
// multipole force (Sect. 4.2), in units of G M / R^2, so the walk can open
// cells at a wider theta and add the predicted residual.
//
// This file holds the training side (residual labels, the tensor-core
// gradient kernel, Adam) and the packing of trained weights for inference;
// inference itself runs inside the gravity walk (rb_walk.cu).
//
// Tensor cores: every layer of the forward and backward pass is a BF16
// mma.sync.m16n8k16 with FP32 accumulation.  Inference gives a warp 16 rows,
// whose hidden activations stay in registers between layers (the FP32
// accumulator fragment of one layer is the BF16 A fragment of the next);
// training gives a block of 8 warps 32 rows.
// Training keeps FP32 master weights (Adam) and hands BF16 copies to the
// kernels.
//
// Parameter layout used inside the library ("padded"): W1 16x64 (rows 12..15
// zero), b1 64, W2 64x64, b2 64, W3 64x64, b3 64, W4 64x8 (cols 3..7 zero),
// b4 8 -- 9928 values; the C ABI exchanges the unpadded 9347 values in the
// order W1 (12x64), b1, W2, b2, W3, b3, W4 (64x3), b4 (row-major, input x
// output).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <vector>

#include "rb_internal.cuh"
#include "rb_mlp.cuh"

namespace rb {
namespace mlp {
namespace {

constexpr int kRows = 32;         // rows of a block's tile in the gradient kernel
constexpr int kMaxPartials = 152; // blocks of the gradient kernel, one per SM
constexpr int kLdH = 72;          // row strides (BF16) of the staged activations and
constexpr int kLdX = 24;          // inputs: ldmatrix reads 8 rows without bank conflicts

// BF16 weights of training as mma B fragments, an entry per MMA and lane: F1..F4
// those of the forward pass, T4..T2 the tiles of W4^T, W3^T and W2^T that take
// an output gradient back to the layer below (B[k][n] = W[n][k]).  One 8-byte
// load per lane and MMA, straight into registers.
struct TrainW {
    uint2 F1[1][8][32], F2[4][8][32], F3[4][8][32], F4[4][1][32];
    uint2 T4[1][8][32], T3[4][8][32], T2[4][8][32];
};

// Writes padded parameter i (value v) into the fragments; biases are read in FP32.
__device__ __forceinline__ void put_weight(TrainW& T, int i, float v) {
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    // element (k, n) of a B operand with nt column tiles
    auto put = [&](uint2* F, int nt, int k, int n) {
        const int lane = 4 * (n & 7) + ((k & 7) >> 1);
        const int at = ((k >> 4) * nt + (n >> 3)) * 32 + lane;
        reinterpret_cast<__nv_bfloat16*>(F + at)[((k >> 3) & 1) * 2 + (k & 1)] = h;
    };
    if (i < kB1) {
        put(&T.F1[0][0][0], 8, i >> 6, i & 63);
    } else if (i >= kW2 && i < kB2) {
        put(&T.F2[0][0][0], 8, (i - kW2) >> 6, (i - kW2) & 63);
        put(&T.T2[0][0][0], 8, (i - kW2) & 63, (i - kW2) >> 6);
    } else if (i >= kW3 && i < kB3) {
        put(&T.F3[0][0][0], 8, (i - kW3) >> 6, (i - kW3) & 63);
        put(&T.T3[0][0][0], 8, (i - kW3) & 63, (i - kW3) >> 6);
    } else if (i >= kW4 && i < kB4) {
        put(&T.F4[0][0][0], 1, (i - kW4) >> 3, (i - kW4) & 7);
        put(&T.T4[0][0][0], 8, (i - kW4) & 7, (i - kW4) >> 3);
    }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const __nv_bfloat16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)) : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t& r0, uint32_t& r1, const __nv_bfloat16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r0), "=r"(r1) : "r"(smem_u32(p)) : "memory");
}

// This lane's row address of each operand tile of a row-major matrix M (ld
// columns): a 16 x 16 A tile at (r0, c0), ...
__device__ __forceinline__ const __nv_bfloat16* at_a(const __nv_bfloat16* M, int ld, int r0, int c0, int lane) {
    return M + (r0 + (lane & 15)) * ld + c0 + (lane >> 4) * 8;
}
// ... the A tile of M^T whose rows are columns c0 .. and whose k are rows r0 .., ...
__device__ __forceinline__ const __nv_bfloat16* at_at(const __nv_bfloat16* M, int ld, int r0, int c0, int lane) {
    return M + (r0 + (lane & 7) + (lane >> 4) * 8) * ld + c0 + ((lane >> 3) & 1) * 8;
}
// ... and two 16 x 8 B tiles at (r0, c0) and (r0, c0 + 8) (the lower 16 lanes: the first).
__device__ __forceinline__ const __nv_bfloat16* at_b(const __nv_bfloat16* M, int ld, int r0, int c0, int lane) {
    return M + (r0 + (lane & 15)) * ld + c0 + (lane >> 4) * 8;
}

// A hidden layer's forward pass for 16 rows and 16 columns of the tile:
// activations to out, GELU's derivatives kept for the backward pass.
template <int KT>
__device__ __forceinline__ void train_hidden(const __nv_bfloat16* in, int ld, const uint2 (&F)[KT][2],
                                             const float2 (&bias)[2], __nv_bfloat16* out, float (&gp)[2][4],
                                             int r0, int c0, int lane) {
    const int g = lane >> 2, q = lane & 3;
    float c[2][4];
#pragma unroll
    for (int j = 0; j < 2; j++) {
        c[j][0] = c[j][2] = bias[j].x;
        c[j][1] = c[j][3] = bias[j].y;
    }
#pragma unroll
    for (int t = 0; t < KT; t++) {
        uint32_t a[4];
        ldsm4(a, at_a(in, ld, r0, 16 * t, lane));
#pragma unroll
        for (int j = 0; j < 2; j++) mma(c[j], a, F[t][j].x, F[t][j].y);
    }
#pragma unroll
    for (int j = 0; j < 2; j++) {
        float h[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const float z = c[j][e];
            const float t = tanhf(kGeluC * (z + 0.044715f * z * z * z));
            h[e] = 0.5f * z * (1.f + t);
            gp[j][e] = 0.5f * (1.f + t) + 0.5f * z * (1.f - t * t) * kGeluC * (1.f + 3.f * 0.044715f * z * z);
        }
        __nv_bfloat16* o = out + (r0 + g) * kLdH + c0 + 8 * j + 2 * q;
        *reinterpret_cast<uint32_t*>(o) = pack2(h[0], h[1]);
        *reinterpret_cast<uint32_t*>(o + 8 * kLdH) = pack2(h[2], h[3]);
    }
}

// dZ = dH gelu'(Z) of the warp's 16 rows and columns: FP32 column sums for the
// bias, BF16 copy for the MMAs.
__device__ __forceinline__ void train_dz(float (&dh)[2][4], const float (&gp)[2][4], float (&sb)[2][2],
                                         __nv_bfloat16* D, int r0, int c0, int lane) {
    const int g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int j = 0; j < 2; j++) {
#pragma unroll
        for (int e = 0; e < 4; e++) dh[j][e] *= gp[j][e];
        sb[j][0] += dh[j][0] + dh[j][2];
        sb[j][1] += dh[j][1] + dh[j][3];
        __nv_bfloat16* o = D + (r0 + g) * kLdH + c0 + 8 * j + 2 * q;
        *reinterpret_cast<uint32_t*>(o) = pack2(dh[j][0], dh[j][1]);
        *reinterpret_cast<uint32_t*>(o + 8 * kLdH) = pack2(dh[j][2], dh[j][3]);
    }
}

// dH of the layer below: the warp's 16 rows and columns of dZ W^T.
__device__ __forceinline__ void train_dh(float (&dh)[2][4], const __nv_bfloat16* D, const uint2 (&T)[4][2], int r0,
                                         int lane) {
#pragma unroll
    for (int j = 0; j < 2; j++) dh[j][0] = dh[j][1] = dh[j][2] = dh[j][3] = 0.f;
#pragma unroll
    for (int t = 0; t < 4; t++) {
        uint32_t a[4];
        ldsm4(a, at_a(D, kLdH, r0, 16 * t, lane));
#pragma unroll
        for (int j = 0; j < 2; j++) mma(dh[j], a, T[t][j].x, T[t][j].y);
    }
}

// acc += a 16-row product: each tile of 16 rows is an MMA of its own, so the
// sum over rows runs in FP32 additions.
__device__ __forceinline__ void add_mma(float (&acc)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    mma(c, a, b0, b1);
#pragma unroll
    for (int e = 0; e < 4; e++) acc[e] += c[e];
}

// Rows r0 .. r0 + 31 of In^T dZ: 16 rows (c0 ..) and 32 columns (n0 ..) of a
// hidden layer's weight gradient.
__device__ __forceinline__ void train_dw(float (&acc)[4][4], const __nv_bfloat16* in, const __nv_bfloat16* D, int c0,
                                         int n0, int lane) {
#pragma unroll
    for (int k = 0; k < 2; k++) {
        uint32_t a[4];
        ldsm4t(a, at_at(in, kLdH, 16 * k, c0, lane));
#pragma unroll
        for (int j = 0; j < 2; j++) {
            uint32_t b[4];
            ldsm4t(b, at_b(D, kLdH, 16 * k, n0 + 16 * j, lane));
            add_mma(acc[2 * j], a, b[0], b[1]);
            add_mma(acc[2 * j + 1], a, b[2], b[3]);
        }
    }
}

struct GradSmem {
    __nv_bfloat16 X[kRows * kLdX];       // inputs (columns 12..15 zero)
    __nv_bfloat16 H[3][kRows * kLdH];    // activations of the hidden layers
    __nv_bfloat16 D[3][kRows * kLdH];    // gradients of their pre-activations
    __nv_bfloat16 D4[kRows * kLdX];      // output gradients (columns 0..7)
    float b[2][200];                     // bias gradients of the two 16-row halves
    float loss[2];
};

// Gradient of the mean squared error over the rows idx[0..n) (all rows of a
// batch of size n_total): forward, then backward through the three hidden
// layers; weight gradients are MMAs of activations^T x output gradients.  A
// block's 8 warps share tiles of 32 rows: each takes 16 rows and 16 columns of
// every layer, and 16 x 32 of a weight gradient, which stays in registers until
// the block's last tile and is then written as the block's part (summed by
// k_mlp_update in a fixed order).
// A batch has too few rows to fill the GPU (2048 rows: 64 blocks), so the time
// is the chain of layers: the weights wait in registers and the layers hand on
// through shared memory.  2048 rows: 7.5 us and 4.8 us for the update; a warp
// per 16 rows with weights, operands and gradient sums (atomics) in shared
// memory took 95 us (training 60,000 rows twice in such batches: 6.34 ms, now
// 2.64 ms, of which 0.8 ms are kernels).
__global__ void __launch_bounds__(256, 1) k_mlp_grad(const TrainW* __restrict__ tw, const float* __restrict__ wf,
                                                     const float* __restrict__ X, const float* __restrict__ Y,
                                                     const int32_t* __restrict__ idx, int n, int n_total,
                                                     float* __restrict__ part, float* __restrict__ lpart) {
    __shared__ __align__(16) GradSmem S;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int r0 = 16 * (w & 1), c0 = 16 * (w >> 1), j0 = c0 / 8;   // layers: rows and columns
    const int m0 = 16 * (w & 3), n0 = 32 * (w >> 2);                // weight gradients
    const bool outw = w < 2;                                        // the output layer's warps
    uint2 f1[1][2], f2[4][2], f3[4][2], f4[4], t4[2], t3[4][2], t2[4][2];
    float2 bias[3][2];
#pragma unroll
    for (int j = 0; j < 2; j++) {
        f1[0][j] = tw->F1[0][j0 + j][lane];
        t4[j] = tw->T4[0][j0 + j][lane];
#pragma unroll
        for (int t = 0; t < 4; t++) {
            f2[t][j] = tw->F2[t][j0 + j][lane];
            f3[t][j] = tw->F3[t][j0 + j][lane];
            t3[t][j] = tw->T3[t][j0 + j][lane];
            t2[t][j] = tw->T2[t][j0 + j][lane];
        }
        const int c = c0 + 8 * j + 2 * q;
        bias[0][j] = *reinterpret_cast<const float2*>(wf + kB1 + c);
        bias[1][j] = *reinterpret_cast<const float2*>(wf + kB2 + c);
        bias[2][j] = *reinterpret_cast<const float2*>(wf + kB3 + c);
    }
#pragma unroll
    for (int t = 0; t < 4; t++) f4[t] = tw->F4[t][0][lane];
    const float2 bias4 = *reinterpret_cast<const float2*>(wf + kB4 + 2 * q);
    float dw1[4] = {0.f}, dw2[4][4] = {{0.f}}, dw3[4][4] = {{0.f}}, dw4[4] = {0.f};
    float sb1[2][2] = {{0.f}}, sb2[2][2] = {{0.f}}, sb3[2][2] = {{0.f}}, sb4[2] = {0.f, 0.f};
    float lsum = 0.f;
    const float scale = 2.f / (3.f * (float)n_total);
    const int ntiles = (n - 1) / kRows + 1;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        __syncthreads();   // the last tile's readers are done
        if (threadIdx.x < 4 * kRows) {
            // four values of a row; columns 12..15 are zero
            const int r = threadIdx.x >> 2, c = threadIdx.x & 3;
            const unsigned row = (unsigned)tile * kRows + r;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row < (unsigned)n && c < 3) v = *reinterpret_cast<const float4*>(X + (size_t)idx[row] * 12 + 4 * c);
            *reinterpret_cast<uint2*>(&S.X[r * kLdX + 4 * c]) = make_uint2(pack2(v.x, v.y), pack2(v.z, v.w));
        }
        float y[4] = {0.f, 0.f, 0.f, 0.f};
        if (outw) {
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const unsigned row = (unsigned)tile * kRows + r0 + g + ((e >> 1) << 3);
                const int c = 2 * q + (e & 1);
                if (row < (unsigned)n && c < 3) y[e] = Y[(size_t)idx[row] * 3 + c];
            }
        }
        __syncthreads();
        float gp1[2][4], gp2[2][4], gp3[2][4], dh[2][4];
        train_hidden<1>(S.X, kLdX, f1, bias[0], S.H[0], gp1, r0, c0, lane);
        __syncthreads();
        train_hidden<4>(S.H[0], kLdH, f2, bias[1], S.H[1], gp2, r0, c0, lane);
        __syncthreads();
        train_hidden<4>(S.H[1], kLdH, f3, bias[2], S.H[2], gp3, r0, c0, lane);
        __syncthreads();
        if (outw) {
            float out[4] = {bias4.x, bias4.y, bias4.x, bias4.y}, dy[4];
#pragma unroll
            for (int t = 0; t < 4; t++) {
                uint32_t a[4];
                ldsm4(a, at_a(S.H[2], kLdH, r0, 16 * t, lane));
                mma(out, a, f4[t].x, f4[t].y);
            }
            // output gradient dY = 2 (P - Y) / (3 n_total), zero outside
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const unsigned row = (unsigned)tile * kRows + r0 + g + ((e >> 1) << 3);
                const int c = 2 * q + (e & 1);
                const float diff = row < (unsigned)n && c < 3 ? out[e] - y[e] : 0.f;
                dy[e] = scale * diff;
                lsum += diff * diff;
            }
            sb4[0] += dy[0] + dy[2];
            sb4[1] += dy[1] + dy[3];
            __nv_bfloat16* o = S.D4 + (r0 + g) * kLdX + 2 * q;
            *reinterpret_cast<uint32_t*>(o) = pack2(dy[0], dy[1]);
            *reinterpret_cast<uint32_t*>(o + 8 * kLdX) = pack2(dy[2], dy[3]);
        }
        __syncthreads();
        // dH3 = dY W4^T (k = the 8 outputs)
        {
            const __nv_bfloat16* d = S.D4 + (r0 + g) * kLdX + 2 * q;
            const uint32_t a[4] = {*reinterpret_cast<const uint32_t*>(d),
                                   *reinterpret_cast<const uint32_t*>(d + 8 * kLdX), 0u, 0u};
#pragma unroll
            for (int j = 0; j < 2; j++) {
                dh[j][0] = dh[j][1] = dh[j][2] = dh[j][3] = 0.f;
                mma(dh[j], a, t4[j].x, 0u);
            }
        }
        train_dz(dh, gp3, sb3, S.D[2], r0, c0, lane);
        __syncthreads();
        train_dh(dh, S.D[2], t3, r0, lane);
        train_dz(dh, gp2, sb2, S.D[1], r0, c0, lane);
        __syncthreads();
        train_dh(dh, S.D[1], t2, r0, lane);
        train_dz(dh, gp1, sb1, S.D[0], r0, c0, lane);
        __syncthreads();
        train_dw(dw3, S.H[1], S.D[2], m0, n0, lane);
        train_dw(dw2, S.H[0], S.D[1], m0, n0, lane);
#pragma unroll
        for (int k = 0; k < 2; k++) {
            uint32_t a[4], b0, b1;
            ldsm4t(a, at_at(S.X, kLdX, 16 * k, 0, lane));
            ldsm2t(b0, b1, at_b(S.D[0], kLdH, 16 * k, 8 * w, lane & 15));
            add_mma(dw1, a, b0, b1);
            if (w < 4) {
                ldsm4t(a, at_at(S.H[2], kLdH, 16 * k, m0, lane));
                ldsm2t(b0, b1, at_b(S.D4, kLdX, 16 * k, 0, lane & 15));
                add_mma(dw4, a, b0, b1);
            }
        }
    }
    // the block's part of the gradient
    float* P = part + (size_t)blockIdx.x * kPad;
    auto put = [&](float* G, int ld, int r, int c, const float(&v)[4]) {
        *reinterpret_cast<float2*>(&G[(r + g) * ld + c + 2 * q]) = make_float2(v[0], v[1]);
        *reinterpret_cast<float2*>(&G[(r + g + 8) * ld + c + 2 * q]) = make_float2(v[2], v[3]);
    };
#pragma unroll
    for (int j = 0; j < 4; j++) {
        put(P + kW2, 64, m0, n0 + 8 * j, dw2[j]);
        put(P + kW3, 64, m0, n0 + 8 * j, dw3[j]);
    }
    put(P + kW1, 64, 0, 8 * w, dw1);
    if (w < 4) put(P + kW4, 8, m0, 0, dw4);
    // bias gradients: over the rows of a warp, then over the two halves
    auto rows = [&](float v) {
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        return v + __shfl_xor_sync(0xffffffffu, v, 16);
    };
#pragma unroll
    for (int j = 0; j < 2; j++)
#pragma unroll
        for (int e = 0; e < 2; e++) {
            const float v1 = rows(sb1[j][e]), v2 = rows(sb2[j][e]), v3 = rows(sb3[j][e]);
            const int c = c0 + 8 * j + 2 * q + e;
            if (g == 0) {
                S.b[w & 1][c] = v1;
                S.b[w & 1][64 + c] = v2;
                S.b[w & 1][128 + c] = v3;
            }
        }
    if (outw) {
        const float v0 = rows(sb4[0]), v1 = rows(sb4[1]);
        if (g == 0) {
            S.b[w][192 + 2 * q] = v0;
            S.b[w][192 + 2 * q + 1] = v1;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0) S.loss[w] = lsum;
    }
    __syncthreads();
    if (threadIdx.x < 200) {
        const int k = threadIdx.x;
        const int at = k < 64 ? kB1 + k : k < 128 ? kB2 + k - 64 : k < 192 ? kB3 + k - 128 : kB4 + k - 192;
        P[at] = S.b[0][k] + S.b[1][k];
    }
    if (threadIdx.x == 0) lpart[blockIdx.x] = S.loss[0] + S.loss[1];
}

// Sum of the blocks' parts (8 warps per 32 parameters, in a fixed order), the
// batch's squared error added to *loss; then the gradient (kAdam false), or
// Adam on the padded FP32 master weights (padding stays zero) and the BF16
// fragments that the next batch reads.
template <bool kAdam>
__global__ void __launch_bounds__(256) k_mlp_update(const float* __restrict__ part, const float* __restrict__ lpart,
                                                    int np, float* __restrict__ loss, float* __restrict__ grad,
                                                    float* __restrict__ w, float* __restrict__ m,
                                                    float* __restrict__ v, TrainW* __restrict__ tw, float lr, float c1,
                                                    float c2) {
    __shared__ float red[8][32];
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31, i = blockIdx.x * 32 + lane;
    float sum = 0.f;
    if (i < kPad) {
#pragma unroll 8
        for (int b = k; b < np; b += 8) sum += part[(size_t)b * kPad + i];
    }
    red[k][lane] = sum;
    __syncthreads();
    if (k == 1 && blockIdx.x == 0) {
        float l = 0.f;
        for (int b = lane; b < np; b += 32) l += lpart[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) *loss += l;
    }
    if (k != 0 || i >= kPad) return;
    float gi = 0.f;
#pragma unroll
    for (int j = 0; j < 8; j++) gi += red[j][lane];
    if (!kAdam) {
        grad[i] = gi;
        return;
    }
    const bool pad = (i < kB1 && (i - kW1) / 64 >= 12) || (i >= kW4 && i < kB4 && (i - kW4) % 8 >= 3) ||
                     (i >= kB4 && i - kB4 >= 3);
    float wi = 0.f;
    if (!pad) {
        const float mi = 0.9f * m[i] + 0.1f * gi;
        const float vi = 0.999f * v[i] + 0.001f * gi * gi;
        m[i] = mi;
        v[i] = vi;
        wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    }
    w[i] = wi;
    put_weight(*tw, i, wi);
}

__global__ void k_mlp_train_weights(const float* __restrict__ w, TrainW* __restrict__ tw) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kPad) put_weight(*tw, i, w[i]);
}

// ---- FP32 debug gradient (canonical layout, no BF16 rounding) ----
// One thread per row: forward and backward of the network in plain FP32
// (inputs, weights, activations and accumulation), products summed in index
// order; the row's gradient of the mean squared error goes to G[row][9347].
// A second launch sums the rows in row order, one thread per parameter, so
// the result does not depend on scheduling.
constexpr int kCW1 = 0, kCB1 = 12 * 64, kCW2 = kCB1 + 64, kCB2 = kCW2 + 64 * 64, kCW3 = kCB2 + 64,
              kCB3 = kCW3 + 64 * 64, kCW4 = kCB3 + 64, kCB4 = kCW4 + 64 * 3, kCN = kCB4 + 3;
static_assert(kCN == 9347, "canonical parameter count");

__device__ __forceinline__ float gelu_grad_f32(float z) {
    const float t = tanhf(kGeluC * (z + 0.044715f * z * z * z));
    return 0.5f * (1.f + t) + 0.5f * z * (1.f - t * t) * kGeluC * (1.f + 3.f * 0.044715f * z * z);
}

__global__ void __launch_bounds__(64) k_mlp_grad_rows_f32(const float* __restrict__ w,
                                                           const float* __restrict__ X,
                                                           const float* __restrict__ Y, int n,
                                                           float* __restrict__ G,
                                                           float* __restrict__ lrow) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    float x[12], z1[64], z2[64], z3[64], h1[64], h2[64], h3[64], pr[3], dy[3];
    for (int k = 0; k < 12; k++) x[k] = X[(size_t)r * 12 + k];
    const int inW[3] = {kCW1, kCW2, kCW3}, inB[3] = {kCB1, kCB2, kCB3}, fan[3] = {12, 64, 64};
    float* zs[3] = {z1, z2, z3};
    float* hs[3] = {h1, h2, h3};
    const float* in = x;
    for (int L = 0; L < 3; L++) {
        for (int j = 0; j < 64; j++) {
            float a = w[inB[L] + j];
            for (int k = 0; k < fan[L]; k++) a = fmaf(in[k], w[inW[L] + k * 64 + j], a);
            zs[L][j] = a;
            hs[L][j] = gelu(a);
        }
        in = hs[L];
    }
    float ls = 0.f;
    for (int c = 0; c < 3; c++) {
        float a = w[kCB4 + c];
        for (int k = 0; k < 64; k++) a = fmaf(h3[k], w[kCW4 + k * 3 + c], a);
        pr[c] = a;
        const float d = a - Y[(size_t)r * 3 + c];
        ls = fmaf(d, d, ls);
        dy[c] = 2.f * d / (3.f * (float)n);
    }
    lrow[r] = ls;
    float* g = G + (size_t)r * kCN;
    for (int c = 0; c < 3; c++) g[kCB4 + c] = dy[c];
    for (int k = 0; k < 64; k++)
        for (int c = 0; c < 3; c++) g[kCW4 + k * 3 + c] = h3[k] * dy[c];
    // layer 3: dZ3 = (W4 dy) * gelu'(Z3), kept in z3
    for (int j = 0; j < 64; j++) {
        float a = 0.f;
        for (int c = 0; c < 3; c++) a = fmaf(w[kCW4 + j * 3 + c], dy[c], a);
        z3[j] = a * gelu_grad_f32(z3[j]);
    }
    // layers 3, 2, 1: weight and bias gradients, then the previous layer's dZ
    const float* dz = z3;
    for (int L = 2; L >= 0; L--) {
        const float* prev = L == 0 ? x : hs[L - 1];
        for (int j = 0; j < 64; j++) g[inB[L] + j] = dz[j];
        for (int k = 0; k < fan[L]; k++)
            for (int j = 0; j < 64; j++) g[inW[L] + k * 64 + j] = prev[k] * dz[j];
        if (L > 0) {
            float* zp = zs[L - 1];
            for (int k = 0; k < 64; k++) {
                float a = 0.f;
                for (int j = 0; j < 64; j++) a = fmaf(w[inW[L] + k * 64 + j], dz[j], a);
                zp[k] = a * gelu_grad_f32(zp[k]);
            }
            dz = zp;
        }
    }
}

__global__ void __launch_bounds__(256) k_mlp_grad_sum_f32(const float* __restrict__ G,
                                                          const float* __restrict__ lrow, int n,
                                                          float* __restrict__ grad, float* __restrict__ loss) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < kCN) {
        float a = 0.f;
        for (int r = 0; r < n; r++) a += G[(size_t)r * kCN + j];
        grad[j] = a;
    }
    if (j == 0) {
        float l = 0.f;
        for (int r = 0; r < n; r++) l += lrow[r];
        *loss = l / (3.f * (float)n);
    }
}

// ---- requests (target slot, image, cell entry) ----

struct CellView {
    double px, py, pz;      // target point (target minus image offset)
    double cx, cy, cz, M, w;
    double Q[6];
    int first, count, level, slot, code;
};

__device__ void req_view(const ReqArgs& A, uint64_t r, CellView& v) {
    v.slot = (int)(r >> 40);
    v.code = (int)((r >> 28) & 0xFFFull);
    const int e = (int)(r & 0xFFFFFFFull);
    const int gx = (v.code & 15) - 7, gy = ((v.code >> 4) & 15) - 7, gz = ((v.code >> 8) & 15) - 7;
    const BoxP bp = A.boxes[A.box[v.slot]];
    const double s = shear_offset(bp, time_of(A.ctl, A.t0, A.half_dt, A.hs));
    double ox, oy, oz;
    image_offset(bp, s, gx, gy, gz, ox, oy, oz);
    v.px = A.x[v.slot] - ox;
    v.py = A.y[v.slot] - oy;
    v.pz = A.z[v.slot] - oz;
    const double4_32a a = A.d_a[e], q0 = A.d_q0[e], q1 = A.d_q1[e];
    v.cx = a.x; v.cy = a.y; v.cz = a.z;
    v.M = q0.x;
    v.Q[0] = q0.y; v.Q[1] = q0.z; v.Q[2] = q0.w; v.Q[3] = q1.x; v.Q[4] = q1.y; v.Q[5] = q1.z;
    v.w = q1.w;
    v.first = A.e_first[e];
    v.count = A.e_count[e];
    v.level = A.e_level[e];
}

// The 12 network inputs (see the oracle's definition) and R^2 = |p - com|^2.
__device__ void req_features(const ReqArgs& A, const CellView& v, float* f, double& R2) {
    const double rx = v.px - v.cx, ry = v.py - v.cy, rz = v.pz - v.cz;
    R2 = rx * rx + ry * ry + rz * rz;
    const double R = sqrt(R2);
    const double hx = rx / R, hy = ry / R, hz = rz / R;
    const BoxP bp = A.boxes[A.box[v.first]];
    const double lo = -0.5 * bp.L;
    const uint64_t key = A.key[v.first];
    const int sh = kMaxDepth - v.level;
    const double ix = (double)(morton_compact3(key >> 2) >> sh);
    const double iy = (double)(morton_compact3(key >> 1) >> sh);
    const double iz = (double)(morton_compact3(key) >> sh);
    const double ccx = lo + (ix + 0.5) * v.w, ccy = lo + (iy + 0.5) * v.w, ccz = lo + (iz + 0.5) * v.w;
    const double sc = 1.0 / (v.M * v.w * v.w);
    const double qxx = v.Q[0] * sc, qyy = v.Q[1] * sc, qzz = v.Q[2] * sc;
    const double qxy = v.Q[3] * sc, qxz = v.Q[4] * sc, qyz = v.Q[5] * sc;
    const double ux = qxx * hx + qxy * hy + qxz * hz;
    const double uy = qxy * hx + qyy * hy + qyz * hz;
    const double uz = qxz * hx + qyz * hy + qzz * hz;
    f[0] = (float)hx; f[1] = (float)hy; f[2] = (float)hz;
    f[3] = (float)(v.w / R);
    f[4] = (float)log10((double)v.count);
    f[5] = (float)((v.cx - ccx) / v.w); f[6] = (float)((v.cy - ccy) / v.w); f[7] = (float)((v.cz - ccz) / v.w);
    f[8] = (float)(hx * ux + hy * uy + hz * uz);
    f[9] = (float)sqrt(ux * ux + uy * uy + uz * uz);
    f[10] = (float)(qxx * qxx + qyy * qyy + qzz * qzz + 2.0 * (qxy * qxy + qxz * qxz + qyz * qyz));
    f[11] = (float)(qxx * (qyy * qzz - qyz * qyz) - qxy * (qxy * qzz - qyz * qxz) +
                    qxz * (qxy * qyz - qyy * qxz));
}

// Residual labels: (exact cell force - multipole force) / (G M / R^2); the
// exact force is Eq. 1 summed over the cell's particles by one warp.
__global__ void __launch_bounds__(256) k_mlp_label(ReqArgs A, float* __restrict__ X,
                                                   float* __restrict__ Y, int64_t* __restrict__ meta) {
    const int nreq = min(*A.req_count, A.req_cap);
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int r = warp; r < nreq; r += nwarps) {
        CellView v;
        req_view(A, A.req[r], v);
        double sx = 0.0, sy = 0.0, sz = 0.0;
        int minid = 0x7fffffff;
        for (int j = v.first + lane; j < v.first + v.count; j += 32) {
            const double dx = A.x[j] - v.px, dy = A.y[j] - v.py, dz = A.z[j] - v.pz;
            const double r2 = dx * dx + dy * dy + dz * dz;
            const double inv = 1.0 / sqrt(r2);
            const double f = source_mass(A.boxes[A.box[j]], A.id[j], A.m[j]) * inv * inv * inv;
            sx += f * dx;
            sy += f * dy;
            sz += f * dz;
            minid = min(minid, A.id[j]);
        }
        for (int o = 16; o > 0; o >>= 1) {
            sx += __shfl_down_sync(0xffffffffu, sx, o);
            sy += __shfl_down_sync(0xffffffffu, sy, o);
            sz += __shfl_down_sync(0xffffffffu, sz, o);
            minid = min(minid, __shfl_down_sync(0xffffffffu, minid, o));
        }
        if (lane == 0) {
            float f[12];
            double R2;
            req_features(A, v, f, R2);
            // multipole force of the cell (monopole + quadrupole, unsoftened)
            const double dx = v.cx - v.px, dy = v.cy - v.py, dz = v.cz - v.pz;
            const double inv = 1.0 / sqrt(R2);
            const double inv3 = inv * inv * inv, inv5 = inv3 * inv * inv;
            const double qx = v.Q[0] * dx + v.Q[3] * dy + v.Q[4] * dz;
            const double qy = v.Q[3] * dx + v.Q[1] * dy + v.Q[5] * dz;
            const double qz = v.Q[4] * dx + v.Q[5] * dy + v.Q[2] * dz;
            const double dqd = dx * qx + dy * qy + dz * qz;
            const double c = 2.5 * dqd * inv5 * inv * inv;
            const double mx = v.M * inv3 * dx + c * dx - inv5 * qx;
            const double my = v.M * inv3 * dy + c * dy - inv5 * qy;
            const double mz = v.M * inv3 * dz + c * dz - inv5 * qz;
            const double unit = v.M / R2;   // G cancels
            for (int k = 0; k < 12; k++) X[(size_t)r * 12 + k] = f[k];
            Y[(size_t)r * 3 + 0] = (float)((sx - mx) / unit);
            Y[(size_t)r * 3 + 1] = (float)((sy - my) / unit);
            Y[(size_t)r * 3 + 2] = (float)((sz - mz) / unit);
            if (meta) {
                meta[(size_t)r * 5 + 0] = A.id[v.slot];
                meta[(size_t)r * 5 + 1] = v.code;
                meta[(size_t)r * 5 + 2] = v.level;
                meta[(size_t)r * 5 + 3] = minid;
                meta[(size_t)r * 5 + 4] = v.count;
            }
        }
    }
}

// Inference layout (Packed) of the padded FP32 weights: one thread per B
// fragment entry, then the biases.
__global__ void k_mlp_pack(const float* __restrict__ w, Packed* __restrict__ P) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    constexpr int n1 = 8 * 32, n2 = 32 * 32, n4 = 4 * 32;
    if (i < n1 + 2 * n2 + n4) {
        int k = i, off, ld, nt;
        uint2* dst;
        if (k < n1) {
            off = kW1; ld = 64; nt = 8; dst = reinterpret_cast<uint2*>(P->B1);
        } else if ((k -= n1) < n2) {
            off = kW2; ld = 64; nt = 8; dst = reinterpret_cast<uint2*>(P->B2);
        } else if ((k -= n2) < n2) {
            off = kW3; ld = 64; nt = 8; dst = reinterpret_cast<uint2*>(P->B3);
        } else {
            k -= n2;
            off = kW4; ld = 8; nt = 1; dst = reinterpret_cast<uint2*>(P->B4);
        }
        const int lane = k & 31, tile = k >> 5, t = tile / nt, j = tile % nt;
        const int g = lane >> 2, q = lane & 3, r = 16 * t + 2 * q, c = 8 * j + g;
        const float* W = w + off;
        uint2 b;
        b.x = pack2(W[r * ld + c], W[(r + 1) * ld + c]);
        b.y = pack2(W[(r + 8) * ld + c], W[(r + 9) * ld + c]);
        dst[nt == 1 ? k : ((t * 4 + (j >> 1)) * 32 + lane) * 2 + (j & 1)] = b;
    } else if ((i -= n1 + 2 * n2 + n4) < 200) {
        if (i < 64) P->b1[i] = w[kB1 + i];
        else if (i < 128) P->b2[i - 64] = w[kB2 + i - 64];
        else if (i < 192) P->b3[i - 128] = w[kB3 + i - 128];
        else P->b4[i - 192] = w[kB4 + i - 192];
    }
}

}  // namespace

void label_async(const ReqArgs& A, float* X, float* Y, int64_t* meta, int max_req, cudaStream_t s) {
    const int blocks = std::max(1, std::min((max_req + 7) / 8, 8 * 152));
    k_mlp_label<<<blocks, 256, 0, s>>>(A, X, Y, meta);
}

void pack_async(const float* w, Packed* packed, cudaStream_t s) {
    constexpr int n = 8 * 32 + 2 * 32 * 32 + 4 * 32 + 200;
    k_mlp_pack<<<(n + 255) / 256, 256, 0, s>>>(w, packed);
}

// ---- host helpers ----

int padded_size() { return kPad; }

// canonical (9347) <-> padded (9928)
void to_padded(const float* c, float* p) {
    std::fill(p, p + kPad, 0.f);
    int k = 0;
    const int in[4] = {12, 64, 64, 64}, out[4] = {64, 64, 64, 3};
    const int offw[4] = {kW1, kW2, kW3, kW4}, offb[4] = {kB1, kB2, kB3, kB4};
    const int ldp[4] = {64, 64, 64, 8};
    for (int L = 0; L < 4; L++) {
        for (int i = 0; i < in[L]; i++)
            for (int o = 0; o < out[L]; o++) p[offw[L] + i * ldp[L] + o] = c[k++];
        for (int o = 0; o < out[L]; o++) p[offb[L] + o] = c[k++];
    }
}

void from_padded(const float* p, float* c) {
    int k = 0;
    const int in[4] = {12, 64, 64, 64}, out[4] = {64, 64, 64, 3};
    const int offw[4] = {kW1, kW2, kW3, kW4}, offb[4] = {kB1, kB2, kB3, kB4};
    const int ldp[4] = {64, 64, 64, 8};
    for (int L = 0; L < 4; L++) {
        for (int i = 0; i < in[L]; i++)
            for (int o = 0; o < out[L]; o++) c[k++] = p[offw[L] + i * ldp[L] + o];
        for (int o = 0; o < out[L]; o++) c[k++] = p[offb[L] + o];
    }
}

size_t train_weights_bytes() { return sizeof(TrainW); }

int grad_blocks(int n) { return std::max(1, std::min((n - 1) / kRows + 1, kMaxPartials)); }

size_t grad_part_floats(int n) { return (size_t)grad_blocks(n) * (kPad + 1); }

// The blocks' parts of the gradient of the mean squared error of the rows
// idx[0..n), with n_total as the mean's denominator, and their squared errors
// behind them.
static cudaError_t grad_parts(const void* tw, const float* wf, const float* X, const float* Y, const int32_t* idx,
                              int n, int n_total, float* part, cudaStream_t s) {
    const int nb = grad_blocks(n);
    k_mlp_grad<<<nb, 256, 0, s>>>(static_cast<const TrainW*>(tw), wf, X, Y, idx, n, n_total, part,
                                  part + (size_t)nb * kPad);
    return cudaGetLastError();
}

cudaError_t grad_async(const void* tw, const float* wf, const float* X, const float* Y, const int32_t* idx, int n,
                       int n_total, float* part, float* grad, float* loss, cudaStream_t s) {
    const cudaError_t e = grad_parts(tw, wf, X, Y, idx, n, n_total, part, s);
    if (e != cudaSuccess) return e;
    const int nb = grad_blocks(n);
    k_mlp_update<false><<<(kPad + 31) / 32, 256, 0, s>>>(part, part + (size_t)nb * kPad, nb, loss, grad, nullptr,
                                                         nullptr, nullptr, nullptr, 0.f, 1.f, 1.f);
    return cudaGetLastError();
}

cudaError_t adam_step_async(float* w, float* m, float* v, void* tw, const float* X, const float* Y,
                            const int32_t* idx, int n, float lr, int step, float* part, float* loss,
                            cudaStream_t s) {
    const cudaError_t e = grad_parts(tw, w, X, Y, idx, n, n, part, s);
    if (e != cudaSuccess) return e;
    const int nb = grad_blocks(n);
    const float c1 = 1.f - powf(0.9f, (float)step), c2 = 1.f - powf(0.999f, (float)step);
    k_mlp_update<true><<<(kPad + 31) / 32, 256, 0, s>>>(part, part + (size_t)nb * kPad, nb, loss, nullptr, w, m, v,
                                                        static_cast<TrainW*>(tw), lr, c1, c2);
    return cudaGetLastError();
}

cudaError_t grad_f32_async(const float* w, const float* X, const float* Y, int n, float* G, float* lrow,
                           float* grad, float* loss, cudaStream_t s) {
    k_mlp_grad_rows_f32<<<(n + 63) / 64, 64, 0, s>>>(w, X, Y, n, G, lrow);
    k_mlp_grad_sum_f32<<<(kCN + 255) / 256, 256, 0, s>>>(G, lrow, n, grad, loss);
    return cudaGetLastError();
}

void train_weights_async(const float* w, void* tw, cudaStream_t s) {
    cudaMemsetAsync(tw, 0, sizeof(TrainW), s);   // the rows of W4^T's tiles beyond the 8 outputs
    k_mlp_train_weights<<<(kPad + 255) / 256, 256, 0, s>>>(w, static_cast<TrainW*>(tw));
}

}  // namespace mlp
}  // namespace rb
