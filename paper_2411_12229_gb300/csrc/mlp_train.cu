// mlp_train.cu -- training kernels of the learned early stop (not in the
// paper): a 16 -> 64 -> 64 -> 1 ReLU MLP over search-state features,
// trained with weighted binary cross-entropy and Adam.
//
// A block takes tiles of 64 samples and runs each as small dense products in
// shared memory:
//   forward  A1 = X W1^T + b1, H1 = relu(A1), A2 = H1 W2^T + b2,
//            H2 = relu(A2), z = H2 W3 + b3
//   backward dz = w (sigmoid(z) - y) / sum(w), D2 = (dz W3^T) .* [A2 > 0],
//            D1 = (D2 W2) .* [A1 > 0]
//   grads    W3: H2^T dz, W2: D2^T H1, W1: D1^T X, biases: column sums
// The gradient stays in registers over the block's tiles and is added to the
// global one with atomics at the end.
//
// What bounds it: in fp32 the products are 14,400 multiply-adds per sample
// (8,192 samples: 3.4 us on all SMs).  Every product gives a thread 4 x 4
// outputs from two 16-byte shared-memory reads per step of the inner
// dimension (operands kept both ways round where two products read them
// along different axes); one output per thread with two 4-byte reads per
// multiply-add, on 64 blocks of 128 samples, took 73 us; this one takes 17 us
// (8,192 samples: 128 blocks, one tile each; two warps per scheduler, so the
// barriers between the products are what is left).
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sqg.h"

namespace {

constexpr int kIn = SQG_MLP_IN, kH = SQG_MLP_HIDDEN, kTile = 64, kThreads = 256;
constexpr int oW1 = 0, ob1 = kH * kIn, oW2 = ob1 + kH, ob2 = oW2 + kH * kH, oW3 = ob2 + kH, ob3 = oW3 + kH;
constexpr int kLd = kH + 4;  // row pitch: 16-byte aligned, rows a bank quad apart

// [a][b]: a = row, b = contiguous.  i: input, h: first hidden layer, o: second
// hidden layer, r: sample.
struct TileSmem {
    float W1ih[kIn][kLd], W2ho[kH][kLd], W2oh[kH][kLd];
    float b1[kH], b2[kH], W3[kH];
    float Xir[kIn][kLd], Xri[kTile][kIn + 4];
    float H1hr[kH][kLd], H1rh[kTile][kLd];
    float D2or[kH][kLd], D2ro[kTile][kLd];
    float D1rh[kTile][kLd];
    float y[kTile], w[kTile];
};

__device__ __forceinline__ float softplus(float z) { return z > 0.f ? z + log1pf(expf(-z)) : log1pf(expf(z)); }

// The sum of the sample weights, and the gradient and the loss cleared for the
// atomics (one block, one launch before the gradient kernel).
constexpr int kPrepThreads = 1024;
__global__ void __launch_bounds__(kPrepThreads) prepare_kernel(const float *__restrict__ w, int n, float *wsum,
                                                               float *grad, float *loss) {
    __shared__ float part[kPrepThreads / 32];
    for (int i = threadIdx.x; i < SQG_MLP_NPARAM; i += kPrepThreads) grad[i] = 0.f;
    if (threadIdx.x == 0 && loss) *loss = 0.f;
    float s = 0.f;
#pragma unroll 8
    for (int i = threadIdx.x; i < n; i += kPrepThreads) s += w[i];
    for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        float t = part[threadIdx.x];
        for (int o = 16; o >= 1; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
        if (threadIdx.x == 0) *wsum = t;
    }
}

// The 4 x 4 values v to dst_ij[r0 + i][c0 + j] and / or dst_ji[c0 + j][r0 + i].
__device__ __forceinline__ void put4(float *dst_ij, float *dst_ji, const float (&v)[4][4], int r0, int c0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        *reinterpret_cast<float4 *>(dst_ij + (r0 + i) * kLd + c0) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
        if (dst_ji)
            *reinterpret_cast<float4 *>(dst_ji + (c0 + i) * kLd + r0) = make_float4(v[0][i], v[1][i], v[2][i], v[3][i]);
    }
}

// acc[i][j] += sum over k of A[k][a0 + i] B[k][b0 + j], k < K.
template <int K>
__device__ __forceinline__ void outer4(float (&acc)[4][4], const float *A, int a0, const float *B, int b0) {
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
        const float4 a = *reinterpret_cast<const float4 *>(A + k * kLd + a0);
        const float4 b = *reinterpret_cast<const float4 *>(B + k * kLd + b0);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
}

__global__ void __launch_bounds__(kThreads) mlp_grad_kernel(const float *__restrict__ P, const float *__restrict__ X,
                                                            const float *__restrict__ y, const float *__restrict__ w,
                                                            int n, const float *__restrict__ wsum,
                                                            float *__restrict__ G, float *__restrict__ loss) {
    extern __shared__ __align__(16) unsigned char raw[];
    TileSmem &s = *reinterpret_cast<TileSmem *>(raw);
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    for (int i = tid; i < kH * kIn; i += kThreads) s.W1ih[i % kIn][i / kIn] = P[oW1 + i];
    for (int i = tid; i < kH * kH; i += kThreads) {
        const float v = P[oW2 + i];
        s.W2oh[i / kH][i % kH] = v;
        s.W2ho[i % kH][i / kH] = v;
    }
    if (tid < kH) {
        s.b1[tid] = P[ob1 + tid];
        s.b2[tid] = P[ob2 + tid];
        s.W3[tid] = P[oW3 + tid];
    }
    const float b3 = P[ob3], inv_w = 1.0f / *wsum;
    // this thread's share of the gradient: W2 rows 4 ty + i, columns 4 tx + j;
    // W1 rows 4 ty + i, column tx; the vectors' entries 4 tx + j over the
    // samples 4 ty + i of every tile
    float gW2[4][4] = {}, gW1[4] = {}, gb1[4] = {}, gb2[4] = {}, gW3[4] = {}, gb3 = 0.f, lsum = 0.f;
    const int ntiles = (n + kTile - 1) / kTile;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int base = tile * kTile, rows = min(kTile, n - base);
        __syncthreads();  // the last tile's reads, and the weights
        for (int i = tid; i < kTile * kIn; i += kThreads) {
            const int r = i / kIn, c = i % kIn;
            const float v = r < rows ? X[(size_t)base * kIn + i] : 0.f;
            s.Xri[r][c] = v;
            s.Xir[c][r] = v;
        }
        if (tid < kTile) {
            s.y[tid] = tid < rows ? y[base + tid] : 0.f;
            s.w[tid] = tid < rows ? w[base + tid] * inv_w : 0.f;
        }
        __syncthreads();
        // A1, H1: samples 4 ty + i, units 4 tx + j
        {
            float a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = s.b1[4 * tx + j];
            outer4<kIn>(a, &s.Xir[0][0], 4 * ty, &s.W1ih[0][0], 4 * tx);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = a[i][j] > 0.f ? a[i][j] : 0.f;
            put4(&s.H1rh[0][0], &s.H1hr[0][0], a, 4 * ty, 4 * tx);
        }
        __syncthreads();
        // A2, z, dz, D2
        {
            float a[4][4], w3[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w3[j] = s.W3[4 * tx + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = s.b2[4 * tx + j];
            outer4<kH>(a, &s.H1hr[0][0], 4 * ty, &s.W2ho[0][0], 4 * tx);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 4 * ty + i;
                float p = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) p = fmaf(w3[j], a[i][j] > 0.f ? a[i][j] : 0.f, p);
#pragma unroll
                for (int o = 8; o >= 1; o >>= 1) p += __shfl_xor_sync(0xFFFFFFFFu, p, o);  // the 16 threads of a sample
                const float z = p + b3, yy = s.y[r], ww = s.w[r];
                // (an absent sample takes no part: its z may overflow where no real one does)
                const bool here = r < rows;
                const float dz = here ? ww * (1.0f / (1.0f + expf(-z)) - yy) : 0.f;
                if (tx == 0 && here) {
                    lsum += ww * (softplus(z) - yy * z);
                    gb3 += dz;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool on = here && a[i][j] > 0.f;
                    const float d2 = on ? dz * w3[j] : 0.f;
                    gW3[j] = fmaf(dz, on ? a[i][j] : 0.f, gW3[j]);
                    gb2[j] += d2;
                    a[i][j] = d2;
                }
            }
            put4(&s.D2ro[0][0], &s.D2or[0][0], a, 4 * ty, 4 * tx);
        }
        __syncthreads();
        outer4<kTile>(gW2, &s.D2ro[0][0], 4 * ty, &s.H1rh[0][0], 4 * tx);
        // D1: samples 4 ty + i, units 4 tx + j
        {
            float a[4][4] = {};
            outer4<kH>(a, &s.D2or[0][0], 4 * ty, &s.W2oh[0][0], 4 * tx);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    a[i][j] = s.H1rh[4 * ty + i][4 * tx + j] > 0.f ? a[i][j] : 0.f;
                    gb1[j] += a[i][j];
                }
            put4(&s.D1rh[0][0], nullptr, a, 4 * ty, 4 * tx);
        }
        __syncthreads();
#pragma unroll 8
        for (int r = 0; r < kTile; ++r) {
            const float4 d1 = *reinterpret_cast<const float4 *>(&s.D1rh[r][4 * ty]);
            const float x = s.Xri[r][tx];
            gW1[0] = fmaf(d1.x, x, gW1[0]);
            gW1[1] = fmaf(d1.y, x, gW1[1]);
            gW1[2] = fmaf(d1.z, x, gW1[2]);
            gW1[3] = fmaf(d1.w, x, gW1[3]);
        }
    }
    const bool aligned = reinterpret_cast<uintptr_t>(G) % 16 == 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float *g2 = G + oW2 + (4 * ty + i) * kH + 4 * tx;
        if (aligned) {
            atomicAdd(reinterpret_cast<float4 *>(g2), make_float4(gW2[i][0], gW2[i][1], gW2[i][2], gW2[i][3]));
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) atomicAdd(g2 + j, gW2[i][j]);
        }
        atomicAdd(&G[oW1 + (4 * ty + i) * kIn + tx], gW1[i]);
    }
    // the vectors: sums over ty through shared memory
    __syncthreads();
    float(*red)[3][kH] = reinterpret_cast<float(*)[3][kH]>(&s.H1hr[0][0]);  // [ty][vector][unit]
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        red[ty][0][4 * tx + j] = gb1[j];
        red[ty][1][4 * tx + j] = gb2[j];
        red[ty][2][4 * tx + j] = gW3[j];
    }
    if (tx == 0) {
        s.y[ty] = lsum;
        s.w[ty] = gb3;
    }
    __syncthreads();
    if (tid < 3 * kH) {
        const int v = tid / kH, u = tid % kH;
        float t = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) t += red[i][v][u];
        atomicAdd(&G[(v == 0 ? ob1 : v == 1 ? ob2 : oW3) + u], t);
    } else if (tid == 3 * kH) {
        float t = 0.f;
        for (int i = 0; i < 16; ++i) t += s.w[i];
        atomicAdd(&G[ob3], t);
    } else if (tid == 3 * kH + 32 && loss) {
        float t = 0.f;
        for (int i = 0; i < 16; ++i) t += s.y[i];
        atomicAdd(loss, t);
    }
}

__global__ void adam_kernel(float *P, const float *G, float *m, float *v, int n, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = G[i];
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

__global__ void __launch_bounds__(kThreads) mlp_forward_kernel(const float *__restrict__ P,
                                                               const float *__restrict__ X, int n,
                                                               float *__restrict__ z) {
    __shared__ float W[SQG_MLP_NPARAM];
    for (int i = threadIdx.x; i < SQG_MLP_NPARAM; i += blockDim.x) W[i] = P[i];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= n) return;
    float x[kIn];
    for (int c = 0; c < kIn; ++c) x[c] = X[(size_t)r * kIn + c];
    float ha = W[ob1 + lane], hb = W[ob1 + lane + 32];
    for (int c = 0; c < kIn; ++c) {
        ha = fmaf(W[oW1 + lane * kIn + c], x[c], ha);
        hb = fmaf(W[oW1 + (lane + 32) * kIn + c], x[c], hb);
    }
    ha = fmaxf(ha, 0.f);
    hb = fmaxf(hb, 0.f);
    float ga = W[ob2 + lane], gb = W[ob2 + lane + 32];
    for (int c = 0; c < kH; ++c) {
        float h = __shfl_sync(0xFFFFFFFFu, c < 32 ? ha : hb, c & 31);
        ga = fmaf(W[oW2 + lane * kH + c], h, ga);
        gb = fmaf(W[oW2 + (lane + 32) * kH + c], h, gb);
    }
    float p = W[oW3 + lane] * fmaxf(ga, 0.f) + W[oW3 + lane + 32] * fmaxf(gb, 0.f);
    for (int o = 16; o >= 1; o >>= 1) p += __shfl_xor_sync(0xFFFFFFFFu, p, o);
    if (lane == 0) z[r] = p + W[ob3];
}

}  // namespace

extern "C" int sqg_mlp_grad(const float *params, const float *x, const float *y, const float *w, int n,
                            float *grad, float *loss, float *scratch, sqg_stream_t stream_) {
    if (!params || !x || !y || !w || !grad || !scratch || n < 1) return SQG_ERR_INVALID_ARG;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    const size_t smem = sizeof(TileSmem);
    if (cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return SQG_ERR_CUDA;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return SQG_ERR_CUDA;
    const int tiles = (n + kTile - 1) / kTile;  // one block per SM holds the tile buffers
    prepare_kernel<<<1, kPrepThreads, 0, stream>>>(w, n, scratch, grad, loss);
    mlp_grad_kernel<<<tiles < sms ? tiles : sms, kThreads, smem, stream>>>(params, x, y, w, n, scratch, grad, loss);
    return cudaGetLastError() == cudaSuccess ? SQG_OK : SQG_ERR_CUDA;
}

extern "C" int sqg_mlp_adam(float *params, const float *grad, float *m, float *v, int step, float lr, float beta1,
                            float beta2, float eps, sqg_stream_t stream_) {
    if (!params || !grad || !m || !v || step < 1 || !(lr > 0.f)) return SQG_ERR_INVALID_ARG;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    adam_kernel<<<(SQG_MLP_NPARAM + 255) / 256, 256, 0, stream>>>(params, grad, m, v, SQG_MLP_NPARAM, lr, beta1,
                                                                  beta2, eps, c1, c2);
    return cudaGetLastError() == cudaSuccess ? SQG_OK : SQG_ERR_CUDA;
}

extern "C" int sqg_mlp_forward(const float *params, const float *x, int n, float *logits, sqg_stream_t stream_) {
    if (!params || !x || !logits || n < 0) return SQG_ERR_INVALID_ARG;
    if (n == 0) return SQG_OK;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    const int wpb = kThreads / 32;
    mlp_forward_kernel<<<(n + wpb - 1) / wpb, kThreads, 0, stream>>>(params, x, n, logits);
    return cudaGetLastError() == cudaSuccess ? SQG_OK : SQG_ERR_CUDA;
}
