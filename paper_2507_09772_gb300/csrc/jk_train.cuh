// Training kernels of the learned precision router (compiled by nvcc into the
// library). Parameters theta (FP32 master copy), flat:
//   W1[16][64] b1[64] W2[64][64] b2[64] W3[64] b3      (5,313 values)
// The forward pass rounds every weight and every layer input (normalised
// features, hidden activations) to BF16 (round to nearest even) and
// accumulates in FP32, as the tensor-core inference in the integral kernels
// does; the backward pass treats each rounding as the identity. The
// loss is the pinball (quantile) loss, which biases the prediction upwards so
// that a quartet is sent to FP32 only when its largest integral is confidently
// small.
#pragma once
#include "jk_router.cuh"

#include <algorithm>

#define JK_RT_OFF_W1 0
#define JK_RT_OFF_B1 (JK_RT_NINP * JK_RT_NH)
#define JK_RT_OFF_W2 (JK_RT_OFF_B1 + JK_RT_NH)
#define JK_RT_OFF_B2 (JK_RT_OFF_W2 + JK_RT_NH * JK_RT_NH)
#define JK_RT_OFF_W3 (JK_RT_OFF_B2 + JK_RT_NH)
#define JK_RT_OFF_B3 (JK_RT_OFF_W3 + JK_RT_NH)
#define JK_RT_NPARAM (JK_RT_OFF_B3 + 1)

__host__ __device__ inline unsigned short jk_f2bf(float f)
{
    unsigned u;
    memcpy(&u, &f, 4);
    if ((u & 0x7f800000u) == 0x7f800000u) return (unsigned short)(u >> 16);   // inf / nan
    u += 0x7fffu + ((u >> 16) & 1u);                                          // nearest even
    return (unsigned short)(u >> 16);
}
__host__ __device__ inline float jk_bf2f(unsigned short b)
{
    unsigned u = ((unsigned)b) << 16;
    float f;
    memcpy(&f, &u, 4);
    return f;
}

// One mini-batch: forward, pinball loss, backward. Sample t of the batch is row
// t of X (seed == JK_GRAD_ROWS) or a hashed one.
//
// Persistent CTAs of 256 threads take tiles of ROWS samples. The three 64 x 64
// products of a tile (hidden layer 2, its backward pass, the gradient of W2) are
// FP32 register tiles over shared memory, and the gradients stay in registers
// (20 per thread) until the CTA's last tile, one FP64 atomic per parameter and CTA.
// Bound by FP32 FMA issue and shared-memory reads: 50,000 rows are 1.5 GFLOP, 20
// us at the FP32 peak. A thread per sample, adding each of its 5,313 products to
// shared memory by atomics that all lanes of a warp aimed at one word, took
// 2.7 ms. Sums over inputs run in the same order as before, so the activations
// and the sign of the residual are the same.
#define JK_GRAD_ROWS 0xffffffffffffffffull
template <int ROWS> struct JkGradSmem {
    float w1[JK_RT_NIN * JK_RT_NH], w2[JK_RT_NH * JK_RT_NH], w2t[JK_RT_NH][JK_RT_NH + 4];
    float w3[JK_RT_NH], b1[JK_RT_NH], b2[JK_RT_NH], b3[4];
    float x[ROWS][JK_RT_NINP];
    float h1[ROWS][JK_RT_NH], h2[ROWS][JK_RT_NH], d[ROWS][JK_RT_NH];   // h2 becomes the first layer's delta
    float g[ROWS], yr[ROWS];
};
template <int ROWS>
__global__ void __launch_bounds__(256) jk_mlp_grad_kernel(const float *__restrict__ theta, const float *__restrict__ mu,
                                                          const float *__restrict__ isd, const float *__restrict__ X,
                                                          const float *__restrict__ y, long long n, int batch,
                                                          unsigned long long seed, float q, double *__restrict__ grad,
                                                          double *__restrict__ loss)
{
    constexpr int H = JK_RT_NH, RT = ROWS / 16;   // rows of a thread's tile
    extern __shared__ __align__(16) unsigned char jk_grad_smem[];
    JkGradSmem<ROWS> &S = *reinterpret_cast<JkGradSmem<ROWS> *>(jk_grad_smem);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int i = tid; i < JK_RT_NIN * H; i += 256) S.w1[i] = jk_bf2f(jk_f2bf(theta[JK_RT_OFF_W1 + i]));
    for (int i = tid; i < H * H; i += 256) {
        const float w = jk_bf2f(jk_f2bf(theta[JK_RT_OFF_W2 + i]));
        S.w2[i] = w;
        S.w2t[i % H][i / H] = w;
    }
    if (tid < H) {
        S.w3[tid] = jk_bf2f(jk_f2bf(theta[JK_RT_OFF_W3 + tid]));
        S.b1[tid] = theta[JK_RT_OFF_B1 + tid];
        S.b2[tid] = theta[JK_RT_OFF_B2 + tid];
        if (tid == 0) S.b3[0] = theta[JK_RT_OFF_B3];
    }
    float gw2[4][4] = {}, gw1[3] = {};
    double gvd = 0.0;   // w3, b2 or b1, summed tile by tile
    int below = 0, above = 0;   // one thread: rows with a negative residual and the others (b3)
    double lsum = 0.0;
    for (int t0 = blockIdx.x * ROWS; t0 < batch; t0 += gridDim.x * ROWS) {
        float gv = 0.0f;
        __syncthreads();
        // normalised features, rounded to BF16 (rows past the batch are zero and carry no weight)
        for (int i = tid; i < ROWS * JK_RT_NINP; i += 256) {
            const int r = i / JK_RT_NINP, k = i % JK_RT_NINP, t = t0 + r;
            float v = 0.0f;
            if (t < batch) {
                const long long row = seed == JK_GRAD_ROWS
                    ? (long long)t
                    : (long long)(jk_mix64(seed * 0x100000001b3ull + (unsigned long long)t) % (unsigned long long)n);
                if (k < JK_RT_NIN)
                    v = jk_bf2f(jk_f2bf(__fmul_rn(__fadd_rn(X[row * JK_RT_NIN + k], -mu[k]), isd[k])));
                else if (k == JK_RT_NIN) S.yr[r] = y[row];
            }
            S.x[r][k] = v;
        }
        __syncthreads();
        // layer 1: rows RT ty .., outputs 4 tx ..
        unsigned pos1 = 0;
        bool odd = false;   // a hidden value that is not finite
        {
            float a[RT][4];
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = S.b1[4 * tx + j];
#pragma unroll
            for (int k = 0; k < JK_RT_NIN; ++k) {
                const float4 w = *reinterpret_cast<const float4 *>(S.w1 + k * H + 4 * tx);
#pragma unroll
                for (int i = 0; i < RT; ++i) {
                    const float v = S.x[RT * ty + i][k];
                    a[i][0] = fmaf(v, w.x, a[i][0]); a[i][1] = fmaf(v, w.y, a[i][1]);
                    a[i][2] = fmaf(v, w.z, a[i][2]); a[i][3] = fmaf(v, w.w, a[i][3]);
                }
            }
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (a[i][j] > 0.0f) pos1 |= 1u << (4 * i + j);
                    const float h = jk_bf2f(jk_f2bf(fmaxf(a[i][j], 0.0f)));
                    odd = odd || !(fabsf(a[i][j]) <= 3.0e38f) || !(h <= 3.0e38f);
                    S.h1[RT * ty + i][4 * tx + j] = h;
                }
        }
        // features or hidden values that are not finite: products with a zero
        // delta count as zero, not as NaN (an inactive unit takes no gradient)
        const bool wild = __syncthreads_or(odd);
        // layer 2
        unsigned pos2 = 0;
        {
            float a[RT][4];
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] = S.b2[4 * tx + j];
#pragma unroll 4
            for (int k = 0; k < H; k += 4) {
                float4 w[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) w[m] = *reinterpret_cast<const float4 *>(S.w2 + (k + m) * H + 4 * tx);
#pragma unroll
                for (int i = 0; i < RT; ++i) {
                    const float4 h = *reinterpret_cast<const float4 *>(&S.h1[RT * ty + i][k]);
                    const float hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        a[i][0] = fmaf(hv[m], w[m].x, a[i][0]); a[i][1] = fmaf(hv[m], w[m].y, a[i][1]);
                        a[i][2] = fmaf(hv[m], w[m].z, a[i][2]); a[i][3] = fmaf(hv[m], w[m].w, a[i][3]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (a[i][j] > 0.0f) pos2 |= 1u << (4 * i + j);
                    S.h2[RT * ty + i][4 * tx + j] = jk_bf2f(jk_f2bf(fmaxf(a[i][j], 0.0f)));
                }
        }
        __syncthreads();
        // output, pinball loss u (q - [u < 0]) and its derivative
        if (tid < ROWS) {
            float out = S.b3[0];
#pragma unroll 8
            for (int o = 0; o < H; ++o) out = fmaf(S.h2[tid][o], S.w3[o], out);
            float gs = 0.0f;
            if (t0 + tid < batch) {
                const float u = S.yr[tid] - out;
                lsum += (double)(u >= 0.0f ? q * u : (q - 1.0f) * u);
                gs = ((u < 0.0f ? 1.0f : 0.0f) - q) / (float)batch;
            }
            S.g[tid] = gs;
        }
        __syncthreads();
        // delta of layer 2
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const float gs = S.g[RT * ty + i];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                S.d[RT * ty + i][4 * tx + j] = (pos2 >> (4 * i + j)) & 1u ? gs * S.w3[4 * tx + j] : 0.0f;
        }
        __syncthreads();
        // gradients of W2 (inputs 4 ty .., outputs 4 tx ..), W3, b2, b3
#pragma unroll 4
        for (int r = 0; r < ROWS; ++r) {
            const float4 h = *reinterpret_cast<const float4 *>(&S.h1[r][4 * ty]);
            const float4 d = *reinterpret_cast<const float4 *>(&S.d[r][4 * tx]);
            float hv[4] = {h.x, h.y, h.z, h.w};
            if (wild) {
                const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (dv[j] != 0.0f && hv[i] != 0.0f) gw2[i][j] = fmaf(hv[i], dv[j], gw2[i][j]);
                continue;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                gw2[i][0] = fmaf(hv[i], d.x, gw2[i][0]); gw2[i][1] = fmaf(hv[i], d.y, gw2[i][1]);
                gw2[i][2] = fmaf(hv[i], d.z, gw2[i][2]); gw2[i][3] = fmaf(hv[i], d.w, gw2[i][3]);
            }
        }
        if (tid < 64) {
#pragma unroll 4
            for (int r = 0; r < ROWS; ++r) gv = fmaf(S.g[r], S.h2[r][tid], gv);
        } else if (tid < 128) {
#pragma unroll 4
            for (int r = 0; r < ROWS; ++r) gv += S.d[r][tid - 64];
        } else if (tid == 192) {
#pragma unroll 4
            for (int r = 0; r < ROWS; ++r) {
                below += S.g[r] > 0.0f;
                above += S.g[r] < 0.0f;
            }
        }
        // delta of layer 1, into h2
        float dh[RT][4] = {};
#pragma unroll 4
        for (int k = 0; k < H; k += 4) {
            float4 w[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) w[m] = *reinterpret_cast<const float4 *>(&S.w2t[k + m][4 * tx]);
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const float4 d = *reinterpret_cast<const float4 *>(&S.d[RT * ty + i][k]);
                const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    dh[i][0] = fmaf(w[m].x, dv[m], dh[i][0]); dh[i][1] = fmaf(w[m].y, dv[m], dh[i][1]);
                    dh[i][2] = fmaf(w[m].z, dv[m], dh[i][2]); dh[i][3] = fmaf(w[m].w, dv[m], dh[i][3]);
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) S.h2[RT * ty + i][4 * tx + j] = (pos1 >> (4 * i + j)) & 1u ? dh[i][j] : 0.0f;
        __syncthreads();
        // gradients of W1 (inputs 3 (tid / 64) .., output tid % 64) and b1
        {
            const int o = tid & 63, k0 = 3 * (tid >> 6);
#pragma unroll 4
            for (int r = 0; r < ROWS; ++r) {
                const float d = S.h2[r][o];
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if (!wild || (d != 0.0f && S.x[r][k0 + k] != 0.0f)) gw1[k] = fmaf(S.x[r][k0 + k], d, gw1[k]);
                if (tid >= 128 && tid < 192) gv += d;
            }
        }
        gvd += (double)gv;
    }
    // b3: the derivative has two values, 1 - q and -q over the batch, which FP32
    // would add with the same rounding error every time
    if (tid == 192) gvd = (double)below * (double)((1.0f - q) / (float)batch) - (double)above * (double)(q / (float)batch);
    // one FP64 atomic per parameter and CTA
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (gw2[i][j] != 0.0f) atomicAdd(&grad[JK_RT_OFF_W2 + (4 * ty + i) * H + 4 * tx + j], (double)gw2[i][j]);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (gw1[k] != 0.0f) atomicAdd(&grad[JK_RT_OFF_W1 + (3 * (tid >> 6) + k) * H + (tid & 63)], (double)gw1[k]);
    if (gvd != 0.0) {
        const int at = tid < 64 ? JK_RT_OFF_W3 + tid
                                : (tid < 128 ? JK_RT_OFF_B2 + tid - 64 : (tid < 192 ? JK_RT_OFF_B1 + tid - 128 : JK_RT_OFF_B3));
        atomicAdd(&grad[at], gvd);
    }
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if ((tid & 31) == 0 && lsum != 0.0) atomicAdd(loss, lsum / batch);
}

// Tiles of 64 rows where they fill the GPU (more arithmetic per shared-memory
// read), of 16 below (a training step of 4,096 samples is 256 of them).
static cudaError_t jk_mlp_grad(const float *theta, const float *mu, const float *isd, const float *X, const float *y,
                               long long n, int batch, unsigned long long seed, float q, double *grad, double *loss,
                               int sms, cudaStream_t st)
{
    if ((batch + 63) / 64 >= sms) {
        const size_t sm = sizeof(JkGradSmem<64>);
        if (cudaError_t e = cudaFuncSetAttribute(jk_mlp_grad_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))
            return e;
        const int grid = std::min((batch + 63) / 64, 2 * sms);
        jk_mlp_grad_kernel<64><<<grid, 256, sm, st>>>(theta, mu, isd, X, y, n, batch, seed, q, grad, loss);
    } else {
        const size_t sm = sizeof(JkGradSmem<16>);
        if (cudaError_t e = cudaFuncSetAttribute(jk_mlp_grad_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))
            return e;
        const int grid = std::min((batch + 15) / 16, 2 * sms);
        jk_mlp_grad_kernel<16><<<grid, 256, sm, st>>>(theta, mu, isd, X, y, n, batch, seed, q, grad, loss);
    }
    return cudaGetLastError();
}

__global__ void jk_adam_kernel(float *__restrict__ theta, const double *__restrict__ grad, float *__restrict__ m1,
                               float *__restrict__ m2, int step, float lr, float b1, float b2, float eps)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= JK_RT_NPARAM) return;
    const float g = (float)grad[i];
    const float a = b1 * m1[i] + (1.0f - b1) * g;
    const float v = b2 * m2[i] + (1.0f - b2) * g * g;
    m1[i] = a;
    m2[i] = v;
    const float ah = a / (1.0f - powf(b1, (float)step));
    const float vh = v / (1.0f - powf(b2, (float)step));
    theta[i] -= lr * ah / (sqrtf(vh) + eps);
}

// Inference over a batch of feature rows with the device weights (the same
// warp-level tensor-core function the integral kernels call). Blocks of 128
// threads; rows past n are evaluated on zero features and not stored.
__global__ void __launch_bounds__(128) jk_mlp_forward_kernel(const JkRouterDev *__restrict__ R,
                                                             const float *__restrict__ X, long long n,
                                                             float *__restrict__ out)
{
    __shared__ __align__(16) unsigned short s_rsm[4 * 32 * JK_RT_NINP];
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    float x[JK_RT_NIN];
    for (int i = 0; i < JK_RT_NIN; ++i) x[i] = t < n ? X[t * JK_RT_NIN + i] : 0.0f;
    const float y = jk_router_warp(R, x, s_rsm + (threadIdx.x >> 5) * 32 * JK_RT_NINP);
    if (t < n) out[t] = y;
}
