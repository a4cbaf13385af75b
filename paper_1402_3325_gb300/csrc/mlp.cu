// mlp.cu -- data, training and evaluation kernels of the learned initial guess.
//
// Training data: for given ordered pairs of a system, the pair's Kepler solve
// is run with the FP64 solver (standard guess) and the features of
// mlp_infer.cuh and the target g = log(s / s_T2) / w are written.
//
// Training (FP32, the project's own kernels), two launches per minibatch:
//   tile kernel: forward and backward pass of 32 samples per block and the
//     block's sums of every gradient;
//   reduce kernel: the blocks' sums added in a fixed order (deterministic, no
//     atomics), then the gradient written or the bias-corrected Adam update
//     of the FP32 master parameters.
// Parameter layout (FP32): W1[64][6], b1[64], W2[64][64], b2[64], W3[64], b3.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>

#include "kepler_fp64.cuh"
#include "mlp_infer.cuh"
#include "pair_batch_fp64.cuh"
#include "step_common.cuh"

namespace sakura {

constexpr int kOffW1 = 0, kOffB1 = 384, kOffW2 = 448, kOffB2 = 4544, kOffW3 = 4608,
              kOffB3 = 4672;

// ---------------------------------------------------------------- data
__global__ void __launch_bounds__(128)
    sample_pairs_kernel(const double *X, int64_t n, double tau, double pre, const int64_t *ids,
                        int64_t count, float *feat, float *target, int *iters_out,
                        double tol, unsigned *status)
{
    const int lane = threadIdx.x & 31;
    const int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - lane;
    const int64_t k = base + lane;
    const bool valid_id = k < count;
    int64_t i = 0, j = 0;
    if (valid_id) {
        i = ids[k] / n;
        j = ids[k] - i * n;
    }
    const bool valid = valid_id && i != j && i >= 0 && i < n;
    PairSolve p;
    double s_t2 = 0.0;
    if (valid) {
        pair_setup(p, tau, X[6 * n + i] + X[6 * n + j], X[i] - X[j], X[n + i] - X[n + j],
                   X[2 * n + i] - X[2 * n + j], X[3 * n + i] - X[3 * n + j],
                   X[4 * n + i] - X[4 * n + j], X[5 * n + i] - X[5 * n + j], pre, 2);
        s_t2 = p.s;
        p.s = p.t * p.ir0;  // solve from the standard guess
    } else {
        p.done = true;
        p.beta = p.s = 0.0;
        p.iters = 0;
        p.status = 0;
    }
    const KeplerParams kp{tol, 50, 1};
    double d[6];
    int it = 0, fb = 0;
    fp64_solve_warp(p, valid, tau, (1.0 - pre) * tau, kp, d, it, fb);
    if (!valid_id) return;
    float f[6] = {0, 0, 0, 0, 0, 0}, w = 0.0f, tg = 0.0f;
    if (valid && guess_features(p.t, p.m, p.r0, p.ir0, p.eta0, p.beta, f, w) && w > 0.0f) {
        const double ratio = p.s / s_t2;
        tg = ratio > 0.0 ? (float)(log(ratio) / (double)w) : 0.0f;
    }
    for (int q = 0; q < 6; ++q) feat[k * 6 + q] = f[q];
    target[k] = tg;
    if (iters_out) iters_out[k] = it;
    if (valid && p.status) atomicOr(status, p.status);
}

// ------------------------------------------------------------- training
// Forward and backward pass of 32 samples at a time, with the tile's
// contribution to every gradient kept in the block's registers until the
// block's last tile; partial [gridDim.x][kMlpGradStride] receives each
// block's sums (the 4673 gradients, then the squared residuals).
//
// Bound: the three 32 x 64 x 64 products of a tile on the FP32 pipe, fed from
// shared memory.  A thread forms 2 x 4 (or 4 x 4) outputs and reads its
// operands as float4 along the summed index, so 6 (8) loads serve 32 (64)
// FMAs; rows are padded to 68 (36) floats, which spreads the 16 rows that a
// warp reads over the banks.  Each pre-activation is one chain of FMAs in
// ascending k from the bias.
// The kernels before took one thread per sample (activations in local memory
// and per-sample arrays in global memory) and one thread per weight walking
// the batch: 455 us per minibatch of 8192, the sums over the batch in
// one chain of 8192 roundings.
constexpr int kMlpTile = 32, kMlpThreads = 256;
constexpr int kMlpRow = 68, kMlpCol = 36;  // padded row lengths
constexpr int kMlpGradStride = 4736;       // floats of a block's sums, 4674 used

struct MlpSmem {
    float W2[64 * kMlpRow], W2T[64 * kMlpRow];           // [o][k], [k][o]
    float hS[kMlpTile * kMlpRow], dS[kMlpTile * kMlpRow];  // [s][k]: h1; h2, then dz2
    float hT[64 * kMlpCol], dT[64 * kMlpCol];            // [k][s]: h1; dz2, then dz1
    float x[kMlpTile * 8], W1[64 * 8], W3[64], b1[64], b2[64], g[kMlpTile], r2[kMlpTile];
};

__device__ __forceinline__ float dot4(float4 a, float4 b, float c)
{
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}

__global__ void __launch_bounds__(kMlpThreads)
    mlp_tile_kernel(const float *P, const float *norm, const float *feat, const float *target,
                    int64_t B, float *partial)
{
    extern __shared__ __align__(16) unsigned char msm[];
    MlpSmem &sm = *reinterpret_cast<MlpSmem *>(msm);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    griddep_wait();    // P from the update before, partial read by it
    griddep_launch();
    for (int e = tid; e < 4096; e += kMlpThreads) {
        const float w = P[kOffW2 + e];
        sm.W2[(e >> 6) * kMlpRow + (e & 63)] = w;
        sm.W2T[(e & 63) * kMlpRow + (e >> 6)] = w;
    }
    for (int e = tid; e < 384; e += kMlpThreads) sm.W1[(e / 6) * 8 + e % 6] = P[kOffW1 + e];
    if (tid < 64) {
        sm.W3[tid] = P[kOffW3 + tid];
        sm.b1[tid] = P[kOffB1 + tid];
        sm.b2[tid] = P[kOffB2 + tid];
    }
    const float b3 = P[kOffB3];
    // gradient sums: W2[ty + 16 i][tx + 16 j]; of the entries of one weight
    // or bias, thread tid's
    float gW2[4][4] = {}, gW1[2] = {0.0f, 0.0f}, gb = 0.0f, gW3 = 0.0f, gb3 = 0.0f, loss = 0.0f;
    for (int64_t t0 = (int64_t)blockIdx.x * kMlpTile; t0 < B;
         t0 += (int64_t)gridDim.x * kMlpTile) {
        __syncthreads();  // the weights; the previous tile's readers
        for (int e = tid; e < kMlpTile * 6; e += kMlpThreads) {
            const int s = e / 6, k = e - 6 * s;
            sm.x[s * 8 + k] = t0 + s < B ? (feat[t0 * 6 + e] - norm[k]) / norm[6 + k] : 0.0f;
        }
        __syncthreads();
        // h1: 8 units of one sample per thread
        {
            const int s = tid >> 3;
            for (int o = tid & 7; o < 64; o += 8) {
                float z = sm.b1[o];
#pragma unroll
                for (int k = 0; k < 6; ++k) z = fmaf(sm.W1[o * 8 + k], sm.x[s * 8 + k], z);
                const float h = tanhf(z);
                sm.hS[s * kMlpRow + o] = h;
                sm.hT[o * kMlpCol + s] = h;
            }
        }
        __syncthreads();
        // h2 of samples 2 ty, 2 ty + 1 and units tx + 16 i
        float z[2][4], h2[2][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) z[0][i] = z[1][i] = sm.b2[tx + 16 * i];
#pragma unroll 4
        for (int k = 0; k < 64; k += 4) {
            const float4 a0 = *(const float4 *)&sm.hS[(2 * ty) * kMlpRow + k];
            const float4 a1 = *(const float4 *)&sm.hS[(2 * ty + 1) * kMlpRow + k];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 w = *(const float4 *)&sm.W2[(tx + 16 * i) * kMlpRow + k];
                z[0][i] = dot4(w, a0, z[0][i]);
                z[1][i] = dot4(w, a1, z[1][i]);
            }
        }
        // y, the residual and dy: the 16 lanes of a half warp hold one sample's units
        float y[2] = {0.0f, 0.0f};
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                h2[u][i] = tanhf(z[u][i]);
                y[u] = fmaf(sm.W3[tx + 16 * i], h2[u][i], y[u]);
                sm.dS[(2 * ty + u) * kMlpRow + tx + 16 * i] = h2[u][i];
            }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            y[0] += __shfl_xor_sync(0xffffffffu, y[0], o);
            y[1] += __shfl_xor_sync(0xffffffffu, y[1], o);
        }
        float dy[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t b = t0 + 2 * ty + u;
            const float r = b < B ? y[u] + b3 - target[b] : 0.0f;
            dy[u] = 2.0f * r / (float)B;
            if (tx == 0) {
                sm.g[2 * ty + u] = dy[u];
                sm.r2[2 * ty + u] = r * r;
            }
        }
        __syncthreads();
        // dW3 (64 threads), db3 and the loss (one warp)
        if (tid < 64) {
            for (int s = 0; s < kMlpTile; ++s)
                gW3 = fmaf(sm.g[s], sm.dS[s * kMlpRow + tid], gW3);
        } else if (tid < 96) {
            gb3 += sm.g[tid - 64];
            loss += sm.r2[tid - 64];
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int o = tx + 16 * i;
                const float d2 = dy[u] * sm.W3[o] * (1.0f - h2[u][i] * h2[u][i]);
                sm.dS[(2 * ty + u) * kMlpRow + o] = d2;
                sm.dT[o * kMlpCol + 2 * ty + u] = d2;
            }
        __syncthreads();
        // dW2[ty + 16 i][tx + 16 j], db2
#pragma unroll 2
        for (int s = 0; s < kMlpTile; s += 4) {
            float4 a[4], h[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = *(const float4 *)&sm.dT[(ty + 16 * i) * kMlpCol + s];
                h[i] = *(const float4 *)&sm.hT[(tx + 16 * i) * kMlpCol + s];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) gW2[i][j] = dot4(a[i], h[j], gW2[i][j]);
        }
        if (tid >= 64 && tid < 128)
            for (int s = 0; s < kMlpTile; ++s) gb += sm.dT[(tid - 64) * kMlpCol + s];
        // dh1 of samples 2 ty, 2 ty + 1 and units tx + 16 i
        float d1[2][4] = {};
#pragma unroll 4
        for (int o = 0; o < 64; o += 4) {
            const float4 a0 = *(const float4 *)&sm.dS[(2 * ty) * kMlpRow + o];
            const float4 a1 = *(const float4 *)&sm.dS[(2 * ty + 1) * kMlpRow + o];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 w = *(const float4 *)&sm.W2T[(tx + 16 * i) * kMlpRow + o];
                d1[0][i] = dot4(w, a0, d1[0][i]);
                d1[1][i] = dot4(w, a1, d1[1][i]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = tx + 16 * i;
                const float h = sm.hS[(2 * ty + u) * kMlpRow + k];
                sm.dT[k * kMlpCol + 2 * ty + u] = d1[u][i] * (1.0f - h * h);
            }
        __syncthreads();
        // dW1 (entries tid and 256 + tid), db1
        if (tid < 64)
            for (int s = 0; s < kMlpTile; ++s) gb += sm.dT[tid * kMlpCol + s];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = tid + 256 * q;
            if (e < 384)
                for (int s = 0; s < kMlpTile; ++s)
                    gW1[q] = fmaf(sm.dT[(e / 6) * kMlpCol + s], sm.x[s * 8 + e % 6], gW1[q]);
        }
    }
    float *out = partial + (int64_t)blockIdx.x * kMlpGradStride;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) out[kOffW2 + (ty + 16 * i) * 64 + tx + 16 * j] = gW2[i][j];
    out[kOffW1 + tid] = gW1[0];
    if (tid + 256 < 384) out[kOffW1 + tid + 256] = gW1[1];
    if (tid < 64) {
        out[kOffB1 + tid] = gb;
        out[kOffW3 + tid] = gW3;
    } else if (tid < 128) {
        out[kOffB2 + tid - 64] = gb;
    }
    if (tid >= 64 && tid < 96) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
            loss += __shfl_xor_sync(0xffffffffu, loss, o);
        }
        if (tid == 64) {
            out[kOffB3] = gb3;
            out[kMlpParams] = loss;
        }
    }
}

// Sums of the blocks' gradients: 32 entries per block of 256 threads, each
// of its 8 warps taking every eighth partial, the warps' sums added in warp
// order.  Then either the gradient is written (grad) or, in training, one
// Adam step taken (m, v; bias corrections 1 - b1t, 1 - b2t).
__global__ void __launch_bounds__(256)
    mlp_reduce_kernel(const float *partial, int blocks, int64_t B, float *grad, float *loss,
                      float *P, float *m, float *v, float lr, float b1t, float b2t)
{
    __shared__ float red[8][32];
    griddep_wait();
    griddep_launch();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int p = blockIdx.x * 32 + lane;
    float s0 = 0.0f, s1 = 0.0f;
    if (p <= kMlpParams) {
        int b = w;
        for (; b + 8 < blocks; b += 16) {
            s0 += partial[(int64_t)b * kMlpGradStride + p];
            s1 += partial[(int64_t)(b + 8) * kMlpGradStride + p];
        }
        if (b < blocks) s0 += partial[(int64_t)b * kMlpGradStride + p];
    }
    red[w][lane] = s0 + s1;
    __syncthreads();
    if (w != 0 || p > kMlpParams) return;
    float gi = red[0][lane];
#pragma unroll
    for (int k = 1; k < 8; ++k) gi += red[k][lane];
    if (p == kMlpParams) {
        *loss = gi / (float)B;
        return;
    }
    if (grad) {
        grad[p] = gi;
        return;
    }
    const float b1 = 0.9f, b2 = 0.999f;
    const float mi = b1 * m[p] + (1.0f - b1) * gi;
    const float vi = b2 * v[p] + (1.0f - b2) * gi * gi;
    m[p] = mi;
    v[p] = vi;
    const float mh = mi / (1.0f - b1t), vh = vi / (1.0f - b2t);
    P[p] -= lr * mh / (sqrtf(vh) + 1e-8f);
}

// ------------------------------------------------------------ inference
__global__ void mlp_eval_kernel(const MlpWeights *Wg, const float *feat, int64_t count,
                                float *out)
{
    __shared__ MlpWeights W;
    __shared__ __nv_bfloat16 stage[4][32 * 16];
    mlp_load_shared(W, Wg);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float f[6] = {0, 0, 0, 0, 0, 0};
    if (k < count)
        for (int q = 0; q < 6; ++q) f[q] = feat[k * 6 + q];
    const float g = mlp_eval_warp(W, stage[wib], f);
    (void)lane;
    if (k < count) out[k] = g;
}

// blob (host FP32, kMlpBlob floats) -> device MlpWeights (BF16 weights)
__global__ void mlp_pack_kernel(const float *blob, MlpWeights *W)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const float *P = blob;
    if (t < 64 * 16) {
        const int n = t / 16, k = t % 16;
        W->W1[t] = __float2bfloat16_rn(k < 6 ? P[kOffW1 + n * 6 + k] : 0.0f);
    }
    if (t < 64 * 64) W->W2[t] = __float2bfloat16_rn(P[kOffW2 + t]);
    if (t < 8 * 64) {
        const int n = t / 64, k = t % 64;
        W->W3[t] = __float2bfloat16_rn(n == 0 ? P[kOffW3 + k] : 0.0f);
    }
    if (t < 64) {
        W->b1[t] = P[kOffB1 + t];
        W->b2[t] = P[kOffB2 + t];
    }
    if (t < 6) {
        W->mean[t] = P[kMlpParams + t];
        W->inv_scale[t] = 1.0f / P[kMlpParams + 6 + t];
    }
    if (t == 0) {
        W->b3 = P[kOffB3];
        W->oscale = P[kMlpParams + 12];
        W->oshift = P[kMlpParams + 13];
    }
}

// --------------------------------------------------------------- launchers
void launch_sample_pairs(const double *X, int64_t n, double tau, double pre, const int64_t *ids,
                         int64_t count, float *feat, float *target, int *iters, double tol,
                         unsigned *status, cudaStream_t s)
{
    const int64_t blocks = (count + 127) / 128;
    sample_pairs_kernel<<<(unsigned)blocks, 128, 0, s>>>(X, n, tau, pre, ids, count, feat, target,
                                                         iters, tol, status);
}

namespace {

// one tile of 32 samples per block, up to two blocks' worth per SM (a block's
// sums are 19 KB of scratch)
int mlp_blocks(int64_t B)
{
    const int64_t tiles = (B + kMlpTile - 1) / kMlpTile;
    return (int)(tiles < 304 ? tiles : 304);
}

}  // namespace

void launch_mlp_step(float *P, const float *norm, const float *feat, const float *target,
                     int64_t B, float *scratch, float *grad, float *loss, float *m, float *v,
                     float lr, float b1t, float b2t, cudaStream_t s)
{
    int blocks = mlp_blocks(B);
    const size_t smem = sizeof(MlpSmem);
    cudaFuncSetAttribute((const void *)mlp_tile_kernel,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const float *Pc = P;
    void *a1[] = {(void *)&Pc, (void *)&norm, (void *)&feat, (void *)&target, (void *)&B,
                  (void *)&scratch};
    launch_pdl((const void *)mlp_tile_kernel, dim3(blocks), dim3(kMlpThreads), a1, smem, s);
    const float *part = scratch;
    void *a2[] = {(void *)&part, (void *)&blocks, (void *)&B, (void *)&grad, (void *)&loss,
                  (void *)&P,    (void *)&m,      (void *)&v, (void *)&lr,   (void *)&b1t,
                  (void *)&b2t};
    launch_pdl((const void *)mlp_reduce_kernel, dim3((kMlpParams + 1 + 31) / 32), dim3(256), a2, 0,
               s);
}

size_t mlp_grad_scratch_floats(int64_t B) { return (size_t)mlp_blocks(B) * kMlpGradStride; }

void launch_mlp_pack(const float *blob, MlpWeights *W, cudaStream_t s)
{
    mlp_pack_kernel<<<(64 * 64 + 127) / 128, 128, 0, s>>>(blob, W);
}

void launch_mlp_eval(const MlpWeights *W, const float *feat, int64_t count, float *out,
                     cudaStream_t s)
{
    mlp_eval_kernel<<<(unsigned)((count + 127) / 128), 128, 0, s>>>(W, feat, count, out);
}

}  // namespace sakura
