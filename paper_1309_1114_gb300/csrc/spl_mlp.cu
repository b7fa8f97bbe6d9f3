// spl_mlp.cu -- the tile-cost network, its inference and training kernels.
//
// 32 -> 64 (ReLU) -> 1 in FP32: y = w2 . relu(W1 x + b1) + b2, trained on
// the render's own per-item timings to predict log(SM cycles).  Loss: mean
// squared error over a batch; gradients by the chain rule through the ReLU;
// optimiser: Adam (Kingma & Ba, Algorithm 1).  The paper has no counterpart:
// it only observes the load imbalance that this network's predictions are
// used to reduce (Sec. 4 Remarks).
#include <cmath>

#include "spl_internal.cuh"

namespace spl {

// y[b] for every sample, one thread each; weights in shared memory.
__global__ void __launch_bounds__(256) mlp_forward_kernel(const float *theta, const float *x,
                                                          int64_t B, float *y) {
    __shared__ float w[kNParam];
    for (int k = threadIdx.x; k < kNParam; k += blockDim.x) w[k] = theta[k];
    __syncthreads();
    const float *W1 = w, *b1 = w + kHid * kFeat, *w2 = b1 + kHid, *b2 = w2 + kHid;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < B;
         b += (int64_t)gridDim.x * blockDim.x) {
        float xv[kFeat];
#pragma unroll
        for (int i = 0; i < kFeat; ++i) xv[i] = x[b * kFeat + i];
        float out = b2[0];
        for (int j = 0; j < kHid; ++j) {
            float z = b1[j];
#pragma unroll
            for (int i = 0; i < kFeat; ++i) z = fmaf(W1[j * kFeat + i], xv[i], z);
            if (z > 0.f) out = fmaf(w2[j], z, out);
        }
        y[b] = out;
    }
}

// Gradient of the loss over a batch, in one pass over the samples.  A CTA takes
// tiles of kGradTile samples: the forward pass as a register-tiled product of the
// staged samples and W1 (a thread: 4 samples x 4 hidden units), the residuals by
// shuffles over a sample's 16 threads, dz = 2 (y - t) / B w2 [z > 0] into shared
// memory, and dW1 += dz^T x as a second register-tiled product (a thread: 4 hidden
// units x 4 features over half of the tile's samples).  dW1, db1, dw2, db2 and the
// loss stay in registers over the CTA's tiles; the CTA writes one partial vector,
// and mlp_reduce_kernel adds the partials in a fixed order, so that a batch gives
// the same gradient every time.
//
// What bounds it: nothing but latency -- 101 MFLOP and 1 MB at 8000 samples are
// microseconds of work.  One thread per parameter running through the whole batch
// (nine CTAs, a serial chain of B global loads each) took 341 us there, with 37 us
// for a pass that wrote dz and h to memory; these two kernels take 6.8 and 4.7 us.
constexpr int kGradTile = 64;
constexpr int kGradPad = kFeat + 4;          // row stride of the staged samples and of W1
constexpr int kDzPad = kHid + 4;

struct GradSmem {
    float w1[kHid * kGradPad], x[kGradTile * kGradPad], dz[kGradTile * kDzPad];
    float b1[kHid], w2[kHid], red[16 * kHid];
};

__global__ void __launch_bounds__(256) mlp_grad_kernel(const float *theta, const float *x,
                                                       const float *t, int64_t B, float *part) {
    extern __shared__ float4 grad_raw[];
    GradSmem &sm = *reinterpret_cast<GradSmem *>(grad_raw);
    const int tid = threadIdx.x, lane = tid & 31, ts = tid >> 4, th = tid & 15;
    for (int k = tid; k < kHid * kFeat; k += 256) sm.w1[(k / kFeat) * kGradPad + k % kFeat] = theta[k];
    if (tid < kHid) {
        sm.b1[tid] = theta[kHid * kFeat + tid];
        sm.w2[tid] = theta[kHid * kFeat + kHid + tid];
    }
    const float b2 = theta[kNParam - 1];
    float gw[4][4] = {}, gb1[4] = {}, gw2[4] = {}, gb2 = 0.f, lsum = 0.f;
    // second product: hidden units j0 .. j0 + 3, features i0 .. i0 + 3, samples half, half + 2, ...
    const int half = tid >> 7, j0 = ((tid >> 3) & 15) * 4, i0 = (tid & 7) * 4;
    const int64_t tiles = (B + kGradTile - 1) / kGradTile;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t s0 = tile * kGradTile;
        const int cnt = (int)(B - s0 < kGradTile ? B - s0 : kGradTile);
        __syncthreads();
        for (int k = tid; k < kGradTile * kFeat; k += 256)
            sm.x[(k / kFeat) * kGradPad + k % kFeat] = k < cnt * kFeat ? x[s0 * kFeat + k] : 0.f;
        __syncthreads();
        float z[4][4];      // samples 4 ts + a, hidden units th + 16 b
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) z[a][b] = sm.b1[th + 16 * b];
#pragma unroll
        for (int k = 0; k < kFeat; k += 4) {
            float4 xv[4], wv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
                xv[a] = *reinterpret_cast<const float4 *>(&sm.x[(4 * ts + a) * kGradPad + k]);
#pragma unroll
            for (int b = 0; b < 4; ++b)
                wv[b] = *reinterpret_cast<const float4 *>(&sm.w1[(th + 16 * b) * kGradPad + k]);
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    z[a][b] = fmaf(wv[b].x, xv[a].x, z[a][b]);
                    z[a][b] = fmaf(wv[b].y, xv[a].y, z[a][b]);
                    z[a][b] = fmaf(wv[b].z, xv[a].z, z[a][b]);
                    z[a][b] = fmaf(wv[b].w, xv[a].w, z[a][b]);
                }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int s = 4 * ts + a;
            float out = 0.f;
#pragma unroll
            for (int b = 0; b < 4; ++b) out = fmaf(sm.w2[th + 16 * b], z[a][b] > 0.f ? z[a][b] : 0.f, out);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) out += __shfl_xor_sync(0xffffffffu, out, o);
            const float res = s < cnt ? out + b2 - t[s0 + s] : 0.f;
            const float d = 2.f * res / (float)B;
            if (th == 0) {
                lsum = fmaf(res, res, lsum);
                gb2 += d;
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float zz = z[a][b];
                const bool on = s < cnt && zz > 0.f;
                const float g = on ? d * sm.w2[th + 16 * b] : 0.f;
                gw2[b] = fmaf(d, on ? zz : 0.f, gw2[b]);
                gb1[b] += g;
                sm.dz[s * kDzPad + th + 16 * b] = g;
            }
        }
        __syncthreads();
#pragma unroll 4
        for (int s = half; s < kGradTile; s += 2) {
            const float4 dv = *reinterpret_cast<const float4 *>(&sm.dz[s * kDzPad + j0]);
            const float4 xv = *reinterpret_cast<const float4 *>(&sm.x[s * kGradPad + i0]);
            const float dj[4] = {dv.x, dv.y, dv.z, dv.w}, xi[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) gw[a][b] = fmaf(dj[a], xi[b], gw[a][b]);
        }
    }
    // the CTA's partial vector: the two sample halves of dW1, then the 16 sample
    // groups of db1 and dw2, then db2 and the loss
    float *out = part + (size_t)blockIdx.x * kGradRow;
    __syncthreads();
    float *stage = sm.x;                      // 64 x 32 of it
    if (half)
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) stage[(j0 + a) * kFeat + i0 + b] = gw[a][b];
#pragma unroll
    for (int b = 0; b < 4; ++b) sm.red[ts * kHid + th + 16 * b] = gb1[b];
    __syncthreads();
    if (!half)
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b)
                out[(j0 + a) * kFeat + i0 + b] = gw[a][b] + stage[(j0 + a) * kFeat + i0 + b];
    if (tid < kHid) {
        float v = 0.f;
        for (int k = 0; k < 16; ++k) v += sm.red[k * kHid + tid];
        out[kHid * kFeat + tid] = v;
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < 4; ++b) sm.red[ts * kHid + th + 16 * b] = gw2[b];
    // db2 and the loss sit in the threads th == 0: lanes 0 and 16 of every warp
    gb2 += __shfl_xor_sync(0xffffffffu, gb2, 16);
    lsum += __shfl_xor_sync(0xffffffffu, lsum, 16);
    if (lane == 0) {
        sm.b1[tid >> 5] = gb2;
        sm.b1[8 + (tid >> 5)] = lsum;
    }
    __syncthreads();
    if (tid < kHid) {
        float v = 0.f;
        for (int k = 0; k < 16; ++k) v += sm.red[k * kHid + tid];
        out[kHid * kFeat + kHid + tid] = v;
    } else if (tid < kHid + 2) {
        float v = 0.f;
        for (int k = 0; k < 8; ++k) v += sm.b1[8 * (tid - kHid) + k];
        out[kNParam - 1 + tid - kHid] = v;
    }
}

// Sum of the CTAs' partial vectors, in a fixed order: 64 columns per CTA, four
// threads per column over every fourth row.  Column kNParam is the loss.
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float *part, int nparts, int64_t B,
                                                         float *grad, float *loss) {
    __shared__ float red[4][64];
    const int c = threadIdx.x & 63, g = threadIdx.x >> 6, p = blockIdx.x * 64 + c;
    float acc = 0.f;
    if (p <= kNParam) {
#pragma unroll 8
        for (int k = g; k < nparts; k += 4) acc += part[(size_t)k * kGradRow + p];
    }
    red[g][c] = acc;
    __syncthreads();
    if (g == 0 && p <= kNParam) {
        const float v = (red[0][c] + red[1][c]) + (red[2][c] + red[3][c]);
        if (p < kNParam)
            grad[p] = v;
        else if (loss)
            *loss = v / (float)B;
    }
}

size_t mlp_work_floats() { return (size_t)kGradBlocks * kGradRow; }

void launch_mlp_forward(const float *theta, const float *x, int64_t B, float *y, cudaStream_t s) {
    if (B <= 0) return;
    int64_t blocks = (B + 255) / 256;
    if (blocks > 1024) blocks = 1024;
    mlp_forward_kernel<<<(unsigned)blocks, 256, 0, s>>>(theta, x, B, y);
    ++g_launches;
}

void launch_mlp_loss_grad(const float *theta, const float *x, const float *t, int64_t B,
                          float *work, float *grad, float *loss, cudaStream_t s) {
    const int64_t tiles = (B + kGradTile - 1) / kGradTile;
    const int blocks = (int)(tiles < kGradBlocks ? tiles : kGradBlocks);
    mlp_grad_kernel<<<blocks, 256, sizeof(GradSmem), s>>>(theta, x, t, B, work);
    ++g_launches;
    mlp_reduce_kernel<<<(kNParam + 1 + 63) / 64, 256, 0, s>>>(work, blocks, B, grad, loss);
    ++g_launches;
}

// theta -= lr * m_hat / (sqrt(v_hat) + eps), step >= 1.
__global__ void mlp_adam_kernel(float *theta, const float *grad, float *m, float *v, int64_t np,
                                float c1, float c2, float lr, float b1, float b2, float eps) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < np;
         k += (int64_t)gridDim.x * blockDim.x) {
        const float g = grad[k];
        const float mk = b1 * m[k] + (1.f - b1) * g;
        const float vk = b2 * v[k] + (1.f - b2) * g * g;
        m[k] = mk;
        v[k] = vk;
        theta[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    }
}

void launch_mlp_adam(float *theta, const float *grad, float *m, float *v, int64_t np, int64_t step,
                     float lr, float b1, float b2, float eps, cudaStream_t s) {
    const float c1 = (float)(1.0 - std::pow((double)b1, (double)step));
    const float c2 = (float)(1.0 - std::pow((double)b2, (double)step));
    mlp_adam_kernel<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(theta, grad, m, v, np, c1, c2, lr,
                                                                   b1, b2, eps);
    ++g_launches;
}

}  // namespace spl
