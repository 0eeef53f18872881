// olb_mlp.cu -- training and inference of the learned WENO-5 weight network
// (olb_mlp.cuh) on the GPU with hand-written kernels.
//
// Objective (per sample s): the interface value v2 + sum_q w_q G_q should be
// the target t; in normalised units the loss is the mean over samples of
// (sum_q w_q Gn_q - tn)^2 with Gn = G / r, tn = (t - v2) / r, r = max - min of
// the stencil.  Inputs: x [S][5] normalised stencils, Gn [S][3], tn [S].
//
// k_mlp_grad: groups of 32 samples, eight threads a sample.  A thread has four of
// the 32 units of each hidden layer (forward, and their derivatives backward); the
// activations of the group sit in shared memory, and the weight gradients, sums
// over its samples, in registers: four entries of W2 a thread, two others.  A CTA
// takes several groups if there are more than CTAs.
// k_adam: the sum over the CTAs' gradients in a fixed order, then the Adam update
// of Kingma & Ba (2015).
// One epoch of 262144 samples in minibatches of 4096: 2.17 -> 1.06 ms (64 pairs of
// launches; a minibatch was 32 CTAs of 128 threads with a sample each, 25 us of serial
// sums, and is 128 CTAs and 9 us, plus 4 us for k_adam).
#include <cmath>
#include <algorithm>
#include <vector>

#include "../../include/olb.h"
#include "olb_mlp.cuh"

using namespace olb;

namespace {

constexpr int GS = 32, GP = 8, GT = GS * GP;  // samples of a group, threads a sample, threads
constexpr int GU = MLP_H / GP;                // units a thread
static_assert(GU == 4, "units are handled as float4");
constexpr int GRAD_STRIDE = 1352;  // floats of one CTA's gradient: MLP_P, the loss, padding

struct GradSmem {
    float th[MLP_P + 1];
    float w2[MLP_H][MLP_H + 4];  // W2 once more, its rows in different banks
    // rows of a sample are 36 floats apart: 16-byte aligned, and the eight samples
    // that a quarter of a warp's float4 accesses touch lie in different banks
    float x[GS][8];
    float h1[GS][MLP_H + 4];
    float h2[GS][MLP_H + 4];
    float dz[GS][4];
    float da2[GS][MLP_H + 4];
    float da1[GS][MLP_H + 4];
    float red[GT / 32];
};

// Gradient (and the loss) of a minibatch: PARTIAL writes each CTA's sums to
// grad[CTA][GRAD_STRIDE], else they are added to grad and *loss.
template <bool PARTIAL>
__global__ void __launch_bounds__(GT) k_mlp_grad(const float *__restrict__ theta, const float *__restrict__ X,
                                                 const float *__restrict__ Gn, const float *__restrict__ tn, int S,
                                                 float inv_S, float *__restrict__ grad, float *__restrict__ loss)
{
    __shared__ __align__(16) GradSmem sm;
    // sample of the group; forward a thread has units c, c + 8, c + 16, c + 24 (rows
    // of W2 in different banks), backward the inputs u .. u + 3 of layer 2
    const int tid = threadIdx.x, s = tid / GP, c = tid % GP, u = c * GU;
    for (int p = tid; p < MLP_P; p += GT) {
        const float v = theta[p];
        sm.th[p] = v;
        if (p >= MLP_W2 && p < MLP_B2) sm.w2[(p - MLP_W2) / MLP_H][(p - MLP_W2) % MLP_H] = v;
    }
    const float *th = sm.th;
    // weight gradients of this thread: W2[j2][k2 .. k2 + 3], and entries tid and tid + GT of the others
    const int j2 = tid / GP, k2 = u;
    float g2[GU] = {0.0f, 0.0f, 0.0f, 0.0f}, go[2] = {0.0f, 0.0f}, sum2 = 0.0f;
    for (long long base = (long long)blockIdx.x * GS; base < S; base += (long long)gridDim.x * GS) {
        const bool valid = base + s < S;
        __syncthreads();  // the parameters; the group before is done with
        if (tid < GS * MLP_IN) {
            const long long at = base * MLP_IN + tid;
            sm.x[tid / MLP_IN][tid % MLP_IN] = at < (long long)S * MLP_IN ? X[at] : 0.0f;
        }
        __syncthreads();
        // forward
        float a[GU];
#pragma unroll
        for (int i = 0; i < GU; ++i) {
            const int j = c + GP * i;
            a[i] = th[MLP_B1 + j];
#pragma unroll
            for (int q = 0; q < MLP_IN; ++q) a[i] = fmaf(th[MLP_W1 + j * MLP_IN + q], sm.x[s][q], a[i]);
            sm.h1[s][j] = tanhf(a[i]);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < GU; ++i) a[i] = th[MLP_B2 + c + GP * i];
#pragma unroll
        for (int k = 0; k < MLP_H; k += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(&sm.h1[s][k]);
#pragma unroll
            for (int i = 0; i < GU; ++i) {
                const float4 w = *reinterpret_cast<const float4 *>(&sm.w2[c + GP * i][k]);
                a[i] = fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, a[i]))));
            }
        }
        float d2[GU], z[MLP_OUT] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < GU; ++i) {
            const int j = c + GP * i;
            d2[i] = tanhf(a[i]);
            sm.h2[s][j] = d2[i];
#pragma unroll
            for (int q = 0; q < MLP_OUT; ++q) z[q] = fmaf(th[MLP_W3 + q * MLP_H + j], d2[i], z[q]);
        }
#pragma unroll
        for (int q = 0; q < MLP_OUT; ++q) {
#pragma unroll
            for (int o = 1; o < GP; o <<= 1) z[q] += __shfl_xor_sync(0xffffffffu, z[q], o);
            z[q] += th[MLP_B3 + q];
        }
        const float zm = fmaxf(z[0], fmaxf(z[1], z[2]));
        float w[MLP_OUT], g[MLP_OUT] = {0.0f, 0.0f, 0.0f}, res = 0.0f;
#pragma unroll
        for (int q = 0; q < MLP_OUT; ++q) w[q] = expf(z[q] - zm);
        const float inv = 1.0f / (w[0] + w[1] + w[2]);
#pragma unroll
        for (int q = 0; q < MLP_OUT; ++q) w[q] *= inv;
        if (valid) {
#pragma unroll
            for (int q = 0; q < MLP_OUT; ++q) g[q] = Gn[(base + s) * MLP_OUT + q];
            res = fmaf(w[0], g[0], fmaf(w[1], g[1], fmaf(w[2], g[2], -tn[base + s])));
        }
        if (c == 0) sum2 = fmaf(res, res, sum2);
        // backward: dL/dw = 2 res G / S; softmax; tanh layers (all zero past the end: res = 0)
        float dz[MLP_OUT], wdw = 0.0f;
#pragma unroll
        for (int q = 0; q < MLP_OUT; ++q) {
            dz[q] = 2.0f * inv_S * res * g[q];
            wdw = fmaf(w[q], dz[q], wdw);
        }
#pragma unroll
        for (int q = 0; q < MLP_OUT; ++q) dz[q] = w[q] * (dz[q] - wdw);
        if (c == 0) *reinterpret_cast<float4 *>(&sm.dz[s][0]) = make_float4(dz[0], dz[1], dz[2], 0.0f);
#pragma unroll
        for (int i = 0; i < GU; ++i) {
            const int j = c + GP * i;
            float b = 0.0f;
#pragma unroll
            for (int q = 0; q < MLP_OUT; ++q) b = fmaf(dz[q], th[MLP_W3 + q * MLP_H + j], b);
            sm.da2[s][j] = b * fmaf(-d2[i], d2[i], 1.0f);
        }
        __syncwarp();
        float b[GU] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 8
        for (int k = 0; k < MLP_H; ++k) {
            const float v = sm.da2[s][k];
            const float4 r = *reinterpret_cast<const float4 *>(&sm.w2[k][u]);
            b[0] = fmaf(v, r.x, b[0]);
            b[1] = fmaf(v, r.y, b[1]);
            b[2] = fmaf(v, r.z, b[2]);
            b[3] = fmaf(v, r.w, b[3]);
        }
        const float4 h = *reinterpret_cast<const float4 *>(&sm.h1[s][u]);
        b[0] *= fmaf(-h.x, h.x, 1.0f);
        b[1] *= fmaf(-h.y, h.y, 1.0f);
        b[2] *= fmaf(-h.z, h.z, 1.0f);
        b[3] *= fmaf(-h.w, h.w, 1.0f);
        *reinterpret_cast<float4 *>(&sm.da1[s][u]) = make_float4(b[0], b[1], b[2], b[3]);
        __syncthreads();
        // weight gradients: sums over the group's samples
#pragma unroll 8
        for (int t = 0; t < GS; ++t) {
            const float v = sm.da2[t][j2];
            const float4 r = *reinterpret_cast<const float4 *>(&sm.h1[t][k2]);
            g2[0] = fmaf(v, r.x, g2[0]);
            g2[1] = fmaf(v, r.y, g2[1]);
            g2[2] = fmaf(v, r.z, g2[2]);
            g2[3] = fmaf(v, r.w, g2[3]);
        }
        // the others: W1 and b1 (192), then b2, W3 and b3
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int q = tid + e * GT, p = q < MLP_W2 ? q : q - MLP_W2 + MLP_B2;
            if (p >= MLP_P) continue;
            const float *l = nullptr, *r = nullptr;  // product of two activations, or one
            int ls = MLP_H + 4, rs = MLP_H + 4;
            if (p < MLP_B1) {
                l = &sm.da1[0][p / MLP_IN];
                r = &sm.x[0][p % MLP_IN];
                rs = 8;
            } else if (p < MLP_W2) {
                l = &sm.da1[0][p - MLP_B1];
            } else if (p < MLP_W3) {
                l = &sm.da2[0][p - MLP_B2];
            } else if (p < MLP_B3) {
                l = &sm.dz[0][(p - MLP_W3) / MLP_H];
                ls = 4;
                r = &sm.h2[0][(p - MLP_W3) % MLP_H];
            } else {
                l = &sm.dz[0][p - MLP_B3];
                ls = 4;
            }
            float acc = go[e];
#pragma unroll 8
            for (int t = 0; t < GS; ++t) acc = fmaf(l[t * ls], r ? r[t * rs] : 1.0f, acc);
            go[e] = acc;
        }
    }
    // the CTA's sums
    for (int o = 16; o > 0; o >>= 1) sum2 += __shfl_xor_sync(0xffffffffu, sum2, o);
    if ((tid & 31) == 0) sm.red[tid >> 5] = sum2;
    __syncthreads();
    auto put = [&](int p, float v) {
        if constexpr (PARTIAL) grad[(long long)blockIdx.x * GRAD_STRIDE + p] = v;
        else atomicAdd(grad + p, v);
    };
#pragma unroll
    for (int i = 0; i < GU; ++i) put(MLP_W2 + j2 * MLP_H + k2 + i, g2[i]);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int q = tid + e * GT, p = q < MLP_W2 ? q : q - MLP_W2 + MLP_B2;
        if (p < MLP_P) put(p, go[e]);
    }
    if (tid == 0) {
        float acc = 0.0f;
        for (int k = 0; k < GT / 32; ++k) acc += sm.red[k];
        if constexpr (PARTIAL) put(MLP_P, acc * inv_S);
        else atomicAdd(loss, acc * inv_S);
    }
}

// part: the gradients of n CTAs.  A block has 32 parameters, each of its warps every
// 32nd CTA's; the loss is "parameter" MLP_P.
constexpr int ADAM_WARPS = 32;
__global__ void __launch_bounds__(ADAM_WARPS * 32) k_adam(float *__restrict__ theta, const float *__restrict__ part, int n,
                                                          float *__restrict__ m, float *__restrict__ v,
                                                          float *__restrict__ loss, float lr, float b1, float b2, float eps,
                                                          float c1, float c2)
{
    __shared__ float red[ADAM_WARPS][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, p0 = blockIdx.x * 32;
    float acc = 0.0f;
    if (p0 + lane <= MLP_P) {
#pragma unroll 4
        for (int c = w; c < n; c += ADAM_WARPS) acc += part[(long long)c * GRAD_STRIDE + p0 + lane];
    }
    red[w][lane] = acc;
    __syncthreads();
    // warp w adds up parameter p0 + w
    float g = red[lane][w];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
    const int p = p0 + w;
    if (lane > 0 || p > MLP_P) return;
    if (p == MLP_P) {
        *loss += g;
        return;
    }
    const float mm = fmaf(b1, m[p], (1.f - b1) * g);
    const float vv = fmaf(b2, v[p], (1.f - b2) * g * g);
    m[p] = mm;
    v[p] = vv;
    theta[p] -= lr * (mm * c1) / (sqrtf(vv * c2) + eps);
}

__global__ void k_mlp_forward(const float *__restrict__ theta, const float *__restrict__ X, int S,
                              float *__restrict__ W)
{
    __shared__ __align__(16) float th[MLP_P + 1];
    for (int p = threadIdx.x; p < MLP_P; p += blockDim.x) th[p] = theta[p];
    __syncthreads();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    float x[MLP_IN], w[MLP_OUT];
    for (int q = 0; q < MLP_IN; ++q) x[q] = X[(long long)s * MLP_IN + q];
    mlp_weights(th, x, w);
    for (int q = 0; q < MLP_OUT; ++q) W[(long long)s * MLP_OUT + q] = w[q];
}

// CTAs for n samples: one for each group of 32, as many as fit on the device at once
int grad_ctas(int n)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 152;
    const int groups = (n + GS - 1) / GS;
    return groups < 4 * sms ? groups : 4 * sms;
}

}  // namespace

extern "C" int olb_mlp_forward(const float *theta, const float *x, int n, float *w, void *stream)
{
    if (!theta || !x || !w || n < 0) return OLB_ERR_ARG;
    if (n == 0) return OLB_OK;
    cudaStream_t s = (cudaStream_t)stream;
    k_mlp_forward<<<(n + 127) / 128, 128, 0, s>>>(theta, x, n, w);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return cuda_status(e);
}

extern "C" int olb_mlp_grad(const float *theta, const float *x, const float *g, const float *t, int n, float *grad,
                            float *loss, void *stream)
{
    if (!theta || !x || !g || !t || !grad || !loss || n < 1) return OLB_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(grad, 0, MLP_P * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(loss, 0, sizeof(float), s);
    if (e == cudaSuccess) {
        k_mlp_grad<false><<<grad_ctas(n), GT, 0, s>>>(theta, x, g, t, n, 1.0f / (float)n, grad, loss);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return cuda_status(e);
}

extern "C" int olb_mlp_train(float *theta, const float *x, const float *g, const float *t, int n, int epochs,
                             int batch, float lr, void *stream, float *loss_history)
{
    if (!theta || !x || !g || !t || n < 1 || epochs < 1 || batch < 1 || !(lr > 0.f)) return OLB_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int ctas = grad_ctas(std::min(batch, n));
    // the CTAs' gradients, then m, v and the per-epoch loss
    const size_t grads = (size_t)ctas * GRAD_STRIDE, state = 2 * MLP_P + epochs + 8;
    // (from the stream's memory pool: cudaMalloc and cudaFree took 0.15 ms of a call)
    float *work = nullptr;
    cudaError_t e = cudaMallocAsync((void **)&work, (grads + state) * sizeof(float), s);
    if (e != cudaSuccess) return cuda_status(e);
    float *m = work + grads, *v = m + MLP_P, *lhist = v + MLP_P;
    e = cudaMemsetAsync(m, 0, state * sizeof(float), s);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    long long step = 0;
    const int nb = (n + batch - 1) / batch;
    for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
        for (int b = 0; b < nb && e == cudaSuccess; ++b) {
            const int off = b * batch, cnt = std::min(batch, n - off), used = grad_ctas(cnt);
            ++step;
            // the loss of minibatch b is weighted by its share of the epoch
            k_mlp_grad<true><<<used, GT, 0, s>>>(theta, x + (long long)off * MLP_IN, g + (long long)off * MLP_OUT, t + off,
                                                 cnt, 1.0f / (float)cnt, work, nullptr);
            const float c1 = 1.f / (1.f - powf(b1, (float)step)), c2 = 1.f / (1.f - powf(b2, (float)step));
            k_adam<<<(MLP_P + 1 + 31) / 32, ADAM_WARPS * 32, 0, s>>>(theta, work, used, m, v, lhist + ep, lr, b1, b2, eps, c1, c2);
            e = cudaGetLastError();
        }
    }
    std::vector<float> h(epochs, 0.f);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), lhist, epochs * sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFreeAsync(work, s);
    if (e != cudaSuccess) return cuda_status(e);
    if (loss_history)
        for (int ep = 0; ep < epochs; ++ep) loss_history[ep] = h[ep] / (float)nb;
    return OLB_OK;
}
