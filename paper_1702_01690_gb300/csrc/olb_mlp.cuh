// olb_mlp.cuh -- the learned WENO-5 weight network on the device.
//
// A 5-32-32-3 MLP (tanh, tanh, softmax) maps the normalised stencil
// x = (v - mean v) / (max v - min v) of an interface to three convex weights
// that replace the Jiang-Shu weights of Eq. weno5_omega.  Parameters, 1347
// floats: W1 [32][5], b1 [32], W2 [32][32], b2 [32], W3 [3][32], b3 [3]
// (row-major, concatenated).
#pragma once

#include "olb_kernels.cuh"

namespace olb {

constexpr int MLP_IN = 5, MLP_H = 32, MLP_OUT = 3;
constexpr int MLP_W1 = 0, MLP_B1 = 160, MLP_W2 = 192, MLP_B2 = 1216, MLP_W3 = 1248, MLP_B3 = 1344;
constexpr int MLP_P = 1347;
// The network acts only where the stencil is not smooth in the Jiang-Shu
// sense: min sigma_q < MLP_GUARD max sigma_q.  Where the three indicators are
// within that factor (smooth data, for which the Jiang-Shu weights approach
// the ideal weights and keep 5th order) the Jiang-Shu weights are used.
constexpr double MLP_GUARD = 0.9;

// tanh(x) = sign(x) (1 - 2 / (exp(2 |x|) + 1)), with exp(2 |x|) = 2^(2 |x| / ln 2)
// and the reciprocal from the special-function unit (ex2.approx.ftz.f32,
// rcp.approx.ftz.f32): 6 instructions instead of an accurate tanhf, with an
// absolute error of ~1e-7 (the network's forward pass is checked against the
// FP64 network at 2e-6 in the tests); exp overflowing to +inf gives 1.
__device__ __forceinline__ float tanh_fast(float x)
{
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(fabsf(x) * 2.8853900817779268f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(e + 1.0f));
    return copysignf(fmaf(-2.0f, r, 1.0f), x);
}

// Weights of one stencil; th points to the parameters, 16-byte aligned.  x: normalised stencil.
__device__ __forceinline__ void mlp_weights(const float *__restrict__ th, const float x[MLP_IN], float w[MLP_OUT])
{
    float h1[MLP_H];
#pragma unroll
    for (int j = 0; j < MLP_H; ++j) {
        float a = th[MLP_B1 + j];
#pragma unroll
        for (int q = 0; q < MLP_IN; ++q) a = fmaf(th[MLP_W1 + j * MLP_IN + q], x[q], a);
        h1[j] = tanh_fast(a);
    }
    float z0 = th[MLP_B3 + 0], z1 = th[MLP_B3 + 1], z2 = th[MLP_B3 + 2];
#pragma unroll 4
    for (int j = 0; j < MLP_H; ++j) {
        const float4 *row = reinterpret_cast<const float4 *>(th + MLP_W2 + j * MLP_H);
        float a = th[MLP_B2 + j];
#pragma unroll
        for (int k4 = 0; k4 < MLP_H / 4; ++k4) {
            const float4 r = row[k4];
            a = fmaf(r.x, h1[4 * k4 + 0], a);
            a = fmaf(r.y, h1[4 * k4 + 1], a);
            a = fmaf(r.z, h1[4 * k4 + 2], a);
            a = fmaf(r.w, h1[4 * k4 + 3], a);
        }
        const float h2 = tanh_fast(a);
        z0 = fmaf(th[MLP_W3 + 0 * MLP_H + j], h2, z0);
        z1 = fmaf(th[MLP_W3 + 1 * MLP_H + j], h2, z1);
        z2 = fmaf(th[MLP_W3 + 2 * MLP_H + j], h2, z2);
    }
    const float zm = fmaxf(z0, fmaxf(z1, z2));
    const float e0 = expf(z0 - zm), e1 = expf(z1 - zm), e2 = expf(z2 - zm);
    const float inv = 1.0f / (e0 + e1 + e2);
    w[0] = e0 * inv;
    w[1] = e1 * inv;
    w[2] = e2 * inv;
}

// Whether the network acts on the stencil with first differences d01 .. d34:
// no smoothness indicator vanishes and min sigma_q < MLP_GUARD max sigma_q
// (otherwise Jiang-Shu with Table tab:weno applies).  The decision is that of
// the population precision.  FP64 spares its FP64 pipe (which bounds that
// kernel): the zero test is on the differences' bits, an FP32 pre-check
// decides away from the threshold, and the FP64 indicators that remain are
// compared on the integer pipe (they are >= 0, and their bit patterns order
// like their values; x == 0 of either sign is a zero pattern without the sign
// bit).
__device__ __forceinline__ bool learned_guard(float d01, float d12, float d23, float d34)
{
    const float a1 = d12 - d01, b1 = fmaf(3.0f, d12, -d01);
    const float a2 = d23 - d12, b2 = d12 + d23;
    const float a3 = d34 - d23, b3 = fmaf(-3.0f, d23, d34);
    const float s1 = fmaf(13.0f * a1, a1, 3.0f * b1 * b1);
    const float s2 = fmaf(13.0f * a2, a2, 3.0f * b2 * b2);
    const float s3 = fmaf(13.0f * a3, a3, 3.0f * b3 * b3);
    const float smin = fminf(s1, fminf(s2, s3)), smax = fmaxf(s1, fmaxf(s2, s3));
    const bool zero = (a1 == 0.0f && b1 == 0.0f) || (a2 == 0.0f && b2 == 0.0f) || (a3 == 0.0f && b3 == 0.0f);
    return !zero && smin < (float)MLP_GUARD * smax;
}
// d: the differences d01 .. d34; e: the same rounded to FP32
__device__ __forceinline__ bool learned_guard(const double d[4], const float e[4])
{
    // a_q = b_q = 0 exactly when both differences of sub-stencil q are 0
    // (a difference of two numbers is 0 only when they are equal, and an
    // FMA is exact before its one rounding)
    auto z = [](double v) { return (__double_as_longlong(v) << 1) == 0; };
    if ((z(d[0]) && z(d[1])) || (z(d[1]) && z(d[2])) || (z(d[2]) && z(d[3]))) return false;
    // FP32 pre-check: each sigma_q is a positive-definite quadratic form in
    // two differences (condition number ~18), so from the differences
    // rounded to FP32 it carries a relative error below ~3e-6; outside a
    // band of 1e-4 around the threshold the FP32 comparison is the FP64
    // one.  Inside the band, or with squares near FP32's range limits,
    // the FP64 test below decides.
    const float fa1 = e[1] - e[0], fb1 = fmaf(3.0f, e[1], -e[0]);
    const float fa2 = e[2] - e[1], fb2 = e[1] + e[2];
    const float fa3 = e[3] - e[2], fb3 = fmaf(-3.0f, e[2], e[3]);
    const float f1 = fmaf(13.0f * fa1, fa1, 3.0f * fb1 * fb1);
    const float f2v = fmaf(13.0f * fa2, fa2, 3.0f * fb2 * fb2);
    const float f3 = fmaf(13.0f * fa3, fa3, 3.0f * fb3 * fb3);
    const float fmn = fminf(f1, fminf(f2v, f3)), fmx = fmaxf(f1, fmaxf(f2v, f3));
    if (fmx > 1e-30f && fmx < 1e30f) {
        if (fmn < (float)(MLP_GUARD * (1.0 - 1e-4)) * fmx) return true;
        if (fmn > (float)(MLP_GUARD * (1.0 + 1e-4)) * fmx) return false;
    }
    const double a1 = d[1] - d[0], b1 = fma(3.0, d[1], -d[0]);
    const double a2 = d[2] - d[1], b2 = d[1] + d[2];
    const double a3 = d[3] - d[2], b3 = fma(-3.0, d[2], d[3]);
    const double s1 = fma(13.0 * a1, a1, 3.0 * b1 * b1);
    const double s2 = fma(13.0 * a2, a2, 3.0 * b2 * b2);
    const double s3 = fma(13.0 * a3, a3, 3.0 * b3 * b3);
    const long long i1 = __double_as_longlong(s1), i2 = __double_as_longlong(s2), i3 = __double_as_longlong(s3);
    const double smin = i1 < i2 ? (i1 < i3 ? s1 : s3) : (i2 < i3 ? s2 : s3);
    const double smax = i1 > i2 ? (i1 > i3 ? s1 : s3) : (i2 > i3 ? s2 : s3);
    const bool zero = (z(a1) && z(b1)) || (z(a2) && z(b2)) || (z(a3) && z(b3));
    return !zero && smin < MLP_GUARD * smax;
}

// An FP64 value rounded to FP32 (to even) on the integer pipe, by conversion (on the
// FP64 pipe) where it is neither zero nor a normal FP32 number.
static __device__ __noinline__ float f32_converted(double v) { return (float)v; }
__device__ __forceinline__ float f32_rounded(double v)
{
    const int hw = __double2hiint(v), e = (hw >> 20) & 0x7ff;
    const unsigned lw = (unsigned)__double2loint(v), sign = (unsigned)hw & 0x80000000u;
    if (e > 1023 - 126 && e < 1023 + 127) {
        const unsigned lr = lw + 0x0fffffffu + ((lw >> 29) & 1u);
        return __uint_as_float((((unsigned)(hw & 0x7fffffff) - (896u << 20) + (lr < lw ? 1u : 0u)) << 3 | lr >> 29) | sign);
    }
    return ((unsigned)hw << 1 | lw) == 0 ? __uint_as_float(sign) : f32_converted(v);
}

// The network's input from the stencil's first differences in FP32: the
// normalised stencil x = (v - mean) / (max - min), taken relative to v0
// (shift invariant); all zero where the network does not act.
__device__ __forceinline__ void learned_input_x(const float e[4], bool acts, float x[MLP_IN])
{
    const float w1 = e[0], w2 = w1 + e[1], w3 = w2 + e[2], w4 = w3 + e[3];
    const float mx = fmaxf(fmaxf(0.0f, w1), fmaxf(fmaxf(w2, w3), w4));
    const float mn = fminf(fminf(0.0f, w1), fminf(fminf(w2, w3), w4));
    const float mean = (((w1 + w2) + w3) + w4) * 0.2f;
    const float ir = acts ? 1.0f / (mx - mn) : 0.0f;
    x[0] = (0.0f - mean) * ir;
    x[1] = (w1 - mean) * ir;
    x[2] = (w2 - mean) * ir;
    x[3] = (w3 - mean) * ir;
    x[4] = (w4 - mean) * ir;
}

// The correction sum_q w_q G_q (the interface value minus v2, Eq. weno5_flux)
// from the network's weights and the first differences, in FP32 (the weights
// carry FP32 error anyway).
__device__ __forceinline__ float learned_corr_from(const float w[MLP_OUT], const float e[4])
{
    const float G1 = fmaf(5.0f / 6.0f, e[1], (-1.0f / 3.0f) * e[0]);
    const float G2 = fmaf(1.0f / 3.0f, e[2], (1.0f / 6.0f) * e[1]);
    const float G3 = fmaf(2.0f / 3.0f, e[2], (-1.0f / 6.0f) * e[3]);
    return fmaf(w[0], G1, fmaf(w[1], G2, w[2] * G3));
}

// The network's correction of a stencil it acts on (per thread).
__device__ __forceinline__ float learned_corr_net(const float *__restrict__ th, const float e[4])
{
    float x[MLP_IN], w[MLP_OUT];
    learned_input_x(e, true, x);
    mlp_weights(th, x, w);
    return learned_corr_from(w, e);
}

// Learned WENO-5 face value of one upwind-ordered stencil: where any
// smoothness indicator vanishes the Jiang-Shu weights with Table tab:weno apply
// (constant ghost layers keep their exact flux), and so do they where the
// stencil is smooth (min sigma_q >= MLP_GUARD max sigma_q); otherwise
// sum_q w_q G_q with the network's weights.  FP64 populations: the guard is
// taken in FP64; the network and sum_q w_q G_q run in FP32 (the weights carry
// FP32 error anyway).  This and weno5_learned_corr: one thread's face, for walls.
__device__ __forceinline__ double weno5_js(const double d[4], double v2)
{
    const double q12 = d[1] * d[1], q23 = d[2] * d[2];
    return weno5_core(d[0], d[1], d[2], d[3], q23, 2.5 * q12, 2.5 * q23, v2);
}
__device__ __forceinline__ double weno5_learned(const float *__restrict__ th, double v0, double v1, double v2, double v3,
                                                double v4)
{
    const double d[4] = {v1 - v0, v2 - v1, v3 - v2, v4 - v3};
    const float e[4] = {(float)d[0], (float)d[1], (float)d[2], (float)d[3]};
    if (!learned_guard(d, e)) return weno5_js(d, v2);
    return v2 + (double)learned_corr_net(th, e);
}

// The same for the compensated FP32 storage: the correction sum_q w_q G_q (the
// interface value minus v2) from the stencil's first differences d01 .. d34,
// which fix the normalised stencil (shift invariant) and the candidates.
__device__ __forceinline__ float weno5_learned_corr(const float *__restrict__ th, float d01, float d12, float d23,
                                                   float d34)
{
    if (!learned_guard(d01, d12, d23, d34)) return weno5_corr(d01, d12, d23, d34);
    const float e[4] = {d01, d12, d23, d34};
    return learned_corr_net(th, e);
}

// ---------------------------------------------------------------- the network of a warp
// Inside the stage kernels the 32 lanes of a warp evaluate the network for 32
// stencils at once.  Lane 4 g + t works on the stencils g, g + 8, g + 16, g + 24
// (the rows of an mma fragment): a weight that it loads from shared memory serves
// four stencils instead of one, and two of them share a packed instruction.
// Every sum takes its terms in a fixed order.
//   FP32 populations: the 32 x 32 layer is a matrix product on the tensor pipe
// (mma.sync m16n8k8 with TF32 operands; each operand split into a TF32 high part
// and a TF32 remainder and the product taken as hi hi + hi lo + lo hi, accurate to
// ~2^-21 like an FP32 dot product).  A lane's layer-1 outputs are its own
// fragment, so nothing goes through shared memory.
//   FP64 populations: FP32 multiply-adds, the layers' outputs exchanged through
// shared memory (mlp_weights' sums: the same results).
// One stage of 1024^2 where the network acts on nearly every face: 4.9 -> 3.1 ms (FP32
// populations) and 6.84 -> 4.9 ms (FP64), from a lane per stencil, whose weights came
// with 576 loads a face (FP64) and whose layer-1 outputs went through shared memory to
// the fragments (FP32).  Bound by instruction issue and latency with the 16 warps that
// 128 registers a thread leave an SM (ncu: FP32 issue 61 %, special functions 22 %,
// tensor pipe 30 %; FP64, before the rows of its scratch were rotated, wavefronts of
// shared memory 90 %).

// What a stage kernel has of the network: its parameters in global memory (wall faces,
// a network a thread), the tables and scratch in shared memory.
struct MlpArg {
    const float *theta;
    float *tables;
};

// Tables in shared memory, in the order of the loads.  Layer 1, for units j = 8 ks +
// 4 u + t at (2 ks + u, part, t): the weights and the bias, each twice (float4
// parts (w0 w0 w1 w1) (w2 w2 w3 w3) (w4 w4 b b)).
constexpr int MLP_T1 = 0, MLP_T1_SIZE = 384;
// FP32: layer 3 and the biases of layer 2, for units j = 8 nt + 2 t + q at (2 nt + q,
// part, t): (w0 w0 w1 w1) (w2 w2 b2 b2); W2 as B fragments (hi hi lo lo) of lane
// (g, t) at (ks, nt, lane): B[k][n] = W2[n][k], k = 8 ks + t (+ 4), n = 8 nt + g; b3
constexpr int MLP_T3 = 384, MLP_TB = 640, MLP_T32_B3 = 2688, MLP_T32_SIZE = 2692;
// FP64: W2 transposed; layer 3's weights (w0 w1 w2 0) of each unit; b2; b3; then
// MLP_WARP_SCRATCH floats a warp (the outputs of a layer, [unit][g][4 stencils])
constexpr int MLP_TW = 384, MLP_T4 = 1408, MLP_T64_B2 = 1536, MLP_T64_B3 = 1568, MLP_T64_SIZE = 1572;
constexpr int MLP_WARP_SCRATCH = 1024;

__device__ __forceinline__ void tf32_split(float v, unsigned &hi, unsigned &lo)
{
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hi) : "f"(v));
    const float r = v - __uint_as_float(hi);
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(lo) : "f"(r));
}

// The same for |v| <= 1 or a NaN, which the low part then carries (two integer
// instructions instead of three for the high part).
__device__ __forceinline__ void tf32_split_unit(float v, unsigned &hi, unsigned &lo)
{
    hi = (__float_as_uint(v) + 0x1000u) & 0xffffe000u;
    const float r = v - __uint_as_float(hi);
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(lo) : "f"(r));
}

// Fill the tables from the parameters theta (all threads of the CTA).
template <typename real>
__device__ __forceinline__ void mlp_tables(float *tb, const float *__restrict__ theta)
{
    for (int i = threadIdx.x; i < 6 * MLP_H; i += blockDim.x) {
        const int j = i / 6, q = i - 6 * j;
        const float v = __ldg(theta + (q < MLP_IN ? MLP_W1 + j * MLP_IN + q : MLP_B1 + j));
        float *o = tb + MLP_T1 + ((j >> 2) * 3 + q / 2) * 16 + (j & 3) * 4 + 2 * (q & 1);
        o[0] = o[1] = v;
    }
    for (int i = threadIdx.x; i < 4 * MLP_H; i += blockDim.x) {
        const int j = i / 4, o = i - 4 * j;
        const float v = __ldg(theta + (o < MLP_OUT ? MLP_W3 + o * MLP_H + j : MLP_B2 + j));
        if constexpr (sizeof(real) == 4) {
            float *p = tb + MLP_T3 + ((2 * (j >> 3) + (j & 1)) * 2 + o / 2) * 16 + (j >> 1 & 3) * 4 + 2 * (o & 1);
            p[0] = p[1] = v;
        } else {
            tb[o < MLP_OUT ? MLP_T4 + i : MLP_T64_B2 + j] = v;
        }
    }
    for (int i = threadIdx.x; i < MLP_H * MLP_H; i += blockDim.x) {
        const int n = i / MLP_H, k = i - MLP_H * n;
        const float v = __ldg(theta + MLP_W2 + i);
        if constexpr (sizeof(real) == 4) {
            unsigned *p = reinterpret_cast<unsigned *>(tb) + MLP_TB +
                          (((k >> 3) * 4 + (n >> 3)) * 32 + 4 * (n & 7) + (k & 3)) * 4 + (k >> 2 & 1);
            tf32_split(v, p[0], p[2]);
        } else {
            tb[MLP_TW + k * MLP_H + n] = v;
        }
    }
    if (threadIdx.x < MLP_OUT)
        tb[(sizeof(real) == 4 ? MLP_T32_B3 : MLP_T64_B3) + threadIdx.x] = __ldg(theta + MLP_B3 + threadIdx.x);
}

// c += a b for one m16n8k8 tile (row-major A, column-major B, FP32 accumulators).
__device__ __forceinline__ void mma_tf32(float c[4], const unsigned a[4], const unsigned b[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// tanh_fast of two values.
__device__ __forceinline__ vf2 tanh_fast(vf2 x)
{
    const float x0 = x[0], x1 = x[1];
    float e0, e1, r0, r1;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(fabsf(x0) * 2.8853900817779268f));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(fabsf(x1) * 2.8853900817779268f));
    const vf2 d = vf2::pair(e0, e1) + vf2::all(1.0f);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(d[0]));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(d[1]));
    const vf2 y = vfma(vf2::all(-2.0f), vf2::pair(r0, r1), vf2::all(1.0f));
    return vf2::pair(copysignf(y[0], x0), copysignf(y[1], x1));
}
__device__ __forceinline__ vf2 vf2_lo(float4 v) { return vf2::pair(v.x, v.y); }
__device__ __forceinline__ vf2 vf2_hi(float4 v) { return vf2::pair(v.z, v.w); }

// The inputs of the four stencils of this lane, as two pairs, from those of each
// lane's own stencil.
__device__ __forceinline__ void mlp_inputs(const float x[MLP_IN], vf2 X[2][MLP_IN])
{
    const int g = (threadIdx.x & 31) >> 2;
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int i = 0; i < MLP_IN; ++i)
            X[p][i] = vf2::pair(__shfl_sync(0xffffffffu, x[i], g + 16 * p), __shfl_sync(0xffffffffu, x[i], g + 16 * p + 8));
}
// Layer 1: outputs of unit j = 4 ju + t for the four stencils of this lane.
__device__ __forceinline__ void mlp_unit1(const float *tb, int ju, const vf2 X[2][MLP_IN], vf2 h[2])
{
    const float4 *r = reinterpret_cast<const float4 *>(tb + MLP_T1) + ju * 12 + (threadIdx.x & 3);
    const float4 r0 = r[0], r1 = r[4], r2 = r[8];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        vf2 a = vfma(vf2_lo(r0), X[p][0], vf2_hi(r2));
        a = vfma(vf2_hi(r0), X[p][1], a);
        a = vfma(vf2_lo(r1), X[p][2], a);
        a = vfma(vf2_hi(r1), X[p][3], a);
        a = vfma(vf2_lo(r2), X[p][4], a);
        h[p] = tanh_fast(a);
    }
}
__device__ __forceinline__ void mlp_softmax(const float z[MLP_OUT], float w[MLP_OUT])
{
    const float zm = fmaxf(z[0], fmaxf(z[1], z[2]));
    const float e0 = expf(z[0] - zm), e1 = expf(z[1] - zm), e2 = expf(z[2] - zm);
    const float inv = 1.0f / (e0 + e1 + e2);
    w[0] = e0 * inv;
    w[1] = e1 * inv;
    w[2] = e2 * inv;
}

// Weights w of this lane's stencil x (FP32 populations); every lane of the warp must
// call it, from one call site (mma.sync.aligned needs the whole warp at the same
// instruction; lanes whose stencil the network does not act on pass any x and
// ignore w).  tb: the tables (mlp_tables<float>).
__device__ __forceinline__ void mlp_weights_warp32(const float *tb, const float x[MLP_IN], float w[MLP_OUT])
{
    const int lane = threadIdx.x & 31, t = lane & 3;
    vf2 X[2][MLP_IN];
    mlp_inputs(x, X);
    // layer 2 accumulators: rows = stencils, 16 per m-tile mt; columns = outputs, 8
    // per n-tile nt; k = the 32 layer-1 outputs, 8 per step ks, each step's layer-1
    // outputs (this lane's part of the A fragments) computed just before it
    float acc[2][4][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[mt][nt][q] = 0.0f;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        unsigned ah[2][4], al[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            vf2 h[2];
            mlp_unit1(tb, 2 * ks + u, X, h);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                tf32_split_unit(h[mt][0], ah[mt][2 * u], al[mt][2 * u]);
                tf32_split_unit(h[mt][1], ah[mt][2 * u + 1], al[mt][2 * u + 1]);
            }
        }
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const uint4 b = reinterpret_cast<const uint4 *>(tb + MLP_TB)[(4 * ks + nt) * 32 + lane];
            const unsigned bh[2] = {b.x, b.y}, bl[2] = {b.z, b.w};
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) mma_tf32(acc[mt][nt], al[mt], bh);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) mma_tf32(acc[mt][nt], ah[mt], bl);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) mma_tf32(acc[mt][nt], ah[mt], bh);
        }
    }
    // h2 = tanh(acc + b2) and layer 3: accumulator q of (mt, nt) holds stencil
    // g + 8 m, m = 2 mt + (q >> 1), output 8 nt + 2 t + (q & 1)
    vf2 z[2][MLP_OUT];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int o = 0; o < MLP_OUT; ++o) z[mt][o] = vf2::all(0.0f);
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float4 *r = reinterpret_cast<const float4 *>(tb + MLP_T3) + (2 * nt + q) * 8 + t;
            const float4 r0 = r[0], r1 = r[4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const vf2 h2 = tanh_fast(vf2::pair(acc[mt][nt][q], acc[mt][nt][q + 2]) + vf2_hi(r1));
                z[mt][0] = vfma(vf2_lo(r0), h2, z[mt][0]);
                z[mt][1] = vfma(vf2_hi(r0), h2, z[mt][1]);
                z[mt][2] = vfma(vf2_lo(r1), h2, z[mt][2]);
            }
        }
    // sum over the four lanes of a row group (t = 0..3), of which lane t keeps m = t:
    // (z_t + z_{t^1}) + (z_{t^2} + z_{t^3})
    float zz[MLP_OUT];
#pragma unroll
    for (int o = 0; o < MLP_OUT; ++o) {
        float s[2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const float keep = t & 1 ? z[mt][o][1] : z[mt][o][0], send = t & 1 ? z[mt][o][0] : z[mt][o][1];
            s[mt] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
        }
        const float keep = t & 2 ? s[1] : s[0], send = t & 2 ? s[0] : s[1];
        zz[o] = (keep + __shfl_xor_sync(0xffffffffu, send, 2)) + tb[MLP_T32_B3 + o];
    }
    float e[MLP_OUT];
    mlp_softmax(zz, e);
    // stencil F sits in lane F; lane 4 (F mod 8) + F / 8 finished it
    const int src = 4 * (lane & 7) + (lane >> 3);
#pragma unroll
    for (int o = 0; o < MLP_OUT; ++o) w[o] = __shfl_sync(0xffffffffu, e[o], src);
}

// The same for FP64 populations, with the results of mlp_weights (every lane of the
// warp must call it).  tb: the tables (mlp_tables<double>); sc: this warp's scratch.
__device__ __forceinline__ void mlp_weights_warp64(const float *tb, const float x[MLP_IN], float w[MLP_OUT], float *sc)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    // (the g of a unit's row rotated by twice the t of the lane that writes it: the
    // eight lanes of a quarter of a 16-byte access fall on all banks)
    float4 *const s4 = reinterpret_cast<float4 *>(sc);
    auto at = [](int unit, int g, int t) { return 8 * unit + ((g + 2 * t) & 7); };
    vf2 X[2][MLP_IN];
    mlp_inputs(x, X);
#pragma unroll 2
    for (int ju = 0; ju < MLP_H / 4; ++ju) {
        vf2 h[2];
        mlp_unit1(tb, ju, X, h);
        s4[at(4 * ju + t, g, t)] = make_float4(h[0][0], h[0][1], h[1][0], h[1][1]);
    }
    __syncwarp();
    // layer 2: the units 8 t .. 8 t + 7 of this lane's four stencils, units in pairs
    vf2 a[4][4];
    const float4 b0 = reinterpret_cast<const float4 *>(tb + MLP_T64_B2)[2 * t],
                 b1 = reinterpret_cast<const float4 *>(tb + MLP_T64_B2)[2 * t + 1];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        a[m][0] = vf2_lo(b0);
        a[m][1] = vf2_hi(b0);
        a[m][2] = vf2_lo(b1);
        a[m][3] = vf2_hi(b1);
    }
#pragma unroll 8
    for (int k = 0; k < MLP_H; ++k) {
        const float4 *r = reinterpret_cast<const float4 *>(tb + MLP_TW + k * MLP_H) + 2 * t;
        const float4 r0 = r[0], r1 = r[1], h = s4[at(k, g, k & 3)];
        const float hm[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const vf2 hh = vf2::all(hm[m]);
            a[m][0] = vfma(vf2_lo(r0), hh, a[m][0]);
            a[m][1] = vfma(vf2_hi(r0), hh, a[m][1]);
            a[m][2] = vfma(vf2_lo(r1), hh, a[m][2]);
            a[m][3] = vfma(vf2_hi(r1), hh, a[m][3]);
        }
    }
    __syncwarp();
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) {
        vf2 h[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) h[m] = tanh_fast(a[m][jp]);
        s4[at(8 * t + 2 * jp, g, t)] = make_float4(h[0][0], h[1][0], h[2][0], h[3][0]);
        s4[at(8 * t + 2 * jp + 1, g, t)] = make_float4(h[0][1], h[1][1], h[2][1], h[3][1]);
    }
    __syncwarp();
    // layer 3 and the softmax: a lane its own stencil
    vf2 z01 = vf2::pair(tb[MLP_T64_B3], tb[MLP_T64_B3 + 1]);
    float z2 = tb[MLP_T64_B3 + 2];
#pragma unroll
    for (int j = 0; j < MLP_H; ++j) {
        const float4 r = reinterpret_cast<const float4 *>(tb + MLP_T4)[j];
        const float h2 = sc[4 * at(j, lane & 7, j >> 3) + (lane >> 3)];
        z01 = vfma(vf2_lo(r), vf2::all(h2), z01);
        z2 = fmaf(r.z, h2, z2);
    }
    const float z[MLP_OUT] = {z01[0], z01[1], z2};
    mlp_softmax(z, w);
    __syncwarp();  // before the next call writes the scratch
}

}  // namespace olb
