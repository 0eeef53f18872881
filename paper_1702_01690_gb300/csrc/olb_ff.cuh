// olb_ff.cuh -- WENO-5 of FP64 populations on the FP32 pipe.
//
// A GB300 SM starts 2 FP64 operations per clock and 128 FP32 ones, so one FP64
// instruction takes the time of 64 FP32 instructions.  The WENO-5 weights and
// corrections are therefore evaluated in float-float arithmetic: a value is the
// unevaluated sum h + l of two floats (~47 significant bits), and an operation
// takes 4 to 7 FP32 instructions.  Only the first differences of the
// populations (exact inputs of everything else, which is a function of
// differences alone) and the sums that go back to FP64 use the FP64 pipe.
//
// Accuracy, relative to the largest difference of the stencil, against 113-bit
// arithmetic on 2e5 stencils each of noise, sines of 16 to 3000 nodes a wave and
// tanh profiles: rms 2^-46.3 to 2^-49.9, at most 2^-42.0.  The FP64 form it took
// the place of normalised its weights with a reciprocal good to 2^-39.9 (rms
// 2^-41 to 2^-42.6), so faces are more accurate than they were.
//
// Measured on a 4096^2 grid (one step, three stages): 236.1 ms with 30 FP64
// operations a face, 106.6 ms with 1.3 differences and 3 more a face.
#pragma once

#include <cuda_runtime.h>

namespace olb {

struct ff {
    float h, l;
};

// FP64 <-> bit patterns and the FP32 seed of a reciprocal.  (Host versions
// exist so that the arithmetic can be checked on a CPU.)
__host__ __device__ __forceinline__ int f64_hi(double v)
{
#ifdef __CUDA_ARCH__
    return __double2hiint(v);
#else
    long long b;
    __builtin_memcpy(&b, &v, 8);
    return (int)(b >> 32);
#endif
}
__host__ __device__ __forceinline__ int f64_lo(double v)
{
#ifdef __CUDA_ARCH__
    return __double2loint(v);
#else
    long long b;
    __builtin_memcpy(&b, &v, 8);
    return (int)b;
#endif
}
__host__ __device__ __forceinline__ double f64_make(int hi, int lo)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double(hi, lo);
#else
    const long long b = ((long long)hi << 32) | (unsigned)lo;
    double v;
    __builtin_memcpy(&v, &b, 8);
    return v;
#endif
}
__host__ __device__ __forceinline__ float f32_make(unsigned b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float v;
    __builtin_memcpy(&v, &b, 4);
    return v;
#endif
}
__host__ __device__ __forceinline__ unsigned f32_bits(float v)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(v);
#else
    unsigned b;
    __builtin_memcpy(&b, &v, 4);
    return b;
#endif
}
__host__ __device__ __forceinline__ float rcp_seed(float v)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
#else
    return (1.0f / v) * 1.00000012f;  // an ulp off, as the hardware's seed may be
#endif
}

// ---------------------------------------------------------------- FP64 to float-float and back
// The differences of one strip of faces are scaled by a common power of two,
// which puts the largest at FF_EXP: squares and weights then stay in FP32's
// range whatever the populations' units.  FfScale holds the scale of a strip
// as the high words of FP64 numbers: emax the exponent field of its largest
// difference, thr the smallest high word that is kept (a difference below
// 2^-132 of the largest, or subnormal, counts as zero).
constexpr int FF_EXP = 157;  // FP32 exponent field of the largest difference
struct FfScale {
    int emax, thr;
};
// top: the largest high word (sign cleared) of the strip's differences.
__host__ __device__ __forceinline__ FfScale ff_scale(int top)
{
    const int emax = top & 0x7ff00000, thr = emax - (132 << 20);
    return {emax, thr > 0x00100000 ? thr : 0x00100000};
}
// d scaled: h its leading 24 bits, l the next 23 (both truncated, so of one sign).
__host__ __device__ __forceinline__ ff ff_split(double d, FfScale s)
{
    const int hw = f64_hi(d);
    const unsigned lw = (unsigned)f64_lo(d);
    const bool keep = (hw & 0x7fffffff) >= s.thr;
    // exponent field e - emax + FF_EXP, formed in the high word and moved to
    // FP32's place by the shift (its upper bits and the sign fall off)
    const unsigned e = (unsigned)(hw - s.emax + (FF_EXP << 20));
    const unsigned b = ((e << 3) | (lw >> 29));
    const unsigned h = (b & 0x7fffffffu) | ((unsigned)hw & 0x80000000u);
    const unsigned base = (h & 0xff800000u) - (23u << 23);
    const float l = f32_make(base | ((lw >> 6) & 0x007fffffu)) - f32_make(base);
    return {keep ? f32_make(h) : 0.0f, keep ? l : 0.0f};
}
// The scaled float v as FP64, scale undone (zero below FP64's normal range).
__host__ __device__ __forceinline__ double ff_widen(float v, FfScale s)
{
    const unsigned b = f32_bits(v), a = b & 0x7fffffffu;
    const int hw = (int)(a >> 3) + (s.emax - (FF_EXP << 20));
    const bool zero = a < 0x00800000u || hw < 0x00100000;
    return f64_make(zero ? 0 : (int)((unsigned)hw | (b & 0x80000000u)), zero ? 0 : (int)(b << 29));
}

// ---------------------------------------------------------------- float-float arithmetic
// (error-free transformations of Dekker and Knuth; -fmad=false keeps every
// product and sum as written)

// (h, l) += b, with the rounding error of the sum kept in l (TwoSum).
__host__ __device__ __forceinline__ void ff_acc(ff &s, float b)
{
    const float r = s.h + b, t = r - s.h;
    s.l += (s.h - (r - t)) + (b - t);
    s.h = r;
}
// (h, l) += k b for a short constant k: the sum's error as in TwoSum, with
// the remainder of the unrounded product k b from an FMA.  Exact up to 2^-47 of
// the larger term where h and k b have one sign, or k is a power of two.
__host__ __device__ __forceinline__ void ff_acck(ff &s, float k, float b)
{
    const float r = fmaf(k, b, s.h), t = r - s.h;
    s.l += (s.h - (r - t)) + fmaf(k, b, -t);
    s.h = r;
}
// (h, l) -= k b where |h| >= |k b| is known (the product split exactly, then
// Fast2Sum: with cancellation k b has to be a float for its sum to be exact).
__host__ __device__ __forceinline__ void ff_subk_small(ff &s, float k, float b)
{
    const float z = k * b, r = s.h - z, t = r - s.h;
    s.l = (s.l - fmaf(k, b, -z)) - (z + t);
    s.h = r;
}
__host__ __device__ __forceinline__ ff ff_norm(ff a)
{
    const float s = a.h + a.l;
    return {s, a.l - (s - a.h)};
}
// a b without the product of the low parts (below 2^-46 of a b)
__host__ __device__ __forceinline__ ff ff_mul(ff a, ff b)
{
    const float p = a.h * b.h;
    return {p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)))};
}
__host__ __device__ __forceinline__ ff ff_sqr(ff a)
{
    const float p = a.h * a.h;
    return {p, fmaf(a.h + a.h, a.l, fmaf(a.h, a.h, -p))};
}
// d0 - 2 d1 + d2
__host__ __device__ __forceinline__ ff ff_diff2(ff d0, ff d1, ff d2)
{
    ff s = {d0.h, fmaf(-2.0f, d1.l, d0.l + d2.l)};
    ff_acc(s, d2.h);
    ff_acck(s, -2.0f, d1.h);
    return ff_norm(s);
}
// a p + b q - c x for the indicators (a, b >= 0, p, q squares, x the product of
// their roots with |c x| <= a p + b q)
__host__ __device__ __forceinline__ ff ff_form(ff p, float b, ff q, float c, ff x)
{
    ff s = {p.h, fmaf(-c, x.l, fmaf(b, q.l, p.l))};
    ff_acck(s, b, q.h);
    ff_subk_small(s, c, x.h);
    return s;
}
// u with u u = (m / s)^2 up to 2^-44, as a float-float square: the seed
// r ~ 1/s leaves e = 1 - r s, and (m r)^2 (1 + 2 e) is (m / s)^2 to O(e^2).
__host__ __device__ __forceinline__ ff ff_inv2(ff s, float m)
{
    const float r = rcp_seed(s.h);
    const float e = fmaf(-r, s.l, fmaf(-r, s.h, 1.0f));
    const float a = m * r, p = a * a;
    return {p, fmaf(p, e + e, fmaf(a, a, -p))};
}

// ---------------------------------------------------------------- WENO-5
// 6 c of one face, c its correction (face value minus the upwind node v2),
// from the first differences d0 .. d3 (v1 - v0, ..., v4 - v3): the candidates
// of Eq. weno5_flux are 6 G_1 = 5 d1 - 2 d0, 6 G_2 = d1 + 2 d2,
// 6 G_3 = 4 d2 - d3, so with the third differences t0 = d0 - 2 d1 + d2 and
// t1 = d1 - 2 d2 + d3
//   6 (G_1 - G_2) = -2 t0,  6 (G_3 - G_2) = -t1,
//   6 c = d1 + 2 d2 - (2 W_1 t0 + W_3 t1) / (W_1 + W_2 + W_3),
// W_q = delta_q / sigma_q^2 (up to a factor) with the indicators of
// Eq. weno5_sigma as the quadratic forms
//   sigma_1 = d0^2 - 11/4 d0 d1 + 5/2 d1^2,  sigma_2 = d1^2 - 5/4 d1 d2 + d2^2,
//   sigma_3 = d3^2 - 11/4 d2 d3 + 5/2 d2^2,
// each positive definite with condition number below 19.  q_j = d_j^2 and
// x_j = d_j d_{j+1} are shared by the faces of a strip.  Weights are scaled by
// the power of two m below the smallest indicator.  Where an indicator
// vanishes (both its differences are zero) the weights are those of Table
// tab:weno: the ideal weights of the vanishing set.
__host__ __device__ __forceinline__ ff weno5_ff(ff d1, ff d2, ff q0, ff q1, ff q2, ff q3, ff x0, ff x1, ff x2, ff t0,
                                                ff t1)
{
    const ff s1 = ff_form(q0, 2.5f, q1, 2.75f, x0);
    const ff s2 = ff_form(q1, 1.0f, q2, 1.25f, x1);
    const ff s3 = ff_form(q3, 2.5f, q2, 2.75f, x2);
    const float lo = fminf(s1.h, fminf(s2.h, s3.h));
    ff w1, w2, w3;  // (m / sigma_q)^2
    if (lo > 0.0f) {
        const float m = f32_make(f32_bits(lo) & 0x7f800000u);
        w1 = ff_inv2(s1, m);
        w2 = ff_inv2(s2, m);
        w3 = ff_inv2(s3, m);
    } else {
        w1 = {s1.h == 0.0f ? 1.0f : 0.0f, 0.0f};
        w2 = {s2.h == 0.0f ? 1.0f : 0.0f, 0.0f};
        w3 = {s3.h == 0.0f ? 1.0f : 0.0f, 0.0f};
    }
    // weights 1 : 6 : 3 times w (delta_q times 10)
    ff den = {w1.h, fmaf(3.0f, w3.l, fmaf(6.0f, w2.l, w1.l))};
    ff_acck(den, 6.0f, w2.h);
    ff_acck(den, 3.0f, w3.h);
    const ff a = ff_mul(w1, t0), b = ff_mul(w3, t1);
    const float b3 = 3.0f * b.h;
    ff num = {a.h + a.h, fmaf(2.0f, a.l, fmaf(3.0f, b.l, fmaf(3.0f, b.h, -b3)))};
    ff_acc(num, b3);
    // num / den: quotient of the leading parts and its remainder
    const float r = rcp_seed(den.h), z = num.h * r;
    const float zl = fmaf(-z, den.l, fmaf(-z, den.h, num.h) + num.l) * r;
    ff c = {d1.h, fmaf(2.0f, d2.l, d1.l) - zl};
    ff_acck(c, 2.0f, d2.h);
    ff_acc(c, -z);
    return ff_norm(c);
}

// The face value v2 + c from a scaled 6 c.
__host__ __device__ __forceinline__ double weno5_value(double v2, ff c6, FfScale s)
{
    return fma(1.0 / 6.0, ff_widen(c6.h, s) + ff_widen(c6.l, s), v2);
}

// The value of one face from its upwind node and first differences.
__host__ __device__ __forceinline__ double weno5_face(double v2, double d0, double d1, double d2, double d3)
{
    const int a0 = f64_hi(d0) & 0x7fffffff, a1 = f64_hi(d1) & 0x7fffffff, a2 = f64_hi(d2) & 0x7fffffff,
              a3 = f64_hi(d3) & 0x7fffffff;
    const int top = max(max(a0, a1), max(a2, a3));
    if (top >= 0x7ff00000) return f64_make(0x7ff80000, 0);  // an infinity or NaN among the differences
    const FfScale s = ff_scale(top);
    const ff f0 = ff_split(d0, s), f1 = ff_split(d1, s), f2 = ff_split(d2, s), f3 = ff_split(d3, s);
    const ff c = weno5_ff(f1, f2, ff_sqr(f0), ff_sqr(f1), ff_sqr(f2), ff_sqr(f3), ff_mul(f0, f1), ff_mul(f1, f2),
                          ff_mul(f2, f3), ff_diff2(f0, f1, f2), ff_diff2(f1, f2, f3));
    return weno5_value(v2, c, s);
}

// S consecutive faces along a row or column, in the upwind direction: the
// stencil v_0 .. v_4 of face j is p[(j + m) step], m = 0..4, and its value goes
// to out[j ostep].  Differences, their squares and products and the third
// differences are formed once per strip; every face has the operations of
// weno5_face on the same operands (up to the common power of two), so that
// strips of any length agree bit for bit.
template <int S>
__device__ __forceinline__ void weno5_strip_ff(const double *p, int step, double *out, int ostep)
{
    double v[S + 4], d[S + 3];
    int top = 0;
    v[0] = p[0];
#pragma unroll
    for (int j = 0; j < S + 3; ++j) {
        v[j + 1] = p[(j + 1) * step];
        d[j] = v[j + 1] - v[j];
        top = max(top, f64_hi(d[j]) & 0x7fffffff);
    }
    if (top >= 0x7ff00000) {  // an infinity or NaN among the differences
#pragma unroll
        for (int j = 0; j < S; ++j) out[j * ostep] = weno5_face(v[j + 2], d[j], d[j + 1], d[j + 2], d[j + 3]);
        return;
    }
    const FfScale s = ff_scale(top);
    ff f0 = ff_split(d[0], s), f1 = ff_split(d[1], s), f2 = ff_split(d[2], s);
    ff q0 = ff_sqr(f0), q1 = ff_sqr(f1), q2 = ff_sqr(f2);
    ff x0 = ff_mul(f0, f1), x1 = ff_mul(f1, f2), t0 = ff_diff2(f0, f1, f2);
#pragma unroll
    for (int j = 0; j < S; ++j) {
        const ff f3 = ff_split(d[j + 3], s);
        const ff q3 = ff_sqr(f3), x2 = ff_mul(f2, f3), t1 = ff_diff2(f1, f2, f3);
        const ff c = weno5_ff(f1, f2, q0, q1, q2, q3, x0, x1, x2, t0, t1);
        out[j * ostep] = weno5_value(v[j + 2], c, s);
        f0 = f1; f1 = f2; f2 = f3;
        q0 = q1; q1 = q2; q2 = q3;
        x0 = x1; x1 = x2;
        t0 = t1;
    }
}

}  // namespace olb
