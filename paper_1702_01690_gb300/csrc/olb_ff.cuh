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
// tanh profiles: rms 2^-46.3 to 2^-49.9, the largest 2^-42.0 (of 4e5 of noise 2^-41.6).
// The FP64 form it took the place of normalised its weights with a reciprocal good to
// 2^-39.9 (rms 2^-41 to 2^-42.6), so faces are more accurate than they were.  But its
// errors were those of the face's own candidates; here a face behind a jump of one
// node, whose weights leave the jump out, still carries 2^-47 of it: two nodes beyond a
// jump of more than 2^46 times their density the first stage of a step is rounding.
//
// Measured on a 4096^2 grid (one step, three stages): 236.1 ms with 30 FP64
// operations a face, 106.6 ms with 1.3 differences and 3 more a face (the force
// and the node updates still in FP64; see olb_stage64.cuh for those).
#pragma once

#include <type_traits>

#include "olb_internal.cuh"

namespace olb {

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
// Values are scaled by a power of two that puts the largest density of a tile
// at 2^45: a tile's differences, from 2^-66 of it (an ulp of a population 2^-13
// of it) to 2^18 times it, then have squares and weights inside FP32's range
// whatever the populations' units.  Where they lie beyond (dilute nodes beside dense
// ones of the next tile) the low parts are not finite, and the stage takes the tile's
// lines again with the scale of its largest population (stage_tile64; grids of one
// launch a stage have that from the start).
constexpr int FF_EXP = 127 + 45;  // FP32 exponent field of the largest density
struct FfScale {
    int off;     // added to an FP64 high word: exponent field e - emax + FF_EXP
    float inf;   // the first scaled value that is beyond FP64 or FP32
    int lo, hi;  // high words of the smallest value that is kept (2^-60 scaled: smaller ones
                 // and zero become it, far below every rounding) and of the first beyond FP32
};
// top: high word (sign cleared) of the largest density.
__host__ __device__ __forceinline__ FfScale ff_scale(int top)
{
    const int off = (FF_EXP << 20) - (top & 0x7ff00000);
    // (densities above 2^941 leave no room beyond FP32: an infinity is then taken as 2^1024)
    const int least = (255 << 20) - 0x7ff00000;
    return {off, f32_make((unsigned)(0x7ff00000 + min(off, least)) << 3), max((67 << 20) - off, 1 << 20), (255 << 20) - max(off, least)};
}
// An int as a float (rounded).
__host__ __device__ __forceinline__ float f32_of(int v)
{
#ifdef __CUDA_ARCH__
    return __int2float_rn(v);
#else
    return (float)v;
#endif
}
// d scaled: h is d rounded to 24 bits, l the rest (29 bits and a sign) rounded
// to 24; not finite for infinities, NaN and what FP32 cannot hold.
// (Zero becomes 2^-60: sigma_q then never vanishes, and nothing divides by
// zero.  Where all differences of a sub-stencil vanish its weight takes over as
// in Table tab:weno, and which of several vanishing ones does is no matter,
// since their candidates agree.)
__host__ __device__ __forceinline__ ff ff_split(double d, FfScale s)
{
    const int hw = f64_hi(d);
    const unsigned lw = (unsigned)f64_lo(d), sign = (unsigned)hw & 0x80000000u;
    const int a = min(max(hw & 0x7fffffff, s.lo), s.hi);
    // half an ulp of h added to the magnitude
    const unsigned lr = lw + 0x10000000u, e = (unsigned)(a + s.off) + (lr < lw ? 1u : 0u);
    const unsigned h = ((e << 3) | (lr >> 29)) | sign;
    // the last 29 bits, less 2^29 where h was rounded up; 8 of their units are 2^-49 of d's leading bit
    const unsigned unit = ((unsigned)(a + s.off - (55 << 20)) << 3) & 0x7f800000u;
    return {f32_make(h), f32_of((int)(lw << 3)) * f32_make(unit | sign)};
}
// A scaled float as FP64, scale undone (FP64's smallest normal number where it
// would be less, no number beyond FP64); l: a low part, whose high part is no number
// where it is none.
__host__ __device__ __forceinline__ double ff_widen(float v, FfScale s, bool l)
{
    const unsigned b = f32_bits(v);
    const int a = (int)(b & 0x7fffffffu), least = (max(s.off, 0) + (1 << 20)) << 3;
    const int m = max(a, least), hw = (m >> 3) - s.off;
    return f64_make(!l && !(fabsf(v) < s.inf) ? 0x7ff80000 : (int)((unsigned)hw | (b & 0x80000000u)), m << 29);
}
// (either part can leave FP32's range alone: where an indicator overflows, its
// weight's high part is zero and only the low part is no number, which the high
// part takes on here)
__host__ __device__ __forceinline__ double ff_widen(ff v, FfScale s)
{
    return ff_widen(fmaf(0.0f, v.l, v.h), s, false) + ff_widen(v.l, s, true);
}

// ---------------------------------------------------------------- one or two floats
// The arithmetic below is written for a vector V of one float or of two (the
// packed instructions fma.rn.f32x2 and so on of sm_100 and later: the same
// operations as two scalar ones in one issue slot; measured on a GB300, FFMA
// starts 114 lanes per clock and SM, FFMA2 63, and a negated operand is free in
// both).  Results do not depend on V.
struct vf1 {
    static constexpr int W = 1;
    float v;
    __host__ __device__ __forceinline__ static vf1 all(float a) { return {a}; }
    __host__ __device__ __forceinline__ static vf1 of(const float *a) { return {a[0]}; }
    __host__ __device__ __forceinline__ float operator[](int) const { return v; }
};
__host__ __device__ __forceinline__ vf1 operator+(vf1 a, vf1 b) { return {a.v + b.v}; }
__host__ __device__ __forceinline__ vf1 operator-(vf1 a, vf1 b) { return {a.v - b.v}; }
__host__ __device__ __forceinline__ vf1 operator*(vf1 a, vf1 b) { return {a.v * b.v}; }
__host__ __device__ __forceinline__ vf1 operator-(vf1 a) { return {-a.v}; }
__host__ __device__ __forceinline__ vf1 vfma(vf1 a, vf1 b, vf1 c) { return {fmaf(a.v, b.v, c.v)}; }

struct vf2 {
    static constexpr int W = 2;
    unsigned long long v;
    __device__ __forceinline__ static vf2 pair(float a, float b)
    {
        vf2 r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
        return r;
    }
    __device__ __forceinline__ static vf2 all(float a) { return pair(a, a); }
    __device__ __forceinline__ static vf2 of(const float *a) { return pair(a[0], a[1]); }
    __device__ __forceinline__ float operator[](int i) const
    {
        float a, b;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
        return i ? b : a;
    }
};
__device__ __forceinline__ vf2 operator+(vf2 a, vf2 b)
{
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(a.v) : "l"(b.v));
    return a;
}
__device__ __forceinline__ vf2 operator-(vf2 a, vf2 b)
{
    asm("sub.rn.f32x2 %0, %0, %1;" : "+l"(a.v) : "l"(b.v));
    return a;
}
__device__ __forceinline__ vf2 operator*(vf2 a, vf2 b)
{
    asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(a.v) : "l"(b.v));
    return a;
}
__device__ __forceinline__ vf2 operator-(vf2 a) { return vf2::pair(-a[0], -a[1]); }
__device__ __forceinline__ vf2 vfma(vf2 a, vf2 b, vf2 c)
{
    vf2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
template <typename V, int = V::W>
__host__ __device__ __forceinline__ V operator*(float a, V b)
{
    return V::all(a) * b;
}
template <typename V, int = V::W>
__host__ __device__ __forceinline__ V vfma(float a, V b, V c)
{
    return vfma(V::all(a), b, c);
}

// W float-floats.
template <typename V>
struct ffv {
    V h, l;
};
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_all(ff a)
{
    return {V::all(a.h), V::all(a.l)};
}
template <typename V>
__host__ __device__ __forceinline__ ff ff_lane(ffv<V> a, int i)
{
    return {a.h[i], a.l[i]};
}
// ff_split of W values
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_split(const double (&d)[V::W], FfScale s)
{
    float h[V::W], l[V::W];
#pragma unroll
    for (int i = 0; i < V::W; ++i) {
        const ff f = ff_split(d[i], s);
        h[i] = f.h;
        l[i] = f.l;
    }
    return {V::of(h), V::of(l)};
}

// ---------------------------------------------------------------- float-float arithmetic
// (error-free transformations of Dekker and Knuth; -fmad=false keeps every
// product and sum as written)

// (h, l) += b, with the rounding error of the sum kept in l (TwoSum).
template <typename V>
__host__ __device__ __forceinline__ void ff_acc(ffv<V> &s, V b)
{
    const V r = s.h + b, t = r - s.h;
    s.l = s.l + ((s.h - (r - t)) + (b - t));
    s.h = r;
}
template <typename V>
__host__ __device__ __forceinline__ void ff_acc(ffv<V> &s, ffv<V> b)
{
    s.l = s.l + b.l;
    ff_acc(s, b.h);
}
// (h, l) += k b for a short constant k: the sum's error as in TwoSum, with
// the remainder of the unrounded product k b from an FMA.  Exact up to 2^-47 of
// the larger term where h and k b have one sign, or k is a power of two.
template <typename V>
__host__ __device__ __forceinline__ void ff_acck(ffv<V> &s, float k, V b)
{
    const V r = vfma(k, b, s.h), t = r - s.h;
    s.l = s.l + ((s.h - (r - t)) + vfma(k, b, -t));
    s.h = r;
}
// (h, l) -= k b where |h| >= |k b| is known (the product split exactly, then
// Fast2Sum: with cancellation k b has to be a float for its sum to be exact).
template <typename V>
__host__ __device__ __forceinline__ void ff_subk_small(ffv<V> &s, float k, V b)
{
    const V z = k * b, r = s.h - z, t = r - s.h;
    s.l = (s.l - vfma(k, b, -z)) - (z + t);
    s.h = r;
}
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_norm(ffv<V> a)
{
    const V s = a.h + a.l;
    return {s, a.l - (s - a.h)};
}
// a b without the product of the low parts (below 2^-46 of a b)
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_mul(ffv<V> a, ffv<V> b)
{
    const V p = a.h * b.h;
    return {p, vfma(a.l, b.h, vfma(a.h, b.l, vfma(a.h, b.h, -p)))};
}
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_mul(ff a, ffv<V> b)
{
    return ff_mul(ff_all<V>(a), b);
}
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_sqr(ffv<V> a)
{
    const V p = a.h * a.h;
    return {p, vfma(a.h + a.h, a.l, vfma(a.h, a.h, -p))};
}
// d0 - 2 d1 + d2
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_diff2(ffv<V> d0, ffv<V> d1, ffv<V> d2)
{
    ffv<V> s = {d0.h, vfma(-2.0f, d1.l, d0.l + d2.l)};
    ff_acc(s, d2.h);
    ff_acck(s, -2.0f, d1.h);
    return s;  // (a sum that cancels leaves l as large as h: both only go into products)
}
// p + b q - c x for the indicators (p, q squares, x the product of their roots
// with |c x| <= p + b q)
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_form(ffv<V> p, float b, ffv<V> q, float c, ffv<V> x)
{
    ffv<V> s = {p.h, vfma(-c, x.l, vfma(b, q.l, p.l))};
    ff_acck(s, b, q.h);
    ff_subk_small(s, c, x.h);
    return s;
}
template <typename V, int = V::W>
__host__ __device__ __forceinline__ V rcp_seed(V a)
{
    float r[V::W];
#pragma unroll
    for (int i = 0; i < V::W; ++i) r[i] = rcp_seed(a[i]);
    return V::of(r);
}
// u with u u = (m / s)^2 up to 2^-44, as a float-float square: the seed
// r ~ 1/s leaves e = 1 - r s, and (m r)^2 (1 + 2 e) is (m / s)^2 to O(e^2).
template <typename V>
__host__ __device__ __forceinline__ ffv<V> ff_inv2(ffv<V> s, V m)
{
    const V r = rcp_seed(s.h);
    const V e = vfma(-r, s.l, vfma(-r, s.h, V::all(1.0f)));
    const V a = m * r, p = a * a;
    return {p, vfma(p, e + e, vfma(a, a, -p))};
}

// ---------------------------------------------------------------- WENO-5
// The part of one face's value that is not linear, from the first differences
// d0 .. d3 (v1 - v0, ..., v4 - v3) of its stencil.  The candidates of Eq.
// weno5_flux are 6 (G_1 - v2) = 5 d1 - 2 d0, 6 (G_2 - v2) = d1 + 2 d2,
// 6 (G_3 - v2) = 4 d2 - d3, so with the third differences t0 = d0 - 2 d1 + d2 and
// t1 = d1 - 2 d2 + d3 the face value F has
//   6 (F - v2) = d1 + 2 d2 - z,  z = (2 W_1 t0 + W_3 t1) / (W_1 + W_2 + W_3),
// W_q = delta_q / sigma_q^2 (up to a factor) with the indicators of
// Eq. weno5_sigma as the quadratic forms
//   sigma_1 = d0^2 - 11/4 d0 d1 + 5/2 d1^2,  sigma_2 = d1^2 - 5/4 d1 d2 + d2^2,
//   sigma_3 = d3^2 - 11/4 d2 d3 + 5/2 d2^2,
// each positive definite with condition number below 19.  q_j = d_j^2 and
// x_j = d_j d_{j+1} are shared by the faces of a line.  Weights are scaled by
// the power of two m below the smallest indicator.  Where an indicator
// vanishes (both its differences are zero) the weights are those of Table
// tab:weno (see ff_split).  Returns z.
template <typename V>
__host__ __device__ __forceinline__ ffv<V> weno5_ff(ffv<V> q0, ffv<V> q1, ffv<V> q2, ffv<V> q3, ffv<V> x0, ffv<V> x1,
                                                    ffv<V> x2, ffv<V> t0, ffv<V> t1)
{
    const ffv<V> s1 = ff_form(q0, 2.5f, q1, 2.75f, x0);
    const ffv<V> s2 = ff_form(q1, 1.0f, q2, 1.25f, x1);
    const ffv<V> s3 = ff_form(q3, 2.5f, q2, 2.75f, x2);
    float mi[V::W];
#pragma unroll
    for (int i = 0; i < V::W; ++i) mi[i] = f32_make(f32_bits(fminf(s1.h[i], fminf(s2.h[i], s3.h[i]))) & 0x7f800000u);
    const V m = V::of(mi);
    const ffv<V> w1 = ff_inv2(s1, m), w2 = ff_inv2(s2, m), w3 = ff_inv2(s3, m);  // (m / sigma_q)^2
    // weights 1 : 6 : 3 times w (delta_q times 10)
    ffv<V> den = {w1.h, vfma(3.0f, w3.l, vfma(6.0f, w2.l, w1.l))};
    ff_acck(den, 6.0f, w2.h);
    ff_acck(den, 3.0f, w3.h);
    const ffv<V> a = ff_mul(w1, t0), b = ff_mul(w3, t1);
    const V b3 = 3.0f * b.h;
    ffv<V> num = {a.h + a.h, vfma(2.0f, a.l, vfma(3.0f, b.l, vfma(3.0f, b.h, -b3)))};
    ff_acc(num, b3);
    // num / den: quotient of the leading parts and its remainder
    const V r = rcp_seed(den.h), z = num.h * r;
    return {z, (vfma(-z, den.l, vfma(-z, den.h, num.h)) + num.l) * r};
}

// The flux difference across a node, in the upwind direction and times 6: the
// value of the face ahead minus that of the face behind, whose non-linear parts
// are z1 and z0.  With v the node, db = v - (node behind), d = the difference
// before db's and da = (node ahead) - v, the linear parts add up to
// 2 da + 5 db - dbb.
template <typename V>
__host__ __device__ __forceinline__ ffv<V> weno5_flux6(ffv<V> dbb, ffv<V> db, ffv<V> da, ffv<V> z0, ffv<V> z1)
{
    const V b5 = 5.0f * db.h;
    ffv<V> s = {2.0f * da.h, vfma(2.0f, da.l, vfma(5.0f, db.l, vfma(5.0f, db.h, -b5))) - dbb.l + (z0.l - z1.l)};
    ff_acc(s, b5);
    ff_acc(s, -dbb.h);
    ff_acc(s, z0.h);
    ff_acc(s, -z1.h);
    return s;
}

// The value of one face from its upwind node and first differences, in FP64.
__host__ __device__ __forceinline__ double weno5_face(double v2, double d0, double d1, double d2, double d3, FfScale s)
{
    using F = ffv<vf1>;
    const double d[4][1] = {{d0}, {d1}, {d2}, {d3}};
    const F f0 = ff_split<vf1>(d[0], s), f1 = ff_split<vf1>(d[1], s), f2 = ff_split<vf1>(d[2], s),
            f3 = ff_split<vf1>(d[3], s);
    const F z = weno5_ff(ff_sqr(f0), ff_sqr(f1), ff_sqr(f2), ff_sqr(f3), ff_mul(f0, f1), ff_mul(f1, f2), ff_mul(f2, f3),
                         ff_diff2(f0, f1, f2), ff_diff2(f1, f2, f3));
    F c = {f1.h, vfma(2.0f, f2.l, f1.l) - z.l};
    ff_acc(c, 2.0f * f2.h);
    ff_acc(c, -z.h);
    return fma(1.0 / 6.0, ff_widen(ff_lane(c, 0), s), v2);
}

// W rows or columns of N nodes (W the floats of V) in the upwind direction, each
// `lane` elements after the one before: p0[0], p0[halo], p0[2 halo] are the three
// nodes behind a line, p1[i step] its nodes, p2[0] and p2[halo] the two ahead.
// store(i, v) takes the flux difference across node i (weno5_flux6).
// Differences, their squares and products and the third differences are formed
// once for the line.  The loop over the faces is unrolled by three: unrolled whole, a
// line is some 2000 instructions and the warps waited for the instruction cache.
template <int N, typename V, typename Store>
__device__ __forceinline__ void weno5_line(const double *p0, const double *p1, const double *p2, int lane, int halo,
                                           int step, FfScale s, Store store)
{
    double v[V::W];
#pragma unroll
    for (int i = 0; i < V::W; ++i) v[i] = p0[i * lane];
    auto next = [&](const double *p) {
        double d[V::W];
#pragma unroll
        for (int i = 0; i < V::W; ++i) {
            const double b = p[i * lane];
            d[i] = b - v[i];
            v[i] = b;
        }
        return ff_split<V>(d, s);
    };
    ffv<V> f0 = next(p0 + halo), f1 = next(p0 + 2 * halo), f2 = next(p1);
    const double *p = p1 + step;
    const V zero = V::all(0.0f);
    ffv<V> z0 = {zero, zero};
    ffv<V> q0 = ff_sqr(f0), q1 = ff_sqr(f1), q2 = ff_sqr(f2), x0 = ff_mul(f0, f1), x1 = ff_mul(f1, f2),
           t0 = ff_diff2(f0, f1, f2);
#pragma unroll 3
    for (int j = 0; j <= N; ++j) {
        if (j == N - 1) {
            p = p2;
            step = halo;
        }
        const ffv<V> f3 = next(p);
        p += step;
        const ffv<V> q3 = ff_sqr(f3), x2 = ff_mul(f2, f3), t1 = ff_diff2(f1, f2, f3);
        const ffv<V> z1 = weno5_ff(q0, q1, q2, q3, x0, x1, x2, t0, t1);
        q0 = q1; q1 = q2; q2 = q3;
        x0 = x1; x1 = x2;
        t0 = t1;
        if (j > 0) store(j - 1, weno5_flux6(f0, f1, f2, z0, z1));
        z0 = z1;
        f0 = f1; f1 = f2; f2 = f3;
    }
}

}  // namespace olb
