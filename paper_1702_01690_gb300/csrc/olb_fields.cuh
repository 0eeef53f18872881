// olb_fields.cuh -- what a stage needs at a node besides its populations: the
// moments (k_fields, one thread per node) and the force (k_force); for grids of at
// most one tile an SM both are taken by the stage's own CTAs (TileFields).
#pragma once

#include <type_traits>

#include "olb_kernels.cuh"

namespace olb {

// n and Delta p as the 49-point stencils read them.  The stencils
// cancel to O(ds^k) of their terms on fine grids, so the FP32 kernel keeps
// each value as an unevaluated sum hi + lo of two floats (hi = the value
// rounded to FP32, lo = the FP64 remainder rounded to FP32): differences of
// neighbouring values then keep ~FP64 accuracy at FP32 cost.
template <typename real>
struct FieldT {
    using type = double;
};
template <>
struct FieldT<float> {
    using type = float2;
};

__device__ __forceinline__ float field_diff(float2 a, float2 b) { return (a.x - b.x) + (a.y - b.y); }
__device__ __forceinline__ float field_val(float2 a) { return a.x + a.y; }

// ---------------------------------------------------------------- moments of a node
// n, u, T and Delta p of one node from its 25 populations (Sec. 2.2; T from
// the trace of Eq. sigmaq_def; Delta p = n T - p^w, Eq. vdw), and whether they
// are admissible (finite, n > 0, T > 0, b n < 1).  get(k) returns population
// k: the value (FP64) or the pair hi + lo (FP32).  SEQ: FP64 sums in FP64, one term
// after the other (olb_stage64l.cuh).
template <typename real>
struct NodeMoments;
template <>
struct NodeMoments<double> {
    double n, dp, ux, uy, T;
    int top;  // high word of the largest |population|, 0 if it is not finite (without SEQ)
    bool ok;
};
template <>
struct NodeMoments<float> {
    float2 n, dp, T, E;  // hi + lo pairs (E = sum |p|^2 f)
    float ux, uy;
    bool ok;
};

template <typename real, bool SEQ = false, typename Get>
__device__ __forceinline__ NodeMoments<real> node_moments(Get get, const Geo &g, const Tab<real> &t)
{
    NodeMoments<real> m;
    if constexpr (sizeof(real) == 8) {
        double n, jx, jy, en;
        if constexpr (SEQ) {
            // row and column sums of the 5 x 5 populations; the middle root is 0
            // (R[2] = R2[2] = 0), so its sums drop out of j and e
            double sx[NQ], sy[NQ];
#pragma unroll
            for (int k1 = 0; k1 < NQ; ++k1) {
                double s = get(NQ * k1);
                if (k1 == 0) sy[0] = s;
                else sy[0] += s;
#pragma unroll
                for (int k2 = 1; k2 < NQ; ++k2) {
                    const double v = get(NQ * k1 + k2);
                    s += v;
                    if (k1 == 0) sy[k2] = v;
                    else sy[k2] += v;
                }
                sx[k1] = s;
            }
            n = sx[0];
            jx = t.R[0] * sx[0];
            jy = t.R[0] * sy[0];
            en = t.R2[0] * (sx[0] + sy[0]);
#pragma unroll
            for (int k = 1; k < NQ; ++k) {
                n += sx[k];
                if (k == 2) continue;
                jx = fma(t.R[k], sx[k], jx);
                jy = fma(t.R[k], sy[k], jy);
                en = fma(t.R2[k], sx[k] + sy[k], en);
            }
        } else {
            const NodeSums s = node_sums64(get);
            m.top = finite_hi(s.top);
            n = s.n;
            jx = fma(t.R[4], s.a4x, t.R[3] * s.a3x);
            jy = fma(t.R[4], s.a4y, t.R[3] * s.a3y);
            en = fma(t.R2[4], s.s4, t.R2[3] * s.s3);
        }
        const double inv_n = recip_nr(n);
        const double ux = jx * inv_n, uy = jy * inv_n;
        const double T = 0.5 * fma(en, inv_n, -fma(ux, ux, uy * uy));
        // Delta p = n T - p^w, p^w = n T / (1 - b n) - a n^2 (Eq. vdw)
        const double nT = n * T;
        m.n = n;
        m.dp = nT - fma(nT, recip_nr(1.0 - g.b * n), -g.a * n * n);
        m.ux = ux;
        m.uy = uy;
        m.T = T;
        m.ok = (n > 0.0) && (T > 0.0) && (g.b * n < 1.0) && isfinite(n) && isfinite(T) && isfinite(ux) && isfinite(uy);
    } else {
        // FP32, compensated storage: row and column sums of the 5 x 5 pairs
        // as double-float values; n and e = sum |p|^2 f from them in
        // double-float arithmetic.  j needs FP32 accuracy of j itself:
        // R_4 (sx_4 - sx_0) + R_3 (sx_3 - sx_1) with the differences of the
        // double-float sums (R_0 = -R_4, R_1 = -R_3, R_2 = 0).
        f2 sx[NQ], sy[NQ];
        {
            float h[NQ], l[NQ];
#pragma unroll
            for (int k1 = 0; k1 < NQ; ++k1) {
#pragma unroll
                for (int k2 = 0; k2 < NQ; ++k2) {
                    const float2 v = get(NQ * k1 + k2);
                    h[k2] = v.x;
                    l[k2] = v.y;
                }
                sx[k1] = pair_sum5(h, l);
            }
#pragma unroll
            for (int k2 = 0; k2 < NQ; ++k2) {
#pragma unroll
                for (int k1 = 0; k1 < NQ; ++k1) {
                    const float2 v = get(NQ * k1 + k2);
                    h[k1] = v.x;
                    l[k1] = v.y;
                }
                sy[k2] = pair_sum5(h, l);
            }
        }
        const f2 one{1.0f, 0.0f};
        const f2 vdw_a = f2_of(g.a), vdw_b = f2_of(g.b);
        const f2 N = f2_add(f2_add(f2_add(sx[0], sx[4]), f2_add(sx[1], sx[3])), sx[2]);
        const float jx = fmaf(t.R[4], pdiff(sx[4].hi, sx[4].lo, sx[0].hi, sx[0].lo),
                              t.R[3] * pdiff(sx[3].hi, sx[3].lo, sx[1].hi, sx[1].lo));
        const float jy = fmaf(t.R[4], pdiff(sy[4].hi, sy[4].lo, sy[0].hi, sy[0].lo),
                              t.R[3] * pdiff(sy[3].hi, sy[3].lo, sy[1].hi, sy[1].lo));
        const f2 S4 = f2_add(f2_add(sx[0], sx[4]), f2_add(sy[0], sy[4]));
        const f2 S3 = f2_add(f2_add(sx[1], sx[3]), f2_add(sy[1], sy[3]));
        const f2 R24{t.R2[4], t.R2lo[4]}, R23{t.R2[3], t.R2lo[3]};
        const f2 Ea = f2_cmul(R24, S4.hi, S4.lo), Eb = f2_cmul(R23, S3.hi, S3.lo);
        const f2 E = f2_add(fast_two_sum(Ea.hi, Ea.lo), fast_two_sum(Eb.hi, Eb.lo));
        // u, T and Delta p = n T - p^w = n^2 (a - b T / (1 - b n)) (Eq. vdw):
        // T and Delta p in double-float arithmetic, so that the stencils of n
        // and Delta p see ~44-bit values without the FP64 pipe
        const f2 IN = f2_div(one, N);
        const float UX = jx * IN.hi, UY = jy * IN.hi;
        const f2 T = f2_scale(f2_add_f(f2_mul(E, IN), -fmaf(UX, UX, UY * UY)), 0.5f);
        const f2 BN = f2_mul(vdw_b, N);
        const f2 Q = f2_div(f2_mul(vdw_b, T), f2_add(one, f2_neg(BN)));
        const f2 DP = f2_mul(f2_mul(N, N), f2_add(vdw_a, f2_neg(Q)));
        m.n = make_float2(N.hi, N.lo);
        m.dp = make_float2(DP.hi, DP.lo);
        m.T = make_float2(T.hi, T.lo);
        m.E = make_float2(E.hi, E.lo);
        m.ux = UX;
        m.uy = UY;
        m.ok = (N.hi > 0.0f) && (T.hi > 0.0f) && (BN.hi < 1.0f) && isfinite(N.hi) && isfinite(T.hi) && isfinite(UX) &&
               isfinite(UY);
    }
    return m;
}

// Fields of the per-node pre-pass (k_fields), [ny][pitch] each: n and
// Delta p (FP32: hi + lo pairs), u_x, u_y, T (FP32: T a pair, and e = sum
// |p|^2 f as a pair for the equilibrium's correction).
template <typename real>
struct StageFields {
    using fld = typename FieldT<real>::type;
    fld *n, *dp, *T, *E;
    real *ux, *uy;
    typename std::conditional<sizeof(real) == 8, ff, float>::type *G[2];  // c F along x and y (k_force)
};

// Pointers of the fields in a buffer of planes of pitch * ny 8-byte elements
// (fields_bytes): FP64 n, Delta p, T, u_x, u_y, c F_x, c F_y; FP32 n, Delta p,
// T, e (float2 each), then u_x and u_y (float) sharing a plane, and c F_x and c
// F_y.
template <typename real>
__host__ __device__ inline StageFields<real> fields_of(void *base, const Geo &g)
{
    StageFields<real> f{};
    char *b = static_cast<char *>(base);
    const size_t plane = (size_t)g.plane * 8;
    f.n = reinterpret_cast<typename FieldT<real>::type *>(b);
    f.dp = reinterpret_cast<typename FieldT<real>::type *>(b + plane);
    f.T = reinterpret_cast<typename FieldT<real>::type *>(b + 2 * plane);
    if constexpr (sizeof(real) == 8) {
        f.E = nullptr;
        f.ux = reinterpret_cast<real *>(b + 3 * plane);
        f.uy = reinterpret_cast<real *>(b + 4 * plane);
        f.G[0] = reinterpret_cast<ff *>(b + 5 * plane);
        f.G[1] = reinterpret_cast<ff *>(b + 6 * plane);
    } else {
        f.E = reinterpret_cast<typename FieldT<real>::type *>(b + 3 * plane);
        f.ux = reinterpret_cast<real *>(b + 4 * plane);
        f.uy = reinterpret_cast<real *>(b + 4 * plane + plane / 2);
        f.G[0] = reinterpret_cast<real *>(b + 5 * plane);
        f.G[1] = reinterpret_cast<real *>(b + 5 * plane + plane / 2);
    }
    return f;
}

// One thread per node: the moments of f_s, stored for the stage kernel,
// which then reads them on its tile and halo instead of recomputing them
// at every halo position; inadmissible moments set bit 0 of the status.
template <typename real, bool SEQ = false>
__global__ void __launch_bounds__(256) k_fields(const real *__restrict__ fs, StageFields<real> out, int *status,
                                                const __grid_constant__ Geo g, const __grid_constant__ Tab<real> t)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)g.nx * g.ny) return;
    const int j = (int)(idx / g.nx), i = (int)(idx - (long long)j * g.nx);
    const long long o = (long long)j * g.pitch + i;
    NodeMoments<real> m;
    if constexpr (sizeof(real) == 8)
        m = node_moments<real, SEQ>([&](int k) { return __ldg(fs + k * g.plane + o); }, g, t);
    else
        m = node_moments<real>(
            [&](int k) { return make_float2(__ldg(fs + k * g.plane + o), __ldg(fs + (NK + k) * g.plane + o)); }, g, t);
    out.n[o] = m.n;
    out.dp[o] = m.dp;
    out.ux[o] = m.ux;
    out.uy[o] = m.uy;
    out.T[o] = m.T;
    if constexpr (sizeof(real) == 4) out.E[o] = m.E;
    if (!m.ok) atomicOr(status, 1);
}

// ---------------------------------------------------------------- batches
// 16-byte aligned and sized: the kernel copies one descriptor into shared
// memory with 16-byte loads, so consecutive array elements must stay aligned
// and the whole struct must be covered by whole int4 words.
template <typename real>
struct __align__(16) BatchRun {
    Geo g;
    Tab<real> t;
    long long off;   // populations: element offset in the three buffers
    long long foff;  // stage fields: byte offset in the fields buffer
    int ntx, pad;
    StageK k[3];  // constants of the three RK-3 stages (FP64)
    long long pad2;
};
static_assert(sizeof(BatchRun<double>) % 16 == 0, "BatchRun<double> must be a whole number of int4 words");
static_assert(sizeof(BatchRun<float>) % 16 == 0, "BatchRun<float> must be a whole number of int4 words");

// The run that item i belongs to: start is the prefix sum of the runs' items.
template <typename I>
__device__ __forceinline__ int run_of(const I *__restrict__ start, int nruns, I i)
{
    int lo = 0, hi = nruns - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(start + mid) <= i) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The moments pre-pass for a batch: one thread per node of every run (a
// grid-stride loop over the prefix sum node_start of the runs' node counts),
// writing each run's fields at its offset of the fields buffer.
template <typename real>
__global__ void __launch_bounds__(256) k_fields_batch(const real *__restrict__ fs, char *fields,
                                                      const BatchRun<real> *__restrict__ runs,
                                                      const long long *__restrict__ node_start, int nruns,
                                                      long long total, int *status)
{
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int lo = run_of(node_start, nruns, idx);
        const BatchRun<real> &run = runs[lo];
        const Geo &g = run.g;
        const long long q = idx - __ldg(node_start + lo);
        const int j = (int)(q / g.nx), i = (int)(q - (long long)j * g.nx);
        const long long o = (long long)j * g.pitch + i;
        const real *f = fs + run.off;
        NodeMoments<real> m;
        if constexpr (sizeof(real) == 8)
            m = node_moments<real>([&](int k) { return __ldg(f + k * g.plane + o); }, g, run.t);
        else
            m = node_moments<real>(
                [&](int k) { return make_float2(__ldg(f + k * g.plane + o), __ldg(f + (NK + k) * g.plane + o)); }, g,
                run.t);
        const StageFields<real> out = fields_of<real>(fields + run.foff, g);
        out.n[o] = m.n;
        out.dp[o] = m.dp;
        out.ux[o] = m.ux;
        out.uy[o] = m.uy;
        out.T[o] = m.T;
        if constexpr (sizeof(real) == 4) out.E[o] = m.E;
        if (!m.ok) atomicOr(status + lo, 1);
    }
}

// ---------------------------------------------------------------- force
// c F = (c/ds) sum_dp / n + (c sigma/ds^3) sum_n at every node from the 49-point
// stencils of Delta p and n (Eqs. F_def, stencil_grad, stencil_glap), in a launch
// of its own between the moments and the stage: inside the stage kernel it took
// 40 % of the time that a tile held its 70 KB of shared memory (loads of the
// halo's fields, differences and sums: 20 k of 46 k cycles a tile, measured with
// clock64), and three tiles are all that an SM holds.  Here blocks are small, 32
// x 8 nodes share a halo, and two nodes a thread keep the FP32 pipe busy.
//
// FP64: differences v(+l) - v(-l), l = 1..3, along x for every row of the block's region
// and along y for every column are taken once in FP64 (a value serves the seven
// nodes of a stencil row) and summed in float-float arithmetic.

// Terms of the 49-point stencils: the offset l of a difference, the row (column)
// m away that it is taken in, and its weight as a whole number, 5040 l w(l, |m|)
// and 2160 c(|m|, l).
struct StencilTerm {
    float w;
    short l, m;
};
__host__ __device__ constexpr float whole(double v) { return (float)(int)(v < 0 ? v - 0.5 : v + 0.5); }
template <bool LAPLACIAN>
struct StencilTerms {
    StencilTerm t[14];
    int n;
    constexpr StencilTerms() : t(), n(0)
    {
        for (int l = 1; l <= 3; ++l)
            for (int m = -3; m <= 3; ++m) {
                const int am = m < 0 ? -m : m;
                const float w = LAPLACIAN ? whole(2160.0 * glap_c(am, l)) : whole(5040.0 * l * grad_w(l, am));
                if (w != 0.0f) t[n++] = {w, (short)(l - 1), (short)m};
            }
    }
};

// The weighted sum for W nodes `lane` elements apart: h and l point to the parts
// of the first difference (l = 1, m = 0) of a node, sl and sm are the strides of
// l and m.
template <bool LAPLACIAN, typename V>
__device__ __forceinline__ ffv<V> stencil_sum(const float *h, const float *lo, int lane, int sl, int sm)
{
    constexpr StencilTerms<LAPLACIAN> c;
    ffv<V> s = {V::all(0.0f), V::all(0.0f)};
#pragma unroll
    for (int i = 0; i < c.n; ++i) {
        const float w = c.t[i].w;
        const int at = c.t[i].l * sl + c.t[i].m * sm;
        float vh[V::W], vl[V::W];
#pragma unroll
        for (int j = 0; j < V::W; ++j) {
            vh[j] = h[at + j * lane];
            vl[j] = lo[at + j * lane];
        }
        const V a = V::of(vh), z = w * a;
        s.l = s.l + vfma(w, V::of(vl), vfma(w, a, -z));
        ff_acc(s, z);
    }
    return s;
}

// Index of a node or of the node that a position beyond a side takes its fields
// from (Sec. 3.4.3): even reflection about walls and mirror planes, else wrapped.
__device__ __forceinline__ int field_index(int i, int n, bool mirror)
{
    if (i >= 0 && i < n) return i;
    if (!mirror) return wrap(i, n);
    return max(0, min(n - 1, i < 0 ? -1 - i : 2 * n - 1 - i));  // (further out: read by no node of the grid)
}

constexpr int FORCE_X = 32, FORCE_Y = 8, FORCE_THREADS = FORCE_X * FORCE_Y / 2;
template <int FX, int FY>
struct ForceSmem {
    static constexpr int HX = FX + 6, HY = FY + 6;
    double v[2][HY][HX];  // Delta p, n
    float dx[2][2][3][HY][FX];
    float dy[2][2][3][FY][HX];
    int top;
};

// differences of the block's fields v, by all NT threads
template <int NT, int FX, int FY>
__device__ __forceinline__ void force_differences(ForceSmem<FX, FY> &sm, FfScale sc)
{
    constexpr int HX = FX + 6, HY = FY + 6;
    // a row of the region, or a row of the block, at a time per warp lane
    for (int e = threadIdx.x; e < 2 * HY * FX; e += NT) {
        const int x = e % FX, r = e / FX % HY, k = e / (FX * HY);
        const double *v = &sm.v[k][r][x + 3];
#pragma unroll
        for (int l = 1; l <= 3; ++l) {
            const ff d = ff_split(v[l] - v[-l], sc);
            sm.dx[k][0][l - 1][r][x] = d.h;
            sm.dx[k][1][l - 1][r][x] = d.l;
        }
    }
    for (int e = threadIdx.x; e < 2 * FY * HX; e += NT) {
        const int x = e % HX, y = e / HX % FY, k = e / (HX * FY);
        const double *v = &sm.v[k][y + 3][x];
#pragma unroll
        for (int l = 1; l <= 3; ++l) {
            const ff d = ff_split(v[l * HX] - v[-l * HX], sc);
            sm.dy[k][0][l - 1][y][x] = d.h;
            sm.dy[k][1][l - 1][y][x] = d.l;
        }
    }
}
// c F along axis a at node (x, y) of the block and, two lanes, (x, y + 4)
template <typename V, int FX, int FY>
__device__ __forceinline__ ffv<V> force_at(const ForceSmem<FX, FY> &sm, FfScale sc, const StageK &c, int a, int x, int y)
{
    constexpr int HX = FX + 6, HY = FY + 6;
    double nd[V::W];
#pragma unroll
    for (int i = 0; i < V::W; ++i) nd[i] = sm.v[1][y + 3 + 4 * i][x + 3];
    const ffv<V> n = ff_split<V>(nd, sc);
    const V r = rcp_seed(n.h);
    const ffv<V> inv = {r, r * vfma(-r, n.l, vfma(-r, n.h, V::all(1.0f)))};
    // kn sum_n is 2^k of the product of its scaled parts
    const int k = c.kn_exp + 127 - 1023 - (sc.off >> 20), k1 = max(-126, min(127, k)), k2 = max(-126, min(127, k - k1));
    const float u1 = f32_make((unsigned)(k1 + 127) << 23), u2 = f32_make((unsigned)(k2 + 127) << 23);
    const float *d = a == 0 ? &sm.dx[0][0][0][y + 3][x] : &sm.dy[0][0][0][y][x + 3];
    constexpr int NX = 3 * HY * FX, NY = 3 * FY * HX;
    const int part = a == 0 ? NX : NY, lane = 4 * (a == 0 ? FX : HX), sr = a == 0 ? FX : 1;
    const ffv<V> sp = stencil_sum<false, V>(d, d + part, lane, part / 3, sr);
    const ffv<V> sn = stencil_sum<true, V>(d + 2 * part, d + 3 * part, lane, part / 3, sr);
    ffv<V> v = ff_mul(c.kp, ff_mul(sp, inv));
    const ffv<V> w = ff_mul(c.kn, sn);
    v.l = v.l + u2 * (u1 * w.l);
    ff_acc(v, u2 * (u1 * w.h));
    return ff_norm(v);
}

__device__ __forceinline__ void force_block(ForceSmem<FORCE_X, FORCE_Y> &sm, const StageFields<double> &f, const Geo &g,
                                            const StageK &c, int x0, int y0)
{
    constexpr int HX = FORCE_X + 6, HY = FORCE_Y + 6;
    const int tid = threadIdx.x;
    if (tid == 0) sm.top = 0;
    __syncthreads();
    int top = 0;
    for (int e = tid; e < HY * HX; e += FORCE_THREADS) {
        const int r = e / HX, x = e - r * HX;
        const long long o = (long long)field_index(y0 - 3 + r, g.ny, g.spec_y) * g.pitch + field_index(x0 - 3 + x, g.nx, g.walls);
        const double n = f.n[o];
        sm.v[0][r][x] = f.dp[o];
        sm.v[1][r][x] = n;
        top = max(top, finite_hi(abs_hi(n)));
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if ((tid & 31) == 0) atomicMax(&sm.top, top);
    __syncthreads();
    const FfScale sc = ff_scale(sm.top);
    force_differences<FORCE_THREADS>(sm, sc);
    __syncthreads();
    const int x = tid % FORCE_X, y = tid / FORCE_X;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const ffv<vf2> v = force_at<vf2>(sm, sc, c, a, x, y);
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (x0 + x < g.nx && y0 + y + 4 * i < g.ny)
                f.G[a][(long long)(y0 + y + 4 * i) * g.pitch + (x0 + x)] = ff_lane(v, i);
    }
}

// FP32: n and Delta p as pairs hi + lo.  grad(Delta p) in FP32 from differences of
// pairs; the capillary stencil cancels its O(ds) terms down to O(ds^3) (a factor
// ~1/(ds k)^2 on fine grids), so its weighted differences are summed in
// double-float arithmetic with double-float weights (exact products of the hi
// parts, TwoSum accumulation): the sum keeps FP32 accuracy of itself, not of its
// terms.
template <int FX, int FY>
struct ForceSmem32 {
    static constexpr int HX = FX + 6, HY = FY + 6;
    float2 dp[HY][HX], n[HY][HX];
};
// sums along x (y) at the node whose field is *v, fields sl apart along the
// direction of the derivative and sm across it
__device__ __forceinline__ float grad_sum32(const float2 *v, int sl, int sm)
{
    float acc = 0.0f;
#pragma unroll
    for (int l = 1; l <= 3; ++l)
#pragma unroll
        for (int m = -3; m <= 3; ++m) {
            const int am = m < 0 ? -m : m;
            if (grad_w(l, am) != 0.0)
                acc = fmaf((float)(l * grad_w(l, am)), field_diff(v[m * sm + l * sl], v[m * sm - l * sl]), acc);
        }
    return acc;
}
__device__ __forceinline__ float glap_sum32(const float2 *v, int sl, int sm)
{
    f2 sum{0.0f, 0.0f};
#pragma unroll
    for (int l = 1; l <= 3; ++l)
#pragma unroll
        for (int m = -3; m <= 3; ++m) {
            const int am = m < 0 ? -m : m;
            if (glap_c(am, l) != 0.0) {
                const float wh = (float)glap_c(am, l);
                const float wl = (float)(glap_c(am, l) - (double)(float)glap_c(am, l));
                const float2 a = v[m * sm + l * sl], b = v[m * sm - l * sl];
                const f2 dh = two_sum(a.x, -b.x);
                const float dl = dh.lo + (a.y - b.y);
                const float p = wh * dh.hi;
                const float e = fmaf(wh, dh.hi, -p);
                const float tl = fmaf(wh, dl, fmaf(wl, dh.hi, e));
                const f2 t2 = two_sum(sum.hi, p);
                sum = f2{t2.hi, t2.lo + (sum.lo + tl)};
            }
        }
    return sum.hi + sum.lo;
}
// c F along axis a at node (x, y) of the block; cc: the stage's coefficient of dt L
template <int FX, int FY>
__device__ __forceinline__ float force_at32(const ForceSmem32<FX, FY> &sm, const Geo &g, float cc, int a, int x, int y)
{
    constexpr int HX = FX + 6;
    const float2 *dp = &sm.dp[y + 3][x + 3], *n = &sm.n[y + 3][x + 3];
    const float dn = (float)g.inv_ds / field_val(*n), sg3 = (float)g.sigma * (float)g.inv_ds3;
    const int sl = a == 0 ? 1 : HX, sm_ = a == 0 ? HX : 1;
    return cc * fmaf(grad_sum32(dp, sl, sm_), dn, sg3 * glap_sum32(n, sl, sm_));
}
__device__ __forceinline__ void force_block32(ForceSmem32<FORCE_X, FORCE_Y> &sm, const StageFields<float> &f, const Geo &g,
                                              float cc, int x0, int y0)
{
    constexpr int HX = FORCE_X + 6, HY = FORCE_Y + 6;
    for (int e = threadIdx.x; e < HY * HX; e += 2 * FORCE_THREADS) {
        const int r = e / HX, x = e - r * HX;
        const long long o = (long long)field_index(y0 - 3 + r, g.ny, g.spec_y) * g.pitch + field_index(x0 - 3 + x, g.nx, g.walls);
        sm.dp[r][x] = f.dp[o];
        sm.n[r][x] = f.n[o];
    }
    __syncthreads();
    const int x = threadIdx.x % FORCE_X, y = threadIdx.x / FORCE_X;
    if (x0 + x >= g.nx || y0 + y >= g.ny) return;
    const long long o = (long long)(y0 + y) * g.pitch + (x0 + x);
    f.G[0][o] = force_at32(sm, g, cc, 0, x, y);
    // (one axis after the other: mixed by the compiler they took 114 registers instead of
    // 42, and k_force of 2048^2 0.180 ms instead of 0.127)
    asm volatile("" ::: "memory");
    f.G[1][o] = force_at32(sm, g, cc, 1, x, y);
}

template <typename real>
struct ForceOf {
    using Smem = ForceSmem<FORCE_X, FORCE_Y>;
    static constexpr int NT = FORCE_THREADS, CTAS = 5;
};
template <>
struct ForceOf<float> {
    using Smem = ForceSmem32<FORCE_X, FORCE_Y>;
    static constexpr int NT = 2 * FORCE_THREADS, CTAS = 4;
};
template <typename real>
__global__ void __launch_bounds__(ForceOf<real>::NT, ForceOf<real>::CTAS) k_force(StageFields<real> f, const __grid_constant__ Geo g,
                                                             const __grid_constant__ StageK c, real cc,
                                                             int row0)
{
    __shared__ typename ForceOf<real>::Smem sm;
    const int x0 = blockIdx.x * FORCE_X, y0 = (row0 + blockIdx.y) * FORCE_Y;
    if constexpr (sizeof(real) == 8) force_block(sm, f, g, c, x0, y0);
    else force_block32(sm, f, g, cc, x0, y0);
}

// the blocks of every run, in the order of force_start (prefix sum of their numbers)
template <typename real>
__global__ void __launch_bounds__(ForceOf<real>::NT, ForceOf<real>::CTAS) k_force_batch(char *fields, const BatchRun<real> *__restrict__ runs,
                                                                   const int *__restrict__ force_start, int nruns, int st,
                                                                   real ccoef)
{
    __shared__ typename ForceOf<real>::Smem sm;
    const int lo = run_of(force_start, nruns, (int)blockIdx.x);
    const BatchRun<real> &run = runs[lo];
    const int b = blockIdx.x - __ldg(force_start + lo), nbx = (run.g.nx + FORCE_X - 1) / FORCE_X;
    const StageFields<real> f = fields_of<real>(fields + run.foff, run.g);
    const int x0 = b % nbx * FORCE_X, y0 = b / nbx * FORCE_Y;
    if constexpr (sizeof(real) == 8) force_block(sm, f, run.g, run.k[st], x0, y0);
    else force_block32(sm, f, run.g, ccoef * (real)run.g.dt, x0, y0);
}

// ---------------------------------------------------------------- fields of one tile
// Moments and stencils' input of an 8 x 8 tile whose CTA takes them itself (stage
// kernels with KP 8): n and Delta p of the 14 x 14 nodes that the stencils of its
// nodes read, the other moments of its nodes.
template <typename real>
struct TileFields;
template <>
struct TileFields<double> {
    ForceSmem<8, 8> force;
    double T[64], ux[64], uy[64];
};
template <>
struct TileFields<float> {
    ForceSmem32<8, 8> force;
    float2 T[64], E[64];
    float ux[64], uy[64];
};
constexpr int OWN_THREADS = 7 * 32;  // 14 x 14 nodes, one a thread
// Threads 0 .. OWN_THREADS - 1, whole warps: the moments of a node (those of k_fields,
// from the nodes that k_force's blocks take), the status of the tile's own nodes; FP64
// the largest population (*top) and density (own.force.top) of the 14 x 14 nodes.
template <typename real>
__device__ __forceinline__ void tile_moments(TileFields<real> &own, int *top, const real *__restrict__ fs, int *status,
                                             const Geo &g, const Tab<real> &t, int x0, int y0)
{
    const int tid = threadIdx.x, r = tid / 14, x = tid - 14 * r;
    int a = 0, an = 0;
    if (r < 14) {
        const real *f = fs + (long long)field_index(y0 - 3 + r, g.ny, g.spec_y) * g.pitch + field_index(x0 - 3 + x, g.nx, g.walls);
        NodeMoments<real> m;
        const bool mine = r >= 3 && r < 11 && x >= 3 && x < 11;
        const int node = 8 * (r - 3) + x - 3;
        if constexpr (sizeof(real) == 8) {
            m = node_moments<real>([&](int k) { return __ldg(f + k * g.plane); }, g, t);
            own.force.v[0][r][x] = m.dp;
            own.force.v[1][r][x] = m.n;
            a = m.top;
            an = finite_hi(abs_hi(m.n));
        } else {
            m = node_moments<real>([&](int k) { return make_float2(__ldg(f + k * g.plane), __ldg(f + (NK + k) * g.plane)); },
                                   g, t);
            own.force.dp[r][x] = m.dp;
            own.force.n[r][x] = m.n;
            if (mine) own.E[node] = m.E;
        }
        if (mine) {
            own.ux[node] = m.ux;
            own.uy[node] = m.uy;
            own.T[node] = m.T;
            if (!m.ok && x0 + x - 3 < g.nx && y0 + r - 3 < g.ny) atomicOr(status, 1);
        }
    }
    if constexpr (sizeof(real) == 8) {
        a = __reduce_max_sync(0xffffffffu, a);
        an = __reduce_max_sync(0xffffffffu, an);
        if ((tid & 31) == 0) {
            atomicMax(top, a);
            atomicMax(&own.force.top, an);
        }
    }
}

}  // namespace olb
