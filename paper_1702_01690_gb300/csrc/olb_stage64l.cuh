// olb_stage64l.cuh -- force and stage of an FP64 tile with learned weights, in FP64.
//
// The network takes its stencil in FP32 and acts behind a guard that is a comparison
// (learned_guard): a last bit of a population that rounds another way moves a weight
// by 1e-7, now and then a face from one set of weights to the other, and a hundred
// steps carry that to 1e-6 of the velocity.  So the populations keep the rounding that
// learned runs have always had: sums, force, faces and node updates are the FP64
// operations of Eqs. rk3, derf and feq in this order, not the float-float arithmetic of
// olb_stage64.cuh (with which two runs of 100 steps of 308 x 4 nodes differed by 1.5e-8
// of u, one of 44 x 188 by 4.5e-8).
//
// One stage of 1024^2 (with moments and force), the network acting on nearly every
// face: 6.84 -> 4.9 ms; on few (a drop): 6.55 -> 5.6 ms.  The network takes most of the
// first (olb_mlp.cuh), with the FP64 operations beside it on the two tiles that an SM
// holds; the second is bound by the FP64 pipe, some 2500 operations a node.  Faces that
// the network leaves to Jiang-Shu among others are gathered for whole warps (5.14 ->
// 4.95 ms, noise); differences are rounded to FP32 on the integer pipe (drop 6.17 ->
// 5.95 ms); a warp of Jiang-Shu faces only takes them at once (5.95 -> 5.6 ms).
#pragma once

#include "olb_tile.cuh"

namespace olb {

// c F at every node, in FP64 (G as doubles).
__device__ __forceinline__ double grad_sum64(const double *v, int sl, int sm)
{
    double acc = 0.0;
#pragma unroll
    for (int l = 1; l <= 3; ++l)
#pragma unroll
        for (int m = -3; m <= 3; ++m) {
            const int am = m < 0 ? -m : m;
            if (grad_w(l, am) != 0.0) acc = fma(l * grad_w(l, am), v[m * sm + l * sl] - v[m * sm - l * sl], acc);
        }
    return acc;
}
__device__ __forceinline__ double glap_sum64(const double *v, int sl, int sm)
{
    double acc = 0.0;
#pragma unroll
    for (int l = 1; l <= 3; ++l)
#pragma unroll
        for (int m = -3; m <= 3; ++m) {
            const int am = m < 0 ? -m : m;
            if (glap_c(am, l) != 0.0) acc = fma(glap_c(am, l), v[m * sm + l * sl] - v[m * sm - l * sl], acc);
        }
    return acc;
}
template <typename real>
__global__ void __launch_bounds__(2 * FORCE_THREADS) k_force_learned(StageFields<real> f, const __grid_constant__ Geo g,
                                                                     real cc, int row0)
{
    constexpr int HX = FORCE_X + 6, HY = FORCE_Y + 6;
    __shared__ double dp[HY][HX], n[HY][HX];
    const int x0 = blockIdx.x * FORCE_X, y0 = (row0 + blockIdx.y) * FORCE_Y;
    for (int e = threadIdx.x; e < HY * HX; e += 2 * FORCE_THREADS) {
        const int r = e / HX, x = e - r * HX;
        const long long o = (long long)field_index(y0 - 3 + r, g.ny, g.spec_y) * g.pitch + field_index(x0 - 3 + x, g.nx, g.walls);
        dp[r][x] = f.dp[o];
        n[r][x] = f.n[o];
    }
    __syncthreads();
    const int x = threadIdx.x % FORCE_X, y = threadIdx.x / FORCE_X;
    if (x0 + x >= g.nx || y0 + y >= g.ny) return;
    const double *d = &dp[y + 3][x + 3], *v = &n[y + 3][x + 3];
    const double dn = g.inv_ds / *v, sg3 = g.sigma * g.inv_ds3;
    const long long o = (long long)(y0 + y) * g.pitch + (x0 + x);
    reinterpret_cast<double *>(f.G[0])[o] = cc * fma(grad_sum64(d, 1, HX), dn, sg3 * glap_sum64(v, 1, HX));
    reinterpret_cast<double *>(f.G[1])[o] = cc * fma(grad_sum64(d, HX, 1), dn, sg3 * glap_sum64(v, HX, 1));
}

// KP (stage_kind) 4: 256 threads, 6: 512.
template <int KP>
struct Smem64L : Staged<double> {
    static constexpr int NT = KP == 6 ? 512 : 256, NFX = (TX + 1) * TY, NFY = TX * (TY + 1), FACES = 20 * (NFX + NFY);
    double E[NQ][NN];   // (c/tau) n g_q(u_x, T)
    double gy[NQ][NN];  // g_q(u_y, T)
    double G[2][NN];    // c F
    // faces of the 20 velocities that move along the axis
    double fx[20][TY][TX + 1];
    double fy[20][TY + 1][TX];
    int njs;                    // faces that the network does not act on
    unsigned short js[FACES];
};

// A face of the tile: velocity k, its stencil's differences in the upwind direction, its
// upwind node and the place of its value.
struct LearnedFace {
    double d[4], v2;
    double *at;
};
template <typename S>
__device__ __forceinline__ bool learned_face(S &sm, const Geo &g, int x0, int y0, int e, LearnedFace &face)
{
    const bool along_x = e < 20 * S::NFX;
    const int e2 = along_x ? e : e - 20 * S::NFX, nf = along_x ? S::NFX : S::NFY, q = e2 / nf, f = e2 - q * nf;
    const int k = line_velocity(along_x, q);
    const int r = along_x ? f / (S::TX + 1) : f / S::TX, c = along_x ? f - r * (S::TX + 1) : f - r * S::TX;
    if (along_x ? (y0 + r >= g.ny || x0 + c > g.nx) : (x0 + c >= g.nx || y0 + r > g.ny)) return false;
    const bool up = along_x ? k / NQ > 2 : k % NQ > 2;
    double v[5];
#pragma unroll
    for (int m = 0; m < 5; ++m)
        v[m] = along_x ? sm.mid[k][r][up ? c + 1 + m : c + 6 - m] : *sm.at(k, up ? r + m : r + 5 - m, 4 + c);
#pragma unroll
    for (int m = 0; m < 4; ++m) face.d[m] = v[m + 1] - v[m];
    face.v2 = v[2];
    face.at = along_x ? &sm.fx[q][r][c] : &sm.fy[q][r][c];
    return true;
}

// One stage of a tile (stage_tile64); ca, cb, cc: the coefficients of f^n, f_s and dt L.
template <int KP>
__device__ __forceinline__ bool stage_tile64l(Smem64L<KP> &sm, const double *__restrict__ fs, const double *fn, double *out,
                                              int *__restrict__ status, const Geo &g, const Tab<double> &t, int x0, int y0,
                                              double ca, double cb, double cc, const MlpArg &net, const TmaMap *tmap,
                                              const StageFields<double> &fields)
{
    using S = Smem64L<KP>;
    constexpr int NT = S::NT, TX = S::TX, TY = S::TY, NN = S::NN;
    const int tid = threadIdx.x;
    const double cit = cc * g.inv_tau, cf = cb - cit, cadv = cc * g.inv_ds;

    // ---- 1. the fields of a node and axis, the populations
    const int a = tid / NN, node = tid % NN, nx = node % TX, ny = node / TX;
    const bool has = tid < 2 * NN && x0 + nx < g.nx && y0 + ny < g.ny;
    double n = 0.0, u = 0.0, T = 1.0, G = 0.0;
    if (has) {
        const long long o = (long long)(y0 + ny) * g.pitch + (x0 + nx);
        n = fields.n[o];
        u = a == 0 ? fields.ux[o] : fields.uy[o];
        T = fields.T[o];
        G = reinterpret_cast<const double *>(a == 0 ? fields.G[0] : fields.G[1])[o];
    }
    if (tid == 0) sm.njs = 0;
    const bool inside = tmap != nullptr && x0 >= 4 && x0 + TX + 4 <= g.nx && y0 >= 3 && y0 + TY + 3 <= g.ny;
    if (inside) tma_issue(sm, tmap, x0, y0);
    else load_region(sm, fs, g, x0, y0);
    __syncthreads();

    // ---- 2. equilibrium factors
    if (tid < 2 * NN) {
        double w[NQ];
        eq_factors<double>(t, u, T, w);
        const double cn = cit * n;
#pragma unroll
        for (int q = 0; q < NQ; ++q) (a == 0 ? sm.E : sm.gy)[q][node] = a == 0 ? cn * w[q] : w[q];
        sm.G[a][node] = G;
    }
    // ---- 3. diffuse walls: fluxes and ghosts of the tile rows
    const bool left = x0 == 0 && g.wall_lo, right = x0 + TX + 3 >= g.nx && g.wall_hi;
    if (left || right) {
        wall_flux<double, true>(sm, g, t, t, net.theta, x0, 2 * NN, left, right);
        __syncthreads();
        wall_ghosts<double>(sm, g, t, x0, 0, left, right);
    }
    if (inside && !tma_finish(sm, status)) return false;
    __syncthreads();

    // ---- 4. faces: those that the network acts on, whole warps; the others, unless they
    // fill a warp, are collected and taken by whole warps then (a warp's FP64 instruction
    // costs the same for one lane as for all)
    float *const scratch = net.tables + MLP_T64_SIZE + (tid >> 5) * MLP_WARP_SCRATCH;
    for (int e = tid; e < (S::FACES + 31) / 32 * 32; e += NT) {
        LearnedFace f{};
        const bool valid = e < S::FACES && learned_face(sm, g, x0, y0, e, f);
        const float d[4] = {f32_rounded(f.d[0]), f32_rounded(f.d[1]), f32_rounded(f.d[2]), f32_rounded(f.d[3])};
        const bool acts = valid && learned_guard(f.d, d);
        float x[MLP_IN], w[MLP_OUT];
        learned_input_x(d, acts, x);
        if (__any_sync(0xffffffffu, acts)) mlp_weights_warp64(net.tables, x, w, scratch);
        if (acts) *f.at = f.v2 + (double)learned_corr_from(w, d);
        const unsigned rest = __ballot_sync(0xffffffffu, valid && !acts);
        if (rest == 0xffffffffu) {
            *f.at = weno5_js(f.d, f.v2);
        } else if (rest) {
            int first = 0;
            if ((tid & 31) == 0) first = atomicAdd(&sm.njs, __popc(rest));
            first = __shfl_sync(0xffffffffu, first, 0);
            if (valid && !acts) sm.js[first + __popc(rest & ((1u << (tid & 31)) - 1u))] = (unsigned short)e;
        }
    }
    __syncthreads();
    for (int i = tid; i < sm.njs; i += NT) {
        LearnedFace f{};
        learned_face(sm, g, x0, y0, sm.js[i], f);
        *f.at = weno5_js(f.d, f.v2);
    }

    // f^n of the column that this thread advances, fetched now
    constexpr int COLS = (NQ * NN + NT - 1) / NT;
    double f0[COLS][NQ];
    if (ca != 0.0)
#pragma unroll
        for (int w = 0; w < COLS; ++w) {
            const int e = tid + w * NT, k2 = e / NN, nd = e - k2 * NN, x = x0 + nd % TX, y = y0 + nd / TX;
            if (e >= NQ * NN || x >= g.nx || y >= g.ny) continue;
#pragma unroll
            for (int k1 = 0; k1 < NQ; ++k1) f0[w][k1] = fn[(NQ * k1 + k2) * g.plane + (long long)y * g.pitch + x];
        }
    __syncthreads();

    // ---- 5. node updates: c L = -c xi.grad f - c F.grad_p f - (c/tau)(f - f^eq) with
    // f^eq = n g g (Eqs. feq, g_alpha), combined with b f (and a f_n) as in Eq. rk3;
    // thread (node, k2) advances the five velocities 5 k1 + k2
#pragma unroll
    for (int w = 0; w < COLS; ++w) {
        const int e = tid + w * NT, k2 = e / NN, nd = e - k2 * NN, x = nd % TX, y = nd / TX;
        if (e >= NQ * NN || x0 + x >= g.nx || y0 + y >= g.ny) continue;
        const double Gx = sm.G[0][nd], Gy = sm.G[1][nd], gyk = sm.gy[k2][nd];
        double col[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) col[q] = sm.mid[NQ * q + k2][y][x + 4];
        double *o = out + k2 * g.plane + (long long)(y0 + y) * g.pitch + (x0 + x);
#pragma unroll
        for (int k1 = 0; k1 < NQ; ++k1) {
            double dx = 0.0, dy = 0.0;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                dx = fma(t.D[k1][q], col[q], dx);
                dy = fma(t.D[k2][q], sm.mid[NQ * k1 + q][y][x + 4], dy);
            }
            double adv = 0.0;
            if (k1 != 2) {
                const double *fx = &sm.fx[NQ * (k1 < 2 ? k1 : k1 - 1) + k2][y][x];
                adv = t.R[k1] * (fx[1] - fx[0]);
            }
            if (k2 != 2) {
                const double *fy = &sm.fy[4 * k1 + (k2 < 2 ? k2 : k2 - 1)][y][x];
                adv = fma(t.R[k2], fy[TX] - fy[0], adv);
            }
            double v = fma(cf, col[k1], fma(sm.E[k1][nd], gyk, -fma(Gx, dx, fma(Gy, dy, cadv * adv))));
            if (ca != 0.0) v = fma(ca, f0[w][k1], v);
            o[NQ * k1 * g.plane] = v;
        }
    }
    return true;
}

}  // namespace olb
