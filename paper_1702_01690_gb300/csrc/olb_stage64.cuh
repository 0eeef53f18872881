// olb_stage64.cuh -- force, fluxes, collision and RK-3 combination of an FP64
// tile (phases 4 and 5 of the stage kernel, olb_fused.cuh).
//
// The stage writes out = f_s + Delta with
//   Delta = ca (f^n - f_s) + (c/tau) (f^eq - f_s) - c xi.grad f - c F.grad_p f,
// c the stage's coefficient of dt L (Eq. rk3; cb = 1 - ca).  Each term of Delta
// is a difference, or is formed from differences, of numbers of the size of f,
// and is small against f.  The FP64 pipe, which starts one operation where the
// FP32 pipe starts 64, therefore only takes the differences themselves (of
// populations along a row, of n and Delta p across a stencil, f^n - f_s,
// f^eq - f_s) and the sum f_s + Delta; what is done with them runs on the FP32
// pipe in float-float arithmetic (olb_ff.cuh), whose 2^-46 of Delta is below
// FP64's rounding of f wherever Delta < f / 128.
//
// Measured, one step (three stages) of a 4096^2 grid: 106.6 ms with the force and
// the node updates in FP64 (1070 FP64 instructions a node and stage beside 60
// differences), 56.8 ms like this (228); 24-run sweep, 8 steps: 39.7 -> 24.1 ms.
// Against 80-bit arithmetic the populations are closer than the FP64 form's
// (12 steps of a 167 x 109 drop: 5.7e-16 instead of 1.2e-15 of their norm, and
// its loss of 1e-15 of the mass is gone): Delta is summed before the one
// rounding at the size of f.
#pragma once

#include "olb_ff.cuh"
#include "olb_internal.cuh"
#include "olb_mlp.cuh"

namespace olb {

// ---------------------------------------------------------------- shared memory
template <int TX, int TY, int KP, bool LEARNED>
struct Smem64 {
    // LS: threads per velocity lane, the tile's nodes rounded up to whole
    // warps; NT threads in all; HP: pitch of a staged row of populations
    static constexpr int HX = TX + 8, HY = TY + 6, NN = TX * TY, LS = (NN + 31) / 32 * 32, NT = LS * KP;
    static constexpr int HP = region_pitch(TX, true);
    static_assert(NN <= 64, "FP64 tiles hold at most 64 nodes");
    // populations of the tile's rows (columns x0 - 4 ...) and of the three rows
    // below and above its nodes
    alignas(128) double mid[NK][TY][HP];
    alignas(128) double below[NK][3][TX];
    alignas(128) double above[NK][3][TX];
    double ex[NQ][NN];  // n g_q(u_x, T) and g_q(u_y, T) of the tile nodes
    double ey[NQ][NN];
    ff G[2][NN];        // c F
    union {
        // phases 2 to 4: fields of the region, and differences v(+l) - v(-l),
        // l = 1..3, of Delta p and n, along x for every row of the region and
        // along y for every column that a stencil of the tile reaches: a value
        // serves the seven nodes of a stencil row
        struct {
            double n[HY][HX];
            double dp[HY][HX];
            double ux[TY][TX];
            double uy[TY][TX];
            double T[TY][TX];
            ff dx[2][3][HY][TX];
            ff dy[2][3][TY][TX + 6];
        };
        // phase 5: flux differences times 6 (weno5_flux6) across the nodes of
        // each row along x and column along y, of the 20 velocities that move
        // along the axis (slot_x, slot_y; learned weights: first the faces'
        // non-linear parts, one more than nodes, which the flux differences then
        // replace); then, in place of one of a velocity's flux differences (inc),
        // the sum of its advection and y force terms
        struct {
            ff ax[20][TY][TX + 1];
            ff ay[20][TX][TY + 1];
            ff rest[NN];
        };
    };
    double wnw[2][TY];        // wall density of each tile row (Eq. nw)
    int top;                  // high word of the largest n of the region (the tile's scale)
    unsigned long long mbar;  // completion barrier of the TMA copies

    // the staged population k at row r and column c of the region; planes lie
    // plane(r) apart; the corners of the region are not staged
    __device__ __forceinline__ double *at(int k, int r, int c)
    {
        return r < 3 ? &below[k][r][c - 4] : r < TY + 3 ? &mid[k][r - 3][c] : &above[k][r - TY - 3][c - 4];
    }
    __device__ __forceinline__ static constexpr bool staged(int r, int c)
    {
        return (r >= 3 && r < TY + 3) || (c >= 4 && c < TX + 4);
    }
    __device__ __forceinline__ static constexpr int plane(int r) { return r >= 3 && r < TY + 3 ? TY * HP : 3 * TX; }
    __device__ __forceinline__ ff &inc(int k1, int k2, int x, int y)
    {
        return k1 != 2 ? ax[NQ * (k1 < 2 ? k1 : k1 - 1) + k2][y][x] : k2 != 2 ? ay[8 + (k2 < 2 ? k2 : k2 - 1)][x][y] : rest[y * TX + x];
    }
};

// Slots of ax for the velocities with xi_x != 0 and of ay for those with xi_y != 0.
__device__ __forceinline__ int slot_x(int k1, int k2) { return NQ * (k1 < 2 ? k1 : k1 - 1) + k2; }
__device__ __forceinline__ int slot_y(int k1, int k2) { return 4 * k1 + (k2 < 2 ? k2 : k2 - 1); }

// ---------------------------------------------------------------- stencils
// The weights of the 49-point stencils (Eqs. stencil_grad, stencil_glap) as
// whole numbers: 5040 l w(l, |m|) and 2160 c(|m|, l).
__host__ __device__ constexpr int whole(double v) { return (int)(v < 0 ? v - 0.5 : v + 0.5); }

// sum over l, m of weight(l, |m|) d(l, m), d giving the difference at offsets
// +l, -l in the row (column) m away
template <bool LAPLACIAN, typename D>
__device__ __forceinline__ ff stencil_sum(D d)
{
    ff s = {0.0f, 0.0f};
#pragma unroll
    for (int l = 1; l <= 3; ++l)
#pragma unroll
        for (int m = -3; m <= 3; ++m) {
            const int am = m < 0 ? -m : m;
            const float w = LAPLACIAN ? (float)whole(2160.0 * glap_c(am, l)) : (float)whole(5040.0 * l * grad_w(l, am));
            if (w != 0.0f) {
                const ff v = d(l, m);
                const float z = w * v.h;
                s.l += fmaf(w, v.l, fmaf(w, v.h, -z));
                ff_acc(s, z);
            }
        }
    return s;
}

// ---------------------------------------------------------------- momentum derivative
// (d_p f)_k of one axis (Eq. derf) from the five populations f of a row or
// column: the matrix is odd under p -> -p, so with a_m = f_{2+m} - f_{2-m} and
// s_m = f_{2+m} + f_{2-m}
//   (d_p f)_{2 +- m} = (E_m2 a_2 + E_m1 a_1) +- (O_m2 s_2 + O_m1 s_1 + O_m0 f_2).
__device__ __forceinline__ void dp_line(const FfTab &t, const ff f[NQ], ff out[NQ])
{
    auto add = [](ff a, ff b) {
        ff s = {a.h, a.l + b.l};
        ff_acc(s, b.h);
        return s;
    };
    auto neg = [](ff a) { return ff{-a.h, -a.l}; };
    auto mul = [](ff c, ff a) {
        const float p = c.h * a.h;
        return ff{p, fmaf(c.l, a.h, fmaf(c.h, a.l, fmaf(c.h, a.h, -p)))};
    };
    const ff a2 = ff_norm(add(f[4], neg(f[0]))), s2 = add(f[4], f[0]);
    const ff a1 = ff_norm(add(f[3], neg(f[1]))), s1 = add(f[3], f[1]);
    out[2] = add(mul(t.E[0][1], a2), mul(t.E[0][0], a1));
#pragma unroll
    for (int m = 1; m <= 2; ++m) {
        const ff e = add(mul(t.E[m][1], a2), mul(t.E[m][0], a1));
        const ff o = add(add(mul(t.O[m - 1][2], s2), mul(t.O[m - 1][1], s1)), mul(t.O[m - 1][0], f[2]));
        out[2 + m] = add(o, e);
        out[2 - m] = add(neg(o), e);
    }
}

// ---------------------------------------------------------------- equilibrium
// g_q(u, T) (eq_factors) by the parity of the Hermite orders: 26 instead of 34
// FP64 operations.
__device__ __forceinline__ void eq_factors64(const Tab<double> &t, double u, double T, double g[NQ])
{
    const double th = T - 1.0, u2 = u * u;
    const double c2 = 0.5 * (u2 + th);
    const double c3 = u * fma(u2, 1.0 / 6.0, 0.5 * th);
    const double c4 = fma(u2, fma(u2, 1.0 / 24.0, 0.25 * th), 0.125 * th * th);
#pragma unroll
    for (int m = 0; m <= 2; ++m) {
        const int k = 2 + m;
        const double even = fma(t.wHe[k][4], c4, fma(t.wHe[k][2], c2, t.wHe[k][0]));
        if (m == 0) {
            g[2] = even;
        } else {
            const double odd = fma(t.wHe[k][3], c3, t.wHe[k][1] * u);
            g[2 + m] = even + odd;
            g[2 - m] = even - odd;
        }
    }
}

// ---------------------------------------------------------------- the stage of one tile
// tid: the thread's index in the CTA; all threads call it.  sm holds the
// fields of phases 1 to 3, and the populations too, unless wait() still has to
// be called for them (it returns false when the copy timed out).
template <int TX, int TY, int KP, bool LEARNED, typename Wait>
__device__ __forceinline__ bool advance64(Smem64<TX, TY, KP, LEARNED> &sm, const double *fn, double *out, const Geo &g,
                                          const Tab<double> &t, const FfTab &ft, const StageK &c, int x0, int y0,
                                          const float *mlp, Wait wait)
{
    using S = Smem64<TX, TY, KP, LEARNED>;
    constexpr int NT = S::NT, NN = S::NN, HY = S::HY, HP = S::HP;
    const int tid = threadIdx.x;
    const FfScale sc = ff_scale(sm.top);

    // ---- 4a. differences of the fields
    constexpr int NX = 3 * HY * TX, NY = 3 * TY * (TX + 6);
    for (int e = tid; e < 2 * (NX + NY); e += NT) {
        const int field = e >= NX + NY;
        const double(*v)[S::HX] = field ? sm.n : sm.dp;
        int q = field ? e - (NX + NY) : e;
        if (q < NX) {
            const int l = q / (HY * TX) + 1, r = q % (HY * TX) / TX, x = q % TX;
            (&sm.dx[field][0][0][0])[q] = ff_split(v[r][x + 4 + l] - v[r][x + 4 - l], sc);
        } else {
            q -= NX;
            const int l = q / (TY * (TX + 6)) + 1, y = q % (TY * (TX + 6)) / (TX + 6), x = q % (TX + 6);
            (&sm.dy[field][0][0][0])[q] = ff_split(v[y + 3 + l][x + 1] - v[y + 3 - l][x + 1], sc);
        }
    }
    __syncthreads();

    // ---- 4b. on the first 128 threads G = c F = (c/ds) sum_dp / n + (c sigma/ds^3)
    // sum_n from the stencil sums of grad(Delta p) and grad(Laplacian n), a node
    // and axis a thread (the scale that the differences carry is taken out of
    // 1/n and sum_n); on the next 128, meanwhile, the equilibrium factors (FP64)
    static_assert(NT >= 256, "phase 4b takes 256 threads");
    if (tid < 2 * NN) {
        const int a = tid / NN, node = tid - a * NN, x = node % TX, y = node / TX;
        ff sp, sn;
        if (a == 0) {
            sp = stencil_sum<false>([&](int l, int m) { return sm.dx[0][l - 1][y + 3 + m][x]; });
            sn = stencil_sum<true>([&](int l, int m) { return sm.dx[1][l - 1][y + 3 + m][x]; });
        } else {
            sp = stencil_sum<false>([&](int l, int m) { return sm.dy[0][l - 1][y][x + 3 + m]; });
            sn = stencil_sum<true>([&](int l, int m) { return sm.dy[1][l - 1][y][x + 3 + m]; });
        }
        const ff n = ff_split(sm.n[y + 3][x + 4], sc);
        const float r = rcp_seed(n.h);
        const ff inv = {r, r * fmaf(-r, n.l, fmaf(-r, n.h, 1.0f))};
        ff v = ff_mul(ff_mul(sp, inv), c.kp);
        const ff w = ff_mul(sn, c.kn);
        // sum_n in the populations' units is 2^k of the scaled one
        const int k = 127 - 1023 - (sc.off >> 20);
        const int k1 = max(-126, min(127, k)), k2 = max(-126, min(127, k - k1));
        const float u1 = f32_make((unsigned)(k1 + 127) << 23), u2 = f32_make((unsigned)(k2 + 127) << 23);
        v.l += w.l * u1 * u2;
        ff_acc(v, w.h * u1 * u2);
        sm.G[a][node] = ff_norm(v);
    } else if (tid >= 128 && tid < 128 + 2 * NN) {
        const int a = (tid - 128) / NN, node = tid - 128 - a * NN, x = node % TX, y = node / TX;
        double w[NQ];
        eq_factors64(t, a == 0 ? sm.ux[y][x] : sm.uy[y][x], sm.T[y][x], w);
        const double n = sm.n[y + 3][x + 4];
#pragma unroll
        for (int q = 0; q < NQ; ++q) (a == 0 ? sm.ex : sm.ey)[q][node] = a == 0 ? n * w[q] : w[q];
    }
    if (!wait()) return false;
    __syncthreads();

    // ---- 5a. flux differences, a tile row or column a thread
    if constexpr (LEARNED) {
        // the faces of the 20 velocities with xi_x != 0, then of the 20 with xi_y != 0
        constexpr int nfx = (TX + 1) * TY, nfy = TX * (TY + 1);
        for (int e = tid; e < 20 * (nfx + nfy); e += NT) {
            const bool along_x = e < 20 * nfx;
            const int e2 = along_x ? e : e - 20 * nfx, nf = along_x ? nfx : nfy, q = e2 / nf, f = e2 - q * nf;
            const int k = along_x ? (q < 2 * NQ ? q : q + NQ) : (q >> 2) * NQ + ((q & 3) < 2 ? (q & 3) : (q & 3) + 1);
            const int r = along_x ? f / (TX + 1) : f / TX, cc = along_x ? f - r * (TX + 1) : f - r * TX;
            if (along_x ? (y0 + r >= g.ny || x0 + cc > g.nx) : (x0 + cc >= g.nx || y0 + r > g.ny)) continue;
            const bool up = along_x ? k / NQ > 2 : k % NQ > 2;
            double v[5];
#pragma unroll
            for (int m = 0; m < 5; ++m)
                v[m] = along_x ? sm.mid[k][r][up ? cc + 1 + m : cc + 6 - m] : *sm.at(k, up ? r + m : r + 5 - m, 4 + cc);
            const double d1 = v[2] - v[1], d2 = v[3] - v[2];
            const ff corr = ff_split(weno5_learned_corr64(mlp, v[1] - v[0], d1, d2, v[4] - v[3]), sc);
            // z = d1 + 2 d2 - 6 (F - v2)
            const ff f1 = ff_split(d1, sc), f2 = ff_split(d2, sc);
            const float c6 = 6.0f * corr.h;
            ff z = {2.0f * f2.h, fmaf(2.0f, f2.l, f1.l) - fmaf(6.0f, corr.l, fmaf(6.0f, corr.h, -c6))};
            ff_acc(z, f1.h);
            ff_acc(z, -c6);
            if (along_x) sm.ax[q][r][cc] = z;
            else sm.ay[q][cc][r] = z;
        }
        __syncthreads();
    }
    // (one call for rows and columns of one length: a second copy of the code
    // would not fit the instruction cache beside the first)
    auto line = [&](auto n, bool along_x, int q, int i) {
        const int k = along_x ? (q < 2 * NQ ? q : q + NQ) : (q >> 2) * NQ + ((q & 3) < 2 ? (q & 3) : (q & 3) + 1);
        const bool up = along_x ? k / NQ > 2 : k % NQ > 2;
        constexpr int N = decltype(n)::value;
        // the three nodes behind the line, its nodes, and the two ahead
        const double *p0, *p1, *p2;
        int step = up ? 1 : -1, halo = step;
        if (along_x) {
            const double *row = &sm.mid[k][i][0];
            p0 = row + (up ? 1 : TX + 6);
            p1 = row + (up ? 4 : TX + 3);
            p2 = row + (up ? TX + 4 : 3);
        } else {
            halo = step * TX;
            step *= HP;
            p0 = up ? &sm.below[k][0][i] : &sm.above[k][2][i];
            p1 = &sm.mid[k][up ? 0 : TY - 1][4 + i];
            p2 = up ? &sm.above[k][0][i] : &sm.below[k][2][i];
        }
        ff *o = along_x ? &sm.ax[q][i][0] : &sm.ay[q][i][0];
        // (the flux difference across a node takes the place of a face that it has used)
        if constexpr (LEARNED)
            weno5_row<N>(p0, p1, p2, halo, step, o + (up ? 0 : N - 1), up ? 1 : -1, sc,
                         [&](int j) { return o[up ? j : N - j]; });
        else
            weno5_row<N>(p0, p1, p2, halo, step, o + (up ? 0 : N - 1), up ? 1 : -1, sc);
    };
    for (int e = tid; e < 20 * (TY + TX); e += NT) {
        const bool along_x = e < 20 * TY;
        const int e2 = along_x ? e : e - 20 * TY, w = along_x ? TY : TX, q = e2 / w, i = e2 - q * w;
        if constexpr (TX == TY) {
            line(std::integral_constant<int, TX>(), along_x, q, i);
        } else {
            if (along_x) line(std::integral_constant<int, TX>(), true, q, i);
            else line(std::integral_constant<int, TY>(), false, q, i);
        }
    }
    __syncthreads();

    // f^n of the velocities that this thread advances in 5c, fetched now (with
    // five lanes it advances one column)
    constexpr int LINES = (NQ * NN + NT - 1) / NT;
    double f0[LINES][NQ];
    if (c.ca.h != 0.0f)
#pragma unroll
        for (int w = 0; w < LINES; ++w) {
            const int e = tid + w * NT, k2 = e / NN, node = e - k2 * NN, x = node % TX, y = node / TX;
            if (e >= NQ * NN || x0 + x >= g.nx || y0 + y >= g.ny) continue;
#pragma unroll
            for (int k1 = 0; k1 < NQ; ++k1)
                f0[w][k1] = fn[(NQ * k1 + k2) * g.plane + (long long)(y0 + y) * g.pitch + (x0 + x)];
        }

    // ---- 5b. a row of velocities (k1; k2 = 0..4) of a node a thread: the y force
    // term and both advection terms of its velocities
    for (int e = tid; e < NQ * NN; e += NT) {
        const int k1 = e / NN, node = e - k1 * NN, x = node % TX, y = node / TX;
        ff f[NQ], d[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) f[q] = ff_split(sm.mid[NQ * k1 + q][y][x + 4], sc);
        dp_line(ft, f, d);
        const ff Gy = sm.G[1][node];
        const ff K1 = c.adv[k1 < 2 ? 2 - k1 : k1 - 2];
#pragma unroll
        for (int k2 = 0; k2 < NQ; ++k2) {
            ff s = ff_mul(Gy, d[k2]);
            if (k2 != 2) {
                const ff v = ff_mul(sm.ay[slot_y(k1, k2)][x][y], c.adv[k2 < 2 ? 2 - k2 : k2 - 2]);
                s.l += v.l;
                ff_acc(s, v.h);
            }
            if (k1 != 2) {
                const ff v = ff_mul(sm.ax[slot_x(k1, k2)][y][x], K1);
                s.l += v.l;
                ff_acc(s, v.h);
            }
            sm.inc(k1, k2, x, y) = s;
        }
    }
    __syncthreads();

    // ---- 5c. a column of velocities (k2; k1 = 0..4) of a node a thread: the x
    // force term, collision and RK-3 combination
#pragma unroll
    for (int w = 0; w < LINES; ++w) {
        const int e = tid + w * NT, k2 = e / NN, node = e - k2 * NN, x = node % TX, y = node / TX;
        if (e >= NQ * NN || x0 + x >= g.nx || y0 + y >= g.ny) continue;
        double fv[NQ];
        ff f[NQ], d[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            fv[q] = sm.mid[NQ * q + k2][y][x + 4];
            f[q] = ff_split(fv[q], sc);
        }
        dp_line(ft, f, d);
        const ff Gx = sm.G[0][node];
        const double gy = sm.ey[k2][node];
        const long long o = (long long)(y0 + y) * g.pitch + (x0 + x);
#pragma unroll
        for (int k1 = 0; k1 < NQ; ++k1) {
            const int k = NQ * k1 + k2;
            const long long at = k * g.plane + o;
            // (c/tau) (f^eq - f)
            ff s = ff_mul(ff_split(fma(sm.ex[k1][node], gy, -fv[k1]), sc), c.cit);
            if (c.ca.h != 0.0f) {
                const ff v = ff_mul(ff_split(f0[w][k1] - fv[k1], sc), c.ca);
                s.l += v.l;
                ff_acc(s, v.h);
            }
            const ff a = sm.inc(k1, k2, x, y), b = ff_mul(Gx, d[k1]);
            s.l -= a.l + b.l;
            ff_acc(s, -a.h);
            ff_acc(s, -b.h);
            out[at] = fv[k1] + ff_widen(ff_norm(s), sc);
        }
    }
    return true;
}

}  // namespace olb
