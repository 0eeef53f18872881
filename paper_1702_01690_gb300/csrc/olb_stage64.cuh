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
// FP64's rounding of f wherever Delta < f / 128.  Where Delta is larger its errors show;
// against 80-bit arithmetic, in units of 2.2e-16 of the largest population (FP64 form ->
// this one): one step of 30 % noise on 32^2 nodes 6.8 -> 2.3, of jumps 0.05 | 1.6 between
// nodes on 32^2 2.9 -> 3.3 (4 steps 16 -> 5), of a drop's interface of three nodes 7.7
// -> 16 (8 steps 91 -> 41).  Only where a step's capillary increment is of the size of f,
// jumps between the nodes of a fine grid (512 x 24), is it the less accurate: 6 -> 105.
//
// Measured, one step (three stages) of a 4096^2 grid: 106.6 ms with the force and
// the node updates in FP64 (1070 FP64 instructions a node and stage beside 60
// differences), 56.8 ms like this (228), 51.8 ms with three CTAs an SM, 46.5 ms
// with the force in a kernel of its own (k_force) and two nodes a thread, 38.7 ms
// with the moments' sums in fixed point (olb_kernels.cuh), 39.1 ms with initial fields
// and moments output as they are now and tiles checked for values beyond their scale.
// Against 80-bit arithmetic the populations are closer than the FP64 form's
// (12 steps of a 167 x 109 drop: 5.7e-16 instead of 1.2e-15 of their norm, and
// its loss of 1e-15 of the mass is gone): Delta is summed before the one
// rounding at the size of f.
//
// What bounds it now (ncu, 2048^2): no pipe; FP64 57-59 %, issue slots 55 %, and
// what three CTAs of five warps leave of latency (three tiles hold 210 of the 228 KB of
// shared memory, and two nodes a thread take 126 registers: 60 of 64 K).
#pragma once

#include "olb_tile.cuh"

namespace olb {

// ---------------------------------------------------------------- shared memory
// A float-float of the nodes (x, y) and (x, y + 4) of the tile: threads that take
// two nodes (vf2) read and write it whole, threads that take one a half of it.
struct __align__(16) ffp {
    float h[2], l[2];
    template <typename V>
    __device__ __forceinline__ ffv<V> get(int half) const
    {
        if constexpr (V::W == 1) return {{h[half]}, {l[half]}};
        else {
            const float4 a = *reinterpret_cast<const float4 *>(this);
            return {vf2::pair(a.x, a.y), vf2::pair(a.z, a.w)};
        }
    }
    template <typename V>
    __device__ __forceinline__ void put(int half, ffv<V> v)
    {
        if constexpr (V::W == 1) {
            h[half] = v.h[0];
            l[half] = v.l[0];
        } else {
            *reinterpret_cast<float4 *>(this) = make_float4(v.h[0], v.h[1], v.l[0], v.l[1]);
        }
    }
};

// Tile of 8 x 8 nodes.  KP selects the threads (stage_kind): 5: 160, two nodes or
// lines a thread; 8: 512, one, which take the tile's moments and force too (OWN).
template <int KP>
struct Plan64 {
    using V = typename std::conditional<KP == 8, vf1, vf2>::type;
    static constexpr int NT = KP == 5 ? 160 : 512;
    static constexpr bool OWN = KP == 8;
};

template <int KP>
struct Smem64 : Staged<double> {
    static constexpr int NT = Plan64<KP>::NT;
    double ex[NQ][NN];  // n g_q(u_x, T) and g_q(u_y, T) of the tile nodes
    double ey[NQ][NN];
    ffp G[2][NN / 2];   // c F
    // flux differences times 6 (weno5_flux6) across the nodes of each row along x
    // and column along y, of the 20 velocities that move along the axis (slot_x,
    // slot_y); then, in place of one of a velocity's flux differences (inc), the sum of
    // its advection and force terms.  Entry i of a column sits in half i / 4 of element i
    // mod 4; the ninth element of a row, the fifth of a column and the one at the end
    // keep the banks of rows and columns apart.
    ffp ax[20][TY / 2][TX + 1];
    ffp ay[20][TX * (TY / 2 + 1) + 1];
    ffp rest[NN / 2];
    int top;            // high word of the largest n of the tile (its scale) or of the largest population

    __device__ __forceinline__ ffp &col(int q, int x, int i) { return ay[q][5 * x + (i & 3)]; }
    // top is at least the largest finite staged population, wall ghosts included (all threads)
    __device__ __noinline__ void raise_top(int tid)
    {
        int a = 0;
        for (int e = tid; e < P * HY * (TX + 6); e += NT) {
            const int k = e / (HY * (TX + 6)), r = e / (TX + 6) % HY, c = 1 + e % (TX + 6);
            const int v = staged(r, c) ? __double2hiint(*at(k, r, c)) & 0x7fffffff : 0;
            a = max(a, v < 0x7ff00000 ? v : 0);
        }
        atomicMax(&top, a);
    }
    __device__ __forceinline__ ffp &inc(int k1, int k2, int x, int y4)
    {
        return k1 != 2   ? ax[NQ * (k1 < 2 ? k1 : k1 - 1) + k2][y4][x]
               : k2 != 2 ? ay[8 + (k2 < 2 ? k2 : k2 - 1)][5 * x + y4]
                         : rest[8 * y4 + x];
    }
};

// Slots of ax for the velocities with xi_x != 0 and of ay for those with xi_y != 0.
__device__ __forceinline__ int slot_x(int k1, int k2) { return NQ * (k1 < 2 ? k1 : k1 - 1) + k2; }
__device__ __forceinline__ int slot_y(int k1, int k2) { return 4 * k1 + (k2 < 2 ? k2 : k2 - 1); }

// ---------------------------------------------------------------- momentum derivative
// (d_p f)_k of one axis (Eq. derf) from the five populations f of a row or
// column: the matrix is odd under p -> -p, so with a_m = f_{2+m} - f_{2-m} and
// s_m = f_{2+m} + f_{2-m}
//   (d_p f)_{2 +- m} = (E_m2 a_2 + E_m1 a_1) +- (O_m2 s_2 + O_m1 s_1 + O_m0 f_2).
template <typename V>
__device__ __forceinline__ void dp_line(const FfTab &t, const ffv<V> f[NQ], ffv<V> out[NQ])
{
    auto add = [](ffv<V> a, ffv<V> b) {
        ff_acc(a, b);
        return a;
    };
    auto neg = [](ffv<V> a) { return ffv<V>{-a.h, -a.l}; };
    const ffv<V> a2 = add(f[4], neg(f[0])), s2 = add(f[4], f[0]);
    const ffv<V> a1 = add(f[3], neg(f[1])), s1 = add(f[3], f[1]);
    out[2] = add(ff_mul(t.E[0][1], a2), ff_mul(t.E[0][0], a1));
#pragma unroll
    for (int m = 1; m <= 2; ++m) {
        const ffv<V> e = add(ff_mul(t.E[m][1], a2), ff_mul(t.E[m][0], a1));
        const ffv<V> o = add(add(ff_mul(t.O[m - 1][2], s2), ff_mul(t.O[m - 1][1], s1)), ff_mul(t.O[m - 1][0], f[2]));
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
// One stage for the tile whose lower-left node is (x0, y0); all threads of the CTA
// call it.  fields: the moments and c F of fs (k_fields, k_force); tw: the table
// of the wall entries; tmap: TMA maps of fs, or nullptr; own: KP 8's room for its own
// fields.  A thread takes V::W nodes
// (y and y + 4 of a column) or lines (rows or columns 4 apart) at a time.
// Returns false when the TMA copy timed out (the CTA must stop).
template <int KP>
__device__ __forceinline__ bool stage_tile64(Smem64<KP> &sm, const double *__restrict__ fs, const double *fn,
                                             double *out, int *__restrict__ status, const Geo &g, const Tab<double> &t,
                                             const Tab<double> &tw, int x0, int y0, const StageK &c, const TmaMap *tmap,
                                              const StageFields<double> &fields,
                                             TileFields<double> *own = nullptr)
{
    using S = Smem64<KP>;
    using V = typename Plan64<KP>::V;
    constexpr int W = V::W, NT = S::NT, TX = S::TX, TY = S::TY, NN = S::NN, NI = NN / W, HP = S::HP;
    const int tid = threadIdx.x;
    const FfTab &ft = t.ff;

    // ---- 1. the fields of a node and axis (threads 0 .. 2 NN - 1), then the
    // populations: copies in flight during phase 2 for a tile inside the grid
    constexpr bool OWN = Plan64<KP>::OWN;
    const int a = tid / NN, node = tid % NN, nx = node % TX, ny = node / TX;
    const bool has = tid < 2 * NN && x0 + nx < g.nx && y0 + ny < g.ny;
    double fn_ = 0.0, fu = 0.0, fT = 1.0;
    ff fG = {0.0f, 0.0f};
    if (!OWN && has) {
        const long long o = (long long)(y0 + ny) * g.pitch + (x0 + nx);
        fn_ = fields.n[o];
        fu = a == 0 ? fields.ux[o] : fields.uy[o];
        fT = fields.T[o];
        fG = (a == 0 ? fields.G[0] : fields.G[1])[o];
    }
    if (tid == 0) {
        sm.top = 0;
        if (OWN) own->force.top = 0;
    }
    const bool inside = tmap != nullptr && x0 >= 4 && x0 + TX + 4 <= g.nx && y0 >= 3 && y0 + TY + 3 <= g.ny;
    if (inside) tma_issue(sm, tmap, x0, y0);
    if constexpr (OWN) {
        __syncthreads();
        if (tid < OWN_THREADS) tile_moments(*own, &sm.top, fs, status, g, t, x0, y0);
        else if (!inside) load_region(sm, fs, g, x0, y0, OWN_THREADS);
        __syncthreads();
        force_differences<NT>(own->force, ff_scale(own->force.top));
        if (has) {
            fn_ = own->force.v[1][ny + 3][nx + 3];
            fu = a == 0 ? own->ux[node] : own->uy[node];
            fT = own->T[node];
        }
    } else if (!inside) {
        load_region(sm, fs, g, x0, y0);
    }
    __syncthreads();

    // ---- 2. equilibrium factors (FP64), the tile's scale (its largest density; OWN: the
    // largest population that the lines read, which costs nothing there)
    if (tid < 2 * NN) {
        double w[NQ];
        eq_factors64(t, fu, fT, w);
#pragma unroll
        for (int q = 0; q < NQ; ++q) (a == 0 ? sm.ex : sm.ey)[q][node] = a == 0 ? fn_ * w[q] : w[q];
        if constexpr (!OWN) {
            ffp &G = sm.G[a][8 * (ny & 3) + nx];
            G.h[ny >> 2] = fG.h;
            G.l[ny >> 2] = fG.l;
            const int hw = __double2hiint(fn_) & 0x7fffffff, top = __reduce_max_sync(0xffffffffu, hw < 0x7ff00000 ? hw : 0);
            if ((tid & 31) == 0) atomicMax(&sm.top, top);
        }
    } else if (OWN && tid < 4 * NN) {
        const ffv<vf1> v = force_at<vf1>(own->force, ff_scale(own->force.top), c, a - 2, nx, ny);
        sm.G[a - 2][8 * (ny & 3) + nx].put(ny >> 2, v);
    }
    // ---- 3. diffuse walls: fluxes and ghosts of the tile rows
    const bool left = x0 == 0 && g.wall_lo, right = x0 + TX + 3 >= g.nx && g.wall_hi;
    if (left || right) {
        wall_flux<double, false>(sm, g, t, tw, nullptr, x0, OWN ? 4 * NN : 2 * NN, left, right);
        __syncthreads();
        wall_ghosts<double>(sm, g, tw, x0, 0, left, right, OWN ? &sm.top : nullptr);
    }
    if (inside && !tma_finish(sm, status)) return false;
    __syncthreads();
    FfScale sc = ff_scale(sm.top);

    // ---- 5a. flux differences, W rows or columns a thread; unless OWN, once more with the
    // scale of the largest population if some were beyond FP32's range (other tiles pay
    // one packed FMA a flux difference for it)
    for (bool again = false;; again = true) {
        V sum = V::all(0.0f);  // of 0 times the low parts: not 0 if one is not finite
        for (int e = tid; e < 40 * (TX / W); e += NT) {
            const bool along_x = e < 20 * (TX / W);
            const int e2 = along_x ? e : e - 20 * (TX / W), q = e2 / (TX / W), i = e2 - q * (TX / W);
            const Line<double> ln = line_of<double>(sm, along_x, q, i);
            const bool up = ln.up;
            auto store = [&](int j, ffv<V> v) {
                const int at = up ? j : TX - 1 - j;
                if constexpr (!OWN) sum = vfma(0.0f, v.l, sum);
                if (along_x) {
                    sm.ax[q][i & 3][at].put(i >> 2, v);
                } else {
#pragma unroll
                    for (int w = 0; w < W; ++w) {
                        ffp &o = sm.col(q, i + 4 * w, at);
                        o.h[at >> 2] = v.h[w];
                        o.l[at >> 2] = v.l[w];
                    }
                }
            };
            weno5_line<TX, V>(ln.p0, ln.p1, ln.p2, along_x ? 4 * HP : 4, ln.halo, ln.step, sc, store);
        }
        if constexpr (OWN) {
            __syncthreads();
            break;
        }
        if (!__syncthreads_or(!(sum[0] == 0.0f && sum[W - 1] == 0.0f)) || again) break;
        const int top = sm.top;
        __syncthreads();
        sm.raise_top(tid);
        __syncthreads();
        if (sm.top == top) break;  // (infinities or NaN among the populations)
        sc = ff_scale(sm.top);
    }

    // (once more, not kept: 5a's registers)
    if (!OWN) sc = ff_scale(*(volatile int *)&sm.top);

    // f^n of the velocities that this thread advances in 5c, fetched now
    constexpr int LINES = (NQ * NI + NT - 1) / NT;
    double f0[LINES][NQ][W];
    if (c.ca.h != 0.0f)
#pragma unroll
        for (int w = 0; w < LINES; ++w) {
            const int e = tid + w * NT, k2 = e / NI, it = e - k2 * NI, x = it % TX, y = it / TX;
#pragma unroll
            for (int i = 0; i < W; ++i) {
                if (e >= NQ * NI || x0 + x >= g.nx || y0 + y + 4 * i >= g.ny) continue;
#pragma unroll
                for (int k1 = 0; k1 < NQ; ++k1)
                    f0[w][k1][i] = fn[(NQ * k1 + k2) * g.plane + (long long)(y0 + y + 4 * i) * g.pitch + (x0 + x)];
            }
        }

    // ---- 5b. a row of velocities (k1; k2 = 0..4) of W nodes a thread: both
    // advection terms, and the y force term; then a column (k2; k1 = 0..4): the x
    // force term, collision and RK-3 combination.  (One loop for both axes: the
    // instructions of a stage have to stay in the cache, see weno5_line.)
#pragma unroll 1
    for (int axis = 1; axis >= 0; --axis) {
#pragma unroll
        for (int w = 0; w < LINES; ++w) {
            const int e = tid + w * NT, line = e / NI, it = e - line * NI, x = it % TX, y = it / TX;
            if (e >= NQ * NI || x0 + x >= g.nx || y0 + y >= g.ny) continue;
            // velocity k0 + q dk is (line, q) in a row, (q, line) in a column
            const int k0 = axis ? NQ * line : line, dk = axis ? 1 : NQ;
            if (axis) {
                const ff K1 = c.adv[line < 2 ? 2 - line : line - 2];
#pragma unroll 1
                for (int k2 = 0; k2 < NQ; ++k2) {
                    ffv<V> s = {V::all(0.0f), V::all(0.0f)};
                    if (line != 2) s = ff_mul(K1, sm.ax[slot_x(line, k2)][y & 3][x].template get<V>(y >> 2));
                    if (k2 != 2)
                        ff_acc(s, ff_mul(c.adv[k2 < 2 ? 2 - k2 : k2 - 2],
                                         sm.ay[slot_y(line, k2)][5 * x + (y & 3)].template get<V>(y >> 2)));
                    sm.inc(line, k2, x, y & 3).put(y >> 2, s);
                }
            }
            double fv[NQ][W];
            ffv<V> f[NQ], d[NQ];
            const double *p = &sm.mid[k0][y][x + 4];
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
#pragma unroll
                for (int i = 0; i < W; ++i) fv[q][i] = p[q * dk * (TY * HP) + 4 * i * HP];
                f[q] = ff_split<V>(fv[q], sc);
            }
            dp_line(ft, f, d);
            const ffv<V> G = sm.G[axis][8 * (y & 3) + x].template get<V>(y >> 2);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                ffp &o = sm.inc(axis ? line : q, axis ? q : line, x, y & 3);
                ffv<V> s = ff_mul(G, d[q]);
                ff_acc(s, o.template get<V>(y >> 2));
                o.put(y >> 2, s);
            }
            if (axis) continue;
            double gy[W];
#pragma unroll
            for (int i = 0; i < W; ++i) gy[i] = sm.ey[line][it + 32 * i];
            double *o = out + line * g.plane + (long long)(y0 + y) * g.pitch + (x0 + x);
#pragma unroll
            for (int k1 = 0; k1 < NQ; ++k1) {
                double q[W];
                // (c/tau) (f^eq - f)
#pragma unroll
                for (int i = 0; i < W; ++i) q[i] = fma(sm.ex[k1][it + 32 * i], gy[i], -fv[k1][i]);
                ffv<V> s = ff_mul(c.cit, ff_split<V>(q, sc));
                if (c.ca.h != 0.0f) {
#pragma unroll
                    for (int i = 0; i < W; ++i) q[i] = f0[w][k1][i] - fv[k1][i];
                    ff_acc(s, ff_mul(c.ca, ff_split<V>(q, sc)));
                }
                const ffv<V> a = sm.inc(k1, line, x, y & 3).template get<V>(y >> 2);
                s.l = s.l - a.l;
                ff_acc(s, -a.h);
#pragma unroll
                for (int i = 0; i < W; ++i)
                    if (i == 0 || y0 + y + 4 * i < g.ny)
                        o[k1 * NQ * g.plane + 4 * i * g.pitch] = fv[k1][i] + ff_widen(ff_lane(s, i), sc);
            }
        }
        if (axis) __syncthreads();
    }
    return true;
}

}  // namespace olb
