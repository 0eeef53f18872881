// olb_stage32.cuh -- one RK-3 stage of an FP32 tile: fluxes, collision and RK-3
// combination.
//
// FP32 keeps every population as a pair hi + lo of floats (compensated storage,
// olb_kernels.cuh): the staged region holds both parts, moments are summed in
// double-float arithmetic, a face is its WENO correction (the face value minus its
// upwind node, a function of first differences of pairs) and the flux difference
// across a node a first difference plus a difference of corrections, the collision
// uses the equilibrium split into its exactly symmetric and antisymmetric parts in
// p (no FP32 rounding of f^eq or of f/tau changes the momentum), and the RK-3
// combination is done in double-float arithmetic.
//
// Bound by its instructions (ncu, 1024^2: issue slots 78 % busy, 7.6 k instructions a
// node, 650 MB of DRAM traffic in 0.26 ms).  Stage kernel on 2048^2: 1.75 -> 1.00 ms
// when a whole line of the tile became one thread's work (flux differences leave it
// instead of faces: 17 shared-memory loads a node and velocity less), the force
// moved to its own kernel (with its 14 x 14 fields a tile), and rows of the staged
// tile got a pitch of 20 floats (57 % of the shared-memory wavefronts were bank
// conflicts); moments and force take 0.22 and 0.13 ms beside it.
#pragma once

#include "olb_tile.cuh"

namespace olb {

// KP (stage_kind) 5: 320 threads, a line of the tile (Line), then a node and velocity
// column, each; 8: 512, which take the tile's moments and force too (OWN); 4: 256,
// with learned weights (whose network needs the registers), 6: 512 with them.
template <int KP, bool LEARNED>
struct Smem32 : Staged<float> {
    static constexpr bool OWN = KP == 8;
    static constexpr int NT = OWN || KP == 6 ? 512 : LEARNED ? 256 : 320;
    // per tile node: the even and odd equilibrium parts n ge_q(u_x, T), n go_q(u_x,
    // T), ge_q(u_y, T), go_q(u_y, T), the correction alpha, beta, gamma
    // (eq_correction), and c F
    float ex[NQ][NN], ox[NQ][NN], ey[NQ][NN], oy[NQ][NN], corr[3][NN], G[2][NN];
    // flux differences across the nodes of each row along x and column along y, of
    // the 20 velocities that move along the axis (line_velocity; learned weights:
    // first the corrections of the faces, one more than nodes, which the flux
    // differences then replace)
    float ax[20][TY][TX + 1];
    float ay[20][TX][TY + 1];
};

// A line of N nodes in the upwind direction (Line; the lo parts lo_p1 elements after
// the hi parts in the tile's rows, lo_halo in those around it): store(i, v) takes
// the flux difference across node i, a first difference of pairs plus the
// difference of the two faces' corrections.  Differences and squares are carried
// from face to face.  Z: gives the correction of face j instead of the Jiang-Shu
// weights.
struct NoCorrections {};
template <int N, typename Store, typename Z = NoCorrections>
__device__ __forceinline__ void weno5_line32(const Line<float> &ln, int lo_p1, int lo_halo, Store store, Z given = {})
{
    constexpr bool JS = std::is_same<Z, NoCorrections>::value;
    float vh = ln.p0[0], vl = ln.p0[lo_halo];
    auto next = [&](const float *p, int lo) {
        const float h = p[0], l = p[lo], d = pdiff(h, l, vh, vl);
        vh = h;
        vl = l;
        return d;
    };
    float d0 = next(ln.p0 + ln.halo, lo_halo), d1 = next(ln.p0 + 2 * ln.halo, lo_halo), d2 = next(ln.p1, lo_p1);
    float h1 = 2.5f * (d1 * d1), c0 = 0.0f;
    const float *p = ln.p1 + ln.step;
    int step = ln.step, lo = lo_p1;
#pragma unroll 3
    for (int j = 0; j <= N; ++j) {
        if (j == N - 1) {
            p = ln.p2;
            step = ln.halo;
            lo = lo_halo;
        }
        const float d3 = next(p, lo);
        p += step;
        float c1;
        if constexpr (JS) {
            const float q2 = d2 * d2, h2 = 2.5f * q2;
            c1 = weno5_core(d0, d1, d2, d3, q2, h1, h2);
            h1 = h2;
        } else {
            c1 = given(j);
        }
        if (j > 0) store(j - 1, d1 + (c1 - c0));
        c0 = c1;
        d0 = d1;
        d1 = d2;
        d2 = d3;
    }
}

// One stage for the tile whose lower-left node is (x0, y0); all threads of the CTA
// call it.  ca, cb, cc: the stage's coefficients of f^n, f_s and dt L (Eq. rk3);
// ca_lo, cb_lo: their remainders (1/3 and 2/3 as double-float constants); tw: the
// table of the wall entries; net: the learned network (LEARNED only); tmap: TMA maps of fs, or nullptr; fields: the moments
// and c F of fs (k_fields, k_force); own: KP 8's room for its own fields.  Returns false when the TMA copy timed out (the CTA must
// stop).
template <int KP, bool LEARNED>
__device__ __forceinline__ bool stage_tile32(Smem32<KP, LEARNED> &sm, const float *__restrict__ fs, const float *fn, float *out,
                                             int *__restrict__ status, const Geo &g, const Tab<float> &t,
                                             const Tab<float> &tw, int x0, int y0, float ca, float cb, float cc, float ca_lo,
                                             float cb_lo, const MlpArg &net, const TmaMap *tmap,
                                             const StageFields<float> &fields, TileFields<float> *own = nullptr)
{
    using S = Smem32<KP, LEARNED>;
    constexpr bool OWN = S::OWN;
    constexpr int NT = S::NT, TX = S::TX, TY = S::TY, NN = S::NN, HP = S::HP;
    const int tid = threadIdx.x;

    // ---- 1. the fields of a node (three threads a node: x factors, y factors,
    // correction), then the populations: copies in flight during phase 2 for a tile
    // inside the grid
    const int part = tid / NN, node = tid % NN, tx = node % TX, ty = node / TX;
    const bool has = part < 3 && x0 + tx < g.nx && y0 + ty < g.ny;
    float2 fN = {1.0f, 0.0f}, fT = {1.0f, 0.0f}, fE = {0.0f, 0.0f};
    float ux = 0.0f, uy = 0.0f, G = 0.0f;
    if (!OWN && has) {
        const long long o = (long long)(y0 + ty) * g.pitch + (x0 + tx);
        fN = fields.n[o];
        fT = fields.T[o];
        ux = fields.ux[o];
        uy = fields.uy[o];
        if (part == 2) fE = fields.E[o];
        else G = (part == 0 ? fields.G[0] : fields.G[1])[o];
    }
    const bool inside = tmap != nullptr && x0 >= 4 && x0 + TX + 4 <= g.nx && y0 >= 3 && y0 + TY + 3 <= g.ny;
    if (inside) tma_issue(sm, tmap, x0, y0);
    if constexpr (OWN) {
        if (tid < OWN_THREADS) tile_moments(*own, nullptr, fs, status, g, t, x0, y0);
        else if (!inside) load_region(sm, fs, g, x0, y0, OWN_THREADS);
        __syncthreads();
        if (has) {
            fN = own->force.n[ty + 3][tx + 3];
            fT = own->T[node];
            ux = own->ux[node];
            uy = own->uy[node];
            if (part == 2) fE = own->E[node];
        }
    } else {
        if (!inside) load_region(sm, fs, g, x0, y0);
        __syncthreads();
    }

    // ---- 2. equilibrium factors and the correction of their rounding
    if (part < 3) {
        float a[NQ], b[NQ];
        if (part != 1) {
            eq_factors_split(t, ux, fT, a, b);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                a[q] = fN.x * a[q];
                b[q] = fN.x * b[q];
            }
        }
        float c[NQ], d[NQ];
        if (part != 0) eq_factors_split(t, uy, fT, c, d);
        if (part == 0) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                sm.ex[q][node] = a[q];
                sm.ox[q][node] = b[q];
            }
        } else if (part == 1) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                sm.ey[q][node] = c[q];
                sm.oy[q][node] = d[q];
            }
        } else {
            eq_correction(t, a, c, fN, fE, ux, uy, sm.corr[0][node], sm.corr[1][node], sm.corr[2][node]);
        }
        if (!OWN && part < 2) sm.G[part][node] = G;
    } else if (OWN && part < 5) {
        sm.G[part - 3][node] = force_at32(own->force, g, cc, part - 3, tx, ty);
    }
    // ---- 3. diffuse walls: fluxes and ghosts of the tile rows
    const bool left = x0 == 0 && g.wall_lo, right = x0 + TX + 3 >= g.nx && g.wall_hi;
    if (left || right) {
        wall_flux<float, LEARNED>(sm, g, t, tw, net.theta, x0, OWN ? 5 * NN : 3 * NN, left, right);
        __syncthreads();
        wall_ghosts<float>(sm, g, tw, x0, 0, left, right);
    }
    if (inside && !tma_finish(sm, status)) return false;
    __syncthreads();

    // ---- 4. flux differences, a row or column a thread
    if constexpr (LEARNED) {
        // every face once, on whole warps: the network of a warp's 32 stencils runs on
        // the tensor pipe, from a single call site (mma.sync needs every lane at the
        // same instruction; items past the end take part in the network only): the
        // x faces of the 20 velocities with xi_x != 0, then the y faces of the 20
        // with xi_y != 0
        constexpr int nfx = (TX + 1) * TY, nfy = TX * (TY + 1), total = 20 * (nfx + nfy);
        for (int e = tid; e < (total + 31) / 32 * 32; e += NT) {
            const int ee = e < total ? e : 0;
            const bool along_x = ee < 20 * nfx;
            const int e2 = along_x ? ee : ee - 20 * nfx, nf = along_x ? nfx : nfy, q = e2 / nf, f = e2 - q * nf;
            const int k = line_velocity(along_x, q);
            const int r = along_x ? f / (TX + 1) : f / TX, c = along_x ? f - r * (TX + 1) : f - r * TX;
            const bool valid = e < total && (along_x ? (y0 + r < g.ny && x0 + c <= g.nx) : (x0 + c < g.nx && y0 + r <= g.ny));
            // first differences of the stencil in the upwind orientation
            const bool up = along_x ? k / NQ > 2 : k % NQ > 2;
            float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (valid) {
                float ph = 0.0f, pl = 0.0f;
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    const int row = along_x ? r + 3 : up ? r + m : r + 5 - m, col = along_x ? (up ? c + 1 + m : c + 6 - m) : 4 + c;
                    const float h = *sm.at(k, row, col), l = *sm.at(NK + k, row, col);
                    if (m > 0) d[m - 1] = pdiff(h, l, ph, pl);
                    ph = h;
                    pl = l;
                }
            }
            const bool acts = learned_guard(d[0], d[1], d[2], d[3]);
            float x[MLP_IN], w[MLP_OUT] = {0.0f, 0.0f, 0.0f};
            learned_input_x(d, acts, x);
            // the whole warp skips the network when none of its stencils needs it
            if (__any_sync(0xffffffffu, acts)) mlp_weights_warp32(net.tables, x, w);
            if (valid) {
                const float res = acts ? learned_corr_from(w, d) : weno5_corr(d[0], d[1], d[2], d[3]);
                if (along_x) sm.ax[q][r][c] = res;
                else sm.ay[q][c][r] = res;
            }
        }
        __syncthreads();
    }
    for (int e = tid; e < 40 * TX; e += NT) {
        const bool along_x = e < 20 * TY;
        const int e2 = along_x ? e : e - 20 * TY, q = e2 / TX, i = e2 % TX;
        const Line<float> ln = line_of<float>(sm, along_x, q, i);
        float *o = along_x ? &sm.ax[q][i][0] : &sm.ay[q][i][0];
        auto store = [&](int j, float v) { o[ln.up ? j : TX - 1 - j] = v; };
        const int lo_p1 = NK * TY * HP, lo_halo = along_x ? lo_p1 : NK * 3 * TX;
        // (learned: the flux difference across a node takes the place of a face that it has used)
        if constexpr (LEARNED)
            weno5_line32<TX>(ln, lo_p1, lo_halo, store, [&](int j) { return o[ln.up ? j : TX - j]; });
        else
            weno5_line32<TX>(ln, lo_p1, lo_halo, store);
    }

    // f^n of the column that this thread advances, fetched now
    constexpr int COLS = (NQ * NN + NT - 1) / NT;
    float fh[COLS][NQ], fl[COLS][NQ];
    if (ca != 0.0f)
#pragma unroll
        for (int w = 0; w < COLS; ++w) {
            const int e = tid + w * NT, k2 = e / NN, nd = e - k2 * NN, x = x0 + nd % TX, y = y0 + nd / TX;
            if (e >= NQ * NN || x >= g.nx || y >= g.ny) continue;
            const float *p = fn + k2 * g.plane + (long long)y * g.pitch + x;
#pragma unroll
            for (int k1 = 0; k1 < NQ; ++k1) {
                fh[w][k1] = p[NQ * k1 * g.plane];
                fl[w][k1] = p[(NK + NQ * k1) * g.plane];
            }
        }
    __syncthreads();

    // ---- 5. node updates: thread (node, k2) advances the five velocities 5 k1 + k2,
    // k1 unrolled, so that the k1 tables are immediate operands and the node's
    // factors are read once
    const float cit = cc * (float)g.inv_tau, cadv = cc * (float)g.inv_ds;
#pragma unroll
    for (int w = 0; w < COLS; ++w) {
        const int e = tid + w * NT, k2 = e / NN, nd = e - k2 * NN, x = nd % TX, y = nd / TX;
        if (e >= NQ * NN || x0 + x >= g.nx || y0 + y >= g.ny) continue;
        const float Gx = sm.G[0][nd], Gy = sm.G[1][nd];
        const float qa = sm.corr[0][nd], qb = sm.corr[1][nd], qc = sm.corr[2][nd];
        const float gyk = sm.ey[k2][nd], oyk = sm.oy[k2][nd];
        float col[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) col[q] = sm.mid[NQ * q + k2][y][x + 4];
        float *o = out + k2 * g.plane + (long long)(y0 + y) * g.pitch + (x0 + x);
#pragma unroll
        for (int k1 = 0; k1 < NQ; ++k1) {
            const int k = NQ * k1 + k2;
            float dx = 0.0f, dy = 0.0f;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                dx = fmaf(t.D[k1][q], col[q], dx);
                dy = fmaf(t.D[k2][q], sm.mid[NQ * k1 + q][y][x + 4], dy);
            }
            // (flux differences are in the upwind direction: times |xi|)
            float adv = 0.0f;
            if (k1 != 2) adv = t.R[k1 < 2 ? 4 - k1 : k1] * sm.ax[NQ * (k1 < 2 ? k1 : k1 - 1) + k2][y][x];
            if (k2 != 2) adv = fmaf(t.R[k2 < 2 ? 4 - k2 : k2], sm.ay[4 * k1 + (k2 < 2 ? k2 : k2 - 1)][x][y], adv);
            // f - f^eq with f^eq = n (ge ge + ge go + go (ge + go)) - c: the
            // exactly symmetric part first, then the parts odd in p_y and in
            // p_x (each exactly odd after rounding), so that FP32 rounding of
            // the equilibrium carries no momentum; c (eq_correction) restores
            // its mass and energy
            const float f = col[k1], fo = sm.mid[NK + k][y][x + 4];
            const float corr =
                (t.wHe[k1][0] * t.wHe[k2][0]) * fmaf(qc, t.R2[k1] - t.R2[k2], fmaf(qb, t.R2[k1] + t.R2[k2], qa));
            const float Ek = sm.ex[k1][nd], oxk = sm.ox[k1][nd];
            const float neq = ((((f - Ek * gyk) + fo) - Ek * oyk) - oxk * (gyk + oyk)) + corr;
            // c L = -c xi.grad f - c F.grad_p f - (c/tau)(f - f^eq), then
            // out = ca f_n + cb f_s + c L (Eq. rk3) in double-float arithmetic
            const float inc = -fmaf(cit, neq, fmaf(Gx, dx, fmaf(Gy, dy, cadv * adv)));
            f2 acc = f2_cmul(f2{cb, cb_lo}, f, fo);
            if (ca != 0.0f) {
                const f2 an = f2_cmul(f2{ca, ca_lo}, fh[w][k1], fl[w][k1]);
                const f2 sh = two_sum(acc.hi, an.hi);
                acc = f2{sh.hi, sh.lo + (acc.lo + an.lo)};
            }
            const f2 si = two_sum(acc.hi, inc);
            const f2 v = fast_two_sum(si.hi, si.lo + acc.lo);
            o[NQ * k1 * g.plane] = v.hi;
            o[(NK + NQ * k1) * g.plane] = v.lo;
        }
    }
    return true;
}

}  // namespace olb
