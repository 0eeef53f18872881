// olb_fused.cuh -- one RK-3 stage of the off-lattice Boltzmann model in a
// single kernel per stage (templated on precision and tile shape).
//
// One CTA owns a TX x TY tile of nodes and stages the populations of the
// tile plus a 3-node halo on every side in shared memory:
//   1. load f_s for the (TX+8) x (TY+6) region (x offset -4 keeps the rows
//      of the region 16-byte aligned; y and periodic x wrap);
//   2. moments n, u, T, Delta p at every fluid node of the region (Sec. 2.2,
//      Eq. vdw), with the even reflection of Delta p and n at walls
//      (Sec. 3.4.3);
//   3. walls (Sec. 3.4.2): extrapolated ghosts for the outgoing velocities,
//      the WENO flux of those velocities at the wall face, summed per tile
//      row into n_w (Eq. nw) by a warp-shuffle reduction over the half-warp
//      that computes the row's ten fluxes, and f^eq_w ghosts for the
//      incoming velocities;
//   4. force F = grad(Delta p)/n + sigma grad(Laplacian n) at the tile nodes
//      from the 49-point stencils (Eqs. F_def, stencil_grad, stencil_glap);
//   5. for KP velocities at a time (one lane of TX*TY threads, rounded up to
//      whole warps, each): every x
//      and y face of the tile once (WENO-5, Eqs. weno5_*), then per node the
//      flux differences, the momentum derivative (Eq. derf), BGK with f^eq
//      (Eqs. feq, g_alpha) and the RK-3 combination of Eq. rk3, written to
//      the output buffer.  KP > 1 gives small tiles enough warps.
//
// FP32 (real = float) keeps every population as a pair hi + lo of floats
// (compensated storage, olb_kernels.cuh): the staged region holds both parts,
// moments are summed in double-float arithmetic, a face stores only its WENO
// correction (the face value minus its upwind node, a function of first
// differences of pairs) so that flux differences are first differences too,
// the collision uses the equilibrium split into its exactly symmetric and
// antisymmetric parts in p (no FP32 rounding of f^eq or of f/tau changes the
// momentum), and the RK-3 combination is done in double-float arithmetic.
#pragma once

#include "olb_fields.cuh"
#include "olb_stage64.cuh"
#include "olb_tile.cuh"

namespace olb {

// Shared memory of an FP32 tile (FP64: Smem64 in olb_stage64.cuh).
template <int TX_, int TY_, int KP>
struct Smem32 {
    // LS: threads per velocity lane, the tile's nodes rounded up to whole
    // warps (so that every lane starts on a warp); NT threads in all;
    // HP: pitch of a staged row of populations (region_pitch)
    static constexpr int TX = TX_, TY = TY_;
    static constexpr int HX = TX + 8, HY = TY + 6, NN = TX * TY, LS = (NN + 31) / 32 * 32, NT = LS * KP;
    static constexpr int HP = region_pitch(TX, false);
    using fld = FieldT<float>::type;
    float pop[NK][HY][HP];
    struct {
        float lo[NK][HY][HP];  // lo parts of the staged populations
    } pl;
    fld n[HY][HX];
    fld dp[HY][HX];
    float ux[TY][TX];
    float uy[TY][TX];
    fld T[TY][TX];    // hi + lo pair
    // e = sum |p|^2 f at the tile nodes as a double-float pair (the target
    // energy of the equilibrium's correction)
    fld eng[TY][TX];
    // per tile node, shared by the KP velocity lanes (with one lane they stay
    // in registers): the stencil sums of grad(Delta p) and grad(Laplacian n),
    // inv_ds / n, the even and odd equilibrium parts n ge_q(u_x, T),
    // n go_q(u_x, T), ge_q(u_y, T), go_q(u_y, T), and, on tiles that keep
    // every face, G_x = c F_x and G_y in L_G, L_G + 1, then the correction
    static constexpr int NEQ = 4;  // equilibrium factor sets
    static constexpr int L_DDX = 0, L_DDY = 1, L_LDX = 2, L_LDY = 3, L_DN = 4, L_E = 5, L_GY = 5 + NQ,
                         L_OX = 5 + 2 * NQ, L_OY = 5 + 3 * NQ, L_G = 5 + NEQ * NQ,
                         L_CA = 7 + NEQ * NQ, L_CB = 8 + NEQ * NQ, L_CC = 9 + NEQ * NQ;
    float loc[KP > 1 ? 10 + NEQ * NQ : 1][KP > 1 ? NN : 1];
    // WENO-5 face values.  Small tiles (at most 64 nodes) hold the faces of
    // all 25 velocities, so one pass computes them all and the node updates
    // follow without further barriers; larger tiles hold KP velocities'.
    static constexpr bool ALL_FACES = TX * TY <= 64;
    static constexpr int KF = ALL_FACES ? NK : KP;
    union {
        float fx[KF][TY][TX + 1];
        // wall density n_w of each tile row at the left and right diffuse wall
        // (Eq. nw): written and read between the moments and the force,
        // before any face value is stored
        float wnw[2][TY];
    };
    float fy[KF][TY + 1][TX];
    unsigned long long mbar;  // completion barrier of the TMA copy of phase 1

    // the staged population k at row r and column c of the region; planes lie
    // plane(r) apart
    __device__ __forceinline__ float *at(int k, int r, int c) { return &pop[k][r][c]; }
    __device__ __forceinline__ static constexpr bool staged(int, int) { return true; }
    __device__ __forceinline__ static constexpr int plane(int) { return HY * HP; }
    static constexpr int TMA_BYTES = 2 * NK * HY * HP * 4;
    __device__ __forceinline__ void tma(const TmaMap *m, int x0, int y0, unsigned mbar)
    {
        tma_load((unsigned)__cvta_generic_to_shared(&pop[0][0][0]), m->bytes[0], x0 - 4, y0 - 3, mbar);
    }
};

template <typename real, int TX, int TY, int KP, bool LEARNED>
struct StageSmem {
    using type = Smem32<TX, TY, KP>;
};
template <int TX, int TY, int KP, bool LEARNED>
struct StageSmem<double, TX, TY, KP, LEARNED> {
    static_assert(TX == 8 && TY == 8, "FP64 tiles are 8 x 8 (stage_shape)");
    using type = Smem64<KP, LEARNED>;
};

template <typename real>
__device__ __forceinline__ real sel5(const real v[NQ], int k)
{
    real r = v[0];
    r = (k == 1) ? v[1] : r;
    r = (k == 2) ? v[2] : r;
    r = (k == 3) ? v[3] : r;
    r = (k == 4) ? v[4] : r;
    return r;
}

// ---------------------------------------------------------------- force and update of an FP32 tile
// Phases 4 and 5 for FP32 populations (FP64: advance64 in olb_stage64.cuh), same
// contract.
template <int TX, int TY, int KP, bool LEARNED, typename Wait>
__device__ __forceinline__ bool advance32(Smem32<TX, TY, KP> &sm, const float *fn, float *out, const Geo &g,
                                          const Tab<float> &t, int x0, int y0, float ca, float cb, float cc, float ca_lo,
                                          float cb_lo, const float *mlp, Wait wait)
{
    using real = float;
    using S = Smem32<TX, TY, KP>;
    constexpr int NT = S::NT, NN = S::NN, HP = S::HP;
    const int tid = threadIdx.x;
    const int node = tid % S::LS, lane_k = tid / S::LS;
    const int tx = node % TX, ty = node / TX;
    const bool active = (node < NN) && (x0 + tx < g.nx) && (y0 + ty < g.ny);

    // ---- 4. force and equilibrium factors at the tile nodes.  The four
    // stencil sums and the two factor sets are split over the velocity lanes
    // (KP = 4: ddx | ddy | ldx, g(u_x) | ldy, g(u_y); KP = 2: x | y parts).
    constexpr int cy = 3, cx = 4;
    auto grad_sum = [&](bool along_x) {
        real acc = 0;
#pragma unroll
        for (int l = 1; l <= 3; ++l)
#pragma unroll
            for (int m = -3; m <= 3; ++m) {
                const int am = m < 0 ? -m : m;
                if (grad_w(l, am) != 0.0) {
                    const real w = real(l * grad_w(l, am));
                    acc = along_x ? fma(w, field_diff(sm.dp[ty + cy + m][tx + cx + l], sm.dp[ty + cy + m][tx + cx - l]), acc)
                                  : fma(w, field_diff(sm.dp[ty + cy + l][tx + cx + m], sm.dp[ty + cy - l][tx + cx + m]), acc);
                }
            }
        return acc;
    };
    auto glap_sum = [&](bool along_x) {
        real acc = 0;
        {
            // the stencil cancels its O(ds) terms down to O(ds^3) (a
            // factor ~1/(ds k)^2 on fine grids), so the weighted differences
            // are summed in double-float arithmetic with double-float weights
            // (exact products of the hi parts, TwoSum accumulation): the sum
            // keeps FP32 accuracy of itself, not of its terms
            f2 sum{0.0f, 0.0f};
#pragma unroll
            for (int l = 1; l <= 3; ++l)
#pragma unroll
                for (int m = -3; m <= 3; ++m) {
                    const int am = m < 0 ? -m : m;
                    if (glap_c(am, l) != 0.0) {
                        const float wh = (float)glap_c(am, l);
                        const float wl = (float)(glap_c(am, l) - (double)(float)glap_c(am, l));
                        const float2 a = along_x ? sm.n[ty + cy + m][tx + cx + l] : sm.n[ty + cy + l][tx + cx + m];
                        const float2 b = along_x ? sm.n[ty + cy + m][tx + cx - l] : sm.n[ty + cy - l][tx + cx + m];
                        const f2 dh = two_sum(a.x, -b.x);
                        const float dl = dh.lo + (a.y - b.y);
                        const float p = wh * dh.hi;
                        const float e = fmaf(wh, dh.hi, -p);
                        const float tl = fmaf(wh, dl, fmaf(wl, dh.hi, e));
                        const f2 t2 = two_sum(sum.hi, p);
                        sum = f2{t2.hi, t2.lo + (sum.lo + tl)};
                    }
                }
            acc = sum.hi + sum.lo;
        }
        return acc;
    };
    // With c the stage's coefficient of dt L (Eq. rk3), the node update below
    // needs per node G = c F and n ge_q(u_x, T), n go_q(u_x, T), ge_q(u_y, T),
    // go_q(u_y, T), the even and odd parts of the factors, in E, Ox, gy, Oy.
    const real sg3 = real(g.sigma) * real(g.inv_ds3);
    const real cit = cc * real(g.inv_tau);
    real Gx = 0, Gy = 0, E[NQ], gy[NQ], Ox[NQ], Oy[NQ];
    real qa = 0, qb = 0, qc = 0;  // alpha, beta, gamma of the equilibrium's correction (eq_correction)
    // equilibrium factor sets of the node at (tx_, ty_): x (scaled by n) into
    // ex, ox and y into ey, oy
    auto eq_sets = [&](bool x_set, real *a, real *b) {
        if (x_set) {
            eq_factors_split(t, sm.ux[ty][tx], sm.T[ty][tx], a, b);
            const real nn = sm.n[ty + 3][tx + 4].x;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                a[q] = nn * a[q];
                b[q] = nn * b[q];
            }
        } else {
            eq_factors_split(t, sm.uy[ty][tx], sm.T[ty][tx], a, b);
        }
    };
    if constexpr (KP == 1) {
        if (active) {
            const real ddx = grad_sum(true), ddy = grad_sum(false);
            const real ldx = glap_sum(true), ldy = glap_sum(false);
            const real nn = field_val(sm.n[ty + cy][tx + cx]);
            const real dn = real(g.inv_ds) / nn;
            Gx = cc * fma(ddx, dn, sg3 * ldx);
            Gy = cc * fma(ddy, dn, sg3 * ldy);
            eq_sets(true, E, Ox);
            eq_sets(false, gy, Oy);
            eq_correction(t, E, gy, sm.n[ty + 3][tx + 4], sm.eng[ty][tx], sm.ux[ty][tx], sm.uy[ty][tx], qa, qb, qc);
        }
    } else {
        static_assert(KP == 2 || KP == 4 || KP == 5 || KP == 8, "velocity lanes: 1, 2, 4, 5 or 8");
        using Sm = Smem32<TX, TY, KP>;
        if (active) {
            // KP = 8: lanes 0..5 take ddx, ddy, ldx, ldy, E, g(u_y);
            // KP = 5: lanes 0..3 ddx, ddy, ldx, ldy, lane 4 E and g(u_y);
            // KP = 4: lane 0 ddx, lane 1 ddy, lane 2 ldx + E, lane 3 ldy + g(u_y);
            // KP = 2: lane 0 the x parts, lane 1 the y parts
            const bool lane_ldx = KP == 2 ? lane_k == 0 : lane_k == 2;
            const bool lane_ldy = KP == 2 ? lane_k == 1 : lane_k == 3;
            const bool lane_gx = KP == 2 ? lane_k == 0 : (KP == 4 ? lane_k == 2 : lane_k == 4);
            const bool lane_gy = KP == 2 ? lane_k == 1 : (KP == 4 ? lane_k == 3 : (KP == 5 ? lane_k == 4 : lane_k == 5));
            if (lane_k == 0) {
                sm.loc[Sm::L_DDX][node] = grad_sum(true);
                sm.loc[Sm::L_DN][node] = real(g.inv_ds) / field_val(sm.n[ty + cy][tx + cx]);
            }
            if (lane_k == 1) sm.loc[Sm::L_DDY][node] = grad_sum(false);
            if (lane_ldx) sm.loc[Sm::L_LDX][node] = glap_sum(true);
            if (lane_ldy) sm.loc[Sm::L_LDY][node] = glap_sum(false);
            if (lane_gx) {
                eq_sets(true, E, Ox);
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    sm.loc[Sm::L_E + q][node] = E[q];
                    sm.loc[Sm::L_OX + q][node] = Ox[q];
                }
            }
            if (lane_gy) {
                eq_sets(false, gy, Oy);
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    sm.loc[Sm::L_GY + q][node] = gy[q];
                    sm.loc[Sm::L_OY + q][node] = Oy[q];
                }
            }
            {
                // the equilibrium's mass and energy correction, on a lane with
                // little else to do (KP = 8: lane 6; KP = 5, 4, 2: lane 1), from
                // the same factors the other lanes store (same operations)
                if (lane_k == (KP == 8 ? 6 : 1)) {
                    real ex[NQ], ox[NQ], ey[NQ], oy[NQ];
                    eq_sets(true, ex, ox);
                    eq_sets(false, ey, oy);
                    eq_correction(t, ex, ey, sm.n[ty + 3][tx + 4], sm.eng[ty][tx], sm.ux[ty][tx], sm.uy[ty][tx], qa,
                                  qb, qc);
                    sm.loc[Sm::L_CA][node] = qa;
                    sm.loc[Sm::L_CB][node] = qb;
                    sm.loc[Sm::L_CC][node] = qc;
                }
            }
        }
        __syncthreads();
        // G = c F at the node: in registers of each lane, or, on tiles that
        // keep every face, once per node in shared memory (read after the
        // barrier that ends the face pass)
        if (active && (!Sm::ALL_FACES || lane_k == 0)) {
            const real dn = sm.loc[Sm::L_DN][node];
            Gx = cc * fma(sm.loc[Sm::L_DDX][node], dn, sg3 * sm.loc[Sm::L_LDX][node]);
            Gy = cc * fma(sm.loc[Sm::L_DDY][node], dn, sg3 * sm.loc[Sm::L_LDY][node]);
            if constexpr (Sm::ALL_FACES) {
                sm.loc[Sm::L_G][node] = Gx;
                sm.loc[Sm::L_G + 1][node] = Gy;
            }
        }
    }

    // ---- 5. advection, collision and RK combination, KP velocities at a time
    const int nfx = (TX + 1) * TY, nfy = TX * (TY + 1);
    const real cadv = cc * real(g.inv_ds);
    using Sf = Smem32<TX, TY, KP>;
    constexpr int KF = Sf::KF;
    // one face value: x face (r, c) or y face (r, c) of velocity k, stored in
    // slot (FP32: its WENO correction, from first differences of the pairs)
    auto face = [&](int k, int slot, bool along_x, int r, int c) {
        const int k1 = k / NQ, k2 = k - NQ * (k / NQ);
        if (along_x) {
            if (y0 + r < g.ny && x0 + c <= g.nx) {
                // face at x = x0 + c: nodes x0+c-3 .. x0+c+2 are columns c+1 .. c+6
                const real *row = &sm.pop[k][3 + r][0];
                const float *lo = &sm.pl.lo[k][3 + r][0];
                auto pd = [&](int a_, int b_) { return pdiff(row[a_], lo[a_], row[b_], lo[b_]); };
                sm.fx[slot][r][c] =
                    (k1 > 2) ? face_corr<LEARNED>(mlp, pd(c + 2, c + 1), pd(c + 3, c + 2), pd(c + 4, c + 3), pd(c + 5, c + 4))
                             : face_corr<LEARNED>(mlp, pd(c + 5, c + 6), pd(c + 4, c + 5), pd(c + 3, c + 4), pd(c + 2, c + 3));
            }
        } else if (x0 + c < g.nx && y0 + r <= g.ny) {
            // face at y = y0 + r: rows y0+r-3 .. y0+r+2 are rows r .. r+5
            const int cc4 = 4 + c;
            const real(*P)[HP] = sm.pop[k];
            const float(*Lo)[HP] = sm.pl.lo[k];
            auto pd = [&](int a_, int b_) { return pdiff(P[a_][cc4], Lo[a_][cc4], P[b_][cc4], Lo[b_][cc4]); };
            sm.fy[slot][r][c] = (k2 > 2) ? face_corr<LEARNED>(mlp, pd(r + 1, r), pd(r + 2, r + 1), pd(r + 3, r + 2), pd(r + 4, r + 3))
                                         : face_corr<LEARNED>(mlp, pd(r + 4, r + 5), pd(r + 3, r + 4), pd(r + 2, r + 3), pd(r + 1, r + 2));
        }
    };
    // learned weights: the face of item (k, slot, along_x,
    // r, c), or none (valid false); every lane of the warp calls it together,
    // from a single call site, since the warp evaluates the network of its 32
    // stencils on the tensor pipe
    float *const mlp_sc = LEARNED ? const_cast<float *>(mlp) + MLP_SCRATCH_OFF + (tid >> 5) * MLP_WARP_SCRATCH : nullptr;
    auto learned_face = [&](int k, int slot, bool along_x, int r, int c, bool valid) {
        const int k1 = k / NQ, k2 = k - NQ * (k / NQ);
        valid = valid && (along_x ? (y0 + r < g.ny && x0 + c <= g.nx) : (x0 + c < g.nx && y0 + r <= g.ny));
        // the stencil v0 .. v4 in the upwind orientation, as positions of the
        // staged region: x faces along row 3 + r, y faces along column 4 + c
        int p0 = 0, step = 1;
        if (along_x) {
            p0 = (k1 > 2) ? c + 1 : c + 6;
            step = (k1 > 2) ? 1 : -1;
        } else {
            p0 = (k2 > 2) ? r : r + 5;
            step = (k2 > 2) ? 1 : -1;
        }
        real d[4] = {0, 0, 0, 0};
        if (valid) {
            const real *P = &sm.pop[k][0][0];
            auto at = [&](int m) { return along_x ? (3 + r) * HP + p0 + m * step : (p0 + m * step) * HP + 4 + c; };
            const float *Lo = &sm.pl.lo[k][0][0];
#pragma unroll
            for (int m = 0; m < 4; ++m) d[m] = pdiff(P[at(m + 1)], Lo[at(m + 1)], P[at(m)], Lo[at(m)]);
        }
        const bool acts = learned_guard(d[0], d[1], d[2], d[3]);
        float x[MLP_IN], w[MLP_OUT] = {0.0f, 0.0f, 0.0f};
        learned_input_x(d, acts, x);
        // the whole warp skips the network when none of its stencils needs it
        if (__any_sync(0xffffffffu, acts)) mlp_weights_warp(mlp, x, w, mlp_sc);
        if (valid) {
            const real res = acts ? learned_corr_from(w, d) : weno5_corr(d[0], d[1], d[2], d[3]);
            if (along_x) sm.fx[slot][r][c] = res;
            else sm.fy[slot][r][c] = res;
        }
    };
    // node update of velocity k (faces in slot) at tile node (tx_, ty_) with
    // Ek = n ge(k1), oxk = n go(k1), gyk = ge(k2), oyk = go(k2)
    auto update = [&](int k1, int k2, int slot, int tx_, int ty_, real Gx_, real Gy_, real Ek, real gyk, real oxk,
                      real oyk, real qa_, real qb_, real qc_) {
        const int k = NQ * k1 + k2;
        const int r = ty_ + 3, c = tx_ + 4;
        real dx = 0, dy = 0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            dx = fma(t.D[k1][q], sm.pop[NQ * q + k2][r][c], dx);
            dy = fma(t.D[k2][q], sm.pop[NQ * k1 + q][r][c], dy);
        }
        const real f = sm.pop[k][r][c];
        const long long o = (long long)(y0 + ty_) * g.pitch + (x0 + tx_);
        // flux difference = difference of the upwind nodes of the two
        // faces (a first difference of pairs) + difference of corrections
        const float(*P)[HP] = sm.pop[k];
        const float(*Lo)[HP] = sm.pl.lo[k];
        float adv = 0.0f;
        if (k1 != 2) {
            const int cu = k1 > 2 ? c : c + 1;
            adv = t.R[k1] * (pdiff(P[r][cu], Lo[r][cu], P[r][cu - 1], Lo[r][cu - 1]) +
                             (sm.fx[slot][ty_][tx_ + 1] - sm.fx[slot][ty_][tx_]));
        }
        if (k2 != 2) {
            const int ru = k2 > 2 ? r : r + 1;
            adv = fmaf(t.R[k2], pdiff(P[ru][c], Lo[ru][c], P[ru - 1][c], Lo[ru - 1][c]) +
                                    (sm.fy[slot][ty_ + 1][tx_] - sm.fy[slot][ty_][tx_]), adv);
        }
        // f - f^eq with f^eq = n (ge ge + ge go + go (ge + go)) - c: the
        // exactly symmetric part first, then the parts odd in p_y and in
        // p_x (each exactly odd after rounding), so that FP32 rounding of
        // the equilibrium carries no momentum; c (eq_correction) restores
        // its mass and energy
        const float fl = Lo[r][c];
        const float corr =
            (t.wHe[k1][0] * t.wHe[k2][0]) * fmaf(qc_, t.R2[k1] - t.R2[k2], fmaf(qb_, t.R2[k1] + t.R2[k2], qa_));
        const float neq = ((((f - Ek * gyk) + fl) - Ek * oyk) - oxk * (gyk + oyk)) + corr;
        // c L = -c xi.grad f - c F.grad_p f - (c/tau)(f - f^eq), then
        // out = ca f_n + cb f_s + c L (Eq. rk3) in double-float arithmetic
        const float inc = -fmaf(cit, neq, fmaf(Gx_, dx, fmaf(Gy_, dy, cadv * adv)));
        f2 acc = f2_cmul(f2{cb, cb_lo}, f, fl);
        if (ca != 0.0f) {
            const f2 an = f2_cmul(f2{ca, ca_lo}, fn[k * g.plane + o], fn[(NK + k) * g.plane + o]);
            const f2 sh = two_sum(acc.hi, an.hi);
            acc = f2{sh.hi, sh.lo + (acc.lo + an.lo)};
        }
        const f2 si = two_sum(acc.hi, inc);
        const f2 v = fast_two_sum(si.hi, si.lo + acc.lo);
        out[k * g.plane + o] = v.hi;
        out[(NK + k) * g.plane + o] = v.lo;
    };
    if (!wait()) return false;  // the populations of phase 1
    for (int kb = 0; kb < NK; kb += KF) {
        __syncthreads();  // loc ready / the previous velocities' faces are consumed
        if constexpr (LEARNED) {
            // learned weights: the network on the tensor pipe, one warp per 32
            // stencils (FP64 evaluates it per thread).  The faces of this pass (all 25 velocities' on small tiles, else
            // those of velocities kb .. kb+KP-1), enumerated as below, on
            // whole warps: items past the end take part in the network only.
            // Small tiles: the x faces of the 20 velocities with xi_x != 0,
            // then the y faces of the 20 with xi_y != 0, located by division
            // (as in the dense pass below); otherwise the KP velocities'
            // faces, located in their prefix table
            int end[KF], total = 0;
            if constexpr (Sf::ALL_FACES) {
                total = 20 * (nfx + nfy);
            } else {
#pragma unroll
                for (int sub = 0; sub < KF; ++sub) {
                    const int k = kb + sub;
                    if (k < NK) total += (k / NQ != 2 ? nfx : 0) + (k % NQ != 2 ? nfy : 0);
                    end[sub] = total;
                }
            }
            const int padded = (total + 31) & ~31;
            for (int e = tid; e < padded; e += NT) {
                int k, sub, f;
                bool valid = e < total;
                if constexpr (Sf::ALL_FACES) {
                    const int ee = valid ? e : 0;
                    if (ee < 20 * nfx) {
                        const int kx = ee / nfx;
                        k = kx < 2 * NQ ? kx : kx + NQ;
                        f = ee - kx * nfx;
                    } else {
                        const int e2 = ee - 20 * nfx, ky = e2 / nfy, q = ky & 3;
                        k = (ky >> 2) * NQ + (q < 2 ? q : q + 1);
                        f = nfx + e2 - ky * nfy;
                    }
                    sub = k;
                } else {
                    int start = 0;
                    sub = 0;
#pragma unroll
                    for (int q = 0; q + 1 < KF; ++q)
                        if (e >= end[q]) {
                            sub = q + 1;
                            start = end[q];
                        }
                    k = kb + sub;
                    f = e - start;
                    if (k / NQ == 2) f += nfx;
                    valid = valid && k < NK;
                }
                const bool along_x = f < nfx;
                const int r = along_x ? f / (TX + 1) : (f - nfx) / TX;
                const int c = along_x ? f - r * (TX + 1) : f - nfx - r * TX;
                // one call site: the warp's network must run as one instruction
                // stream (mma.sync needs every lane at the same instruction)
                learned_face(k, sub, along_x, valid ? r : 0, valid ? c : 0, valid);
            }
        } else if constexpr (Sf::ALL_FACES) {
            // (issue-bound) every face of every velocity once, in strips
            // of SX (SY) consecutive faces along a tile row (column), each
            // strip in the upwind direction of its velocity: the x strips of
            // the 20 velocities with xi_x != 0 (k1 != 2), then the y strips of
            // the 20 with xi_y != 0 (k2 != 2).
            constexpr int SX = (TX + 1) % 4 == 0 ? 4 : ((TX + 1) % 3 == 0 ? 3 : 1);
            constexpr int SY = (TY + 1) % 4 == 0 ? 4 : ((TY + 1) % 3 == 0 ? 3 : 1);
            constexpr int NSX = (TX + 1) / SX, NSY = (TY + 1) / SY;    // strips per row, per column
            constexpr int nsx = NSX * TY, nsy = NSY * TX;              // strips per velocity
            for (int e = tid; e < 20 * (nsx + nsy); e += NT) {
                if (e < 20 * nsx) {
                    const int kx = e / nsx, f = e - kx * nsx;
                    const int k = kx < 2 * NQ ? kx : kx + NQ;
                    const int r = f / NSX, cs = (f - r * NSX) * SX;
                    // face at x = x0 + c reads columns c+1 .. c+5 (xi_x > 0) or c+6 .. c+2
                    const real *row = &sm.pop[k][3 + r][0];
                    const real *rlo = &sm.pl.lo[k][3 + r][0];
                    if (k / NQ > 2) weno5_strip_c<SX>(row + cs + 1, rlo + cs + 1, 1, &sm.fx[k][r][cs], 1);
                    else weno5_strip_c<SX>(row + cs + SX + 5, rlo + cs + SX + 5, -1, &sm.fx[k][r][cs + SX - 1], -1);
                } else {
                    const int e2 = e - 20 * nsx, ky = e2 / nsy, f = e2 - ky * nsy, q = ky & 3;
                    const int k = (ky >> 2) * NQ + (q < 2 ? q : q + 1);
                    const int rs = (f / TX) * SY, c = f - (f / TX) * TX;
                    // face at y = y0 + r reads rows r .. r+4 (xi_y > 0) or r+5 .. r+1
                    if (k % NQ > 2)
                        weno5_strip_c<SY>(&sm.pop[k][rs][4 + c], &sm.pl.lo[k][rs][4 + c], HP, &sm.fy[k][rs][c], TX);
                    else
                        weno5_strip_c<SY>(&sm.pop[k][rs + SY + 4][4 + c], &sm.pl.lo[k][rs + SY + 4][4 + c], -HP,
                                          &sm.fy[k][rs + SY - 1][c], -TX);
                }
            }
            // (faces outside the grid are computed from staged values and never read)
        } else {
            // faces of the KP velocities kb .. kb+KP-1, each computed once and
            // enumerated densely: x faces of the tile rows unless xi_x = 0
            // (k1 = 2), then y faces of the tile columns unless xi_y = 0 (k2 = 2)
            int end[KP], total = 0;
#pragma unroll
            for (int sub = 0; sub < KP; ++sub) {
                const int k = kb + sub;
                if (k < NK) total += (k / NQ != 2 ? nfx : 0) + (k % NQ != 2 ? nfy : 0);
                end[sub] = total;
            }
            for (int e = tid; e < total; e += NT) {
                int sub = 0, start = 0;
#pragma unroll
                for (int q = 0; q + 1 < KP; ++q)
                    if (e >= end[q]) {
                        sub = q + 1;
                        start = end[q];
                    }
                const int k = kb + sub;
                int f = e - start;
                if (k / NQ == 2) f += nfx;
                if (f < nfx) {
                    const int r = f / (TX + 1);
                    face(k, sub, true, r, f - r * (TX + 1));
                } else {
                    const int r = (f - nfx) / TX;
                    face(k, sub, false, r, f - nfx - r * TX);
                }
            }
        }
        __syncthreads();
        if constexpr (Sf::ALL_FACES && KP == NQ) {
            // (issue-bound) node updates with five lanes: thread (node,
            // lane k2) advances the five velocities 5 k1 + k2, k1 unrolled,
            // so that the k1 tables are immediate operands and the node's
            // factors are read once
            if (active) {
                const int k2 = lane_k;
                const real Gx_ = sm.loc[Sf::L_G][node], Gy_ = sm.loc[Sf::L_G + 1][node];
                const real qa_ = sm.loc[Sf::L_CA][node], qb_ = sm.loc[Sf::L_CB][node], qc_ = sm.loc[Sf::L_CC][node];
                const real gyk = sm.loc[Sf::L_GY + k2][node], oyk = sm.loc[Sf::L_OY + k2][node];
#pragma unroll
                for (int k1 = 0; k1 < NQ; ++k1)
                    update(k1, k2, NQ * k1 + k2, tx, ty, Gx_, Gy_, sm.loc[Sf::L_E + k1][node], gyk,
                           sm.loc[Sf::L_OX + k1][node], oyk, qa_, qb_, qc_);
            }
        } else if constexpr (Sf::ALL_FACES) {
            // node updates, enumerated densely over (velocity, tile node)
            for (int e = tid; e < NK * NN; e += NT) {
                const int k = e / NN, nd = e - k * NN;
                const int tx_ = nd % TX, ty_ = nd / TX;
                if (x0 + tx_ >= g.nx || y0 + ty_ >= g.ny) continue;
                const int k1 = k / NQ, k2 = k - NQ * (k / NQ);
                update(k1, k2, k, tx_, ty_, sm.loc[Sf::L_G][nd], sm.loc[Sf::L_G + 1][nd], sm.loc[Sf::L_E + k1][nd],
                       sm.loc[Sf::L_GY + k2][nd], sm.loc[Sf::L_OX + k1][nd], sm.loc[Sf::L_OY + k2][nd],
                       sm.loc[Sf::L_CA][nd], sm.loc[Sf::L_CB][nd], sm.loc[Sf::L_CC][nd]);
            }
        } else {
            const int k = kb + lane_k;
            if (active && k < NK) {
                const int k1 = k / NQ, k2 = k - NQ * (k / NQ);
                real Ek, gyk, oxk = 0, oyk = 0, qa_ = qa, qb_ = qb, qc_ = qc;
                if constexpr (KP > 1) {
                    Ek = sm.loc[Sf::L_E + k1][node];
                    gyk = sm.loc[Sf::L_GY + k2][node];
                    oxk = sm.loc[Sf::L_OX + k1][node];
                    oyk = sm.loc[Sf::L_OY + k2][node];
                    qa_ = sm.loc[Sf::L_CA][node];
                    qb_ = sm.loc[Sf::L_CB][node];
                    qc_ = sm.loc[Sf::L_CC][node];
                } else {
                    Ek = sel5(E, k1);
                    gyk = sel5(gy, k2);
                    oxk = sel5(Ox, k1);
                    oyk = sel5(Oy, k2);
                }
                update(k1, k2, lane_k, tx, ty, Gx, Gy, Ek, gyk, oxk, oyk, qa_, qb_, qc_);
            }
        }
    }
    return true;
}

// One stage for the tile whose lower-left node is (x0, y0); all threads of
// the CTA call it (it synchronises).  ca, cb, cc: the stage's coefficients of
// f^n, f_s and dt L (Eq. rk3), in FP32; ca_lo, cb_lo: their remainders (1/3 and
// 2/3 as double-float constants).  g and t may live in parameter space (single
// grid) or shared memory (batch); tw: the table of the wall entries (geqw,
// inv_den), t itself for a single grid, the run's own in a batch, whose velocity
// tables t are common to all runs and passed as a kernel parameter; mlp: the
// learned network's parameters in shared memory (LEARNED only); tmap: TMA map of
// fs (of this run, in a batch) for this tile shape, or nullptr; fields: the
// moments of fs from k_fields.  Returns false when the TMA copy timed out (the
// CTA must stop).
template <int TX, int TY, int KP, bool LEARNED>
__device__ __forceinline__ bool stage_tile32(Smem32<TX, TY, KP> &sm, const float *__restrict__ fs, const float *fn,
                                             float *out, int *__restrict__ status, const Geo &g, const Tab<float> &t,
                                             const Tab<float> &tw, int x0, int y0, float ca, float cb, float cc,
                                             float ca_lo, float cb_lo, const float *mlp, const TmaMap *tmap,
                                             const StageFields<float> &fields)
{
    using S = Smem32<TX, TY, KP>;
    constexpr int NT = S::NT, HX = S::HX, HY = S::HY;
    const int tid = threadIdx.x;

    // ---- 1. populations of the region (c <-> x = x0 - 4 + c, r <-> y = y0 - 3 + r)
    const bool inside = tmap != nullptr && x0 >= 4 && x0 + TX + 4 <= g.nx && y0 >= 3 && y0 + TY + 3 <= g.ny;
    // the pre-pass fields of this thread's first position (phase 2's item e = tid)
    // are fetched into registers now, so that their latency overlaps the staging
    // of the populations
    using fld = FieldT<float>::type;
    fld pf_n{}, pf_dp{}, pf_T{}, pf_E{};
    float pf_ux = 0, pf_uy = 0;
    bool pf_ok = false, pf_node = false;
    int pf_r = 0, pf_c = 0;
    if (tid < HY * (HX - 2)) {
        pf_r = tid / (HX - 2);
        pf_c = tid - pf_r * (HX - 2) + 1;
        const int gx = x0 - 4 + pf_c, gyr = y0 - 3 + pf_r;
        pf_ok = !(g.walls && (gx < 0 || gx >= g.nx)) && !(g.spec_y && (gyr < 0 || gyr >= g.ny));
        if (pf_ok) {
            const long long o = (long long)wrap(gyr, g.ny) * g.pitch + wrap(gx, g.nx);
            pf_n = fields.n[o];
            pf_dp = fields.dp[o];
            const int tr = pf_r - 3, tc = pf_c - 4;
            pf_node = tr >= 0 && tr < TY && tc >= 0 && tc < TX;
            if (pf_node) {
                pf_ux = fields.ux[o];
                pf_uy = fields.uy[o];
                pf_T = fields.T[o];
                pf_E = fields.E[o];
            }
        }
    }
    // A tile inside the grid touches its staged populations first in the face
    // pass (no walls, no sides), so phases 2-4 run while the copy is in flight
    if (inside) tma_issue(sm, tmap, x0, y0);
    else load_region(sm, fs, g, x0, y0);
    __syncthreads();

    // ---- 2. fields at every fluid position of the region that the 7 x 7
    // force stencils reach (columns 1 .. HX-2; ghost positions of walls and
    // specular sides take the reflected fields in phase 3): n and Delta p on the
    // region, u, T and e at the tile nodes.  A tile at a diffuse wall also
    // computes here, on warps of their own, its wall fluxes.
    const bool x_lo = g.walls && x0 == 0;                // ghost columns at x = 0
    const bool x_hi = g.walls && (x0 + TX + 3 >= g.nx);  // ghost columns at x = nx ds
    const bool left_wall = x_lo && g.wall_lo;
    const bool right_wall = x_hi && g.wall_hi;
    if (pf_ok) {
        sm.n[pf_r][pf_c] = pf_n;
        sm.dp[pf_r][pf_c] = pf_dp;
        if (pf_node) {
            sm.ux[pf_r - 3][pf_c - 4] = pf_ux;
            sm.uy[pf_r - 3][pf_c - 4] = pf_uy;
            sm.T[pf_r - 3][pf_c - 4] = pf_T;
            sm.eng[pf_r - 3][pf_c - 4] = pf_E;
        }
    }
    for (int e = tid + NT; e < HY * (HX - 2); e += NT) {
        const int r = e / (HX - 2), c = e - r * (HX - 2) + 1;
        const int gx = x0 - 4 + c, gyr = y0 - 3 + r;
        if (g.walls && (gx < 0 || gx >= g.nx)) continue;
        if (g.spec_y && (gyr < 0 || gyr >= g.ny)) continue;
        const long long o = (long long)wrap(gyr, g.ny) * g.pitch + wrap(gx, g.nx);
        sm.n[r][c] = fields.n[o];
        sm.dp[r][c] = fields.dp[o];
        const int tr = r - 3, tc = c - 4;
        if (tr >= 0 && tr < TY && tc >= 0 && tc < TX) {
            sm.ux[tr][tc] = fields.ux[o];
            sm.uy[tr][tc] = fields.uy[o];
            sm.T[tr][tc] = fields.T[o];
            sm.eng[tr][tc] = fields.E[o];
        }
    }
    // wall-flux items start on the first warp after the field positions
    if (left_wall || right_wall)
        wall_flux<float, LEARNED>(sm, g, t, tw, mlp, x0, (HY * (HX - 2) + 31) / 32 * 32, left_wall, right_wall);

    // ---- 3. sides: n and Delta p reflected evenly into the ghost layers of
    // walls and specular planes (Sec. 3.4.3; y first, then x over every row,
    // which makes the corners a double reflection); the incoming ghosts at walls
    if (g.spec_y && (y0 == 0 || y0 + TY + 2 >= g.ny)) {
        __syncthreads();
        for (int e = tid; e < HY * HX; e += NT) {
            const int r = e / HX, c = e - r * HX;
            const int gyr = y0 - 3 + r;
            if (gyr >= 0 && gyr < g.ny) continue;
            if ((gyr < 0 ? -1 - gyr : gyr - g.ny) > 2) continue;
            const int rm = (gyr < 0 ? -1 - gyr : 2 * g.ny - 1 - gyr) - (y0 - 3);
            sm.n[r][c] = sm.n[rm][c];
            sm.dp[r][c] = sm.dp[rm][c];
        }
    }
    if (x_lo || x_hi) {
        __syncthreads();
        for (int e = tid; e < HY * HX; e += NT) {
            const int r = e / HX, c = e - r * HX;
            const int gx = x0 - 4 + c;
            if (gx >= 0 && gx < g.nx) continue;
            const bool right = gx >= g.nx;
            if ((right ? gx - g.nx : -1 - gx) > 2) continue;  // beyond ghost layer 2
            const int cm = (right ? 2 * g.nx - 1 - gx : -1 - gx) - (x0 - 4);
            sm.n[r][c] = sm.n[r][cm];
            sm.dp[r][c] = sm.dp[r][cm];
        }
        wall_ghosts<float>(sm, g, tw, x0, (HY * HX + 31) / 32 * 32, left_wall, right_wall);
    }
    __syncthreads();

    // ---- 4, 5. force, fluxes, collision and RK-3 combination
    return advance32<TX, TY, KP, LEARNED>(sm, fn, out, g, t, x0, y0, ca, cb, cc, ca_lo, cb_lo, mlp,
                                          [&] { return !inside || tma_finish(sm, status); });
}

// Shared memory of the single-grid kernel: the tile staging, then (learned
// weights only) the network's parameters at a 16-byte aligned offset and the
// warps' scratch for the network's tensor-pipe layer.
template <typename real, int TX, int TY, int KP>
constexpr size_t mlp_offset()
{
    return (sizeof(typename StageSmem<real, TX, TY, KP, true>::type) + 15) / 16 * 16;
}
template <typename real, int TX, int TY, int KP, bool LEARNED>
constexpr size_t fused_smem_bytes()
{
    // learned: the parameters; FP32 also the split W2 and MLP_WARP_SCRATCH
    // floats per warp
    using S = typename StageSmem<real, TX, TY, KP, LEARNED>::type;
    constexpr size_t mlp_floats = sizeof(real) == 4 ? MLP_SCRATCH_OFF + S::NT / 32 * MLP_WARP_SCRATCH : MLP_P + 1;
    return LEARNED ? mlp_offset<real, TX, TY, KP>() + mlp_floats * sizeof(float) : sizeof(S);
}
// Threads of a shape's CTA: FP32: KP lanes of the tile's nodes, rounded up to
// warps; FP64: Plan64.
template <typename real, int TX, int TY, int KP>
constexpr int stage_threads()
{
    return StageSmem<real, TX, TY, KP, false>::type::NT;
}

// CTAs per SM that the register allocation must leave room for: as many as
// the shared memory (228 KB per SM, 1 KB of it reserved per CTA) and the
// 2048 threads of an SM allow.  Without this bound the compiler may take
// more registers than that occupancy leaves (e.g. 80 for a 512-thread CTA
// that could otherwise share its SM), capped at cap when cap > 0.
constexpr int fused_min_ctas(size_t smem_bytes, int threads, int cap = 0)
{
    const int by_smem = (int)((228 * 1024) / (smem_bytes + 1024)), by_threads = 2048 / threads;
    const int n = by_smem < by_threads ? by_smem : by_threads;
    return n < 1 ? 1 : (cap > 0 && n > cap ? cap : n);
}

// Single grid: one CTA per tile.  Learned-weight instances leave their network the registers
// it needs: FP32 (tensor-pipe network) at most two CTAs per SM, FP64 (per-thread
// network) one.
template <typename real, int TX, int TY, int KP, bool LEARNED>
__global__ void __launch_bounds__((stage_threads<real, TX, TY, KP>()),
                                  fused_min_ctas(fused_smem_bytes<real, TX, TY, KP, LEARNED>(),
                                                 stage_threads<real, TX, TY, KP>(),
                                                 LEARNED ? (sizeof(real) == 4 ? 2 : 1) : 0))
k_fused(const real *__restrict__ fs, const real *fn, real *out, int *__restrict__ status,
        const __grid_constant__ Geo g, const __grid_constant__ Tab<real> t, real ca, real cb, real cc, real ca_lo,
        real cb_lo, const __grid_constant__ StageK sk, const float *__restrict__ mlp, const __grid_constant__ TmaArg tma,
        const __grid_constant__ StageFields<real> fields)
{
    // 128-byte aligned: the TMA copy of phase 1 lands at offset 0
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto &sm = *reinterpret_cast<typename StageSmem<real, TX, TY, KP, LEARNED>::type *>(smem_raw);
    float *mlp_sm = nullptr;
    if constexpr (LEARNED) {
        mlp_sm = reinterpret_cast<float *>(smem_raw + mlp_offset<real, TX, TY, KP>());
        for (int p = threadIdx.x; p < MLP_P; p += blockDim.x) mlp_sm[p] = __ldg(mlp + p);
        if constexpr (sizeof(real) == 4) {
            __syncthreads();
            mlp_split_w2(mlp_sm);
        }
        // made visible by the first barrier inside stage_tile
    }
    const TmaMap *tm = tma.on ? &tma.map : nullptr;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    if constexpr (sizeof(real) == 8)
        stage_tile64<KP, LEARNED>(sm, fs, fn, out, status, g, t, t, x0, y0, sk, mlp_sm, tm, fields);
    else
        stage_tile32<TX, TY, KP, LEARNED>(sm, fs, fn, out, status, g, t, t, x0, y0, ca, cb, cc, ca_lo, cb_lo, mlp_sm, tm,
                                          fields);
}

// Batch of independent runs (uneven grid sizes, own parameters): one CTA per
// (run, tile) work item, in the order of the items, so that the hardware
// dispatches neighbouring tiles together and their halos stay in L2 (a
// persistent grid-stride loop let the CTAs drift apart and measured slower);
// tile_start[r] is the first item of run r (prefix sum, tile_start[nruns] =
// total).  Each run has its populations at offset `off` of the three shared
// buffers and its own status word.
template <typename real, int TX, int TY, int KP>
__global__ void __launch_bounds__((stage_threads<real, TX, TY, KP>()),
                                  fused_min_ctas(fused_smem_bytes<real, TX, TY, KP, false>() + sizeof(BatchRun<real>),
                                                 stage_threads<real, TX, TY, KP>()))
k_fused_batch(const real *__restrict__ fs, const real *fn, real *out, int *__restrict__ status,
              const BatchRun<real> *__restrict__ runs, const int *__restrict__ tile_start, int nruns,
              const __grid_constant__ Tab<real> tv, real ca, real cb, real ccoef, real ca_lo, real cb_lo, int st,
              char *fields, const TmaMap *__restrict__ tmaps)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto &sm = *reinterpret_cast<typename StageSmem<real, TX, TY, KP, false>::type *>(smem_raw);
    __shared__ __align__(16) BatchRun<real> run;
    const int item = blockIdx.x;
    const int lo = run_of(tile_start, nruns, item);
    {
        const int4 *src = reinterpret_cast<const int4 *>(runs + lo);
        int4 *dst = reinterpret_cast<int4 *>(&run);
        for (int w = threadIdx.x; w < (int)(sizeof(BatchRun<real>) / sizeof(int4)); w += blockDim.x)
            dst[w] = __ldg(src + w);
    }
    __syncthreads();
    const int lt = item - __ldg(tile_start + lo);
    const int x0 = (lt % run.ntx) * TX, y0 = (lt / run.ntx) * TY;
    const StageFields<real> fl = fields_of<real>(fields + run.foff, run.g);
    // the run's tensor map of fs lives in global memory, written by the host
    // before the launch: acquire it for the tensormap proxy before the thread
    // that issues the copy uses it
    const TmaMap *tm = tmaps ? tmaps + lo : nullptr;
    if (tm && threadIdx.x == 0)
        for (int k = 0; k < 2; ++k)
            asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(tm->bytes[k]) : "memory");
    if constexpr (sizeof(real) == 8)
        stage_tile64<KP, false>(sm, fs + run.off, fn + run.off, out + run.off, status + lo, run.g, tv, run.t, x0, y0,
                                run.k[st], nullptr, tm, fl);
    else
        stage_tile32<TX, TY, KP, false>(sm, fs + run.off, fn + run.off, out + run.off, status + lo, run.g, tv, run.t, x0,
                                        y0, ca, cb, ccoef * (real)run.g.dt, ca_lo, cb_lo, nullptr, tm, fl);
}

template <typename real, int TX, int TY, int KP, bool LEARNED = false>
cudaError_t fused_prepare_one()
{
    cudaError_t e = cudaFuncSetAttribute(k_fused<real, TX, TY, KP, LEARNED>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)fused_smem_bytes<real, TX, TY, KP, LEARNED>());
    if constexpr (!LEARNED)
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_fused_batch<real, TX, TY, KP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)fused_smem_bytes<real, TX, TY, KP, false>());
    return e;
}

template <typename real, int TX, int TY, int KP, bool LEARNED = false>
cudaError_t fused_launch_one(const real *fs, const real *fn, real *out, int *status, const Geo &g,
                             const Tab<real> &t, StageCoef c, const float *mlp, const TmaMap *tmap, void *fields,
                             cudaStream_t s)
{
    dim3 grid((g.nx + TX - 1) / TX, (g.ny + TY - 1) / TY);
    TmaArg tma{};
    if (tmap) {
        tma.map = *tmap;
        tma.on = 1;
    }
    // the moments of fs first (one thread per node), then the stage
    const StageFields<real> fl = fields_of<real>(fields, g);
    const long long N = (long long)g.nx * g.ny;
    k_fields<real><<<(unsigned)((N + 255) / 256), 256, 0, s>>>(fs, fl, status, g, t);
    StageK sk{};
    if constexpr (sizeof(real) == 8) {
        sk = stage_constants(g, c);
        k_force<<<dim3((g.nx + FORCE_X - 1) / FORCE_X, (g.ny + FORCE_Y - 1) / FORCE_Y), FORCE_THREADS, 0, s>>>(fl, g, sk);
    }
    k_fused<real, TX, TY, KP, LEARNED><<<grid, stage_threads<real, TX, TY, KP>(), fused_smem_bytes<real, TX, TY, KP, LEARNED>(), s>>>(
        fs, fn, out, status, g, t, (real)c.ca, (real)c.cb, (real)c.cc, (real)(c.ca - (double)(real)c.ca),
        (real)(c.cb - (double)(real)c.cb), sk, mlp, tma, fl);
    return cudaGetLastError();
}

template <typename real, int TX, int TY, int KP>
cudaError_t fused_batch_launch_one(const real *fs, const real *fn, real *out, int *status, const void *runs,
                                   const int *tile_start, int nruns, int total, const Tab<real> &t, StageCoef c,
                                   int st, void *fields, const long long *node_start, long long total_nodes,
                                   const int *force_start, int force_blocks, const TmaMap *tmaps, cudaStream_t s)
{
    if (total < 1) return cudaSuccess;
    if (total_nodes > 0) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const long long want = (total_nodes + 255) / 256, cap = 8LL * sms * 8;
        k_fields_batch<real><<<(unsigned)(want < cap ? want : cap), 256, 0, s>>>(
            fs, static_cast<char *>(fields), static_cast<const BatchRun<real> *>(runs), node_start, nruns, total_nodes,
            status);
    }
    if constexpr (sizeof(real) == 8)
        k_force_batch<<<force_blocks, FORCE_THREADS, 0, s>>>(
            static_cast<char *>(fields), static_cast<const BatchRun<double> *>(runs), force_start, nruns, st);
    k_fused_batch<real, TX, TY, KP><<<total, stage_threads<real, TX, TY, KP>(), fused_smem_bytes<real, TX, TY, KP, false>(), s>>>(
        fs, fn, out, status, static_cast<const BatchRun<real> *>(runs), tile_start, nruns, t, (real)c.ca, (real)c.cb,
        (real)c.cc, (real)(c.ca - (double)(real)c.ca), (real)(c.cb - (double)(real)c.cb), st, static_cast<char *>(fields),
        tmaps);
    return cudaGetLastError();
}

// Shapes compiled for each precision: TX x TY nodes per CTA, KP velocities
// advanced at once (KP lanes of TX*TY threads rounded up to whole warps).  FP32:
// those of TILE_X/TILE_Y/TILE_K in olb_internal.cuh; FP64: those that
// stage_shape maps them to.  OLB_FUSED_LEARNED_*: with learned weights.
#define OLB_FUSED_SHAPES_float(DO) \
    DO(float, 8, 8, 4) DO(float, 16, 8, 2) DO(float, 16, 8, 1) DO(float, 32, 8, 1) DO(float, 32, 16, 1) \
    DO(float, 8, 8, 8) DO(float, 7, 8, 8) DO(float, 8, 8, 5)
#define OLB_FUSED_SHAPES_double(DO) DO(double, 8, 8, 8) DO(double, 8, 8, 5)
#define OLB_FUSED_LEARNED_float(DO) DO(float, 8, 8, 4) DO(float, 16, 8, 2) DO(float, 32, 16, 1)
#define OLB_FUSED_LEARNED_double(DO) DO(double, 8, 8, 4)
#define OLB_FUSED_PREP_CASE(real, A, B, C) \
    if (!learned && sh.tx == A && sh.ty == B && sh.kp == C) return fused_prepare_one<real, A, B, C>();
#define OLB_FUSED_PREP_LEARNED(real, A, B, C) \
    if (learned && sh.tx == A && sh.ty == B && sh.kp == C) return fused_prepare_one<real, A, B, C, true>();
#define OLB_FUSED_LAUNCH_CASE(real, A, B, C)                  \
    if (!mlp && sh.tx == A && sh.ty == B && sh.kp == C)        \
        return fused_launch_one<real, A, B, C>(fs, fn, out, status, g, t, c, mlp, tma, fields, s);
#define OLB_FUSED_LAUNCH_LEARNED(real, A, B, C)               \
    if (mlp && sh.tx == A && sh.ty == B && sh.kp == C)         \
        return fused_launch_one<real, A, B, C, true>(fs, fn, out, status, g, t, c, mlp, tma, fields, s);
#define OLB_FUSED_BATCH_CASE(real, A, B, C)                                                                  \
    if (sh.tx == A && sh.ty == B && sh.kp == C)                                                              \
        return fused_batch_launch_one<real, A, B, C>(fs, fn, out, status, runs, tile_start, nruns, total, t,     \
                                                     c, st, fields, node_start, total_nodes, force_start,       \
                                                     force_blocks, tmaps, s);
#define OLB_DEFINE_FUSED(real)                                                                                \
    cudaError_t prepare_fused(real *, int tx, int ty, int kp, bool learned)                                   \
    {                                                                                                         \
        const Shape sh = stage_shape(sizeof(real) == 8, learned, tx, ty, kp);                                 \
        OLB_FUSED_SHAPES_##real(OLB_FUSED_PREP_CASE)                                                          \
        OLB_FUSED_LEARNED_##real(OLB_FUSED_PREP_LEARNED)                                                      \
        return cudaErrorInvalidValue;                                                                         \
    }                                                                                                         \
    cudaError_t launch_fused(const real *fs, const real *fn, real *out, int *status, const Geo &g,            \
                             const Tab<real> &t, StageCoef c, int tx, int ty, int kp, const float *mlp,       \
                             const TmaMap *tma, void *fields, cudaStream_t s)                                 \
    {                                                                                                         \
        const Shape sh = stage_shape(sizeof(real) == 8, mlp != nullptr, tx, ty, kp);                          \
        OLB_FUSED_SHAPES_##real(OLB_FUSED_LAUNCH_CASE)                                                        \
        OLB_FUSED_LEARNED_##real(OLB_FUSED_LAUNCH_LEARNED)                                                    \
        return cudaErrorInvalidValue;                                                                         \
    }                                                                                                         \
    cudaError_t launch_fused_batch(const real *fs, const real *fn, real *out, int *status, const void *runs,  \
                                   const int *tile_start, int nruns, int total, const Tab<real> &t,         \
                                   StageCoef c, int st, int tx, int ty, int kp, void *fields,                 \
                                   const long long *node_start, long long total_nodes, const int *force_start, int force_blocks, const TmaMap *tmaps,   \
                                   cudaStream_t s)                                                            \
    {                                                                                                         \
        const Shape sh = stage_shape(sizeof(real) == 8, false, tx, ty, kp);                                   \
        OLB_FUSED_SHAPES_##real(OLB_FUSED_BATCH_CASE)                                                         \
        return cudaErrorInvalidValue;                                                                         \
    }                                                                                                         \
    size_t batch_run_bytes(real *) { return sizeof(BatchRun<real>); }                                         \
    void batch_run_fill(real *, void *dst, const Geo &g, const Tab<real> &t, long long off, long long foff,   \
                        int ntx)                                                                              \
    {                                                                                                         \
        BatchRun<real> r{};                                                                                   \
        r.g = g;                                                                                              \
        r.t = t;                                                                                              \
        r.off = off;                                                                                          \
        r.foff = foff;                                                                                        \
        r.ntx = ntx;                                                                                          \
        const StageCoef c[3] = {{0.0, 1.0, g.dt}, {0.75, 0.25, 0.25 * g.dt}, {1.0 / 3.0, 2.0 / 3.0, 2.0 / 3.0 * g.dt}}; \
        if (sizeof(real) == 8)                                                                                \
            for (int st = 0; st < 3; ++st) r.k[st] = stage_constants(g, c[st]);                               \
        *static_cast<BatchRun<real> *>(dst) = r;                                                              \
    }

}  // namespace olb
