// olb_tile.cuh -- staging of a tile's populations in shared memory (TMA for tiles
// inside the grid, else element by element) and the diffuse walls (Sec. 3.4.2),
// for the stage kernels of both precisions.
#pragma once

#include "olb_fields.cuh"
#include "olb_mlp.cuh"

namespace olb {

// Face value of one upwind-ordered FP64 stencil: Jiang-Shu weights, or the
// learned network's (parameters mlp) when LEARNED.
template <bool LEARNED>
__device__ __forceinline__ double face_value(const float *mlp, double v0, double v1, double v2, double v3, double v4)
{
    if constexpr (LEARNED)
        return weno5_learned(mlp, v0, v1, v2, v3, v4);
    else
    {
        auto high = [](double v) { return __double2hiint(v) & 0x7fffffff; };
        const FfScale s = ff_scale(max(max(max(high(v0), high(v1)), max(high(v3), high(v4))), high(v2)));
        return weno5_face(v2, v1 - v0, v2 - v1, v3 - v2, v4 - v3, s);
    }
}

// FP32 pairs: the correction c (face value minus the upwind node v2) of the
// stencil with first differences d01 .. d34.
template <bool LEARNED>
__device__ __forceinline__ float face_corr(const float *mlp, float d01, float d12, float d23, float d34)
{
    if constexpr (LEARNED)
        return weno5_learned_corr(mlp, d01, d12, d23, d34);
    else
        return weno5_corr(d01, d12, d23, d34);
}

// ---------------------------------------------------------------- TMA staging
// Iterations of the bounded wait for the copy (each try_wait suspends for at
// most a short, hardware-defined time): far above the microseconds a copy of
// a tile's region takes, far below a hang.
constexpr int TMA_WAIT_LIMIT = 1 << 16;

__device__ __forceinline__ bool mbar_wait(unsigned mbar, unsigned parity)
{
    for (int i = 0; i < TMA_WAIT_LIMIT; ++i) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Phase 1 for a tile whose staged region lies inside the grid: TMA copies of the
// boxes of the tensor maps (TmaMap) into the staging arrays, completion tracked by
// an mbarrier.  tma_issue starts the copies (all threads call it; it
// synchronises); tma_finish waits for them with the bounded wait.  If the wait
// runs out, bit 1 of the status word is set, the copies are waited for once more
// (bounded) and false is returned: the caller leaves the tile untouched and the
// CTA stops.  After completed copies the barrier is invalidated.
__device__ __forceinline__ void tma_load(unsigned dst, const unsigned char *map, int x, int y, unsigned mbar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(0), "r"(mbar)
        : "memory");
}
template <typename Smem>
__device__ __forceinline__ void tma_issue(Smem &sm, const TmaMap *tmap, int x0, int y0)
{
    const unsigned mbar = (unsigned)__cvta_generic_to_shared(&sm.mbar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"((unsigned)Smem::TMA_BYTES) : "memory");
        sm.tma(tmap, x0, y0, mbar);
    }
    __syncthreads();  // the barrier is initialised before anyone waits on it
}
template <typename Smem>
__device__ __forceinline__ bool tma_finish(Smem &sm, int *status)
{
    const unsigned mbar = (unsigned)__cvta_generic_to_shared(&sm.mbar);
    const bool ok = mbar_wait(mbar, 0);
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) atomicOr(status, 2);
        mbar_wait(mbar, 0);
        return false;
    }
    // every thread has passed its wait (the barrier above)
    if (threadIdx.x == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(mbar) : "memory");
    return true;
}

// Staged populations of an 8 x 8 tile: P planes (FP64 25; FP32 25 hi, then 25 lo)
// of the tile's rows (columns x0 - 4 ...) and of the three rows below and above
// its nodes.
template <typename real>
struct Staged {
    static constexpr int TX = 8, TY = 8, HX = TX + 8, HY = TY + 6, NN = TX * TY, P = pop_planes<real>();
    static constexpr int HP = region_pitch(TX, sizeof(real) == 8);  // pitch of a staged row
    alignas(128) real mid[P][TY][HP];
    alignas(128) real below[P][3][TX];
    alignas(128) real above[P][3][TX];
    real wnw[2][TY];          // wall density of each tile row (Eq. nw)
    unsigned long long mbar;  // completion barrier of the TMA copies

    // plane k at row r and column c of the region (r: y = y0 - 3 + r, c: x = x0 - 4 +
    // c); planes lie plane(r) apart; the corners of the region are not staged
    __device__ __forceinline__ real *at(int k, int r, int c)
    {
        return r < 3 ? &below[k][r][c - 4] : r < TY + 3 ? &mid[k][r - 3][c] : &above[k][r - TY - 3][c - 4];
    }
    __device__ __forceinline__ static constexpr bool staged(int r, int c)
    {
        return (r >= 3 && r < TY + 3) || (c >= 4 && c < TX + 4);
    }
    __device__ __forceinline__ static constexpr int plane(int r) { return r >= 3 && r < TY + 3 ? TY * HP : 3 * TX; }
    static constexpr int TMA_BYTES = P * (TY * HP + 6 * TX) * (int)sizeof(real);
    __device__ __forceinline__ void tma(const TmaMap *m, int x0, int y0, unsigned bar)
    {
        tma_load((unsigned)__cvta_generic_to_shared(&mid[0][0][0]), m->bytes[0], x0 - 4, y0, bar);
        tma_load((unsigned)__cvta_generic_to_shared(&below[0][0][0]), m->bytes[1], x0, y0 - 3, bar);
        tma_load((unsigned)__cvta_generic_to_shared(&above[0][0][0]), m->bytes[1], x0, y0 + TY, bar);
    }
};

// A line of an 8 x 8 tile in the upwind direction of a velocity: row i (20
// velocities with xi_x != 0) or column i (20 with xi_y != 0), q counting the
// velocities.  p0[0], p0[halo], p0[2 halo] are the three nodes behind it, p1[j
// step] its nodes, p2[0] and p2[halo] the two ahead.
template <typename real>
struct Line {
    const real *p0, *p1, *p2;
    int halo, step;
    bool up;
};
__device__ __forceinline__ int line_velocity(bool along_x, int q)
{
    return along_x ? (q < 2 * NQ ? q : q + NQ) : (q >> 2) * NQ + ((q & 3) < 2 ? (q & 3) : (q & 3) + 1);
}
template <typename real>
__device__ __forceinline__ Line<real> line_of(const Staged<real> &sm, bool along_x, int q, int i)
{
    constexpr int TX = Staged<real>::TX, TY = Staged<real>::TY, HP = Staged<real>::HP;
    const int k = line_velocity(along_x, q);
    Line<real> l;
    l.up = along_x ? k / NQ > 2 : k % NQ > 2;
    l.step = l.halo = l.up ? 1 : -1;
    if (along_x) {
        const real *row = &sm.mid[k][i][0];
        l.p0 = row + (l.up ? 1 : TX + 6);
        l.p1 = row + (l.up ? 4 : TX + 3);
        l.p2 = row + (l.up ? TX + 4 : 3);
    } else {
        l.halo *= TX;
        l.step *= HP;
        l.p0 = l.up ? &sm.below[k][0][i] : &sm.above[k][2][i];
        l.p1 = &sm.mid[k][l.up ? 0 : TY - 1][4 + i];
        l.p2 = l.up ? &sm.above[k][0][i] : &sm.below[k][2][i];
    }
    return l;
}

// ---------------------------------------------------------------- element by element
// Phase 1 for the other tiles (region position (r, c): y = y0 - 3 + r, x = x0 - 4 +
// c): periodic sides wrap.  Ghost layers 0..2 of a specular side hold the
// populations of the first three nodes inside with the normal velocity component
// reversed (Sec. 3.4.1); diffuse-wall ghosts are set later; anything further out
// is never read and holds 0.  By the threads from `first` on.
template <typename real, typename S>
__device__ __forceinline__ void load_region(S &sm, const real *__restrict__ fs, const Geo &g, int x0, int y0, int first = 0)
{
    constexpr int HX = S::HX, HY = S::HY, NT = S::NT;
    for (int e = (int)threadIdx.x - first; e < HY * HX; e += NT - first) {
        const int r = e / HX, c = e - r * HX;
        if (!S::staged(r, c)) continue;
        real *dst = sm.at(0, r, c);
        const int dp = S::plane(r);
        int gy = y0 - 3 + r, gx = x0 - 4 + c;
        bool flip_x = false, flip_y = false, zero = false;
        if (gy < 0 || gy >= g.ny) {
            if (!g.spec_y) {
                gy = wrap(gy, g.ny);
            } else if ((gy < 0 ? -1 - gy : gy - g.ny) <= 2) {
                gy = gy < 0 ? -1 - gy : 2 * g.ny - 1 - gy;
                flip_y = true;
            } else {
                zero = true;
            }
        }
        if (gx < 0 || gx >= g.nx) {
            const bool lo = gx < 0;
            if (!g.walls) {
                gx = wrap(gx, g.nx);
            } else if ((lo ? g.spec_lo : g.spec_hi) && (lo ? -1 - gx : gx - g.nx) <= 2) {
                gx = lo ? -1 - gx : 2 * g.nx - 1 - gx;
                flip_x = true;
            } else {
                zero = true;
            }
        }
        if (zero) {
#pragma unroll 5
            for (int k = 0; k < NK; ++k) {
                dst[k * dp] = real(0);
                if constexpr (sizeof(real) == 4) dst[(NK + k) * dp] = 0.0f;
            }
            continue;
        }
        const real *src = fs + (long long)gy * g.pitch + gx;
        if (!flip_x && !flip_y) {
#pragma unroll 5
            for (int k = 0; k < NK; ++k) {
                dst[k * dp] = __ldg(src + k * g.plane);
                if constexpr (sizeof(real) == 4) dst[(NK + k) * dp] = __ldg(src + (NK + k) * g.plane);
            }
        } else {
#pragma unroll
            for (int k1 = 0; k1 < NQ; ++k1)
#pragma unroll
                for (int k2 = 0; k2 < NQ; ++k2) {
                    const int kk = NQ * (flip_x ? NQ - 1 - k1 : k1) + (flip_y ? NQ - 1 - k2 : k2);
                    dst[(NQ * k1 + k2) * dp] = __ldg(src + kk * g.plane);
                    if constexpr (sizeof(real) == 4) dst[(NK + NQ * k1 + k2) * dp] = __ldg(src + (NK + kk) * g.plane);
                }
        }
    }
}

// ---------------------------------------------------------------- diffuse walls
// The wall-face flux of every outgoing velocity in every tile row (the WENO-5 face
// value at the wall from the three nearest fluid nodes and the two ghosts
// extrapolated from them), summed into the row's wall density n_w (Eq. nw); the
// two ghosts are stored.  Items start on thread `first` (a multiple of 32).  Each
// tile row of a wall takes a half-warp: lanes v = 0..9 compute the flux of
// outgoing velocity v (the half-range p_x < 0 at x = 0, p_x > 0 at x = nx ds),
// lanes 10..15 add 0, and a shuffle reduction over the half-warp gives the row's
// sum.
template <typename real, bool LEARNED, typename S>
__device__ __forceinline__ void wall_flux(S &sm, const Geo &g, const Tab<real> &t, const Tab<real> &tw, const float *mlp,
                                          int x0, int first, bool left_wall, bool right_wall)
{
    constexpr int HX = S::HX, TY = S::TY, NT = S::NT;
    const int tid = threadIdx.x;
    const int nflux = ((int)left_wall + (int)right_wall) * TY * 16;
    for (int f = (tid - first % NT + NT) % NT; f < nflux; f += NT) {
        // (wall, tile row tr, outgoing velocity v); the left wall's items first
        const int side = (f >= TY * 16 || !left_wall) ? 1 : 0;
        const int fr = f >= TY * 16 ? f - TY * 16 : f;
        const int tr = fr >> 4, v = fr & 15;
        const int k1 = side ? 3 + v / 5 : v / 5;
        const int k = NQ * k1 + v % 5;
        // nearest three fluid nodes, nearest first; ghost layers 0 and 1
        // are the next two columns outwards
        const int c0 = side ? g.nx - 1 - (x0 - 4) : 0 - (x0 - 4);
        const int dc = side ? -1 : 1;
        real wf = 0;
        if (v >= 10) {
            // idle lane of the row's half-warp
        } else if constexpr (sizeof(real) == 8) {
            const real a0 = *sm.at(k, tr + 3, c0), a1 = *sm.at(k, tr + 3, c0 + dc);
            const real a2 = *sm.at(k, tr + 3, c0 + 2 * dc);
            const real g0 = fma(real(3), a0 - a1, a2);
            const real g1 = fma(real(6), a0, fma(real(-8), a1, real(3) * a2));
            if (c0 - dc >= 0 && c0 - dc < HX) *sm.at(k, tr + 3, c0 - dc) = g0;
            if (c0 - 2 * dc >= 0 && c0 - 2 * dc < HX) *sm.at(k, tr + 3, c0 - 2 * dc) = g1;
            wf = t.R[k1] * face_value<LEARNED>(mlp, a2, a1, a0, g0, g1);
        } else {
            // pairs: the ghosts 3a0 - 3a1 + a2 and 6a0 - 8a1 + 3a2 as a0 plus
            // combinations of the differences D1 = a0 - a1, D2 = a1 - a2, and
            // the stencil (a2, a1, a0, g0, g1) by its first differences
            // (D2, D1, 2 D1 - D2, 3 D1 - 2 D2)
            const int row = tr + 3;
            const float h0 = *sm.at(k, row, c0), l0 = *sm.at(NK + k, row, c0);
            const float h1 = *sm.at(k, row, c0 + dc), l1 = *sm.at(NK + k, row, c0 + dc);
            const float h2 = *sm.at(k, row, c0 + 2 * dc), l2 = *sm.at(NK + k, row, c0 + 2 * dc);
            const float D1 = pdiff(h0, l0, h1, l1), D2 = pdiff(h1, l1, h2, l2);
            const float e0 = fmaf(2.0f, D1, -D2), e1 = fmaf(5.0f, D1, -3.0f * D2);
            const f2 G0 = f2_add_f(f2{h0, l0}, e0), G1 = f2_add_f(f2{h0, l0}, e1);
            if (c0 - dc >= 0 && c0 - dc < HX) {
                *sm.at(k, row, c0 - dc) = G0.hi;
                *sm.at(NK + k, row, c0 - dc) = G0.lo;
            }
            if (c0 - 2 * dc >= 0 && c0 - 2 * dc < HX) {
                *sm.at(k, row, c0 - 2 * dc) = G1.hi;
                *sm.at(NK + k, row, c0 - 2 * dc) = G1.lo;
            }
            const float corr = face_corr<LEARNED>(mlp, D2, D1, e0, fmaf(3.0f, D1, -2.0f * D2));
            wf = t.R[k1] * (h0 + (l0 + corr));
        }
        const unsigned half = (tid & 16) ? 0xffff0000u : 0x0000ffffu;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) wf += __shfl_xor_sync(half, wf, o);
        if (v == 0) sm.wnw[side][tr] = -wf * tw.inv_den[side];
    }
}

// The incoming ghosts of the tile rows at a wall, f^eq_w = n_w g g (Eq.
// diffuse_flux); items start on thread `first`.  top: the high word of the largest staged
// value, kept up to date, or nullptr.
template <typename real, typename S>
__device__ __forceinline__ void wall_ghosts(S &sm, const Geo &g, const Tab<real> &tw, int x0, int first, bool left_wall,
                                            bool right_wall, int *top = nullptr)
{
    constexpr int HX = S::HX, TY = S::TY, NT = S::NT;
    const int nin = ((int)left_wall + (int)right_wall) * TY * 30;
    for (int f = ((int)threadIdx.x - first % NT + NT) % NT; f < nin; f += NT) {
        // (wall, tile row tr, ghost layer m, incoming velocity v)
        const int side = (f >= TY * 30 || !left_wall) ? 1 : 0;
        const int fr = f >= TY * 30 ? f - TY * 30 : f;
        const int tr = fr / 30, m = (fr - 30 * tr) / 10, v = fr - 30 * tr - 10 * m;
        const int c = side ? g.nx + m - (x0 - 4) : -1 - m - (x0 - 4);
        if (c < 0 || c >= HX) continue;
        const int k = NQ * (side ? v / 5 : 3 + v / 5) + v % 5;
        const real ghost = sm.wnw[side][tr] * tw.geqw[side][k];
        *sm.at(k, tr + 3, c) = ghost;
        if constexpr (sizeof(real) == 8)
            if (top) atomicMax(top, finite_hi(abs_hi(ghost)));
        if constexpr (sizeof(real) == 4) *sm.at(NK + k, tr + 3, c) = 0.0f;
    }
}

}  // namespace olb
