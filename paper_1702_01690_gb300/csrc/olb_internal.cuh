// olb_internal.cuh -- types shared by the library's translation units.
//
// Device data layout (all arrays owned by the context):
//   populations  FP64: double f[25][ny][pitch]   kappa = 5*k1 + k2 (x-major
//                velocity index), pitch = nx rounded up to 32 elements so
//                every row starts on a 128/256-byte boundary
//                FP32: float f[2][25][ny][pitch], the value of population
//                kappa held as the unevaluated sum hi + lo of plane kappa
//                (hi, the value rounded to FP32) and plane 25 + kappa (lo,
//                the remainder rounded to FP32): compensated storage, so that
//                an RK increment far below FP32 resolution of f survives
//   status       int                     bit 0: invalid moment seen; bit 1: a
//                                        bounded wait for a TMA copy ran out
//   fields       moments and force of the nodes (StageFields in olb_fields.cuh, 56 or
//                48 bytes a node), for grids of more tiles than SMs
// The stage kernel keeps what else it needs of its tile (equilibrium factors, wall
// densities, flux differences) in shared memory.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

struct olb_params;

namespace olb {

constexpr int NQ = 5;   // Gauss-Hermite points per axis (Table trots)
constexpr int NK = 25;  // velocities

// Planes of one population buffer: 25 in FP64; 50 in FP32 (hi planes, then
// the lo planes of the compensated storage).
template <typename real>
constexpr int pop_planes()
{
    return sizeof(real) == 8 ? NK : 2 * NK;
}

// Geometry and physical parameters, passed by value to every kernel.
struct Geo {
    int nx, ny, pitch;
    int walls;           // 1: the x sides are not periodic (walls or specular)
    int wall_lo, wall_hi;  // diffuse wall at x = 0 / at x = nx ds (Sec. 3.4.2)
    int spec_lo, spec_hi;  // specular plane at x = 0 / at x = nx ds (Sec. 3.4.1)
    int spec_y;            // specular planes at y = 0 and y = ny ds
    long long plane;     // pitch * ny
    double ds, inv_ds, inv_ds3, dt, inv_tau, sigma, a, b;
};

// An unevaluated sum h + l of two floats (olb_ff.cuh).
struct ff {
    float h, l;
};

// The matrix D of the momentum derivative by parity, for FP64's stage kernel
// (dp_line in olb_stage64.cuh), and the constants of one of its RK-3 stages, as
// float-floats.
struct FfTab {
    ff E[3][2], O[2][3];
};
struct StageK {
    ff cit;     // c / tau, c the coefficient of dt L
    ff ca;      // the coefficient of f^n (cb = 1 - ca)
    ff kp, kn;  // c / (5040 ds), c sigma / (2160 ds^3) / 2^kn_exp (one over a density: beyond FP32's
    int kn_exp; // range in many units, so its binary exponent is kept beside it)
    ff adv[3];  // c |xi| / (6 ds), |xi| the roots 2, 3, 4
};
template <typename real>
struct TabFf {
};
template <>
struct TabFf<double> {
    FfTab ff;
};

// Velocity-space tables (Sec. 2.2, 2.3), in the population precision.
template <typename real>
struct Tab : TabFf<real> {
    real R[NQ];          // roots of He_5, ascending
    real R2[NQ];         // R^2
    real R2lo[NQ];       // R^2 - R2 (the remainder of R^2 in this precision; 0 in FP64)
    real D[NQ][NQ];      // (d_p f)_k = sum_k' D[k][k'] f_k'   (Eq. derf)
    real wHe[NQ][NQ];    // w_k He_l(p_k), l = 0..4            (Eq. g_alpha)
    real geqw[2][NK];    // g_{k1}(0, Tw) g_{k2}(uw, Tw) per wall
    real inv_den[2];     // 1 / sum_incoming g g p per wall    (Eq. nw)
};

// Host-side tables in FP64 (computed once from the closed forms).
struct HostTables {
    double R[NQ], W[NQ], D[NQ][NQ], wHe[NQ][NQ];
};
void host_tables(HostTables *t);
double host_g(const HostTables &t, int k, double u, double T);

template <typename real>
void fill_tab(Tab<real> *tab, const HostTables &h, const double Tw[2], const double uw[2]);
ff ff_of(double v);

// Parameter validation of olb_create (OLB_OK / OLB_ERR_ARG / OLB_ERR_CFL)
// and the mapping of CUDA errors to status codes (olb_api.cu).
int validate_params(const ::olb_params *p);
// Host fields [N] admissible as an initial state: n > 0, b n < 1, T > 0, all
// finite (olb_api.cu; large arrays are checked by several host threads).
bool fields_admissible(const double *n, const double *ux, const double *uy, const double *T, size_t N, double b);
void set_sides(Geo *g, const ::olb_params *p);
int cuda_status(cudaError_t e);

// TMA tensor maps (CUtensorMap, 128 bytes, 64-byte aligned) over one population
// buffer as a 3-D tensor [planes][ny][nx] with row stride pitch: a box of the rows
// of a tile, (pitch of a staged row) x TY x planes, and one of the three rows
// above or below its nodes, TX x 3 x planes.  The corners of the region, which no
// face reads, are left out (39 KB instead of 51 KB for an FP64 tile, and three
// CTAs on an SM instead of two).
struct alignas(64) TmaMap {
    unsigned char bytes[2][128];
};
// Kernel argument: the maps and whether to use them (tiles whose staged region
// lies inside the grid are loaded by TMA when on != 0).
struct alignas(64) TmaArg {
    TmaMap map;
    int on;
};
// Pitch (elements) of a staged row of a tile's region, TX + 8 nodes wide, with two
// (FP64) or four (FP32) more: the lines of the eight rows of a tile then start in
// different banks (rows of TX + 8 are whole multiples of the 32 banks or halves of
// it, and the lines of a warp would queue for one or two).
__host__ __device__ constexpr int region_pitch(int tx, bool fp64) { return tx + 8 + (fp64 ? 2 : 4); }
// Encode the maps of buffer `base` for tile shape tx x ty (olb_api.cu); false
// if the shape's rows are not a multiple of 16 bytes or the driver refuses.
bool tma_encode(TmaMap *out, const void *base, bool fp64, const Geo &g, int tx, int ty);

// All grids are advanced as tiles of 8 x 8 nodes, whatever shape was set (their flux
// differences and factors fit in shared memory beside the populations; larger shapes
// kept one velocity's faces at a time and recomputed per-node terms 25 times: FP32
// 4096^2 14 ms a stage with 32 x 16 against 8).
constexpr int STAGE_TX = 8, STAGE_TY = 8;
inline int stage_tiles(int nx, int ny) { return ((nx + STAGE_TX - 1) / STAGE_TX) * ((ny + STAGE_TY - 1) / STAGE_TY); }
// The compiled stage that advances so many tiles.  At most one tile an SM, 8: one launch of 512 threads a tile that take the moments and the
// force of the tile too (of its 14 x 14 nodes, three times the work of k_fields);
// else 5: three launches.  A stage, three launches and one, FP64: 8 tiles 27.3 and
// 15.2 us, 128 tiles 27.1 and 15.6, 256 tiles 32.6 and 30.3, 384 tiles 35.5 and 44.9,
// 4096 tiles 210 and 407; FP32: 13.9 and 7.4, 13.7 and 8.0, 15.8 and 15.1, 18.0 and
// 21.7, 93 and 188 (the lines cross between two and two and a half tiles an SM; the rule
// stops at one, up to which one launch is always the faster by far).  Learned weights: at
// most one tile an SM, 6 (512 threads a tile), else 4 (256, two tiles an SM): 39 tiles
// 70.8 (4) and 59.6 us (6) in FP64, 42.5 and 37.7 in FP32; 200 tiles 113 and 122, 68 and 72.
int stage_kind(bool learned, int tiles);

// Shapes that olb_set_tile accepts with learned weights.
inline bool learned_shape(int tx, int ty, int kp)
{
    return (tx == 8 && ty == 8 && kp == 4) || (tx == 16 && ty == 8 && kp == 2) || (tx == 32 && ty == 16 && kp == 1);
}

// RK-3 stage coefficients: out = ca f^n + cb f_s + cc L[f_s] (Eq. rk3).
struct StageCoef {
    double ca, cb, cc;
};
StageK stage_constants(const Geo &g, StageCoef c);

// Launchers, one set per precision (olb_fp64.cu, olb_fp32.cu).  Output
// pointers of launch_moments_out may be NULL to skip a field.  launch_fused
// runs the per-node moments pre-pass into fields (a buffer of fields_bytes(g)),
// then the stage kernel, which reads them.
#define OLB_DECLARE_LAUNCHERS(real)                                                                    \
    cudaError_t prepare_fused(real *, int tx, int ty, int kp, bool learned, int tiles);                \
    cudaError_t launch_fused(const real *fs, const real *fn, real *out, int *status, const Geo &g,     \
                             const Tab<real> &t, StageCoef c, const float *mlp,                        \
                             const TmaMap *tma, void *fields, cudaStream_t s);                         \
    cudaError_t launch_fused_batch(const real *fs, const real *fn, real *out, int *status,             \
                                   const void *runs, const int *tile_start, int nruns, int total,      \
                                   const Tab<real> &t, StageCoef c, int st, void *fields,              \
                                   const long long *node_start, long long total_nodes,                 \
                                   const int *force_start, int force_blocks,                           \
                                   const TmaMap *tmaps, cudaStream_t s);                               \
    size_t batch_run_bytes(real *);                                                                    \
    void batch_run_fill(real *, void *dst, const Geo &g, const Tab<real> &t, long long off,            \
                        long long foff, int ntx);                                                      \
    cudaError_t launch_init(real *f, const double *n, const double *ux, const double *uy,              \
                            const double *T, const Geo &g, const Tab<double> &t, cudaStream_t s);       \
    cudaError_t launch_moments_out(const real *f, double *n, double *ux, double *uy, double *T,        \
                                   const Geo &g, const Tab<double> &t, cudaStream_t s);                 \
    cudaError_t launch_to_f64(const real *f, double *dst, const Geo &g, cudaStream_t s);               \
    cudaError_t launch_from_f64(real *f, const double *src, const Geo &g, cudaStream_t s);             \
    cudaError_t launch_totals(const real *f, double *partial, double *out, const Geo &g,               \
                              const Tab<double> &t, cudaStream_t s);

OLB_DECLARE_LAUNCHERS(double)
OLB_DECLARE_LAUNCHERS(float)

// Bytes of the per-node fields of the stage (fields_of in olb_fields.cuh): 7
// (FP64) or 6 planes of pitch * ny 8-byte elements.
inline size_t fields_bytes(const Geo &g, bool fp64) { return (size_t)(fp64 ? 7 : 6) * g.plane * 8; }
// Blocks of the force kernel (32 x 8 nodes each) of a grid.
inline int force_blocks(const Geo &g) { return ((g.nx + 31) / 32) * ((g.ny + 7) / 8); }

// Global sums (olb_totals): fixed grid of the first reduction pass, whose
// per-block partial sums (4 each) the second pass adds in a fixed order.
constexpr int TOTALS_BLOCKS = 1024, TOTALS_THREADS = 256;

// Shapes that olb_set_tile accepts: TX x TY nodes and KP velocities at once
// (all are advanced as tiles of STAGE_TX x STAGE_TY).
constexpr int NUM_TILES = 8;
constexpr int TILE_X[NUM_TILES] = {8, 16, 16, 32, 32, 8, 7, 8};
constexpr int TILE_Y[NUM_TILES] = {8, 8, 8, 8, 16, 8, 8, 8};
constexpr int TILE_K[NUM_TILES] = {4, 2, 1, 1, 1, 8, 8, 5};

}  // namespace olb
