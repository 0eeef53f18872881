// olb_fused.cuh -- the stage kernels: one RK-3 stage of the off-lattice Boltzmann
// model for a grid (k_fused) or a batch of grids (k_fused_batch), and their
// launches.
//
// A stage is three launches (one on small grids, see stage_kind).  k_fields computes the moments n, u, T, Delta p of f_s
// once per node (Sec. 2.2, Eq. vdw), k_force the force F = grad(Delta p)/n + sigma
// grad(Laplacian n) from the 49-point stencils (Eqs. F_def, stencil_grad,
// stencil_glap; Sec. 3.4.3 at walls and mirror planes), both in olb_fields.cuh.
// Then one CTA per tile of 8 x 8 nodes (olb_stage64.cuh, olb_stage32.cuh, FP64 with
// learned weights olb_stage64l.cuh):
//   1. stages the populations of the tile and three nodes around it in shared
//      memory (olb_tile.cuh; TMA for tiles inside the grid);
//   2. forms the equilibrium factors of its nodes (Eqs. feq, g_alpha);
//   3. at walls (Sec. 3.4.2): extrapolated ghosts for the outgoing velocities, the
//      WENO flux of those velocities at the wall face, summed per tile row into n_w
//      (Eq. nw), and f^eq_w ghosts for the incoming velocities;
//   4. takes the WENO-5 fluxes (Eqs. weno5_*) along every row and column of the
//      tile, a line a thread, and from them the flux differences across its nodes;
//   5. adds advection, momentum derivative (Eq. derf), BGK and the RK-3
//      combination of Eq. rk3, and writes the output buffer.
#pragma once

#include "olb_fields.cuh"
#include "olb_stage32.cuh"
#include "olb_stage64.cuh"
#include "olb_stage64l.cuh"
#include "olb_tile.cuh"

namespace olb {

template <typename real, int KP, bool LEARNED>
struct StageSmem {
    using type = Smem32<KP, LEARNED>;
};
template <int KP>
struct StageSmem<double, KP, false> {
    using type = Smem64<KP>;
};
template <int KP>
struct StageSmem<double, KP, true> {
    using type = Smem64L<KP>;
};

// Shared memory of the single-grid kernel: the tile staging, then (learned
// weights only) the network's tables at a 16-byte aligned offset and, FP64, a
// scratch of each warp (olb_mlp.cuh).
template <typename real, int KP>
constexpr size_t mlp_offset()
{
    return (sizeof(typename StageSmem<real, KP, true>::type) + 15) / 16 * 16;
}
// KP 8: the CTA's own fields.
template <typename real>
constexpr size_t own_offset()
{
    return (sizeof(typename StageSmem<real, 8, false>::type) + 15) / 16 * 16;
}
template <typename real, int KP, bool LEARNED>
constexpr size_t fused_smem_bytes()
{
    using S = typename StageSmem<real, KP, LEARNED>::type;
    constexpr size_t mlp_floats = sizeof(real) == 4 ? MLP_T32_SIZE : MLP_T64_SIZE + S::NT / 32 * MLP_WARP_SCRATCH;
    return LEARNED   ? mlp_offset<real, KP>() + mlp_floats * sizeof(float)
           : KP == 8 ? own_offset<real>() + sizeof(TileFields<real>)
                     : sizeof(S);
}
template <typename real, int KP, bool LEARNED>
constexpr int stage_threads()
{
    return StageSmem<real, KP, LEARNED>::type::NT;
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

// Single grid: one CTA per tile.  Learned-weight instances leave their network the
// registers it needs: 512 threads per SM.
template <typename real, int KP, bool LEARNED>
__global__ void __launch_bounds__((stage_threads<real, KP, LEARNED>()),
                                  fused_min_ctas(fused_smem_bytes<real, KP, LEARNED>(),
                                                 stage_threads<real, KP, LEARNED>(),
                                                 KP == 4 ? 2 : KP == 5 ? 0 : 1))
k_fused(const real *__restrict__ fs, const real *fn, real *out, int *__restrict__ status,
        const __grid_constant__ Geo g, const __grid_constant__ Tab<real> t, real ca, real cb, real cc, real ca_lo,
        real cb_lo, const __grid_constant__ StageK sk, const float *__restrict__ mlp, const __grid_constant__ TmaArg tma,
        const __grid_constant__ StageFields<real> fields, int row0)
{
    // 128-byte aligned: the TMA copy of phase 1 lands at offset 0
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto &sm = *reinterpret_cast<typename StageSmem<real, KP, LEARNED>::type *>(smem_raw);
    MlpArg net = {nullptr, nullptr};
    if constexpr (LEARNED) {
        net = {mlp, reinterpret_cast<float *>(smem_raw + mlp_offset<real, KP>())};
        mlp_tables<real>(net.tables, mlp);  // made visible by the first barrier inside stage_tile
    }
    TileFields<real> *own = KP == 8 ? reinterpret_cast<TileFields<real> *>(smem_raw + own_offset<real>()) : nullptr;
    const TmaMap *tm = tma.on ? &tma.map : nullptr;
    const int x0 = blockIdx.x * 8;
    // (masked: not negative as the compiler sees it; 0.8 % of a stage of 2048^2 otherwise)
    const int y0 = (int)(((unsigned)row0 & 0x0fffffffu) + blockIdx.y) * 8;
    if constexpr (sizeof(real) == 8 && LEARNED)
        stage_tile64l<KP>(sm, fs, fn, out, status, g, t, x0, y0, ca, cb, cc, net, tm, fields);
    else if constexpr (sizeof(real) == 8)
        stage_tile64<KP>(sm, fs, fn, out, status, g, t, t, x0, y0, sk, tm, fields, own);
    else
        stage_tile32<KP, LEARNED>(sm, fs, fn, out, status, g, t, t, x0, y0, ca, cb, cc, ca_lo, cb_lo, net, tm, fields, own);
}

// Batch of independent runs (uneven grid sizes, own parameters): one CTA per
// (run, tile) work item, in the order of the items, so that the hardware
// dispatches neighbouring tiles together and their halos stay in L2 (a
// persistent grid-stride loop let the CTAs drift apart and measured slower);
// tile_start[r] is the first item of run r (prefix sum, tile_start[nruns] =
// total).  Each run has its populations at offset `off` of the three shared
// buffers and its own status word.
template <typename real, int KP>
__global__ void __launch_bounds__((stage_threads<real, KP, false>()),
                                  fused_min_ctas(fused_smem_bytes<real, KP, false>() + sizeof(BatchRun<real>),
                                                 stage_threads<real, KP, false>(), KP == 8 ? 1 : 0))
k_fused_batch(const real *__restrict__ fs, const real *fn, real *out, int *__restrict__ status,
              const BatchRun<real> *__restrict__ runs, const int *__restrict__ tile_start, int nruns,
              const __grid_constant__ Tab<real> tv, real ca, real cb, real ccoef, real ca_lo, real cb_lo, int st,
              char *fields, const TmaMap *__restrict__ tmaps)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    auto &sm = *reinterpret_cast<typename StageSmem<real, KP, false>::type *>(smem_raw);
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
    const int x0 = (lt % run.ntx) * 8, y0 = (lt / run.ntx) * 8;
    const StageFields<real> fl = fields_of<real>(fields + run.foff, run.g);
    // the run's tensor map of fs lives in global memory, written by the host
    // before the launch: acquire it for the tensormap proxy before the thread
    // that issues the copy uses it
    const TmaMap *tm = tmaps ? tmaps + lo : nullptr;
    if (tm && threadIdx.x == 0)
        for (int k = 0; k < 2; ++k)
            asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(tm->bytes[k]) : "memory");
    TileFields<real> *own = KP == 8 ? reinterpret_cast<TileFields<real> *>(smem_raw + own_offset<real>()) : nullptr;
    if constexpr (sizeof(real) == 8)
        stage_tile64<KP>(sm, fs + run.off, fn + run.off, out + run.off, status + lo, run.g, tv, run.t, x0, y0,
                                run.k[st], tm, fl, own);
    else
        stage_tile32<KP, false>(sm, fs + run.off, fn + run.off, out + run.off, status + lo, run.g, tv, run.t, x0, y0, ca, cb,
                            ccoef * (real)run.g.dt, ca_lo, cb_lo, MlpArg{}, tm, fl, own);
}

template <typename real, int KP, bool LEARNED = false>
cudaError_t fused_prepare_one()
{
    cudaError_t e = cudaFuncSetAttribute(k_fused<real, KP, LEARNED>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)fused_smem_bytes<real, KP, LEARNED>());
    if constexpr (!LEARNED)
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_fused_batch<real, KP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)fused_smem_bytes<real, KP, false>());
    return e;
}

// A launch has at most 65535 blocks along y: launch(first row of blocks, rows) for each
// so many.
template <typename Launch>
void for_rows(int rows, Launch launch)
{
    for (int row0 = 0; row0 < rows; row0 += 65535) launch(row0, rows - row0 < 65535 ? rows - row0 : 65535);
}

template <typename real, int KP, bool LEARNED = false>
cudaError_t fused_launch_one(const real *fs, const real *fn, real *out, int *status, const Geo &g,
                             const Tab<real> &t, StageCoef c, const float *mlp, const TmaMap *tmap, void *fields,
                             cudaStream_t s)
{
    TmaArg tma{};
    if (tmap) {
        tma.map = *tmap;
        tma.on = 1;
    }
    // the moments of fs first (one thread per node) and the force, then the stage
    const StageFields<real> fl = fields_of<real>(fields, g);
    const StageK sk = sizeof(real) == 8 ? stage_constants(g, c) : StageK{};
    if (KP != 8) {
        const long long N = (long long)g.nx * g.ny;
        constexpr bool SEQ = LEARNED && sizeof(real) == 8;
        k_fields<real, SEQ><<<(unsigned)((N + 255) / 256), 256, 0, s>>>(fs, fl, status, g, t);
        for_rows((g.ny + FORCE_Y - 1) / FORCE_Y, [&](int row0, int rows) {
            const dim3 blocks((g.nx + FORCE_X - 1) / FORCE_X, rows);
            if constexpr (SEQ) k_force_learned<real><<<blocks, 2 * FORCE_THREADS, 0, s>>>(fl, g, c.cc, row0);
            else k_force<real><<<blocks, ForceOf<real>::NT, 0, s>>>(fl, g, sk, (real)c.cc, row0);
        });
    }
    for_rows((g.ny + 7) / 8, [&](int row0, int rows) {
        k_fused<real, KP, LEARNED><<<dim3((g.nx + 7) / 8, rows), stage_threads<real, KP, LEARNED>(),
                                     fused_smem_bytes<real, KP, LEARNED>(), s>>>(
            fs, fn, out, status, g, t, (real)c.ca, (real)c.cb, (real)c.cc, (real)(c.ca - (double)(real)c.ca),
            (real)(c.cb - (double)(real)c.cb), sk, mlp, tma, fl, row0);
    });
    return cudaGetLastError();
}

template <typename real, int KP>
cudaError_t fused_batch_launch_one(const real *fs, const real *fn, real *out, int *status, const void *runs,
                                   const int *tile_start, int nruns, int total, const Tab<real> &t, StageCoef c,
                                   int st, void *fields, const long long *node_start, long long total_nodes,
                                   const int *force_start, int force_blocks, const TmaMap *tmaps, cudaStream_t s)
{
    if (total < 1) return cudaSuccess;
    if (KP != 8 && total_nodes > 0) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const long long want = (total_nodes + 255) / 256, cap = 8LL * sms * 8;
        k_fields_batch<real><<<(unsigned)(want < cap ? want : cap), 256, 0, s>>>(
            fs, static_cast<char *>(fields), static_cast<const BatchRun<real> *>(runs), node_start, nruns, total_nodes,
            status);
    }
    if (KP != 8)
        k_force_batch<real><<<force_blocks, ForceOf<real>::NT, 0, s>>>(
            static_cast<char *>(fields), static_cast<const BatchRun<real> *>(runs), force_start, nruns, st, (real)c.cc);
    k_fused_batch<real, KP><<<total, stage_threads<real, KP, false>(), fused_smem_bytes<real, KP, false>(), s>>>(
        fs, fn, out, status, static_cast<const BatchRun<real> *>(runs), tile_start, nruns, t, (real)c.ca, (real)c.cb,
        (real)c.cc, (real)(c.ca - (double)(real)c.ca), (real)(c.cb - (double)(real)c.cb), st, static_cast<char *>(fields),
        tmaps);
    return cudaGetLastError();
}

// Compiled instances (stage_kind): KP 8 and 5, 6 and 4 with learned weights.
#define OLB_DEFINE_FUSED(real)                                                                                \
    cudaError_t prepare_fused(real *, int tx, int ty, int kp, bool learned, int tiles)                        \
    {                                                                                                         \
        if (learned && !learned_shape(tx, ty, kp)) return cudaErrorInvalidValue;                              \
        const int kind = stage_kind(learned, tiles);                                                          \
        return kind == 4   ? fused_prepare_one<real, 4, true>()                                               \
               : kind == 6 ? fused_prepare_one<real, 6, true>()                                               \
               : kind == 8 ? fused_prepare_one<real, 8>()                                                     \
                           : fused_prepare_one<real, 5>();                                                    \
    }                                                                                                         \
    cudaError_t launch_fused(const real *fs, const real *fn, real *out, int *status, const Geo &g,            \
                             const Tab<real> &t, StageCoef c, const float *mlp, const TmaMap *tma,            \
                             void *fields, cudaStream_t s)                                                    \
    {                                                                                                         \
        const int kind = stage_kind(mlp != nullptr, stage_tiles(g.nx, g.ny));                                 \
        if (kind == 4) return fused_launch_one<real, 4, true>(fs, fn, out, status, g, t, c, mlp, tma, fields, s); \
        if (kind == 6) return fused_launch_one<real, 6, true>(fs, fn, out, status, g, t, c, mlp, tma, fields, s); \
        return kind == 8 ? fused_launch_one<real, 8>(fs, fn, out, status, g, t, c, nullptr, tma, fields, s)   \
                         : fused_launch_one<real, 5>(fs, fn, out, status, g, t, c, nullptr, tma, fields, s);  \
    }                                                                                                         \
    cudaError_t launch_fused_batch(const real *fs, const real *fn, real *out, int *status, const void *runs,  \
                                   const int *tile_start, int nruns, int total, const Tab<real> &t,           \
                                   StageCoef c, int st, void *fields, const long long *node_start,            \
                                   long long total_nodes, const int *force_start, int force_blocks,           \
                                   const TmaMap *tmaps, cudaStream_t s)                                       \
    {                                                                                                         \
        const auto go = stage_kind(false, total) == 8 ? fused_batch_launch_one<real, 8> : fused_batch_launch_one<real, 5>; \
        return go(fs, fn, out, status, runs, tile_start, nruns, total, t, c, st, fields, node_start, total_nodes, \
                  force_start, force_blocks, tmaps, s);                                                       \
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
