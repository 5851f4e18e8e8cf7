/* Batched kernels of the 2D compact GKS over tile lists spanning every grid:
 * a block of a stage kernel takes one tile, a thread one item.  The per-item
 * arithmetic is the single-grid step path's (kernels.cuh,
 * step_flux.cuh), so a grid of a batch and the same grid alone run the same
 * formulas.  Mixed precision ran each stage as one fused kernel sweeping
 * strips through shared memory before the face flux took a thread per face;
 * with that flux in both, 2 steps of 1.8 M cells in 12 grids, states copied in
 * and out, take 2.96 ms against the sweep's 3.63 ms (registers and the
 * sweep's barriers held it at 16 warps per SM); the FP64 batch of 6 grids 4.67
 * ms against 5.54 ms with its tile loops over the per-point flux.  With chained
 * launches, the alternating block order and states in and out by one kernel
 * 2.37 ms and 3.49 ms.
 */
#include "batch.h"
#include "step_flux.cuh"

namespace gks {

template <typename R> __device__ __forceinline__ Src<R> stage_src_of(const GridDesc &g, int stage);
template <> __device__ __forceinline__ Src<double> stage_src_of<double>(const GridDesc &g, int stage)
{
    return stage == 1 ? Src<double>{g.W, g.G} : Src<double>{g.Ws, g.Gs};
}
template <> __device__ __forceinline__ Src<float> stage_src_of<float>(const GridDesc &g, int stage)
{
    const Shadow &s = stage == 1 ? g.s0 : g.s1;
    return Src<float>{s.hi, s.lo, s.g};
}

template <typename R>
__global__ void __launch_bounds__(256) bk_speed(const GridDesc *__restrict__ gd, const Tile *__restrict__ tiles, int ntiles,
                                                long tile, unsigned long long *__restrict__ smax)
{
    __shared__ double red[8];
    for (int ti = blockIdx.x; ti < ntiles; ti += gridDim.x) {
        const Tile T = tiles[ti];
        const unsigned grid = T.grid_kind >> 1;
        const KP &P = gd[grid].P;
        const long end = T.begin + tile < P.ncell ? T.begin + tile : P.ncell;
        /* the FP64 state, or its FP32 shadow in mixed precision */
        const R *W;
        if constexpr (sizeof(R) == sizeof(float)) W = gd[grid].s0.hi;
        else W = gd[grid].W;
        const R gam = R(P.gamma);
        R sr = R(0);
        for (long c = T.begin + threadIdx.x; c < end; c += blockDim.x) {
            const R rho = W[c];
            const R u = W[P.ncell + c] / rho, v = W[2 * P.ncell + c] / rho;
            const R p = (gam - R(1)) * (W[3 * P.ncell + c] - R(0.5) * rho * (u * u + v * v));
            sr = fmax(sr, fmax(fabs(u), fabs(v)) + sqrt(gam * p / rho));
        }
        double s = (double)sr;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double m = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, red[w]);
            atomicMax(&smax[grid], (unsigned long long)__double_as_longlong(isnan(m) ? 1e300 : m));
        }
        __syncthreads();
    }
}

__global__ void bk_dt(const GridDesc *__restrict__ gd, int nb, double cfl, const unsigned long long *__restrict__ smax,
                      double *__restrict__ dt, float *__restrict__ updc)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const KP &P = gd[b].P;
    const double d = cfl * P.h / __longlong_as_double((long long)smax[b]);
    dt[2 * b] = d;
    dt[2 * b + 1] = 1.0 / d;
    if (updc) store_updc(updc + 10 * b, make_updc(d, updc_cw(P, 2)));
}

/* The parameter block of one grid: the scheme constants and boundary types,
 * which the grids of a batch share, from the launch parameter (constant
 * bank), the geometry from the grid's descriptor. */
__device__ __forceinline__ KP grid_kp(const KP &common, const KP &g)
{
    KP P = common;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        P.n[a] = g.n[a];
        P.nface[a] = g.nface[a];
        P.foff[a] = g.foff[a];
        P.ext[a] = g.ext[a];
        P.dn[a] = g.dn[a];
        P.dface[a][0] = g.dface[a][0];
        P.dface[a][1] = g.dface[a][1];
    }
    P.ncell = g.ncell;
    P.nftot = g.nftot;
    P.next = g.next;
    P.h = g.h;
    P.ih = g.ih;
    P.fh = g.fh;
    P.fih = g.fih;
    P.dext[0] = g.dext[0];
    P.dext[1] = g.dext[1];
    return P;
}

/* One block per tile, one item per thread: no loop whose invariants (the
 * grid's geometry, the addresses) would be held in registers across items. */
template <typename R>
__global__ void __launch_bounds__(128) bk_poly(const KP common, const GridDesc *__restrict__ gd,
                                               const Tile *__restrict__ tiles, int stage)
{
    after_previous();
    const Tile T = tiles[block_in_order(stage == 2)];
    const GridDesc &g = gd[T.grid_kind >> 1];
    const KP P = grid_kp(common, g.P);
    const unsigned t = T.begin + threadIdx.x;
    /* FP64: a thread per variable too (spread_cells) */
    if (t < P.next)
        cell_poly_item<R, 2, true, sizeof(R) == sizeof(double)>(P, stage_src_of<R>(g, stage), (R *)g.B, t, (int)blockIdx.y);
}

/* block size and register cap of the single-grid face flux; FP32 spills 124 / 132
 * bytes at it (the single grid 16 / 16), most likely for the grid's parameters, which
 * are registers here and the constant bank there */
template <typename R>
__global__ void __launch_bounds__(kStepFluxBlock, (kStepFluxMinBlocks<R, 2, false>))
    bk_flux(const KP common, const GridDesc *__restrict__ gd, const Tile *__restrict__ tiles,
            const double *dt, int *status, bool rev)
{
    after_previous();
    __shared__ typename FaceV<R>::V slots[kFaceStash<R, 2> * kStepFluxBlock];
    typename FaceV<R>::V *stash = slots + threadIdx.x;
    const Tile T = tiles[block_in_order(rev)];
    const unsigned grid = T.grid_kind >> 1;
    const GridDesc &g = gd[grid];
    const KP P = grid_kp(common, g.P);
    const R d = R(dt[2 * grid]), id = R(dt[2 * grid + 1]);
    const unsigned fl = T.begin + threadIdx.x;
    if (T.grid_kind & 1u) {
        if (fl < P.nface[1])
            step_face_item<R, 2, 1, false, kStepFluxBlock>(P, (const R *)g.B, d, id, (R *)g.ff, status + grid, fl, stash);
    } else {
        if (fl < P.nface[0])
            step_face_item<R, 2, 0, false, kStepFluxBlock>(P, (const R *)g.B, d, id, (R *)g.ff, status + grid, fl, stash);
    }
}

template <typename R, int STAGE>
__global__ void __launch_bounds__(128) bk_update(const KP common, const GridDesc *__restrict__ gd,
                                                 const Tile *__restrict__ tiles, const double *dt,
                                                 const float *updc, int *status)
{
    after_previous();
    const Tile T = tiles[block_in_order(STAGE == 2)];
    const unsigned grid = T.grid_kind >> 1;
    const GridDesc &g = gd[grid];
    const KP P = grid_kp(common, g.P);
    UpdC uc;
    if constexpr (sizeof(R) == sizeof(float)) uc = load_updc(updc + 10 * grid);
    const unsigned c = T.begin + threadIdx.x;
    R wn[4];
    if (c < P.ncell)
        step_update_item<R, 2, STAGE>(P, (const R *)g.ff, dt[2 * grid], g.W, g.G, g.Ws, g.Gs, g.Acc, g.s0, g.s1,
                                      status + grid, c, uc, wn);
}

template <typename R> cudaError_t batch_speed(const BatchLaunch &L, const LaunchShape &S, cudaStream_t st)
{
    bk_speed<R><<<S.blocks, S.block, 0, st>>>(L.gd, L.tiles, L.ntiles, S.tile, L.smax);
    return cudaGetLastError();
}
template <typename R> cudaError_t batch_poly(const BatchLaunch &L, const LaunchShape &S, int stage, cudaStream_t st)
{
    return launch_chained(bk_poly<R>, dim3(S.blocks, sizeof(R) == sizeof(double) ? 4 : 1), S.block, st, *L.common, L.gd, L.tiles, stage);
}
template <typename R> cudaError_t batch_flux(const BatchLaunch &L, const LaunchShape &S, int stage, cudaStream_t st)
{
    if (S.block != kStepFluxBlock) return cudaErrorInvalidConfiguration;
    static const bool prep = (smem_carveout_for(bk_flux<R>, kStepFluxMinBlocks<R, 2, false>), true);
    (void)prep;
    return launch_chained(bk_flux<R>, S.blocks, S.block, st, *L.common, L.gd, L.tiles, L.dt, L.status, stage == 1);
}
template <typename R> cudaError_t batch_update(const BatchLaunch &L, const LaunchShape &S, int stage, cudaStream_t st)
{
    return launch_chained(stage == 1 ? bk_update<R, 1> : bk_update<R, 2>, S.blocks, S.block, st, *L.common, L.gd, L.tiles, L.dt, L.updc,
                          L.status);
}
cudaError_t batch_shadow(const GridDesc &g, cudaStream_t st)
{
    const long want = (g.P.ncell + 255) / 256;
    shadow_kernel<2><<<(unsigned)(want < 4096 ? (want > 0 ? want : 1) : 4096), 256, 0, st>>>(g.P, g.W, g.G, g.s0);
    return cudaGetLastError();
}

cudaError_t batch_widen_grad(const GridDesc &g, cudaStream_t st)
{
    const long n = 2L * 4 * g.P.ncell;
    const long want = (n + 255) / 256;
    widen_grad_kernel<<<(unsigned)(want < 4096 ? (want > 0 ? want : 1) : 4096), 256, 0, st>>>(g.s0.g, g.G, n);
    return cudaGetLastError();
}

cudaError_t batch_dt(const GridDesc *gd, int nb, double cfl, const unsigned long long *smax, double *dt, float *updc,
                     cudaStream_t st)
{
    bk_dt<<<(nb + 127) / 128, 128, 0, st>>>(gd, nb, cfl, smax, dt, updc);
    return cudaGetLastError();
}

/* resident blocks per SM of the wave-speed kernel at a block size */
int batch_occupancy(int precision, int block)
{
    int n = 0;
    if (precision) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, bk_speed<float>, block, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, bk_speed<double>, block, 0);
    return n;
}

#define GKS_BATCH_INST(R)                                                                             \
    template cudaError_t batch_speed<R>(const BatchLaunch &, const LaunchShape &, cudaStream_t);       \
    template cudaError_t batch_poly<R>(const BatchLaunch &, const LaunchShape &, int, cudaStream_t);   \
    template cudaError_t batch_flux<R>(const BatchLaunch &, const LaunchShape &, int, cudaStream_t);   \
    template cudaError_t batch_update<R>(const BatchLaunch &, const LaunchShape &, int, cudaStream_t);
GKS_BATCH_INST(float)
GKS_BATCH_INST(double)

} // namespace gks
