/* Batched 2D mode: many independent grids of uneven sizes advanced by
 * kernels over tile work lists, one step captured in a CUDA graph.
 * Internal declarations (the C ABI is in include/genogks.h). */
#pragma once
#include "internal.h"

namespace gks {

/* per-grid device descriptor: parameters and buffer bases */
struct GridDesc {
    KP P;
    double *W, *G, *Ws, *Gs, *Acc;
    void *B, *ff;
    Shadow s0, s1; /* FP32 shadows (mixed precision only; Ws, Gs: FP64 only) */
};

/* a contiguous range of one kernel's index space on one grid, from item
 * `begin` for the class's tile size or to the end of the space */
struct Tile {
    unsigned grid_kind; /* 2 grid + face direction (flux; others 0) */
    unsigned begin;
};

/* BK_STAGE: the three stage kernels, of the mixed-precision batch, as one entry */
enum BatchKernel { BK_SPEED = 0, BK_POLY = 1, BK_FLUX = 2, BK_UPDATE = 3, BK_STAGE = 4, BK_COUNT = 5 };

struct LaunchShape {
    int block;   /* threads per block */
    long tile;   /* items per tile */
    int blocks;  /* grid size (wave speed: persistent blocks; stage kernels: one block per tile) */
};

struct BatchLaunch {
    const GridDesc *gd;         /* device */
    const Tile *tiles;
    int ntiles;
    double *dt;                 /* per grid: dt[2 g] the time step, dt[2 g + 1] = 1 / dt */
    float *updc;                /* per grid: the mixed update's stage constants (UpdC, 10 floats) */
    unsigned long long *smax;   /* per grid */
    int *status;                /* per grid: status[g] */
    const KP *common;           /* host: the scheme constants every grid shares */
};

template <typename R> cudaError_t batch_speed(const BatchLaunch &L, const LaunchShape &S, cudaStream_t st);
template <typename R> cudaError_t batch_poly(const BatchLaunch &L, const LaunchShape &S, int stage, cudaStream_t st);
template <typename R> cudaError_t batch_flux(const BatchLaunch &L, const LaunchShape &S, int stage, cudaStream_t st);
template <typename R> cudaError_t batch_update(const BatchLaunch &L, const LaunchShape &S, int stage, cudaStream_t st);
cudaError_t batch_dt(const GridDesc *gd, int nb, double cfl, const unsigned long long *smax, double *dt, float *updc,
                     cudaStream_t st);
cudaError_t batch_shadow(const GridDesc &g, cudaStream_t st);
/* FP64 gradients of grid g from its FP32 shadow (mixed precision) */
cudaError_t batch_widen_grad(const GridDesc &g, cudaStream_t st);
int batch_occupancy(int precision, int block);

} // namespace gks
