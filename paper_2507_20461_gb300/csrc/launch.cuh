/* Launch wrappers of the stage kernels for one dimension M; included by the
 * per-dimension translation units k1d.cu, k2d.cu, k3d.cu. */
#pragma once
#include "internal.h"
#include "step_flux.cuh"

namespace gks {

template <typename R> Src<R> stage_src(gks_ctx *c, int input);
template <> inline Src<double> stage_src<double>(gks_ctx *c, int input)
{
    return input ? Src<double>{c->Ws, c->Gs} : Src<double>{c->W, c->G};
}
template <> inline Src<float> stage_src<float>(gks_ctx *c, int input)
{
    const Shadow &s = input ? c->s1 : c->s0;
    return Src<float>{s.hi, s.lo, s.g};
}

inline int sm_count()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return n;
}
/* Small grids, as blocks per SM: a thread per (cell, variable) in the
 * reconstruction, a lane per Gauss point in the flux.  With too few blocks to
 * hide a thread's chain of instructions the work of one is spread over several;
 * past the lines below the repeated index work and evaluations cost more.  The
 * FP64 reconstruction is always spread: its index work runs beside the FP64 pipe.
 * Measured (GB300, us a step, plain / spread, then plain / split):
 *   FP32 2D: 160^2 (1.4 recon, 5.3 flux blocks per SM) 44.9 / 40.5, 44.9 / 37.2;
 *     224^2 (2.6, 10.4) 47.7 / 45.1, 47.7 / 44.9; 320^2 (5.3, 21) 63.9 / 60.3, 63.7 / 65.1;
 *     448^2 (10.4, 41) 97.9 / 98.4, equal;
 *   FP32 3D: 26^3 (1.1, 5.6) 88 / 71, 88 / 68; 32^3 (2.0, 10.4) 97 / 93, 97 / 90;
 *     40 x 36^2 (3.1, 16) 117.6 / 117.1, 117.3 / 115.1; 48 x 40^2 (4.5, 24) 139 / 151, 139 / 152;
 *   FP64 2D: 160^2 565 / 454, 565 / 590; 3D: 20^3 (0.6, 2.6) 986 / 669, 986 / 707;
 *     26^3 1360 / 1110, 1360 / 1507; 64 x 50^2 (9.2, 50) 8451 / 8354; 512^2 (13.6) 3210 / 3148. */
template <typename R, int M> inline bool spread_cells(unsigned blocks)
{
    if constexpr (sizeof(R) == sizeof(double)) return true;
    else return blocks <= (unsigned)((M == 2 ? 6 : 3) * sm_count());
}
template <typename R> inline bool split_faces(unsigned blocks) { return blocks <= (unsigned)((sizeof(R) == sizeof(double) ? 3 : 12) * sm_count()); }

/* interface states into fs_dev */
template <typename R, int M> static cudaError_t states_impl(gks_ctx *c, int input, double *fs_dev)
{
    const KP &P = c->kp;
    if constexpr (M == 1) {
        if (c->order != 8) return nc_launch_faces(c, input, fs_dev, false);
        ProfScope ps(c, GKS_KC_FACE);
        face1d_kernel<R, false><<<blocks_for(P.n[0] + 1, 32), 32, 0, c->stream>>>(P, input ? c->Ws : c->W, input ? c->Gs : c->G, c->dt, fs_dev, nullptr, c->status);
    } else {
        constexpr int NG = (M == 2) ? 2 : 4;
        R *B = (R *)c->B;
        const Src<R> src = stage_src<R>(c, input);
        {
            ProfScope ps(c, GKS_KC_RECON);
            cell_poly_kernel<R, M><<<blocks_for(P.next), kBlock, 0, c->stream>>>(P, src, B);
        }
        for (int d = 0; d < M; ++d) {
            const unsigned nb = blocks_for(P.nface[d] * NG);
            ProfScope ps(c, GKS_KC_FACE);
#define GKS_FACE(D)                                                                                           \
    if (d == D) {                                                                                             \
        face_flux_prepare<R, M, D, false>();                                                                  \
        face_flux_kernel<R, M, D, false><<<nb, kBlock, 0, c->stream>>>(P, src, B, c->dt, fs_dev, nullptr, c->status); \
    }
            GKS_FACE(0)
            GKS_FACE(1)
            if constexpr (M == 3) { GKS_FACE(2) }
#undef GKS_FACE
        }
    }
    return cudaGetLastError();
}

template <typename R, int M, bool NS, bool SPLIT, bool POINTS> static cudaError_t face_flux_launch(gks_ctx *c, int input)
{
    const KP &P = c->kp;
    constexpr int BT = kStepFluxBlock, FB = SPLIT ? BT / (M == 3 ? 4 : 2) : BT;
    static const bool prep = SPLIT || (smem_carveout_for(step_flux_kernel<R, M, NS, SPLIT, POINTS>, kStepFluxMinBlocks<R, M, NS>), true);
    (void)prep;
    unsigned nb[3], total = 0, runs = M == 2 ? ~0u : 0u;
    for (int d = 0; d < M; ++d) {
        nb[d] = blocks_for(P.nface[d], FB);
        total += nb[d];
        if (nb[d] / kFaceRun < runs) runs = nb[d] / kFaceRun;
    }
    const FaceOrder order{runs, {nb[0] - runs * kFaceRun, nb[1] - runs * kFaceRun}};
    ProfScope ps(c, GKS_KC_FACE);
    launch_chained(step_flux_kernel<R, M, NS, SPLIT, POINTS>, total, BT, c->stream, P, (const R *)c->B, c->dt, (R *)c->ff, c->status, order, input == 0);
    return cudaGetLastError();
}

/* reconstruction and face fluxes (step_flux.cuh): summed over the Gauss points
 * (the step), or per point (gks_flux) */
template <typename R, int M, bool NS, bool POINTS> static cudaError_t flux_impl(gks_ctx *c, int input)
{
    const KP &P = c->kp;
    R *B = (R *)c->B;
    {
        ProfScope ps(c, GKS_KC_RECON);
        const unsigned nb = blocks_for(P.next);
        if (spread_cells<R, M>(nb))
            launch_chained(cell_poly_kernel<R, M, true, true>, dim3(nb, M + 2), kBlock, c->stream, P, stage_src<R>(c, input), B, input != 0);
        else if constexpr (sizeof(R) == sizeof(float))
            launch_chained(cell_poly_kernel<R, M, true>, nb, kBlock, c->stream, P, stage_src<R>(c, input), B, input != 0);
    }
    return split_faces<R>(blocks_for(P.nftot, kStepFluxBlock)) ? face_flux_launch<R, M, NS, true, POINTS>(c, input)
                                                            : face_flux_launch<R, M, NS, false, POINTS>(c, input);
}

template <int M> cudaError_t launch_states(gks_ctx *c, int input, double *fs_dev)
{
    return c->precision ? states_impl<float, M>(c, input, fs_dev) : states_impl<double, M>(c, input, fs_dev);
}

template <typename R, int M> static cudaError_t flux_of(gks_ctx *c, int input, bool sums)
{
    const KP &P = c->kp;
    const bool ns = P.fp.mu > 0.0;
    if constexpr (M == 1) {
        if (c->order != 8) return nc_launch_faces(c, input, nullptr, true);
        const unsigned nb = blocks_for(P.n[0] + 1, 32);
        const double *W = input ? c->Ws : c->W, *G = input ? c->Gs : c->G;
        ProfScope ps(c, GKS_KC_FACE);
        if (ns) face1d_kernel<R, true, true><<<nb, 32, 0, c->stream>>>(P, W, G, c->dt, nullptr, (R *)c->ff, c->status);
        else face1d_kernel<R, true><<<nb, 32, 0, c->stream>>>(P, W, G, c->dt, nullptr, (R *)c->ff, c->status);
        return cudaGetLastError();
    } else {
        if (sums) return ns ? flux_impl<R, M, true, false>(c, input) : flux_impl<R, M, false, false>(c, input);
        return ns ? flux_impl<R, M, true, true>(c, input) : flux_impl<R, M, false, true>(c, input);
    }
}

template <int M> cudaError_t launch_flux(gks_ctx *c, int input, bool sums)
{
    return c->precision ? flux_of<float, M>(c, input, sums) : flux_of<double, M>(c, input, sums);
}

template <typename R, int M, int STAGE, bool SPEED> static void update_launch(gks_ctx *c, unsigned long long *smax)
{
    launch_chained(step_update_kernel<R, M, STAGE, SPEED>, blocks_for(c->kp.ncell, 256), 256, c->stream, c->kp, (const R *)c->ff, c->dt, c->W, c->G, c->Ws, c->Gs, c->Acc, c->s0, c->s1, c->status, c->updc, smax, STAGE == 2);
}

template <typename R, int M> static cudaError_t update_impl(gks_ctx *c, int stage, unsigned long long *smax)
{
    ProfScope ps(c, GKS_KC_UPDATE);
    if (stage == 1) update_launch<R, M, 1, false>(c, nullptr);
    else if (smax) update_launch<R, M, 2, true>(c, smax);
    else update_launch<R, M, 2, false>(c, nullptr);
    return cudaGetLastError();
}

template <int M> cudaError_t launch_update(gks_ctx *c, int stage, unsigned long long *smax)
{
    if constexpr (M == 1) return cudaErrorInvalidValue; /* the 1D stages update in the kernel that evaluates the fluxes */
    else return c->precision ? update_impl<float, M>(c, stage, smax) : update_impl<double, M>(c, stage, smax);
}

template <int M> cudaError_t launch_wavespeed(gks_ctx *c)
{
    cudaError_t e = cudaMemsetAsync(c->smax, 0, 2 * sizeof(unsigned long long), c->stream);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    long want = (c->kp.ncell + 255) / 256;
    long cap = (long)nsm * 8;
    const unsigned nb = (unsigned)(want < cap ? (want > 0 ? want : 1) : cap);
    ProfScope ps(c, GKS_KC_DT);
    if (c->shadows) wavespeed_kernel<M, float><<<nb, 256, 0, c->stream>>>(c->kp, c->s0.hi, c->smax);
    else wavespeed_kernel<M, double><<<nb, 256, 0, c->stream>>>(c->kp, c->W, c->smax);
    return cudaGetLastError();
}

/* the time step of wave speed slot in; clears the slot that the step's last stage adds to */
template <int M> cudaError_t launch_dt(gks_ctx *c, double cfl, const unsigned long long *in, unsigned long long *clear)
{
    /* viscous limit cfl h^2 / (2 (m - 1) nu): passed as the factor
     * 2 (m - 1) mu / h that turns max(1 / rho) into the rate cfl h / dt */
    const double visc = c->kp.fp.mu > 0.0 ? 2.0 * (M > 1 ? M - 1 : 1) * c->kp.fp.mu / c->h : 0.0;
    ProfScope ps(c, GKS_KC_DT);
    launch_chained(dt_from_speed_kernel, 1, 1, c->stream, in, cfl * c->h, visc, c->dt, c->shadows ? c->updc : nullptr,
                                                 updc_cw(c->kp, M), clear);
    return cudaGetLastError();
}

template <int M> cudaError_t launch_shadow(gks_ctx *c)
{
    if (!c->shadows) return cudaSuccess;
    const long want = (c->kp.ncell + 255) / 256;
    shadow_kernel<M><<<(unsigned)(want < 4096 ? (want > 0 ? want : 1) : 4096), 256, 0, c->stream>>>(c->kp, c->W, c->G,
                                                                                                   c->s0);
    return cudaGetLastError();
}

#define GKS_INSTANTIATE(M)                                                                                \
    template cudaError_t launch_states<M>(gks_ctx *, int, double *);                                      \
    template cudaError_t launch_flux<M>(gks_ctx *, int, bool);                                            \
    template cudaError_t launch_update<M>(gks_ctx *, int, unsigned long long *);                          \
    template cudaError_t launch_wavespeed<M>(gks_ctx *);                                                  \
    template cudaError_t launch_dt<M>(gks_ctx *, double, const unsigned long long *, unsigned long long *); \
    template cudaError_t launch_shadow<M>(gks_ctx *);

} // namespace gks
