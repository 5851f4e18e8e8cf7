/* Kernels of the 1D compact GKS with GENO reconstruction (FP64 and mixed precision). */
#include "launch.cuh"
#include "step_1d.cuh"

namespace gks {
GKS_INSTANTIATE(1)

template <typename R, bool NS> static cudaError_t step1d(gks_ctx *c, const StepClock &first, const StepClock &last)
{
    const unsigned nb = blocks_for(c->kp.n[0], kCells1d);
    {
        ProfScope ps(c, GKS_KC_FACE);
        launch_chained(step1d_kernel<R, NS, 1>, nb, 32, c->stream, c->kp, c->W, c->G, c->W, c->G, c->Ws, c->Gs, c->Acc, c->status, first);
    }
    ProfScope ps(c, GKS_KC_FACE);
    launch_chained(step1d_kernel<R, NS, 2>, nb, 32, c->stream, c->kp, c->Ws, c->Gs, c->W, c->G, c->Ws, c->Gs, c->Acc, c->status, last);
    return cudaGetLastError();
}

template <bool NS> static cudaError_t step1d_short(gks_ctx *c, const StepClock &first, const StepClock &last)
{
    const unsigned nb = blocks_for(c->kp.n[0], kCellsShort);
    {
        ProfScope ps(c, GKS_KC_FACE);
        launch_chained(step1d_short_kernel<NS, 1>, nb, 128, c->stream, c->kp, c->W, c->G, c->W, c->G, c->Ws, c->Gs, c->Acc, c->status, first);
    }
    ProfScope ps(c, GKS_KC_FACE);
    launch_chained(step1d_short_kernel<NS, 2>, nb, 128, c->stream, c->kp, c->Ws, c->Gs, c->W, c->G, c->Ws, c->Gs, c->Acc, c->status, last);
    return cudaGetLastError();
}

cudaError_t launch_step1d(gks_ctx *c, const StepClock &first, const StepClock &last)
{
    const bool ns = c->kp.fp.mu > 0.0;
    if (!c->precision && short_1d(c->kp.n[0])) return ns ? step1d_short<true>(c, first, last) : step1d_short<false>(c, first, last);
    if (c->precision) return ns ? step1d<float, true>(c, first, last) : step1d<float, false>(c, first, last);
    return ns ? step1d<double, true>(c, first, last) : step1d<double, false>(c, first, last);
}
}
