/* 1D non-compact GENO schemes (Sec. 4.1): 5th order (the 5th-order WENO
 * stencils) and 6th order (six-cell stencil symmetric about the face), with
 * the HLLC flux and classical four-stage RK4 (Sec. 2).  FP64.
 *
 * Face f (0..n) lies between cells f-1 and f.  The left state is
 * reconstructed in cell f-1 from the averages at offsets -2..3; the right
 * state in cell f from the mirrored stencil, so both use the same map
 * (nc5_left / nc6_left, generated in exact arithmetic).
 *
 * The kernels are bound by the FP64 pipe (two lanes per SM and clock), so they
 * are arranged for few FP64 instructions: the maps take averages relative to
 * the cell, the resolved parts skip the weights (chi_is_one), the low-order
 * weights share one division, and a stage's fluxes and RK update are one
 * kernel (step_1d.cuh: a warp's faces and the cells between them).
 * GB300, one RK4 step of 10^6 cells, order 6: 10.6 to 4.5 ms. */
#include "internal.h"
#include "step_1d.cuh"

namespace gks {

namespace {

/* GENO blend of the left value from averages relative to the reconstruction
 * cell (u[2] = 0): chi qH + (1 - chi) sum_k omega_k p_k, with IS^H = max,
 * IS^L = min, IS^tau = |(IS_first + IS_last)/2 - IS_2|, r = 2, and d = C0 on the
 * sub-stencil centred on the cell (index 1). */
template <int ORDER>
__device__ __forceinline__ double nc_value(const KP &P, const double *u)
{
    constexpr int K = (ORDER == 5) ? 3 : 4;
    double qH, p[K], IS[K];
    if constexpr (ORDER == 5) nc5_left<double>(u, qH, p, IS);
    else nc6_left<double>(u, qH, p, IS);
    if (P.limiter == 1) return qH;
    double ISL = IS[0];
#pragma unroll
    for (int k = 1; k < K; ++k) ISL = fmin(ISL, IS[k]);
    /* outer-left, outer-right and centred sub-stencils (6th order: S_1, S_4,
     * S_2; S_1..S_3 would never see the stencil's last cell) */
    const double ISt = fabs(0.5 * (IS[0] + IS[K - 1]) - IS[1]);
    if (chi_is_one<double>(P, ISt, ISL, 2)) return qH;
    double ISH = IS[0];
#pragma unroll
    for (int k = 1; k < K; ++k) ISH = fmax(ISH, IS[k]);
    const double chi = chi_of<double>(P, ISt, ISH, ISL, 2);
    /* weights d_k / (IS_k + eps)^2, all multiplied by the product of the
     * (IS_j + eps)^2: no division but that of the sums; outside the safe
     * range of the products (overflow, underflow) with a division each */
    double x[K], c[K], ws = 0.0, ql = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) x[k] = IS[k] + P.eps;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        c[k] = 1.0;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if (j != k) c[k] *= x[j];
        const double w = ((k == 1) ? P.C0 : 1.0) * (c[k] * c[k]);
        ws += w;
        ql += w * p[k];
    }
    if (!(ws > 1e-250 && ws < 1e250)) {
        ws = ql = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const double w = ((k == 1) ? P.C0 : 1.0) / (x[k] * x[k]);
            ws += w;
            ql += w * p[k];
        }
    }
    return chi * qH + (1.0 - chi) * (ql / ws);
}

/* a / b, given ib = 1 / b: the product corrected by its remainder, as good as a
 * division (one rounding but for ib's in the remainder) for two more operations.
 * With the plain product the 10^6-cell step's error against 64 bits was 15% larger
 * (4.6e-17 for 4.0e-17, 4.43 ms); with divisions 4.0e-17 and 4.61 ms; so 4.0e-17 and
 * 4.50 ms. */
__device__ __forceinline__ double quotient(double a, double b, double ib)
{
    const double q = a * ib;
    return fma(fma(-q, b, a), ib, q);
}

/* HLLC flux (Toro) with the Davis wave-speed bounds; false if a state is
 * not admissible */
__device__ __forceinline__ bool hllc(double gamma, const double *L, const double *R, double *F)
{
    const double il = 1.0 / L[0], ir = 1.0 / R[0];
    const double rl = L[0], ul = quotient(L[1], rl, il), pl = (gamma - 1.0) * (L[2] - 0.5 * rl * ul * ul);
    const double rr = R[0], ur = quotient(R[1], rr, ir), pr = (gamma - 1.0) * (R[2] - 0.5 * rr * ur * ur);
    if (!(rl > 0.0) || !(rr > 0.0) || !(pl > 0.0) || !(pr > 0.0)) return false;
    const double cl = sqrt(quotient(gamma * pl, rl, il)), cr = sqrt(quotient(gamma * pr, rr, ir));
    const double SL = fmin(ul - cl, ur - cr), SR = fmax(ul + cl, ur + cr);
    const double Ss = (pr - pl + rl * ul * (SL - ul) - rr * ur * (SR - ur)) / (rl * (SL - ul) - rr * (SR - ur));
    if (0.0 <= SL) {
        F[0] = rl * ul;
        F[1] = rl * ul * ul + pl;
        F[2] = ul * (L[2] + pl);
    } else if (0.0 <= Ss) {
        const double k = rl * (SL - ul) / (SL - Ss);
        const double Us[3] = {k, k * Ss, k * (quotient(L[2], rl, il) + (Ss - ul) * (Ss + pl / (rl * (SL - ul))))};
        const double FL[3] = {rl * ul, rl * ul * ul + pl, ul * (L[2] + pl)};
#pragma unroll
        for (int v = 0; v < 3; ++v) F[v] = FL[v] + SL * (Us[v] - L[v]);
    } else if (0.0 <= SR) {
        const double k = rr * (SR - ur) / (SR - Ss);
        const double Us[3] = {k, k * Ss, k * (quotient(R[2], rr, ir) + (Ss - ur) * (Ss + pr / (rr * (SR - ur))))};
        const double FR[3] = {rr * ur, rr * ur * ur + pr, ur * (R[2] + pr)};
#pragma unroll
        for (int v = 0; v < 3; ++v) F[v] = FR[v] + SR * (Us[v] - R[v]);
    } else {
        F[0] = rr * ur;
        F[1] = rr * ur * ur + pr;
        F[2] = ur * (R[2] + pr);
    }
    return true;
}

/* both states of face f, after the admissibility fallback */
template <int ORDER>
__device__ __forceinline__ void nc_states(const KP &P, const double *W, int f, double (*st)[3])
{
    double w[6][3]; /* cells f - 3 .. f + 2 */
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        int flip[3];
        const long c = cell_lin<1>(P, f - 3 + i, 0, 0, flip);
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const double x = W[v * P.ncell + c];
            w[i][v] = ghost_sign<1>(P, flip, v) < 0 ? -x : x;
        }
    }
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const double *own = w[side ? 3 : 2];
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            double u[6]; /* u[2] = 0 is not read */
#pragma unroll
            for (int i = 0; i < 6; ++i) u[i] = w[side ? 5 - i : i][v] - own[v];
            st[side][v] = own[v] + nc_value<ORDER>(P, u);
        }
        if (!admissible<double, 1>(st[side], own, P.adm)) {
#pragma unroll
            for (int v = 0; v < 3; ++v) st[side][v] = own[v];
        }
    }
}

template <int ORDER>
__device__ __forceinline__ void nc_flux(const KP &P, const double *W, int f, int *status, double *F)
{
    double st[2][3];
    nc_states<ORDER>(P, W, f, st);
    if (!hllc(P.gamma, st[0], st[1], F)) {
        atomicOr(status, ST_FLUX);
        F[0] = F[1] = F[2] = 0.0;
    }
    /* walls are at rest and adiabatic: no mass or energy flux */
    if ((f == 0 && P.bcs[0][0] >= 2) || (f == P.n[0] && P.bcs[0][1] >= 2)) F[0] = F[2] = 0.0;
}

/* FLUX = false: face states fs[side][v][c][face] (c = 0 value, 1 derivative,
 * which this scheme does not reconstruct: 0).  FLUX = true: ff[q][v][face]
 * with q = 0 the HLLC flux and q = 1, 2 zero (no time derivative, no
 * interface state). */
template <int ORDER, bool FLUX>
__global__ void __launch_bounds__(32) nc_face_kernel(KP P, const double *__restrict__ W, double *__restrict__ fs,
                                                     double *__restrict__ ff, int *__restrict__ status)
{
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f > P.n[0]) return;
    const long nf = P.nftot;
    if (!FLUX) {
        double st[2][3];
        nc_states<ORDER>(P, W, f, st);
#pragma unroll
        for (int side = 0; side < 2; ++side)
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                fs[((long)(side * 3 + v) * 2 + 0) * nf + f] = st[side][v];
                fs[((long)(side * 3 + v) * 2 + 1) * nf + f] = 0.0;
            }
        return;
    }
    double F[3];
    nc_flux<ORDER>(P, W, f, status, F);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
        ff[(long)(0 * 3 + v) * nf + f] = F[v];
        ff[(long)(1 * 3 + v) * nf + f] = 0.0;
        ff[(long)(2 * 3 + v) * nf + f] = 0.0;
    }
}

/* The RK update of one cell from the fluxes of its faces; returns the new state. */
template <int STAGE>
__device__ __forceinline__ void nc_update(const KP &P, double dt, const double *F, const double *up, double *W0,
                                          double *Wout, double *Acc, int *status,
                                          long cell, double *out)
{
    /* loads before stores (chain.cuh) */
    double u0[3], acc[3];
#pragma unroll
    for (int v = 0; v < 3; ++v) {
        u0[v] = W0[v * P.ncell + cell];
        acc[v] = STAGE == 1 ? 0.0 : Acc[v * P.ncell + cell];
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) {
        const double L = -(up[v] - F[v]) * P.ih;
        const long i = (long)v * P.ncell + cell;
        if (STAGE == 1) {
            Acc[i] = L;
            out[v] = Wout[i] = u0[v] + 0.5 * dt * L;
        } else if (STAGE == 2) {
            Acc[i] = acc[v] + 2.0 * L;
            out[v] = Wout[i] = u0[v] + 0.5 * dt * L;
        } else if (STAGE == 3) {
            Acc[i] = acc[v] + 2.0 * L;
            out[v] = Wout[i] = u0[v] + dt * L;
        } else {
            out[v] = W0[i] = u0[v] + dt / 6.0 * (acc[v] + L);
        }
    }
    const double p = P.fp.gm1 * (out[2] - 0.5 * out[1] * out[1] / out[0]);
    int st = 0;
    if (!(out[0] > 0.0)) st |= ST_RHO;
    if (!(p > 0.0)) st |= ST_P;
    if (!isfinite(p) || !isfinite(out[0])) st |= ST_NAN;
    if (st) atomicOr(status, st);
}

/* one stage of classical RK4 with L(U)_j = -(F_{j+1/2} - F_{j-1/2}) / h, the
 * stage's input Win, its output Wout (another buffer: the neighbours' stencils
 * still read Win):
 *   stage 1: Acc = L(U0),   U1 = U0 + dt/2 L(U0)
 *   stage 2: Acc += 2 L(U1), U2 = U0 + dt/2 L(U1)
 *   stage 3: Acc += 2 L(U2), U3 = U0 + dt L(U2)
 *   stage 4: U0 += dt/6 (Acc + L(U3)) */
template <int ORDER, int STAGE>
__global__ void __launch_bounds__(32) nc_stage_kernel(KP P, const double *Win, double *W0, double *Wout, double *Acc,
                                                      int *status, StepClock clk)
{
    after_previous();
    const int lane = threadIdx.x, n = P.n[0];
    const int f = min((int)blockIdx.x * kCells1d + lane, n); /* lanes past the last face repeat it */
    const double dt = clock_dt(clk);
    if (STAGE == 1 && clk.clear && blockIdx.x == 0 && lane < 2) clk.clear[lane] = 0ull;
    double F[3], up[3];
    nc_flux<ORDER>(P, Win, f, status, F);
#pragma unroll
    for (int v = 0; v < 3; ++v) up[v] = __shfl_down_sync(0xffffffffu, F[v], 1);
    const long cell = (long)blockIdx.x * kCells1d + lane;
    const bool own = lane < kCells1d && cell < n;
    double out[3] = {1.0, 0.0, 0.0};
    if (own) nc_update<STAGE>(P, dt, F, up, W0, Wout, Acc, status, cell, out);
    if (STAGE == 4 && clk.out) speed_max<double>(own ? speed_of<1, double>(out, P.gamma) : 0.0, 0.0, clk.out);
}

/* the same stage for short grids: eight lanes per face, six of them
 * reconstructing one variable of one side each (step_1d.cuh) */
template <int ORDER, int STAGE>
__global__ void __launch_bounds__(128) nc_short_kernel(KP P, const double *Win, double *W0, double *Wout, double *Acc,
                                                       int *status, StepClock clk)
{
    after_previous();
    __shared__ double q[kShortFaces][3];
    const int n = P.n[0], sub = threadIdx.x & 7, face = threadIdx.x >> 3;
    const int f = min((int)blockIdx.x * kCellsShort + face, n); /* past the last face: the last face again */
    const double dt = clock_dt(clk);
    if (STAGE == 1 && clk.clear && blockIdx.x == 0 && threadIdx.x < 2) clk.clear[threadIdx.x] = 0ull;
    double val = 0.0, own = 0.0;
    if (sub < 6) {
        const int side = sub / 3, v = sub % 3;
        double u[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            int flip[3];
            const long c = cell_lin<1>(P, side ? f + 2 - i : f - 3 + i, 0, 0, flip);
            const double x = Win[v * P.ncell + c];
            u[i] = ghost_sign<1>(P, flip, v) < 0 ? -x : x;
        }
        own = u[2];
#pragma unroll
        for (int i = 0; i < 6; ++i) u[i] -= own;
        val = own + nc_value<ORDER>(P, u);
    }
    __syncwarp();
    double st[2][3], cw[3];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        gather3(val, (threadIdx.x & 24) + 3 * side, st[side]);
        gather3(own, (threadIdx.x & 24) + 3 * side, cw);
        if (!admissible<double, 1>(st[side], cw, P.adm)) {
#pragma unroll
            for (int v = 0; v < 3; ++v) st[side][v] = cw[v];
        }
    }
    double F[3];
    if (!hllc(P.gamma, st[0], st[1], F)) {
        if (sub == 0) atomicOr(status, ST_FLUX);
        F[0] = F[1] = F[2] = 0.0;
    }
    /* walls are at rest and adiabatic: no mass or energy flux */
    if ((f == 0 && P.bcs[0][0] >= 2) || (f == n && P.bcs[0][1] >= 2)) F[0] = F[2] = 0.0;
    if (sub == 0) {
#pragma unroll
        for (int v = 0; v < 3; ++v) q[face][v] = F[v];
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int l = threadIdx.x;
    const long cell = (long)blockIdx.x * kCellsShort + l;
    const bool mine = l < kCellsShort && cell < n;
    double out[3] = {1.0, 0.0, 0.0};
    if (mine) nc_update<STAGE>(P, dt, q[l], q[l + 1], W0, Wout, Acc, status, cell, out);
    if (STAGE == 4 && clk.out) speed_max<double>(mine ? speed_of<1, double>(out, P.gamma) : 0.0, 0.0, clk.out);
}

template <int ORDER, int STAGE>
void nc_stage(gks_ctx *c, const double *in, double *out, const StepClock &clk)
{
    const KP &P = c->kp;
    ProfScope ps(c, GKS_KC_FACE);
    if (short_1d(P.n[0]))
        launch_chained(nc_short_kernel<ORDER, STAGE>, blocks_for(P.n[0], kCellsShort), 128, c->stream, P, in, c->W, out, c->Acc, c->status, clk);
    else
        launch_chained(nc_stage_kernel<ORDER, STAGE>, blocks_for(P.n[0], kCells1d), 32, c->stream, P, in, c->W, out, c->Acc, c->status, clk);
}

template <int ORDER> cudaError_t nc_step(gks_ctx *c, const StepClock &first, const StepClock &mid, const StepClock &last)
{
    /* U1 and U3 in Ws, U2 in Gs (of the same size in 1D) */
    nc_stage<ORDER, 1>(c, c->W, c->Ws, first);
    nc_stage<ORDER, 2>(c, c->Ws, c->Gs, mid);
    nc_stage<ORDER, 3>(c, c->Gs, c->Ws, mid);
    nc_stage<ORDER, 4>(c, c->Ws, nullptr, last);
    return cudaGetLastError();
}

} // namespace

cudaError_t nc_launch_faces(gks_ctx *c, int input, double *fs_dev, bool flux)
{
    const KP &P = c->kp;
    const double *W = input ? c->Ws : c->W;
    const unsigned nb = blocks_for(P.n[0] + 1, 32);
    double *ff = (double *)c->ff;
    ProfScope ps(c, GKS_KC_FACE);
    if (c->order == 5) {
        if (flux) nc_face_kernel<5, true><<<nb, 32, 0, c->stream>>>(P, W, nullptr, ff, c->status);
        else nc_face_kernel<5, false><<<nb, 32, 0, c->stream>>>(P, W, fs_dev, nullptr, c->status);
    } else {
        if (flux) nc_face_kernel<6, true><<<nb, 32, 0, c->stream>>>(P, W, nullptr, ff, c->status);
        else nc_face_kernel<6, false><<<nb, 32, 0, c->stream>>>(P, W, fs_dev, nullptr, c->status);
    }
    return cudaGetLastError();
}

cudaError_t nc_launch_step(gks_ctx *c, const StepClock &first, const StepClock &mid, const StepClock &last)
{
    return c->order == 5 ? nc_step<5>(c, first, mid, last) : nc_step<6>(c, first, mid, last);
}

} // namespace gks
