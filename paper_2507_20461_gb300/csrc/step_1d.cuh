/*
 * One stage of the 1D schemes (arXiv 2507.20461, Sec. 4.1, Sec. 4.2) as one
 * kernel: the faces and the update of the cells between them.
 *
 * FP64 is issued at two lanes per SM and clock, and an FP64 instruction holds
 * its warp's scheduler for 64 clocks however many lanes are active (4 warps of
 * an SM, one per scheduler: 76; measured with chains of DFMA).  A stage of a
 * grid that does not fill the schedulers therefore takes 31 ns per FP64
 * instruction of one warp, and is split accordingly:
 *   - long grids, step1d_kernel: a lane takes face f0 + l and then cell f0 + l, the
 *     upper face's fluxes coming from the next lane by shuffle; the last
 *     lane's face is the next warp's first (both evaluate it from the same
 *     inputs by the same instructions, so its flux leaves one cell and enters
 *     the other to the bit).  One warp per block: warps spread over the SMs;
 *   - short FP64 grids, step1d_short_kernel: eight lanes take a face.  Six
 *     reconstruct one variable of one side each, then each lane takes the half
 *     stream of one side, so a warp issues about a quarter of the instructions.
 *     A block's four warps take 16 faces and update the 15 cells between.
 * The time step of a CFL run comes from the wave speed that the previous
 * step's last stage left (two words: max |u| + c and max 1 / rho): every thread
 * divides for itself, so a step is two launches (RK4: four) with no reduction,
 * time-step or memory-set launch between.  The first stage clears the slot
 * that the last stage adds to.
 * Against separate face (128 threads a block), update, wave-speed, time-step
 * and memset launches: 20 steps of 400 cells 3.56 to 1.15 ms (long form 2.43 ms; 0.96 ms with chained
 * launches and the flux's table).
 */
#pragma once
#include "kernels.cuh"

namespace gks {

/* where a step's dt comes from and where the next step's wave speed goes */
struct StepClock {
    const double *dt;             /* given time step, or */
    const unsigned long long *in; /* wave speed of the step's input (dt = nullptr) */
    unsigned long long *clear;    /* slot to zero (first stage), or nullptr */
    unsigned long long *out;      /* slot of the new state's wave speed (last stage), or nullptr */
    double cfl_h, visc;
};

__device__ __forceinline__ double clock_dt(const StepClock &k) { return k.dt ? k.dt[0] : dt_of_speed(k.in, k.cfl_h, k.visc); }

/* cells of a block: its faces less the one shared with the next block */
constexpr int kCells1d = 31, kShortFaces = 16, kCellsShort = kShortFaces - 1;

/* The short form up to three blocks per SM: with n blocks' worth of warps per
 * scheduler it takes about n times its one-wave time, the long form does not
 * change until 31 cells per scheduler.  Short / long measured (us a step, order
 * 8): 400 cells 55 / 121, 4000 86 / 121, 6500 118 / 121, 9000 149 / 121; order 6
 * (RK4): 74 / 186, 102 / 186, 133 / 190, 165 / 190.  The line is where order 8
 * meets. */
inline bool short_1d(int n)
{
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
    return (n + kCellsShort - 1) / kCellsShort <= 3 * nsm;
}

/* one variable of one side of face f (value, physical derivative, and the
 * cell's own average): the left reconstruction of the stencil, mirrored for
 * the right side (derivatives change sign) */
__device__ __forceinline__ void recon1d_side(const KP &P, const double *W, const double *G, int f,
                                             int side, int v, double &val, double &der, double &own)
{
    double w[4], d[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int flip[3];
        const long c = cell_lin<1>(P, side ? f + 1 - q : f - 2 + q, 0, 0, flip);
        const double x = W[v * P.ncell + c], g = G[v * P.ncell + c] * P.h;
        const bool neg = ghost_sign<1>(P, flip, v) < 0;
        w[q] = neg ? -x : x;
        d[q] = (neg != ((flip[0] & 1) != 0)) != (side != 0) ? -g : g;
    }
    own = w[1];
    const double wm1 = w[0] - own, w1 = w[2] - own, w2 = w[3] - own;
    double qv, qd, a[3][2], pv[3], pd[3];
    p7_face<double>(wm1, 0.0, w1, w2, d[0], d[1], d[2], d[3], qv, qd);
    sub_quadratics<double>(wm1, w1, w2, d[0], a, pv, pd);
    geno1d_blend<double>(P, a, pv, pd, qv, qd, val, der);
    val += own;
    der = (side ? -der : der) * P.ih;
}

/* values of the group's lanes as one array: x[v] of side s from lane base + 3 s + v */
__device__ __forceinline__ void gather3(double x, int from, double *o)
{
#pragma unroll
    for (int v = 0; v < 3; ++v) o[v] = __shfl_sync(0xffffffffu, x, from + v);
}

template <bool NS, int STAGE>
__global__ void __launch_bounds__(128) step1d_short_kernel(KP P, const double *Win, const double *Gin, double *W,
                                                           double *G, double *Ws, double *Gs, double *Acc, int *status,
                                                           StepClock clk)
{
    after_previous();
    __shared__ double q[kShortFaces][9];
    const int n = P.n[0], sub = threadIdx.x & 7, face = threadIdx.x >> 3;
    const int f = min((int)blockIdx.x * kCellsShort + face, n); /* past the last face: the last face again */
    const double dt = clock_dt(clk);
    if (STAGE == 1 && clk.clear && blockIdx.x == 0 && threadIdx.x < 2) clk.clear[threadIdx.x] = 0ull;
    double val = 0.0, der = 0.0, own = 0.0;
    if (sub < 6) recon1d_side(P, Win, Gin, f, sub / 3, sub % 3, val, der, own);
    __syncwarp();
    /* this lane's side: even left, odd right */
    const int side = sub & 1, from = (threadIdx.x & 24) + 3 * side;
    double Wq[3], dW[1][3], cw[3];
    gather3(val, from, Wq);
    gather3(der, from, dW[0]);
    gather3(own, from, cw);
    if (!admissible<double, 1>(Wq, cw, P.adm)) {
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            Wq[v] = cw[v];
            dW[0][v] = 0.0;
        }
    }
    HalfStream<double, 1> hs;
    bool ok = half_stream<double, 1, NS>(Wq, primitive_of<double, 1>(Wq, P.fp.gm1), dW, P.fp.gm1, P.fp.Ntot, side ? -1.0 : 1.0, hs);
    if (!ok) hs = HalfStream<double, 1>{};
    ok = __shfl_xor_sync(0xffffffffu, (int)ok, 1) && ok;
    Streams<double, 1> s;
    auto both = [](double x) { return x + __shfl_xor_sync(0xffffffffu, x, 1); };
#pragma unroll
    for (int v = 0; v < 3; ++v) {
        s.W0[v] = both(hs.W0[v]);
        s.Fk[v] = both(hs.Fk[v]);
        s.WT[v] = both(hs.WT[v]);
        s.FT[v] = both(hs.FT[v]);
        if constexpr (NS) {
            s.WA[v] = both(hs.WA[v]);
            s.FA[v] = both(hs.FA[v]);
        }
        s.S[0][v] = both(dW[0][v]);
    }
    s.pl = hs.p; /* the pair's pressures enter by |pl - pr| and pl + pr */
    s.pr = __shfl_xor_sync(0xffffffffu, hs.p, 1);
    double F[3], Ft[3], Wh[3];
    if (ok) ok = flux_of_streams<double, 1, NS>(P.fp, dt, 1.0 / dt, 1.0, s, F, Ft, Wh);
    if (!ok) {
        if (sub == 0) atomicOr(status, ST_FLUX);
#pragma unroll
        for (int v = 0; v < 3; ++v) F[v] = Ft[v] = Wh[v] = 0.0;
    }
    /* walls (slip or no-slip) are at rest and adiabatic: neither mass nor energy crosses them */
    if ((f == 0 && P.bcs[0][0] >= 2) || (f == n && P.bcs[0][1] >= 2)) F[0] = F[2] = Ft[0] = Ft[2] = 0.0;
    if (sub == 0) {
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            q[face][v] = F[v];
            q[face][3 + v] = Ft[v];
            q[face][6 + v] = Wh[v];
        }
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int l = threadIdx.x;
    const long cell = (long)blockIdx.x * kCellsShort + l;
    const bool mine = l < kCellsShort && cell < n;
    double Wn[3] = {1.0, 0.0, 0.0};
    if (mine) {
        auto fsum = [&](int i, int v, int, int plus) -> double { return q[l + plus][3 * i + v]; };
        fp64_update_cell<1, STAGE>(P, fsum, 1.0, dt, W, G, Ws, Gs, Acc, status, cell, Wn);
    }
    if (STAGE == 2 && clk.out) speed_max<double>(mine ? speed_of<1, double>(Wn, P.gamma) : 0.0, mine ? 1.0 / Wn[0] : 0.0, clk.out);
}

template <typename R, bool NS, int STAGE>
__global__ void __launch_bounds__(32) step1d_kernel(KP P, const double *Win, const double *Gin, double *W, double *G,
                                                    double *Ws, double *Gs, double *Acc, int *status, StepClock clk)
{
    after_previous();
    const int lane = threadIdx.x, n = P.n[0];
    const int f = min((int)blockIdx.x * kCells1d + lane, n); /* lanes past the last face repeat it */
    const double dt = clock_dt(clk);
    if (STAGE == 1 && clk.clear && blockIdx.x == 0 && lane < 2) clk.clear[lane] = 0ull;
    R q[3][3], up[3][3];
    flux1d_face<R, NS>(P, Win, Gin, f, R(dt), status, q[0], q[1], q[2]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int v = 0; v < 3; ++v) up[i][v] = __shfl_down_sync(0xffffffffu, q[i][v], 1);
    const long cell = (long)blockIdx.x * kCells1d + lane;
    const bool own = lane < kCells1d && cell < n;
    double Wn[3] = {1.0, 0.0, 0.0};
    if (own) {
        auto fsum = [&](int i, int v, int, int plus) -> double { return (double)(plus ? up[i][v] : q[i][v]); };
        fp64_update_cell<1, STAGE>(P, fsum, 1.0, dt, W, G, Ws, Gs, Acc, status, cell, Wn);
    }
    if (STAGE == 2 && clk.out) speed_max<double>(own ? speed_of<1, double>(Wn, P.gamma) : 0.0, own ? 1.0 / Wn[0] : 0.0, clk.out);
}

} // namespace gks
