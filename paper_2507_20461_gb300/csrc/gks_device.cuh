/*
 * Gas-kinetic interface flux for the Euler and Navier-Stokes equations
 * (device code).
 *
 * The paper (Sec. 2) takes the flux from the time-dependent gas distribution
 * function of the GKS and defers its formulas to earlier work; this is the
 * BGK solution at an interface Gauss point in the face frame (velocity
 * component 0 and derivative axis 0 along the face normal):
 *
 *   f(0,t) = (1-e) g0 + t e (T0 g0) + t (A0 g0)
 *          + e [ (1 - t T_l) H(u) g_l + (1 - t T_r) H(-u) g_r ],   e = exp(-t/tau_n),
 *
 * with T = sum_e a_e u_e the spatial micro-slopes (left, right, and the
 * equilibrium one from the mean of the left/right derivatives), A0 the
 * equilibrium time slope from the compatibility condition, the physical
 * collision time 0 (Euler) in the Chapman-Enskog terms and the numerical one
 * tau_n = C1 dt + C2 |pl - pr| / (pl + pr) dt in the relaxation factor.
 *
 * Closed forms used here (all exact rearrangements of the velocity
 * integrals):
 *   rho0 <u psi>_0        = Euler flux of W0;
 *   rho0 <T0 psi>_0       = sum_e dF_e/dx_e(W0) = -dW0/dt;
 *   rho0 <A0 u psi>_0     = dF_n/dt = F_n'(W0) dW0/dt;
 *   time integrals over [0, d]: int (1-e) = d - ie, int t e = ite,
 *     ie = tau_n (1 - e_d), ite = tau_n^2 - tau_n (d + tau_n) e_d.
 * With the integrated fluxes over dt/2 and dt, F = (4 F(dt/2) - F(dt)) / dt
 * and dF/dt = 4 (F(dt) - 2 F(dt/2)) / dt^2 reduce to
 *   F  = F0 + (4 ie_h - ie_1)/dt (Fk - F0) + (4 ite_h - ite_1)/dt (FT0 - FTk),
 *   Ft = FA0 + 4 (ie_1 - 2 ie_h)/dt^2 (Fk - F0) + 4 (ite_1 - 2 ite_h)/dt^2 (FT0 - FTk),
 * and the interface state W(dt/2) = W0 + t (1 - e_t) dW0/dt - t e_t WTk.
 *
 * Navier-Stokes (Sec. 2, viscous flux of the same scheme; Prandtl number 1):
 * the general BGK solution with physical collision time tau > 0,
 *   f(0,t) = (1-e) g0 + ((t+tau) e - tau) T0 g0 + (t - tau + tau e) A0 g0
 *          + e [ (1 - (t+tau) T_l - tau A_l) H(u) g_l + (same, r) H(-u) g_r ],
 * tau = mu / p0 and e = exp(-t/(tau_n + tau)); A_l, A_r the time slopes of
 * the two initial states from their own compatibility conditions.  The tau
 * terms of the integrals add tau (cF1 D - V) to F, tau cT1 D to Ft and
 * -tau e_t (WTk + WAk) to W(dt/2), with V = rho0 <u psi (T0 + A0)>_0 and
 * D = V - FTk - FAk (FAk, WAk: the two half-space moments of A_l, A_r).
 *
 * The FP32 flux evaluates the left and the right Maxwellian together
 * on lane pairs (lr2.cuh: one packed two-lane instruction for both sides);
 * the arithmetic of each lane is the scalar code's.
 */
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "erfc_table.cuh"
#include "fpsplit.cuh"
#include "lr2.cuh"

namespace gks {

/* The half-space moments take h = erfc(a) and e = exp(-a^2) of the same
 * argument.
 * FP64, |a| < 3 (Mach 3.5 normal to the face): degree-8 polynomials about a point
 * x_k near the nearest k/32 from a 15 KB table (gen_erfc.py; truncation below
 * 2^-55), 20 FP64 instructions for both where the library's erfc and exp take about
 * 71; the table's loads run beside the FP64 pipe, which bounds the kernel (2D 512^2
 * face flux 1.52 to 1.27 ms a stage).  The interval comes from an exact add of 1.5
 * 2^47, whose unit is 1/32.  Both functions are all but doubles at x_k, so the
 * constant terms carry no rounding: error 0.76 and 0.61 ulp at most, 0.31 and 0.29
 * rms, where correct rounding has 0.29 (with x_k = k/32 1.3 and 1.2, 0.39 and 0.40).
 * Above, the library.
 * FP32: the library's erfc; e is the hardware exponential (__expf, about 2 + 1.2 x
 * ulp, x = a^2; it multiplies terms that vanish as x grows).  A polynomial in
 * 1 / (1 + |a|/2) times e, lanes together, raised the error of W(dt/2) by a third
 * and is not taken. */
template <typename R> struct RT;
template <> struct RT<double> {
    __device__ static double exp_(double x) { return exp(x); }
    __device__ static double sqrt_(double x) { return sqrt(x); }
    __device__ static double rsqrt_(double x) { return rsqrt(x); }
    __device__ static double tanh_(double x) { return tanh(x); }
    __device__ static double abs_(double x) { return fabs(x); }
    __device__ __forceinline__ static void erfc_exp(double a, double &h, double &e)
    {
        const uint64_t bits = fps::dbits(a);
        const uint32_t hi = (uint32_t)(bits >> 32) & 0x7fffffffu;
        const double x = fps::bitsd(bits & 0x7fffffffffffffffull);
        if (hi < 0x40080000u) { /* |a| < 3 */
            const double m = 211106232532992.0; /* 1.5 2^47 */
            const double *row = erfc_rows[(uint32_t)fps::dbits(x + m) & 127u];
            const double d = x - row[2 * ERFC_DEG + 2];
            double p = row[ERFC_DEG], q = row[2 * ERFC_DEG + 1];
#pragma unroll
            for (int j = ERFC_DEG - 1; j >= 0; --j) {
                p = p * d + row[j];
                q = q * d + row[ERFC_DEG + 1 + j];
            }
            h = p;
            e = q;
        } else {
            h = erfc(x);
            e = exp(-x * x);
        }
        if (bits >> 63) h = 2.0 - h;
    }
};
/* FP32: the exponentials of the flux (erfc_exp and the relaxation factor) take
 * the hardware exponential; the 2048^2 mixed step is 1.3% shorter */
template <> struct RT<float> {
    __device__ static float exp_(float x) { return __expf(x); }
    __device__ static float sqrt_(float x) { return sqrtf(x); }
    __device__ static float rsqrt_(float x) { return rsqrtf(x); }
    __device__ static float tanh_(float x) { return tanhf(x); }
    __device__ static float abs_(float x) { return fabsf(x); }
    __device__ __forceinline__ static void erfc_exp(float a, float &h, float &e)
    {
        e = __expf(-a * a);
        h = erfcf(a);
    }
};

/* left/right pairs: the transcendentals per lane */
template <> struct RT<LR> {
    __device__ static LR rsqrt_(LR x) { return LR(rsqrtf(x.l()), rsqrtf(x.r())); }
    __device__ __forceinline__ static void erfc_exp(LR a, LR &h, LR &e)
    {
        const LR x = LR(a * a);
        e = LR(__expf(-x.l()), __expf(-x.r()));
        h = LR(erfcf(a.l()), erfcf(a.r()));
    }
};

/* x > 0 (every lane of a pair) */
__device__ __forceinline__ bool positive(double x) { return x > 0.0; }
__device__ __forceinline__ bool positive(float x) { return x > 0.f; }
__device__ __forceinline__ bool positive(LR x) { return x.l() > 0.f && x.r() > 0.f; }

/* The two half streams of the initial state at t = 0, one of them per call
 * (or both at once on left/right lane pairs): density-weighted half-space
 * moments of the Maxwellian (W0: <psi>, Fk: <u psi>), of its spatial slope term
 * T = sum_e u_e a_e (WT, FT) and, for Navier-Stokes, of its time slope A (WA,
 * FA).  s = +1 takes u > 0 (left state), -1 takes u < 0.
 *
 * What bounds this code is the number of arithmetic instructions (FP64: two
 * per SM per clock; FP32: issue), so the velocity integrals are arranged for
 * few of them:
 *   - primitive slopes.  With theta = p / rho and tau_e = d_e theta / theta,
 *     a_e = d_e rho / rho - (N/2) tau_e + c.d_e U / theta + (c^2 + xi^2) tau_e /
 *     (2 theta), c = u - U; in powers of the normal velocity and the transverse
 *     peculiar velocities v' = v - V,
 *     a_e = P + Q u + h (u^2 + S^2) + sum_s d_e U_s v'_s / theta,
 *     S^2 = v'^2 + xi^2, h = tau / (2 theta);
 *   - transverse peculiar velocities: their odd moments vanish and <S^2> =
 *     (N-1) theta, <v'^2 S^2> = (N+1) theta^2, <S^4> = (N-1)(N+1) theta^2, so
 *     <T>, <S^2 T> and <v' T> are short polynomials in u (A, A with the extra
 *     terms x0 + x1 u, B below); the raw moments follow by the shift by V;
 *   - the density is folded into the first two half-space moments, and
 *     <u psi_0 T> = <psi_1 T> is taken once.
 * Against raw transverse moments with tabulated expectations and general
 * slope vectors, and the equilibrium below in the same form (GB300, one step):
 * FP64 2D 512^2 5.5 to 4.4 ms, Navier-Stokes 390 x 195 2.1 to 1.55 ms; mixed
 * 256^3 54.5 to 40.9 ms, 2D 2048^2 2.6 to 2.42 ms.  (Registers and spills of the
 * flux kernels: step_flux.cuh.)
 */
template <typename R, int M> struct HalfStream {
    R W0[M + 2], Fk[M + 2], WT[M + 2], FT[M + 2], WA[M + 2], FA[M + 2], p;
};

/* 1 / rho, velocity, rho |U|^2 and pressure of a state (rho |U|^2 from m U: in
 * range wherever the state is) */
template <typename R, int M> struct Primitive {
    R inv, U[M], ke, p;
};
template <typename R, int M> __device__ __forceinline__ Primitive<R, M> primitive_of(const R *W, R gm1)
{
    Primitive<R, M> q;
    q.inv = R(1) / W[0];
    q.ke = R(0);
#pragma unroll
    for (int i = 0; i < M; ++i) {
        q.U[i] = W[1 + i] * q.inv;
        q.ke += q.U[i] * W[1 + i];
    }
    q.p = gm1 * (W[M + 1] - R(0.5) * q.ke);
    return q;
}

template <typename R, int M, bool NS>
__device__ __forceinline__ bool half_stream(const R *W, const Primitive<R, M> &prim, const R (*dW)[M + 2], R gm1, R Ntot, R s,
                                            HalfStream<R, M> &o)
{
    const R inv = prim.inv, p = prim.p, *U = prim.U;
    const R hUU = R(0.5) * prim.ke * inv; /* |U|^2 / 2 */
    if (!positive(W[0]) || !positive(p)) return false;
    o.p = p;
    const R th = p * inv;
    const R y = RT<R>::rsqrt_(th), ith = y * y; /* 1 / theta */
    const R U0 = U[0];

    /* rho <u^k> over the half space; sqrt(lambda) = y / sqrt(2), 1 / sqrt(lambda) = sqrt(2) theta y */
    R u[7];
    {
        const R x = R(0.70710678118654752) * y * U0;
        R h, e;
        RT<R>::erfc_exp(-s * x, h, e);
        u[0] = R(0.5) * W[0] * h;
        u[1] = U0 * u[0] + s * (R(0.39894228040143268) * W[0] * th * y) * e;
#pragma unroll
        for (int k = 0; k < 5; ++k) u[k + 2] = U0 * u[k + 1] + R(k + 1) * th * u[k];
    }
    /* rho <u^k (u^2 + S^2)> */
    const R kt = (Ntot - R(1)) * th;
    R E[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) E[k] = u[k + 2] + kt * u[k];
    R vv = R(0);
#pragma unroll
    for (int t = 1; t < M; ++t) vv += U[t] * U[t];
    o.W0[0] = u[0];
    o.W0[1] = u[1];
    o.Fk[0] = u[1];
    o.Fk[1] = u[2];
#pragma unroll
    for (int t = 1; t < M; ++t) {
        o.W0[1 + t] = U[t] * u[0];
        o.Fk[1 + t] = U[t] * u[1];
    }
    o.W0[M + 1] = R(0.5) * (E[0] + vv * u[0]);
    o.Fk[M + 1] = R(0.5) * (E[1] + vv * u[1]);

    /* primitive slopes; P^ = P + <S^2> h */
    R r0[M], dU[M][M], tau[M], Q[M], h[M], Ph[M];
    const R gip = gm1 * inv * ith, hith = R(0.5) * ith;
#pragma unroll
    for (int e = 0; e < M; ++e) {
        r0[e] = dW[e][0] * inv;
        R dE = dW[e][M + 1] - hUU * dW[e][0];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const R sv = dW[e][1 + i] - U[i] * dW[e][0];
            dE -= U[i] * sv;
            dU[e][i] = sv * inv;
        }
        tau[e] = gip * dE - r0[e];
        h[e] = hith * tau[e];
        const R g = U0 * h[e], al = dU[e][0] * ith;
        Q[e] = al - R(2) * g;
        Ph[e] = r0[e] - R(0.5) * tau[e] - U0 * (al - g);
    }
    /* <T> = A0 + A1 u + A2 u^2 + A3 u^3; <S^2 T> = (N-1) theta <T> + x0 + x1 u */
    R A[4], x0 = R(0), x1 = kt * tau[0];
    A[0] = R(0);
    A[1] = Ph[0];
    A[2] = Q[0];
    A[3] = h[0];
#pragma unroll
    for (int t = 1; t < M; ++t) {
        A[0] += U[t] * Ph[t] + dU[t][t];
        A[1] += U[t] * Q[t];
        A[2] += U[t] * h[t];
        x0 += kt * U[t] * tau[t] + R(2) * th * dU[t][t];
    }
    R w0 = u[1] * A[1] + u[2] * A[2] + u[3] * A[3];
    R f0 = u[2] * A[1] + u[3] * A[2] + u[4] * A[3];
    R f1 = u[3] * A[1] + u[4] * A[2] + u[5] * A[3];
    R we = E[1] * A[1] + E[2] * A[2] + E[3] * A[3] + x1 * u[1];
    R fe = E[2] * A[1] + E[3] * A[2] + E[4] * A[3] + x1 * u[2];
    if constexpr (M > 1) {
        w0 += u[0] * A[0];
        f0 += u[1] * A[0];
        f1 += u[2] * A[0];
        we += E[0] * A[0] + x0 * u[0];
        fe += E[1] * A[0] + x0 * u[1];
    }
    we = R(0.5) * we;
    fe = R(0.5) * fe;
#pragma unroll
    for (int r = 1; r < M; ++r) {
        /* <v'_r T> = B0 + B1 u + B2 u^2 */
        R B0 = th * (Ph[r] + tau[r]);
#pragma unroll
        for (int t = 1; t < M; ++t) B0 += U[t] * dU[t][r];
        const R B1 = dU[0][r] + th * Q[r], B2 = th * h[r];
        const R wr = u[0] * B0 + u[1] * B1 + u[2] * B2;
        const R fr = u[1] * B0 + u[2] * B1 + u[3] * B2;
        o.WT[1 + r] = wr + U[r] * w0;
        o.FT[1 + r] = fr + U[r] * f0;
        we += U[r] * (wr + R(0.5) * U[r] * w0);
        fe += U[r] * (fr + R(0.5) * U[r] * f0);
    }
    o.WT[0] = w0;
    o.WT[1] = f0;
    o.FT[0] = f0;
    o.FT[1] = f1;
    o.WT[M + 1] = we;
    o.FT[M + 1] = fe;
    if constexpr (NS) {
        /* time slope A of this state from its own compatibility condition
         * <psi (T + A) g> = 0 over all velocities: the Euler time derivatives */
        R div = R(0), rt = R(0), tt = R(0);
#pragma unroll
        for (int e = 0; e < M; ++e) {
            div += dU[e][e];
            rt += U[e] * r0[e];
            tt += U[e] * tau[e];
        }
        rt = -(rt + div);
        tt = -(tt + gm1 * div);
        R Ut[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            R c = th * (tau[i] + r0[i]);
#pragma unroll
            for (int e = 0; e < M; ++e) c += U[e] * dU[e][i];
            Ut[i] = -c;
        }
        const R ha = hith * tt, g = U0 * ha, al = Ut[0] * ith;
        const R qa = al - R(2) * g, pa = rt - R(0.5) * tt - U0 * (al - g), xa = kt * tt;
        const R a0 = pa * u[0] + qa * u[1] + ha * u[2], a1 = pa * u[1] + qa * u[2] + ha * u[3];
        R wa = R(0.5) * (pa * E[0] + qa * E[1] + ha * E[2] + xa * u[0]);
        R fa = R(0.5) * (pa * E[1] + qa * E[2] + ha * E[3] + xa * u[1]);
#pragma unroll
        for (int r = 1; r < M; ++r) {
            const R wr = Ut[r] * u[0], fr = Ut[r] * u[1];
            o.WA[1 + r] = wr + U[r] * a0;
            o.FA[1 + r] = fr + U[r] * a1;
            wa += U[r] * (wr + R(0.5) * U[r] * a0);
            fa += U[r] * (fr + R(0.5) * U[r] * a1);
        }
        o.WA[0] = a0;
        o.WA[1] = a1;
        o.FA[0] = a1;
        o.FA[1] = pa * u[2] + qa * u[3] + ha * u[4];
        o.WA[M + 1] = wa;
        o.FA[M + 1] = fa;
    }
    return true;
}

/* Flux constants, precomputed on the host in both precisions so that an
 * FP32 kernel issues no FP64 instruction for them (fill with fill_flux). */
struct FluxParams {
    double gamma, c1, c2;
    double gm1, Ntot, c8N; /* gamma - 1, 2 / (gamma - 1), 8 / Ntot */
    double mu;             /* dynamic viscosity (Navier-Stokes flux only) */
    float fgm1, fNtot, fc8N, fc1, fc2, fmu;
};

/* the constant in the precision R */
template <typename R> __host__ __device__ __forceinline__ R pick(double d, float f)
{
    if constexpr (sizeof(R) == sizeof(float)) return f;
    else return d;
}

inline void fill_flux(FluxParams &fp, double gamma, double c1, double c2)
{
    fp.gamma = gamma;
    fp.c1 = c1;
    fp.c2 = c2;
    fp.gm1 = gamma - 1.0;
    fp.Ntot = 2.0 / (gamma - 1.0);
    fp.c8N = 8.0 / fp.Ntot;
    fp.fgm1 = (float)fp.gm1;
    fp.fNtot = (float)fp.Ntot;
    fp.fc8N = (float)fp.c8N;
    fp.fc1 = (float)c1;
    fp.fc2 = (float)c2;
    fp.fmu = (float)fp.mu;
}

/* The two half streams of a point together: the equilibrium state W0 and its
 * flux Fk from their collision, the sums of their slope (and time slope)
 * moments, and the sums S[e] of the two sides' derivatives. */
template <typename R, int M> struct Streams {
    R W0[M + 2], Fk[M + 2], WT[M + 2], FT[M + 2], WA[M + 2], FA[M + 2], S[M][M + 2], pl, pr;
};

/* FP32: both sides at once on left/right lane pairs (packed two-lane instructions) */
template <int M, bool NS>
__device__ __forceinline__ bool streams_of(const FluxParams &fp, const LR *W, const Primitive<LR, M> &prim,
                                           const LR (*dW)[M + 2], Streams<float, M> &o)
{
    HalfStream<LR, M> q;
    if (!half_stream<LR, M, NS>(W, prim, dW, LR(fp.fgm1), LR(fp.fNtot), LR(1.f, -1.f), q)) return false;
    o.pl = q.p.l();
    o.pr = q.p.r();
#pragma unroll
    for (int b = 0; b < M + 2; ++b) {
        o.W0[b] = q.W0[b].sum();
        o.Fk[b] = q.Fk[b].sum();
        o.WT[b] = q.WT[b].sum();
        o.FT[b] = q.FT[b].sum();
        if constexpr (NS) {
            o.WA[b] = q.WA[b].sum();
            o.FA[b] = q.FA[b].sum();
        }
#pragma unroll
        for (int e = 0; e < M; ++e) o.S[e][b] = dW[e][b].sum();
    }
    return true;
}

/* FP64: one side after the other; prim(g) gives the primitive state of side g */
template <int M, bool NS, typename Prim>
__device__ __forceinline__ bool streams_of(const FluxParams &fp, const double *Wl, const double *Wr, const Prim &prim,
                                           const double (*dWl)[M + 2], const double (*dWr)[M + 2], Streams<double, M> &o)
{
    HalfStream<double, M> q;
    if (!half_stream<double, M, NS>(Wl, prim(0), dWl, fp.gm1, fp.Ntot, 1.0, q)) return false;
    o.pl = q.p;
#pragma unroll
    for (int b = 0; b < M + 2; ++b) {
        o.W0[b] = q.W0[b];
        o.Fk[b] = q.Fk[b];
        o.WT[b] = q.WT[b];
        o.FT[b] = q.FT[b];
        if constexpr (NS) {
            o.WA[b] = q.WA[b];
            o.FA[b] = q.FA[b];
        }
    }
    if (!half_stream<double, M, NS>(Wr, prim(1), dWr, fp.gm1, fp.Ntot, -1.0, q)) return false;
    o.pr = q.p;
#pragma unroll
    for (int b = 0; b < M + 2; ++b) {
        o.W0[b] += q.W0[b];
        o.Fk[b] += q.Fk[b];
        o.WT[b] += q.WT[b];
        o.FT[b] += q.FT[b];
        if constexpr (NS) {
            o.WA[b] += q.WA[b];
            o.FA[b] += q.FA[b];
        }
#pragma unroll
        for (int e = 0; e < M; ++e) o.S[e][b] = dWl[e][b] + dWr[e][b];
    }
    return true;
}

/* The flux of one interface point from its half streams; derivatives in units
 * of 1 / ih (ih = 1 for physical derivatives, 1 / h for cell units: the scale
 * enters the time coefficients instead of every derivative); idt = 1 / dt.
 * Returns false (and leaves outputs untouched) when the equilibrium is not
 * admissible.
 * NS = false: the Euler flux (physical collision time 0 in the Chapman-Enskog
 * terms).  NS = true: the Navier-Stokes flux with Prandtl number 1, physical
 * collision time tau = mu / p0 of the interface equilibrium, added to the
 * numerical one in the relaxation factor. */
template <typename R, int M, bool NS>
__device__ __forceinline__ bool flux_of_streams(const FluxParams &fp, R dt, R idt, R ih, const Streams<R, M> &q, R *F,
                                                R *Ft, R *Wh)
{
    constexpr int NV = M + 2;
    const R gm1 = pick<R>(fp.gm1, fp.fgm1);
    const R Ntot = pick<R>(fp.Ntot, fp.fNtot);
    const R *W0 = q.W0, *Fk = q.Fk, *WTs = q.WT, *FTs = q.FT, *WA = q.WA, *FA = q.FA, pl = q.pl, pr = q.pr;

    /* Equilibrium.  Its slope and time-slope moments have closed forms in the
     * primitive derivatives:
     *   rho0 <psi T0>_0 = -dW0/dt by the Euler equations, rho0 <psi A0>_0 = dW0/dt,
     *   rho0 <u psi A0>_0 = dF_n/dt = F_n'(W0) dW0/dt,
     *   rho0 <u psi (T0 + A0)>_0 = V, the first-order Chapman-Enskog moment over
     *   tau: the stress p (d_i U_n + d_n U_i - (gamma - 1) delta div U), its work,
     *   and the heat flux (N + 2)/2 p d_n theta;
     * so <u psi T0> = V - dF_n/dt without any velocity integral.  The mean
     * derivatives enter as the sums of the two sides' (the factor 1/2 is in
     * the coefficients of the last loop: W0t, FAe and V carry a factor 2). */
    R U[M], ke = R(0);
    const R inv = R(1) / W0[0];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        U[i] = W0[1 + i] * inv;
        ke += U[i] * W0[1 + i];
    }
    const R rho = W0[0], p0 = gm1 * (W0[M + 1] - R(0.5) * ke);
    if (!positive(rho) || !positive(p0)) return false;
    const R hUU = R(0.5) * ke * inv;
    R W0t[NV], FAe[NV], V[NV];
    {
        R dr[M], dp[M], dU[M][M], div = R(0);
#pragma unroll
        for (int e = 0; e < M; ++e) {
            dr[e] = q.S[e][0];
            R dE = q.S[e][M + 1] - hUU * dr[e];
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const R sv = q.S[e][1 + i] - U[i] * dr[e];
                dE -= U[i] * sv;
                dU[e][i] = sv * inv;
            }
            dp[e] = gm1 * dE;
            div += dU[e][e];
        }
        R rt = rho * div, pt = (gm1 + R(1)) * p0 * div;
#pragma unroll
        for (int e = 0; e < M; ++e) {
            rt += U[e] * dr[e];
            pt += U[e] * dp[e];
        }
        rt = -rt;
        pt = -pt;
        R Et = R(0.5) * Ntot * pt + hUU * rt, Ut0 = R(0);
        W0t[0] = rt;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            R c = dp[i] * inv;
#pragma unroll
            for (int e = 0; e < M; ++e) c += U[e] * dU[e][i];
            const R z = rho * c; /* -rho dU_i/dt */
            Et -= U[i] * z;
            W0t[1 + i] = U[i] * rt - z;
            if (i == 0) Ut0 = -c;
        }
        W0t[M + 1] = Et;
        FAe[0] = W0t[1];
        FAe[1] = W0t[1] * U[0] + W0[1] * Ut0 + pt;
#pragma unroll
        for (int i = 1; i < M; ++i) FAe[1 + i] = W0t[1 + i] * U[0] + W0[1 + i] * Ut0;
        FAe[M + 1] = Ut0 * (W0[M + 1] + p0) + U[0] * (Et + pt);
        V[0] = R(0);
        V[1] = p0 * (R(2) * dU[0][0] - gm1 * div);
        V[M + 1] = (R(0.5) * Ntot + R(1)) * (p0 * inv) * (dp[0] - p0 * inv * dr[0]) + U[0] * V[1];
#pragma unroll
        for (int i = 1; i < M; ++i) {
            V[1 + i] = p0 * (dU[0][i] + dU[i][0]);
            V[M + 1] += U[i] * V[1 + i];
        }
    }
    R F0[NV];
    F0[0] = W0[1];
    F0[1] = W0[1] * U[0] + p0;
#pragma unroll
    for (int i = 1; i < M; ++i) F0[1 + i] = W0[1 + i] * U[0];
    F0[M + 1] = U[0] * (W0[M + 1] + p0);

    /* relaxation time over dt, kappa = tau_n / dt, and the time integrals */
    R kap, eh = R(0), tau = R(0);
    if constexpr (std::is_same_v<R, double> && !NS) {
        /* kappa = y / S and 1 / (2 kappa) from one reciprocal of S y, or by a
         * division each where S y is 0 or outside 2^-1000 .. 2^1000 */
        const double S = pl + pr, y = fp.c1 * S + fp.c2 * fabs(pl - pr), Sy = S * y;
        double z;
        if ((uint32_t)(fps::dbits(Sy) >> 32) - 0x01700000u < 0x7e700000u - 0x01700000u) {
            const double q = 1.0 / Sy;
            kap = y * y * q;
            z = -0.5 * S * S * q;
        } else {
            kap = fp.c1 + fp.c2 * fabs(pl - pr) / S;
            z = kap > 0.0 ? -0.5 / kap : -1e3; /* exp(-1e3) = 0 */
        }
        eh = exp(z);
    } else {
        kap = pick<R>(fp.c1, fp.fc1) + pick<R>(fp.c2, fp.fc2) * RT<R>::abs_(pl - pr) / (pl + pr);
        if constexpr (NS) {
            tau = pick<R>(fp.mu, fp.fmu) / p0;
            kap += tau * idt;
            tau *= ih;
        }
        if (kap > R(0)) eh = RT<R>::exp_(R(-0.5) / kap);
    }
    const R e1 = eh * eh; /* exp(-dt/tn) */
    const R ie_h = kap * (R(1) - eh), ie_1 = kap * (R(1) - e1);
    const R ite_h = kap * (kap - (R(0.5) + kap) * eh), ite_1 = kap * (kap - (R(1) + kap) * e1);
    const R cF1 = R(4) * ie_h - ie_1, cF2 = (R(4) * ite_h - ite_1) * (dt * ih);
    const R cT1 = R(4) * (ie_1 - R(2) * ie_h) * idt, cT2 = R(4) * (ite_1 - R(2) * ite_h) * ih;
    const R hih = R(0.5) * ih, hw = hih * dt, cW1 = R(0.5) * hw * (R(1) - eh), cW2 = -hw * eh;
#pragma unroll
    for (int b = 0; b < NV; ++b) {
        const R dk = Fk[b] - F0[b];
        const R dT = R(0.5) * (V[b] - FAe[b]) - FTs[b];
        F[b] = F0[b] + cF1 * dk + cF2 * dT;
        Ft[b] = hih * FAe[b] + cT1 * dk + cT2 * dT;
        Wh[b] = W0[b] + cW1 * W0t[b] + cW2 * WTs[b];
        if constexpr (NS) {
            /* the tau terms of the time integrals: with V = <u psi (T0 + A0) g0>
             * (the equilibrium's viscous part) and D = V - (left + right
             * half-space <u psi (T + A) g>), F gains tau (cF1 D - V) and Ft
             * gains tau cT1 D; the interface state gains -tau e (the two
             * sides' half-space <psi (T + A) g>), since <psi (T0 + A0) g0> = 0 */
            const R v = R(0.5) * V[b], D = v - FTs[b] - FA[b];
            F[b] += tau * (cF1 * D - v);
            Ft[b] += tau * cT1 * D;
            Wh[b] -= tau * eh * (WTs[b] + WA[b]);
        }
    }
    return true;
}

/* one interface point: states and derivatives (units of 1 / ih) of the two sides */
template <typename R, int M, bool NS = false>
__device__ __forceinline__ bool gks_point_scaled(const FluxParams &fp, R dt, R idt, R ih, const R *Wl, const R *Wr,
                                                 const R (*dWl)[M + 2], const R (*dWr)[M + 2], R *F, R *Ft, R *Wh)
{
    Streams<R, M> q;
    if constexpr (std::is_same_v<R, float>) {
        LR W[M + 2], dW[M][M + 2];
#pragma unroll
        for (int b = 0; b < M + 2; ++b) {
            W[b] = LR(Wl[b], Wr[b]);
#pragma unroll
            for (int e = 0; e < M; ++e) dW[e][b] = LR(dWl[e][b], dWr[e][b]);
        }
        if (!streams_of<M, NS>(fp, W, primitive_of<LR, M>(W, LR(fp.fgm1)), dW, q)) return false;
    } else {
        auto prim = [&](int g) { return primitive_of<R, M>(g ? Wr : Wl, fp.gm1); };
        if (!streams_of<M, NS>(fp, Wl, Wr, prim, dWl, dWr, q)) return false;
    }
    return flux_of_streams<R, M, NS>(fp, dt, idt, ih, q, F, Ft, Wh);
}

/* the same from physical derivatives */
template <typename R, int M, bool NS = false>
__device__ __forceinline__ bool gks_point(const FluxParams &fp, R dt, const R *Wl, const R *Wr, const R (*dWl)[M + 2],
                                          const R (*dWr)[M + 2], R *F, R *Ft, R *Wh)
{
    return gks_point_scaled<R, M, NS>(fp, dt, R(1) / dt, R(1), Wl, Wr, dWl, dWr, F, Ft, Wh);
}

} // namespace gks
