/*
 * The stage kernels of the multi-D step path (arXiv 2507.20461, Sec. 2-4):
 * face fluxes with one thread per face, and the layouts they share with the
 * reconstruction and the update.
 *
 * One thread takes a face with all its Gauss points (2 in 2D, 4 in 3D):
 *   - a cubic's values and derivatives at two Gauss points +-a of a face differ
 *     only in the sign of the terms odd in that tangential coordinate, so a
 *     pair costs little more than one point (face_pair: 22 operations in 2D and
 *     41 in 3D per variable and side against 42 and 90 for two separate
 *     evaluations);
 *   - the Gauss points are summed in registers: no exchange between threads,
 *     no barrier, one decomposition of the face index;
 *   - FP32 evaluates both sides at once on left/right lane pairs, which the
 *     flux takes as they are; FP64 evaluates side after side.
 * The second point of a pair waits in shared memory (private slots of the
 * thread: no barrier, no bank conflicts).
 * Against one thread per (face, Gauss point), coefficients staged per block by
 * cp.async and the sums exchanged through shared memory, one launch per
 * direction (GB300): 2048^2 mixed 0.77 to 0.48 ms a stage, 256^3 mixed 16.9
 * to 8.0 ms, 99 x 64 x 50 Navier-Stokes 0.39 to 0.20 ms, FP64 512^2 1.87 to
 * 1.50 ms (0.456, 7.97, 0.197 and 1.236 ms with the flux arithmetic, slots and
 * block order of now).
 *
 * Layouts (step path only): groups of 32 consecutive extended cells, or faces,
 * with the record fields of a group in rows of 32, so that every field of an
 * item lies at a constant offset from one address (loads and stores with
 * immediate offsets, still coalesced):
 *   B  : per cell NV (NC + 1) fields, the blended cubic and the (mirrored)
 *        average of each variable, so the flux needs no ghost mapping;
 *   ff : per face 3 NV fields, F, dF/dt and W(dt/2) summed over the Gauss points.
 * In FP64 the sum over a face's points is rounded at the face value's size, where
 * the difference of two neighbouring faces' points would be exact: a step's error
 * against 64 bits is 5% to 8% larger than with every point kept (3.3e-15 for 3.1e-15,
 * 390 x 195 viscous).  Kept, the points double ff and the update's FP64 work: 512^2
 * 6.17 to 6.21 ms a pass of two steps, 20^3 609 to 628 us and 12 x 9 x 10 230 to 297 us a step.
 */
#pragma once
#include "kernels.cuh"

namespace gks {

/* fields of a cell's record in B: v (NC + 1) + k, k = NC the average */
template <int M> constexpr int kCellFields = (M + 2) * (Cubic<float, M>::NC + 1);
template <int M> constexpr int kFaceFields = 3 * (M + 2);
/* offset of field 0 of item i of a layout with F fields; field k follows at 32 k */
template <int F> __host__ __device__ __forceinline__ size_t group_off(unsigned i)
{
    return (size_t)(i >> 5) * (F * 32) + (i & 31u);
}
__host__ __device__ __forceinline__ size_t group_elems(size_t items, int fields) { return (items + 31) / 32 * 32 * fields; }

/* index of the monomial x^e0 y^e1 z^e2 in the generated coefficient order:
 * by degree, then lexicographic in (e0, e1, e2), x y z absent in 3D */
template <int M> constexpr int mono_index(int e0, int e1, int e2)
{
    int n = 0;
    for (int deg = 1; deg <= 3; ++deg)
        for (int a = 0; a <= deg; ++a)
            for (int b = 0; b <= (M == 3 ? deg - a : deg); ++b) {
                const int c = M == 3 ? deg - a - b : 0;
                if (M == 2 && a + b != deg) continue;
                if (a == 1 && b == 1 && c == 1) continue;
                if (a == e0 && b == e1 && c == e2) return n;
                ++n;
            }
    return -1;
}

/* index of n^i t1^j t2^k, n the face normal D, t1 < t2 the other axes */
template <int M, int D> constexpr int face_mono(int i, int j, int k)
{
    int e[3] = {0, 0, 0};
    e[D] = i;
    e[D == 0 ? 1 : 0] = j;
    if (M == 3) e[D == 2 ? 1 : 2] = k;
    return mono_index<M>(e[0], e[1], e[2]);
}

template <int M, int D, int I, int J, int K> struct FaceMono {
    static constexpr int at = face_mono<M, D>(I, J, K);
};

/* Value and derivatives (face frame: normal, tangential ascending; cell units)
 * of w + cubic at the two Gauss points t1 = -a (o0) and t1 = +a (o1) of the
 * face at n = s/2, t2 = sa (3D; sa = -+a), a = 1/(2 sqrt 3), a^2 = 1/12. */
template <typename V, int M, int D>
__device__ __forceinline__ void face_pair(const V *c, V w, V s, V sa, V *o0, V *o1)
{
    constexpr double A = 0.28867513459481287;
    const V a = V(A);
#define C(i, j, k) c[FaceMono<M, D, i, j, k>::at]
    V q1 = C(0, 1, 0) + V(0.5) * s * C(1, 1, 0);
    q1 += V(0.25) * C(2, 1, 0);
    V r = C(1, 2, 0), dn = C(1, 0, 0) + s * C(2, 0, 0), d1o, vo;
    if constexpr (M == 3) {
        q1 += V(1.0 / 12.0) * C(0, 1, 2);
        q1 += sa * C(0, 1, 1);
        r += C(1, 0, 2);
        dn += sa * (C(1, 0, 1) + s * C(2, 0, 1));
    }
    dn += V(1.0 / 12.0) * r;
    dn += V(0.75) * C(3, 0, 0);
    V v = V(0.5) * s * C(1, 0, 0);
    v += V(1.0 / 6.0) * C(2, 0, 0);
    v += V(0.125) * s * C(3, 0, 0);
    v += V(1.0 / 24.0) * s * r;
    vo = a * (q1 + V(1.0 / 12.0) * C(0, 3, 0));
    const V d1 = q1 + V(0.25) * C(0, 3, 0);
    const V dno = a * (C(1, 1, 0) + s * C(2, 1, 0));
    d1o = V(2.0 * A) * C(0, 2, 0) + V(A) * s * C(1, 2, 0);
    if constexpr (M == 3) {
        V q2 = C(0, 0, 1) + V(0.5) * s * C(1, 0, 1);
        q2 += V(0.25) * C(2, 0, 1);
        q2 += V(1.0 / 12.0) * C(0, 2, 1);
        v += sa * (q2 + V(1.0 / 12.0) * C(0, 0, 3));
        d1o += V(2.0 * A) * sa * C(0, 2, 1);
        V d2 = q2 + V(0.25) * C(0, 0, 3);
        d2 += sa * (V(2.0) * C(0, 0, 2) + s * C(1, 0, 2));
        const V d2o = a * C(0, 1, 1) + V(2.0 * A) * sa * C(0, 1, 2);
        o0[3] = d2 - d2o;
        o1[3] = d2 + d2o;
    }
#undef C
    /* the average last: the increments round at their own size */
    o0[0] = w + (v - vo);
    o1[0] = w + (v + vo);
    o0[1] = dn - dno;
    o1[1] = dn + dno;
    o0[2] = d1 - d1o;
    o1[2] = d1 + d1o;
}

/* FP32: one group of left/right lane pairs; FP64: two groups, left and right */
template <typename R> struct FaceV;
template <> struct FaceV<float> {
    using V = LR;
    static constexpr int G = 1;
    __device__ __forceinline__ static V sign(int) { return LR(1.f, -1.f); }
    __device__ __forceinline__ static V load(const float *l, const float *r, int, int off) { return LR(l[off], r[off]); }
};
template <> struct FaceV<double> {
    using V = double;
    static constexpr int G = 2;
    __device__ __forceinline__ static V sign(int g) { return g ? -1.0 : 1.0; }
    __device__ __forceinline__ static V load(const double *l, const double *r, int g, int off) { return (g ? r : l)[off]; }
};

/* values a thread keeps in its shared slots: the second point of a pair */
template <typename R, int M> constexpr int kFaceStash = FaceV<R>::G * (M + 2) * (M + 1);

/* The pointer as an opaque value: loads through it stay where they are
 * written, instead of being hoisted (and their values spilled) out of the
 * loops over the Gauss points. */
template <typename R> __device__ __forceinline__ const R *opaque(const R *p)
{
#ifdef __CUDA_ARCH__
    asm volatile("" : "+l"(p));
#endif
    return p;
}

/* The flux of one Gauss point from the face-frame states and derivatives
 * W[g][v], dW[g][e][v] (cell units) of both sides, after the admissibility
 * fallback: a side whose density rho or pressure p is not above adm times its
 * cell's, rho_c and p_c, takes the cell average (average(g, v)) with zero slopes.
 * The test is
 *   FP64: rho > rref = adm rho_c and p > plim = adm p_c, p from the half streams'
 *         own primitive state (no operation but the comparisons);
 *   FP32: with rref = 1 / rho_c, r = rho rref > adm and r E - (m rref) m / 2 >
 *         plim r, plim = adm p_c / (gamma - 1) (reversed where rho_c < 0), which
 *         does not wait for the state's reciprocal: 2048^2 456 us a launch, 256^3
 *         7.97 ms, 99 x 64 x 50 viscous 197 us (with the primitive state's p 453
 *         us, 8.04 ms, 200 us).
 * Both have the range of the flux itself.  Products without rref, rho E - |m|^2 / 2
 * against plim rho, leave FP32's range at rho E below 2^-126, and FP64's, with
 * rho_c as a third factor, at rho^2 E below 2^-1022, where the state does not (they
 * took 452 us, 7.89 ms, 197 us; FP64 512^2 1.264 ms a launch against 1.241 ms).
 * False: a state the flux could not use. */
template <typename R, int M, bool NS, typename Average>
__device__ __forceinline__ bool face_point(const FluxParams &fp, R adm, R dt, R idt, R ih,
                                           typename FaceV<R>::V (&W)[FaceV<R>::G][M + 2],
                                           typename FaceV<R>::V (&dW)[FaceV<R>::G][M][M + 2],
                                           const typename FaceV<R>::V (&rref)[FaceV<R>::G],
                                           const typename FaceV<R>::V (&plim)[FaceV<R>::G], const Average &average, R *F,
                                           R *Ft, R *Wh)
{
    using V = typename FaceV<R>::V;
    constexpr int NV = M + 2, G = FaceV<R>::G;
    /* the primitive state of group g after the fallback */
    auto admitted = [&](int g) -> Primitive<V, M> {
        if constexpr (G == 1) {
            const V r = W[g][0] * rref[g];
            V ke = V(0);
#pragma unroll
            for (int i = 1; i <= M; ++i) ke += W[g][i] * V(W[g][i] * rref[g]);
            const V t = r * W[g][M + 1] - V(0.5) * ke, z = t - plim[g] * r;
            bool okl = r.l() > adm && z.l() > 0.f, okr = r.r() > adm && z.r() > 0.f;
            if (!okl || !okr) {
                okl = okl || (rref[g].l() < 0.f && r.l() < adm && z.l() < 0.f);
                okr = okr || (rref[g].r() < 0.f && r.r() < adm && z.r() < 0.f);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const V c = average(g, v);
                    W[g][v] = V(okl ? W[g][v].l() : c.l(), okr ? W[g][v].r() : c.r());
#pragma unroll
                    for (int e = 0; e < M; ++e) dW[g][e][v] = V(okl ? dW[g][e][v].l() : 0.f, okr ? dW[g][e][v].r() : 0.f);
                }
            }
            return primitive_of<V, M>(W[g], V(fp.fgm1));
        } else {
            Primitive<V, M> q = primitive_of<V, M>(W[g], fp.gm1);
            if (!(W[g][0] > rref[g] && q.p > plim[g])) {
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    W[g][v] = average(g, v);
#pragma unroll
                    for (int e = 0; e < M; ++e) dW[g][e][v] = V(0);
                }
                q = primitive_of<V, M>(W[g], fp.gm1);
            }
            return q;
        }
    };
    Streams<R, M> s;
    if constexpr (G == 1) {
        const Primitive<V, M> q = admitted(0);
        if (!streams_of<M, NS>(fp, W[0], q, dW[0], s)) return false;
    } else {
        if (!streams_of<M, NS>(fp, W[0], W[G - 1], admitted, dW[0], dW[G - 1], s)) return false;
    }
    return flux_of_streams<R, M, NS>(fp, dt, idt, ih, s, F, Ft, Wh);
}

/* One face of direction D: fl its index among that direction's faces; stash the
 * thread's first shared slot, SS the slot stride.
 * SPLIT: each of 2 (3D: 4) neighbouring lanes takes one Gauss point of the face,
 * all lanes of the warp call it, and the sums go over shuffles (no stash); lanes
 * past the last face pass it again with store = false.
 * POINTS: the fluxes of every Gauss point into ff[q][v][g][face] (gks_flux)
 * instead of their sums. */
template <typename R, int M, int D, bool NS, int SS, bool SPLIT = false, bool POINTS = false>
__device__ __forceinline__ void step_face_item(const KP &P, const R *B, R dt, R idt, R *ff,
                                               int *status, unsigned fl, typename FaceV<R>::V *stash, bool store = true)
{
    using FV = FaceV<R>;
    using V = typename FV::V;
    constexpr int NV = M + 2, NC = Cubic<R, M>::NC, G = FV::G, REC = kCellFields<M>;
    unsigned q0, q1 = 0;
    int idx[3];
    idx[0] = (int)fdivmod(P.dface[D][0], fl, q0);
    idx[1] = (int)fdivmod(P.dface[D][1], q0, q1);
    idx[2] = (M >= 3) ? (int)q1 : 0;
    /* extended index of the plus-side cell (one ghost layer), and of the minus side */
    unsigned er = (unsigned)((idx[1] + 1) * P.ext[0] + idx[0] + 1);
    if (M >= 3) er += (unsigned)(idx[2] + 1) * (unsigned)P.ext[0] * (unsigned)P.ext[1];
    const unsigned el = er - (D == 0 ? 1u : (D == 1 ? (unsigned)P.ext[0] : (unsigned)P.ext[0] * (unsigned)P.ext[1]));
    const R *pl = B + group_off<REC>(el), *pr = B + group_off<REC>(er);
    constexpr int A1 = (D == 0) ? 1 : 0, A2 = (D == 2) ? 1 : 2;
    constexpr int ax[3] = {D, A1, A2};
    const R adm = pick<R>(P.adm, P.fadm), ih = pick<R>(P.ih, P.fih);

    R F[NV], Ft[NV], Wh[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) F[v] = Ft[v] = Wh[v] = R(0);
    /* walls (slip or no-slip) are at rest and adiabatic: neither mass nor
     * energy crosses them (exactly, whatever the rounding of the two sides) */
    auto wall = [&] { return (idx[D] == 0 && P.bcs[D][0] >= 2) || (idx[D] == P.n[D] && P.bcs[D][1] >= 2); };
    /* FP32 2D: during the second point the first one's sums wait in the slots
     * that its values left (80 registers spill 16 bytes instead of 180; in 3D,
     * where they live through the loop, and in FP64 this added spills) */
    constexpr bool PARK = G == 1 && M == 2 && !SPLIT && !POINTS;
    bool bad = false;
    constexpr int NG = M == 3 ? 4 : 2;
    const int point = SPLIT ? (int)(threadIdx.x % NG) : 0; /* SPLIT: this lane's Gauss point */
    const int b0 = SPLIT ? point >> 1 : 0, b1 = SPLIT ? b0 + 1 : NG / 2;
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
        const V sa = V(b ? 0.28867513459481287 : -0.28867513459481287);
        pl = opaque(pl);
        pr = opaque(pr);
        /* face frame: W[g][v], dW[g][e][v]; rref, plim: the cell averages' side of the admissibility test */
        V W[G][NV], dW[G][M][NV], rref[G], plim[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            V kc = V(0), Ec = V(0), r0 = V(0), i0 = V(0);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int gv = (v >= 1 && v <= M) ? 1 + ax[v - 1] : v; /* global variable */
                V c[NC], w, o0[M + 1], o1[M + 1];
#pragma unroll
                for (int k = 0; k < NC; ++k) c[k] = FV::load(pl, pr, g, (gv * (NC + 1) + k) * 32);
                w = FV::load(pl, pr, g, (gv * (NC + 1) + NC) * 32);
                if (v == 0) {
                    r0 = w;
                    i0 = V(1) / w;
                } else if (v <= M) kc += w * (w * i0);
                else Ec = w;
                face_pair<V, M, D>(c, w, FV::sign(g), sa, o0, o1);
                if constexpr (SPLIT) {
                    W[g][v] = point & 1 ? o1[0] : o0[0];
#pragma unroll
                    for (int e = 0; e < M; ++e) dW[g][e][v] = point & 1 ? o1[1 + e] : o0[1 + e];
                } else {
                    W[g][v] = o0[0];
                    stash[(g * NV + v) * (M + 1) * SS] = o1[0];
#pragma unroll
                    for (int e = 0; e < M; ++e) {
                        dW[g][e][v] = o0[1 + e];
                        stash[((g * NV + v) * (M + 1) + 1 + e) * SS] = o1[1 + e];
                    }
                }
            }
            rref[g] = G == 1 ? i0 : V(V(adm) * r0);
            plim[g] = V(G == 1 ? adm : R(adm * P.fp.gm1)) * (Ec - V(0.5) * kc);
        }
#pragma unroll
        for (int p = 0; p < (SPLIT ? 1 : 2); ++p) {
            if (p) {
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        W[g][v] = stash[(g * NV + v) * (M + 1) * SS];
#pragma unroll
                        for (int e = 0; e < M; ++e) dW[g][e][v] = stash[((g * NV + v) * (M + 1) + 1 + e) * SS];
                    }
                if constexpr (PARK) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        stash[3 * v * SS] = V(F[v], Ft[v]);
                        stash[(3 * v + 1) * SS] = V(Wh[v], 0.f);
                    }
                }
            }
            auto average = [&](int g, int v) -> V {
                const int gv = (v >= 1 && v <= M) ? 1 + ax[v - 1] : v;
                return FV::load(opaque(pl), opaque(pr), g, (gv * (NC + 1) + NC) * 32);
            };
            R f[NV], ft[NV], wh[NV];
            const bool ok = face_point<R, M, NS>(P.fp, adm, dt, idt, ih, W, dW, rref, plim, average, f, ft, wh);
            if constexpr (POINTS) {
                const int point_at = SPLIT ? point : p + 2 * b;
                if (store) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const int gv = (v >= 1 && v <= M) ? 1 + ax[v - 1] : v;
                        const bool none = !ok || (wall() && (v == 0 || v == NV - 1));
                        R *o = ff + ((long)gv * NG + point_at) * P.nftot + (unsigned)P.foff[D] + fl;
                        o[0] = none ? R(0) : f[v];
                        o[(long)NV * NG * P.nftot] = none ? R(0) : ft[v];
                        o[2l * NV * NG * P.nftot] = ok ? wh[v] : R(0);
                    }
                }
            } else {
                if constexpr (PARK) {
                    if (p) {
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            const V a = stash[3 * v * SS];
                            F[v] = a.l();
                            Ft[v] = a.r();
                            Wh[v] = stash[(3 * v + 1) * SS].l();
                        }
                    }
                }
                if (ok) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        F[v] += f[v];
                        Ft[v] += ft[v];
                        Wh[v] += wh[v];
                    }
                }
            }
            bad = bad || !ok;
        }
    }
    if (bad) atomicOr(status, ST_FLUX);
    if constexpr (POINTS) return;
    if constexpr (SPLIT) {
#pragma unroll
        for (int o = 1; o < NG; o <<= 1)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                F[v] += __shfl_xor_sync(0xffffffffu, F[v], o);
                Ft[v] += __shfl_xor_sync(0xffffffffu, Ft[v], o);
                Wh[v] += __shfl_xor_sync(0xffffffffu, Wh[v], o);
            }
        if (!store || point != 0) return;
    }
    if (wall()) F[0] = F[NV - 1] = Ft[0] = Ft[NV - 1] = R(0);
    R *o = ff + group_off<kFaceFields<M>>((unsigned)P.foff[D] + fl);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const int gv = (v >= 1 && v <= M) ? 1 + ax[v - 1] : v;
        o[gv * 32] = F[v];
        o[(NV + gv) * 32] = Ft[v];
        o[(2 * NV + gv) * 32] = Wh[v];
    }
}

/* All faces of a stage in one launch, in the order of FaceOrder.
 * Threads per block and resident blocks asked of the compiler, measured: 64
 * threads spread a small grid over twice the SMs of 128 (equal on large
 * ones).  FP32 2D Euler 12 blocks (80 registers: 0.481 ms per 2048^2 launch;
 * 10 and 16 blocks 0.49 and 0.55), 3D 8 (128 registers: 8.0 ms per 256^3 launch;
 * 6 and 10 blocks 9.7 and 10.0), Navier-Stokes 8 (0.203 ms per 99 x 64 x 50
 * launch; 10 blocks 0.25).  Spilled at these caps (bytes stored / loaded): 2D Euler
 * 16 / 16, 3D Euler 4 / 4, 3D Navier-Stokes 28 / 40, with every point written (gks_flux)
 * 20 / 20, 0 and 44 / 60; the batch's copy of the 2D flux 124 / 132 (k2d_batch.cu).  The points of a pair are
 * unrolled: as a loop the packed constants stay in registers across it (2D
 * 0.54, 3D 9.0 ms).  FP64 is bound by its pipe: 4 to 6 blocks are equal, but
 * for spills (2D Navier-Stokes 4 blocks, 174 registers; 5 and 6 both cap at 168
 * and spill 190 bytes, as warps come in fours).  FP64 registers: 2D 158 (a lane per
 * point 132), Navier-Stokes 174 (148), 3D 224 (210), Navier-Stokes 255 with 4 bytes
 * spilled (210). */
constexpr int kStepFluxBlock = 64;
template <typename R, int M, bool NS>
constexpr int kStepFluxMinBlocks = sizeof(R) == sizeof(float) ? (M == 2 && !NS ? 12 : 8) : (M == 2 && !NS ? 6 : 4);

/* The order of the flux blocks.  2D: runs of kFaceRun blocks of one direction,
 * then the same run of the other, which finds its cells' records in L2 (2048
 * blocks: 20 MB of records); what is left after the shorter direction's whole
 * runs follows direction by direction.  FP32 2048^2 467 to 455 us a launch,
 * 1003 x 777 99 to 92 us.  3D: direction by direction (in runs, whose records
 * are 50 MB, 256^3 takes 8.59 ms for 7.88). */
constexpr unsigned kFaceRun = 2048;
struct FaceOrder {
    unsigned runs;    /* whole runs of every direction */
    unsigned left[2]; /* blocks of directions 0 and 1 past them */
    template <int M> __device__ __forceinline__ void at(unsigned b, unsigned &dir, unsigned &block) const
    {
        const unsigned whole = runs * (M * kFaceRun);
        if (b < whole) {
            const unsigned r = b / kFaceRun;
            dir = r % M;
            block = (r / M) * kFaceRun + b % kFaceRun;
            return;
        }
        b -= whole;
        dir = b < left[0] ? 0 : (M == 2 || b < left[0] + left[1] ? 1 : 2);
        block = runs * kFaceRun + b - (dir == 0 ? 0 : left[0]) - (dir == 2 ? left[1] : 0);
    }
};

/* SPLIT: a lane per Gauss point, 64 / NG faces a block */
template <typename R, int M, bool NS, bool SPLIT, bool POINTS = false>
__global__ void __launch_bounds__(kStepFluxBlock, (kStepFluxMinBlocks<R, M, NS>))
    step_flux_kernel(KP P, const R *B, const double *dtp, R *ff, int *status, FaceOrder order, bool rev)
{
    constexpr int BT = kStepFluxBlock, PER = SPLIT ? (M == 3 ? 4 : 2) : 1, FB = BT / PER;
    __shared__ typename FaceV<R>::V slots[SPLIT ? 1 : kFaceStash<R, M> * BT];
    after_previous();
    typename FaceV<R>::V *stash = SPLIT ? slots : slots + threadIdx.x;
    const R dt = R(dtp[0]), idt = R(dtp[1]);
    unsigned dir, block;
    order.at<M>(block_in_order(rev), dir, block);
    auto face = [&](auto dir, unsigned block) {
        constexpr int D = decltype(dir)::value;
        const unsigned fl = block * FB + threadIdx.x / PER, n = (unsigned)P.nface[D];
        if constexpr (SPLIT) step_face_item<R, M, D, NS, BT, true, POINTS>(P, B, dt, idt, ff, status, fl < n ? fl : n - 1, stash, fl < n);
        else if (fl < n) step_face_item<R, M, D, NS, BT, false, POINTS>(P, B, dt, idt, ff, status, fl, stash);
    };
    if (dir == 0) face(std::integral_constant<int, 0>{}, block);
    else if (M == 2 || dir == 1) face(std::integral_constant<int, 1>{}, block);
    else if constexpr (M == 3) face(std::integral_constant<int, 2>{}, block);
}

/* the stage update from the face sums of step_face_item; wn receives the new averages */
template <typename R, int M, int STAGE>
__device__ __forceinline__ void step_update_item(const KP &P, const R *ff, double dt, double *W,
                                                 double *G, double *Ws, double *Gs,
                                                 double *Acc, const Shadow &s0, const Shadow &s1,
                                                 int *status, long cell, const UpdC &uc, R *wn)
{
    constexpr int NV = M + 2;
    unsigned q0, q1;
    const int i = (int)fdivmod(P.dn[0], (unsigned)cell, q0);
    const int j = (int)fdivmod(P.dn[1], q0, q1);
    const int k = (M >= 3) ? (int)q1 : 0;
    const R *fm[M], *fp[M];
#pragma unroll
    for (int d = 0; d < M; ++d) {
        fm[d] = ff + group_off<kFaceFields<M>>((unsigned)face_of<M>(P, d, i, j, k, 0));
        fp[d] = ff + group_off<kFaceFields<M>>((unsigned)face_of<M>(P, d, i, j, k, 1));
    }
    auto fsum = [&](int q, int v, int d, int plus) -> R { return (plus ? fp[d] : fm[d])[(q * NV + v) * 32]; };
    if constexpr (sizeof(R) == sizeof(float))
        mixed_update_cell<M, STAGE>(P, fsum, uc, W, (float *)Acc, s0, s1, status, cell, wn);
    else
        fp64_update_cell<M, STAGE>(P, fsum, 1.0 / (M == 2 ? 2 : 4), dt, W, G, Ws, Gs, Acc, status, cell, wn);
}

/* SPEED: the new state's wave speed into smax as well (the last stage of a CFL
 * step that another follows), from the values that wavespeed_kernel would read */
template <typename R, int M, int STAGE, bool SPEED>
__global__ void __launch_bounds__(256) step_update_kernel(KP P, const R *ff, const double *dtp, double *W, double *G,
                                                          double *Ws, double *Gs, double *Acc, Shadow s0, Shadow s1,
                                                          int *status, const float *updc, unsigned long long *smax, bool rev)
{
    after_previous();
    UpdC uc;
    if constexpr (sizeof(R) == sizeof(float)) uc = load_updc(updc);
    const long cell = (long)block_in_order(rev) * blockDim.x + threadIdx.x;
    R wn[M + 2], s = R(0), ir = R(0);
    if (cell < P.ncell) {
        step_update_item<R, M, STAGE>(P, ff, dtp[0], W, G, Ws, Gs, Acc, s0, s1, status, cell, uc, wn);
        if constexpr (SPEED) {
            s = fmax(R(0), speed_of<M, R>(wn, pick<R>(P.gamma, (float)(P.fgm1 + 1.0f)))); /* a NaN counts as 0 */
            ir = fmax(R(0), R(1) / wn[0]);
        }
    }
    if constexpr (SPEED) block_speed_max<R>(s, ir, smax);
}

} // namespace gks
