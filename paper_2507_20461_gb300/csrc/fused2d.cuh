/*
 * One stage of the 2D compact GKS with GENO reconstruction as a single
 * kernel (arXiv 2507.20461, Sec. 2: reconstruct, evolve the gas distribution
 * at the interfaces, update the averages by Eq. semifvs and the averaged
 * gradients by Eq. slope), mixed precision: FP32 reconstruction and flux,
 * exact FP32 face sums and double-float / FP64 accumulation.
 *
 * A block owns a strip of TX columns and sweeps it row by row over a chunk
 * of rows, keeping everything between the stage input and the stage output
 * in shared memory:
 *   - a ring of four rows of the stage input (FP32 shadow: hi, lo, grad x,
 *     grad y of the four variables; the strip plus two ghost columns on
 *     each side, mapped and sign-flipped by the boundary conditions),
 *     filled with cp.async one row ahead of its use;
 *   - a ring of two rows of blended GENO cubics (blend_cubic; the strip
 *     plus one column on each side);
 *   - the face values (F, dF/dt, W(dt/2) per Gauss point) of the x faces of
 *     one row and a ring of two rows of y faces.
 * Per row j, two phases separated by block barriers:
 *   A  the cubics of row j + 1 and the stage update of row j - 1
 *      (mixed_update_var), each one item per (cell, variable);
 *   B  the faces of row j: its TX + 1 x faces and the TX y faces between
 *      rows j and j + 1, a face with both its Gauss points per thread
 *      (face_pair, face_point); TX = 62 and 128 threads make it one round.
 * Only the first cubic rows and y faces of a chunk, and the two columns on
 * each side of a strip, are evaluated twice (by both blocks that touch them,
 * from the same inputs by the same instructions, so both get the same bits
 * and every face's flux still leaves one cell and enters the other exactly:
 * the sums of the averages stay conserved to FP64 rounding).  Neither the
 * cubic coefficients nor the face fluxes go through device memory.
 */
#pragma once
#include "step_flux.cuh"

namespace gks {

template <int TX_> struct SweepStrip {
    static constexpr int TX = TX_;
    static constexpr int NV = 4, NC = GENO_NC2;
    /* stage-input rows: the strip plus two ghost columns on each side */
    static constexpr int WX = TX + 4;
    static constexpr int NFIELD = 16; /* hi[v], lo[v], g_x[v], g_y[v] */
    static constexpr int SROW = NFIELD * WX;
    static constexpr int NSLOT = 4;
    /* cubic rows: the strip plus one column on each side */
    static constexpr int CX = TX + 2;
    static constexpr int REC = NV * NC;
    static constexpr int BROW = CX * REC, WROW = CX * NV;
    /* face values: per face F, dF/dt, W(dt/2) of the four variables summed
     * over its Gauss points, global variable order */
    static constexpr int FV = 3 * NV;
    static constexpr int NXF = TX + 1, NYF = TX;
    static constexpr int XROW = NXF * FV, YROW = NYF * FV;
    /* flux work: 32-face blocks of x faces, then of y faces */
    static constexpr int NXB = (NXF + 31) / 32, NYB = (NYF + 31) / 32;
    static constexpr int O_STATE = 0, O_B = O_STATE + NSLOT * SROW, O_W0 = O_B + 2 * BROW, O_XF = O_W0 + 2 * WROW,
                         O_YF = O_XF + XROW, FLOATS = O_YF + 2 * YROW;
    static constexpr size_t SMEM = sizeof(float) * (size_t)FLOATS;
    static_assert(SROW % 4 == 0 && BROW % 4 == 0 && WROW % 4 == 0 && XROW % 4 == 0 && YROW % 4 == 0,
                  "16-byte aligned regions");
};

/* plane of field f of a stage input: f = v (hi), 4 + v (lo), 8 + 4 a + v
 * (gradient along a) */
__device__ __forceinline__ const float *sweep_plane(const Shadow &s, long nc, int f)
{
    return (f < 4) ? s.hi + (long)f * nc : (f < 8) ? s.lo + (long)(f - 4) * nc : s.g + (long)(f - 8) * nc;
}

/* Geometry of one grid: the fields of its parameter block that differ
 * between the grids of a batch (which share every scheme constant). */
struct FusedGeo {
    int nx, ny;
    long nc;
    double ih;
    float fh, fih;
};

/* The stage on the strip of columns x0 .. x0 + TX - 1, rows y0 .. y0 + rows
 * - 1 (clipped to the grid), by the NT threads of the calling block; P holds
 * the scheme constants and boundary types, geo the grid's geometry; smem
 * holds SweepStrip<TX>::FLOATS floats, uc is block-shared.  Every thread of
 * the block calls it. */
template <int STAGE, bool NS, int TX, int NT>
__device__ __forceinline__ void fused2d_strip(const KP &P, const FusedGeo &geo, const Shadow &s0, const Shadow &s1,
                                              double *__restrict__ W, float *__restrict__ acc, double dt,
                                              int *__restrict__ status, int x0, int y0, int rows, float *smem,
                                              UpdC &uc)
{
    using T = SweepStrip<TX>;
    constexpr int NV = T::NV, NC = T::NC, WX = T::WX, CX = T::CX;
    static_assert(NT % 32 == 0, "the four variables of a cell are updated by neighbouring lanes");
    float *const S = smem + T::O_STATE; /* [slot][field][WX] */
    float *const Bc = smem + T::O_B;    /* [slot][cx][v * NC + k] */
    float *const W0 = smem + T::O_W0;   /* [slot][cx][v] signed cell averages (FP32 hi) */
    float *const XF = smem + T::O_XF;   /* [ix][g][12] */
    float *const YF = smem + T::O_YF;   /* [slot][ix][g][12] */

    const Shadow &sin = (STAGE == 1) ? s0 : s1;
    const int nx = geo.nx, ny = geo.ny;
    const long nc = geo.nc;
    const int y1 = min(y0 + rows, ny);
    const int tid = threadIdx.x;
    if (tid == 0) uc = make_updc(dt, geo.ih / 2);
    const bool xin = x0 >= 2 && x0 + TX + 2 <= nx; /* every column of the strip's rows is inside */

    /* stage-input row r into its ring slot; cells that need no sign change
     * are copied with cp.async (completed by cp_wait), mirrored ghost cells
     * whose sign changes are read, negated and stored */
    auto load_row = [&](int r) {
        float *dst = S + (r & 3) * T::SROW;
        const bool rin = r >= 0 && r < ny;
        for (int it = tid; it < T::SROW; it += NT) {
            const int f = it / WX, wx = it - f * WX;
            const int gx = x0 - 2 + wx;
            const float *plane = sweep_plane(sin, nc, f);
            long src;
            bool neg = false;
            if (rin && xin) {
                src = (long)r * nx + gx;
            } else {
                int flip[3] = {0, 0, 0};
                const int ii = map_idx(gx, nx, P.bcs[0][0], P.bcs[0][1], flip[0]);
                const int jj = map_idx(r, ny, P.bcs[1][0], P.bcs[1][1], flip[1]);
                src = (long)jj * nx + ii;
                neg = ghost_sign<2>(P, flip, f & 3) < 0;
                if (f >= 8 && (flip[(f - 8) >> 2] & 1)) neg = !neg;
            }
            if (!neg) {
                const unsigned d = (unsigned)__cvta_generic_to_shared(dst + it);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(plane + src) : "memory");
            } else {
                dst[it] = -plane[src];
            }
        }
    };
    auto cp_wait = [] { asm volatile("cp.async.wait_all;\n" ::: "memory"); };

    /* blended cubic of item it of cubic row r (state rows r - 1 .. r + 1 in the ring) */
    auto recon_item = [&](int r, int it) {
        const int v = it / CX, cx = it - v * CX;
        const float *rm = S + ((r - 1) & 3) * T::SROW, *r0 = S + (r & 3) * T::SROW, *rp = S + ((r + 1) & 3) * T::SROW;
        const int wx = cx + 1;
        const float hr = geo.fh;
        const int fh = v, fl = 4 + v, fgx = 8 + v, fgy = 12 + v;
        const float h0 = r0[fh * WX + wx], l0 = r0[fl * WX + wx];
        float d[GENO_ND2];
        /* q = 2 e + (side > 0): x-, x+, y-, y+ */
        const float *row[4] = {r0, r0, rm, rp};
        const int col[4] = {wx - 1, wx + 1, wx, wx};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            d[q * 3] = (row[q][fh * WX + col[q]] - h0) + (row[q][fl * WX + col[q]] - l0);
            d[q * 3 + 1] = row[q][fgx * WX + col[q]] * hr;
            d[q * 3 + 2] = row[q][fgy * WX + col[q]] * hr;
        }
        d[12] = r0[fgx * WX + wx] * hr;
        d[13] = r0[fgy * WX + wx] * hr;
        float b[NC];
        blend_cubic<float, 2>(P, d, b);
        float *o = Bc + (r & 1) * T::BROW + cx * T::REC + v * NC;
#pragma unroll
        for (int k = 0; k < NC; ++k) o[k] = b[k];
        W0[(r & 1) * T::WROW + cx * NV + v] = h0;
    };

    /* face it of row j (its direction is warp-uniform), both Gauss points.
     * y_only: the y faces between rows j - 1 and j; else the x faces of row j
     * (it < 32 NXB), then the y faces between rows j and j + 1 */
    const float dtf = (float)dt, idt = 1.f / dtf;
    auto flux_item = [&](int j, int it, bool y_only) {
        const bool xd = !y_only && it < 32 * T::NXB;
        const int ix = (xd || y_only) ? it : it - 32 * T::NXB;
        if (xd ? ix >= T::NXF : ix >= T::NYF) return;
        const int yr = y_only ? j : j + 1; /* row of the y faces' upper cells */
        const int fi = x0 + ix;
        if (xd ? (fi > nx || j >= ny) : (fi >= nx || yr > ny)) return;
        const float *cL, *cR, *wL, *wR;
        if (xd) {
            cL = Bc + (j & 1) * T::BROW + ix * T::REC;
            cR = cL + T::REC;
            wL = W0 + (j & 1) * T::WROW + ix * NV;
            wR = wL + NV;
        } else {
            cL = Bc + ((yr - 1) & 1) * T::BROW + (ix + 1) * T::REC;
            cR = Bc + (yr & 1) * T::BROW + (ix + 1) * T::REC;
            wL = W0 + ((yr - 1) & 1) * T::WROW + (ix + 1) * NV;
            wR = W0 + (yr & 1) * T::WROW + (ix + 1) * NV;
        }
        const bool wall = xd ? ((fi == 0 && P.bcs[0][0] >= 2) || (fi == nx && P.bcs[0][1] >= 2))
                             : ((yr == 0 && P.bcs[1][0] >= 2) || (yr == ny && P.bcs[1][1] >= 2));
        /* one copy of the code for both directions: a y face of the cubic
         * P(x, y) is the x face of P(y, x), whose coefficients are P's with x
         * and y swapped (monomials y, x, y^2, xy, x^2, y^3, xy^2, x^2y, x^3),
         * its momenta swapped (selects on the warp-uniform direction) */
        constexpr int swp[NC] = {1, 0, 4, 3, 2, 8, 7, 6, 5};
        LR Wp[2][1][NV], dWp[2][1][2][NV], rc[1], dqc[1];
        {
            float rl[T::REC], rr[T::REC];
#pragma unroll
            for (int k = 0; k < T::REC / 4; ++k) {
                const float4 l = reinterpret_cast<const float4 *>(cL)[k], q = reinterpret_cast<const float4 *>(cR)[k];
                rl[4 * k] = l.x, rl[4 * k + 1] = l.y, rl[4 * k + 2] = l.z, rl[4 * k + 3] = l.w;
                rr[4 * k] = q.x, rr[4 * k + 1] = q.y, rr[4 * k + 2] = q.z, rr[4 * k + 3] = q.w;
            }
            const float4 al = *reinterpret_cast<const float4 *>(wL), ar = *reinterpret_cast<const float4 *>(wR);
            const LR w[NV] = {LR(al.x, ar.x), xd ? LR(al.y, ar.y) : LR(al.z, ar.z), xd ? LR(al.z, ar.z) : LR(al.y, ar.y),
                              LR(al.w, ar.w)};
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int u = (v == 1 || v == 2) ? 3 - v : v; /* the swapped variable */
                LR c[NC], o0[3], o1[3];
#pragma unroll
                for (int k = 0; k < NC; ++k)
                    c[k] = LR(xd ? rl[v * NC + k] : rl[u * NC + swp[k]], xd ? rr[v * NC + k] : rr[u * NC + swp[k]]);
                face_pair<LR, 2, 0>(c, w[v], LR(1.f, -1.f), LR(0.f), o0, o1);
                Wp[0][0][v] = o0[0];
                Wp[1][0][v] = o1[0];
                dWp[0][0][0][v] = o0[1];
                dWp[1][0][0][v] = o1[1];
                dWp[0][0][1][v] = o0[2];
                dWp[1][0][1][v] = o1[2];
            }
            const LR kc = w[1] * w[1] + w[2] * w[2];
            rc[0] = w[0];
            dqc[0] = LR(P.fadm) * (w[0] * w[3] - LR(0.5f) * kc);
        }
        float q[3][NV];
        bool bad = false;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            auto average = [&](int, int v) -> LR {
                const int u = (v == 1 || v == 2) && !xd ? 3 - v : v;
                return LR(wL[u], wR[u]);
            };
            float F[NV], Ft[NV], Wh[NV];
            if (!face_point<float, 2, NS>(P.fp, P.fadm, dtf, idt, geo.fih, Wp[p], dWp[p], rc, dqc, average, F, Ft, Wh)) {
                bad = true;
#pragma unroll
                for (int v = 0; v < NV; ++v) F[v] = Ft[v] = Wh[v] = 0.f;
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                q[0][v] = p ? q[0][v] + F[v] : F[v];
                q[1][v] = p ? q[1][v] + Ft[v] : Ft[v];
                q[2][v] = p ? q[2][v] + Wh[v] : Wh[v];
            }
        }
        if (bad) atomicOr(status, ST_FLUX);
        if (wall) q[0][0] = q[0][NV - 1] = q[1][0] = q[1][NV - 1] = 0.f;
        float *base = xd ? XF : YF + (yr & 1) * T::YROW;
        float4 *o = reinterpret_cast<float4 *>(base + ix * T::FV);
#pragma unroll
        for (int r = 0; r < 3; ++r)
            o[r] = make_float4(q[r][0], xd ? q[r][1] : q[r][2], xd ? q[r][2] : q[r][1], q[r][3]);
    };

    /* stage update of row j, one item per (cell, variable): item t is
     * variable t % 4 of cell t / 4 (the four variables of a cell in four
     * neighbouring lanes, which then gather the new state for its
     * admissibility flags).  Faces: x faces of row j, y faces below (slot of
     * row j) and above (slot of row j + 1).  Every thread of the block calls it. */
    auto update_row = [&](int j) {
        for (int it = tid; it < (NV * TX + NT - 1) / NT * NT; it += NT) {
            const int tx = it >> 2, v = it & 3;
            const int gx = x0 + tx;
            const bool valid = it < NV * TX && gx < nx && j < ny;
            float wn = 1.f;
            if (valid) {
                const float *ylo = YF + (j & 1) * T::YROW, *yhi = YF + ((j + 1) & 1) * T::YROW;
                auto fsum = [&](int q, int vv, int d, int plus) -> float {
                    const float *p = d == 0 ? XF + (tx + plus) * T::FV : (plus ? yhi : ylo) + tx * T::FV;
                    return p[q * NV + vv];
                };
                wn = mixed_update_var<2, STAGE>(nc, geo.fih, fsum, uc, W, acc, s0, s1, (long)j * nx + gx, v);
            }
            const int base = (tid & 31) & ~3;
            float w4[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) w4[k] = __shfl_sync(0xffffffffu, wn, base + k);
            if (valid && v == 0) mixed_state_flags<2>(P, w4, status);
        }
    };

    /* The sweep, one loop for the whole chunk.  Iteration j: phase A, the
     * cubics of row j + 1 and the update of row j - 1; phase B, the load of
     * input row j + 3 and the faces of row j (the x faces of row j and the y
     * faces between rows j and j + 1).  The first two iterations are the
     * prologue (j = y0 - 2: cubic row y0 - 1 only; j = y0 - 1: cubic row y0
     * and the y faces below row y0), the last one the epilogue (j = y1: the
     * update of row y1 - 1 only).  A cubic row or a face on a chunk's edge
     * is also computed by the neighbouring chunk, and conservation needs
     * both results bit-identical: every cubic and every face therefore comes
     * from the one copy of recon_item / flux_item in this loop.  The row
     * index and its phase are opaque values, so the compiler can neither
     * peel the first iterations nor specialise a copy of the code for them. */
    for (int r = y0 - 2; r <= y0; ++r) load_row(r);
    cp_wait();
    __syncthreads();
#pragma unroll 1
    for (int jl = y0 - 2; jl <= y1; ++jl) {
        int j = jl;
        asm volatile("" : "+r"(j));
        /* 0: a full row; 1: cubics and the y faces below row y0; 2: cubics
         * only; 3: the last update only */
        int phase = j >= y1 ? 3 : (j >= y0 ? 0 : (j == y0 - 1 ? 1 : 2));
        asm volatile("" : "+r"(phase));
        /* A: cubics of row j + 1; update of row j - 1 */
        if (phase != 3)
            for (int it = tid; it < NV * CX; it += NT) recon_item(j + 1, it);
        if (j > y0) update_row(j - 1);
        if (phase == 3) break;
        __syncthreads();
        /* B: faces of row j; input row j + 3 in flight meanwhile (the slot
         * of row j - 1, which phase A no longer reads) */
        if (j + 1 < y1) load_row(j + 3);
        if (phase != 2) {
            const bool yo = phase == 1;
            const int nfi = 32 * (yo ? T::NYB : T::NXB + T::NYB);
            for (int it = tid; it < nfi; it += NT) flux_item(yo ? y0 : j, it, yo);
        }
        cp_wait();
        __syncthreads();
    }
}

} // namespace gks
