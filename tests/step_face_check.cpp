// Host build of the step path's per-face flux (csrc/step_flux.cuh,
// step_face_item: all Gauss points of a face, evaluated in pairs, summed) for
// the CPU tests, through the test-only CUDA stand-in in tests/hostshim,
// against the per-point flux (face_flux_item) of the same state summed over
// the Gauss points.  Arguments: M n0 n1 n2 h limiter mu dt prec, then the six
// boundary types (prec 0: the FP64 items; 1: the FP32 items from the FP32
// shadow of the state, against the FP64 per-point flux).
// stdin: W[nv][cells], G[M][nv][cells].  stdout: per quantity (F, dF/dt,
// W(dt/2)) the largest difference and the largest magnitude, then the two
// status words.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include <cuda_runtime.h>

#include "step_flux.cuh"

template <int M, int D, bool NS> static void reference(const gks::KP &P, const gks::Src<double> &src, const double *B, double dt, double *ff, int *st)
{
    for (long t = 0; t < P.nface[D] * (M == 2 ? 2 : 4); ++t) gks::face_flux_item<double, M, D, true, NS>(P, src, B, dt, nullptr, ff, st, t);
}

template <typename R, int M, int D, bool NS> static void faces(const gks::KP &P, const R *B, double dt, R *ff, int *st)
{
    typename gks::FaceV<R>::V stash[gks::kFaceStash<R, M>];
    for (long f = 0; f < P.nface[D]; ++f)
        gks::step_face_item<R, M, D, NS, 1>(P, B, (R)dt, (R)(1.0 / dt), ff, st, (unsigned)f, stash);
}

template <typename R, int M, bool NS>
static void run(const gks::KP &P, const gks::Src<R> &src, const gks::Src<double> &src64, double dt)
{
    constexpr int NV = M + 2, NG = M == 2 ? 2 : 4, NC = gks::Cubic<double, M>::NC;
    std::vector<double> B((size_t)NV * NC * P.next), ref((size_t)3 * NV * NG * P.nftot);
    std::vector<R> Bs(gks::group_elems(P.next, gks::kCellFields<M>)), ff(gks::group_elems(P.nftot, gks::kFaceFields<M>));
    int s0 = 0, s1 = 0;
    for (long t = 0; t < P.next; ++t) {
        gks::cell_poly_item<double, M>(P, src64, B.data(), t);
        gks::cell_poly_item<R, M, true>(P, src, Bs.data(), t);
    }
    reference<M, 0, NS>(P, src64, B.data(), dt, ref.data(), &s0);
    reference<M, 1, NS>(P, src64, B.data(), dt, ref.data(), &s0);
    faces<R, M, 0, NS>(P, Bs.data(), dt, ff.data(), &s1);
    faces<R, M, 1, NS>(P, Bs.data(), dt, ff.data(), &s1);
    if constexpr (M == 3) {
        reference<M, 2, NS>(P, src64, B.data(), dt, ref.data(), &s0);
        faces<R, M, 2, NS>(P, Bs.data(), dt, ff.data(), &s1);
    }
    for (int q = 0; q < 3; ++q) {
        double far = 0, big = 0;
        for (int v = 0; v < NV; ++v)
            for (long f = 0; f < P.nftot; ++f) {
                double a = 0;
                for (int g = 0; g < NG; ++g) a += ref[((long)(q * NV + v) * NG + g) * P.nftot + f];
                const double b = ff[gks::group_off<gks::kFaceFields<M>>((unsigned)f) + (q * NV + v) * 32];
                far = std::max(far, std::isfinite(b) ? std::fabs(a - b) : HUGE_VAL);
                big = std::max(big, std::fabs(a));
            }
        std::printf("%.17g %.17g\n", far, big);
    }
    std::printf("%d %d\n", s0, s1);
}

template <int M> static void go(gks::KP &P, double dt, int prec, const std::vector<double> &W, const std::vector<double> &G)
{
    std::vector<float> hi(W.size()), lo(W.size()), g(G.begin(), G.end());
    std::vector<double> W32(W.size()), G32(g.begin(), g.end());
    for (size_t i = 0; i < W.size(); ++i) {
        gks::split(W[i], hi[i], lo[i]);
        W32[i] = (double)hi[i] + (double)lo[i];
    }
    const bool ns = P.fp.mu > 0;
    const gks::Src<double> d{W.data(), G.data()}, d32{W32.data(), G32.data()};
    const gks::Src<float> f{hi.data(), lo.data(), g.data()};
    if (prec) ns ? run<float, M, true>(P, f, d32, dt) : run<float, M, false>(P, f, d32, dt);
    else ns ? run<double, M, true>(P, d, d, dt) : run<double, M, false>(P, d, d, dt);
}

int main(int argc, char **argv)
{
    if (argc < 16) return 2;
    const int m = std::atoi(argv[1]), prec = std::atoi(argv[9]);
    gks::KP P{};
    long ncell = 1, next = 1;
    for (int a = 0; a < 3; ++a) {
        P.n[a] = a < m ? std::atoi(argv[2 + a]) : 1;
        P.ext[a] = a < m ? P.n[a] + 2 : 1;
        ncell *= P.n[a];
        next *= P.ext[a];
    }
    P.ncell = ncell;
    P.next = next;
    long off = 0;
    for (int d = 0; d < m; ++d) {
        long f = 1;
        for (int a = 0; a < m; ++a) f *= (a == d) ? P.n[a] + 1 : P.n[a];
        P.nface[d] = f;
        P.foff[d] = off;
        off += f;
    }
    P.nftot = off;
    for (int a = 0; a < 3; ++a)
        for (int s = 0; s < 2; ++s) P.bcs[a][s] = a < m ? std::atoi(argv[10 + 2 * a + s]) : 0;
    P.limiter = std::atoi(argv[6]);
    P.h = std::atof(argv[5]);
    P.ih = 1.0 / P.h;
    P.gamma = 1.4;
    P.C = 20.0;
    P.itanhC = 1.0 / std::tanh(20.0);
    P.eps = 1e-15;
    P.C0 = 8.0;
    P.adm = 0.3;
    P.d0 = 0.85;
    P.ct = 1e-6;
    P.fp.gamma = 1.4;
    P.fp.c1 = 0.05;
    P.fp.c2 = 1.0;
    P.fp.mu = std::atof(argv[7]);
    gks::finalize_kp(P);
    std::vector<double> W((size_t)(m + 2) * ncell), G((size_t)m * (m + 2) * ncell);
    for (double &x : W)
        if (std::scanf("%lf", &x) != 1) return 2;
    for (double &x : G)
        if (std::scanf("%lf", &x) != 1) return 2;
    if (m == 2) go<2>(P, std::atof(argv[8]), prec, W, G);
    else go<3>(P, std::atof(argv[8]), prec, W, G);
    return 0;
}
