// Host build of the step path's face flux (csrc/step_flux.cuh, step_face_item;
// 1D: csrc/kernels.cuh, flux1d_face) for the CPU tests, through the test-only
// CUDA stand-in in tests/hostshim: the same state twice, as given and with
// every average, gradient and the viscosity times 2^k.  Arguments: M n0 n1 n2 h
// limiter mu dt prec k, then the six boundary types (prec 1: the FP32 items on
// the state's FP32 shadow).  stdin: W[nv][cells], G[M][nv][cells].
// stdout: per quantity (F, dF/dt, W(dt/2)) the largest difference of the second
// run's result over 2^k from the first's, and the largest magnitude, then the
// two status words.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include <cuda_runtime.h>

#include "step_flux.cuh"

template <typename R, int M, int D, bool NS> static void faces(const gks::KP &P, const R *B, double dt, R *ff, int *st)
{
    typename gks::FaceV<R>::V stash[gks::kFaceStash<R, M>];
    for (long f = 0; f < P.nface[D]; ++f)
        gks::step_face_item<R, M, D, NS, 1>(P, B, (R)dt, (R)(1.0 / dt), ff, st, (unsigned)f, stash);
}

// out[q][v][face]
template <typename R, int M, bool NS>
static std::vector<double> fluxes(const gks::KP &P, double dt, const std::vector<double> &W, const std::vector<double> &G, int *st)
{
    constexpr int NV = M + 2;
    std::vector<double> out((size_t)3 * NV * P.nftot);
    if constexpr (M == 1) {
        for (long f = 0; f < P.nftot; ++f) {
            R q[3][3];
            gks::flux1d_face<R, NS>(P, W.data(), G.data(), (int)f, (R)dt, st, q[0], q[1], q[2]);
            for (int i = 0; i < 9; ++i) out[(size_t)i * P.nftot + f] = q[i / 3][i % 3];
        }
    } else {
        std::vector<float> hi(W.size()), lo(W.size()), g(G.begin(), G.end());
        for (size_t i = 0; i < W.size(); ++i) gks::split(W[i], hi[i], lo[i]);
        gks::Src<R> src;
        if constexpr (sizeof(R) == sizeof(float)) src = gks::Src<float>{hi.data(), lo.data(), g.data()};
        else src = gks::Src<double>{W.data(), G.data()};
        std::vector<R> B(gks::group_elems(P.next, gks::kCellFields<M>)), ff(gks::group_elems(P.nftot, gks::kFaceFields<M>));
        for (long t = 0; t < P.next; ++t) gks::cell_poly_item<R, M, true>(P, src, B.data(), t);
        faces<R, M, 0, NS>(P, B.data(), dt, ff.data(), st);
        faces<R, M, 1, NS>(P, B.data(), dt, ff.data(), st);
        if constexpr (M == 3) faces<R, M, 2, NS>(P, B.data(), dt, ff.data(), st);
        for (int i = 0; i < 3 * NV; ++i)
            for (long f = 0; f < P.nftot; ++f)
                out[(size_t)i * P.nftot + f] = ff[gks::group_off<gks::kFaceFields<M>>((unsigned)f) + i * 32];
    }
    return out;
}

template <typename R, int M> static void go(gks::KP P, double dt, int k, std::vector<double> W, std::vector<double> G)
{
    const bool ns = P.fp.mu > 0;
    int s0 = 0, s1 = 0;
    const std::vector<double> a = ns ? fluxes<R, M, true>(P, dt, W, G, &s0) : fluxes<R, M, false>(P, dt, W, G, &s0);
    for (double &x : W) x = std::ldexp(x, k);
    for (double &x : G) x = std::ldexp(x, k);
    P.fp.mu = std::ldexp(P.fp.mu, k);
    gks::finalize_kp(P);
    const std::vector<double> b = ns ? fluxes<R, M, true>(P, dt, W, G, &s1) : fluxes<R, M, false>(P, dt, W, G, &s1);
    const size_t part = a.size() / 3;
    for (int q = 0; q < 3; ++q) {
        double far = 0, big = 0;
        for (size_t i = q * part; i < (q + 1) * part; ++i) {
            far = std::max(far, std::isfinite(b[i]) ? std::fabs(std::ldexp(b[i], -k) - a[i]) : HUGE_VAL);
            big = std::max(big, std::fabs(a[i]));
        }
        std::printf("%.17g %.17g\n", far, big);
    }
    std::printf("%d %d\n", s0, s1);
}

int main(int argc, char **argv)
{
    if (argc < 17) return 2;
    const int m = std::atoi(argv[1]), prec = std::atoi(argv[9]), k = std::atoi(argv[10]);
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
        for (int s = 0; s < 2; ++s) P.bcs[a][s] = a < m ? std::atoi(argv[11 + 2 * a + s]) : 0;
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
    const double dt = std::atof(argv[8]);
    if (m == 1) prec ? go<float, 1>(P, dt, k, W, G) : go<double, 1>(P, dt, k, W, G);
    else if (m == 2) prec ? go<float, 2>(P, dt, k, W, G) : go<double, 2>(P, dt, k, W, G);
    else prec ? go<float, 3>(P, dt, k, W, G) : go<double, 3>(P, dt, k, W, G);
    return 0;
}
