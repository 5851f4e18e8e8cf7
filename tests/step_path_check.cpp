// Host build of a multi-D step from the item functions that the step's kernels
// run (csrc/kernels.cuh, cell_poly_item in its grouped layout; csrc/step_flux.cuh,
// step_face_item and step_update_item) for the CPU tests, through the test-only
// CUDA stand-in in tests/hostshim: both stages item by item in plain loops.
// Arguments: M n0 n1 n2 h limiter mu prec, then the six boundary types (prec 1:
// mixed precision, FP32 items and shadows and the FP64 state).  stdin: dt,
// W[nv][cells], G[M][nv][cells].  stdout: W then G after the step (one line
// each), then the status word.
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

template <typename R, int M, bool NS> static int step(gks::KP &P, double dt, std::vector<double> &W, std::vector<double> &G)
{
    const long nc = P.ncell;
    std::vector<double> Ws(W.size()), Gs(G.size()), Acc(W.size());
    std::vector<float> h0(W.size()), l0(W.size()), g0(G.begin(), G.end()), h1(W.size()), l1(W.size()), g1(G.size());
    for (size_t i = 0; i < W.size(); ++i) gks::split(W[i], h0[i], l0[i]);
    const gks::Shadow s0{h0.data(), l0.data(), g0.data()}, s1{h1.data(), l1.data(), g1.data()};
    std::vector<R> B(gks::group_elems(P.next, gks::kCellFields<M>)), ff(gks::group_elems(P.nftot, gks::kFaceFields<M>));
    const gks::UpdC uc = gks::make_updc(dt, gks::updc_cw(P, M));
    int status = 0;
    for (int stage = 1; stage <= 2; ++stage) {
        gks::Src<R> src;
        if constexpr (sizeof(R) == sizeof(float)) src = stage == 1 ? gks::Src<float>{s0.hi, s0.lo, s0.g} : gks::Src<float>{s1.hi, s1.lo, s1.g};
        else src = stage == 1 ? gks::Src<double>{W.data(), G.data()} : gks::Src<double>{Ws.data(), Gs.data()};
        for (long t = 0; t < P.next; ++t) gks::cell_poly_item<R, M, true>(P, src, B.data(), t);
        faces<R, M, 0, NS>(P, B.data(), dt, ff.data(), &status);
        faces<R, M, 1, NS>(P, B.data(), dt, ff.data(), &status);
        if constexpr (M == 3) faces<R, M, 2, NS>(P, B.data(), dt, ff.data(), &status);
        R wn[M + 2];
        for (long c = 0; c < nc; ++c) {
            if (stage == 1)
                gks::step_update_item<R, M, 1>(P, ff.data(), dt, W.data(), G.data(), Ws.data(), Gs.data(), Acc.data(), s0, s1, &status, c, uc, wn);
            else
                gks::step_update_item<R, M, 2>(P, ff.data(), dt, W.data(), G.data(), Ws.data(), Gs.data(), Acc.data(), s0, s1, &status, c, uc, wn);
        }
    }
    if (sizeof(R) == sizeof(float))
        for (size_t i = 0; i < G.size(); ++i) G[i] = g0[i];
    return status;
}

template <int M> static int go(gks::KP &P, int prec, double dt, std::vector<double> &W, std::vector<double> &G)
{
    const bool ns = P.fp.mu > 0;
    if (prec) return ns ? step<float, M, true>(P, dt, W, G) : step<float, M, false>(P, dt, W, G);
    return ns ? step<double, M, true>(P, dt, W, G) : step<double, M, false>(P, dt, W, G);
}

int main(int argc, char **argv)
{
    if (argc < 15) return 2;
    const int m = std::atoi(argv[1]), prec = std::atoi(argv[8]);
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
        for (int s = 0; s < 2; ++s) P.bcs[a][s] = a < m ? std::atoi(argv[9 + 2 * a + s]) : 0;
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
    double dt;
    if (std::scanf("%lf", &dt) != 1) return 2;
    std::vector<double> W((size_t)(m + 2) * ncell), G((size_t)m * (m + 2) * ncell);
    for (double &x : W)
        if (std::scanf("%lf", &x) != 1) return 2;
    for (double &x : G)
        if (std::scanf("%lf", &x) != 1) return 2;
    const int st = m == 2 ? go<2>(P, prec, dt, W, G) : go<3>(P, prec, dt, W, G);
    for (size_t i = 0; i < W.size(); ++i) std::printf("%.17g%c", W[i], i + 1 < W.size() ? ' ' : '\n');
    for (size_t i = 0; i < G.size(); ++i) std::printf("%.17g%c", G[i], i + 1 < G.size() ? ' ' : '\n');
    std::printf("%d\n", st);
    return 0;
}
