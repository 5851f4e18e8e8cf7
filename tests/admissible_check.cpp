// Host check of the admissibility test (csrc/kernels.cuh, admissible<double, M>:
// products where they surely decide, divisions elsewhere) against its definition
// in long double, through the test-only CUDA stand-in in tests/hostshim: random
// states and averages of magnitudes from 2^-500 to 2^500, averages that are not
// physical among them.  stdout: the number of decisions, how many the definition
// accepts, and how many differ where it is not within 1e-9 of its limits.
#include <cmath>
#include <cstdio>
#include <random>
#include <cuda_runtime.h>

#include "kernels.cuh"

template <int M> static void run(std::mt19937_64 &g, long *count)
{
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    for (int it = 0; it < 100000; ++it) {
        const int k = (int)(500 * u(g)), ke = k + (int)(20 * u(g)); /* densities near 2^k, energies near 2^ke */
        double w[M + 2], c[M + 2];
        for (double *s : {w, c}) {
            s[0] = std::ldexp(1.0 + 0.9 * u(g), k);
            s[M + 1] = std::ldexp(1.0 + 0.9 * u(g), ke);
            const double m = std::sqrt(std::ldexp(s[0], -k) * std::ldexp(s[M + 1], -ke)) * 1.6;
            for (int a = 0; a < M; ++a) s[1 + a] = std::ldexp(m * u(g) * std::sqrt((k + ke) & 1 ? 2.0 : 1.0), (k + ke) >> 1);
        }
        if (it % 10 == 0) c[0] = -c[0];
        if (it % 10 == 1) w[0] = -w[0];
        const double delta = it % 7 ? 0.3 : 0.0;
        long double p = 0, pc = 0;
        for (int a = 0; a < M; ++a) {
            p += (long double)w[1 + a] * w[1 + a];
            pc += (long double)c[1 + a] * c[1 + a];
        }
        p = w[M + 1] - p / w[0] / 2;
        pc = c[M + 1] - pc / c[0] / 2;
        const long double dr = w[0] - (long double)delta * c[0], dp = p - delta * pc, tiny = 1e-9L;
        if (std::fabs(dr) < tiny * std::fabs(w[0]) || std::fabs(dp) < tiny * std::fabs(w[M + 1])) continue;
        ++count[0];
        const bool want = dr > 0 && dp > 0;
        count[1] += want;
        count[2] += want != gks::admissible<double, M>(w, c, delta);
    }
}

int main()
{
    std::mt19937_64 g(20);
    long count[3] = {0, 0, 0};
    run<1>(g, count);
    run<2>(g, count);
    run<3>(g, count);
    std::printf("%ld %ld %ld\n", count[0], count[1], count[2]);
    return 0;
}
