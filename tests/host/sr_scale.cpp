// The relativistic recoveries on states in other units, on the host: argv =
// exponent k (rho, p, m, E by 4^k, B by 2^k), states, seed.  Nothing but the
// exponents may change.  Prints the values of sr_prim64 and sr_prim_mixed (either
// equation of state) that differ from the unscaled state's, scaled.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <random>

#include "sr_df.cuh"

using namespace ctu;

int main(int argc, char **argv)
{
    const int k = std::atoi(argv[1]);
    const long count = std::atol(argv[2]);
    const double s2 = std::ldexp(1.0, 2 * k), s1 = std::ldexp(1.0, k);
    std::mt19937_64 gen(std::atoi(argv[3]));
    auto uni = [&] { return (double)(gen() >> 11) / 9007199254740992.0; };
    auto sym = [&](double s) { return s * (2.0 * uni() - 1.0); };
    long wrong[2] = {0, 0};
    for (long i = 0; i < count; ++i) {
        const double gam = i & 1 ? 4.0 / 3.0 : 0.0;
        const double sp = std::pow(uni(), 0.3) * 0.995, c = sym(1.0), f = 6.283185307179586 * uni();
        const double r = std::sqrt(1.0 - c * c), b = std::exp(3.0 * uni() - 3.0);
        float V[9] = {(float)std::exp(2.0 * uni() - 1.0), (float)(sp * r * std::cos(f)), (float)(sp * r * std::sin(f)),
                      (float)(sp * c), (float)std::exp(6.0 * uni() - 5.0)};
        for (int q = 5; q < 9; ++q) V[q] = (float)(b * sym(1.0));
        double U[9], X[9], a[9], v[9];
        sr_cons<double, float>(V, gam, U);
        for (int q = 0; q < 9; ++q) X[q] = U[q] * (q < 5 ? s2 : s1);
        const double W0 = i % 3 ? (U[4] + U[0]) * (0.5 + 0.6 * uni()) : 0.0;
        for (int m = 0; m < 2; ++m) {
            const unsigned sa = m ? sr_prim_mixed(U, gam, a, W0) : sr_prim64(U, gam, a, W0);
            const unsigned sv = m ? sr_prim_mixed(X, gam, v, W0 * s2) : sr_prim64(X, gam, v, W0 * s2);
            wrong[m] += sa != 0 || sv != 0;
            for (int q = 0; q < 9; ++q) wrong[m] += v[q] != (q == 0 || q == 4 ? a[q] * s2 : q >= 5 ? X[q] : a[q]);
        }
    }
    std::printf("%ld %ld\n", wrong[0], wrong[1]);
    return 0;
}
