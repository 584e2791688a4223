// The FP64 path's relativistic recovery (sr_prim_fp64) and the float64 iteration
// (sr_prim64) on the host, against Newton's iteration in long double: argv =
// largest Lorentz factor, states, seed.  Prints the failures and the mean
// relative error of rho and p of both.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <random>

#include "sr_df.cuh"

using namespace ctu;
using ld = long double;

static void solve(const double (&U)[9], ld gam, ld W, ld &rho, ld &p)
{
    const ld D = U[0], tau = (ld)U[4] + U[0], g1 = (gam - 1) / gam;
    ld m2 = 0, B2 = 0, S = 0, v2, s;
    for (int k = 0; k < 3; ++k) {
        m2 += (ld)U[1 + k] * U[1 + k];
        B2 += (ld)U[5 + k] * U[5 + k];
        S += (ld)U[1 + k] * U[5 + k];
    }
    for (int it = 0; it < 40; ++it) {
        const ld t = S / W;
        v2 = (m2 + t * t * (2 * W + B2)) / ((W + B2) * (W + B2));
        s = std::sqrt(1 - v2);
        rho = D * s;
        p = g1 * (W * (1 - v2) - rho);
        const ld dv2 = -2 * (v2 + t * t / W) / (W + B2), dp = g1 * (1 - v2 + dv2 * (D / (2 * s) - W));
        W -= (W - tau + B2 * (1 + v2) / 2 - p - t * t / 2) / (1 - dp + B2 * dv2 / 2 + t * t / W);
    }
}

int main(int argc, char **argv)
{
    const double top = std::atof(argv[1]), gam = 4.0 / 3.0, g1 = (gam - 1.0) / gam;
    const long count = std::atol(argv[2]);
    std::mt19937_64 gen(std::atoi(argv[3]));
    auto uni = [&] { return (double)(gen() >> 11) / 9007199254740992.0; };
    auto sym = [&](double s) { return s * (2.0 * uni() - 1.0); };
    long failed[2] = {0, 0};
    double err[2] = {0.0, 0.0};
    for (long i = 0; i < count; ++i) {
        const double lor = 1.0 + (top - 1.0) * (0.5 + 0.5 * uni()), sp = std::sqrt(1.0 - 1.0 / (lor * lor));
        const double c = sym(1.0), f = 6.283185307179586 * uni(), r = std::sqrt(1.0 - c * c), b = std::exp(4.0 * uni() - 3.0);
        double V[9] = {std::exp(4.0 * uni() - 2.0), sp * r * std::cos(f), sp * r * std::sin(f), sp * c, std::exp(8.0 * uni() - 6.0),
                       b * sym(1.0), b * sym(1.0), b * sym(1.0), 0.0};
        double U[9], got[2][9];
        sr_cons<double, double>(V, gam, U);
        const double W = (V[0] + V[4] / g1) * lor * lor, W0 = W * (1.0 + sym(1e-3));
        const unsigned st[2] = {sr_prim64(U, gam, got[0], W0),
                                sr_prim_fp64(U, gam, g1, df{(float)g1, (float)(g1 - (double)(float)g1)}, (float)W0, got[1])};
        ld rho, p;
        solve(U, gam, W, rho, p);
        for (int k = 0; k < 2; ++k) {
            failed[k] += st[k] != 0;
            err[k] += std::fmax((double)std::fabs((got[k][0] - rho) / rho), (double)std::fabs((got[k][4] - p) / p)) / count;
        }
    }
    std::printf("%ld %ld %.3e %.3e\n", failed[0], failed[1], err[0], err[1]);
    return 0;
}
