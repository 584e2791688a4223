// The double-float recovery (sr_recover) against the float64 iteration
// (sr_prim_mixed) on states in other units, on the host as the device runs it:
// float32 denormals flushed (linked so), the approximate reciprocal and root up to
// SEED_ULPS off.  argv = exponent k (rho, p by 4^k, B by 2^k), states, seed.
// Prints: denormals flushed, physical states, undecided among them, values that differ.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <random>

#include "sr_df.cuh"

using namespace ctu;

int main(int argc, char **argv)
{
    const double s2 = std::ldexp(1.0, 2 * std::atoi(argv[1])), s1 = std::ldexp(1.0, std::atoi(argv[1]));
    const long count = std::atol(argv[2]);
    std::mt19937_64 gen(std::atoi(argv[3]));
    auto uni = [&] { return (double)(gen() >> 11) / 9007199254740992.0; };
    auto sym = [&](double s) { return s * (2.0 * uni() - 1.0); };
    const double gam = 4.0 / 3.0;
    auto pair = [](double x) { return df{(float)x, (float)(x - (double)(float)x)}; };
    const df g1 = pair((gam - 1.0) / gam), ig = pair(gam / (gam - 1.0));
    volatile float tiny = 1.2e-38f;
    const int flushed = (float)(tiny * 0.5f) == 0.0f;
    long undecided = 0, wrong = 0, physical = 0;
    for (long i = 0; i < count; ++i) {
        float V[9], T[9];
        if (i & 1) {  // the beam's edge
            const double prof = uni(), lor = 1.0 + 9.0 * prof, off = 0.05 * std::fmin(prof, 0.2);
            const double v[9] = {0.01 + 0.99 * prof, sym(off), sym(off), std::sqrt(1.0 - 1.0 / (lor * lor)) * (1.0 - 0.001 * prof),
                                 0.01 * (1.0 + sym(0.5)), sym(0.3), sym(0.3), 3.225 + sym(0.1), sym(0.01)};
            for (int q = 0; q < 9; ++q) V[q] = (float)v[q];
        } else {  // any direction, speed, temperature and magnetisation
            const double sp = std::pow(uni(), 0.3) * 0.995, c = sym(1.0), f = 6.283185307179586 * uni();
            const double r = std::sqrt(1.0 - c * c), b = std::exp(5.0 * uni() - 4.0);
            V[0] = (float)std::exp(6.0 * uni() - 3.0);
            V[1] = (float)(sp * r * std::cos(f));
            V[2] = (float)(sp * r * std::sin(f));
            V[3] = (float)(sp * c);
            V[4] = (float)std::exp(10.0 * uni() - 7.0);
            for (int q = 5; q < 9; ++q) V[q] = (float)(b * sym(1.0));
        }
        V[0] *= (float)s2;
        V[4] *= (float)s2;
        for (int q = 5; q < 9; ++q) V[q] *= (float)s1;
        double Uc[9], U[9], ref[9];
        sr_cons<double, float>(V, gam, Uc);
        for (int q = 0; q < 9; ++q) {
            T[q] = (float)(sym(1e-5) * Uc[q]);
            U[q] = Uc[q] + (double)T[q];
        }
        const double W0 = sr_w<double>(V[0], V[4], gam) *
                          rcp64(1.0 - ((double)V[1] * V[1] + (double)V[2] * V[2] + (double)V[3] * V[3]));
        SrState u;
        float w0 = 0.0f, got[5];
        unsigned st;
        if (i % 3) {  // from a predicted state, with its W as the guess
            st = sr_prim_mixed(U, gam, ref, W0);
            sr_state_of(V, T, ig, u, w0);
        } else {  // from a stored float64 state, without a guess
            st = sr_prim_mixed(U, gam, ref, 0.0);
            u.D = sr_split(U[0]);
            u.tau = d_add(sr_split(U[4]), u.D);
            for (int k = 0; k < 3; ++k) {
                u.m[k] = sr_split(U[1 + k]);
                u.b[k] = sr_split(U[5 + k]);
            }
        }
        physical += st == 0;
        if (!sr_recover(u, w0, g1, got)) {
            undecided += st == 0;
            continue;
        }
        wrong += st != 0;
        for (int q = 0; q < 5; ++q) wrong += (float)ref[q] != got[q];
    }
    std::printf("%d %ld %ld %ld\n", flushed, physical, undecided, wrong);
    return 0;
}
