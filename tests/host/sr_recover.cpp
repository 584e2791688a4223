// Relativistic recovery in double-float (sr_recover) against the float64
// iteration it stands for (sr_prim_mixed), on the host: argv = family, states,
// seed.  Prints: states, undecided among the physical ones, values that differ.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <random>

#include "sr_df.cuh"

using namespace ctu;

int main(int argc, char **argv)
{
    const int family = std::atoi(argv[1]);
    const long count = std::atol(argv[2]);
    std::mt19937_64 gen(std::atoi(argv[3]));
    auto uni = [&] { return (double)(gen() >> 11) / 9007199254740992.0; };
    auto sym = [&](double s) { return s * (2.0 * uni() - 1.0); };
    const double gam = family == 3 ? 5.0 / 3.0 : 4.0 / 3.0;
    auto pair = [](double x) { return df{(float)x, (float)(x - (double)(float)x)}; };
    const df g1 = pair((gam - 1.0) / gam), ig = pair(gam / (gam - 1.0));
    long undecided = 0, wrong = 0, physical = 0, fwrong = 0;
    for (long i = 0; i < count; ++i) {
        double v[9];
        if (family <= 2) {  // beam, its edge, the ambient medium beside it
            const double prof = family == 0 ? 0.95 + 0.1 * uni() : family == 1 ? uni() : uni() < 0.3 ? 0.0 : std::exp(-38.0 * uni());
            const double lor = 1.0 + 9.0 * prof, off = family == 2 ? 0.01 : 0.05;
            v[0] = (0.01 + 0.99 * prof) * (1.0 + sym(0.01));
            v[1] = sym(off) * std::fmin(prof, 0.2);
            v[2] = sym(off) * std::fmin(prof, 0.2);
            v[3] = std::sqrt(1.0 - 1.0 / (lor * lor)) * (1.0 - 0.001 * prof);
            v[4] = 0.01 * (1.0 + sym(family == 2 ? 0.0 : 0.5));
            v[5] = family == 2 ? 0.0 : sym(0.3);
            v[6] = family == 2 ? 0.0 : sym(0.3);
            v[7] = 3.225 + sym(family == 2 ? 0.0 : 0.1);
            v[8] = sym(0.01);
        } else {  // any direction, speed, temperature and magnetisation
            const double s = std::pow(uni(), 0.3) * 0.995, c = sym(1.0), f = 6.283185307179586 * uni();
            const double r = std::sqrt(1.0 - c * c), b = std::exp(5.0 * uni() - 4.0);
            v[0] = std::exp(6.0 * uni() - 3.0);
            v[1] = s * r * std::cos(f);
            v[2] = s * r * std::sin(f);
            v[3] = s * c;
            v[4] = std::exp(10.0 * uni() - 7.0);
            for (int k = 5; k < 9; ++k) v[k] = b * sym(1.0);
        }
        float V[9], T[9];
        for (int q = 0; q < 9; ++q) V[q] = (float)v[q];
        double Uc[9], U[9], ref[9];
        sr_cons<double, float>(V, gam, Uc);
        for (int q = 0; q < 9; ++q) {
            T[q] = (float)(sym(family == 2 && (i & 1) ? 0.0 : 1e-5) * Uc[q]);
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
        fwrong += d2f_int(U[4]) != (float)U[4];
        physical += st == 0;
        if (!sr_recover(u, w0, g1, got)) {
            undecided += st == 0;
            continue;
        }
        wrong += st != 0;
        for (int q = 0; q < 5; ++q) wrong += (float)ref[q] != got[q];
    }
    std::printf("%ld %ld %ld %ld\n", physical, undecided, wrong, fwrong);
    return 0;
}
