// The float64 forms of mhd_fp64.cuh on the host beside the generic functions they
// stand for (mhd_device.cuh), instantiated in long double.
// Every number of the inputs in turn is a quiet nan of either sign; prints the
// outputs that are numbers here and nans there, and those that are nans in both.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <limits>
#include <random>

using std::copysign;
using std::sqrt;
using ld = long double;
#include "mhd_fp64.cuh"

namespace ctu {
template <> struct Tol<ld> {
    static ld bt() { return 1.0e-24L; }
    static ld hlld() { return 1.0e-12L; }
};
} // namespace ctu
using namespace ctu;

template <class R> static void predict(const double (&vs)[5][NV], bool ppm, bool hyb, int mode, int lim, R (&P)[NV], R (&M)[NV])
{
    R v[5][NV];
    for (int m = 0; m < 5; ++m)
        for (int q = 0; q < NV; ++q) v[m][q] = vs[m][q];
    const R gam = R(5.0 / 3.0), ch = R(3.0), dtdx = R(0.0625);
    if (hyb)
        char_predict<R, RECON_PPM_HYB>(v, gam, ch, dtdx, mode, lim, R(0), P, M);
    else if (ppm)
        char_predict<R, RECON_PPM>(v, gam, ch, dtdx, mode, lim, R(0), P, M);
    else
        char_predict<R, RECON_MC>(v, gam, ch, dtdx, mode, lim, R(0), P, M);
}

struct Gen {
    std::mt19937_64 gen;
    double uni() { return (double)(gen() >> 11) / 9007199254740992.0; }
    double sym(double s) { return s * (2.0 * uni() - 1.0); }
    void state(double (&V)[NV], const double (&c)[NV], double s)
    {
        for (int q = 0; q < NV; ++q) V[q] = c[q] + sym(s);
        V[0] = std::exp(0.5 * V[0]);
        V[4] = std::exp(0.5 * V[4]);
    }
    void center(double (&c)[NV])
    {
        for (double &x : c) x = sym(2.0);
    }
};

int main()
{
    Gen g;
    long lost = 0, both = 0;
    for (int it = 0; it < 200; ++it) {
        double c[NV], vs[5][NV];
        g.center(c);
        for (auto &v : vs) g.state(v, c, 0.5);
        for (int k = 0; k < 5 * NV * 2; ++k) {
            const double keep = vs[k / 2 / NV][k / 2 % NV];
            vs[k / 2 / NV][k / 2 % NV] = copysign(std::numeric_limits<double>::quiet_NaN(), k & 1 ? -1.0 : 1.0);
            for (int kind = 0; kind < 4; ++kind) {
                double P[NV], M[NV];
                ld Pl[NV], Ml[NV];
                predict<double>(vs, kind > 0, kind > 1, it & 1, kind == 3 ? 2 : 0, P, M);
                predict<ld>(vs, kind > 0, kind > 1, it & 1, kind == 3 ? 2 : 0, Pl, Ml);
                for (int q = 0; q < NV; ++q) {
                    lost += (Pl[q] != Pl[q] && P[q] == P[q]) + (Ml[q] != Ml[q] && M[q] == M[q]);
                    both += (Pl[q] != Pl[q] && P[q] != P[q]) + (Ml[q] != Ml[q] && M[q] != M[q]);
                }
            }
            if (k < 4 * NV) {
                double F[NV];
                ld L[NV], R[NV], Fl[NV];
                for (int q = 0; q < NV; ++q) {
                    L[q] = vs[0][q];
                    R[q] = vs[1][q];
                }
                const bool b = riemann_hlld(vs[0], vs[1], 5.0 / 3.0, 3.0, F);
                const bool bl = riemann_hlld<ld>(L, R, ld(5.0 / 3.0), 3.0L, Fl);
                lost += bl && !b;
                for (int q = 0; q < NV; ++q) {
                    lost += Fl[q] != Fl[q] && F[q] == F[q];
                    both += Fl[q] != Fl[q] && F[q] != F[q];
                }
            }
            vs[k / 2 / NV][k / 2 % NV] = keep;
        }
    }
    std::printf("%ld %ld\n", lost, both);
    return 0;
}
