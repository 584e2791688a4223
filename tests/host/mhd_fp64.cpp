// The float64 forms of mhd_fp64.cuh on the host beside the generic functions they
// stand for (mhd_device.cuh), instantiated in long double.
//   nan: every number of the inputs in turn a quiet nan of either sign; prints the
//        outputs that are finite here and nan there, and those of both that are nan
//   err: random states (argv: count, seed); prints the mean relative error of the
//        fluxes and of the predicted states, IEEE double forms and these, against
//        long double
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

// IEEE double arithmetic in the generic functions (double itself takes the forms)
struct alignas(16) Ieee {
    double v;
    Ieee() = default;
    Ieee(double x) : v(x) {}
    explicit operator double() const { return v; }
};
static Ieee operator+(Ieee a, Ieee b) { return a.v + b.v; }
static Ieee operator-(Ieee a, Ieee b) { return a.v - b.v; }
static Ieee operator*(Ieee a, Ieee b) { return a.v * b.v; }
static Ieee operator/(Ieee a, Ieee b) { return a.v / b.v; }
static Ieee operator-(Ieee a) { return -a.v; }
static Ieee &operator+=(Ieee &a, Ieee b) { return a = a + b; }
static bool operator<(Ieee a, Ieee b) { return a.v < b.v; }
static bool operator>(Ieee a, Ieee b) { return a.v > b.v; }
static bool operator<=(Ieee a, Ieee b) { return a.v <= b.v; }
static bool operator>=(Ieee a, Ieee b) { return a.v >= b.v; }
static Ieee fabs(Ieee a) { return std::fabs(a.v); }
static Ieee sqrt(Ieee a) { return std::sqrt(a.v); }
static Ieee fmin(Ieee a, Ieee b) { return std::fmin(a.v, b.v); }
static Ieee fmax(Ieee a, Ieee b) { return std::fmax(a.v, b.v); }
static Ieee copysign(Ieee a, Ieee b) { return std::copysign(a.v, b.v); }
namespace ctu {
template <> struct Tol<Ieee> : Tol<double> {};
} // namespace ctu

template <class R> static ld rel(const R (&a)[NV], const ld (&b)[NV])
{
    ld n = 0, d = 0;
    for (int q = 0; q < NV; ++q) {
        n += ((ld)(double)a[q] - b[q]) * ((ld)(double)a[q] - b[q]);
        d += b[q] * b[q];
    }
    return sqrt(n / d);
}

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

int main(int argc, char **argv)
{
    const bool nan = argv[1][0] == 'n';
    Gen g;
    if (nan) {
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
    const long count = std::atol(argv[2]);
    g.gen.seed(std::atoi(argv[3]));
    ld err[3][2] = {};
    for (long it = 0; it < count; ++it) {
        double c[NV], vs[5][NV], P[2][NV];
        ld Pl[2][NV], L[NV], R[NV], Fl[NV];
        Ieee Pi[2][NV], Li[NV], Ri[NV], Fi[NV];
        double F[NV];
        g.center(c);
        const double s = std::exp(-6.0 * g.uni());
        for (auto &v : vs) g.state(v, c, s);
        for (int kind = 0; kind < 2; ++kind) {
            predict<double>(vs, kind, false, it & 1, 0, P[0], P[1]);
            predict<Ieee>(vs, kind, false, it & 1, 0, Pi[0], Pi[1]);
            predict<ld>(vs, kind, false, it & 1, 0, Pl[0], Pl[1]);
            for (int e = 0; e < 2; ++e) {
                err[kind][0] += rel(Pi[e], Pl[e]) / (2 * count);
                err[kind][1] += rel(P[e], Pl[e]) / (2 * count);
            }
        }
        for (int q = 0; q < NV; ++q) {
            L[q] = Li[q].v = vs[1][q];
            R[q] = Ri[q].v = vs[2][q];
        }
        riemann_hlld(vs[1], vs[2], 5.0 / 3.0, 3.0, F);
        riemann_hlld<Ieee>(Li, Ri, 5.0 / 3.0, 3.0, Fi);
        riemann_hlld<ld>(L, R, ld(5.0 / 3.0), 3.0L, Fl);
        err[2][0] += rel(Fi, Fl) / count;
        err[2][1] += rel(F, Fl) / count;
    }
    for (auto &e : err) std::printf("%.3Le %.3Le\n", e[0], e[1]);
    return 0;
}
