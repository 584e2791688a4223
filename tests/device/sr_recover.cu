// The mixed relativistic recoveries on the device: the double-float ones
// (sr_interface_call, sr_recover) against the float64 iterations they stand for
// (sr_interface_slow, sr_prim_slow).  argv = exponent k (rho, p by 4^k, B by 2^k),
// states.  Prints: physical states, values that differ, states sr_recover decides.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "sr_df.cuh"

using namespace ctu;

__global__ void k_compare(const SrFace *f, int n, double gam, df g1, df ig1, unsigned long long *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long wrong = 0, decided = 0, physical;
    const SrOut a = sr_interface_call(f[i], g1, ig1, gam), b = sr_interface_slow(f[i], gam);
    physical = b.st == 0u;
    wrong += a.st != b.st;
    for (int q = 0; q < NV; ++q) wrong += b.st == 0u && __float_as_uint(a.V[q]) != __float_as_uint(b.V[q]);
    SrCons c;
    double U[NV];
    sr_cons<double, float>(f[i].V, gam, U);
    for (int q = 0; q < NV; ++q) c.U[q] = U[q] + (double)f[i].T[q];
    SrState u;
    float v[5];
    u.D = sr_split(c.U[0]);
    u.tau = d_add(sr_split(c.U[4]), u.D);
    for (int k = 0; k < 3; ++k) {
        u.m[k] = sr_split(c.U[1 + k]);
        u.b[k] = sr_split(c.U[5 + k]);
    }
    if (sr_recover(u, 0.0f, g1, v)) {
        const SrOut o = sr_prim_slow(c, gam, 0.0);
        decided = 1;
        wrong += o.st != 0u;
        for (int q = 0; q < 5; ++q) wrong += __float_as_uint(v[q]) != __float_as_uint(o.V[q]);
    }
    atomicAdd(out, physical);
    atomicAdd(out + 1, wrong);
    atomicAdd(out + 2, decided);
}

int main(int argc, char **argv)
{
    const float s2 = std::ldexp(1.0f, 2 * std::atoi(argv[1])), s1 = std::ldexp(1.0f, std::atoi(argv[1]));
    const int n = std::atoi(argv[2]);
    std::mt19937_64 gen(3);
    auto uni = [&] { return (double)(gen() >> 11) / 9007199254740992.0; };
    auto sym = [&](double s) { return s * (2.0 * uni() - 1.0); };
    std::vector<SrFace> f(n);
    for (int i = 0; i < n; ++i) {
        double v[9];
        if (i & 1) {  // the beam and its edge
            const double prof = uni(), lor = 1.0 + 9.0 * prof, off = 0.05 * std::fmin(prof, 0.2);
            const double w[9] = {0.01 + 0.99 * prof, sym(off), sym(off), std::sqrt(1.0 - 1.0 / (lor * lor)) * (1.0 - 0.001 * prof),
                                 0.01 * (1.0 + sym(0.5)), sym(0.3), sym(0.3), 3.225 + sym(0.1), sym(0.01)};
            for (int q = 0; q < 9; ++q) v[q] = w[q];
        } else {  // any direction, speed, temperature and magnetisation
            const double sp = std::pow(uni(), 0.3) * 0.995, c = sym(1.0), p = 6.283185307179586 * uni();
            const double r = std::sqrt(1.0 - c * c), b = std::exp(5.0 * uni() - 4.0);
            v[0] = std::exp(6.0 * uni() - 3.0);
            v[1] = sp * r * std::cos(p);
            v[2] = sp * r * std::sin(p);
            v[3] = sp * c;
            v[4] = std::exp(10.0 * uni() - 7.0);
            for (int q = 5; q < 9; ++q) v[q] = b * sym(1.0);
        }
        for (int q = 0; q < 9; ++q) {
            f[i].V[q] = (float)v[q] * (q == 0 || q == 4 ? s2 : q >= 5 ? s1 : 1.0f);
            f[i].T[q] = (float)(sym(1e-5) * (q < 5 ? v[0] * s2 : v[q] * s1));
        }
    }
    const double gam = 4.0 / 3.0;
    auto pair = [](double x) { return df{(float)x, (float)(x - (double)(float)x)}; };
    SrFace *d;
    unsigned long long *o, h[3];
    if (cudaMalloc(&d, n * sizeof(SrFace)) != cudaSuccess || cudaMalloc(&o, sizeof(h)) != cudaSuccess) return 1;
    cudaMemcpy(d, f.data(), n * sizeof(SrFace), cudaMemcpyHostToDevice);
    cudaMemset(o, 0, sizeof(h));
    k_compare<<<(n + 127) / 128, 128>>>(d, n, gam, pair((gam - 1.0) / gam), pair(gam / (gam - 1.0)), o);
    if (cudaMemcpy(h, o, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    std::printf("%llu %llu %llu\n", h[0], h[1], h[2]);
    return 0;
}
