// d_rcp64 and d_roots64 on the device against long double: prints the largest
// relative error of 1/x, 1/sqrt(x) and sqrt(x) in units of 2^-53, and the values of
// the roots of 0 and of a denormal.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "mhd_fp64.cuh"

__global__ void k_roots(const double *x, double *r, double *y, double *s, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = ctu::d_rcp64(x[i]);
    ctu::d_roots64(x[i], y[i], s[i]);
}

int main()
{
    const int n = 1 << 22;
    std::vector<double> x(n), o[3];
    std::mt19937_64 gen(1);
    x[0] = 0.0;
    x[1] = 1e-310;
    for (int i = 2; i < n; ++i)
        x[i] = std::ldexp(1.0 + (double)(gen() >> 12) / 4503599627370496.0, i & 1 ? (int)(gen() % 2040) - 1020 : (int)(gen() % 8) - 4);
    double *d[4];
    for (auto &p : d)
        if (cudaMalloc(&p, n * sizeof(double)) != cudaSuccess) return 1;
    cudaMemcpy(d[0], x.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    k_roots<<<n / 256, 256>>>(d[0], d[1], d[2], d[3], n);
    for (int k = 0; k < 3; ++k) {
        o[k].resize(n);
        if (cudaMemcpy(o[k].data(), d[k + 1], n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    }
    long double e[3] = {0, 0, 0};
    for (int i = 2; i < n; ++i) {
        const long double t[3] = {1.0L / x[i], 1.0L / std::sqrt((long double)x[i]), std::sqrt((long double)x[i])};
        for (int k = 0; k < 3; ++k) e[k] = std::fmax(e[k], std::fabs(o[k][i] / t[k] - 1.0L));
    }
    for (int k = 0; k < 3; ++k) std::printf("%.4Lf ", std::ldexp(e[k], 53));
    std::printf("%g %g %g %g\n", o[1][0], o[2][0], o[1][1], o[2][1]);
    return 0;
}
