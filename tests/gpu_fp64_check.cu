// The FP64 primitives of the closed form (csrc/fp64.cuh) and the FP32 pass's
// angle (csrc/quad32.cuh) against a host reference in long double: per function
// its name, its largest error in units of its bound, and the sample count.  The bounds sum the roundings:
//   sqrt64     2^-52 relative;
//   log_ratio  4e-16 + 2.3e-16 |log| (num s, the table's log, the FP32 tail of
//              the series, and the sum's own rounding);
//   angle64    6e-16 (the table's angle, the rounded pi, two sums of size <= pi);
//   angle_q1   4 x 2^-24 relative (the difference, the reciprocal, the product, the sum).
// Built and run by tests/test_gpu_fp64_primitives.py.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include <cuda_runtime.h>

#include "fp64.cuh"
#include "quad32.cuh"

__global__ void eval(int n, const double *a, const double *b, double *s, double *l, double *t, double *g)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double p = fabs(a[i]), q = fabs(b[i]);
    s[i] = em::sqrt64(p);
    l[i] = p > 0.0 && q > 0.0 ? em::log_ratio(p, q, em::kLogTab) : 0.0;
    t[i] = em::angle64(a[i], b[i], em::kAtanTab);
    const float x = (float)q, y = (float)p;
    g[i] = x > 1e-30f && x < 1e30f && y < 1e30f ? (double)emq::angle_q1(y, x) : 0.0;
}

int main()
{
    std::vector<double> a, b;
    auto add = [&](double u, double v) {
        a.push_back(u);
        b.push_back(v);
    };
    std::mt19937_64 rng(7);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    for (int i = 0; i < 200000; ++i) add(U(rng), U(rng));
    for (int i = 0; i < 100000; ++i) add(U(rng) * std::exp2(60 * U(rng)), U(rng) * std::exp2(60 * U(rng)));
    for (int i = 0; i < 100000; ++i) {   // ratios near 1, and next to the tables' breakpoints
        const double u = 1.0 + U(rng) * std::exp2(-1 - i % 50);
        add(u, 1.0);
        const double c = (2 * (i % 64) + 1) / 128.0;
        add(c * u, 1.0);
        add(1.0 + i % 65 / 64.0 * u, 1.0 + 1e-3 * U(rng));
    }
    const double edge[] = {0.0, -0.0, 1.0, -1.0, 1e-290, 1e-160, -1e-160, 1e100, 4.0, 2.0};
    for (double u : edge)
        for (double v : edge) add(u, v);
    const int n = (int)a.size();
    double *d[6];
    std::vector<double> r[4];
    for (auto &p : d) cudaMalloc(&p, n * sizeof(double));
    cudaMemcpy(d[0], a.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemcpy(d[1], b.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    eval<<<(n + 255) / 256, 256>>>(n, d[0], d[1], d[2], d[3], d[4], d[5]);
    for (int k = 0; k < 4; ++k) {
        r[k].resize(n);
        if (cudaMemcpy(r[k].data(), d[2 + k], n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    }
    double worst[4] = {0, 0, 0, 0};
    for (int i = 0; i < n; ++i) {
        const double p = std::fabs(a[i]), q = std::fabs(b[i]);
        const long double s = sqrtl((long double)p);
        worst[0] = std::fmax(worst[0], s > 0 ? (double)(fabsl(r[0][i] - s) / s) / 0x1p-52 : (r[0][i] == 0.0 ? 0.0 : 1e9));
        if (p > 0.0 && q > 0.0) {
            const long double l = logl((long double)p) - logl((long double)q);
            worst[1] = std::fmax(worst[1], (double)fabsl(r[1][i] - l) / (4e-16 + 2.3e-16 * (double)fabsl(l)));
        }
        // the zero vector's angle is 0 whatever its signs
        const long double t = p == 0.0 && q == 0.0 ? 0.0L : atan2l((long double)a[i], (long double)b[i]);
        worst[2] = std::fmax(worst[2], (double)fabsl(r[2][i] - t) / 6e-16);
        const float x = (float)q, y = (float)p;
        if (x > 1e-30f && x < 1e30f && y > 1e-30f && y < 1e30f && y / x > 1e-30f) {
            const long double g = atan2l((long double)y, (long double)x);
            worst[3] = std::fmax(worst[3], (double)(fabsl(r[3][i] - g) / g) / 0x1p-22);
        }
        for (auto &v : r)
            if (!std::isfinite(v[i])) worst[2] = 1e9;
    }
    std::printf("sqrt64 %g %d\nlog_ratio %g %d\nangle64 %g %d\nangle_q1 %g %d\n", worst[0], n, worst[1], n, worst[2], n, worst[3], n);
    return 0;
}
