// Largest relative error of r_rsqrt (csrc/newton_common.cuh) over 2^-52, against long double.
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <random>
#include <vector>

#include "newton_common.cuh"

__global__ void run(const double *a, double *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = kitrt_dev::r_rsqrt(a[i]);
}

int main()
{
    std::vector<double> a;
    std::mt19937_64 g(1);
    std::uniform_real_distribution<double> u(0.0, 1.0);
    for (int i = 0; i < 1 << 20; ++i) a.push_back(exp2(u(g) * 2000.0 - 1000.0) * (1.0 + u(g)));
    for (int i = 0; i < 1 << 18; ++i) a.push_back(0.25 + 3.75 * u(g));
    // both sides of the branch at the ends of the FP32 range, and powers of two
    for (double b : {1e-37, 1e37})
        for (int k = -1000; k <= 1000; ++k) a.push_back(b * (1.0 + k * 1e-12));
    for (int k = -1000; k <= 1000; ++k) a.push_back(exp2((double)k));
    const int n = (int)a.size();
    double *da, *dy;
    std::vector<double> y(n);
    if (cudaMalloc(&da, n * 8) || cudaMalloc(&dy, n * 8)) return 1;
    if (cudaMemcpy(da, a.data(), n * 8, cudaMemcpyHostToDevice)) return 1;
    run<<<(n + 255) / 256, 256>>>(da, dy, n);
    if (cudaMemcpy(y.data(), dy, n * 8, cudaMemcpyDeviceToHost)) return 1;
    long double worst = 0;
    for (int i = 0; i < n; ++i) worst = std::max(worst, fabsl((long double)y[i] * sqrtl((long double)a[i]) - 1));
    printf("%.6Lf\n", ldexpl(worst, 52));
    return 0;
}
