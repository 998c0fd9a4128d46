// quotient() of csrc/common.cuh against IEEE division: random mantissas at every exponent of the range in
// which it approximates (both ends and the powers of two among them), and the divisors that take the
// division (subnormal, tiny, huge, zero, infinite, NaN), where the results must be the same.
//   nvcc -gencode arch=compute_103a,code=sm_103a -O3 -std=c++17 -I<include> -I<csrc> quotient_check.cu
// Bar: both the product with the approximation and the last step round once (2^-53 each), what the cubic
// step leaves is below 2^-57 (an approximation to 2^-19), the division itself rounds by 2^-54 here where the
// relative size is smallest: 2.25 x 2^-53 of the quotient, compared in long double.
#include "common.cuh"

#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>
#include <vector>

__global__ void quotient_kernel(int n, const double *v, const double *d, double *q) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) q[i] = ot::quotient(v[i], d[i]);
}

int main() {
    std::mt19937_64 rng(1);
    std::vector<double> v, d;
    auto mant = [&] { return 1.0 + (double)(rng() >> 12) * 0x1p-52; };
    for (int e = -1000; e <= 999; ++e)
        for (int k = 0; k < 512; ++k) {
            const double m = k == 0 ? 1.0 : k == 1 ? 2.0 - 0x1p-52 : k == 2 ? 1.0 + 0x1p-52 : k == 3 ? 1.5 : mant();
            d.push_back(std::ldexp(k & 4 ? -m : m, e));
            // quotients from 2^-20 to 2^20, well inside the range
            v.push_back(std::ldexp(mant(), std::max(-1000, std::min(1000, e + (int)(rng() % 41) - 20))));
        }
    const size_t approx = d.size();
    const double inf = INFINITY, nan = NAN;
    for (double x : {0.0, -0.0, 0x1p-1074, 3 * 0x1p-1070, 0x1p-1022, 0x1.8p-1010, -0x1p-1001, 0x1.fp1001, 0x1p1022,
                     -0x1.9p1023, inf, -inf, nan})
        for (double y : {0.0, 1.0, -3.0, 0x1p-1060, 0x1.4p-1020, 0x1.7p1020, inf, nan}) {
            d.push_back(x);
            v.push_back(y);
        }
    const int n = (int)d.size();
    double *gv, *gd, *gq;
    std::vector<double> q(n);
    if (cudaMalloc(&gv, 8 * n) || cudaMalloc(&gd, 8 * n) || cudaMalloc(&gq, 8 * n)) return 2;
    cudaMemcpy(gv, v.data(), 8 * n, cudaMemcpyHostToDevice);
    cudaMemcpy(gd, d.data(), 8 * n, cudaMemcpyHostToDevice);
    quotient_kernel<<<256, 256>>>(n, gv, gd, gq);
    if (cudaMemcpy(q.data(), gq, 8 * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    long double worst = 0;
    int bad = 0;
    for (int i = 0; i < n; ++i) {
        if ((size_t)i < approx) {
            const long double want = (long double)v[i] / (long double)d[i];
            const long double err = std::fabs(((long double)q[i] - want) / want) * 0x1p53L;
            if (!(err <= 2.25L)) ++bad;
            if (!(err <= worst)) worst = err;
        } else {
            const double want = v[i] / d[i];
            if (!(q[i] == want || (std::isnan(q[i]) && std::isnan(want)))) {
                printf("%a / %a = %a, not %a\n", v[i], d[i], want, q[i]);
                ++bad;
            }
        }
    }
    printf("%d quotients, worst error %.3Lf x 2^-53, %d wrong\n", n, worst, bad);
    if (bad) return 1;
    printf("OK\n");
    return 0;
}
