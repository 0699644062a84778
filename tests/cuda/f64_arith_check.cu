// Standalone GPU check of the FP64 reciprocal, roots and power-of-two scalings
// of swe_f64.cuh against CUDA's correctly rounded division and square root
// and its cube root, over log-uniform values of the range that the step meets
// and far beyond it.  Prints one line per function with the largest relative
// error in units of 2^-52, then "special" with the number of wrong results on
// zero, denormals, infinities and NaN.
#include <cmath>
#include <cstdio>
#include <limits>
#include <vector>

#include "swe_kernels.cuh"

using namespace swe;

__device__ double ulps(double got, double ref) { return fabs(got - ref) / fabs(ref) * 4503599627370496.0; }

__device__ void note(double* slot, double v) {   // non-negative doubles order like their bits
    if (!(v >= 0.0)) v = 1e30;                   // NaN
    atomicMax((unsigned long long*)slot, (unsigned long long)__double_as_longlong(v));
}

__global__ void check(const double* xs, int n, double* worst) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = xs[i];
    note(worst + 0, ulps(f64::rcp(x), 1.0 / x));
    note(worst + 1, ulps(f64::rcp(-x), -1.0 / x));
    double y;
    note(worst + 2, ulps(f64::sqrt_rsqrt(x, y), sqrt(x)));
    note(worst + 3, ulps(y, 1.0 / sqrt(x)));
    if (x > 1.2e-38 && x < 3e38) note(worst + 4, ulps(f64::rcbrt(x), 1.0 / cbrt(x)));
    note(worst + 5, ulps(f64::twice(x), 2.0 * x) + ulps(f64::half(-x), -0.5 * x) + ulps(f64::four_times(x), 4.0 * x));
}

__global__ void special(int* wrong) {
    const double inf = __longlong_as_double(0x7FF0000000000000LL), nan = __longlong_as_double(0x7FF8000000000000LL);
    const double tiny = __longlong_as_double(1LL);
    int bad = 0;
    double y;
    bad += f64::sqrt_rsqrt(0.0, y) != 0.0 || y != 0.0;
    bad += f64::sqrt_(-0.0) != 0.0;
    bad += f64::sqrt_(tiny) != 0.0;
    bad += !isnan(f64::sqrt_(nan));
    bad += !isnan(f64::rcp(nan));
    bad += f64::twice(0.0) != 0.0 || f64::half(0.0) != 0.0;
    bad += f64::twice(inf) != inf || f64::half(-inf) != -inf || !isnan(f64::twice(nan)) || !isnan(f64::half(nan));
    bad += f64::twice(tiny) != tiny;
    *wrong = bad;
}

int main() {
    const int n = 1 << 20;
    std::vector<double> xs(n);
    unsigned long long s = 88172645463325252ULL;
    for (int i = 0; i < n; ++i) {
        s ^= s << 13; s ^= s >> 7; s ^= s << 17;
        const double u = (double)(s >> 11) / 9007199254740992.0;
        xs[i] = std::pow(10.0, i % 4 ? -8.0 + 16.0 * u : -300.0 + 600.0 * u);
    }
    double *dx, *dw;
    int* db;
    const int kChecks = 6;
    cudaMalloc(&dx, n * sizeof(double));
    cudaMalloc(&dw, kChecks * sizeof(double));
    cudaMalloc(&db, sizeof(int));
    cudaMemcpy(dx, xs.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemset(dw, 0, kChecks * sizeof(double));
    check<<<n / 256, 256>>>(dx, n, dw);
    special<<<1, 1>>>(db);
    double w[kChecks];
    int bad = -1;
    cudaMemcpy(w, dw, sizeof w, cudaMemcpyDeviceToHost);
    cudaMemcpy(&bad, db, sizeof bad, cudaMemcpyDeviceToHost);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    const char* names[kChecks] = {"rcp", "rcp_negative", "sqrt", "rsqrt", "rcbrt", "scale"};
    for (int k = 0; k < kChecks; ++k) std::printf("%s %.6f\n", names[k], w[k]);
    std::printf("special %d\n", bad);
    return 0;
}
