// Standalone GPU check of the FP64 products, reciprocals, roots and power-of-two
// scalings of swe_f64.cuh.  Hard (FP64 pipe) and Soft (integer unit)
// reciprocals and roots against CUDA's correctly rounded division and square
// root and its cube root, over log-uniform values of the range that the step
// meets and far beyond it: one line per function with the largest relative
// error in units of 2^-52.  Then the number of Soft products that differ from
// the correctly rounded ones ("mul"; half of the factors have 26 to 28
// significant bits, so that exact halves occur), and of wrong results on zero,
// denormals, infinities and NaN ("special").
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <vector>

#include "swe_kernels.cuh"

using namespace swe;

__device__ double ulps(double got, double ref) { return fabs(got - ref) / fabs(ref) * 4503599627370496.0; }

__device__ void note(double* slot, double v) {   // non-negative doubles order like their bits
    if (!(v >= 0.0)) v = 1e30;                   // NaN
    atomicMax((unsigned long long*)slot, (unsigned long long)__double_as_longlong(v));
}

template <class A>
__device__ void check_one(double x, double* worst) {
    note(worst + 0, ulps(A::rcp(x), 1.0 / x));
    note(worst + 1, ulps(A::rcp(-x), -1.0 / x));
    double y;
    note(worst + 2, ulps(A::sqrt_(x), sqrt(x)));
    note(worst + 3, ulps(A::sqrt_rsqrt(x, y), sqrt(x)));
    note(worst + 4, ulps(y, 1.0 / sqrt(x)));
    if (x > 1.2e-38 && x < 3e38) note(worst + 5, ulps(f64::rcbrt<A>(x), 1.0 / cbrt(x)));
}

__global__ void check(const double* xs, int n, double* worst, unsigned long long* bad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = xs[i];
    check_one<f64::Hard>(x, worst);
    check_one<f64::Soft>(x, worst + 6);
    note(worst + 12, ulps(f64::twice(x), 2.0 * x) + ulps(f64::half(-x), -0.5 * x) + ulps(f64::four_times(x), 4.0 * x));
    for (int k = 1; k <= 64; ++k) {
        double y = xs[(i + 7919LL * k) % n];
        if (k & 1) y = -y;
        const double p = __dmul_rn(x, y);
        if (!(fabs(p) > 1e-307 && fabs(p) < 1e307)) continue;   // a normal product
        if (__double_as_longlong(f64::Soft::mul(x, y)) != __double_as_longlong(p)) atomicAdd(bad, 1ULL);
    }
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
    bad += f64::Soft::sqrt_rsqrt(0.0, y) != 0.0 || y != 0.0 || f64::Soft::sqrt_(-0.0) != 0.0;
    bad += f64::Soft::sqrt_(tiny) != 0.0 || f64::Soft::sqrt_(1.0) != 1.0 || f64::Soft::sqrt_(4.0) != 2.0;
    bad += f64::Soft::rcp(1.0) != 1.0 || f64::Soft::rcp(-8.0) != -0.125;
    bad += __double_as_longlong(f64::Soft::mul(0.0, -3.0)) != __double_as_longlong(-0.0);
    bad += __double_as_longlong(f64::Soft::mul(-2.5, -0.0)) != 0LL || f64::Soft::mul(0.0, 0.0) != 0.0;
    bad += !f64::in_range<-64, 24>(0.0) || !f64::in_range<-64, 24>(-0.0) || f64::in_range<-64, 24>(nan);
    bad += f64::in_range<-64, 24>(inf) || f64::in_range<-64, 24>(tiny) || f64::in_range<-64, 24>(16777216.0);
    bad += !f64::in_range<-64, 24>(-16777215.0) || !f64::in_range<-64, 24>(5.5e-20) || f64::in_range<-64, 24>(5.4e-20);
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
        if (i & 1) {   // 26 to 28 significant bits
            unsigned long long b;
            std::memcpy(&b, &xs[i], 8);
            b &= ~((1ULL << (25 + (i >> 1) % 3)) - 1ULL);
            std::memcpy(&xs[i], &b, 8);
        } else if (i % 64 == 0) {   // significands next to 1 and 2
            unsigned long long b;
            std::memcpy(&b, &xs[i], 8);
            b = (b & 0xFFF0000000000000ULL) | ((i / 64) % 2 ? (unsigned long long)(i / 128 % 5)
                                                            : 0xFFFFFFFFFFFFFULL - (unsigned long long)(i / 128 % 5));
            std::memcpy(&xs[i], &b, 8);
        }
    }
    double *dx, *dw;
    int* db;
    unsigned long long *dm, m = ~0ULL;
    const int kChecks = 13;
    cudaMalloc(&dx, n * sizeof(double));
    cudaMalloc(&dw, kChecks * sizeof(double));
    cudaMalloc(&db, sizeof(int));
    cudaMalloc(&dm, sizeof m);
    cudaMemset(dm, 0, sizeof m);
    cudaMemcpy(dx, xs.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemset(dw, 0, kChecks * sizeof(double));
    check<<<n / 256, 256>>>(dx, n, dw, dm);
    special<<<1, 1>>>(db);
    double w[kChecks];
    int bad = -1;
    cudaMemcpy(w, dw, sizeof w, cudaMemcpyDeviceToHost);
    cudaMemcpy(&bad, db, sizeof bad, cudaMemcpyDeviceToHost);
    cudaMemcpy(&m, dm, sizeof m, cudaMemcpyDeviceToHost);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    const char* names[kChecks] = {"rcp",      "rcp_negative",      "sqrt",      "sqrt_with_inverse",      "rsqrt",      "rcbrt",
                                  "soft_rcp", "soft_rcp_negative", "soft_sqrt", "soft_sqrt_with_inverse", "soft_rsqrt", "soft_rcbrt",
                                  "scale"};
    for (int k = 0; k < kChecks; ++k) std::printf("%s %.6f\n", names[k], w[k]);
    std::printf("mul %llu\nspecial %d\n", m, bad);
    return 0;
}
