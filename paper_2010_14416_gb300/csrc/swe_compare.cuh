// swe_compare.cuh -- comparisons and selections of the flux path.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

namespace swe {

template <typename T>
__device__ __forceinline__ T tmax(T a, T b) { return a > b ? a : b; }
template <typename T>
__device__ __forceinline__ T tmin(T a, T b) { return a < b ? a : b; }

// ---- comparisons of the flux path ------------------------------------------------
// On GB300 the FP64 unit (2 operations per clock per SM) executes compares and
// min/max of doubles as well as their arithmetic, and it bounds the FP64 step.
// For doubles each helper below forms exactly the IEEE result of its
// comparison (NaN, infinities and signed zeros included) from the bit
// patterns, with 64-bit integer operations, which the FP64 kernels leave
// idle; the selects return the same operand the plain expression returns, so
// results are bit for bit those of the plain operators.  Other scalars (float,
// the adjoint's dual numbers) use the plain operators.
namespace cmp {
constexpr unsigned long long kPosInf = 0x7FF0000000000000ULL;   // bits of +inf
constexpr unsigned long long kNegZero = 0x8000000000000000ULL;  // bits of -0
__device__ __forceinline__ unsigned long long bits(double x) { return (unsigned long long)__double_as_longlong(x); }
template <typename T>
constexpr bool kInt = std::is_same<T, double>::value;
}  // namespace cmp

// x > c for c finite and > 0
template <typename T>
__device__ __forceinline__ bool gt_pos(T x, T c) {
    if constexpr (cmp::kInt<T>) {
        const unsigned long long xb = cmp::bits(x), cb = cmp::bits(c);
        return xb - cb - 1ULL < cmp::kPosInf - cb;          // c < x <= +inf
    } else {
        return x > c;
    }
}
// x <= c for c finite and > 0
template <typename T>
__device__ __forceinline__ bool le_pos(T x, T c) {
    if constexpr (cmp::kInt<T>) {
        const unsigned long long xb = cmp::bits(x), cb = cmp::bits(c);
        return xb <= cb || xb - cmp::kNegZero <= cmp::kPosInf;   // +0 <= x <= c, or -inf <= x <= -0
    } else {
        return x <= c;
    }
}
// x < c for c finite and > 0
template <typename T>
__device__ __forceinline__ bool lt_pos(T x, T c) {
    if constexpr (cmp::kInt<T>) {
        const unsigned long long xb = cmp::bits(x), cb = cmp::bits(c);
        return xb < cb || xb - cmp::kNegZero <= cmp::kPosInf;
    } else {
        return x < c;
    }
}
// |x| < c for c finite and > 0
template <typename T>
__device__ __forceinline__ bool abs_lt_pos(T x, T c) {
    if constexpr (cmp::kInt<T>) {
        return (cmp::bits(x) & ~cmp::kNegZero) < cmp::bits(c);
    } else {
        return fabs(x) < c;
    }
}
template <typename T>
__device__ __forceinline__ bool gt_zero(T x) {
    if constexpr (cmp::kInt<T>) return cmp::bits(x) - 1ULL < cmp::kPosInf;            // smallest denormal .. +inf
    else return x > T(0);
}
template <typename T>
__device__ __forceinline__ bool ge_zero(T x) {
    if constexpr (cmp::kInt<T>) {
        const unsigned long long xb = cmp::bits(x);
        return xb <= cmp::kPosInf || xb == cmp::kNegZero;
    } else {
        return x >= T(0);
    }
}
template <typename T>
__device__ __forceinline__ bool le_zero(T x) {
    if constexpr (cmp::kInt<T>) {
        const unsigned long long xb = cmp::bits(x);
        return xb == 0ULL || xb - cmp::kNegZero <= cmp::kPosInf;
    } else {
        return x <= T(0);
    }
}
template <typename T>
__device__ __forceinline__ bool lt_zero(T x) {
    if constexpr (cmp::kInt<T>) return cmp::bits(x) - (cmp::kNegZero + 1ULL) < cmp::kPosInf;  // -inf .. -denormal
    else return x < T(0);
}
// tmax(0, x)
template <typename T>
__device__ __forceinline__ T max_zero(T x) {
    if constexpr (cmp::kInt<T>) return lt_zero(x) ? T(0) : x;
    else return tmax(T(0), x);
}
// tmin(a, b) for a, b >= +0 (or +inf), e.g. CFL candidates and depths
template <typename T>
__device__ __forceinline__ T min_nonneg(T a, T b) {
    if constexpr (cmp::kInt<T>) return cmp::bits(a) < cmp::bits(b) ? a : b;
    else return tmin(a, b);
}
// tmax(a, b) for finite a, b (bed elevations)
template <typename T>
__device__ __forceinline__ T max_finite(T a, T b) {
    if constexpr (cmp::kInt<T>) {
        // the sign-magnitude bits, turned into a two's-complement key, order
        // finite doubles except that -0 sorts below +0, where IEEE has a tie
        const long long ab = __double_as_longlong(a), bb = __double_as_longlong(b);
        const long long ka = ab ^ ((ab >> 63) & 0x7FFFFFFFFFFFFFFFLL), kb = bb ^ ((bb >> 63) & 0x7FFFFFFFFFFFFFFFLL);
        const bool both_zero = (((unsigned long long)ab | (unsigned long long)bb) << 1) == 0ULL;
        return (ka > kb && !both_zero) ? a : b;
    } else {
        return tmax(a, b);
    }
}

}  // namespace swe
