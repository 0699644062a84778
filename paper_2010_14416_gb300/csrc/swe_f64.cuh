// swe_f64.cuh -- the FP64 arithmetic of one cell update (Eq 12-37).
//
// What bounds it.  An SM of GB300 completes one FP64 warp instruction in 19
// clocks, a lone warp one in 64, whatever the number of active lanes or of
// independent operations (measured), so every FP64 kernel here is bound by the
// number of instructions it puts on that pipe: memory, integer and FP32 units
// idle.  Hence:
//   - products, reciprocals and roots run on the integer unit (Soft below), so
//     the FP64 pipe is left with the additions and fused multiply-adds;
//   - comparisons, selects and powers of two run on the integer unit too
//     (swe_compare.cuh, scale2 below);
//   - the wave speeds need no star depth where Eq 21 chooses the
//     two-rarefaction estimate (Eq 22): there h* <= min(h_L, h_R), so both
//     factors of Eq 20 are 1;
//   - where they do, a_K p_K = sqrt(g h* (h* + h_K) / (2 h_K)) is formed at once;
//   - Eq 24 needs only the sign of S*.  Eq 25's numerator is minus Eq 18's
//     numerator of the mass flux and its denominator is negative, so between
//     S_L and S_R that is the sign of the mass flux;
//   - an edge's flux and its two bed source terms are combined per edge into
//     what each of its cells subtracts (5 numbers per unit length), so a cell
//     takes three fused multiply-adds per edge.
// Measured against IEEE division and square root with the textbook order of
// operations, all on the FP64 pipe: 2^20 Riemann problems 418 us, 215 with the
// shorter formulas and roots, 90 with Soft; a step of the 1M-cell canal with
// the edge pass 480, 317 and 182 us.
// Every operation is explicitly rounded (the compiler may neither fuse nor
// split it), so each kernel that inlines these functions rounds alike and
// their results agree bit for bit.
//
#pragma once

#include "swe_compare.cuh"

namespace swe {
namespace f64 {

__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dadd_rn(a, -b); }
__device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double neg(double a) { return -a; }

// a 2^K by the exponent bits, for a normal a whose product is normal; zero,
// denormals, infinities and NaN give themselves
template <int K>
__device__ __forceinline__ double scale2(double a) {
    const int hi = __double2hiint(a);
    return __hiloint2double(((hi + 0x00100000) & 0x7FE00000) ? hi + K * 0x00100000 : hi, __double2loint(a));
}
__device__ __forceinline__ double twice(double a) { return scale2<1>(a); }
__device__ __forceinline__ double four_times(double a) { return scale2<2>(a); }
__device__ __forceinline__ double half(double a) { return scale2<-1>(a); }

// ---- products, reciprocals and roots -----------------------------------------------------
// Two implementations.  Hard puts them on the FP64 pipe.  Soft forms them on
// the integer unit from the significands, for operands in a range that the
// callers check (in_range): a lone warp's FP64 instruction takes 64 clocks and
// an SM completes one per 19, while its integer unit stands idle, so a product
// of about 35 integer instructions, spread over the four SM quarters, takes
// half the pipe's time and runs beside it; a reciprocal takes 40 in place of 3
// FP64 instructions, a root 55 in place of 6.  Additions and fused
// multiply-adds stay on the FP64 pipe.  A product is the correctly rounded
// one of either; reciprocals and roots are within 0.52 ulp, Soft's within
// 0.505.

// |x| in [2^lo, 2^hi), or zero
template <int LO, int HI>
__device__ __forceinline__ bool in_range(double x) {
    const unsigned h = (unsigned)__double2hiint(x) & 0x7FFFFFFFu;
    return h - ((unsigned)(1023 + LO) << 20) < ((unsigned)(HI - LO) << 20) || (h | (unsigned)__double2loint(x)) == 0u;
}

struct Hard {
    static constexpr bool kRare = false;
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    // seeds: the documented approximations of 1/x and 1/sqrt(x) that read the
    // upper word of x and write the upper word of the result
    static __device__ __forceinline__ double rcp_seed(double x) {
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        return y;
    }
    static __device__ __forceinline__ double rsqrt_seed(double x) {
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        // zero, denormals and negative values: 0, so that sqrt_(0) is 0
        return __double2hiint(x) < 0x00100000 ? 0.0 : y;
    }
    // 1/x for normal x: y0 (1 + e + e^2), e = 1 - x y0 (Householder's third
    // order; the error e^3 < 2^-60 is under the last operation's rounding)
    static __device__ __forceinline__ double rcp(double x) {
        const double y = rcp_seed(x);
        const double e = __fma_rn(-x, y, 1.0);
        return __fma_rn(__fma_rn(e, e, e), y, y);
    }
    // sqrt(x) (0 for x below the normal range): Heron's step for the root
    // t = x y0 and its inverse together, then the residual x - t^2 (Markstein)
    static __device__ __forceinline__ double sqrt_half_rsqrt(double x, double& h1) {
        const double y0 = rsqrt_seed(x);
        const double t = __dmul_rn(x, y0), h = half(y0);
        const double r = __fma_rn(-t, h, 0.5);
        const double t1 = __fma_rn(t, r, t);
        h1 = __fma_rn(h, r, h);                       // 1 / (2 sqrt(x)) to about 2^-40
        return __fma_rn(__fma_rn(-t1, t1, x), h1, t1);
    }
    static __device__ __forceinline__ double sqrt_(double x) {
        double h;
        return sqrt_half_rsqrt(x, h);
    }
    // and, as y, 1/sqrt(x) (0 there): one Newton step more, from the root
    static __device__ __forceinline__ double sqrt_rsqrt(double x, double& y) {
        double h;
        const double s = sqrt_half_rsqrt(x, h);
        const double y1 = twice(h);
        y = __fma_rn(__fma_rn(-s, y1, 1.0), y1, y1);
        return s;
    }
};

struct Soft {
    static constexpr bool kRare = false;
    // 32 x 32 -> 64 bits, plus c
    static __device__ __forceinline__ unsigned long long wide(unsigned a, unsigned b, unsigned long long c = 0ULL) {
        return (unsigned long long)a * b + c;
    }
    static __device__ __forceinline__ unsigned significand_hi(int hi) { return ((unsigned)hi & 0xFFFFFu) | 0x100000u; }

    // a b, rounded to nearest even: zero operands, or normal ones with a normal
    // product; with FLUSH a smaller product gives zero
    template <bool FLUSH>
    static __device__ __forceinline__ double product(double a, double b) {
        const unsigned ah = (unsigned)__double2hiint(a), al = (unsigned)__double2loint(a);
        const unsigned bh = (unsigned)__double2hiint(b), bl = (unsigned)__double2loint(b);
        const unsigned bm = significand_hi(bh);
        const unsigned Ah = __funnelshift_l(al, significand_hi(ah), 11), Al = al << 11;
        // the significands' product times 2^11, 117 bits: the result's 52 or 53
        // bits above 64, the remainder below
        const unsigned long long p0 = wide(Al, bl);
        const unsigned long long p1 = wide(Al, bm, p0 >> 32);
        const unsigned long long p2 = wide(Ah, bl, p1 & 0xFFFFFFFFULL);
        const unsigned long long p3 = wide(Ah, bm, p1 >> 32) + (p2 >> 32);
        unsigned h1 = (unsigned)(p3 >> 32), h0 = (unsigned)p3, l1 = (unsigned)p2, l0 = (unsigned)p0;
        const unsigned ea = ah & 0x7FF00000u, eb = bh & 0x7FF00000u;
        const unsigned top = h1 & 0x100000u;            // the product of the significands is at least 2
        const unsigned s = top ? 0u : 1u;
        h1 = __funnelshift_l(h0, h1, s);
        h0 = __funnelshift_l(l1, h0, s);
        l1 = __funnelshift_l(l0, l1, s);
        l0 <<= s;
        // up when the remainder exceeds one half, or is one half and the result odd
        const unsigned q = (l0 != 0u) | (h0 & 1u);
        const unsigned long long r = (((unsigned long long)h1 << 32) | h0) + (l1 >= 0x80000001u - q ? 1ULL : 0ULL);
        unsigned rh = (unsigned)(r >> 32) + ea + eb + top - (1024u << 20), rl = (unsigned)r;
        if (ea == 0u || eb == 0u || (FLUSH && ea + eb <= (1024u << 20))) { rh = 0u; rl = 0u; }
        return __hiloint2double((int)(rh | ((ah ^ bh) & 0x80000000u)), (int)rl);
    }
    static __device__ __forceinline__ double mul(double a, double b) { return product<false>(a, b); }

    // an FP32 seed in (1/2, 1] as a 32-bit fraction
    static __device__ __forceinline__ unsigned fraction(float r) {
        const unsigned b = min(max(__float_as_uint(r), 0x3F000000u), 0x3F7FFFFFu);
        return (b << 8) | 0x80000000u;
    }
    // R (1 + c) for a 32-bit fraction R (even) and c in units of 2^-(31 + SHIFT) / 2^31, as a 64-bit
    // fraction, less 8 units so that 1 does not overflow; then rounded to 53 bits
    // with the exponent field `field`
    template <int SHIFT>
    static __device__ __forceinline__ double scaled_fraction(unsigned R, long long c, unsigned field) {
        const unsigned h = R >> 1;
        const long long v = (long long)(int)(c >> 32) * (int)h;
        const unsigned long long u = wide(h, (unsigned)c);
        const unsigned long long Y =
            ((unsigned long long)R << 32) + (unsigned long long)(v << (32 - SHIFT)) + (u >> SHIFT) - 8ULL;
        const unsigned long long m = (Y >> 11) + ((Y >> 10) & 1ULL);
        return __longlong_as_double((long long)(((unsigned long long)field << 32) + m));
    }

    // 1/x for normal x with a normal reciprocal
    static __device__ __forceinline__ double rcp(double x) {
        const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
        const unsigned Xh = __funnelshift_l(lo, significand_hi(hi), 11), Xl = lo << 11;   // m 2^63, m in [1, 2)
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float((Xh >> 8) + 0x3F000000u)));
        const unsigned R = fraction(r);
        // e = 1 - m r in units of 2^-63, |e| < 2^-21
        const unsigned long long p = wide(Xh, R, wide(Xl, R) >> 32);
        const long long e = (long long)(0x8000000000000000ULL - p);
        const int es = (int)(e >> 11);
        const long long c = e + (((long long)es * es) >> 41);                             // e + e^2
        const unsigned field = (2044u << 20) - (hi & 0x7FF00000u);
        const double y = scaled_fraction<30>(R, c, field);
        return __hiloint2double(__double2hiint(y) | (int)(hi & 0x80000000u), __double2loint(y));
    }

    // sqrt(x) and, as y, 1/sqrt(x), for normal x; both 0 for x = 0 and below the normal range
    template <bool INVERSE>
    static __device__ __forceinline__ double root(double x, double& y) {
        const int hi = __double2hiint(x);
        const unsigned lo = (unsigned)__double2loint(x);
        const unsigned e = (unsigned)hi >> 20;
        const unsigned odd = e & 1u;                         // an even power of two: x' = m, else x' = 2 m
        const unsigned s = 11u - odd;
        const unsigned Xh = __funnelshift_l(lo, significand_hi(hi), s), Xl = lo << s;     // x' 2^62, x' in [1, 4)
        const unsigned frac = __funnelshift_l(lo, (unsigned)hi, 3) & 0x7FFFFFu;
        float r;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(frac | (0x40000000u - (odd << 23)))));
        const unsigned R = fraction(r);
        const unsigned long long t = wide(Xh, R, wide(Xl, R) >> 32);                      // x' r, units of 2^-62
        const unsigned th = (unsigned)(t >> 32), tl = (unsigned)t;
        const long long d = (long long)(0x4000000000000000ULL - wide(th, R, wide(tl, R) >> 32));   // 1 - x' r^2
        const int ds = (int)(d >> 11);
        const long long c = (d >> 1) + (((((long long)ds * ds) >> 40) * 3) >> 3);         // d/2 + 3/8 d^2
        const int ch = (int)(c >> 32);
        const unsigned long long S = t + (unsigned long long)(((long long)(int)th * ch) << 2) +
                                     (wide(th, (unsigned)c) >> 30) +
                                     (unsigned long long)(((long long)(int)(tl >> 1) * ch) >> 29);
        const unsigned long long m = (S >> 10) + ((S >> 9) & 1ULL);
        const unsigned er = (e + 1023u) >> 1;
        const bool none = hi < 0x00100000;
        if constexpr (INVERSE) {
            y = scaled_fraction<29>(R, c, (2044u - er) << 20);
            if (none) y = 0.0;
        }
        const double v = __longlong_as_double((long long)(((unsigned long long)((er - 1u) << 20) << 32) + m));
        return none ? 0.0 : v;
    }
    static __device__ __forceinline__ double sqrt_(double x) {
        double y;
        return root<false>(x, y);
    }
    static __device__ __forceinline__ double sqrt_rsqrt(double x, double& y) { return root<true>(x, y); }
};

// Soft's values with products on the FP64 pipe, for a kernel that runs a warp
// or less per SM quarter: there a chain of products takes 64 clocks each on
// the pipe and about 130 on the integer unit.
struct SoftRoots : Soft {
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
};

// For adjoints, whose products may become as small as they like.
struct SoftFlush : Soft {
    static __device__ __forceinline__ double mul(double a, double b) { return product<true>(a, b); }
};

// CUDA's operations, for the operands that neither takes: denormal numbers,
// infinities, exponents near the ends of the range.
struct Rare {
    static constexpr bool kRare = true;
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
    static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
};

// Hard's, for normal operands and zero
__device__ __forceinline__ double rcp(double x) { return Hard::rcp(x); }
__device__ __forceinline__ double sqrt_(double x) { return Hard::sqrt_(x); }
__device__ __forceinline__ double sqrt_rsqrt(double x, double& y) { return Hard::sqrt_rsqrt(x, y); }

// x^(-1/3) for a normal x in the FP32 range: y0 (1 + e/3 + 2/9 e^2) from the
// FP32 reciprocal cube root (about 2^-22), the conversions by their bits
template <typename A = Hard>
__device__ __forceinline__ double rcbrt(double x) {
    const long long rebias = 896LL << 23;                      // (1023 - 127) at the FP32 exponent's place
    const float xf = __int_as_float((int)((__double_as_longlong(x) >> 29) - rebias));
    const double y = __longlong_as_double(((long long)__float_as_int(rcbrtf(xf)) + rebias) << 29);
    const double e = fma(-x, A::mul(A::mul(y, y), y), 1.0);
    const double p = A::mul(fma(2.0 / 9.0, e, 1.0 / 3.0), e);
    return fma(y, p, y);
}

// ---- Riemann flux in the edge-normal frame (Eq 14, 17-26) ------------------------------
// Readings as in riemann_hllc.  PL, PR receive g h_K^2 / 2; `speeds`, if given,
// S_L, S_R, S*.
template <typename A>
__device__ __forceinline__ void riemann(double hL, double unL, double utL, double hR, double unR, double utR,
                                        double g2, double h_dry, double& G1, double& G2, double& G3, double& PL,
                                        double& PR, double* speeds, bool hll_only) {
    const bool wetL = gt_pos(hL, h_dry), wetR = gt_pos(hR, h_dry);
    const double ghL = A::mul(g2, hL), ghR = A::mul(g2, hR);
    PL = A::mul(ghL, hL);
    PR = A::mul(ghR, hR);
    if (!wetL && !wetR) {
        G1 = 0.0; G2 = 0.0; G3 = 0.0;
        if (speeds) { speeds[0] = 0.0; speeds[1] = 0.0; speeds[2] = 0.0; }
        return;
    }
    double aL, aR;
    if constexpr (A::kRare) {
        aL = A::sqrt_(A::mul(add(g2, g2), hL));
        aR = A::sqrt_(A::mul(add(g2, g2), hR));
    } else {
        aL = A::sqrt_(twice(ghL));
        aR = A::sqrt_(twice(ghR));
    }
    double SL, SR;
    if (wetL && wetR) {
        SL = sub(unL, aL);                                                     // Eq 19 with p = 1
        SR = add(unR, aR);
        const double asum = add(aL, aR), hsum = add(hL, hR), du = sub(unR, unL);
        // h0 = hsum w / (4 asum), w = 2 asum - du (Eq 21): h0 > min(h_L, h_R) without dividing
        const double w = fma(2.0, asum, -du), hmin = min_nonneg(hL, hR);
        bool shock;
        double rh0 = 0.0;
        if constexpr (A::kRare) {   // by quotients, which neither under- nor overflow first
            const double q = w / asum;
            shock = hsum / hmin * q > 4.0;
            if (shock) rh0 = 4.0 / q / hsum;
        } else {
            const double hw = A::mul(hsum, w), asum4 = four_times(asum);
            shock = gt_pos(hw, A::mul(hmin, asum4));
            if (shock) rh0 = A::mul(asum4, A::rcp(hw));
        }
        if (shock) {                                                           // Eq 23
            const double rL = A::rcp(hL), rR = A::rcp(hR);
            const double gL = A::sqrt_(A::mul(g2, add(rh0, rL))), gR = A::sqrt_(A::mul(g2, add(rh0, rR)));
            const double hs = A::mul(fma(hL, gL, fma(hR, gR, -du)), A::rcp(add(gL, gR)));
            const double ghs = A::mul(g2, hs);
            if (gt_pos(hs, hL)) SL = sub(unL, A::sqrt_(A::mul(ghs, fma(hs, rL, 1.0))));   // Eq 20
            if (gt_pos(hs, hR)) SR = add(unR, A::sqrt_(A::mul(ghs, fma(hs, rR, 1.0))));
        }
    } else if (wetL) {                                                         // Eq 26
        SL = sub(unL, aL);
        SR = fma(2.0, aL, unL);
    } else {
        SL = fma(-2.0, aR, unR);
        SR = add(unR, aR);
    }
    const double qL = A::mul(hL, unL), qR = A::mul(hR, unR);
    const bool supL = ge_zero(SL), supR = !supL && le_zero(SR);
    bool upL = supL;
    if (supL) {                                                                // Eq 17
        G1 = qL;
        G2 = fma(qL, unL, PL);
        if (hll_only) G3 = A::mul(G1, utL);
    } else if (supR) {
        G1 = qR;
        G2 = fma(qR, unR, PR);
        if (hll_only) G3 = A::mul(G1, utR);
        upL = wetL && !wetR && ge_zero(SR);
    } else {                                                                   // Eq 18
        const double r = A::rcp(sub(SR, SL));
        const double ss = A::kRare ? SR * r * SL : A::mul(SR, SL);
        const double fL = fma(qL, unL, PL), fR = fma(qR, unR, PR);
        if constexpr (A::kRare) {   // the weights first: S F may overflow
            const double wL = SR * r, wR = -SL * r;
            G1 = fma(ss, sub(hR, hL), fma(wR, qR, wL * qL));
            G2 = fma(ss, sub(qR, qL), fma(wR, fR, wL * fL));
            if (hll_only) G3 = fma(ss, hR * utR - hL * utL, fma(wR, qR * utR, wL * (qL * utL)));
        } else {
            G1 = A::mul(fma(ss, sub(hR, hL), fma(-SL, qR, A::mul(SR, qL))), r);
            G2 = A::mul(fma(ss, sub(qR, qL), fma(-SL, fR, A::mul(SR, fL))), r);
            if (hll_only) {
                const double tL = A::mul(qL, utL), tR = A::mul(qR, utR);
                G3 = A::mul(fma(ss, sub(A::mul(hR, utR), A::mul(hL, utL)), fma(-SL, tR, A::mul(SR, tL))), r);
            }
        }
        upL = wetL && (!wetR || ge_zero(G1));
    }
    if (!hll_only) G3 = A::mul(G1, upL ? utL : utR);                              // Eq 24
    if (speeds) {
        speeds[0] = SL;
        speeds[1] = SR;
        if (wetL && wetR) {                                                    // Eq 25
            const double mL = A::mul(hL, sub(unL, SL)), mR = A::mul(hR, sub(unR, SR));
            speeds[2] = A::mul(fma(SL, mR, -A::mul(SR, mL)), A::rcp(sub(mR, mL)));
        } else {
            speeds[2] = wetL ? SR : SL;
        }
    }
}

// The flux of inputs that Hard does not take, out of line.
struct FluxAndSpeeds { double G1, G2, G3, S[3]; };
static __device__ __noinline__ FluxAndSpeeds riemann_rare(double hL, double unL, double utL, double hR, double unR,
                                                          double utR, double g2, double h_dry, bool hll_only) {
    FluxAndSpeeds r;
    double PL, PR;
    riemann<Rare>(hL, unL, utL, hR, unR, utR, g2, h_dry, r.G1, r.G2, r.G3, PL, PR, r.S, hll_only);
    return r;
}

// Per unit length, for any states.  Hard takes reciprocals and roots of normal
// numbers in its range, and its products keep clear of under- and overflow
// where they are compared.  (A mesh's wet depths are 2^-126 at least, so its
// cells and edges need no test for it; the flux alone may be asked for any
// depth and dry threshold.)
__device__ __forceinline__ void riemann_any(double hL, double unL, double utL, double hR, double unR, double utR,
                                            double g2, double h_dry, double& G1, double& G2, double& G3, double* speeds,
                                            bool hll_only) {
    double PL, PR;
    const bool g_ok = __double2hiint(g2) >= 0;   // (roots of negative numbers: NaN in Rare only)
    if (in_range<-64, 24>(hL) && in_range<-64, 24>(hR) && in_range<-100, 40>(unL) && in_range<-100, 40>(utL) &&
        in_range<-100, 40>(unR) && in_range<-100, 40>(utR) && in_range<-64, 24>(g2) && g_ok) {
        riemann<Soft>(hL, unL, utL, hR, unR, utR, g2, h_dry, G1, G2, G3, PL, PR, speeds, hll_only);
    } else if (in_range<-200, 100>(hL) && in_range<-200, 100>(hR) && in_range<-400, 100>(unL) &&
               in_range<-400, 100>(utL) && in_range<-400, 100>(unR) && in_range<-400, 100>(utR) &&
               in_range<-64, 64>(g2) && g_ok) {
        riemann<Hard>(hL, unL, utL, hR, unR, utR, g2, h_dry, G1, G2, G3, PL, PR, speeds, hll_only);
    } else {
        const FluxAndSpeeds r = riemann_rare(hL, unL, utL, hR, unR, utR, g2, h_dry, hll_only);
        G1 = r.G1; G2 = r.G2; G3 = r.G3;
        if (speeds) { speeds[0] = r.S[0]; speeds[1] = r.S[1]; speeds[2] = r.S[2]; }
    }
}

template <typename A>
__device__ __forceinline__ void velocity_by(double h, double hu, double hv, double h_dry, double& u, double& v) {
    u = 0.0;
    v = 0.0;
    if (gt_pos(h, h_dry)) {
        const double r = A::rcp(h);
        u = A::mul(hu, r);
        v = A::mul(hv, r);
    }
}

template <class S = Soft>
__device__ __forceinline__ void velocity(double h, double hu, double hv, double h_dry, double& u, double& v) {
    if (in_range<-64, 24>(h) && in_range<-64, 24>(hu) && in_range<-64, 24>(hv)) velocity_by<S>(h, hu, hv, h_dry, u, v);
    else velocity_by<Hard>(h, hu, hv, h_dry, u, v);
}

// One side of an edge: depth, velocity, bed.
struct Side { double h, u, v, z; };

// What an edge adds to each of its cells' sums, per unit length: the flux
// leaving the cell less its bed source term (Eq 30 with 1/2).  The mass part is
// m for the left cell and -m for the right one; the momentum parts are (xL, yL)
// and -(xR, yR).  The cell's sum multiplies by the length in a fused
// multiply-add: a product rounded per edge would show, since the edges of a
// cell nearly cancel.
struct EdgeTerms { double m, xL, yL, xR, yR; };

// One interior edge in its canonical orientation (L is the cell with the lower
// caller index, (n1, n2) its outward unit normal).  Flux and bed source of
// side K along the normal are G2 - (g/2)(h*_K^2 - h_K^2), so both sides share
// the rotation of G3.
template <typename A>
__device__ __forceinline__ void edge_by(const Side& L, const Side& R, double n1, double n2, double g2, double h_dry,
                                        bool hll_only, EdgeTerms& t) {
    // hydrostatic reconstruction (Eq 28): z* = max(z_L, z_R)
    const double zs = max_finite(L.z, R.z);
    const double hL = max_zero(sub(add(L.h, L.z), zs)), hR = max_zero(sub(add(R.h, R.z), zs));
    // the edge frame (Eq 12)
    const double unL = fma(L.u, n1, A::mul(L.v, n2)), utL = fma(L.v, n1, -A::mul(L.u, n2));
    const double unR = fma(R.u, n1, A::mul(R.v, n2)), utR = fma(R.v, n1, -A::mul(R.u, n2));
    double G1, G2, G3, PL, PR;
    riemann<A>(hL, unL, utL, hR, unR, utR, g2, h_dry, G1, G2, G3, PL, PR, nullptr, hll_only);
    const double sL = fma(-A::mul(g2, L.h), L.h, PL), sR = fma(-A::mul(g2, R.h), R.h, PR);
    const double pL = sub(G2, sL), pR = sub(G2, sR);
    const double t1 = A::mul(G3, n2), t2 = A::mul(G3, n1);
    t.m = G1;
    t.xL = fma(pL, n1, -t1);
    t.yL = fma(pL, n2, t2);
    t.xR = fma(pR, n1, -t1);
    t.yR = fma(pR, n2, t2);
}


// The ranges in which every product of Soft's edge is zero or normal (the
// smallest and the largest have under 16 such factors and their cancelled
// differences: 2^-800 and 2^300), for states far beyond any flow's.
__device__ __forceinline__ bool soft_side(const Side& s) {
    return in_range<-64, 24>(s.h) && in_range<-100, 40>(s.u) && in_range<-100, 40>(s.v) && in_range<-64, 24>(s.z);
}
__device__ __forceinline__ bool soft_edge(double n1, double n2, double g2) {
    return in_range<-64, 1>(n1) && in_range<-64, 1>(n2) && in_range<-64, 24>(g2);
}
static __device__ __noinline__ EdgeTerms edge_hard(Side L, Side R, double n1, double n2, double g2, double h_dry,
                                            bool hll_only) {
    EdgeTerms t;
    edge_by<Hard>(L, R, n1, n2, g2, h_dry, hll_only, t);
    return t;
}
template <class S = Soft>
__device__ __forceinline__ void edge(const Side& L, const Side& R, double n1, double n2, double g2, double h_dry,
                                     bool hll_only, EdgeTerms& t) {
    if (soft_side(L) && soft_side(R) && soft_edge(n1, n2, g2))
        edge_by<S>(L, R, n1, n2, g2, h_dry, hll_only, t);
    else
        t = edge_hard(L, R, n1, n2, g2, h_dry, hll_only);
}

// The momentum part of an edge whose cells are both dry (no flux, only the bed
// source term), for the cell (h, z) with outward unit normal (n1, n2): bit
// for bit what edge() gives that cell.
__device__ __forceinline__ void dry_edge(double h, double z, double zk, double n1, double n2, double g2, double& x,
                                         double& y) {
    const double zs = max_finite(z, zk);
    const double hs = max_zero(sub(add(h, z), zs));
    const double p = -fma(-Hard::mul(g2, h), h, Hard::mul(Hard::mul(g2, hs), hs));
    x = fma(p, n1, 0.0);
    y = fma(p, n2, 0.0);
}

// A boundary edge (Section 3.1): the flux leaving cell c, per unit length, in
// the edge frame.
__device__ __forceinline__ void boundary_flux(int kind, double value, const Side& c, double un, double ut, double g2,
                                              double h_dry, bool hll_only, double& G1, double& G2, double& G3) {
    const double p = Hard::mul(Hard::mul(g2, c.h), c.h);
    if (kind == 0) {                                            // wall
        G1 = 0.0; G2 = p; G3 = 0.0;
    } else if (kind == 1) {                                     // inflow, q per unit length
        G1 = -value;
        G2 = gt_pos(c.h, h_dry) ? fma(Hard::mul(value, value), Hard::rcp(c.h), p) : p;
        G3 = 0.0;
    } else {                                                    // transmissive, fixed stage
        const double hg = kind == 3 ? max_zero(sub(value, c.z)) : c.h;
        double PL, PR;
        riemann<Hard>(c.h, un, ut, hg, un, ut, g2, h_dry, G1, G2, G3, PL, PR, nullptr, hll_only);
    }
}

// A boundary edge's addition to its cell's sums, per unit length.
__device__ __forceinline__ void boundary(int kind, double value, const Side& c, double n1, double n2, double g2,
                                         double h_dry, bool hll_only, double& m, double& x, double& y) {
    const double un = fma(c.u, n1, Hard::mul(c.v, n2)), ut = fma(c.v, n1, -Hard::mul(c.u, n2));
    double G2, G3;
    boundary_flux(kind, value, c, un, ut, g2, h_dry, hll_only, m, G2, G3);
    x = fma(G2, n1, -Hard::mul(G3, n2));
    y = fma(G2, n2, Hard::mul(G3, n1));
}

// ---- the end of one cell update (Eq 37 with friction Eq 33-36, the clamps) ----------------
// From the sums (m, x, y) of the edges' terms: the new (h, qx, qy) into out.
// The friction factor is c = g m^2 h^(-7/3); (1 + a|q|) I + a q q^T/|q| with
// a = dt c / 2 has eigenvalue 1 + 2a|q| along q and 1 + a|q| across it.
template <typename A>
__device__ __forceinline__ void update_by(double h, double qx, double qy, double m, double x, double y, double ia,
                                       double gm2, double dt, double h_dry, double& oh, double& ox, double& oy) {
    const double k = A::mul(dt, ia);
    const double dh = -A::mul(m, k);
    double dx = -A::mul(x, k), dy = -A::mul(y, k);
    if (gt_pos(h, h_dry) && gt_zero(gm2)) {
        const double qq = fma(qx, qx, A::mul(qy, qy));
        if (gt_pos(qq, 1e-300)) {
            double ry;
            const double qn = A::sqrt_rsqrt(qq, ry);                           // |q|, 1/|q|
            const double r = rcbrt<A>(h);
            const double r3 = A::mul(A::mul(r, r), r);                            // 1/h
            const double dtc = A::mul(dt, A::mul(gm2, A::mul(A::mul(r3, r3), r)));      // dt c
            const double c1 = A::mul(dtc, qn);                                 // 2 a |q|
            // rhs: dt (R_q + S_f) + dt/2 J_qh dh, S_f = -c|q|q, J_qh = (7/3) c |q| q / h
            const double kq = A::mul(c1, fma(A::mul(7.0 / 6.0, dh), r3, -1.0));
            const double bx = fma(kq, qx, dx), by = fma(kq, qy, dy);
            const double rd1 = A::rcp(fma(0.5, c1, 1.0)), rd2 = A::rcp(add(c1, 1.0));
            const double w = A::mul(fma(bx, qx, A::mul(by, qy)), A::mul(A::mul(half(dtc), ry), rd2));
            dx = A::mul(fma(-w, qx, bx), rd1);
            dy = A::mul(fma(-w, qy, by), rd1);
        }
    }
    oh = add(h, dh);
    ox = add(qx, dx);
    oy = add(qy, dy);
}

// (the ranges as for edge(): Soft's products stay within 2^-900 and 2^740)
template <class S = Soft>
__device__ __forceinline__ void update(double h, double qx, double qy, double m, double x, double y, double ia,
                                       double gm2, double dt, double h_dry, double& oh, double& ox, double& oy) {
    if (in_range<-64, 24>(h) && in_range<-64, 24>(qx) && in_range<-64, 24>(qy) && in_range<-128, 64>(m) &&
        in_range<-128, 64>(x) && in_range<-128, 64>(y) && in_range<-64, 64>(ia) && in_range<-64, 16>(gm2) &&
        in_range<-64, 24>(dt))
        update_by<S>(h, qx, qy, m, x, y, ia, gm2, dt, h_dry, oh, ox, oy);
    else
        update_by<Hard>(h, qx, qy, m, x, y, ia, gm2, dt, h_dry, oh, ox, oy);
}

// The CFL candidate R h / (h sqrt(g h) + |q|) = R / (sqrt(g h) + |u|) (Eq 15) of a wet state.
template <typename A>
__device__ __forceinline__ double cfl_by(double h, double qx, double qy, double rin, double g) {
    const double qm = A::sqrt_(fma(qx, qx, A::mul(qy, qy)));
    return A::mul(A::mul(rin, h), A::rcp(fma(h, A::sqrt_(A::mul(g, h)), qm)));
}
template <class S = Soft>
__device__ __forceinline__ double cfl_candidate(double h, double qx, double qy, double rin, double g) {
    if (in_range<-64, 24>(h) && in_range<-64, 24>(qx) && in_range<-64, 24>(qy) && in_range<-64, 64>(rin) &&
        in_range<-64, 24>(g))
        return cfl_by<S>(h, qx, qy, rin, g);
    return cfl_by<Hard>(h, qx, qy, rin, g);
}

}  // namespace f64
}  // namespace swe
