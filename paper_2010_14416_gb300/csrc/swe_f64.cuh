// swe_f64.cuh -- the FP64 arithmetic of one cell update (Eq 12-37).
//
// What bounds it.  GB300 executes 2 FP64 operations per clock per SM (a warp
// instruction holds the pipe for 16 clocks), so every FP64 kernel here is
// bound by the number of instructions it puts on that pipe: memory, integer
// and FP32 units idle.  Hence:
//   - reciprocals, square roots and h^(-1/3) are one third-order (Householder)
//     correction of a hardware seed good to 2^-20 or better: with
//     e = 1 - x y0 (reciprocal), 1 - x y0^2 (root) or 1 - x y0^3 (cube root),
//     the error left is of order e^3 < 2^-60, under the rounding of the last
//     operation.  3, 5 and 6 FP64 instructions; IEEE division and square root
//     take 8 to 10 with their range checks;
//   - comparisons, selects and powers of two run on the integer unit
//     (swe_compare.cuh, twice() and four_times() below);
//   - the wave speeds need no star depth where Eq 21 chooses the
//     two-rarefaction estimate (Eq 22): there h* <= min(h_L, h_R), so both
//     factors of Eq 20 are 1;
//   - where they do, a_K p_K = sqrt(g h* (h* + h_K) / (2 h_K)) is formed at once;
//   - Eq 24 needs only the sign of S*.  Eq 25's numerator is minus Eq 18's
//     numerator of the mass flux and its denominator is negative, so between
//     S_L and S_R that is the sign of the mass flux;
//   - an edge's flux and its two bed source terms are combined per edge, times
//     the edge's length, into what each of its cells subtracts (5 numbers), so
//     a cell adds three numbers per edge.
// Measured on GB300 against IEEE division and square root with the textbook
// order of operations: 2^20 Riemann problems 418 -> 215 us, a step of the
// 1M-cell canal with the edge pass 480 -> 317 us, an adjoint step of a
// 250k-cell reach 1,181 -> 568 us.
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

// seeds: the documented approximations of 1/x and 1/sqrt(x) that read the
// upper word of x and write the upper word of the result
__device__ __forceinline__ double rcp_seed(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    // zero, denormals and negative values: 0, so that sqrt_(0) is 0
    return __double2hiint(x) < 0x00100000 ? 0.0 : y;
}

// 1/x for normal x: y0 (1 + e + e^2)
__device__ __forceinline__ double rcp(double x) {
    const double y = rcp_seed(x);
    const double e = fma(-x, y, 1.0);
    return fma(fma(e, e, e), y, y);
}

// sqrt(x) (0 for x below the normal range) and, as y, 1/sqrt(x) (0 there):
// y0 (1 + e/2 + 3/8 e^2)
__device__ __forceinline__ double sqrt_rsqrt(double x, double& y) {
    const double y0 = rsqrt_seed(x);
    const double t = mul(x, y0);
    const double e = fma(-t, y0, 1.0);
    const double p = mul(fma(0.375, e, 0.5), e);
    y = fma(y0, p, y0);
    return fma(t, p, t);
}
__device__ __forceinline__ double sqrt_(double x) {
    double y;
    return sqrt_rsqrt(x, y);
}

// x^(-1/3) for a normal x in the FP32 range: y0 (1 + e/3 + 2/9 e^2) from the
// FP32 reciprocal cube root (about 2^-22), the conversions by their bits
__device__ __forceinline__ double rcbrt(double x) {
    const long long rebias = 896LL << 23;                      // (1023 - 127) at the FP32 exponent's place
    const float xf = __int_as_float((int)((__double_as_longlong(x) >> 29) - rebias));
    const double y = __longlong_as_double(((long long)__float_as_int(rcbrtf(xf)) + rebias) << 29);
    const double e = fma(-x, mul(mul(y, y), y), 1.0);
    const double p = mul(fma(2.0 / 9.0, e, 1.0 / 3.0), e);
    return fma(y, p, y);
}

// ---- Riemann flux in the edge-normal frame (Eq 14, 17-26), times `len` -----------------
// Readings as in riemann_hllc.  PL, PR receive g h_K^2 / 2.  Without SCALED
// the flux is per unit length.  `speeds`, if given, receives S_L, S_R, S*.
template <bool SCALED>
__device__ __forceinline__ void riemann(double hL, double unL, double utL, double hR, double unR, double utR,
                                        double g2, double h_dry, double len, double& G1, double& G2, double& G3,
                                        double& PL, double& PR, double* speeds, bool hll_only) {
    const bool wetL = gt_pos(hL, h_dry), wetR = gt_pos(hR, h_dry);
    const double ghL = mul(g2, hL), ghR = mul(g2, hR);
    PL = mul(ghL, hL);
    PR = mul(ghR, hR);
    if (!wetL && !wetR) {
        G1 = 0.0; G2 = 0.0; G3 = 0.0;
        if (speeds) { speeds[0] = 0.0; speeds[1] = 0.0; speeds[2] = 0.0; }
        return;
    }
    const double aL = sqrt_(twice(ghL)), aR = sqrt_(twice(ghR));
    double SL, SR;
    if (wetL && wetR) {
        SL = sub(unL, aL);                                                     // Eq 19 with p = 1
        SR = add(unR, aR);
        const double asum = add(aL, aR), hsum = add(hL, hR), du = sub(unR, unL);
        // h0 = hsum w / (4 asum), w = 2 asum - du (Eq 21): h0 > min(h_L, h_R) without dividing
        const double hw = mul(hsum, fma(2.0, asum, -du));
        const double asum4 = four_times(asum);
        if (gt_pos(hw, mul(min_nonneg(hL, hR), asum4))) {                      // Eq 23
            const double rh0 = mul(asum4, rcp(hw)), rL = rcp(hL), rR = rcp(hR);
            const double gL = sqrt_(mul(g2, add(rh0, rL))), gR = sqrt_(mul(g2, add(rh0, rR)));
            const double hs = mul(fma(hL, gL, fma(hR, gR, -du)), rcp(add(gL, gR)));
            const double ghs = mul(g2, hs);
            if (gt_pos(hs, hL)) SL = sub(unL, sqrt_(mul(ghs, fma(hs, rL, 1.0))));   // Eq 20
            if (gt_pos(hs, hR)) SR = add(unR, sqrt_(mul(ghs, fma(hs, rR, 1.0))));
        }
    } else if (wetL) {                                                         // Eq 26
        SL = sub(unL, aL);
        SR = fma(2.0, aL, unL);
    } else {
        SL = fma(-2.0, aR, unR);
        SR = add(unR, aR);
    }
    const double qL = mul(hL, unL), qR = mul(hR, unR);
    const bool supL = ge_zero(SL), supR = !supL && le_zero(SR);
    bool upL = supL;
    if (supL) {                                                                // Eq 17
        G1 = SCALED ? mul(qL, len) : qL;
        G2 = fma(qL, unL, PL);
        if (SCALED) G2 = mul(G2, len);
        if (hll_only) G3 = mul(G1, utL);
    } else if (supR) {
        G1 = SCALED ? mul(qR, len) : qR;
        G2 = fma(qR, unR, PR);
        if (SCALED) G2 = mul(G2, len);
        if (hll_only) G3 = mul(G1, utR);
        upL = wetL && !wetR && ge_zero(SR);
    } else {                                                                   // Eq 18
        double r = rcp(sub(SR, SL));
        if (SCALED) r = mul(r, len);
        const double ss = mul(SR, SL);
        const double fL = fma(qL, unL, PL), fR = fma(qR, unR, PR);
        G1 = mul(fma(ss, sub(hR, hL), fma(-SL, qR, mul(SR, qL))), r);
        G2 = mul(fma(ss, sub(qR, qL), fma(-SL, fR, mul(SR, fL))), r);
        if (hll_only) {
            const double tL = mul(qL, utL), tR = mul(qR, utR);
            G3 = mul(fma(ss, sub(mul(hR, utR), mul(hL, utL)), fma(-SL, tR, mul(SR, tL))), r);
        }
        upL = wetL && (!wetR || ge_zero(G1));
    }
    if (!hll_only) G3 = mul(G1, upL ? utL : utR);                              // Eq 24
    if (speeds) {
        speeds[0] = SL;
        speeds[1] = SR;
        if (wetL && wetR) {                                                    // Eq 25
            const double mL = mul(hL, sub(unL, SL)), mR = mul(hR, sub(unR, SR));
            speeds[2] = mul(fma(SL, mR, -mul(SR, mL)), rcp(sub(mR, mL)));
        } else {
            speeds[2] = wetL ? SR : SL;
        }
    }
}

__device__ __forceinline__ void velocity(double h, double hu, double hv, double h_dry, double& u, double& v) {
    u = 0.0;
    v = 0.0;
    if (gt_pos(h, h_dry)) {
        const double r = rcp(h);
        u = mul(hu, r);
        v = mul(hv, r);
    }
}

// One side of an edge: depth, velocity, bed.
struct Side { double h, u, v, z; };

// What an edge adds to each of its cells' sums: the flux leaving the cell less
// its bed source term (Eq 30 with 1/2), times the edge's length.  The mass
// part is m for the left cell and -m for the right one; the momentum parts
// are (xL, yL) and -(xR, yR).
struct EdgeTerms { double m, xL, yL, xR, yR; };

// One interior edge in its canonical orientation (L is the cell with the lower
// caller index, (n1, n2) its outward unit normal).  Flux and bed source of
// side K along the normal are G2 - (g/2)(h*_K^2 - h_K^2), so both sides share
// the rotation of G3.
__device__ __forceinline__ void edge(const Side& L, const Side& R, double n1, double n2, double len, double g2,
                                     double h_dry, bool hll_only, EdgeTerms& t) {
    // hydrostatic reconstruction (Eq 28): z* = max(z_L, z_R)
    const double zs = max_finite(L.z, R.z);
    const double hL = max_zero(sub(add(L.h, L.z), zs)), hR = max_zero(sub(add(R.h, R.z), zs));
    // the edge frame (Eq 12)
    const double unL = fma(L.u, n1, mul(L.v, n2)), utL = fma(L.v, n1, -mul(L.u, n2));
    const double unR = fma(R.u, n1, mul(R.v, n2)), utR = fma(R.v, n1, -mul(R.u, n2));
    double G1, G2, G3, PL, PR;
    riemann<true>(hL, unL, utL, hR, unR, utR, g2, h_dry, len, G1, G2, G3, PL, PR, nullptr, hll_only);
    const double sL = fma(-mul(g2, L.h), L.h, PL), sR = fma(-mul(g2, R.h), R.h, PR);
    const double pL = fma(-sL, len, G2), pR = fma(-sR, len, G2);
    const double t1 = mul(G3, n2), t2 = mul(G3, n1);
    t.m = G1;
    t.xL = fma(pL, n1, -t1);
    t.yL = fma(pL, n2, t2);
    t.xR = fma(pR, n1, -t1);
    t.yR = fma(pR, n2, t2);
}

// The momentum part of an edge whose cells are both dry (no flux, only the bed
// source term), for the cell (h, z) with outward unit normal (n1, n2): bit
// for bit what edge() gives that cell.
__device__ __forceinline__ void dry_edge(double h, double z, double zk, double n1, double n2, double len, double g2,
                                         double& x, double& y) {
    const double zs = max_finite(z, zk);
    const double hs = max_zero(sub(add(h, z), zs));
    const double p = fma(-fma(-mul(g2, h), h, mul(mul(g2, hs), hs)), len, 0.0);
    x = fma(p, n1, 0.0);
    y = fma(p, n2, 0.0);
}

// A boundary edge (Section 3.1): the flux leaving cell c, per unit length, in
// the edge frame.
__device__ __forceinline__ void boundary_flux(int kind, double value, const Side& c, double un, double ut, double g2,
                                              double h_dry, bool hll_only, double& G1, double& G2, double& G3) {
    const double p = mul(mul(g2, c.h), c.h);
    if (kind == 0) {                                            // wall
        G1 = 0.0; G2 = p; G3 = 0.0;
    } else if (kind == 1) {                                     // inflow, q per unit length
        G1 = -value;
        G2 = gt_pos(c.h, h_dry) ? fma(mul(value, value), rcp(c.h), p) : p;
        G3 = 0.0;
    } else {                                                    // transmissive, fixed stage
        const double hg = kind == 3 ? max_zero(sub(value, c.z)) : c.h;
        double PL, PR;
        riemann<false>(c.h, un, ut, hg, un, ut, g2, h_dry, 1.0, G1, G2, G3, PL, PR, nullptr, hll_only);
    }
}

// A boundary edge's addition to its cell's sums.
__device__ __forceinline__ void boundary(int kind, double value, const Side& c, double n1, double n2, double len,
                                         double g2, double h_dry, bool hll_only, double& m, double& x, double& y) {
    const double un = fma(c.u, n1, mul(c.v, n2)), ut = fma(c.v, n1, -mul(c.u, n2));
    double G1, G2, G3;
    boundary_flux(kind, value, c, un, ut, g2, h_dry, hll_only, G1, G2, G3);
    const double p = mul(G2, len), s = mul(G3, len);
    m = mul(G1, len);
    x = fma(p, n1, -mul(s, n2));
    y = fma(p, n2, mul(s, n1));
}

// ---- the end of one cell update (Eq 37 with friction Eq 33-36, the clamps) ----------------
// From the sums (m, x, y) of the edges' terms: the new (h, qx, qy) into out.
// The friction factor is c = g m^2 h^(-7/3); (1 + a|q|) I + a q q^T/|q| with
// a = dt c / 2 has eigenvalue 1 + 2a|q| along q and 1 + a|q| across it.
__device__ __forceinline__ void update(double h, double qx, double qy, double m, double x, double y, double ia,
                                       double gm2, double dt, double h_dry, double& oh, double& ox, double& oy) {
    const double k = mul(dt, ia);
    const double dh = -mul(m, k);
    double dx = -mul(x, k), dy = -mul(y, k);
    if (gt_pos(h, h_dry) && gt_zero(gm2)) {
        const double qq = fma(qx, qx, mul(qy, qy));
        if (gt_pos(qq, 1e-300)) {
            double ry;
            const double qn = sqrt_rsqrt(qq, ry);                           // |q|, 1/|q|
            const double r = rcbrt(h);
            const double r3 = mul(mul(r, r), r);                            // 1/h
            const double dtc = mul(dt, mul(gm2, mul(mul(r3, r3), r)));      // dt c
            const double c1 = mul(dtc, qn);                                 // 2 a |q|
            // rhs: dt (R_q + S_f) + dt/2 J_qh dh, S_f = -c|q|q, J_qh = (7/3) c |q| q / h
            const double kq = mul(c1, fma(mul(7.0 / 6.0, dh), r3, -1.0));
            const double bx = fma(kq, qx, dx), by = fma(kq, qy, dy);
            const double rd1 = rcp(fma(0.5, c1, 1.0)), rd2 = rcp(add(c1, 1.0));
            const double w = mul(fma(bx, qx, mul(by, qy)), mul(mul(half(dtc), ry), rd2));
            dx = mul(fma(-w, qx, bx), rd1);
            dy = mul(fma(-w, qy, by), rd1);
        }
    }
    oh = add(h, dh);
    ox = add(qx, dx);
    oy = add(qy, dy);
}

// The CFL candidate R h / (h sqrt(g h) + |q|) = R / (sqrt(g h) + |u|) (Eq 15) of a wet state.
__device__ __forceinline__ double cfl_candidate(double h, double qx, double qy, double rin, double g) {
    const double qm = sqrt_(fma(qx, qx, mul(qy, qy)));
    return mul(mul(rin, h), rcp(fma(h, sqrt_(mul(g, h)), qm)));
}

}  // namespace f64
}  // namespace swe
