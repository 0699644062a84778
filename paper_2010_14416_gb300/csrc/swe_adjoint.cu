// swe_adjoint.cu -- discrete adjoint of the FP64 step (swe_adjoint), frozen-dt
// stepping (swe_step_dt) and parameter updates (swe_set_fields).
//
// The loss is L = sum_g (h_g^N - target_g)^2 after N steps with the step
// sizes frozen at the forward run's values.  With U^{n+1} = F(U^n; z, m) the
// adjoint state lambda^n = (dF/dU^n)^T lambda^{n+1} runs backwards from
// lambda^N = dL/dU^N, accumulating dL/dz and dL/dm on the way.  Cell i's
// update is U_i + Phi(U_i, m_i, R_i), R_i = (1/|Omega_i|) sum_e E_ie, where
// E_ie is the edge's flux-and-bed-source contribution (Eq 13, 30, 37).  One
// reverse step, without atomics:
//   phase 1 (cell i): R_i again, from the edge terms that the forward kept or
//     inline; the transpose of Phi -> own term a_i, dL/dm_i,
//     nu_i = (dPhi/dR)^T lambda / |Omega_i|
//   phase 2:
//     lambda^n_j = a_j + sum_e (dE_je)^T nu_j + (dE_ie)^T nu_i,  dL/dz_j likewise.
// By default the transposes are written out by hand and phase 2 takes each
// interior edge once for both of its cells, then sums a cell's edges in the
// same kernel as the step before's phase 1.  SWE_ADJOINT_DUAL differentiates
// the forward's formulas on dual numbers instead (seven components for Phi,
// four for an edge, from both cells), as a check.  Either follows the branches
// that the forward takes.  Where the states of all steps do not fit, they are
// recomputed segment by segment from checkpoints.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <utility>
#include <vector>

#include "swe_dual.cuh"
#include "swe_internal.h"

using namespace swe;

namespace {

using D4 = Dual<4>;
using D7 = Dual<7>;

struct AdjArgs {
    const V4<double>* __restrict__ U;     // state U^n, internal order
    const V4<double>* __restrict__ geoA;
    const V4<double>* __restrict__ geoB;
    const V4<double>* __restrict__ geoR;  // lengths of the three edges
    const int4* __restrict__ topo;
    const double* __restrict__ gm2;
    V4<double>* __restrict__ lam;         // lambda (h, hu, hv, -)
    V4<double>* __restrict__ aw;          // own term of phase 1
    V4<double>* __restrict__ nu;          // (dPhi/dR)^T lambda / |Omega|
    double* __restrict__ gm;              // dL/d(g m^2), accumulated
    double* __restrict__ gz;              // dL/dz, accumulated
    long long n;
    double dt, g, h_dry;
    int hll;
    BcTable bc;
    // phase 1 with the edge pass: the interior fluxes of U^n from edge_flux_kernel
    const V4<double>* __restrict__ eflux;
    const double* __restrict__ esrc;
    const int4* __restrict__ eidx;
    long long n_edges;
    // phase 2 on transposes: the interior edges (canonical orientation), their
    // unit normals and lengths, and per edge the adjoints of its two cells' states
    const int2* __restrict__ ecells;
    const double* __restrict__ eln;
    const double* __restrict__ erl;
    V4<double>* __restrict__ ed;
    // debug checks: neighbour codes and edge indices are checked before use
    int debug;
    int n_groups;
    unsigned* status;
};

// a neighbour code of cell i checked before use when debug checks are on: an
// unusable one is flagged and taken as a wall (group 0)
__device__ __forceinline__ int adj_code(const AdjArgs& a, int c) {
    if (a.debug && !code_ok(c, a.n, a.n_groups)) {
        atomicOr(a.status, kStatusBadIndex);
        return -1;
    }
    return c;
}

// the outward unit normal and length of local edge j
__device__ __forceinline__ void edge_geo(const V4<double>& gA, const V4<double>& gB, const V4<double>& gR, int j,
                                         double& n1, double& n2, double& len) {
    n1 = j == 0 ? gA.x : (j == 1 ? gA.z : gB.x);
    n2 = j == 0 ? gA.y : (j == 1 ? gA.w : gB.y);
    len = j == 0 ? gR.x : (j == 1 ? gR.y : gR.z);
}

// Reverse of the semi-implicit friction update (f64::update, Eq 33-37) at
// (h, qx, qy, g m^2, Rh, Rx, Ry): for the adjoints (bdh, bdqx, bdqy) of
// (dh, dqx, dqy), the adjoints w[0..6] of the seven inputs, in the order of
// the dual-number seeds.  Reciprocals and roots as in the forward
// (swe_f64.cuh): the FP64 pipe bounds this kernel too.
template <class A>
__device__ __forceinline__ void friction_rev(double hi, double qx, double qy, double gm2, double Rh, double Rx,
                                             double Ry, double dt, double h_dry, double bdh, double bdqx, double bdqy,
                                             double w[7]) {
    using f64::add, f64::fma;
    const double qq = fma(qx, qx, A::mul(qy, qy));
    const bool act = gt_pos(hi, h_dry) && gt_zero(gm2) && gt_pos(qq, 1e-300);
#pragma unroll
    for (int k = 0; k < 7; ++k) w[k] = 0.0;
    if (!act) {
        w[4] = A::mul(bdh, dt); w[5] = A::mul(bdqx, dt); w[6] = A::mul(bdqy, dt);
        return;
    }
    const double dh = A::mul(dt, Rh);
    // forward
    double rq;
    const double qn = A::sqrt_rsqrt(qq, rq);                    // |q|, 1/|q|
    const double r = f64::rcbrt<A>(hi);
    const double rh = A::mul(A::mul(r, r), r);                  // 1/h
    const double p = A::mul(A::mul(rh, rh), r);                 // h^(-7/3)
    const double cf = A::mul(gm2, p);
    const double dtc = A::mul(dt, cf), al = f64::half(dtc);
    const double dhr = A::mul(dh, rh);
    const double P = fma(7.0 / 6.0, dhr, -1.0);
    const double c1 = A::mul(dtc, qn), k = A::mul(c1, P);
    const double bx = fma(k, qx, A::mul(dt, Rx)), by = fma(k, qy, A::mul(dt, Ry));
    const double rd1 = A::rcp(fma(0.5, c1, 1.0)), rd2 = A::rcp(add(1.0, c1));
    const double alq = A::mul(al, A::mul(rq, rd2));             // al / (|q| d2)
    const double S = fma(bx, qx, A::mul(by, qy));
    const double proj = A::mul(S, alq);
    // reverse: dq = (b - proj q) / d1
    const double ox = A::mul(fma(-proj, qx, bx), rd1), oy = A::mul(fma(-proj, qy, by), rd1);
    double b_bx = A::mul(bdqx, rd1), b_by = A::mul(bdqy, rd1);
    const double bd1 = -fma(b_bx, ox, A::mul(b_by, oy));        // of d1, through 1/d1
    const double b_proj = -fma(b_bx, qx, A::mul(b_by, qy));
    double b_qx = -A::mul(b_bx, proj), b_qy = -A::mul(b_by, proj);
    // proj = S al / (|q| d2)
    const double b_S = A::mul(b_proj, alq);
    const double b_pp = A::mul(b_proj, proj);
    const double b_d2 = -A::mul(b_pp, rd2);
    double b_qn = -A::mul(b_pp, rq);
    // al in proj, and in d1 = 1 + al |q|, d2 = d1 + al |q|
    const double b_aq = fma(2.0, b_d2, bd1);
    const double b_al = fma(b_aq, qn, A::mul(A::mul(b_proj, S), A::mul(rq, rd2)));
    b_qn = fma(b_aq, al, b_qn);
    b_bx = fma(b_S, qx, b_bx); b_qx = fma(b_S, bx, b_qx);
    b_by = fma(b_S, qy, b_by); b_qy = fma(b_S, by, b_qy);
    // b = dt R_q + k q
    const double b_k = fma(b_bx, qx, A::mul(b_by, qy));
    b_qx = fma(b_bx, k, b_qx); b_qy = fma(b_by, k, b_qy);
    // k = dt c |q| P, P = (7/6) dh / h - 1
    const double b_kP = A::mul(b_k, P);
    const double b_cf = A::mul(dt, fma(b_kP, qn, f64::half(b_al)));
    b_qn = fma(b_kP, dtc, b_qn);
    const double b_P = A::mul(A::mul(b_k, c1), 7.0 / 6.0);
    const double b_dh = fma(b_P, rh, bdh);
    // c = g m^2 h^(-7/3), 1/h, |q|
    const double b_qq = A::mul(b_qn, rq);
    w[0] = -A::mul(rh, fma(b_P, dhr, A::mul(7.0 / 3.0, A::mul(b_cf, cf))));
    w[1] = fma(b_qq, qx, b_qx);
    w[2] = fma(b_qq, qy, b_qy);
    w[3] = A::mul(b_cf, p);
    w[4] = A::mul(b_dh, dt); w[5] = A::mul(b_bx, dt); w[6] = A::mul(b_by, dt);
}

// The ranges that SoftFlush takes; beyond them the FP64 pipe.  Its products
// must stay below 2^1024 (smaller ones than 2^-1022 become 0): with adjoints
// below 2^100, wet depths from 2^-40 (so h_dry at least that) to 2^24, |u|
// below 2^20, g/2 within 2^-16 to 2^16, lengths below 2^40 and, in the friction
// update, |q| and dt below 2^24, g m^2 below 2^16 and right-hand sides below
// 2^64, multiplying the factors' bounds along the chains, with a_K and 1/a_K of
// the smallest and largest depth, 1/(S_R - S_L) <= 1/max|S_K| and rcp(1 + x) <= 1,
// gives at most 2^716 through an edge and 2^880 through the friction update.
__device__ __forceinline__ bool soft_adjoint(double x) { return f64::in_range<-400, 100>(x); }
__device__ __forceinline__ bool soft_scheme(double g2, double h_dry) {
    return f64::in_range<-16, 16>(g2) && f64::in_range<-40, 24>(h_dry);
}
// |q| / h < 2^20 by the exponents (a dry cell's velocity is not formed)
__device__ __forceinline__ bool slow(double q, double h) {
    return (__double2hiint(q) & 0x7FF00000) - (__double2hiint(h) & 0x7FF00000) < (20 << 20);
}

// EDGES reads R_i's interior fluxes from the edge pass (the forward's own
// edge-pass arithmetic) instead of evaluating them; R_i is the same bit for bit.
// TRANSPOSE transposes the friction update by hand (friction_rev) instead of
// running it on seven-component duals.
// `st` is the step whose update is transposed, L the cell's lambda after it.
struct AdjStep {
    const V4<double>* U;               // state U^n
    const V4<double>* eflux;           // edge terms of U^n, with the edge pass
    const double* esrc;
    double dt;
};
template <bool EDGES, bool TRANSPOSE>
__device__ __forceinline__ void adj_phase1(const AdjArgs& a, const AdjStep& st, long long i, const V4<double>& L) {
    if (TRANSPOSE && ((__double_as_longlong(L.x) | __double_as_longlong(L.y) | __double_as_longlong(L.z)) << 1) == 0LL &&
        !a.debug) {
        // a cell that no gauge's influence has reached yet passes nothing on
        V4<double> zero;
        zero.x = zero.y = zero.z = zero.w = 0.0;
        a.aw[i] = zero;
        a.nu[i] = zero;
        return;
    }
    const double g = a.g, h_dry = a.h_dry;
    const V4<double> own = st.U[i];
    const V4<double> gA = a.geoA[i], gB = a.geoB[i], gR = a.geoR[i];
    const int4 tp = a.topo[i];
    const int code[3] = {adj_code(a, tp.x), adj_code(a, tp.y), adj_code(a, tp.z)};
    const double hi = own.x, zi = own.w;
    double ui, vi;
    cell_velocity<double>(hi, own.y, own.z, h_dry, ui, vi);
    // the forward's explicit right-hand side R_i
    const double g2 = f64::mul(0.5, g);
    const f64::Side own_side{hi, ui, vi, zi};
    double m = 0.0, x = 0.0, y = 0.0;
    int4 ei = make_int4(-1, -1, -1, 0);
    if constexpr (EDGES) ei = a.eidx[i];
    for (int j = 0; j < 3; ++j) {
        double n1, n2, len;
        edge_geo(gA, gB, gR, j, n1, n2, len);
        double tm = 0.0, tx, ty;
        const int c = code[j];
        if (c >= 0) {
            const V4<double> o = st.U[c & kNbrMask];
            const bool flip = (c & kFlipBit) != 0;
            if constexpr (EDGES) {
                if (!gt_pos(hi, h_dry) && !gt_pos(o.x, h_dry)) {
                    f64::dry_edge(hi, zi, o.w, n1, n2, g2, tx, ty);
                } else {
                    int e = j == 0 ? ei.x : (j == 1 ? ei.y : ei.z);
                    if (a.debug && !(e >= 0 && e < a.n_edges)) {
                        atomicOr(a.status, kStatusBadIndex);
                        e = 0;
                    }
                    const V4<double> fl = st.eflux[e];
                    tm = flip ? -fl.x : fl.x;
                    tx = flip ? -fl.w : fl.y;
                    ty = flip ? -st.esrc[e] : fl.z;
                }
            } else {
                f64::Side other{o.x, 0.0, 0.0, o.w};
                f64::velocity(o.x, o.y, o.z, h_dry, other.u, other.v);
                f64::EdgeTerms t;
                f64::edge(flip ? other : own_side, flip ? own_side : other, flip ? -n1 : n1, flip ? -n2 : n2, g2, h_dry,
                          a.hll != 0, t);
                tm = flip ? -t.m : t.m;
                tx = flip ? -t.xR : t.xL;
                ty = flip ? -t.yR : t.yL;
            }
        } else {
            const int grp = -1 - c;
            f64::boundary(a.bc.kind[grp], a.bc.value[grp], own_side, n1, n2, g2, h_dry, a.hll != 0, tm, tx, ty);
        }
        m = f64::fma(len, tm, m);
        x = f64::fma(len, tx, x);
        y = f64::fma(len, ty, y);
    }
    const double ia = gB.z;
    const double Rh = -m * ia, Rx = -x * ia, Ry = -y * ia;
    double lh = L.x, lx_ = L.y, ly_ = L.z;
    double w[7];
    if constexpr (TRANSPOSE) {
        // the forward's clamps (h < 0 zeroes the cell, h <= h_dry zeroes momentum) on
        // the new depth, then the friction update's transpose
        const double hn = f64::add(hi, -f64::mul(m, f64::mul(st.dt, ia)));   // f64::update
        if (hn < 0.0) { lh = 0.0; lx_ = 0.0; ly_ = 0.0; }
        else if (hn <= h_dry) { lx_ = 0.0; ly_ = 0.0; }
        const double gm2 = a.gm2[i];
        if (f64::in_range<-64, 24>(hi) && f64::in_range<-64, 24>(own.y) && f64::in_range<-64, 24>(own.z) &&
            f64::in_range<-64, 16>(gm2) && f64::in_range<-64, 24>(st.dt) && f64::in_range<-192, 64>(Rh) &&
            f64::in_range<-192, 64>(Rx) && f64::in_range<-192, 64>(Ry) && soft_adjoint(lh) && soft_adjoint(lx_) &&
            soft_adjoint(ly_) && soft_scheme(g2, h_dry))
            friction_rev<f64::SoftFlush>(hi, own.y, own.z, gm2, Rh, Rx, Ry, st.dt, h_dry, lh, lx_, ly_, w);
        else
            friction_rev<f64::Hard>(hi, own.y, own.z, gm2, Rh, Rx, Ry, st.dt, h_dry, lh, lx_, ly_, w);
    } else {
        // Phi on duals: seeds h, hu, hv, g m^2, Rh, Rx, Ry
        D7 dh, dqx, dqy;
        friction_update<D7>(D7::seed(hi, 0), D7::seed(own.y, 1), D7::seed(own.z, 2), D7::seed(a.gm2[i], 3),
                            D7::seed(Rh, 4), D7::seed(Rx, 5), D7::seed(Ry, 6), D7(st.dt), D7(h_dry), dh, dqx, dqy);
        // the forward's clamps: h < 0 zeroes the cell, h <= h_dry zeroes momentum
        const double hn = hi + dh.v;
        if (hn < 0.0) { lh = 0.0; lx_ = 0.0; ly_ = 0.0; }
        else if (hn <= h_dry) { lx_ = 0.0; ly_ = 0.0; }
#pragma unroll
        for (int k = 0; k < 7; ++k) w[k] = lh * dh.d[k] + lx_ * dqx.d[k] + ly_ * dqy.d[k];
    }
    V4<double> own_term;
    own_term.x = lh + w[0];
    own_term.y = lx_ + w[1];
    own_term.z = ly_ + w[2];
    own_term.w = 0.0;
    a.aw[i] = own_term;
    a.gm[i] += w[3];
    V4<double> nu;
    nu.x = w[4] * ia;
    nu.y = w[5] * ia;
    nu.z = w[6] * ia;
    nu.w = 0.0;
    a.nu[i] = nu;
}

template <bool EDGES, bool TRANSPOSE>
__global__ void __launch_bounds__(128) adj_phase1_kernel(const AdjArgs a) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    adj_phase1<EDGES, TRANSPOSE>(a, AdjStep{a.U, a.eflux, a.esrc, a.dt}, i, a.lam[i]);
}

__global__ void __launch_bounds__(128) adj_phase2_kernel(const AdjArgs a) {
    const long long jc = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (jc >= a.n) return;
    const double g = a.g, h_dry = a.h_dry;
    const V4<double> own = a.U[jc];
    const V4<double> gA = a.geoA[jc], gB = a.geoB[jc], gR = a.geoR[jc];
    const int4 tp = a.topo[jc];
    const int code[3] = {adj_code(a, tp.x), adj_code(a, tp.y), adj_code(a, tp.z)};
    const V4<double> nuj = a.nu[jc];
    const D4 H = D4::seed(own.x, 0), QX = D4::seed(own.y, 1), QY = D4::seed(own.z, 2), Z = D4::seed(own.w, 3);
    D4 U, V;
    cell_velocity<D4>(H, QX, QY, D4(h_dry), U, V);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int j = 0; j < 3; ++j) {
        double n1, n2, len;
        edge_geo(gA, gB, gR, j, n1, n2, len);
        const double lx = len * n1, ly = len * n2;
        const int c = code[j];
        D4 F0, F1, F2;
        if (c >= 0) {
            const long long i = c & kNbrMask;
            const V4<double> o = a.U[i];
            D4 src;
            edge_interior<D4>(H, U, V, Z, D4(o.x), D4(o.y), D4(o.z), D4(o.w), D4(n1), D4(n2), (c & kFlipBit) != 0,
                              D4(g), D4(h_dry), F0, F1, F2, src, a.hll != 0);
            // this cell's term E_je = (-len F0, -len F1 + src lx, -len F2 + src ly)
            // the neighbour's E_ie = (len F0, len F1 - src_i lx, len F2 - src_i ly),
            // src_i = (g/2)(h**_i^2 - h_i^2) with z* = max(z_i, z_j) as the neighbour forms it
            const D4 zs_i = tmax(D4(o.w), Z);
            const D4 hs_i = tmax(D4(0.0), D4(o.x) + D4(o.w) - zs_i);
            const D4 src_i = D4(0.5 * g) * (hs_i * hs_i - D4(o.x * o.x));
            const V4<double> nui = a.nu[i];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double e0 = -len * F0.d[k];
                const double e1 = -len * F1.d[k] + src.d[k] * lx;
                const double e2 = -len * F2.d[k] + src.d[k] * ly;
                const double o0 = len * F0.d[k];
                const double o1 = len * F1.d[k] - src_i.d[k] * lx;
                const double o2 = len * F2.d[k] - src_i.d[k] * ly;
                acc[k] += nuj.x * e0 + nuj.y * e1 + nuj.z * e2 + nui.x * o0 + nui.y * o1 + nui.z * o2;
            }
        } else {
            const int grp = -1 - c;
            edge_boundary<D4>(a.bc.kind[grp], a.bc.value[grp], H, U, V, Z, D4(n1), D4(n2), D4(g), D4(h_dry), F0, F1,
                              F2, a.hll != 0);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                acc[k] += -len * (nuj.x * F0.d[k] + nuj.y * F1.d[k] + nuj.z * F2.d[k]);
        }
    }
    const V4<double> aw = a.aw[jc];
    V4<double> out;
    out.x = aw.x + acc[0];
    out.y = aw.y + acc[1];
    out.z = aw.z + acc[2];
    out.w = 0.0;
    a.lam[jc] = out;
    a.gz[jc] += acc[3];
}

// ---- hand-written transposes of the edge flux (the default reverse step) ----------
// The reverse of one interior edge's contribution to both of its cells:
// with E_L = (-len F0, -len F1 + src_L lx, -len F2 + src_L ly) the edge's term
// in the left cell's (-f0, sx - f1, sy - f2) and E_R the right cell's
// (its flux is -F, its L n is -(lx, ly)), the step's adjoint needs
// d(nu_L . E_L + nu_R . E_R) / d(h, hu, hv, z) of both cells.  One forward
// evaluation of the edge and one reverse sweep through it give both, where
// the dual-number kernels evaluate the edge from each side on four-component
// duals.  The forward is recomputed here with the arithmetic of swe_f64.cuh,
// whose reciprocals and inverse roots the reverse uses again (no division),
// and every branch is taken as the forward takes it; the derivative of a max
// at a tie is that of the operand the forward returns.  The FP64 pipe bounds
// these kernels too: products, reciprocals and roots run on the integer unit
// (f64::SoftFlush), and an edge or cell whose adjoints are still zero is
// passed over (48 steps back, 64 gauges have reached half of 250k cells):
// 375k edges 188 us before, 1,181 us a step of that adjoint at first, 390
// before these two, 192 with them.

// Reverse of f64::riemann (Eq 17-26) at (hL, unL, utL, hR, unR, utR): adds
// the adjoints of the six inputs for the flux adjoints (bG1, bG2, bG3).
template <class A>
__device__ __forceinline__ void riemann_rev(double hL, double unL, double utL, double hR, double unR, double utR,
                                            double g2, double h_dry, bool hll_only, double bG1, double bG2, double bG3,
                                            double& bhL, double& bunL, double& butL, double& bhR, double& bunR,
                                            double& butR) {
    using f64::add, f64::sub, f64::fma;
    const bool wetL = gt_pos(hL, h_dry), wetR = gt_pos(hR, h_dry);
    if (!wetL && !wetR) return;   // no flux on either side
    const bool wet = wetL && wetR;
    // ---- forward values
    const double ghL = A::mul(g2, hL), ghR = A::mul(g2, hR);
    double yL, yR;                                                              // 1/a_K (0 where a_K = 0)
    const double aL = A::sqrt_rsqrt(f64::twice(ghL), yL), aR = A::sqrt_rsqrt(f64::twice(ghR), yR);
    double SL, SR;
    double w = 0.0, hsum = 0.0, rhw = 0.0, rh0 = 0.0, rL = 0.0, rR = 0.0, gL = 0.0, gR = 0.0, ygL = 0.0, ygR = 0.0,
           rDg = 0.0, hs = 0.0, ycL = 0.0, ycR = 0.0;
    bool shock = false, shL = false, shR = false;
    if (wet) {
        SL = sub(unL, aL);
        SR = add(unR, aR);
        const double asum = add(aL, aR);
        hsum = add(hL, hR);
        const double du = sub(unR, unL);
        w = fma(2.0, asum, -du);
        const double hw = A::mul(hsum, w);
        const double asum4 = f64::four_times(asum);
        shock = gt_pos(hw, A::mul(min_nonneg(hL, hR), asum4));                  // Eq 21
        if (shock) {                                                            // Eq 23
            rhw = A::rcp(hw);
            rh0 = A::mul(asum4, rhw);
            rL = A::rcp(hL);
            rR = A::rcp(hR);
            gL = A::sqrt_rsqrt(A::mul(g2, add(rh0, rL)), ygL);
            gR = A::sqrt_rsqrt(A::mul(g2, add(rh0, rR)), ygR);
            rDg = A::rcp(add(gL, gR));
            hs = A::mul(fma(hL, gL, fma(hR, gR, -du)), rDg);
            const double ghs = A::mul(g2, hs);
            shL = gt_pos(hs, hL);
            shR = gt_pos(hs, hR);
            if (shL) SL = sub(unL, A::sqrt_rsqrt(A::mul(ghs, fma(hs, rL, 1.0)), ycL));   // Eq 20
            if (shR) SR = add(unR, A::sqrt_rsqrt(A::mul(ghs, fma(hs, rR, 1.0)), ycR));
        }
    } else if (wetL) {                                                          // Eq 26
        SL = sub(unL, aL);
        SR = fma(2.0, aL, unL);
    } else {
        SL = fma(-2.0, aR, unR);
        SR = add(unR, aR);
    }
    const double qL = A::mul(hL, unL), qR = A::mul(hR, unR);
    const bool supL = ge_zero(SL), supR = !supL && le_zero(SR);               // Eq 17
    // ---- reverse
    double bSL = 0.0, bSR = 0.0, bqL = 0.0, bqR = 0.0, bPL = 0.0, bPR = 0.0;
    if (supL || supR) {
        // G3 = q ut for either flux; where S* = S_R = 0 the left side's ut (Eq 24)
        const bool left_ut = supL || (!hll_only && wetL && !wetR && ge_zero(SR));
        const double q = supL ? qL : qR;
        const double bq = fma(bG3, left_ut ? utL : utR, bG1);
        if (left_ut) butL = fma(bG3, q, butL);
        else butR = fma(bG3, q, butR);
        if (supL) { bqL = bq; bPL = bG2; }
        else { bqR = bq; bPR = bG2; }
    } else {
        const double r = A::rcp(sub(SR, SL));
        const double ss = A::mul(SR, SL);
        const double fL = fma(qL, unL, A::mul(ghL, hL)), fR = fma(qR, unR, A::mul(ghR, hR));
        const double dh = sub(hR, hL), dq = sub(qR, qL);
        const double SRqL = A::mul(SR, qL);
        const double G1 = A::mul(fma(ss, dh, fma(-SL, qR, SRqL)), r);
        const double G2 = A::mul(fma(ss, dq, fma(-SL, fR, A::mul(SR, fL))), r);
        if (!hll_only) {                                                        // Eq 24
            const bool upL = wetL && (!wetR || ge_zero(G1));
            bG1 = fma(bG3, upL ? utL : utR, bG1);
            if (upL) butL = fma(bG3, G1, butL);
            else butR = fma(bG3, G1, butR);
        } else {
            const double tL = A::mul(qL, utL), tR = A::mul(qR, utR), dt3 = fma(hR, utR, -A::mul(hL, utL));
            const double G3 = A::mul(fma(ss, dt3, fma(-SL, tR, A::mul(SR, tL))), r);
            const double bN3 = A::mul(bG3, r);
            bSR = fma(bN3, sub(fma(SL, dt3, tL), G3), bSR);
            bSL = fma(bN3, add(fma(SR, dt3, -tR), G3), bSL);
            bqL = fma(A::mul(bN3, SR), utL, bqL);
            bqR = fma(-A::mul(bN3, SL), utR, bqR);
            butL = fma(bN3, fma(-ss, hL, SRqL), butL);
            butR = fma(bN3, fma(ss, hR, -A::mul(SL, qR)), butR);
            const double b3s = A::mul(bN3, ss);
            bhR = fma(b3s, utR, bhR);
            bhL = fma(-b3s, utL, bhL);
        }
        // G = N / (S_R - S_L)
        const double bN1 = A::mul(bG1, r), bN2 = A::mul(bG2, r);
        bSR = fma(bN1, sub(fma(SL, dh, qL), G1), fma(bN2, sub(fma(SL, dq, fL), G2), bSR));
        bSL = fma(bN1, add(fma(SR, dh, -qR), G1), fma(bN2, add(fma(SR, dq, -fR), G2), bSL));
        const double b2s = A::mul(bN2, ss), b1s = A::mul(bN1, ss);
        bqL = add(bqL, fma(bN1, SR, -b2s));
        bqR = add(bqR, fma(-bN1, SL, b2s));
        bPL = A::mul(bN2, SR);
        bPR = -A::mul(bN2, SL);
        bhR = add(bhR, b1s);
        bhL = sub(bhL, b1s);
    }
    // f_K = q_K un_K + g h_K^2 / 2, q_K = h_K un_K
    bqL = fma(bPL, unL, bqL);
    bunL = fma(bPL, qL, fma(bqL, hL, bunL));
    bhL = fma(f64::twice(ghL), bPL, fma(bqL, unL, bhL));
    bqR = fma(bPR, unR, bqR);
    bunR = fma(bPR, qR, fma(bqR, hR, bunR));
    bhR = fma(f64::twice(ghR), bPR, fma(bqR, unR, bhR));
    double baL = 0.0, baR = 0.0;
    if (wet) {
        bunL = add(bunL, bSL);
        bunR = add(bunR, bSR);
        if (!shL) baL = -bSL;
        if (!shR) baR = bSR;
        if (shock) {
            double bhs = 0.0;
            if (shL) {   // c_L = sqrt(g/2 (h*^2 / h_L + h*))
                const double t = A::mul(A::mul(-bSL, g2), f64::half(ycL)), x = A::mul(hs, rL);
                bhs = A::mul(t, fma(2.0, x, 1.0));
                bhL = fma(-A::mul(t, x), x, bhL);
            }
            if (shR) {
                const double t = A::mul(A::mul(bSR, g2), f64::half(ycR)), x = A::mul(hs, rR);
                bhs = fma(t, fma(2.0, x, 1.0), bhs);
                bhR = fma(-A::mul(t, x), x, bhR);
            }
            // h* = N / (g_L + g_R), N = h_L g_L + h_R g_R - du
            const double bN = A::mul(bhs, rDg), bNg = A::mul(bN, g2);
            // g_K = sqrt(g/2 (1/h0 + 1/h_K))
            const double xL = A::mul(A::mul(bNg, sub(hL, hs)), f64::half(ygL));
            const double xR = A::mul(A::mul(bNg, sub(hR, hs)), f64::half(ygR));
            // 1/h0 = 4 asum / (hsum w), w = 2 asum - du
            const double b0 = add(xL, xR), b0r = A::mul(A::mul(b0, rh0), rhw);
            const double bw = -A::mul(b0r, hsum);
            bhL = fma(bN, gL, fma(-A::mul(xL, rL), rL, fma(-b0r, w, bhL)));
            bhR = fma(bN, gR, fma(-A::mul(xR, rR), rR, fma(-b0r, w, bhR)));
            const double ba = fma(4.0, A::mul(b0, rhw), f64::twice(bw));
            const double bdu = add(bN, bw);   // of -du
            baL = add(baL, ba); baR = add(baR, ba);
            bunR = sub(bunR, bdu); bunL = add(bunL, bdu);
        }
    } else if (wetL) {                                                          // Eq 26
        bunL = add(bunL, add(bSL, bSR));
        baL = fma(2.0, bSR, -bSL);
    } else {
        bunR = add(bunR, add(bSL, bSR));
        baR = fma(-2.0, bSL, bSR);
    }
    bhL = fma(A::mul(baL, g2), yL, bhL);                                        // a_K = sqrt(g h_K)
    bhR = fma(A::mul(baR, g2), yR, bhR);
}

// Reverse of one interior edge in canonical orientation (left cell L, its
// outward unit normal (n1, n2)): for the adjoints (wF0, wF1, wF2) of the flux
// leaving L and (sL, sR) of the two cells' bed source factors, the adjoints
// of (h, hu, hv, z) of L in dL and of R in dR.
template <class A>
__device__ __forceinline__ void edge_interior_rev(const V4<double>& L, const V4<double>& R, double n1, double n2,
                                                  double len, double g2, double h_dry, bool hll_only,
                                                  const V4<double>& nl, const V4<double>& nr, V4<double>& dL,
                                                  V4<double>& dR) {
    using f64::add, f64::sub, f64::fma;
    // adjoints of the flux leaving L (F in the left cell's term -len F, +len F
    // in the right cell's) and of the bed source factors
    const double bG1 = A::mul(len, sub(nr.x, nl.x));
    const double d1 = A::mul(len, sub(nr.y, nl.y)), d2 = A::mul(len, sub(nr.z, nl.z));
    const double gl = A::mul(f64::twice(g2), len);
    const double gsL = A::mul(gl, fma(nl.y, n1, A::mul(nl.z, n2))), gsR = -A::mul(gl, fma(nr.y, n1, A::mul(nr.z, n2)));
    // forward: velocities (R9), hydrostatic reconstruction (Eq 28), rotation (Eq 12)
    const bool wL = gt_pos(L.x, h_dry), wR = gt_pos(R.x, h_dry);
    const double rL = wL ? A::rcp(L.x) : 0.0, rR = wR ? A::rcp(R.x) : 0.0;
    const double uL = A::mul(L.y, rL), vL = A::mul(L.z, rL), uR = A::mul(R.y, rR), vR = A::mul(R.z, rR);
    const double zs = max_finite(L.w, R.w);   // a tie takes z_R, as the forward
    const bool zleft = __double_as_longlong(zs) != __double_as_longlong(R.w);
    const double xL = sub(add(L.x, L.w), zs), xR = sub(add(R.x, R.w), zs);
    const bool pL = !lt_zero(xL), pR = !lt_zero(xR);
    const double hL = pL ? xL : 0.0, hR = pR ? xR : 0.0;
    const double unL = fma(uL, n1, A::mul(vL, n2)), utL = fma(vL, n1, -A::mul(uL, n2));
    const double unR = fma(uR, n1, A::mul(vR, n2)), utR = fma(vR, n1, -A::mul(uR, n2));
    // reverse: back from (x, y) (Eq 12 inverse)
    const double bG2 = fma(d1, n1, A::mul(d2, n2)), bG3 = fma(d2, n1, -A::mul(d1, n2));
    // bed source factors (Eq 30 with 1/2): src_K = (g/2)(h**_K^2 - h_K^2)
    double bhL = A::mul(gsL, hL), bunL = 0.0, butL = 0.0, bhR = A::mul(gsR, hR), bunR = 0.0, butR = 0.0;
    riemann_rev<A>(hL, unL, utL, hR, unR, utR, g2, h_dry, hll_only, bG1, bG2, bG3, bhL, bunL, butL, bhR, bunR, butR);
    // rotation and velocities (r_K = 0 on a dry side)
    dL.y = A::mul(fma(bunL, n1, -A::mul(butL, n2)), rL);
    dL.z = A::mul(fma(bunL, n2, A::mul(butL, n1)), rL);
    dR.y = A::mul(fma(bunR, n1, -A::mul(butR, n2)), rR);
    dR.z = A::mul(fma(bunR, n2, A::mul(butR, n1)), rR);
    // reconstruction: h*_K = h_K + z_K - z*, z* the higher bed
    if (!pL) bhL = 0.0;
    if (!pR) bhR = 0.0;
    dL.x = fma(-gsL, L.x, fma(-dL.y, uL, fma(-dL.z, vL, bhL)));
    dR.x = fma(-gsR, R.x, fma(-dR.y, uR, fma(-dR.z, vR, bhR)));
    dL.w = zleft ? -bhR : bhL;
    dR.w = zleft ? bhR : -bhL;
}

__device__ __forceinline__ bool soft_state(const V4<double>& s) {
    return f64::in_range<-64, 24>(s.x) && f64::in_range<-64, 24>(s.y) && f64::in_range<-64, 24>(s.z) &&
           f64::in_range<-64, 24>(s.w) && slow(s.y, s.x) && slow(s.z, s.x);
}

// Reverse of a boundary edge's flux (f64::boundary_flux): adds to d the
// adjoints of cell c's (h, hu, hv, z) for the adjoints of the flux leaving it.
// (Out of line: 20 registers less for the cells without one.)
__device__ __noinline__ void boundary_rev(int kind, double value, const V4<double>& c, double n1, double n2,
                                             double g2, double h_dry, bool hll_only, double wF0, double wF1, double wF2,
                                             double d[4]) {
    const double bG1 = wF0, bG2 = wF1 * n1 + wF2 * n2;
    const double gh = f64::twice(g2) * c.x;
    if (kind == kBcWall) {
        d[0] += bG2 * gh;
        return;
    }
    const double r = gt_pos(c.x, h_dry) ? f64::rcp(c.x) : 0.0;
    const double bG3 = wF2 * n1 - wF1 * n2;
    if (kind == kBcInflow) {   // G2 = g h^2 / 2 + q^2 / h
        const double qr = value * r;
        d[0] += bG2 * (gh - qr * qr);
        return;
    }
    const double u = f64::mul(c.y, r), v = f64::mul(c.z, r);
    const double un = f64::fma(u, n1, f64::mul(v, n2)), ut = f64::fma(v, n1, -f64::mul(u, n2));
    const double x = f64::sub(value, c.w);
    const double hg = kind == kBcStage ? max_zero(x) : c.x;
    double bh = 0.0, bun = 0.0, but = 0.0, bhg = 0.0, bung = 0.0, butg = 0.0;
    // (on the FP64 pipe: few warps come here, and a lone warp's chain of Soft
    // operations takes longer than of FP64 instructions)
    riemann_rev<f64::Hard>(c.x, un, ut, hg, un, ut, g2, h_dry, hll_only, bG1, bG2, bG3, bh, bun, but, bhg, bung, butg);
    bun += bung;
    but += butg;
    if (kind == kBcStage) {
        if (!lt_zero(x)) d[3] -= bhg;
    } else {
        bh += bhg;
    }
    const double bx = (bun * n1 - but * n2) * r, by = (bun * n2 + but * n1) * r;
    d[0] += bh - (bx * u + by * v);
    d[1] += bx;
    d[2] += by;
}

__device__ __forceinline__ bool zero3(const V4<double>& v) {
    return ((__double_as_longlong(v.x) | __double_as_longlong(v.y) | __double_as_longlong(v.z)) << 1) == 0LL;
}
// Phase 2, edges: each interior edge once, the adjoints of both cells' states
// through it, into ed[2 e] (left cell) and ed[2 e + 1] (right cell).
__global__ void __launch_bounds__(128) adj_edge_kernel(const AdjArgs a) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < a.n_edges; e += stride) {
        int2 lr = a.ecells[e];
        V4<double> dl, dr;
        dl.x = dl.y = dl.z = dl.w = 0.0;
        dr.x = dr.y = dr.z = dr.w = 0.0;
        if (a.debug && !(lr.x >= 0 && lr.x < a.n && lr.y >= 0 && lr.y < a.n)) {
            atomicOr(a.status, kStatusBadIndex);
            a.ed[2 * e] = dl;
            a.ed[2 * e + 1] = dr;
            continue;
        }
        // both cells' adjoints zero (no gauge's influence has come this far back):
        // so is the edge's
        const V4<double> nl = a.nu[lr.x], nr = a.nu[lr.y];
        if (zero3(nl) && zero3(nr)) {
            a.ed[2 * e] = dl;
            a.ed[2 * e + 1] = dr;
            continue;
        }
        const V4<double> L = a.U[lr.x], R = a.U[lr.y];
        const double n1 = a.eln[2 * e], n2 = a.eln[2 * e + 1], len = a.erl[e];
        const double g2 = f64::mul(0.5, a.g);
        if (soft_state(L) && soft_state(R) && f64::soft_edge(n1, n2, g2) && soft_scheme(g2, a.h_dry) &&
            f64::in_range<-64, 40>(len) && soft_adjoint(nl.x) &&
            soft_adjoint(nl.y) && soft_adjoint(nl.z) && soft_adjoint(nr.x) && soft_adjoint(nr.y) && soft_adjoint(nr.z))
            edge_interior_rev<f64::SoftFlush>(L, R, n1, n2, len, g2, a.h_dry, a.hll != 0, nl, nr, dl, dr);
        else
            edge_interior_rev<f64::Hard>(L, R, n1, n2, len, g2, a.h_dry, a.hll != 0, nl, nr, dl, dr);
        a.ed[2 * e] = dl;
        a.ed[2 * e + 1] = dr;
    }
}

// Phase 2, cells: lambda^n_j = own term + the contributions of j's interior
// edges (in local edge order) + its boundary edges' (own state only);
// dL/dz_j likewise.
__device__ __forceinline__ V4<double> adj_cell(const AdjArgs& a, long long jc) {
    const int4 tp = a.topo[jc];
    const int code[3] = {adj_code(a, tp.x), adj_code(a, tp.y), adj_code(a, tp.z)};
    const int4 ei = a.eidx[jc];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    bool any_boundary = false;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int c = code[j];
        if (c >= 0) {
            int e = j == 0 ? ei.x : (j == 1 ? ei.y : ei.z);
            if (a.debug && !(e >= 0 && e < a.n_edges)) {
                atomicOr(a.status, kStatusBadIndex);
                continue;
            }
            const V4<double> d = a.ed[2 * (long long)e + ((c & kFlipBit) ? 1 : 0)];
            acc[0] += d.x; acc[1] += d.y; acc[2] += d.z; acc[3] += d.w;
        } else {
            any_boundary = true;
        }
    }
    if (any_boundary) {
        const V4<double> own = a.U[jc];
        const V4<double> gA = a.geoA[jc], gB = a.geoB[jc], gR = a.geoR[jc];
        const V4<double> nuj = a.nu[jc];
        for (int j = 0; j < 3; ++j) {
            const int c = code[j];
            if (c >= 0) continue;
            double n1, n2, len;
            edge_geo(gA, gB, gR, j, n1, n2, len);
            const int grp = -1 - c;
            boundary_rev(a.bc.kind[grp], a.bc.value[grp], own, n1, n2, 0.5 * a.g, a.h_dry, a.hll != 0, -len * nuj.x,
                         -len * nuj.y, -len * nuj.z, acc);
        }
    }
    const V4<double> aw = a.aw[jc];
    V4<double> out;
    out.x = aw.x + acc[0];
    out.y = aw.y + acc[1];
    out.z = aw.z + acc[2];
    out.w = 0.0;
    a.gz[jc] += acc[3];
    return out;
}

__global__ void __launch_bounds__(128, 4) adj_cell_kernel(const AdjArgs a) {
    const long long jc = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (jc < a.n) a.lam[jc] = adj_cell(a, jc);
}

// adj_cell_kernel of one step and adj_phase1_kernel of the step before it: the
// cell's lambda passes from one to the other in registers, and a reverse step
// is two launches in place of three, half of each latency on 20,000 cells (a
// reverse step's kernels 38 -> 34 us).
template <bool EDGES>
__global__ void __launch_bounds__(128, 4) adj_cell_phase1_kernel(const AdjArgs a, const AdjStep before) {
    const long long jc = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (jc >= a.n) return;
    const V4<double> lam = adj_cell(a, jc);
    adj_phase1<EDGES, true>(a, before, jc, lam);
}

// loss += sum_g (h_g - target_g)^2 for one observation (one thread: fixed order)
__global__ void adj_loss_kernel(const V4<double>* __restrict__ U, const long long* __restrict__ gauges,
                                const double* __restrict__ target, int n_gauges, double* __restrict__ loss) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double L = *loss;
        for (int k = 0; k < n_gauges; ++k) {
            const double r = U[gauges[k]].x - target[k];
            L += r * r;
        }
        *loss = L;
    }
}

// lambda^n += d(observation)/dU^n: 2 (h_g - target_g) on the gauges' depths
__global__ void adj_inject_kernel(const V4<double>* __restrict__ U, const long long* __restrict__ gauges,
                                  const double* __restrict__ target, int n_gauges, V4<double>* __restrict__ lam) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int k = 0; k < n_gauges; ++k) {
            const long long c = gauges[k];
            lam[c].x += 2.0 * (U[c].x - target[k]);
        }
    }
}

// caller-order gradients: dL/dm = dL/d(g m^2) * 2 g m, dL/dz as is
__global__ void adj_output_kernel(const double* __restrict__ gm, const double* __restrict__ gz,
                                  const double* __restrict__ gm2, const unsigned* __restrict__ inv, double g,
                                  double* __restrict__ out_m, double* __restrict__ out_z, long long n) {
    const long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (o < n) {
        const long long c = inv[o];
        // g m = sqrt(g * g m^2) for m >= 0
        if (out_m) out_m[o] = gm[c] * 2.0 * sqrt(g * gm2[c]);
        if (out_z) out_z[o] = gz[c];
    }
}

template <typename T>
__global__ void set_z_kernel(V4<T>* __restrict__ s0, V4<T>* __restrict__ s1, const T* __restrict__ z, long long n) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) {
        s0[c].w = z[c];
        s1[c].w = z[c];
    }
}

int afail(cudaError_t e, const char* what) {
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return SWE_ECUDA;
}

struct DevBuf {
    void* p = nullptr;
    ~DevBuf() { if (p) cudaFree(p); }
};

// The buffers of one adjoint call, laid out in one allocation that the mesh
// keeps (up to kAdjKeep, all meshes of the process together up to kAdjKeepAll)
// for its next call: allocating and freeing them took 0.4 ms a call and more
// with the checkpoints' size.
constexpr size_t kAdjKeep = (size_t)3 << 29;      // 1.5 GiB of the device's 280
constexpr size_t kAdjKeepAll = (size_t)6 << 30;   // 6 GiB
std::atomic<size_t> adj_kept_all{0};
bool keep_arena(swe_mesh* m) {
    if (m->adj_kept) return true;   // counted
    size_t all = adj_kept_all.load();
    do {
        if (m->adj_bytes > kAdjKeep || all + m->adj_bytes > kAdjKeepAll) return false;
    } while (!adj_kept_all.compare_exchange_weak(all, all + m->adj_bytes));
    m->adj_kept = m->adj_bytes;
    return true;
}
struct AdjArena {
    swe_mesh* m;
    std::vector<std::pair<void**, size_t>> parts;   // (pointer, offset)
    size_t bytes = 0;
    explicit AdjArena(swe_mesh* mesh) : m(mesh) {}
    void add(void** p, size_t b) {
        parts.push_back({p, bytes});
        bytes += (std::max<size_t>(b, 16) + 255) / 256 * 256;
    }
    cudaError_t place() {
        cudaError_t e = cudaSuccess;
        if (m->adj_bytes < bytes) {
            drop_adjoint_workspace(m);
            e = cudaMalloc(&m->adj_arena, bytes);
            if (e != cudaSuccess) {
                m->adj_arena = nullptr;
                return e;
            }
            m->adj_bytes = bytes;
            m->device_bytes += (int64_t)bytes;
        }
        for (auto& q : parts) *q.first = (char*)m->adj_arena + q.second;
        return e;
    }
    // nothing uses the buffers after the call (it may leave early, and the
    // mesh may change its stream before the next)
    ~AdjArena() {
        cudaStreamSynchronize(m->stream);
        if (!keep_arena(m)) drop_adjoint_workspace(m);
    }
};

struct AdjDeviceGuard {
    int prev = -1;
    explicit AdjDeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~AdjDeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

__global__ void small_init_kernel(unsigned long long* small) {
    if (threadIdx.x < kSmallWords) small[threadIdx.x] = threadIdx.x < 3 ? kInfBits : 0ULL;
}

// Observations every obs_every steps (obs_every divides nsteps); targets:
// [nsteps / obs_every][n_gauges].
int adjoint_impl(swe_mesh* m, int64_t nsteps, double cfl, const int32_t* gauge_cells, int n_gauges,
                 const double* targets, int64_t obs_every, int checkpoint_every, double* loss,
                 double* grad_manning, double* grad_bathy, int where, double* dts_out) {
    if (!m || nsteps < 1 || !(cfl > 0.0) || !gauge_cells || n_gauges < 1 || !targets || !loss ||
        (where != SWE_HOST && where != SWE_DEVICE) || checkpoint_every < 0 || obs_every < 1 ||
        nsteps % obs_every != 0) {
        set_error("swe_adjoint: bad arguments");
        return SWE_EINVAL;
    }
    const int64_t n_obs = nsteps / obs_every;
    if (m->cfg.precision != SWE_FP64) { set_error("swe_adjoint: the adjoint runs on FP64 meshes"); return SWE_EINVAL; }
    if (!m->have_state) { set_error("swe_adjoint: no state set"); return SWE_EINVAL; }
    const int64_t n = m->hm.n_cells;
    std::vector<long long> gint(n_gauges);
    for (int k = 0; k < n_gauges; ++k) {
        if (gauge_cells[k] < 0 || gauge_cells[k] >= n) { set_error("swe_adjoint: gauge cell out of range"); return SWE_EINVAL; }
        gint[k] = m->hm.inv[gauge_cells[k]];
    }
    AdjDeviceGuard dg(m->cfg.device);
    int rc = flush_mesh_bc(m);
    if (rc) return rc;
    cudaStream_t st = m->stream;
    const size_t sb = (size_t)n * sizeof(V4<double>);
    const bool transposes = m->adjoint_method == SWE_ADJOINT_TRANSPOSE;
    if (transposes) {   // the interior edge list of the edge-by-edge reverse step
        rc = build_edges(m);
        if (rc) return rc;
    }
    // With the edge pass, a segment's steps keep their edge terms (40 B per
    // interior edge and step), so phase 1 reads those of U^n that the step
    // n -> n+1 formed instead of running the edge pass again; without room for
    // them, phase 1 runs it.
    const bool edges = m->plain.edges && m->eflux;
    const size_t Eb = (size_t)std::max<int64_t>(m->n_edges, 1);
    bool keep = edges && transposes;
    void *p_ckpt, *p_seg, *p_dtlog, *p_small, *p_lam, *p_aw, *p_nu, *p_gm, *p_gz, *p_idx, *p_target, *p_loss, *p_ed,
        *p_flux = nullptr, *p_src = nullptr;
    cudaError_t e = cudaSuccess;
    AdjArena arena(m);
    // K steps a segment, segments recomputed from their checkpoints in reverse:
    // one segment of all steps (nothing recomputed, the same bits) where its
    // states and edge terms fit the kept workspace, else what was asked for.
    const int K_asked = checkpoint_every > 0 ? checkpoint_every : 50;
    int64_t K = K_asked;
    auto layout = [&](int64_t k, bool with_flux) {
        K = k;
        arena.parts.clear();
        arena.bytes = 0;
        arena.add(&p_ckpt, (size_t)((nsteps + K - 1) / K) * sb);
        arena.add(&p_seg, (size_t)K * sb);
        arena.add(&p_dtlog, nsteps * sizeof(double));
        arena.add(&p_small, kSmallWords * sizeof(unsigned long long));
        for (void** p : {&p_lam, &p_aw, &p_nu}) arena.add(p, sb);
        for (void** p : {&p_gm, &p_gz}) arena.add(p, n * sizeof(double));
        arena.add(&p_idx, n_gauges * sizeof(long long));
        arena.add(&p_target, (size_t)n_obs * n_gauges * sizeof(double));
        arena.add(&p_loss, sizeof(double));
        arena.add(&p_ed, transposes ? Eb * 2 * sizeof(V4<double>) : 0);
        if (with_flux) {
            arena.add(&p_flux, (size_t)K * Eb * sizeof(V4<double>));
            arena.add(&p_src, (size_t)K * Eb * sizeof(double));
        }
    };
    auto place = [&]() {
        e = arena.place();
        if (e != cudaSuccess) (void)cudaGetLastError();   // clear the failed allocation's error
        return e == cudaSuccess;
    };
    layout(nsteps, keep);
    if (nsteps <= K_asked || arena.bytes > kAdjKeep || !place()) {
        layout(std::min<int64_t>(K_asked, nsteps), keep);
        if (!place() && keep) {
            keep = false;
            layout(std::min<int64_t>(K_asked, nsteps), false);
            place();
        }
    }
    if (e != cudaSuccess) {
        set_error(std::string("swe_adjoint: device allocation failed: ") + cudaGetErrorString(e));
        return SWE_ENOMEM;
    }
    const int64_t nseg = (nsteps + K - 1) / K;
    if (e == cudaSuccess) e = cudaMemsetAsync(p_loss, 0, sizeof(double), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(p_idx, gint.data(), n_gauges * sizeof(long long), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p_target, targets, (size_t)n_obs * n_gauges * sizeof(double), cudaMemcpyHostToDevice, st);
    const long long* gi = (const long long*)p_idx;
    const double* tg = (const double*)p_target;
    V4<double>* const sflux = (V4<double>*)p_flux;
    double* const ssrc = (double*)p_src;
    // forward run: checkpoints every K steps, step sizes logged, loss summed
    // over the observations.  The last segment's states (and, with the edge
    // pass, the fluxes its steps form) are kept as the reverse sweep's segment
    // buffer: recomputing them would give the same bits (the same kernels and
    // step sizes), so the reverse sweep starts without a recomputation.
    const int64_t last0 = (nseg - 1) * K;   // first step of the last segment
    char* const segp = (char*)p_seg;
    for (int64_t s = 0; s < nsteps && e == cudaSuccess; ++s) {
        void* cur = m->state[m->nstep % 2];
        void* nxt = m->state[(m->nstep + 1) % 2];
        if (s % K == 0) e = cudaMemcpyAsync((char*)p_ckpt + (s / K) * sb, cur, sb, cudaMemcpyDeviceToDevice, st);
        // in the last segment the steps go from one of its states to the next
        const bool in_last = s >= last0;
        const void* in = in_last ? segp + (s - last0) * sb : cur;
        void* out = in_last && s + 1 < nsteps ? segp + (s + 1 - last0) * sb : nxt;
        if (e == cudaSuccess && s == last0)
            e = cudaMemcpyAsync(segp, cur, sb, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess)
            e = launch_step_raw(m, in, out, m->small, m->nstep, cfl, nullptr, (double*)p_dtlog + s, st, false,
                                keep && in_last ? (void*)(sflux + (s - last0) * Eb) : nullptr,
                                keep && in_last ? (void*)(ssrc + (s - last0) * Eb) : nullptr);
        // and the mesh is left with the last two
        if (e == cudaSuccess && in_last && s + 1 == nsteps && s > last0)
            e = cudaMemcpyAsync(cur, in, sb, cudaMemcpyDeviceToDevice, st);
        ++m->nstep;
        m->act_valid = false;   // stepped without the activity bytes
        if (e == cudaSuccess && (s + 1) % obs_every == 0) {
            adj_loss_kernel<<<1, 32, 0, st>>>((const V4<double>*)out, gi, tg + ((s + 1) / obs_every - 1) * n_gauges,
                                             n_gauges, (double*)p_loss);
            e = cudaGetLastError();
        }
    }
    if (e != cudaSuccess) return afail(e, "swe_adjoint: forward");
    std::vector<double> dts(nsteps);
    std::vector<unsigned long long> fstat(kSmallWords);
    e = cudaMemcpyAsync(dts.data(), p_dtlog, nsteps * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(fstat.data(), m->small, kSmallWords * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return afail(e, "swe_adjoint: forward");
    if (fstat[kSlotStatus] & kStatusBadIndex) {
        set_error("swe_adjoint: an index or boundary group out of range in the forward run (debug checks)");
        return SWE_EMESH;
    }
    if (fstat[kSlotStatus] & kStatusStall) return status_code(fstat[kSlotStatus]);
    if (fstat[kSlotStatus] & kStatusNonFinite) { set_error("swe_adjoint: forward run is not finite"); return SWE_ENONFINITE; }
    for (double d : dts)
        if (!std::isfinite(d)) { set_error("swe_adjoint: forward run went dry"); return SWE_EDRY; }
    if (dts_out) std::memcpy(dts_out, dts.data(), nsteps * sizeof(double));
    // lambda^N = d(last observation)/dU^N
    e = cudaMemsetAsync(p_lam, 0, sb, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(p_gm, 0, n * sizeof(double), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(p_gz, 0, n * sizeof(double), st);
    if (e == cudaSuccess) {
        adj_inject_kernel<<<1, 32, 0, st>>>((const V4<double>*)m->state[m->nstep % 2], gi,
                                           tg + (n_obs - 1) * n_gauges, n_gauges, (V4<double>*)p_lam);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) { small_init_kernel<<<1, 32, 0, st>>>((unsigned long long*)p_small); e = cudaGetLastError(); }
    if (e != cudaSuccess) return afail(e, "swe_adjoint: loss");
    AdjArgs a;
    a.geoA = (const V4<double>*)m->geoA;
    a.geoB = (const V4<double>*)m->geoB;
    a.geoR = (const V4<double>*)m->geoR;
    a.topo = m->topo;
    a.gm2 = (const double*)m->gm2;
    a.lam = (V4<double>*)p_lam;
    a.aw = (V4<double>*)p_aw;
    a.nu = (V4<double>*)p_nu;
    a.gm = (double*)p_gm;
    a.gz = (double*)p_gz;
    a.n = n;
    a.g = m->cfg.g;
    a.h_dry = m->cfg.h_dry;
    a.hll = m->cfg.flux == SWE_FLUX_HLL ? 1 : 0;
    a.bc = m->bc;
    a.n_edges = m->n_edges;
    a.debug = m->cfg.debug_checks;
    a.n_groups = m->n_groups;
    a.status = (unsigned*)((unsigned long long*)p_small + kSlotStatus);
    // with the edge pass, phase 1 takes R's interior fluxes from one evaluation per edge
    a.eflux = edges ? (const V4<double>*)m->eflux : nullptr;
    a.esrc = edges ? (const double*)m->esrc : nullptr;
    a.eidx = m->eidx;
    a.ecells = m->ecells;
    a.eln = (const double*)m->eln;
    a.erl = (const double*)m->erl;
    a.ed = (V4<double>*)p_ed;
    StepArgs<double> ea{};
    if (edges) {
        ea.ecells = m->ecells;
        ea.eln = (const double*)m->eln;
        ea.erl = (const double*)m->erl;
        ea.eflux = (V4<double>*)m->eflux;
        ea.esrc = (double*)m->esrc;
        ea.n_edges = m->n_edges;
        ea.g = m->cfg.g;
        ea.h_dry = m->cfg.h_dry;
        ea.hll = a.hll;
        ea.n = n;
        ea.debug = a.debug;
        ea.n_groups = a.n_groups;
        ea.status = a.status;
    }
    // one-warp blocks on a small mesh: 128 threads leave some SMs with twice the
    // others' share (step_threads has the measurements)
    const unsigned eblock = m->n_edges <= kSpreadCells ? 32 : 128, block = n <= kSpreadCells ? 32 : 128;
    const unsigned egrid =
        (unsigned)std::min<int64_t>((std::max<int64_t>(m->n_edges, 1) + eblock - 1) / eblock, 65535);
    const unsigned grid = (unsigned)((n + block - 1) / block);
    // reverse sweep, segment by segment
    for (int64_t sgi = nseg - 1; sgi >= 0 && e == cudaSuccess; --sgi) {
        const int64_t n0 = sgi * K, n1 = std::min<int64_t>(n0 + K, nsteps);
        const bool from_forward = sgi == nseg - 1;   // the forward run kept this segment
        if (!from_forward)
            e = cudaMemcpyAsync(segp, (char*)p_ckpt + sgi * sb, sb, cudaMemcpyDeviceToDevice, st);
        for (int64_t k = 0; !from_forward && k + 1 < n1 - n0 && e == cudaSuccess; ++k)
            e = launch_step_raw(m, segp + k * sb, segp + (k + 1) * sb, (unsigned long long*)p_small, k, cfl,
                                (const double*)p_dtlog + n0 + k, nullptr, st, false,
                                keep ? (void*)(sflux + k * Eb) : nullptr, keep ? (void*)(ssrc + k * Eb) : nullptr);
        if (keep && !from_forward && e == cudaSuccess) {   // the segment's last state has no recomputed step
            const int64_t k = n1 - n0 - 1;
            ea.s_in = (const V4<double>*)(segp + k * sb);
            ea.eflux = sflux + k * Eb;
            ea.esrc = ssrc + k * Eb;
            e = Launch<double>::edge_flux(ea, st);
        }
        bool phase1_done = false;   // by the launch before
        for (int64_t k = n1 - n0 - 1; k >= 0 && e == cudaSuccess; --k) {
            a.U = (const V4<double>*)(segp + k * sb);
            a.dt = dts[n0 + k];
            if (keep) {
                a.eflux = sflux + k * Eb;
                a.esrc = ssrc + k * Eb;
                if (!phase1_done) adj_phase1_kernel<true, true><<<grid, block, 0, st>>>(a);
            } else if (edges) {
                ea.s_in = a.U;
                e = Launch<double>::edge_flux(ea, st);
                if (e != cudaSuccess) break;
                if (transposes) adj_phase1_kernel<true, true><<<grid, block, 0, st>>>(a);
                else adj_phase1_kernel<true, false><<<grid, block, 0, st>>>(a);
            } else if (!phase1_done) {
                if (transposes) adj_phase1_kernel<false, true><<<grid, block, 0, st>>>(a);
                else adj_phase1_kernel<false, false><<<grid, block, 0, st>>>(a);
            }
            // the step before follows at once where its edge terms are at hand and no
            // observation enters lambda in between
            phase1_done = transposes && (keep || !edges) && k > 0 && (n0 + k) % obs_every != 0;
            if (transposes) {
                adj_edge_kernel<<<egrid, eblock, 0, st>>>(a);
                const AdjStep before{(const V4<double>*)(segp + (k - 1) * sb), keep ? sflux + (k - 1) * Eb : nullptr,
                                     keep ? ssrc + (k - 1) * Eb : nullptr, phase1_done ? dts[n0 + k - 1] : 0.0};
                if (phase1_done && keep) adj_cell_phase1_kernel<true><<<grid, block, 0, st>>>(a, before);
                else if (phase1_done) adj_cell_phase1_kernel<false><<<grid, block, 0, st>>>(a, before);
                else adj_cell_kernel<<<grid, block, 0, st>>>(a);
            } else {
                adj_phase2_kernel<<<grid, block, 0, st>>>(a);
            }
            const int64_t nn = n0 + k;  // lambda now holds lambda^nn
            if (nn > 0 && nn % obs_every == 0)
                adj_inject_kernel<<<1, 32, 0, st>>>(a.U, gi, tg + (nn / obs_every - 1) * n_gauges, n_gauges, a.lam);
            e = cudaGetLastError();
        }
    }
    if (e != cudaSuccess) return afail(e, "swe_adjoint: reverse sweep");
    if (m->cfg.debug_checks) {
        unsigned long long rs[kSmallWords];
        e = cudaMemcpyAsync(rs, p_small, sizeof rs, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return afail(e, "swe_adjoint: reverse sweep status");
        if (rs[kSlotStatus] & kStatusBadIndex) {
            set_error("swe_adjoint: an index or boundary group out of range in the reverse sweep (debug checks)");
            return SWE_EMESH;
        }
    }
    // outputs
    if (where == SWE_DEVICE) {
        adj_output_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const double*)p_gm, (const double*)p_gz,
                                                                       (const double*)m->gm2, m->inv, m->cfg.g,
                                                                       grad_manning, grad_bathy, n);
        e = cudaGetLastError();
    } else {
        DevBuf om, oz;
        e = cudaMalloc(&om.p, n * sizeof(double));
        if (e == cudaSuccess) e = cudaMalloc(&oz.p, n * sizeof(double));
        if (e == cudaSuccess) {
            adj_output_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const double*)p_gm, (const double*)p_gz,
                                                                           (const double*)m->gm2, m->inv, m->cfg.g,
                                                                           (double*)om.p, (double*)oz.p, n);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess && grad_manning)
            e = cudaMemcpyAsync(grad_manning, om.p, n * sizeof(double), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess && grad_bathy)
            e = cudaMemcpyAsync(grad_bathy, oz.p, n * sizeof(double), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(loss, p_loss, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return afail(e, "swe_adjoint: output");
    return SWE_OK;
}

}  // namespace

void swe::drop_adjoint_workspace(swe_mesh* m) {
    if (m->adj_arena) cudaFree(m->adj_arena);
    m->adj_arena = nullptr;
    m->device_bytes -= (int64_t)m->adj_bytes;
    adj_kept_all -= m->adj_kept;
    m->adj_bytes = m->adj_kept = 0;
}

extern "C" {

int swe_adjoint(swe_mesh* m, int64_t nsteps, double cfl, const int32_t* gauge_cells, int n_gauges,
                const double* target_h, int checkpoint_every, double* loss, double* grad_manning,
                double* grad_bathy, int where, double* dts_out) {
    NvtxRange nvtx_range("swe_adjoint");
    return adjoint_impl(m, nsteps, cfl, gauge_cells, n_gauges, target_h, nsteps, checkpoint_every, loss,
                        grad_manning, grad_bathy, where, dts_out);
}

int swe_adjoint_series(swe_mesh* m, int64_t nsteps, double cfl, const int32_t* gauge_cells, int n_gauges,
                       const double* targets, int64_t obs_every, int checkpoint_every, double* loss,
                       double* grad_manning, double* grad_bathy, int where, double* dts_out) {
    NvtxRange nvtx_range("swe_adjoint_series");
    return adjoint_impl(m, nsteps, cfl, gauge_cells, n_gauges, targets, obs_every, checkpoint_every, loss,
                        grad_manning, grad_bathy, where, dts_out);
}

int swe_step_dt(swe_mesh* m, int64_t nsteps, const double* dts, double* t_out) {
    NvtxRange nvtx_range("swe_step_dt");
    if (!m || nsteps < 0 || (nsteps > 0 && !dts)) { set_error("swe_step_dt: bad arguments"); return SWE_EINVAL; }
    if (!m->have_state) { set_error("swe_step_dt: no state set"); return SWE_EINVAL; }
    for (int64_t s = 0; s < nsteps; ++s)
        if (!(dts[s] > 0.0) || !std::isfinite(dts[s])) { set_error("swe_step_dt: step sizes must be > 0"); return SWE_EINVAL; }
    AdjDeviceGuard dg(m->cfg.device);
    int rc = flush_mesh_bc(m);
    if (rc) return rc;
    cudaStream_t st = m->stream;
    DevBuf d;
    cudaError_t e = cudaMalloc(&d.p, (nsteps ? nsteps : 1) * sizeof(double));
    if (e == cudaSuccess && nsteps)
        e = cudaMemcpyAsync(d.p, dts, nsteps * sizeof(double), cudaMemcpyHostToDevice, st);
    for (int64_t s = 0; s < nsteps && e == cudaSuccess; ++s) {
        e = launch_step_raw(m, m->state[m->nstep % 2], m->state[(m->nstep + 1) % 2], m->small, m->nstep, 1.0,
                            (const double*)d.p + s, (double*)(m->small + kSlotDtLast), st);
        ++m->nstep;
        m->act_valid = false;   // stepped without the activity bytes
    }
    unsigned long long sm[kSmallWords];
    if (e == cudaSuccess) e = cudaMemcpyAsync(sm, m->small, sizeof sm, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return afail(e, "swe_step_dt");
    if (t_out) std::memcpy(t_out, &sm[kSlotT], sizeof(double));
    if (sm[kSlotStatus] & kStatusBadIndex) {
        set_error("swe_step_dt: an index or boundary group out of range (debug checks)");
        return SWE_EMESH;
    }
    if (sm[kSlotStatus] & kStatusStall) return status_code(sm[kSlotStatus]);
    if (sm[kSlotStatus] & kStatusNonFinite) { set_error("swe_step_dt: non-finite state"); return SWE_ENONFINITE; }
    return SWE_OK;
}

int swe_adjoint_method(swe_mesh* m, int method) {
    if (!m) { set_error("swe_adjoint_method: NULL mesh"); return SWE_EINVAL; }
    if (method != SWE_ADJOINT_TRANSPOSE && method != SWE_ADJOINT_DUAL) {
        set_error("swe_adjoint_method: unknown method");
        return SWE_EINVAL;
    }
    m->adjoint_method = method;
    return SWE_OK;
}

int swe_set_fields(swe_mesh* m, const double* bathy, const double* manning) {
    if (!m) { set_error("swe_set_fields: NULL mesh"); return SWE_EINVAL; }
    const int64_t n = m->hm.n_cells;
    if (manning)
        for (int64_t c = 0; c < n; ++c)
            if (!(manning[c] >= 0.0) || !std::isfinite(manning[c])) {
                set_error("swe_set_fields: negative or non-finite Manning coefficient");
                return SWE_EINVAL;
            }
    if (bathy)
        for (int64_t c = 0; c < n; ++c)
            if (!std::isfinite(bathy[c])) { set_error("swe_set_fields: non-finite bed"); return SWE_EINVAL; }
    AdjDeviceGuard dg(m->cfg.device);
    cudaStream_t st = m->stream;
    cudaError_t e = cudaStreamSynchronize(st);
    for (int64_t c = 0; c < n; ++c) {
        const int64_t o = m->hm.perm[c];
        if (bathy) m->hm.z[c] = bathy[o];
        if (manning) m->hm.m[c] = manning[o];
    }
    const bool f32 = m->cfg.precision == SWE_FP32;
    const unsigned grid = (unsigned)((n + 255) / 256);
    if (e == cudaSuccess && bathy) {
        if (f32) {
            std::vector<float> zt(n);
            for (int64_t c = 0; c < n; ++c) zt[c] = (float)m->hm.z[c];
            e = cudaMemcpy(m->zdev, zt.data(), n * sizeof(float), cudaMemcpyHostToDevice);
            if (e == cudaSuccess) {
                set_z_kernel<float><<<grid, 256, 0, st>>>((V4<float>*)m->state[0], (V4<float>*)m->state[1],
                                                         (const float*)m->zdev, n);
                e = cudaGetLastError();
            }
        } else {
            e = cudaMemcpy(m->zdev, m->hm.z.data(), n * sizeof(double), cudaMemcpyHostToDevice);
            if (e == cudaSuccess) {
                set_z_kernel<double><<<grid, 256, 0, st>>>((V4<double>*)m->state[0], (V4<double>*)m->state[1],
                                                          (const double*)m->zdev, n);
                e = cudaGetLastError();
            }
        }
    }
    if (e == cudaSuccess && manning) {
        if (f32) {
            std::vector<float> g(n);
            for (int64_t c = 0; c < n; ++c) g[c] = (float)(m->cfg.g * m->hm.m[c] * m->hm.m[c]);
            e = cudaMemcpy(m->gm2, g.data(), n * sizeof(float), cudaMemcpyHostToDevice);
            m->topo_dirty = true;  // topo.w carries g m^2 in FP32
        } else {
            std::vector<double> g(n);
            for (int64_t c = 0; c < n; ++c) g[c] = m->cfg.g * m->hm.m[c] * m->hm.m[c];
            e = cudaMemcpy(m->gm2, g.data(), n * sizeof(double), cudaMemcpyHostToDevice);
        }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return afail(e, "swe_set_fields");
    return flush_mesh_bc(m);
}

}  // extern "C"
