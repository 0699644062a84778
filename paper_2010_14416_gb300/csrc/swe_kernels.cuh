// swe_kernels.cuh -- device code of the fused shallow-water step (sm_103a).
//
// One thread owns one cell (in the locality order chosen at mesh build time)
// and gathers its three neighbours, so every cell's sum of edge fluxes is
// formed in a fixed order without atomics.  Each interior edge has a
// canonical orientation: the cell with the lower caller index is the left
// state and its outward normal is the edge normal.  Both cells of an edge
// evaluate the same device function on the same operands (the right cell
// passes them swapped back into canonical order) and apply the result with
// opposite signs, so the two contributions cancel (exactly, as long as the
// compiler emits the same instruction sequence for each unrolled edge slot),
// and the result does not depend on the cell ordering.
//
// Method: Delmas & Soulaimani, Sections 2-3 (Eq 12-37); readings of the
// garbled equations are the same as the oracle's and are listed where used.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "swe_compare.cuh"
#include "swe_f32.cuh"
#include "swe_f64.cuh"

namespace swe {

constexpr int kMaxGroups = 64;
constexpr int kNbrMask = 0x3FFFFFFF;   // neighbour index bits
constexpr int kFlipBit = 0x40000000;   // set when this cell is the right side of the edge
constexpr int kStaticBit = (int)0x80000000;  // in topo.w: the cell has an inflow or fixed-stage edge
constexpr unsigned long long kInfBits = 0x7FF0000000000000ULL;  // +inf as double bits

// status word bits
constexpr unsigned kStatusNonFinite = 1u;
constexpr unsigned kStatusDry = 2u;
constexpr unsigned kStatusStall = 8u;      // a wait of the step loop gave up
constexpr unsigned kStatusBadIndex = 4u;   // debug checks: an index or boundary group out of range

// Debug checks: whether a neighbour code can be used on a mesh of n cells with
// n_groups boundary groups -- an interior code (>= 0) whose cell index is below
// n, or a boundary code (< 0) whose group -1 - code is below n_groups.
__host__ __device__ __forceinline__ bool code_ok(int code, long long n, int n_groups) {
    if (code >= 0) return (long long)(code & 0x3FFFFFFF) < n;
    return -1 - (long long)code < (long long)n_groups;
}

constexpr int kBcWall = 0, kBcInflow = 1, kBcTransmissive = 2, kBcStage = 3;

constexpr int kScanBlock = 256;   // threads of act_scan_kernel, 16 cells each
constexpr int kScanLog = 12;      // a block's span: 2^kScanLog = 16 kScanBlock cells
constexpr int kEnsPad = 256;  // ensemble members are padded to whole multiples of this many cells

template <typename T>
struct alignas(4 * sizeof(T)) V4 {
    T x, y, z, w;
};

// Boundary groups: for group g, kind[g] and value[g] = q (m^2/s, inflow per
// unit length) or eta_s (m, stage).
struct BcTable {
    int kind[kMaxGroups];
    double value[kMaxGroups];
};

template <typename T>
struct StepArgs {
    const V4<T>* __restrict__ s_in;    // (h, hu, hv, z) per cell
    V4<T>* __restrict__ s_out;
    const V4<T>* __restrict__ geoA;    // (L n)_0 x, y, (L n)_1 x, y : outward normals times length (FP64: n alone)
    const V4<T>* __restrict__ geoB;    // (L n)_2 x, y (FP64: n), 1/|Omega|, inscribed radius
    const V4<T>* __restrict__ geoR;    // FP64: the three edges' lengths L (x, y, z)
    const int4* __restrict__ topo;     // neighbour codes of the 3 edges; .w = g m^2 bits (FP32)
    const T* __restrict__ gm2;         // g m^2 per cell (Manning factor of Eq 32), FP64 only
    const double* dt_read;             // min_i R_i/(c_i+|u_i|) of the current state
    unsigned long long* dt_write;      // same quantity for the new state (atomicMin on bits)
    unsigned long long* dt_reset;      // slot cleared to +inf for the step after next
    double* t;                         // simulated time
    unsigned* status;                  // kStatus* bits
    unsigned long long* n_clamped;     // cells clamped from h < 0
    unsigned long long* n_active;      // cells that ran the full flux path (diagnostic)
    long long n;                       // number of cells
    unsigned grid;                     // blocks launched (grid-stride)
    double cfl;
    int hll;                           // 1: HLL flux for all components, 0: HLLC
    const double* dt_fixed;            // if set: the step size to take (frozen time steps)
    double* dt_log;                    // if set: receives the step size taken
    // activity bytes (step_kernel_act only): read, marked for the next step,
    // cleared for the step after next
    const unsigned char* act_in;
    unsigned char* act_next;
    unsigned char* act_clear;
    // one flag per 2^kScanLog cells and buffer: 0 if none of the span's bytes is
    // set; and the spans next to each (itself among them)
    const unsigned char* span_in;
    unsigned char* span_next;
    unsigned char* span_clear;
    const unsigned* span_first;
    const unsigned* span_adj;
    unsigned* act_list;                // cells that run the flux path (act_scan_kernel), in [0, *act_count)
    unsigned* act_count;               // and a count of the blocks that have used it; both 0 between steps
    // edge pass (step_kernel with EDGES): interior edges in canonical orientation,
    // evaluated once per step by edge_flux_kernel before the cell pass
    const int2* ecells;                // (left, right) cell of each interior edge
    const T* eln;                      // [E][2] L n of the edge (FP64: n alone), outward from the left cell
    const T* erl;                      // FP64: the edge's length
    V4<T>* eflux;                      // (F0, F1, F2, bed source factor of the left cell) per edge; FP64: m, xL, yL, xR
    T* esrc;                           // bed source factor of the right cell per edge; FP64: yR
    const int4* eidx;                  // per cell: the interior edge of each local edge (x, y, z)
    long long n_edges;
    T g, h_dry;
    BcTable bc;
    int debug;                         // 1: check indices and groups before use (kStatusBadIndex)
    int n_groups;                      // boundary groups in use
    __device__ __forceinline__ int bc_kind(int grp) const { return bc.kind[grp]; }
    __device__ __forceinline__ double bc_value(int grp) const { return bc.value[grp]; }
    __device__ __forceinline__ long long cell_bound() const { return n; }
};

// Arguments of the batched ensemble step: the members' cells are concatenated,
// each member padded to a whole multiple of kEnsPad cells (padding cells are
// dry and walled in, so they take the quiet path).  A block works on tiles of
// BLOCK cells (BLOCK divides kEnsPad), so every tile belongs to one member.
template <typename T>
struct EnsArgs {
    const V4<T>* __restrict__ s_in;
    V4<T>* __restrict__ s_out;
    const V4<T>* __restrict__ geoA;
    const V4<T>* __restrict__ geoB;
    const V4<T>* __restrict__ geoR;    // FP64: the three edges' lengths
    const int4* __restrict__ topo;     // neighbour codes offset to the concatenated numbering
    const T* __restrict__ gm2;         // FP64 only
    const int* __restrict__ tile_member;               // member of each kEnsPad-cell span
    const long long* __restrict__ member_first_tile;   // first kEnsPad-cell span of each member
    const double* __restrict__ cfl;    // per member
    unsigned long long* small;         // per member: 8 words (dt slots 0..2, t, status, clamps, -, -)
    const int* __restrict__ kind_;     // global boundary groups (0 = wall)
    const double* __restrict__ value_;
    unsigned long long* n_active;      // all members (diagnostic)
    long long n_total;                 // cells of the padded layout (a multiple of kEnsPad)
    // split step: the first pair_spans kEnsPad-cell spans belong to the members
    // the cell-pair kernel updates; the other kernels then update the cells
    // from cell_lo = pair_spans * kEnsPad on (otherwise both are 0)
    long long cell_lo;
    unsigned pair_spans;
    int chunk_log2;                    // tiles per round-robin chunk = 2^chunk_log2
    // dynamic chunks (ensemble_step_kernel_dyn): three rotating counters; the
    // step takes chunks from sched[sched_slot] and zeroes sched[sched_reset]
    unsigned* sched;
    int sched_slot, sched_reset;
    // activity bytes over the concatenated layout (ensemble_step_kernel_act)
    const unsigned char* act_in;
    unsigned char* act_next;
    unsigned char* act_clear;
    // list mode: span flags, the spans beside each span, the list of cells that
    // run the flux path, its count (and one of blocks), each member's step size
    const unsigned char* span_in;
    unsigned char* span_next;
    unsigned char* span_clear;
    const unsigned* span_first;
    const unsigned* span_adj;
    unsigned* act_list;
    unsigned* act_count;
    T* member_dt;
    int n_members;
    // edge pass over the concatenated members (ensemble_step_kernel with EDGES)
    const int2* ecells;
    const T* eln;
    const T* erl;
    V4<T>* eflux;
    T* esrc;
    const int4* eidx;
    long long n_edges;
    int slot_read, slot_write, slot_reset;
    int hll;
    T g, h_dry;
    int debug;                         // 1: check indices and groups before use (kStatusBadIndex)
    int n_groups;                      // global boundary groups in use
    __device__ __forceinline__ int bc_kind(int grp) const { return kind_[grp]; }
    __device__ __forceinline__ double bc_value(int grp) const { return value_[grp]; }
    __device__ __forceinline__ long long cell_bound() const { return n_total; }
};

// ---- precision-specific arithmetic ------------------------------------------------
// The FP32 instantiation is compiled with fast-math: division, reciprocal and
// square root map to the hardware approximations (a few ulp), which the
// 1e-4 FP32 tolerance absorbs.  The double one (IEEE division and square root)
// serves the first CFL step of a state; the FP64 steps have their own
// arithmetic (swe_f64.cuh).
template <typename T> struct Ar;
template <> struct Ar<float> {
    static __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
    static __device__ __forceinline__ float div_(float a, float b) { return __fdividef(a, b); }
    static __device__ __forceinline__ float rcp_(float x) { return __fdividef(1.0f, x); }
};
template <> struct Ar<double> {
    static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
    static __device__ __forceinline__ double div_(double a, double b) { return a / b; }
    static __device__ __forceinline__ double rcp_(double x) { return 1.0 / x; }
};

// h^(-1/3) in double, for the friction factor h^(-7/3) = r^7 and 1/h = r^3
// (Eq 33-35): positive normal h in the FP32 range.
__device__ __forceinline__ double inv_cbrt_newton(double h) { return f64::rcbrt(h); }

// |L n|^2 of an edge, written as one fused multiply-add so that every kernel
// (and both cells of an edge, whose L n differ only in sign) forms the same
// value.
template <typename T>
__device__ __forceinline__ T edge_l2(T lx, T ly) { return fma(lx, lx, ly * ly); }

// ---- Riemann flux in the edge-normal frame (Eq 14, 17-26) -------------------------
// Input U_K = (h_K, h_K un_K, h_K ut_K) given as depth and normal/tangential
// velocity.  Readings: Eq 20 p_K = sqrt(h*(h*+h_K)/2)/h_K; Eq 21-22 use the
// normal velocity jump; the two-rarefaction base is clamped at 0; Eq 24 is
// upwinded (ut_L when S* >= 0); Eq 26 line 2 is the right-dry case; both dry
// gives no flux.
// With hll_only the third component is the HLL flux of U_3 = h ut (Eq 18
// applied to it) instead of the HLLC upwinding of Eq 24.
template <typename T>
__device__ __forceinline__ void riemann_hllc(T hL, T unL, T utL, T hR, T unR, T utR, T g, T h_dry,
                                             T& G1, T& G2, T& G3, T* speeds = nullptr, bool hll_only = false) {
    if constexpr (std::is_same<T, float>::value) {   // FP32: swe_f32.cuh, branch-free and explicitly rounded
        f32::riemann<float>(hL, unL, utL, hR, unR, utR, g, f32::mul(0.5f, g), h_dry, G1, G2, G3, speeds, hll_only);
        return;
    } else if constexpr (std::is_same<T, double>::value) {   // FP64: swe_f64.cuh
        f64::riemann_any(hL, unL, utL, hR, unR, utR, 0.5 * g, h_dry, G1, G2, G3, speeds, hll_only);
        return;
    } else {
    using A = Ar<T>;
    const bool wetL = gt_pos(hL, h_dry), wetR = gt_pos(hR, h_dry);
    if (!wetL && !wetR) {
        G1 = T(0); G2 = T(0); G3 = T(0);
        if (speeds) { speeds[0] = T(0); speeds[1] = T(0); speeds[2] = T(0); }
        return;
    }
    const T aL = A::sqrt_(g * hL), aR = A::sqrt_(g * hR);
    T SL, SR, Ss;
    if (!wetL) {
        SL = unR - T(2) * aR; SR = unR + aR; Ss = SL;
    } else if (!wetR) {
        SL = unL - aL; SR = unL + T(2) * aL; Ss = SR;
    } else {
        const T hsum = hL + hR;
        const T h0 = T(0.5) * hsum - T(0.25) * A::div_((unR - unL) * hsum, aL + aR);  // Eq 21
        T pL = T(1), pR = T(1);                                                     // Eq 20
        // Eq 22's two-rarefaction estimate is at most min(h_L, h_R) where Eq 21
        // chooses it: p_L = p_R = 1 there
        if (!le_pos(h0, min_nonneg(hL, hR))) {                                       // Eq 23
            const T r2h0 = A::rcp_(T(2) * h0);
            const T gL = A::sqrt_(g * (h0 + hL) * r2h0 * A::rcp_(hL));
            const T gR = A::sqrt_(g * (h0 + hR) * r2h0 * A::rcp_(hR));
            const T hs = A::div_(hL * gL + hR * gR + unL - unR, gL + gR);
            if (gt_pos(hs, hL)) pL = A::div_(A::sqrt_(T(0.5) * hs * (hs + hL)), hL);
            if (gt_pos(hs, hR)) pR = A::div_(A::sqrt_(T(0.5) * hs * (hs + hR)), hR);
        }
        SL = unL - aL * pL;                                                          // Eq 19
        SR = unR + aR * pR;
        const T mL = hL * (unL - SL), mR = hR * (unR - SR);
        Ss = A::div_(SL * mR - SR * mL, mR - mL);                                    // Eq 25
    }
    const T qL = hL * unL, qR = hR * unR;
    const T PL = qL * unL + T(0.5) * g * hL * hL;
    const T PR = qR * unR + T(0.5) * g * hR * hR;
    if (ge_zero(SL)) {                                                               // Eq 17
        G1 = qL; G2 = PL;
        if (hll_only) G3 = qL * utL;
    } else if (le_zero(SR)) {
        G1 = qR; G2 = PR;
        if (hll_only) G3 = qR * utR;
    } else {                                                                         // Eq 18
        const T r = A::rcp_(SR - SL);
        const T ss = SR * SL;
        G1 = (SR * qL - SL * qR + ss * (hR - hL)) * r;
        G2 = (SR * PL - SL * PR + ss * (qR - qL)) * r;
        if (hll_only) G3 = (SR * (qL * utL) - SL * (qR * utR) + ss * (hR * utR - hL * utL)) * r;
    }
    if (!hll_only) G3 = G1 * (ge_zero(Ss) ? utL : utR);                              // Eq 24
    if (speeds) { speeds[0] = SL; speeds[1] = SR; speeds[2] = Ss; }
    }
}

// Threads of a step kernel's block.  FP64 blocks may be launched with fewer than
// BLOCK (step_threads); asking for it costs an FP32 step 1 % (1M-cell canal
// 17.27 us, 17.08 with the constant).
template <typename T, int BLOCK>
__device__ __forceinline__ int block_threads() {
    return sizeof(T) == 8 ? (int)blockDim.x : BLOCK;
}

template <typename T>
__device__ __forceinline__ T inf_of();
template <>
__device__ __forceinline__ float inf_of<float>() { return __int_as_float(0x7F800000); }
template <>
__device__ __forceinline__ double inf_of<double>() { return __longlong_as_double((long long)kInfBits); }

// ---- the step size, formed once per warp ------------------------------------------
// dt = cfl * (min of the previous state) in double, and its rounding to the
// state precision, made by lane 0 and broadcast (all 32 lanes must call):
// FP32 kernels then run no FP64 instruction per thread for it.  dt is
// non-negative or +inf, so "has a step" is an integer compare of its bits.
template <typename T>
struct WarpDt {
    double d;
    T t;
    bool have;
};
template <typename T>
__device__ __forceinline__ WarpDt<T> warp_step_dt(double cfl, const double* dt_read, const double* dt_fixed) {
    double v = 0.0;
    T vt = T(0);
    if ((threadIdx.x & 31) == 0) {
        v = dt_fixed ? *dt_fixed : cfl * (*dt_read);
        vt = T(v);
    }
    WarpDt<T> r;
    r.d = __shfl_sync(0xffffffffu, v, 0);
    r.t = __shfl_sync(0xffffffffu, vt, 0);
    r.have = (unsigned long long)__double_as_longlong(r.d) < kInfBits;
    return r;
}

// ---- block min of a non-negative candidate, published with one atomicMin ----------
// The minimum is taken in the candidate's own precision and widened to double
// once (exact and monotone, so the result equals a double minimum): an FP32
// kernel keeps its reduction off the FP64 pipe.  Non-negative doubles order
// like their bit patterns, so the 64-bit atomicMin is exact.  Optionally also
// sums a per-thread counter into *count_dst (one atomicAdd per block).
template <int BLOCK, typename T>
__device__ __forceinline__ void block_min_publish(T cand, unsigned long long* dst, unsigned cnt = 0u,
                                                  unsigned long long* count_dst = nullptr) {
    __shared__ T warp_min[BLOCK / 32];
    __shared__ unsigned warp_cnt[BLOCK / 32];
    for (int o = 16; o > 0; o >>= 1) cand = min_nonneg(cand, __shfl_xor_sync(0xffffffffu, cand, o));
    if (count_dst) cnt = __reduce_add_sync(0xffffffffu, cnt);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { warp_min[wid] = cand; warp_cnt[wid] = cnt; }
    __syncthreads();
    if (wid == 0) {
        const int warps = block_threads<T, BLOCK>() / 32;
        T v = lane < warps ? warp_min[lane] : inf_of<T>();
        unsigned c = lane < warps ? warp_cnt[lane] : 0u;
        for (int o = 16; o > 0; o >>= 1) v = min_nonneg(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (count_dst) c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0 && v < inf_of<T>())
            atomicMin(dst, (unsigned long long)__double_as_longlong((double)v));
        if (lane == 0 && count_dst && c) atomicAdd(count_dst, (unsigned long long)c);
    }
}

// ---- Manning factor g m^2: packed in topo.w (FP32) or its own array (FP64) --------
// (the sign bit of topo.w is the static-activity flag; g m^2 >= 0 leaves it free)
template <typename Args>
__device__ __forceinline__ float load_gm2(const Args&, long long, const int4& tp, float) {
    return __int_as_float(tp.w & 0x7FFFFFFF);
}
template <typename Args>
__device__ __forceinline__ double load_gm2(const Args& a, long long i, const int4&, double) {
    return a.gm2[i];
}

// ---- asynchronous global -> shared copies (cp.async, 16 B, L2 only) ------------------
// Each thread stages its own future cells' records; it alone reads them back,
// so the per-thread wait_group is the only synchronisation needed.
template <int BYTES>
__device__ __forceinline__ void cp_async_record(void* smem_dst, const void* gmem_src) {
    static_assert(BYTES % 16 == 0, "records are whole 16-byte chunks");
    const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
#pragma unroll
    for (int b = 0; b < BYTES; b += 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + b),
                     "l"((const char*)gmem_src + b)
                     : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(PENDING) : "memory");
}

// ---- a cell update's view of the mesh: states in, state out, geometry ----------------
template <typename Args>
__device__ __forceinline__ auto load_state(const Args& a, long long i) {
    return a.s_in[i];
}
template <typename Args, typename V>
__device__ __forceinline__ void store_state(const Args& a, long long i, const V& v) {
    a.s_out[i] = v;
}
template <typename Args, typename V>
__device__ __forceinline__ void load_geometry(const Args& a, long long i, V& gA, V& gB) {
    gA = a.geoA[i];
    gB = a.geoB[i];
}

// ---- pieces of one cell update, shared by the step kernels and the adjoint ----------
// Templated on the scalar so the discrete adjoint can run them on forward-mode
// dual numbers: it then differentiates exactly the arithmetic, and takes
// exactly the branches, of the forward step.

template <typename T>
__device__ __forceinline__ void cell_velocity(T h, T hu, T hv, T h_dry, T& u, T& v) {
    if constexpr (std::is_same<T, double>::value) {
        f64::velocity(h, hu, hv, h_dry, u, v);
    } else {
        u = T(0);
        v = T(0);
        if (gt_pos(h, h_dry)) { const T r = Ar<T>::rcp_(h); u = hu * r; v = hv * r; }
    }
}

// Flux leaving cell i through an interior edge (per unit length, x-y frame)
// and the edge's bed source factor (g/2)(h**_i^2 - h_i^2) (Eq 30 with 1/2).
// (n1, n2) is cell i's outward unit normal; flip says cell i is the right
// state of the edge's canonical orientation.
template <typename T>
__device__ __forceinline__ void edge_interior(T hi, T ui, T vi, T zi, T hk, T huk, T hvk, T zk, T n1, T n2,
                                              bool flip, T g, T h_dry, T& F0, T& F1, T& F2, T& src,
                                              bool hll_only = false, T* src_k = nullptr) {
    if constexpr (std::is_same<T, float>::value) {   // FP32: swe_f32.cuh
        f32::edge_interior<float>(hi, ui, vi, zi, hk, huk, hvk, zk, n1, n2, flip, g, f32::mul(0.5f, g), h_dry, F0, F1,
                                  F2, src, hll_only, src_k);
        return;
    }
    static_assert(!std::is_same<T, double>::value, "FP64 edges: f64::edge");
    T uk, vk;
    cell_velocity<T>(hk, huk, hvk, h_dry, uk, vk);
    // hydrostatic reconstruction (Eq 28): z* = max(z_i, z_k)
    const T zs = max_finite(zi, zk);
    const T hsi = max_zero(hi + zi - zs);
    const T hsk = max_zero(hk + zk - zs);
    // canonical orientation: left = lower caller index
    const T hL = flip ? hsk : hsi, hR = flip ? hsi : hsk;
    const T uL = flip ? uk : ui, vL = flip ? vk : vi;
    const T uR = flip ? ui : uk, vR = flip ? vi : vk;
    const T c1 = flip ? -n1 : n1, c2 = flip ? -n2 : n2;
    // rotate into the edge frame (Eq 12)
    const T unL = uL * c1 + vL * c2, utL = vL * c1 - uL * c2;
    const T unR = uR * c1 + vR * c2, utR = vR * c1 - uR * c2;
    T G1, G2, G3;
    riemann_hllc<T>(hL, unL, utL, hR, unR, utR, g, h_dry, G1, G2, G3, nullptr, hll_only);
    // back to (x, y) (Eq 12 inverse), as the flux leaving this cell
    const T s = flip ? T(-1) : T(1);
    F0 = s * G1;
    F1 = s * (G2 * c1 - G3 * c2);
    F2 = s * (G2 * c2 + G3 * c1);
    src = T(0.5) * g * (hsi * hsi - hi * hi);
    if (src_k) *src_k = T(0.5) * g * (hsk * hsk - hk * hk);   // the other cell's bed source factor
}

// Flux leaving cell i through a boundary edge of the given kind (Section 3.1).
template <typename T>
__device__ __forceinline__ void edge_boundary(int kind, double value, T hi, T ui, T vi, T zi, T n1, T n2, T g,
                                              T h_dry, T& F0, T& F1, T& F2, bool hll_only = false) {
    if constexpr (std::is_same<T, float>::value) {   // FP32: swe_f32.cuh
        f32::edge_boundary(kind, value, hi, ui, vi, zi, n1, n2, g, f32::mul(0.5f, g), h_dry, F0, F1, F2, hll_only);
        return;
    } else if constexpr (std::is_same<T, double>::value) {   // FP64: swe_f64.cuh
        const f64::Side c{hi, ui, vi, zi};
        const double un = f64::fma(ui, n1, f64::mul(vi, n2)), ut = f64::fma(vi, n1, -f64::mul(ui, n2));
        double G1, G2, G3;
        f64::boundary_flux(kind, value, c, un, ut, 0.5 * g, h_dry, hll_only, G1, G2, G3);
        F0 = G1;
        F1 = f64::fma(G2, n1, -f64::mul(G3, n2));
        F2 = f64::fma(G2, n2, f64::mul(G3, n1));
        return;
    } else {
    const T un = ui * n1 + vi * n2, ut = vi * n1 - ui * n2;
    T G1, G2, G3;
    if (kind == kBcWall) {
        G1 = T(0); G2 = T(0.5) * g * hi * hi; G3 = T(0);
    } else if (kind == kBcInflow) {
        const T q = T(value);
        G1 = -q;
        G2 = T(0.5) * g * hi * hi + (gt_pos(hi, h_dry) ? Ar<T>::div_(q * q, hi) : T(0));
        G3 = T(0);
    } else {
        T hg = hi;
        if (kind == kBcStage) hg = max_zero(T(value) - zi);
        riemann_hllc<T>(hi, un, ut, hg, un, ut, g, h_dry, G1, G2, G3, nullptr, hll_only);
    }
    F0 = G1;
    F1 = G2 * n1 - G3 * n2;
    F2 = G2 * n2 + G3 * n1;
    }
}

// Semi-implicit friction (Eq 33-37), for the adjoint's duals: dU solving [I - dt/2 J_f] dU = dt (R + S_f)
// with R = (Rh, Rx, Ry) the explicit right-hand side per unit area.
template <typename T>
__device__ __forceinline__ void friction_update(T hi, T qx, T qy, T gm2, T Rh, T Rx, T Ry, T dt, T h_dry, T& dh,
                                                T& dqx, T& dqy) {
    using A = Ar<T>;
    dh = dt * Rh;
    dqx = dt * Rx;
    dqy = dt * Ry;
    if (gt_pos(hi, h_dry) && gt_zero(gm2)) {
        const T qq = qx * qx + qy * qy;
        if (gt_zero(qq)) {
            const T qn = A::sqrt_(qq);
            const T cf = gm2 * A::pow_m73(hi), rh = A::rcp_(hi);   // c = g m^2 h^(-7/3), 1/h
            const T al = T(0.5) * dt * cf;                  // alpha = dt c / 2
            // rhs: dt (R_q + S_f) + dt/2 J_qh dh, with S_f = -c|q|q and
            // J_qh = (7/3) c |q| q / h
            const T k = dt * cf * qn * (T(7.0 / 6.0) * dh * rh - T(1));
            const T bx = dqx + k * qx, by = dqy + k * qy;
            // (1 + a|q|) I + a q q^T/|q| has eigenvalue 1 + 2a|q| along q
            // and 1 + a|q| across it
            const T d1 = T(1) + al * qn, d2 = d1 + al * qn;
            const T rqd2 = A::rcp_(qn * d2), rd1 = A::rcp_(d1);
            const T proj = (bx * qx + by * qy) * al * rqd2;
            dqx = (bx - proj * qx) * rd1;
            dqy = (by - proj * qy) * rd1;
        }
    }
}

// ---- the end of one FP64 cell update --------------------------------------------------
// From the sums of the edges' terms (f64::EdgeTerms) to the new state, its
// checks, and the cell's next CFL candidate R_i/(sqrt(g h)+|u|) (Eq 15; +inf
// when the new state is dry).  Every FP64 cell kernel ends here.
template <class S = f64::Soft, typename Args>
__device__ __forceinline__ double finish_cell(const Args& a, long long i, const V4<double>& own, double m, double x,
                                              double y, double ia, double rin, double gm2, double dt,
                                              unsigned long long* n_clamped, unsigned* status) {
    const double g = a.g, h_dry = a.h_dry;
    V4<double> out;
    out.w = own.w;
    f64::update<S>(own.x, own.y, own.z, m, x, y, ia, gm2, dt, h_dry, out.x, out.y, out.z);
    if (lt_zero(out.x)) {
        out.x = 0.0; out.y = 0.0; out.z = 0.0;
        atomicAdd(n_clamped, 1ULL);
    } else if (le_pos(out.x, h_dry)) {
        out.y = 0.0; out.z = 0.0;
    }
    const double big = 3.0e38;
    if (!lt_pos(out.x, big) || !abs_lt_pos(out.y, big) || !abs_lt_pos(out.z, big))
        atomicOr(status, kStatusNonFinite);
    store_state(a, i, out);
    return gt_pos(out.x, h_dry) ? f64::cfl_candidate<S>(out.x, out.y, out.z, rin, g) : inf_of<double>();
}

// ---- one FP32 cell of the fused step -------------------------------------------------
// update_cell for FP32: the same loads, quiet test and edge loop, with the
// arithmetic of swe_f32.cuh, every operation explicitly rounded, so that every
// FP32 kernel and launch shape gives the same bits.
// Pairs of cells sharing their local edge 0 (step_kernel_pair): with PAIR 1
// the first cell hands the flux of that edge to the second (pmode kPairGive ->
// kPairGiven, pe = the flux leaving the first cell); with PAIR 2 the second
// takes its negative (pmode kPairTake) instead of evaluating the edge.
struct PairEdge { float F0, F1, F2; };
constexpr int kPairNone = 0, kPairGive = 1, kPairGiven = 2, kPairTake = 3;

template <bool GEO_EARLY, bool EDGES, int PAIR = 0, typename Args>
__device__ __forceinline__ float update_cell_f32(const Args& a, long long i, const V4<float>& own, const int4& tp,
                                                 float dt, unsigned& active, unsigned long long* n_clamped,
                                                 unsigned* status, int* pmode = nullptr,
                                                 volatile PairEdge* pe = nullptr) {
    const float g = a.g, h_dry = a.h_dry, g2 = f32::mul(0.5f, g);
    const float hi = own.x, zi = own.w;
    int code[3] = {tp.x, tp.y, tp.z};
    if (a.debug) {   // an unusable code is flagged and taken as a wall (group 0)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (!code_ok(code[j], a.cell_bound(), a.n_groups)) {
                atomicOr(status, kStatusBadIndex);
                code[j] = -1;
            }
    }
    V4<float> nb[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) nb[j] = code[j] >= 0 ? load_state(a, code[j] & kNbrMask) : own;
    V4<float> gA, gB;
    float gm2;
    if constexpr (GEO_EARLY) {
        load_geometry(a, i, gA, gB);
        gm2 = load_gm2(a, i, tp, 0.0f);
    }
    bool quiet = !(hi > h_dry);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        if (code[j] >= 0) {
            quiet = quiet && !(nb[j].x > h_dry);
        } else {
            const int kind = a.bc_kind(-1 - code[j]);
            quiet = quiet && (kind == kBcWall || kind == kBcTransmissive);
        }
    }
    V4<float> out;
    out.w = zi;
    if (quiet) {
        out.x = hi; out.y = 0.0f; out.z = 0.0f;
        store_state(a, i, out);
        return inf_of<float>();
    }
    active += 1u;
    if constexpr (!GEO_EARLY) {
        load_geometry(a, i, gA, gB);
        gm2 = load_gm2(a, i, tp, 0.0f);
    }
    float ui, vi;
    f32::velocity(hi, own.y, own.z, h_dry, ui, vi);
    float f0 = 0.0f, f1 = 0.0f, f2 = 0.0f, sx = 0.0f, sy = 0.0f;
    int4 ei = make_int4(-1, -1, -1, 0);
    if constexpr (EDGES) ei = a.eidx[i];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int c = j == 0 ? code[0] : (j == 1 ? code[1] : code[2]);
        const V4<float> o = j == 0 ? nb[0] : (j == 1 ? nb[1] : nb[2]);
        const float lx = j == 0 ? gA.x : (j == 1 ? gA.z : gB.x);
        const float ly = j == 0 ? gA.y : (j == 1 ? gA.w : gB.y);
        const float l2 = edge_l2(lx, ly);
        const float rl = rsqrtf(l2);
        const float len = f32::mul(l2, rl);
        const float n1 = f32::mul(lx, rl), n2 = f32::mul(ly, rl);   // this cell's outward unit normal
        float F0, F1, F2;
        if (c >= 0) {
            float src;
            if constexpr (EDGES) {
                if (!(hi > h_dry) && !(o.x > h_dry)) {
                    const float zs = f32::vmax(zi, o.w);
                    const float hsi = f32::max0(f32::sub(f32::add(hi, zi), zs));
                    F0 = 0.0f; F1 = 0.0f; F2 = 0.0f;
                    f32::bed_src(hsi, hi, g2, src);
                } else {
                    int e = j == 0 ? ei.x : (j == 1 ? ei.y : ei.z);
                    if (a.debug && !(e >= 0 && e < a.n_edges)) {
                        atomicOr(status, kStatusBadIndex);
                        e = 0;
                    }
                    const V4<float> fl = a.eflux[e];
                    if (c & kFlipBit) {
                        F0 = -fl.x; F1 = -fl.y; F2 = -fl.z;
                        src = a.esrc[e];
                    } else {
                        F0 = fl.x; F1 = fl.y; F2 = fl.z;
                        src = fl.w;
                    }
                }
            } else if (PAIR == 2 && j == 0 && *pmode == kPairTake) {
                // the first cell's evaluation of this edge, seen from this side;
                // the bed source factor is this cell's own (Eq 30)
                const float zs = f32::vmax(zi, o.w);
                const float hsi = f32::max0(f32::sub(f32::add(hi, zi), zs));
                f32::bed_src(hsi, hi, g2, src);
                F0 = -pe->F0; F1 = -pe->F1; F2 = -pe->F2;
            } else {
                f32::edge_interior<float>(hi, ui, vi, zi, o.x, o.y, o.z, o.w, n1, n2, (c & kFlipBit) != 0, g, g2,
                                          h_dry, F0, F1, F2, src, a.hll != 0);
                if (PAIR == 1 && j == 0 && *pmode == kPairGive) {
                    pe->F0 = F0; pe->F1 = F1; pe->F2 = F2;
                    *pmode = kPairGiven;
                }
            }
            sx = f32::fma(src, lx, sx);
            sy = f32::fma(src, ly, sy);
        } else {
            const int grp = -1 - c;
            f32::edge_boundary(a.bc_kind(grp), a.bc_value(grp), hi, ui, vi, zi, n1, n2, g, g2, h_dry, F0, F1, F2,
                               a.hll != 0);
        }
        f0 = f32::fma(len, F0, f0);
        f1 = f32::fma(len, F1, f1);
        f2 = f32::fma(len, F2, f2);
    }
    bool clamped, nonfinite;
    const float cand = f32::finish<float>(hi, f32::rcp_(hi), own.y, own.z, f0, f1, f2, sx, sy, gB.z, gB.w, gm2, dt, g,
                                          h_dry, out.x, out.y, out.z, clamped, nonfinite);
    if (clamped) atomicAdd(n_clamped, 1ULL);
    if (nonfinite) atomicOr(status, kStatusNonFinite);
    store_state(a, i, out);
    return cand;
}

// ---- one cell of the fused step -----------------------------------------------------
// Returns the cell's CFL candidate R_i/(sqrt(g h)+|u|) of the new state (+inf
// when the new state is dry); sets `active` when the full flux path ran.
//
// A dry cell whose neighbours are all dry and whose boundary edges are walls
// or transmissive is "quiet": every mass flux it sees is exactly +-0 (both
// sides dry give G = 0; walls carry no mass), so its depth is unchanged, and
// its momentum is set to zero by the dry-cell rule after the update.  Its new
// state is therefore (h, 0, 0) bit for bit whatever the momentum terms were,
// and the edge loop, geometry and friction are skipped.
//
// GEO_EARLY issues the cell's geometry loads together with the neighbour
// gathers (one memory round trip fewer for a cell that runs the flux path,
// at the price of geometry traffic for quiet cells too); otherwise they are
// issued after the quiet test.  Both give the same results.
//
// EDGES takes the interior edges' terms from the edge pass (edge_flux_kernel,
// the same arithmetic evaluated once per edge) instead of evaluating them
// here; an edge with both cells dry has no flux and its bed source term is
// formed inline, with the same bits.

// The FP64 cell of the edge-pass step.  It reads its neighbours' depths only,
// and normals only for boundary edges and edges with both cells dry: with whole neighbour and geometry records the kernel held 138 registers
// (12 warps an SM) and waited on its chain of operations (48 us for 250k wet
// cells; a step of the 1M-cell canal 182 us then, 163 now).
template <typename Args>
__device__ __forceinline__ double update_cell_edges(const Args& a, long long i, const V4<double>& own, const int4& tp,
                                                    double dt, unsigned& active, unsigned long long* n_clamped,
                                                    unsigned* status) {
    const double h_dry = a.h_dry;
    const double hi = own.x, zi = own.w;
    int code[3] = {tp.x, tp.y, tp.z};
    if (a.debug) {   // an unusable code is flagged and taken as a wall (group 0)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (!code_ok(code[j], a.cell_bound(), a.n_groups)) {
                atomicOr(status, kStatusBadIndex);
                code[j] = -1;
            }
    }
    const int4 ei = a.eidx[i];
    const bool wet = gt_pos(hi, h_dry);
    bool flux[3];   // the edge pass evaluated the edge
    bool quiet = !wet;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        flux[j] = false;
        if (code[j] >= 0) {
            flux[j] = wet || gt_pos(a.s_in[code[j] & kNbrMask].x, h_dry);
            quiet = quiet && !flux[j];
        } else {
            const int kind = a.bc_kind(-1 - code[j]);
            quiet = quiet && (kind == kBcWall || kind == kBcTransmissive);
        }
    }
    if (quiet) {
        V4<double> out;
        out.x = hi; out.y = 0.0; out.z = 0.0; out.w = zi;
        a.s_out[i] = out;
        return inf_of<double>();
    }
    active += 1u;
    const double2 tail = ((const double2*)&a.geoB[i])[1];   // 1/|Omega|, R
    const double gm2 = a.gm2[i];
    const V4<double> gR = a.geoR[i];                        // the edges' lengths
    double m = 0.0, x = 0.0, y = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int c = code[j];
        double tm = 0.0, tx, ty;
        if (flux[j]) {
            int e = j == 0 ? ei.x : (j == 1 ? ei.y : ei.z);
            if (a.debug && !(e >= 0 && e < a.n_edges)) {
                atomicOr(status, kStatusBadIndex);
                e = 0;
            }
            const V4<double> fl = a.eflux[e];
            const bool flip = (c & kFlipBit) != 0;
            tm = flip ? -fl.x : fl.x;
            tx = flip ? -fl.w : fl.y;
            ty = flip ? -a.esrc[e] : fl.z;
        } else {
            const double2 n = j == 2 ? *(const double2*)&a.geoB[i] : ((const double2*)&a.geoA[i])[j];
            const double g2 = f64::mul(0.5, a.g);
            if (c >= 0) {
                f64::dry_edge(hi, zi, a.s_in[c & kNbrMask].w, n.x, n.y, g2, tx, ty);
            } else {
                const int grp = -1 - c;
                f64::Side side{hi, 0.0, 0.0, zi};
                f64::velocity(hi, own.y, own.z, h_dry, side.u, side.v);
                f64::boundary(a.bc_kind(grp), a.bc_value(grp), side, n.x, n.y, g2, h_dry, a.hll != 0, tm, tx, ty);
            }
        }
        const double len = j == 0 ? gR.x : (j == 1 ? gR.y : gR.z);
        m = f64::fma(len, tm, m);
        x = f64::fma(len, tx, x);
        y = f64::fma(len, ty, y);
    }
    return finish_cell(a, i, own, m, x, y, tail.x, tail.y, gm2, dt, n_clamped, status);
}

template <typename T, bool GEO_EARLY, bool EDGES = false, typename Args>
__device__ __forceinline__ T update_cell(const Args& a, long long i, const V4<T>& own, const int4& tp, T dt,
                                         unsigned& active, unsigned long long* n_clamped, unsigned* status) {
    if constexpr (std::is_same<T, float>::value) {
        return update_cell_f32<GEO_EARLY, EDGES>(a, i, own, tp, dt, active, n_clamped, status);
    } else if constexpr (EDGES) {
        return update_cell_edges(a, i, own, tp, dt, active, n_clamped, status);
    } else {
    const double h_dry = a.h_dry, g2 = f64::mul(0.5, a.g);
    const double hi = own.x, zi = own.w;
    int code[3] = {tp.x, tp.y, tp.z};
    if (a.debug) {   // an unusable code is flagged and taken as a wall (group 0)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (!code_ok(code[j], a.cell_bound(), a.n_groups)) {
                atomicOr(status, kStatusBadIndex);
                code[j] = -1;
            }
    }
    // issue the three neighbour gathers before any arithmetic
    V4<double> nb[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) nb[j] = code[j] >= 0 ? a.s_in[code[j] & kNbrMask] : own;
    V4<double> gA, gB, gR;   // unit normals, 1/|Omega| and R, lengths
    double gm2;
    if constexpr (GEO_EARLY) {
        gA = a.geoA[i];
        gB = a.geoB[i];
        gR = a.geoR[i];
        gm2 = a.gm2[i];
    }
    bool quiet = !gt_pos(hi, h_dry);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        if (code[j] >= 0) {
            quiet = quiet && !gt_pos(nb[j].x, h_dry);
        } else {
            const int kind = a.bc_kind(-1 - code[j]);
            quiet = quiet && (kind == kBcWall || kind == kBcTransmissive);
        }
    }
    if (quiet) {
        V4<double> out;
        out.x = hi; out.y = 0.0; out.z = 0.0; out.w = zi;
        a.s_out[i] = out;
        return inf_of<double>();
    }
    active += 1u;
    if constexpr (!GEO_EARLY) {
        gA = a.geoA[i];
        gB = a.geoB[i];
        gR = a.geoR[i];
        gm2 = a.gm2[i];
    }
    f64::Side own_side{hi, 0.0, 0.0, zi};
    f64::velocity(hi, own.y, own.z, h_dry, own_side.u, own_side.v);
    double m = 0.0, x = 0.0, y = 0.0;
#pragma unroll 1   // an edge's evaluation is some 2,500 instructions
    for (int j = 0; j < 3; ++j) {
        const int c = j == 0 ? code[0] : (j == 1 ? code[1] : code[2]);
        const V4<double> o = j == 0 ? nb[0] : (j == 1 ? nb[1] : nb[2]);
        const double n1 = j == 0 ? gA.x : (j == 1 ? gA.z : gB.x);   // this cell's outward unit normal
        const double n2 = j == 0 ? gA.y : (j == 1 ? gA.w : gB.y);
        const double len = j == 0 ? gR.x : (j == 1 ? gR.y : gR.z);
        double tm = 0.0, tx, ty;
        if (c >= 0) {
            const bool flip = (c & kFlipBit) != 0;
            f64::Side nb_side{o.x, 0.0, 0.0, o.w};
            f64::velocity(o.x, o.y, o.z, h_dry, nb_side.u, nb_side.v);
            f64::Side L, R;   // the canonical orientation: left = lower caller index
            L.h = flip ? nb_side.h : own_side.h; R.h = flip ? own_side.h : nb_side.h;
            L.u = flip ? nb_side.u : own_side.u; R.u = flip ? own_side.u : nb_side.u;
            L.v = flip ? nb_side.v : own_side.v; R.v = flip ? own_side.v : nb_side.v;
            L.z = flip ? nb_side.z : own_side.z; R.z = flip ? own_side.z : nb_side.z;
            f64::EdgeTerms t;
            f64::edge(L, R, flip ? -n1 : n1, flip ? -n2 : n2, g2, h_dry, a.hll != 0, t);
            tm = flip ? -t.m : t.m;
            tx = flip ? -t.xR : t.xL;
            ty = flip ? -t.yR : t.yL;
        } else {
            const int grp = -1 - c;
            f64::boundary(a.bc_kind(grp), a.bc_value(grp), own_side, n1, n2, g2, h_dry, a.hll != 0, tm, tx, ty);
        }
        m = f64::fma(len, tm, m);
        x = f64::fma(len, tx, x);
        y = f64::fma(len, ty, y);
    }
    return finish_cell(a, i, own, m, x, y, gB.z, gB.w, gm2, dt, n_clamped, status);
    }
}

// Blocks per SM that a step kernel's registers are held to.  The FP64 cell
// pass after the edge pass is a chain of integer and FP64 operations: the more
// warps the better until it spills (20 an SM, 96 registers; 16 for the
// ensemble's).
template <typename T, bool EDGES, bool ENSEMBLE>
__host__ __device__ constexpr int min_blocks_of(int block, int min_blocks) {
    return sizeof(T) == 8 && EDGES ? (ENSEMBLE ? 16 : 20) * 32 / block : min_blocks;
}

// ---- the fused step: fluxes + bed source + BCs + friction + update + next dt ------
// Grid-stride over cells with about one resident wave of blocks, so the block
// reduction (and its barrier) runs once per block.  With STAGES > 1 each
// thread keeps its next STAGES-1 cells' state and topology records in flight
// through cp.async into its own shared-memory slots.
template <typename T, int BLOCK, int MINB, int STAGES, bool GEO_EARLY, bool EDGES = false>
__global__ void __launch_bounds__(BLOCK, (min_blocks_of<T, EDGES, false>(BLOCK, MINB))) step_kernel(const StepArgs<T> a) {
    const WarpDt<T> wdt = warp_step_dt<T>(a.cfl, a.dt_read, a.dt_fixed);
    const double dt_d = wdt.d;
    const bool have_dt = wdt.have;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.dt_reset = kInfBits;
        if (have_dt) *a.t += dt_d;
        else atomicOr(a.status, kStatusDry);
        if (a.dt_log) *a.dt_log = dt_d;
    }
    T cand = inf_of<T>();
    unsigned active = 0u;
    const int threads = block_threads<T, BLOCK>();
    const long long stride = (long long)gridDim.x * threads;
    long long i = (long long)blockIdx.x * threads + threadIdx.x;
    if (!have_dt) {
        for (; i < a.n; i += stride) a.s_out[i] = a.s_in[i];
    } else if constexpr (STAGES <= 1) {
        const T dt = wdt.t;
        for (; i < a.n; i += stride) {
            const V4<T> own = a.s_in[i];
            const int4 tp = a.topo[i];
            cand = min_nonneg(cand, update_cell<T, GEO_EARLY, EDGES>(a, i, own, tp, dt, active, a.n_clamped, a.status));
        }
    } else {
        __shared__ V4<T> st_own[STAGES][BLOCK];
        __shared__ int4 st_topo[STAGES][BLOCK];
        const T dt = wdt.t;
        const int tid = threadIdx.x;
#pragma unroll
        for (int s = 0; s < STAGES - 1; ++s) {
            const long long c = i + (long long)s * stride;
            if (c < a.n) {
                cp_async_record<sizeof(V4<T>)>(&st_own[s][tid], &a.s_in[c]);
                cp_async_record<16>(&st_topo[s][tid], &a.topo[c]);
            }
            cp_async_commit();
        }
        int slot = 0;
        for (; i < a.n; i += stride) {
            const long long c = i + (long long)(STAGES - 1) * stride;
            const int fill = slot == 0 ? STAGES - 1 : slot - 1;
            if (c < a.n) {
                cp_async_record<sizeof(V4<T>)>(&st_own[fill][tid], &a.s_in[c]);
                cp_async_record<16>(&st_topo[fill][tid], &a.topo[c]);
            }
            cp_async_commit();
            cp_async_wait<STAGES - 1>();
            const V4<T> own = st_own[slot][tid];
            const int4 tp = st_topo[slot][tid];
            cand = min_nonneg(cand, update_cell<T, GEO_EARLY, EDGES>(a, i, own, tp, dt, active, a.n_clamped, a.status));
            slot = slot == STAGES - 1 ? 0 : slot + 1;
        }
        cp_async_wait<0>();
    }
    block_min_publish<BLOCK>(cand, a.dt_write, active, a.n_active);
}

// ---- the fused step over pairs of adjacent cells (FP32) -----------------------------
// Thread work item p is the cell pair (2p, 2p+1).  The mesh's pairing order
// puts two cells that share an edge at such positions, with that edge as
// local edge 0 of both, for most cells.  The edge's flux is then evaluated
// once, by the first cell, and the second takes its negative: bit for bit
// what it would evaluate itself (the edge's canonical evaluation, rotated with
// the exactly opposite normal), while each cell still sums its edges in local
// order, so the results equal the one-cell kernels'.  Five Riemann problems
// per pair instead of six.  Unmatched cells come in whole warps of their own.
template <int BLOCK, int MINB, bool GEO_EARLY>
__global__ void __launch_bounds__(BLOCK, MINB) step_kernel_pair(const StepArgs<float> a) {
    const WarpDt<float> wdt = warp_step_dt<float>(a.cfl, a.dt_read, a.dt_fixed);
    const bool have_dt = wdt.have;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.dt_reset = kInfBits;
        if (have_dt) *a.t += wdt.d;
        else atomicOr(a.status, kStatusDry);
        if (a.dt_log) *a.dt_log = wdt.d;
    }
    float cand = inf_of<float>();
    unsigned active = 0u;
    // 32-bit pair indices (a mesh has fewer than 2^30 cells): fewer live registers
    const unsigned stride = gridDim.x * BLOCK;
    const unsigned np = (unsigned)((a.n + 1) >> 1);
    unsigned p = blockIdx.x * BLOCK + threadIdx.x;
    __shared__ PairEdge slot[BLOCK];
    volatile PairEdge* pe = &slot[threadIdx.x];
    if (!have_dt) {
        for (long long i = p; i < a.n; i += (long long)gridDim.x * BLOCK) a.s_out[i] = a.s_in[i];
    } else {
        const float dt = wdt.t;
        for (; p < np; p += stride) {
            const long long iA = 2 * (long long)p, iB = iA + 1;
            const bool hasB = iB < a.n;
            const V4<float> ownA = a.s_in[iA];
            const int4 tpA = a.topo[iA];
            const int cB = hasB ? __ldg(&a.topo[iB].x) : -1;
            const bool shared = tpA.x >= 0 && cB >= 0 && (long long)(tpA.x & kNbrMask) == iB &&
                                (long long)(cB & kNbrMask) == iA;
            // the first cell gives its edge 0; the handed-over flux waits in shared
            // memory, not in registers, through the first cell's other edges
            int mode = shared ? kPairGive : kPairNone;
            cand = min_nonneg(cand, update_cell_f32<GEO_EARLY, false, 1>(a, iA, ownA, tpA, dt, active, a.n_clamped,
                                                                         a.status, &mode, pe));
            if (hasB) {
                // the second cell's records are read after the first cell's update
                // (fewer live registers)
                const V4<float> ownB = a.s_in[iB];
                const int4 tpB = a.topo[iB];
                int modeB = mode == kPairGiven ? kPairTake : kPairNone;
                cand = min_nonneg(cand, update_cell_f32<GEO_EARLY, false, 2>(a, iB, ownB, tpB, dt, active,
                                                                             a.n_clamped, a.status, &modeB, pe));
            }
        }
    }
    block_min_publish<BLOCK>(cand, a.dt_write, active, a.n_active);
}

// ---- edge pass: each interior edge's flux once per step ----------------------------
// The canonical evaluation of an interior edge (from its left cell, Eq 12-30)
// is the one both of its cells make in step_kernel; here one thread makes it
// and stores, FP32, the flux leaving the left cell and both cells' bed source
// factors, or, FP64, both cells' terms (f64::EdgeTerms), which the cell pass
// (step_kernel with EDGES) applies with the left/right sign.  Edges with both cells dry are skipped: the cells form
// them inline.  Worth it where the flux arithmetic, not memory, bounds the
// step (the FP64 pipe).
template <typename T, int BLOCK>
__global__ void __launch_bounds__(BLOCK) edge_flux_kernel(const StepArgs<T> a) {
    const T g = a.g, h_dry = a.h_dry;
    const int threads = block_threads<T, BLOCK>();
    const long long stride = (long long)gridDim.x * threads;
    for (long long e = (long long)blockIdx.x * threads + threadIdx.x; e < a.n_edges; e += stride) {
        const int2 lr = a.ecells[e];
        if (a.debug && !(lr.x >= 0 && lr.x < a.n && lr.y >= 0 && lr.y < a.n)) {
            atomicOr(a.status, kStatusBadIndex);
            continue;
        }
        const V4<T> L = a.s_in[lr.x], R = a.s_in[lr.y];
        if (!gt_pos(L.x, h_dry) && !gt_pos(R.x, h_dry)) continue;
        V4<T> f;
        T sr;
        if constexpr (sizeof(T) == 8) {
            f64::Side l{L.x, 0.0, 0.0, L.w}, r{R.x, 0.0, 0.0, R.w};
            f64::velocity(L.x, L.y, L.z, h_dry, l.u, l.v);
            f64::velocity(R.x, R.y, R.z, h_dry, r.u, r.v);
            f64::EdgeTerms t;
            f64::edge(l, r, a.eln[2 * e], a.eln[2 * e + 1], f64::mul(0.5, g), h_dry, a.hll != 0, t);
            f.x = t.m; f.y = t.xL; f.z = t.yL; f.w = t.xR;
            sr = t.yR;
        } else {
            const T lx = a.eln[2 * e], ly = a.eln[2 * e + 1];
            const T rl = rsqrtf(edge_l2(lx, ly));
            T ui, vi;
            cell_velocity<T>(L.x, L.y, L.z, h_dry, ui, vi);
            edge_interior<T>(L.x, ui, vi, L.w, R.x, R.y, R.z, R.w, lx * rl, ly * rl, false, g, h_dry, f.x, f.y, f.z,
                             f.w, a.hll != 0, &sr);
        }
        a.eflux[e] = f;
        a.esrc[e] = sr;
    }
}

// ---- the fused step with activity bytes ------------------------------------------
// One byte per cell in three rotating buffers.  In the buffer a step reads, a
// cell's byte is non-zero exactly when the cell is not quiet: it is wet, or a
// neighbour is wet, or it has an inflow or fixed-stage edge.  The step marks
// in the next buffer (plain stores of 1, so concurrent marks of one byte
// agree) every cell that is wet after its update together with its
// neighbours, and every cell with an inflow/stage edge; and it clears each
// cell's byte in the third buffer, which the step after next fills.  A cell
// whose byte is 0 takes the quiet update (h, 0, 0) without its topology
// record or its neighbours' states -- the same result the neighbour test of
// update_cell gives, bit for bit.
//
// Over a list, in two launches: act_scan_kernel reads the bytes (2 per cell, 16 cells a
// thread, a block's 4,096 at a time, and none of a span whose flags say that
// they are all 0) and gathers the cells that run the flux path into a list, a
// span's cells in their order; a quiet cell costs it nothing more unless its
// state has to be written: where the cell was quiet in the previous step too,
// the output buffer (the state of two steps ago, itself dry at rest with the
// same h) holds it already.  step_kernel_act then updates the listed cells,
// dealt evenly to the threads.  On a mostly dry mesh the channel's cells lie
// together in the mesh order, so dealing out the cells by their place instead
// leaves some SMs with several times the average work and makes every quiet
// cell cost a state record read: that kernel, a cp.async pipeline over all
// cells, took 96 us a step on the 13M-cell river, 6 % of it wet; the two take
// 10 and 24 us.
//
// scan_span: one block's span, its threads' 16 cells from c0 on; `in` says that
// the thread's cells take part, `step` that they step (else state and activity
// carry over unchanged).
template <typename T, typename Args>
__device__ __forceinline__ void scan_span(const Args& a, unsigned sp, long long c0, long long n, bool in, bool step) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ unsigned total[kScanBlock / 32], base;
    uint4 now = make_uint4(0u, 0u, 0u, 0u), prev = now;
    if (in) {
        now = *(const uint4*)(a.act_in + c0);      // the buffers reach past n in whole 32 bytes
        prev = *(const uint4*)(a.act_clear + c0);
    }
    // bit 0 of a byte: the cell runs the flux path in this step; a previous
    // byte that is not 0: it ran it in the previous step, or the bytes were
    // rebuilt less than two steps ago
    const unsigned w[4] = {now.x, now.y, now.z, now.w}, v[4] = {prev.x, prev.y, prev.z, prev.w};
    // the low bits of a word's four bytes, as a 4-bit number
    auto low_bits = [](unsigned x) { return ((x & 0x01010101u) * 0x01020408u) >> 24; };
    unsigned runs = 0u, rewrite = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        runs |= low_bits(w[q]) << (4 * q);
        rewrite |= low_bits(v[q] | (v[q] >> 1)) << (4 * q);   // bytes are 0 to 3
    }
    if (rewrite) *(uint4*)(a.act_clear + c0) = make_uint4(0u, 0u, 0u, 0u);
    bool carry = false;
    if (in && !step) {
        carry = (w[0] | w[1] | w[2] | w[3]) != 0u;
        *(uint4*)(a.act_next + c0) = now;
        for (long long c = c0; c < c0 + 16 && c < n; ++c) a.s_out[c] = a.s_in[c];
        runs = 0u;
        rewrite = 0u;
    }
    rewrite &= ~runs;
    // a warp whose 512 cells are all to be rewritten (the two steps after the
    // bytes are rebuilt) copies them side by side
    if (__all_sync(0xffffffffu, rewrite == 0xFFFFu && c0 + 16 <= n)) {
        const long long w0 = c0 - 16 * lane;
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
            V4<T> s = a.s_in[w0 + 32 * k + lane];
            s.y = T(0); s.z = T(0);
            a.s_out[w0 + 32 * k + lane] = s;
        }
    } else {
        for (unsigned m = rewrite; m; m &= m - 1u) {
            const long long c = c0 + __ffs(m) - 1;
            if (c < n) {
                V4<T> s = a.s_in[c];
                s.y = T(0); s.z = T(0);
                a.s_out[c] = s;
            }
        }
    }
    const unsigned cnt = __popc(runs);
    unsigned pos = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned up = __shfl_up_sync(0xffffffffu, pos, o);
        if (lane >= o) pos += up;
    }
    if (lane == 31) total[warp] = pos;
    const bool any_carry = __syncthreads_or(carry);   // (and every thread has read the span's flags)
    unsigned before = 0u, all = 0u;
#pragma unroll
    for (int q = 0; q < kScanBlock / 32; ++q) {
        if (q == warp) before = all;
        all += total[q];
    }
    if (threadIdx.x == 0) {
        if (all) base = atomicAdd(a.act_count, all);
        a.span_clear[sp] = 0;
    }
    // the cells that this step will mark lie in this span or one beside it (the
    // marking kernel's own stores to a few hot flags took it from 24 to 33 us)
    if (all || any_carry)
        for (unsigned q = a.span_first[sp] + threadIdx.x; q < a.span_first[sp + 1]; q += kScanBlock)
            a.span_next[a.span_adj[q]] = 1;
    __syncthreads();
    unsigned at = base + before + pos - cnt;
    for (unsigned m = runs; m; m &= m - 1u) a.act_list[at++] = (unsigned)c0 + __ffs(m) - 1;
}

template <typename T>
__global__ void __launch_bounds__(kScanBlock) act_scan_kernel(const StepArgs<T> a) {
    // whether there is a step (warp_step_dt), by the bits alone: in thousands of
    // warps an FP64 product each takes microseconds
    const double dt = a.dt_fixed ? *a.dt_fixed : *a.dt_read;
    const bool have_dt = (unsigned long long)__double_as_longlong(dt) < kInfBits;
    const unsigned sp = blockIdx.x;   // the block's span
    if (!(a.span_in[sp] | a.span_clear[sp])) return;
    const long long c0 = ((long long)sp << kScanLog) + threadIdx.x * 16;
    scan_span<T>(a, sp, c0, a.n, c0 < a.n, have_dt);
}

// The listed cells' update and marks.  Each thread keeps the state and
// topology records of its next PF - 1 entries in flight through cp.async into
// its own shared-memory slots.
template <typename T, int BLOCK, int MINB, bool GEO_EARLY, int PF>
__global__ void __launch_bounds__(BLOCK, MINB) step_kernel_act(const StepArgs<T> a) {
    static_assert(BLOCK % 32 == 0, "warps of whole cells");
    static_assert(PF >= 2, "at least one entry ahead");
    const WarpDt<T> wdt = warp_step_dt<T>(a.cfl, a.dt_read, a.dt_fixed);
    const bool have_dt = wdt.have;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.dt_reset = kInfBits;
        if (have_dt) *a.t += wdt.d;
        else atomicOr(a.status, kStatusDry);
        if (a.dt_log) *a.dt_log = wdt.d;
    }
    T cand = inf_of<T>();
    unsigned active = 0u;
    const int tid = threadIdx.x;
    const unsigned stride = gridDim.x * BLOCK;
    const unsigned n_list = have_dt ? *(volatile const unsigned*)a.act_count : 0u;
    __shared__ V4<T> st_own[PF][BLOCK];
    __shared__ int4 st_topo[PF][BLOCK];
    __shared__ unsigned st_cell[PF][BLOCK];
    auto fetch = [&](int slot, unsigned k) {
        if (k < n_list) {
            const unsigned c = a.act_list[k];
            st_cell[slot][tid] = c;
            cp_async_record<sizeof(V4<T>)>(&st_own[slot][tid], &a.s_in[c]);
            cp_async_record<16>(&st_topo[slot][tid], &a.topo[c]);
        }
        cp_async_commit();
    };
    unsigned k = blockIdx.x * BLOCK + tid;   // host: n < 2^29, so k + PF stride < 2^32
#pragma unroll
    for (int s = 0; s < PF - 1; ++s) fetch(s, k + s * stride);
    const T dt = wdt.t;
    int slot = 0;
    for (; k < n_list; k += stride) {
        fetch(slot == 0 ? PF - 1 : slot - 1, k + (PF - 1) * stride);
        cp_async_wait<PF - 1>();
        const unsigned c = st_cell[slot][tid];
        const V4<T> own = st_own[slot][tid];
        const T r = update_cell<T, GEO_EARLY>(a, c, own, st_topo[slot][tid], dt, active, a.n_clamped, a.status);
        cand = min_nonneg(cand, r);
        const bool wet = r < inf_of<T>();
        // the topology record and the cell are read again from shared memory
        // rather than kept live in registers across the update
        const volatile int* tv = (const volatile int*)&st_topo[slot][tid];
        if (wet || (tv[3] & kStaticBit)) a.act_next[((const volatile unsigned*)st_cell[slot])[tid]] = 1;
        if (wet) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int code = tv[j];
                if (code >= 0 && (!a.debug || code_ok(code, a.n, a.n_groups))) a.act_next[code & kNbrMask] = 1;
            }
        }
        slot = slot == PF - 1 ? 0 : slot + 1;
    }
    cp_async_wait<0>();
    block_min_publish<BLOCK>(cand, a.dt_write, active, a.n_active);   // (a barrier: every thread has read the count)
    // the last block to get here empties the list for the next scan
    if (tid == 0 && atomicAdd(a.act_count + 1, 1u) == gridDim.x - 1) {
        a.act_count[0] = 0u;
        a.act_count[1] = 0u;
    }
}

// The same in one launch over all cells, FP32, for meshes where two launches and
// the list cost more than going through the quiet cells (list_activity has the
// measurements).  Per-thread cp.async pipeline over the thread's cells
// c_k = i0 + k stride:
// iteration k issues the topology of c_{k+1} (only if its byte is set), then
// the activity bytes of c_{k+PF+1} (8 lanes copy the warp's 32 bytes) and the
// state record of c_{k+PF}; it then processes c_k.  PF (the prefetch
// distance of the streamed state, >= 2) is a compiled shape parameter.
template <int BLOCK, int MINB, bool GEO_EARLY, int PF>
__global__ void __launch_bounds__(BLOCK, MINB) step_kernel_act_all(const StepArgs<float> a) {
    using T = float;
    static_assert(BLOCK % 32 == 0, "warps of whole cells");
    static_assert(PF >= 2, "the wait counts below assume a prefetch distance of at least two cells");
    constexpr int NS = PF + 1;  // state and activity slots
    const WarpDt<T> wdt = warp_step_dt<T>(a.cfl, a.dt_read, a.dt_fixed);
    const double dt_d = wdt.d;
    const bool have_dt = wdt.have;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.dt_reset = kInfBits;
        if (have_dt) *a.t += dt_d;
        else atomicOr(a.status, kStatusDry);
        if (a.dt_log) *a.dt_log = dt_d;
    }
    T cand = inf_of<T>();
    unsigned active = 0u;
    // 32-bit cell indices: the host allows this kernel only for n < 2^29, so
    // c + (PF + 1) stride < 2^32 with stride <= n + BLOCK and PF <= 5
    const unsigned stride = gridDim.x * BLOCK;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned i0 = blockIdx.x * BLOCK + tid;
    const unsigned n = (unsigned)a.n;
    if (!have_dt) {
        // no step: the state and its activity carry over unchanged
        for (unsigned c = i0; c < n; c += stride) {
            a.s_out[c] = a.s_in[c];
            a.act_next[c] = a.act_in[c];
            a.act_clear[c] = 0;
        }
    } else {
        static_assert(PF <= 5, "32-bit indices");
        __shared__ V4<T> st_own[NS][BLOCK];
        __shared__ int4 st_topo[2][BLOCK];
        __shared__ unsigned st_act[NS][BLOCK / 4];  // 32 activity bytes per warp per stage
        __shared__ unsigned st_prev[NS][BLOCK / 4]; // and the previous step's (act_clear) bytes
        const T dt = wdt.t;
        // warp w of the block owns st_act[.][8 w .. 8 w + 7]; lanes 0..7 copy 4 bytes each
        auto act_copy = [&](int slot, unsigned c) {
            const unsigned base = c - lane;
            if (lane < 8 && base < n) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                                 (unsigned)__cvta_generic_to_shared(&st_act[slot][warp * 8 + lane])),
                             "l"(a.act_in + base + 4 * lane)
                             : "memory");
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                                 (unsigned)__cvta_generic_to_shared(&st_prev[slot][warp * 8 + lane])),
                             "l"(a.act_clear + base + 4 * lane)
                             : "memory");
            }
        };
        // bit 0: the cell runs the flux path in this step (bit 0 of its byte);
        // bit 1: the previous step's byte is not 0 (the cell ran the flux path
        // then, or the bytes were rebuilt less than two steps ago)
        auto act_byte = [&](int slot) -> unsigned {
            return (((const unsigned char*)&st_act[slot][warp * 8])[lane] & 1u) |
                   (((const unsigned char*)&st_prev[slot][warp * 8])[lane] ? 2u : 0u);
        };
        // prologue: activity of c_0 .. c_PF and states of c_0 .. c_{PF-1}; then topology of c_0
#pragma unroll
        for (int q = 0; q <= PF; ++q) act_copy(q, i0 + q * stride);
#pragma unroll
        for (int q = 0; q < PF; ++q)
            if (i0 + q * stride < n) cp_async_record<sizeof(V4<T>)>(&st_own[q][tid], &a.s_in[i0 + q * stride]);
        cp_async_commit();
        cp_async_wait<0>();
        __syncwarp();
        unsigned f_cur = act_byte(0);
        if ((f_cur & 1u) && i0 < n) cp_async_record<16>(&st_topo[0][tid], &a.topo[i0]);
        cp_async_commit();                                       // T_{-1}
        cp_async_commit();                                       // H_{-1} (empty: its copies were in the first group)
        int ks = 0, k2 = 0;  // k mod NS, k mod 2
        for (unsigned c = i0; c - lane < n; c += stride) {
            const int ks1 = ks + 1 == NS ? 0 : ks + 1;          // slot of c_{k+1}
            const int ksp = ks == 0 ? NS - 1 : ks - 1;          // slot of c_{k+PF} (c_{k-1}'s, consumed)
            // groups so far: ..., T_{k-1}, H_{k-1}; H_{k-PF} and older (activity of
            // c_{k+1}, state of c_k) must be complete, which H_{k-2} implies
            cp_async_wait<2>();
            __syncwarp();
            const unsigned f_next = act_byte(ks1);
            const unsigned c1 = c + stride, cp = c + PF * stride, cp1 = c + (PF + 1) * stride;
            if ((f_next & 1u) && c1 < n) cp_async_record<16>(&st_topo[k2 ^ 1][tid], &a.topo[c1]);
            cp_async_commit();                                   // T_k
            __syncwarp();                                        // every lane has read slot ks before it refills
            act_copy(ks, cp1);
            if (cp < n) cp_async_record<sizeof(V4<T>)>(&st_own[ksp][tid], &a.s_in[cp]);
            cp_async_commit();                                   // H_k
            cp_async_wait<3>();                                  // T_{k-1}: the topology of c_k
            if (c < n) {
                const V4<T> own = st_own[ks][tid];
                if (!(f_cur & 1u)) {
                    // quiet: the new state is (h, 0, 0); if the cell was quiet in the
                    // previous step too, the output buffer (the state of two steps
                    // ago, itself dry at rest with the same h) holds it already
                    if (f_cur & 2u) {
                        V4<T> out;
                        out.x = own.x; out.y = T(0); out.z = T(0); out.w = own.w;
                        a.s_out[c] = out;
                    }
                } else {
                    const T r = update_cell<T, GEO_EARLY>(a, c, own, st_topo[k2][tid], dt, active, a.n_clamped,
                                                          a.status);
                    cand = min_nonneg(cand, r);
                    const bool wet = r < inf_of<T>();
                    // the topology record is read again from shared memory rather than kept
                    // live in registers across the update
                    const volatile int* tv = (const volatile int*)&st_topo[k2][tid];
                    if (wet || (tv[3] & kStaticBit)) a.act_next[c] = 1;
                    if (wet) {
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            const int code = tv[j];
                            if (code >= 0 && (!a.debug || code_ok(code, a.n, a.n_groups)))
                                a.act_next[code & kNbrMask] = 1;
                        }
                    }
                }
                a.act_clear[c] = 0;
            }
            f_cur = f_next;
            ks = ks1;
            k2 ^= 1;
        }
        cp_async_wait<0>();
    }
    block_min_publish<BLOCK>(cand, a.dt_write, active, a.n_active);
}

// Activity bytes of a state (into a buffer filled with 2): a wet cell marks
// itself and its neighbours, a cell with an inflow/stage edge marks itself.
// Bit 0 says that the cell runs the flux path; bit 1, set in every rebuilt
// byte, keeps the step after next from leaving a quiet state in place (its
// output buffer holds the state that was set, not a step's result).
template <typename T>
__global__ void act_init_kernel(const V4<T>* __restrict__ s, const int4* __restrict__ topo, long long n, T h_dry,
                                unsigned char* __restrict__ act) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    const bool wet = s[c].x > h_dry;
    const int4 tp = topo[c];
    if (wet || (tp.w & kStaticBit)) act[c] = 3;
    if (wet) {   // (an out-of-range index is skipped here; the step's debug checks report it)
        if (tp.x >= 0 && (tp.x & kNbrMask) < n) act[tp.x & kNbrMask] = 3;
        if (tp.y >= 0 && (tp.y & kNbrMask) < n) act[tp.y & kNbrMask] = 3;
        if (tp.z >= 0 && (tp.z & kNbrMask) < n) act[tp.z & kNbrMask] = 3;
    }
}

// ---- batched ensemble step -------------------------------------------------------
// Members advance together, each with its own CFL step: one launch covers every
// member's cells.  When a block moves on to another member, its warps publish
// the finished member's CFL minimum (warp shuffle, one atomicMin per warp, no
// barrier).
// The warp minimum is taken in the state precision and widened once (exact:
// widening is monotone), which keeps FP32 kernels off the FP64 pipe.
template <typename T>
__device__ __forceinline__ void warp_min_publish(T cand, unsigned long long* dst) {
    for (int o = 16; o > 0; o >>= 1) cand = min_nonneg(cand, __shfl_xor_sync(0xffffffffu, cand, o));
    if ((threadIdx.x & 31) == 0 && cand < inf_of<T>())
        atomicMin(dst, (unsigned long long)__double_as_longlong((double)cand));
}

// Tiles are dealt to blocks in round-robin chunks of 2^chunk_log2 tiles,
// which balances wet (expensive) and dry (cheap) members across the GPU while
// the member still changes only at chunk or member boundaries.  The chunk
// size, the tile size BLOCK and the grid are launch shapes chosen by the
// autotuner; none of them changes any cell's arithmetic.
__device__ __forceinline__ long long ens_tile_of(long long k, long long nchunk_stride, long long b, int cl2) {
    const long long mask = (1LL << cl2) - 1;
    return ((b + (k >> cl2) * nchunk_stride) << cl2) + (k & mask);
}

template <typename T, int BLOCK, int MINB, int STAGES, bool GEO_EARLY, bool EDGES = false>
__global__ void __launch_bounds__(BLOCK, (min_blocks_of<T, EDGES, true>(BLOCK, MINB))) ensemble_step_kernel(const EnsArgs<T> a) {
    static_assert(kEnsPad % BLOCK == 0, "a tile must not straddle two members");
    const long long G = gridDim.x, b = blockIdx.x;
    const int cl2 = a.chunk_log2;
    const long long t_lo = a.cell_lo / BLOCK;              // tiles from cell_lo on
    const long long n_tiles = (a.n_total - a.cell_lo) / BLOCK;
    const long long n_chunks = (n_tiles + (1LL << cl2) - 1) >> cl2;
    // this block's chunks: b, b + G, b + 2G, ... ; k counts its tiles
    const long long my_chunks = b < n_chunks ? (n_chunks - 1 - b) / G + 1 : 0;
    const long long k_end = my_chunks << cl2;
    const int tid = threadIdx.x;
    int member = -1;
    unsigned long long* sm = nullptr;
    bool have_dt = false;
    T dt = T(0);
    T cand = inf_of<T>();
    unsigned active = 0u;
    __shared__ V4<T> st_own[STAGES > 1 ? STAGES : 1][BLOCK];
    __shared__ int4 st_topo[STAGES > 1 ? STAGES : 1][BLOCK];
    if constexpr (STAGES > 1) {
#pragma unroll
        for (int s = 0; s < STAGES - 1; ++s) {
            const long long tile = ens_tile_of(s, G, b, cl2);
            if (s < k_end && tile < n_tiles) {
                const long long c = (tile + t_lo) * BLOCK + tid;
                cp_async_record<sizeof(V4<T>)>(&st_own[s][tid], &a.s_in[c]);
                cp_async_record<16>(&st_topo[s][tid], &a.topo[c]);
            }
            cp_async_commit();
        }
    }
    int slot = 0;
    for (long long k = 0; k < k_end; ++k) {
        const long long tile = ens_tile_of(k, G, b, cl2);
        if (tile >= n_tiles) break;                        // ragged last chunk
        const long long cell0 = (tile + t_lo) * BLOCK;
        const int mk = a.tile_member[cell0 / kEnsPad];     // uniform across the block
        if (mk != member) {
            if (member >= 0) warp_min_publish<T>(cand, sm + a.slot_write);
            cand = inf_of<T>();
            member = mk;
            sm = a.small + 8 * (long long)mk;
            // mk is uniform across the block, so every lane is here
            const WarpDt<T> wdt = warp_step_dt<T>(a.cfl[mk], (const double*)(sm + a.slot_read), nullptr);
            const double dt_d = wdt.d;
            have_dt = wdt.have;
            dt = wdt.t;
            if (cell0 == a.member_first_tile[mk] * kEnsPad && tid == 0) {
                sm[a.slot_reset] = kInfBits;
                if (have_dt) *(double*)(sm + 3) += dt_d;
                else atomicOr((unsigned*)(sm + 4), kStatusDry);
            }
        }
        const long long i = cell0 + tid;
        V4<T> own;
        int4 tp;
        if constexpr (STAGES > 1) {
            const long long kn = k + STAGES - 1;
            const long long nt = ens_tile_of(kn, G, b, cl2);
            const int fill = slot == 0 ? STAGES - 1 : slot - 1;
            if (kn < k_end && nt < n_tiles) {
                const long long c = (nt + t_lo) * BLOCK + tid;
                cp_async_record<sizeof(V4<T>)>(&st_own[fill][tid], &a.s_in[c]);
                cp_async_record<16>(&st_topo[fill][tid], &a.topo[c]);
            }
            cp_async_commit();
            cp_async_wait<STAGES - 1>();
            own = st_own[slot][tid];
            tp = st_topo[slot][tid];
            slot = slot == STAGES - 1 ? 0 : slot + 1;
        } else {
            own = a.s_in[i];
            tp = a.topo[i];
        }
        if (have_dt)
            cand = min_nonneg(cand, update_cell<T, GEO_EARLY, EDGES>(a, i, own, tp, dt, active, sm + 5, (unsigned*)(sm + 4)));
        else
            a.s_out[i] = own;
    }
    if constexpr (STAGES > 1) cp_async_wait<0>();
    if (member >= 0) warp_min_publish<T>(cand, sm + a.slot_write);
    active = __reduce_add_sync(0xffffffffu, active);
    if ((tid & 31) == 0 && active) atomicAdd(a.n_active, (unsigned long long)active);
}

// ---- batched ensemble step with dynamically taken chunks ------------------------------
// Each block takes its next chunk of 2^chunk_log2 tiles from a per-step
// counter (one atomicAdd per chunk, taken one chunk ahead), so blocks that
// drew cheap (dry) chunks take more of them and the grid finishes together.
// Which block updates a cell changes nothing in the cell's arithmetic, and the
// per-member minimum and the counters are order-independent: the results are
// those of the static schedule bit for bit.
template <typename T, int BLOCK, int MINB, bool GEO_EARLY>
__global__ void __launch_bounds__(BLOCK, MINB) ensemble_step_kernel_dyn(const EnsArgs<T> a) {
    static_assert(kEnsPad % BLOCK == 0, "a tile must not straddle two members");
    const int cl2 = a.chunk_log2;
    const long long t_lo = a.cell_lo / BLOCK;              // tiles from cell_lo on
    const long long n_tiles = (a.n_total - a.cell_lo) / BLOCK;
    const unsigned n_chunks = (unsigned)((n_tiles + (1LL << cl2) - 1) >> cl2);
    const int tid = threadIdx.x;
    __shared__ unsigned s_chunk[2];
    if (blockIdx.x == 0 && tid == 0) a.sched[a.sched_reset] = 0u;   // the counter of the step after next
    if (tid == 0) s_chunk[0] = atomicAdd(&a.sched[a.sched_slot], 1u);
    __syncthreads();
    int member = -1;
    unsigned long long* sm = nullptr;
    bool have_dt = false;
    T dt = T(0);
    T cand = inf_of<T>();
    unsigned active = 0u;
    unsigned chunk = s_chunk[0];
    for (int it = 0; chunk < n_chunks; ++it) {
        if (tid == 0) s_chunk[(it + 1) & 1] = atomicAdd(&a.sched[a.sched_slot], 1u);   // the next chunk, ahead
        const long long t0 = (long long)chunk << cl2;
        for (int q = 0; q < (1 << cl2); ++q) {
            const long long tile = t0 + q;
            if (tile >= n_tiles) break;                    // ragged last chunk
            const long long cell0 = (tile + t_lo) * BLOCK;
            const int mk = a.tile_member[cell0 / kEnsPad];  // uniform across the block
            if (mk != member) {
                if (member >= 0) warp_min_publish<T>(cand, sm + a.slot_write);
                cand = inf_of<T>();
                member = mk;
                sm = a.small + 8 * (long long)mk;
                const WarpDt<T> wdt = warp_step_dt<T>(a.cfl[mk], (const double*)(sm + a.slot_read), nullptr);
                have_dt = wdt.have;
                dt = wdt.t;
                if (cell0 == a.member_first_tile[mk] * kEnsPad && tid == 0) {
                    sm[a.slot_reset] = kInfBits;
                    if (have_dt) *(double*)(sm + 3) += wdt.d;
                    else atomicOr((unsigned*)(sm + 4), kStatusDry);
                }
            }
            const long long i = cell0 + tid;
            const V4<T> own = a.s_in[i];
            const int4 tp = a.topo[i];
            if (have_dt)
                cand = min_nonneg(cand, update_cell<T, GEO_EARLY>(a, i, own, tp, dt, active, sm + 5, (unsigned*)(sm + 4)));
            else
                a.s_out[i] = own;
        }
        __syncthreads();   // the next chunk's index is visible, and every thread has read this one
        chunk = s_chunk[(it + 1) & 1];
    }
    if (member >= 0) warp_min_publish<T>(cand, sm + a.slot_write);
    active = __reduce_add_sync(0xffffffffu, active);
    if ((tid & 31) == 0 && active) atomicAdd(a.n_active, (unsigned long long)active);
}

// ---- batched ensemble step over a list of its active cells ---------------------------
// The list mode of the ensemble (QUEUE): the mesh's two launches (act_scan_kernel,
// step_kernel_act) over the concatenated members.  The scan also forms each
// member's step size and does its bookkeeping; cells before cell_lo belong to
// the cell-pair kernel.  24 canal and river members of 3.7M cells in all, half
// of them fully wet: 85 to 89 us a step with any kernel that goes through all
// river cells (40 us for those), 61 with this one behind the cell-pair kernel.
template <typename T>
__global__ void __launch_bounds__(kScanBlock) ens_scan_kernel(const EnsArgs<T> a) {
    if (blockIdx.x == 0) {
        for (int mk = threadIdx.x; mk < a.n_members; mk += kScanBlock) {
            if (a.member_first_tile[mk] * kEnsPad < a.cell_lo) continue;
            unsigned long long* sm = a.small + 8 * (long long)mk;
            const double d = a.cfl[mk] * __longlong_as_double((long long)sm[a.slot_read]);
            a.member_dt[mk] = T(d);
            sm[a.slot_reset] = kInfBits;
            if ((unsigned long long)__double_as_longlong(d) < kInfBits) *(double*)(sm + 3) += d;
            else atomicOr((unsigned*)(sm + 4), kStatusDry);
        }
    }
    const unsigned sp = (unsigned)(a.cell_lo >> kScanLog) + blockIdx.x;
    if (!(a.span_in[sp] | a.span_clear[sp])) return;
    const long long c0 = ((long long)sp << kScanLog) + threadIdx.x * 16;
    const bool in = c0 >= a.cell_lo && c0 < a.n_total;   // (both ends are whole tiles)
    bool step = true;
    if (in) step = a.small[8 * (long long)a.tile_member[c0 / kEnsPad] + a.slot_read] < kInfBits;
    scan_span<T>(a, sp, c0, a.n_total, in, step);
}

// One lane's CFL minimum to its member's slot; the warp's at once where all
// lanes have the same member.
template <typename T>
__device__ __forceinline__ void publish_member(const EnsArgs<T>& a, int member, T cand) {
    const int m0 = __shfl_sync(0xffffffffu, member, 0);
    if (__all_sync(0xffffffffu, member == m0)) {
        if (m0 >= 0) warp_min_publish<T>(cand, a.small + 8 * (long long)m0 + a.slot_write);
    } else if (member >= 0 && cand < inf_of<T>()) {
        atomicMin(a.small + 8 * (long long)member + a.slot_write,
                  (unsigned long long)__double_as_longlong((double)cand));
    }
}

// The listed cells: a block takes an even share of the list in one piece (DYN:
// pieces of BLOCK << chunk_log2 entries as they come), so that its cells lie
// together and their member rarely changes.
template <typename T, int BLOCK, bool GEO_EARLY, bool DYN>
__device__ __forceinline__ void ens_list_steps(const EnsArgs<T>& a) {
    constexpr int PF = 2;
    __shared__ V4<T> st_own[PF][BLOCK];
    __shared__ int4 st_topo[PF][BLOCK];
    __shared__ unsigned st_cell[PF][BLOCK];
    __shared__ unsigned s_piece;
    const int tid = threadIdx.x;
    const unsigned n_list = *(volatile const unsigned*)a.act_count;
    if (DYN && blockIdx.x == 0 && tid == 0) a.sched[a.sched_reset] = 0u;   // the counter of the step after next
    int member = -1;
    T cand = inf_of<T>(), dt = T(0);
    unsigned active = 0u;
    unsigned lo, hi;
    const unsigned share = DYN ? (unsigned)BLOCK << a.chunk_log2
                               : ((n_list + gridDim.x - 1) / gridDim.x + 31u) & ~31u;
    for (unsigned piece = blockIdx.x;;) {
        if constexpr (DYN) {
            __syncthreads();   // every thread has read the last piece
            if (tid == 0) s_piece = atomicAdd(&a.sched[a.sched_slot], 1u);
            __syncthreads();
            piece = s_piece;
        }
        const unsigned long long first = (unsigned long long)piece * share;
        if (first >= n_list) break;
        lo = (unsigned)first;
        hi = n_list - lo > share ? lo + share : n_list;
        auto fetch = [&](int slot, unsigned k) {
            if (k < hi) {
                const unsigned c = a.act_list[k];
                st_cell[slot][tid] = c;
                cp_async_record<sizeof(V4<T>)>(&st_own[slot][tid], &a.s_in[c]);
                cp_async_record<16>(&st_topo[slot][tid], &a.topo[c]);
            }
            cp_async_commit();
        };
        fetch(0, lo + tid);
        int slot = 0;
        for (unsigned k0 = lo; k0 < hi; k0 += BLOCK) {     // uniform across the block
            const unsigned k = k0 + tid;
            fetch(slot ^ 1, k + BLOCK);
            cp_async_wait<1>();
            int mk = member;
            if (k < hi) mk = a.tile_member[st_cell[slot][tid] / kEnsPad];
            if (__any_sync(0xffffffffu, mk != member)) {
                publish_member<T>(a, member, cand);
                cand = inf_of<T>();
                member = mk;
                if (mk >= 0) dt = a.member_dt[mk];
            }
            if (k < hi) {
                const unsigned c = st_cell[slot][tid];
                unsigned long long* sm = a.small + 8 * (long long)mk;
                const T r = update_cell<T, GEO_EARLY>(a, c, st_own[slot][tid], st_topo[slot][tid], dt, active, sm + 5,
                                                      (unsigned*)(sm + 4));
                cand = min_nonneg(cand, r);
                const bool wet = r < inf_of<T>();
                const volatile int* tv = (const volatile int*)&st_topo[slot][tid];
                if (wet || (tv[3] & kStaticBit)) a.act_next[((const volatile unsigned*)st_cell[slot])[tid]] = 1;
                if (wet) {
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        const int code = tv[j];
                        if (code >= 0 && (!a.debug || code_ok(code, a.n_total, a.n_groups)))
                            a.act_next[code & kNbrMask] = 1;
                    }
                }
            }
            slot ^= 1;
        }
        cp_async_wait<0>();
        if constexpr (!DYN) break;
    }
    publish_member<T>(a, member, cand);
    __shared__ unsigned s_active;
    if (tid == 0) s_active = 0u;
    __syncthreads();
    active = __reduce_add_sync(0xffffffffu, active);
    if ((tid & 31) == 0 && active) atomicAdd(&s_active, active);
    __syncthreads();
    if (tid == 0 && s_active) atomicAdd(a.n_active, (unsigned long long)s_active);
    // the last block to get here empties the list for the next scan
    if (tid == 0 && atomicAdd(a.act_count + 1, 1u) == gridDim.x - 1) {
        a.act_count[0] = 0u;
        a.act_count[1] = 0u;
    }
}

// ---- batched ensemble step with activity bytes ----------------------------------------
// The activity mode of step_kernel_act over the concatenated members: the same
// bytes, marks and per-thread cp.async pipeline, with the thread's cells taken
// tile by tile in the ensemble's round-robin chunk order.  Tiles are whole
// (members are padded), so a tile is valid for every lane or for none.  Cells
// are indexed with 32 bits (the host allows this kernel below 2^29 cells).
//
// DYN takes the chunks dynamically, as ensemble_step_kernel_dyn does: the
// block's j-th chunk is s_ch[j mod 3], drawn from the step's counter two
// chunks ahead by thread 0 at the start of chunk j - 2 and published by the
// barrier that starts chunk j - 1, so the pipeline's look-ahead of three
// cells (into chunk j + 1 at most, chunks being at least 4 tiles) always
// finds its tile.  The slot refilled at the start of chunk j held chunk
// j - 1, which nothing reads after that barrier.
template <typename T, int BLOCK, int MINB, bool GEO_EARLY, bool DYN = false, bool QUEUE = false>
__global__ void __launch_bounds__(BLOCK, MINB) ensemble_step_kernel_act(const EnsArgs<T> a) {
    static_assert(kEnsPad % BLOCK == 0, "a tile must not straddle two members");
    if constexpr (QUEUE) {
        ens_list_steps<T, BLOCK, GEO_EARLY, DYN>(a);
        return;
    } else {
    constexpr unsigned kNone = 0xFFFFFFFFu;
    const unsigned G = gridDim.x, b = blockIdx.x;
    const int cl2 = a.chunk_log2;                   // >= 2 with DYN (the host checks)
    const unsigned t_lo = (unsigned)(a.cell_lo / BLOCK);           // tiles from cell_lo on
    const unsigned n_tiles = (unsigned)((a.n_total - a.cell_lo) / BLOCK);
    const unsigned n_chunks = (n_tiles + (1u << cl2) - 1) >> cl2;
    const unsigned my_chunks = b < n_chunks ? (n_chunks - 1 - b) / G + 1 : 0;
    const unsigned k_end = DYN ? kNone : my_chunks << cl2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ unsigned s_ch[3];
    if constexpr (DYN) {
        if (b == 0 && tid == 0) a.sched[a.sched_reset] = 0u;   // the counter of the step after next
        if (tid == 0) {
            s_ch[0] = atomicAdd(&a.sched[a.sched_slot], 1u);
            s_ch[1] = atomicAdd(&a.sched[a.sched_slot], 1u);
        }
        __syncthreads();
    }
    // this thread's cell in the block's k-th tile (kNone past the end)
    auto cell_of = [&](unsigned k) -> unsigned {
        if constexpr (DYN) {
            const unsigned ch = s_ch[(k >> cl2) % 3];
            if (ch >= n_chunks) return kNone;
            const unsigned t = (ch << cl2) + (k & ((1u << cl2) - 1));
            return t < n_tiles ? (t + t_lo) * BLOCK + tid : kNone;
        } else {
            if (k >= k_end) return kNone;
            const unsigned t = ((b + (k >> cl2) * G) << cl2) + (k & ((1u << cl2) - 1));
            return t < n_tiles ? (t + t_lo) * BLOCK + tid : kNone;
        }
    };
    __shared__ V4<T> st_own[3][BLOCK];
    __shared__ int4 st_topo[2][BLOCK];
    // per warp: the 32 activity bytes of its cells in 3 stages (lanes 0..7 copy
    // 4 each).  Unlike step_kernel_act, this kernel writes every quiet state:
    // leaving those quiet in two steps in place measured slower here (the
    // kernel is bound by instruction issue, not by its bytes).
    __shared__ unsigned st_act[3][BLOCK / 4];
    auto act_copy = [&](int slot, unsigned c) {
        if (lane < 8 && c != kNone)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(
                             (unsigned)__cvta_generic_to_shared(&st_act[slot][warp * 8 + lane])),
                         "l"(a.act_in + (c - lane) + 4 * lane)
                         : "memory");
    };
    // whether the cell runs the flux path (bit 0 of its byte)
    auto act_byte = [&](int slot) -> unsigned {
        return ((const unsigned char*)&st_act[slot][warp * 8])[lane] & 1u;
    };
    int member = -1;
    unsigned long long* sm = nullptr;
    bool have_dt = false;
    T dt = T(0);
    T cand = inf_of<T>();
    unsigned active = 0u;
    {
        const unsigned c0 = cell_of(0), c1 = cell_of(1), c2 = cell_of(2);
        act_copy(0, c0);
        act_copy(1, c1);
        act_copy(2, c2);
        if (c0 != kNone) cp_async_record<sizeof(V4<T>)>(&st_own[0][tid], &a.s_in[c0]);
        if (c1 != kNone) cp_async_record<sizeof(V4<T>)>(&st_own[1][tid], &a.s_in[c1]);
        cp_async_commit();
        cp_async_wait<0>();
        __syncwarp();
    }
    unsigned f_cur = act_byte(0);
    {
        const unsigned c0 = cell_of(0);
        if (f_cur && c0 != kNone) cp_async_record<16>(&st_topo[0][tid], &a.topo[c0]);
    }
    cp_async_commit();                                           // T_{-1}
    cp_async_commit();                                           // H_{-1} (empty)
    int k3 = 0, k2 = 0;
    for (unsigned k = 0; k < k_end; ++k) {
        if constexpr (DYN) {
            if ((k & ((1u << cl2) - 1)) == 0) {                  // a chunk starts (block-uniform)
                if (k) __syncthreads();
                if (tid == 0) s_ch[((k >> cl2) + 2) % 3] = atomicAdd(&a.sched[a.sched_slot], 1u);
            }
        }
        const unsigned c = cell_of(k);
        if (c == kNone) break;                                   // ragged last chunk (block-uniform)
        const int mk = a.tile_member[(c - tid) / kEnsPad];       // uniform across the block
        if (mk != member) {
            if (member >= 0) warp_min_publish<T>(cand, sm + a.slot_write);
            cand = inf_of<T>();
            member = mk;
            sm = a.small + 8 * (long long)mk;
            const WarpDt<T> wdt = warp_step_dt<T>(a.cfl[mk], (const double*)(sm + a.slot_read), nullptr);
            have_dt = wdt.have;
            dt = wdt.t;
            if ((long long)(c - tid) == a.member_first_tile[mk] * kEnsPad && tid == 0) {
                sm[a.slot_reset] = kInfBits;
                if (have_dt) *(double*)(sm + 3) += wdt.d;
                else atomicOr((unsigned*)(sm + 4), kStatusDry);
            }
        }
        const int k3n = k3 == 2 ? 0 : k3 + 1, k3nn = k3n == 2 ? 0 : k3n + 1;
        cp_async_wait<2>();
        __syncwarp();
        const unsigned f_next = act_byte(k3n);
        const unsigned c1 = cell_of(k + 1), c2 = cell_of(k + 2), c3 = cell_of(k + 3);
        if (f_next && c1 != kNone) cp_async_record<16>(&st_topo[k2 ^ 1][tid], &a.topo[c1]);
        cp_async_commit();                                       // T_k
        __syncwarp();
        act_copy(k3, c3);
        if (c2 != kNone) cp_async_record<sizeof(V4<T>)>(&st_own[k3nn][tid], &a.s_in[c2]);
        cp_async_commit();                                       // H_k
        cp_async_wait<3>();                                      // T_{k-1}: the topology of c_k
        const V4<T> own = st_own[k3][tid];
        if (!have_dt) {
            a.s_out[c] = own;
            a.act_next[c] = (unsigned char)f_cur;
        } else if (!f_cur) {
            V4<T> out;
            out.x = own.x; out.y = T(0); out.z = T(0); out.w = own.w;
            a.s_out[c] = out;
        } else {
            const T r = update_cell<T, GEO_EARLY>(a, c, own, st_topo[k2][tid], dt, active, sm + 5,
                                                  (unsigned*)(sm + 4));
            cand = min_nonneg(cand, r);
            const bool wet = r < inf_of<T>();
            const volatile int* tv = (const volatile int*)&st_topo[k2][tid];
            if (wet || (tv[3] & kStaticBit)) a.act_next[c] = 1;
            if (wet) {
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const int code = tv[j];
                    if (code >= 0 && (!a.debug || code_ok(code, a.n_total, a.n_groups)))
                        a.act_next[code & kNbrMask] = 1;
                }
            }
        }
        a.act_clear[c] = 0;
        f_cur = f_next;
        k3 = k3n;
        k2 ^= 1;
    }
    cp_async_wait<0>();
    if (member >= 0) warp_min_publish<T>(cand, sm + a.slot_write);
    active = __reduce_add_sync(0xffffffffu, active);
    if ((tid & 31) == 0 && active) atomicAdd(a.n_active, (unsigned long long)active);
    }
}

// ---- batched ensemble step over cell pairs (FP32) ------------------------------------
// A split ensemble places the members that are mostly wet at creation first in
// its layout; this kernel updates their spans [0, pair_spans), and one of the
// other ensemble kernels the rest (from cell_lo on) in the same step.  A block
// takes a contiguous run of spans (the wet members cost about the same per
// cell, so equal runs balance, and a block changes member rarely); its thread
// t updates the pair (2t, 2t+1) of the span (BLOCK pairs = kEnsPad cells)
// exactly as step_kernel_pair does, so the members' results are those of the
// plain solver bit for bit.
template <int BLOCK, int MINB, bool GEO_EARLY>
__global__ void __launch_bounds__(BLOCK, MINB) ensemble_step_kernel_pair(const EnsArgs<float> a) {
    static_assert(2 * BLOCK == kEnsPad, "a block's pairs are one span");
    const unsigned ns = a.pair_spans;
    const unsigned lo = (unsigned)((unsigned long long)ns * blockIdx.x / gridDim.x);
    const unsigned hi = (unsigned)((unsigned long long)ns * (blockIdx.x + 1) / gridDim.x);
    const int tid = threadIdx.x;
    __shared__ PairEdge slot[BLOCK];
    volatile PairEdge* pe = &slot[tid];
    unsigned active = 0u;
    // runs of spans of one member: the member's step size, then its spans; the
    // member's status block is addressed from its index where used
    for (unsigned t = lo; t < hi;) {
        const int mk = a.tile_member[t];       // uniform across the block
        unsigned long long* sm = a.small + 8 * mk;
        const WarpDt<float> wdt = warp_step_dt<float>(a.cfl[mk], (const double*)(sm + a.slot_read), nullptr);
        if ((long long)t == a.member_first_tile[mk] && tid == 0) {
            sm[a.slot_reset] = kInfBits;
            if (wdt.have) *(double*)(sm + 3) += wdt.d;
            else atomicOr((unsigned*)(sm + 4), kStatusDry);
        }
        if (!wdt.have) {
            for (; t < hi && a.tile_member[t] == mk; ++t) {
                const unsigned iA = t * kEnsPad + 2 * tid;
                a.s_out[iA] = a.s_in[iA];
                a.s_out[iA + 1] = a.s_in[iA + 1];
            }
            continue;
        }
        const float dt = wdt.t;
        float cand = inf_of<float>();
        for (; t < hi && a.tile_member[t] == mk; ++t) {
            const unsigned iA = t * kEnsPad + 2 * tid, iB = iA + 1;
            const V4<float> ownA = a.s_in[iA];
            const int4 tpA = a.topo[iA];
            const int cB = __ldg(&a.topo[iB].x);
            const bool shared = tpA.x >= 0 && cB >= 0 && (unsigned)(tpA.x & kNbrMask) == iB &&
                                (unsigned)(cB & kNbrMask) == iA;
            int mode = shared ? kPairGive : kPairNone;
            cand = min_nonneg(cand, update_cell_f32<GEO_EARLY, false, 1>(a, iA, ownA, tpA, dt, active,
                                                                         a.small + 8 * mk + 5,
                                                                         (unsigned*)(a.small + 8 * mk + 4), &mode,
                                                                         pe));
            const V4<float> ownB = a.s_in[iB];
            const int4 tpB = a.topo[iB];
            int modeB = mode == kPairGiven ? kPairTake : kPairNone;
            cand = min_nonneg(cand, update_cell_f32<GEO_EARLY, false, 2>(a, iB, ownB, tpB, dt, active,
                                                                         a.small + 8 * mk + 5,
                                                                         (unsigned*)(a.small + 8 * mk + 4), &modeB,
                                                                         pe));
        }
        warp_min_publish<float>(cand, a.small + 8 * mk + a.slot_write);
    }
    active = __reduce_add_sync(0xffffffffu, active);
    if ((tid & 31) == 0 && active) atomicAdd(a.n_active, (unsigned long long)active);
}

// ---- CFL min of a given state (used after swe_set_state), and its wet cells where
// n_wet is given ----------------------------------------------------------------------
template <typename T, int BLOCK>
__global__ void __launch_bounds__(BLOCK) dt_kernel(const V4<T>* __restrict__ s, const V4<T>* __restrict__ geoB,
                                                   long long n, T g, T h_dry, unsigned long long* dt_write,
                                                   unsigned long long* n_wet) {
    using A = Ar<T>;
    const long long i = (long long)blockIdx.x * BLOCK + threadIdx.x;
    T cand = inf_of<T>();
    unsigned wet = 0u;
    if (i < n) {
        const V4<T> c = s[i];
        if (c.x > h_dry) {
            wet = 1u;
            const T r = A::rcp_(c.x);
            const T u = c.y * r, v = c.z * r;
            cand = A::div_(geoB[i].w, A::sqrt_(g * c.x) + A::sqrt_(u * u + v * v));
        }
    }
    block_min_publish<BLOCK>(cand, dt_write, wet, n_wet);
}

// ---- layout conversion between caller arrays and the packed internal state --------
// Each direction makes its random accesses reads (13M cells numbered by an
// unstructured mesher): packing gathers the caller's three values by internal
// order, perm[internal] = caller (scattering whole records by the caller's
// order took 420 us, 16-byte writes into 32-byte sectors); unpacking gathers a
// record by the caller's order, inv[caller] = internal, and writes side by
// side (204 us).
template <typename T>
__global__ void pack_state_kernel(const T* __restrict__ h, const T* __restrict__ hu, const T* __restrict__ hv,
                                  const unsigned* __restrict__ perm, const T* __restrict__ z, V4<T>* __restrict__ s,
                                  long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const unsigned o = perm[i];
        V4<T> v;
        v.x = h[o]; v.y = hu[o]; v.z = hv[o]; v.w = z[i];
        s[i] = v;
    }
}

template <typename T>
__global__ void unpack_state_kernel(const V4<T>* __restrict__ s, const unsigned* __restrict__ inv, T* __restrict__ h,
                                    T* __restrict__ hu, T* __restrict__ hv, long long n) {
    const long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (o < n) {
        const V4<T> v = s[inv[o]];
        h[o] = v.x; hu[o] = v.y; hv[o] = v.z;
    }
}

// ---- batched Riemann flux (parity entry point) --------------------------------------
template <typename T>
__global__ void riemann_batch_kernel(long long n, const T* __restrict__ hL, const T* __restrict__ unL,
                                     const T* __restrict__ utL, const T* __restrict__ hR,
                                     const T* __restrict__ unR, const T* __restrict__ utR, T g, T h_dry,
                                     T* __restrict__ G1, T* __restrict__ G2, T* __restrict__ G3, T* __restrict__ S,
                                     int hll) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        T a, b, c, sp[3];
        riemann_hllc<T>(hL[i], unL[i], utL[i], hR[i], unR[i], utR[i], g, h_dry, a, b, c, sp, hll != 0);
        G1[i] = a; G2[i] = b; G3[i] = c;
        if (S) { S[3 * i] = sp[0]; S[3 * i + 1] = sp[1]; S[3 * i + 2] = sp[2]; }
    }
}

// ---- blocks of the FP64 step kernels on small meshes ------------------------------------
// A grid of more blocks than full ones cover the cells with means smaller
// blocks: whole warps, as few as still cover them.  Up to kSpreadCells FP64
// cells (or edges) the default is one-warp blocks: a lone warp's FP64
// instruction holds its SM quarter for 64 clocks, four quarters together reach
// one per 19, so warps should be spread evenly (4,000 cells: 9,663 -> 9,134 us
// for 500 steps).  FP32 steps measured the same to 2 % slower with it.
constexpr long long kSpreadCells = 152LL * 12 * 32;   // 12 one-warp blocks on each of GB300's 152 SMs
template <typename T>
__host__ __device__ inline unsigned step_threads(long long n, unsigned grid, int block) {
    if (sizeof(T) == 4) return (unsigned)block;
    const long long per = (n + grid - 1) / grid;
    const long long t = (per + 31) / 32 * 32;
    return (unsigned)(t < block ? (t < 32 ? 32 : t) : block);
}
inline unsigned spread_grid(long long n) { return (unsigned)((n + 31) / 32); }

// ---- host-side launchers, one set per precision ------------------------------------
template <typename T>
struct LoopArgs;

template <typename T>
struct Launch {
    // (block, min_blocks) pairs with a compiled kernel; see step_variants()
    // with a.act_in set, the activity kernel (stages ignored) runs
    static cudaError_t step(const StepArgs<T>& a, int block, int min_blocks, int stages, int geo_early,
                            cudaStream_t st);
    // with a.eflux set (and a.act_in not), the edge pass then the cell pass run
    static cudaError_t resident_blocks(int block, int min_blocks, int stages, int geo_early, int activity,
                                       int edges, int* per_sm);
    // compiled (block, min_blocks, stages, geo_early) shapes of the cell pass of the edge-pass step
    static int edge_variants(int (*out)[4], int max);
    // the edge pass alone (interior fluxes of a.s_in into a.eflux, a.esrc)
    static cudaError_t edge_flux(const StepArgs<T>& a, cudaStream_t st);
    // compiled (block, min_blocks, geo_early, stages = prefetch distance + 1) shapes of the activity kernel
    static int act_variants(int (*out)[4], int max);
    static cudaError_t act_init(const V4<T>* s, const int4* topo, long long n, T h_dry, unsigned char* act,
                                cudaStream_t st);
    // compiled (block, min_blocks, stages, geo_early) shapes of the step kernel; returns their number
    static int step_variants(int (*out)[4], int max);
    // the step over cell pairs (FP32 only; cudaErrorInvalidValue otherwise) with one of its
    // compiled (block, min_blocks, geo_early, stages) shapes; a.grid blocks of `block` threads,
    // each thread a pair at a time
    static cudaError_t step_pair(const StepArgs<T>& a, int block, int min_blocks, int geo_early, int stages,
                                 cudaStream_t st);
    static cudaError_t pair_resident_blocks(int block, int min_blocks, int geo_early, int stages, int* per_sm);
    static int pair_variants(int (*out)[4], int max);
    // batched ensemble step with one of its compiled (block, min_blocks, stages, geo_early) shapes
    static cudaError_t ensemble_step(const EnsArgs<T>& a, int block, int min_blocks, int stages, int geo_early,
                                     unsigned grid, cudaStream_t st);
    static cudaError_t ensemble_resident_blocks(int block, int min_blocks, int stages, int geo_early, int* per_sm);
    static int ensemble_variants(int (*out)[4], int max);
    // activity kernel of the ensemble: compiled (block, min_blocks, geo_early) shapes,
    // with round-robin (dynamic 0) or dynamically taken (dynamic 1) chunks
    // (queue 1, FP32: the cells that run the flux path are gathered per warp into
    // full warps first; compiled shapes from ensemble_actq_variants)
    static cudaError_t ensemble_step_act(const EnsArgs<T>& a, int block, int min_blocks, int geo_early,
                                         unsigned grid, cudaStream_t st, int dynamic = 0, int queue = 0);
    static cudaError_t ensemble_act_resident_blocks(int block, int min_blocks, int geo_early, int* per_sm,
                                                    int dynamic = 0, int queue = 0);
    static int ensemble_act_variants(int (*out)[3], int max);
    static int ensemble_actq_variants(int (*out)[3], int max);
    // edge pass of the ensemble (a.eflux set): edge kernel, then the cell pass of
    // one of its compiled (block, min_blocks, stages, geo_early) shapes
    static int ensemble_edge_variants(int (*out)[4], int max);
    // dynamically scheduled ensemble kernel: compiled (block, min_blocks, geo_early) shapes
    static cudaError_t ensemble_step_dyn(const EnsArgs<T>& a, int block, int min_blocks, int geo_early,
                                         unsigned grid, cudaStream_t st);
    static cudaError_t ensemble_dyn_resident_blocks(int block, int min_blocks, int geo_early, int* per_sm);
    static int ensemble_dyn_variants(int (*out)[3], int max);
    static cudaError_t ensemble_edge_resident_blocks(int block, int min_blocks, int stages, int geo_early,
                                                     int* per_sm);
    // cell-pair kernel of a split ensemble (FP32 only): 128-thread blocks, compiled
    // (min_blocks, geo_early) shapes
    static cudaError_t ensemble_step_pair(const EnsArgs<T>& a, int min_blocks, int geo_early, unsigned grid,
                                          cudaStream_t st);
    static cudaError_t ensemble_pair_resident_blocks(int min_blocks, int geo_early, int* per_sm);
    static int ensemble_pair_variants(int (*out)[2], int max);
    static void ensemble_default(int* block, int* min_blocks, int* stages, int* geo_early);
    static int default_min_blocks(int block);
    // many steps in one cooperative launch (swe_loop.cuh): the largest mesh whose
    // grid is resident, and the launch
    static cudaError_t loop_capacity(int device, long long* cells);
    static cudaError_t loop(const LoopArgs<T>& a, cudaStream_t st);
    static cudaError_t dt(const V4<T>* s, const V4<T>* geoB, long long n, T g, T h_dry,
                          unsigned long long* dt_write, unsigned long long* n_wet,
                          cudaStream_t st);
    static cudaError_t pack(const T* h, const T* hu, const T* hv, const unsigned* perm, const T* z,
                            V4<T>* s, long long n, cudaStream_t st);
    static cudaError_t unpack(const V4<T>* s, const unsigned* inv, T* h, T* hu, T* hv, long long n,
                              cudaStream_t st);
    static cudaError_t riemann(long long n, const T* hL, const T* unL, const T* utL, const T* hR,
                               const T* unR, const T* utR, T g, T h_dry, T* G1, T* G2, T* G3, T* S,
                               int hll, cudaStream_t st);
};

}  // namespace swe
