// swe_loop.cuh -- many steps of a small mesh in one launch.
//
// A step of a few thousand cells is all latency: launching its kernel, reading
// the step size, the gathers, and the block reductions cost 4.6 us on 20,000
// FP32 cells and 13 us on 4,000 FP64 cells with the edge pass's two kernels,
// against under 1 us of arithmetic.  Here one cooperative launch runs all the
// steps of a call: a cell (FP32), or the cells of a block and the edges that
// touch them (FP64), stays with its thread, which keeps its static data and
// its own state in registers, and the grid meets once per step.  The cells'
// arithmetic is that of the other kernels, so are the bits.
#pragma once

#include "swe_kernels.cuh"

namespace swe {

// Limit of the polls of one wait (under 2 s; a step takes microseconds).  A
// grid that gives up sets kStatusStall and leaves, and no loop starts on a
// status block that has it.
constexpr unsigned kMaxPolls = 1u << 22;
// words of the status block
constexpr int kLoopSlotT = 3, kLoopSlotStatus = 4, kLoopSlotClamp = 5, kLoopSlotActive = 6, kLoopSlotDtLast = 7;

template <typename T>
struct LoopArgs {
    V4<T>* state[2];                   // the states' ping-pong pair
    const V4<T>* geoA;
    const V4<T>* geoB;
    const V4<T>* geoR;
    const int4* topo;
    const T* gm2;
    unsigned long long* small;         // status block
    unsigned* barrier;                 // arrivals, 0 at launch
    long long n;
    long long step0;                   // index of the first step
    int steps;
    unsigned max_polls;                // of one wait
    int one_block_sms;                 // FP64: no SM has more than one block
    double cfl;
    T g, h_dry;
    int hll, debug, n_groups;
    BcTable bc;
    // FP64: per block kLoopEdges slots, the edges that touch its cells
    // ((left, right) cell, left < 0: none; unit normal), and per cell
    // the slots of its three edges
    const int2* ecell;
    const double* egeo;                // [block][2][kLoopEdges]
    const uchar4* eslot;
};

constexpr int kLoopCells = 32;         // FP64 cells of a block: one warp's
constexpr int kLoopEdges = 96;         // at most three each

// A state written by another SM in the step before: from L2.
__device__ __forceinline__ V4<float> load_l2(const V4<float>* p) {
    const float4 v = __ldcg((const float4*)p);
    V4<float> r;
    r.x = v.x; r.y = v.y; r.z = v.z; r.w = v.w;
    return r;
}
__device__ __forceinline__ V4<double> load_l2(const V4<double>* p) {
    const double2 a = __ldcg((const double2*)p), b = __ldcg((const double2*)p + 1);
    V4<double> r;
    r.x = a.x; r.y = a.y; r.z = b.x; r.w = b.y;
    return r;
}

// What update_cell_f32 and finish_cell take as their arguments: one cell's view
// of the loop.  The cell's new state stays here for the next step.
template <typename T>
struct LoopCell {
    const LoopArgs<T>& a;
    const V4<T>* s_in;
    V4<T>* s_out;
    V4<T> gA, gB;                      // FP32: the cell's geometry
    V4<T>* next;
    T g, h_dry;
    int hll, debug, n_groups;
    __device__ __forceinline__ int bc_kind(int grp) const { return a.bc.kind[grp]; }
    __device__ __forceinline__ double bc_value(int grp) const { return a.bc.value[grp]; }
    __device__ __forceinline__ long long cell_bound() const { return a.n; }
};
template <typename T>
__device__ __forceinline__ V4<T> load_state(const LoopCell<T>& a, long long i) { return load_l2(a.s_in + i); }
template <typename T>
__device__ __forceinline__ void store_state(const LoopCell<T>& a, long long i, const V4<T>& v) {
    *a.next = v;
    a.s_out[i] = v;
}
template <typename T>
__device__ __forceinline__ void load_geometry(const LoopCell<T>& a, long long, V4<T>& gA, V4<T>& gB) {
    gA = a.gA;
    gB = a.gB;
}

// Every block's writes before, its reads after: the block's threads meet,
// thread 0 releases them with its arrival and waits for the others'.  Returns
// whether all arrived.
__device__ __forceinline__ bool grid_meet(unsigned* barrier, unsigned target, unsigned max_polls, unsigned* status,
                                          int* failed) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(barrier, 1u);
        unsigned seen = 0u;
        for (unsigned polls = 0u; seen < target && polls < max_polls; ++polls)
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(barrier) : "memory");
        if (seen < target) {
            atomicOr(status, kStatusStall);
            *failed = 1;
        }
    }
    __syncthreads();
    return *failed == 0;
}

// Whether an earlier loop gave up on this status block (the whole block calls).
__device__ __forceinline__ bool loop_stalled(const unsigned* status) {
    return __syncthreads_or((int)(*(const volatile unsigned*)status & kStatusStall)) != 0;
}

// One step's size from the slot that the step before has filled.
template <typename T>
__device__ __forceinline__ WarpDt<T> loop_dt(double cfl, const unsigned long long* slot) {
    const double v = cfl * __longlong_as_double((long long)__ldcg(slot));
    WarpDt<T> r;
    r.d = v;
    r.t = T(v);
    r.have = (unsigned long long)__double_as_longlong(v) < kInfBits;
    return r;
}

// The bookkeeping of a step, by one thread of the grid (as in step_kernel).
template <typename T>
__device__ __forceinline__ void loop_book(const LoopArgs<T>& a, int p3, const WarpDt<T>& dt) {
    a.small[(p3 + 2) % 3] = kInfBits;
    double* t = (double*)(a.small + kLoopSlotT);
    if (dt.have) *t += dt.d;
    else atomicOr((unsigned*)(a.small + kLoopSlotStatus), kStatusDry);
    *(double*)(a.small + kLoopSlotDtLast) = dt.d;
}

// FP32: a cell per thread.
template <int BLOCK, int MINB>
__global__ void __launch_bounds__(BLOCK, MINB) step_loop_f32(const LoopArgs<float> a) {
    __shared__ int failed;
    if (threadIdx.x == 0) failed = 0;
    const long long i = (long long)blockIdx.x * BLOCK + threadIdx.x;
    const bool in = i < a.n;
    unsigned* const status = (unsigned*)(a.small + kLoopSlotStatus);
    if (loop_stalled(status)) return;
    V4<float> own{}, next{};
    int4 tp = make_int4(-1, -1, -1, 0);
    LoopCell<float> v{a, nullptr, nullptr, {}, {}, &next, a.g, a.h_dry, a.hll, a.debug, a.n_groups};
    if (in) {
        own = a.state[a.step0 % 2][i];
        tp = a.topo[i];
        v.gA = a.geoA[i];
        v.gB = a.geoB[i];
    }
    int p2 = (int)(a.step0 % 2), p3 = (int)(a.step0 % 3);
    unsigned active = 0u;
    unsigned long long active_sum = 0ULL;
    for (int s = 0; s < a.steps; ++s) {
        const WarpDt<float> dt = loop_dt<float>(a.cfl, a.small + p3);
        if (i == 0) loop_book(a, p3, dt);
        float cand = inf_of<float>();
        if (in) {
            if (dt.have) {
                v.s_in = a.state[p2];
                v.s_out = a.state[1 - p2];
                cand = update_cell_f32<true, false>(v, i, own, tp, dt.t, active, a.small + kLoopSlotClamp, status);
                own = next;
            } else {
                a.state[1 - p2][i] = own;
            }
        }
        p2 = 1 - p2;
        p3 = p3 == 2 ? 0 : p3 + 1;
        block_min_publish<BLOCK>(cand, a.small + p3);   // the slot that the next step reads
        if (!grid_meet(a.barrier, (unsigned)(s + 1) * gridDim.x, a.max_polls, status, &failed)) break;
    }
    active_sum = __reduce_add_sync(0xffffffffu, active);
    if ((threadIdx.x & 31) == 0 && active_sum) atomicAdd(a.small + kLoopSlotActive, active_sum);
}

// FP64: three warps evaluate the edges that touch the block's 32 cells, an edge
// per thread, into shared memory; the first updates the cells.  An edge
// between two blocks is evaluated by both, the others once.
// S: f64::SoftRoots while an SM has one block (a warp per quarter), else Soft.
template <int MINB, class S>
__global__ void __launch_bounds__(kLoopEdges, MINB) step_loop_f64(const LoopArgs<double> a) {
    __shared__ int failed;
    __shared__ double term[5][kLoopEdges];
    __shared__ unsigned char wet_edge[kLoopEdges];
    const int tid = threadIdx.x;
    if (tid == 0) failed = 0;
    unsigned* const status = (unsigned*)(a.small + kLoopSlotStatus);
    if (loop_stalled(status)) return;
    const double h_dry = a.h_dry, g2 = f64::mul(0.5, a.g);
    const int2 lr = a.ecell[(long long)blockIdx.x * kLoopEdges + tid];
    const double* const eg = a.egeo + (long long)blockIdx.x * 2 * kLoopEdges + tid;
    double n1 = 0.0, n2 = 0.0;
    if (lr.x >= 0) { n1 = eg[0]; n2 = eg[kLoopEdges]; }
    const long long i = (long long)blockIdx.x * kLoopCells + tid;
    const bool in = tid < kLoopCells && i < a.n;
    V4<double> own{}, next{};
    int4 tp = make_int4(-1, -1, -1, 0);
    uchar4 slot = make_uchar4(0, 0, 0, 0);
    double ia = 0.0, rin = 0.0, gm2 = 0.0;
    V4<double> gR{};                   // the edges' lengths
    bool open = false;                 // a boundary edge that keeps the cell out of the quiet path
    LoopCell<double> v{a, nullptr, nullptr, {}, {}, &next, a.g, a.h_dry, a.hll, a.debug, a.n_groups};
    if (in) {
        own = a.state[a.step0 % 2][i];
        tp = a.topo[i];
        slot = a.eslot[i];
        ia = a.geoB[i].z;
        rin = a.geoB[i].w;
        gm2 = a.gm2[i];
        gR = a.geoR[i];
        open = (tp.w & kStaticBit) != 0;
    }
    int p2 = (int)(a.step0 % 2), p3 = (int)(a.step0 % 3);
    unsigned active = 0u;
    for (int s = 0; s < a.steps; ++s) {
        const WarpDt<double> dt = loop_dt<double>(a.cfl, a.small + p3);
        if (blockIdx.x == 0 && tid == 0) loop_book(a, p3, dt);
        const V4<double>* const s_in = a.state[p2];
        if (lr.x >= 0) {
            const V4<double> L = load_l2(s_in + lr.x), R = load_l2(s_in + lr.y);
            f64::Side l{L.x, 0.0, 0.0, L.w}, r{R.x, 0.0, 0.0, R.w};
            f64::velocity<S>(L.x, L.y, L.z, h_dry, l.u, l.v);
            f64::velocity<S>(R.x, R.y, R.z, h_dry, r.u, r.v);
            f64::EdgeTerms t;
            f64::edge<S>(l, r, n1, n2, g2, h_dry, a.hll != 0, t);
            term[0][tid] = t.m; term[1][tid] = t.xL; term[2][tid] = t.yL; term[3][tid] = t.xR; term[4][tid] = t.yR;
            wet_edge[tid] = gt_pos(L.x, h_dry) || gt_pos(R.x, h_dry);
        }
        __syncthreads();
        double cand = inf_of<double>();
        if (in) {
            v.s_out = a.state[1 - p2];
            if (!dt.have) {
                v.s_out[i] = own;
            } else {
                const int code[3] = {tp.x, tp.y, tp.z};
                bool quiet = !gt_pos(own.x, h_dry) && !open;
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const int e = j == 0 ? slot.x : (j == 1 ? slot.y : slot.z);
                    if (code[j] >= 0 && wet_edge[e]) quiet = false;
                }
                if (quiet) {
                    own.y = 0.0; own.z = 0.0;
                    v.s_out[i] = own;
                } else {
                    active += 1u;
                    double m = 0.0, x = 0.0, y = 0.0;
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        const int c = code[j], e = j == 0 ? slot.x : (j == 1 ? slot.y : slot.z);
                        double tm, tx, ty;
                        if (c >= 0) {
                            const bool flip = (c & kFlipBit) != 0;
                            const double um = term[0][e], ux = term[flip ? 3 : 1][e], uy = term[flip ? 4 : 2][e];
                            tm = flip ? -um : um; tx = flip ? -ux : ux; ty = flip ? -uy : uy;
                        } else {
                            const double2 n = j == 2 ? *(const double2*)&a.geoB[i] : ((const double2*)&a.geoA[i])[j];
                            const int grp = -1 - c;
                            f64::Side side{own.x, 0.0, 0.0, own.w};
                            f64::velocity<S>(own.x, own.y, own.z, h_dry, side.u, side.v);
                            f64::boundary(a.bc.kind[grp], a.bc.value[grp], side, n.x, n.y, g2, h_dry, a.hll != 0, tm,
                                          tx, ty);
                        }
                        const double len = j == 0 ? gR.x : (j == 1 ? gR.y : gR.z);
                        m = f64::fma(len, tm, m);
                        x = f64::fma(len, tx, x);
                        y = f64::fma(len, ty, y);
                    }
                    cand = finish_cell<S>(v, i, own, m, x, y, ia, rin, gm2, dt.t, a.small + kLoopSlotClamp, status);
                    own = next;
                }
            }
        }
        p2 = 1 - p2;
        p3 = p3 == 2 ? 0 : p3 + 1;
        if (tid < 32) warp_min_publish<double>(cand, a.small + p3);
        if (!grid_meet(a.barrier, (unsigned)(s + 1) * gridDim.x, a.max_polls, status, &failed)) break;
    }
    if (tid < 32) {
        active = __reduce_add_sync(0xffffffffu, active);
        if (tid == 0 && active) atomicAdd(a.small + kLoopSlotActive, (unsigned long long)active);
    }
}

}  // namespace swe
