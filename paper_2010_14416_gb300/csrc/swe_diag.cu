// swe_diag.cu -- diagnostics of a mesh's state (swe_diagnostics) and a
// steady-state driver (swe_run_to_steady).
//
// The paper computes inflow and outflow rates during its runs and copies
// them to the host on a side stream (Section 5.3.2), and it first runs to a
// stabilised solution before the production runs (Section 6.3.2).  Here:
//   - cell reductions (stored volume, largest depth change over the last step,
//     largest depth and speed, wet cells) in per-block partials on a fixed
//     grid, summed by one block: deterministic;
//   - the outward discharge through each boundary group, evaluated with the
//     step kernel's own boundary flux on the current state (the mass that
//     leaves through those edges in the next step per unit time), one value
//     per boundary edge, summed per group on the host in a fixed order.
// Interior fluxes cancel, so volume^{n+1} - volume^n = -dt_n * sum of the
// discharges evaluated on U^n.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "swe_internal.h"

using namespace swe;

namespace {

constexpr int kDiagBlock = 256;
constexpr int kDiagMaxBlocks = 1024;
constexpr int kDiagWords = 5;  // volume, dh_max, h_max, speed_max, n_wet

template <typename T>
__global__ void __launch_bounds__(kDiagBlock)
diag_cells_kernel(const V4<T>* __restrict__ cur, const V4<T>* __restrict__ prev, const V4<T>* __restrict__ geoB,
                  long long n, double h_dry, int have_prev, double* __restrict__ partial) {
    double vol = 0.0, dh = 0.0, hmax = 0.0, spd = 0.0, wet = 0.0;
    for (long long i = (long long)blockIdx.x * kDiagBlock + threadIdx.x; i < n; i += (long long)gridDim.x * kDiagBlock) {
        const V4<T> c = cur[i];
        const double h = (double)c.x;
        vol += h / (double)geoB[i].z;
        if (have_prev) dh = fmax(dh, fabs(h - (double)prev[i].x));
        hmax = fmax(hmax, h);
        if (h > h_dry) {
            wet += 1.0;
            const double u = (double)c.y / h, v = (double)c.z / h;
            spd = fmax(spd, sqrt(u * u + v * v));
        }
    }
    __shared__ double red[kDiagWords][kDiagBlock];
    red[0][threadIdx.x] = vol; red[1][threadIdx.x] = dh; red[2][threadIdx.x] = hmax;
    red[3][threadIdx.x] = spd; red[4][threadIdx.x] = wet;
    __syncthreads();
    for (int s = kDiagBlock / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[0][threadIdx.x] += red[0][threadIdx.x + s];
            red[1][threadIdx.x] = fmax(red[1][threadIdx.x], red[1][threadIdx.x + s]);
            red[2][threadIdx.x] = fmax(red[2][threadIdx.x], red[2][threadIdx.x + s]);
            red[3][threadIdx.x] = fmax(red[3][threadIdx.x], red[3][threadIdx.x + s]);
            red[4][threadIdx.x] += red[4][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x < kDiagWords) partial[blockIdx.x * kDiagWords + threadIdx.x] = red[threadIdx.x][0];
}

// The blocks' partials (one per thread, kDiagMaxBlocks threads) reduced in a
// fixed tree.  One thread adding them in turn took 0.1 ms for 400 blocks: a
// chain of dependent FP64 sums with a load in each link.
__global__ void __launch_bounds__(kDiagMaxBlocks) diag_final_kernel(const double* __restrict__ partial, int nb,
                                                                     double* __restrict__ out) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    double v[kDiagWords];
#pragma unroll
    for (int w = 0; w < kDiagWords; ++w) v[w] = t < nb ? partial[t * kDiagWords + w] : 0.0;
    __shared__ double red[kDiagWords][kDiagMaxBlocks / 32];
    auto fold = [&]() {
        for (int o = 16; o > 0; o >>= 1) {
            v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
            v[1] = fmax(v[1], __shfl_down_sync(0xffffffffu, v[1], o));
            v[2] = fmax(v[2], __shfl_down_sync(0xffffffffu, v[2], o));
            v[3] = fmax(v[3], __shfl_down_sync(0xffffffffu, v[3], o));
            v[4] += __shfl_down_sync(0xffffffffu, v[4], o);
        }
    };
    fold();
    if (lane == 0)
        for (int w = 0; w < kDiagWords; ++w) red[w][warp] = v[w];
    __syncthreads();
    if (warp == 0) {
        for (int w = 0; w < kDiagWords; ++w) v[w] = red[w][lane];
        fold();
        if (lane == 0)
            for (int w = 0; w < kDiagWords; ++w) out[w] = v[w];
    }
}

// Largest depth change over the last step: what run_to_steady tests between
// its runs of steps.  Depth differences are non-negative doubles, which order
// like their bits.
template <typename T>
__global__ void __launch_bounds__(kDiagBlock)
diag_change_kernel(const V4<T>* __restrict__ cur, const V4<T>* __restrict__ prev, long long n,
                   unsigned long long* __restrict__ out) {
    double dh = 0.0;
    for (long long i = (long long)blockIdx.x * kDiagBlock + threadIdx.x; i < n; i += (long long)gridDim.x * kDiagBlock)
        dh = fmax(dh, fabs((double)cur[i].x - (double)prev[i].x));
    for (int o = 16; o > 0; o >>= 1) dh = fmax(dh, __shfl_xor_sync(0xffffffffu, dh, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(dh));
}

// one boundary edge per thread: L * (outward mass flux) with the step's
// boundary treatment (Section 3.1)
template <typename T>
__global__ void diag_boundary_kernel(const V4<T>* __restrict__ cur, const V4<T>* __restrict__ geoA,
                                     const V4<T>* __restrict__ geoB, const V4<T>* __restrict__ geoR,
                                     const long long* __restrict__ slots,
                                     const int* __restrict__ groups, long long nb, BcTable bc, T g, T h_dry,
                                     int hll, double* __restrict__ q) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nb) return;
    const long long s = slots[k];
    const long long i = s / 3;
    const int j = (int)(s % 3);
    const V4<T> c = cur[i];
    const V4<T> gA = geoA[i], gB = geoB[i];
    const T lx = j == 0 ? gA.x : (j == 1 ? gA.z : gB.x);
    const T ly = j == 0 ? gA.y : (j == 1 ? gA.w : gB.y);
    T len, n1, n2;   // the step's own
    if constexpr (sizeof(T) == 8) {
        const V4<T> gR = geoR[i];
        len = j == 0 ? gR.x : (j == 1 ? gR.y : gR.z);
        n1 = lx;
        n2 = ly;
    } else {
        const T l2 = edge_l2(lx, ly);
        const T rl = rsqrtf(l2);
        len = l2 * rl;
        n1 = lx * rl;
        n2 = ly * rl;
    }
    T ui, vi;
    cell_velocity<T>(c.x, c.y, c.z, h_dry, ui, vi);
    const int grp = groups[k];
    T F0, F1, F2;
    edge_boundary<T>(bc.kind[grp], bc.value[grp], c.x, ui, vi, c.w, n1, n2, g, h_dry, F0, F1, F2, hll != 0);
    q[k] = (double)len * (double)F0;
}

int dfail(cudaError_t e, const char* what) {
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return SWE_ECUDA;
}

struct DiagDeviceGuard {
    int prev = -1;
    explicit DiagDeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DiagDeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

// The mesh's diagnostics workspace: device words [results | status block | q of
// the boundary edges], their pinned host copy, and the boundary edges (slot,
// group) in a fixed order.  Laid out on the first call; a change of boundary
// groups renews the groups.
int diag_workspace(swe_mesh* m) {
    if (m->diag_dev) {
        if (!m->diag_groups_old) return SWE_OK;
        const size_t nb = m->diag_edge_group.size();
        for (size_t k = 0; k < nb; ++k) m->diag_edge_group[k] = -1 - m->hm.code[m->diag_edge[k]];
        if (nb) {
            const cudaError_t e = cudaMemcpyAsync(m->diag_groups, m->diag_edge_group.data(), nb * sizeof(int),
                                                  cudaMemcpyHostToDevice, m->stream);
            if (e != cudaSuccess) return dfail(e, "swe_diagnostics: boundary groups");
        }
        m->diag_groups_old = false;
        return SWE_OK;
    }
    std::vector<long long> slots;
    std::vector<int> groups;
    try {
        for (int64_t s = 0; s < 3 * m->hm.n_cells; ++s)   // (internal cell, local edge)
            if (m->hm.code[s] < 0) {
                slots.push_back(s);
                groups.push_back(-1 - m->hm.code[s]);
            }
    } catch (const std::bad_alloc&) {
        set_error("swe_diagnostics: out of host memory");
        return SWE_ENOMEM;
    }
    const size_t nb = slots.size(), words = kDiagWords + kSmallWords + nb;
    cudaError_t e = cudaMalloc((void**)&m->diag_dev, words * sizeof(double));
    if (e == cudaSuccess) e = cudaMallocHost((void**)&m->diag_host, words * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->diag_partial, kDiagMaxBlocks * kDiagWords * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->diag_slots, std::max<size_t>(nb, 1) * sizeof(long long));
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->diag_groups, std::max<size_t>(nb, 1) * sizeof(int));
    if (e == cudaSuccess && nb)
        e = cudaMemcpyAsync(m->diag_slots, slots.data(), nb * sizeof(long long), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess && nb)
        e = cudaMemcpyAsync(m->diag_groups, groups.data(), nb * sizeof(int), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) {
        drop_diag_workspace(m);
        return dfail(e, "swe_diagnostics: workspace");
    }
    m->diag_edge_group.swap(groups);
    m->diag_edge.swap(slots);
    m->diag_groups_old = false;
    m->diag_bytes = (int64_t)(words * sizeof(double) + kDiagMaxBlocks * kDiagWords * sizeof(double) +
                              std::max<size_t>(nb, 1) * (sizeof(long long) + sizeof(int)));
    m->device_bytes += m->diag_bytes;
    return SWE_OK;
}

template <typename T>
int diagnostics_t(swe_mesh* m, swe_diag* out) {
    const int64_t n = m->hm.n_cells;
    cudaStream_t st = m->stream;
    int rc = diag_workspace(m);
    if (rc) return rc;
    const long long nb = (long long)m->diag_edge_group.size();
    const int nblk = (int)std::min<long long>(kDiagMaxBlocks, (n + kDiagBlock - 1) / kDiagBlock);
    double* const dq = m->diag_dev + kDiagWords + kSmallWords;
    const V4<T>* cur = (const V4<T>*)m->state[m->nstep % 2];
    const V4<T>* prev = (const V4<T>*)m->state[(m->nstep + 1) % 2];
    diag_cells_kernel<T><<<nblk, kDiagBlock, 0, st>>>(cur, prev, (const V4<T>*)m->geoB, n, m->cfg.h_dry,
                                                     m->nstep > 0 ? 1 : 0, m->diag_partial);
    diag_final_kernel<<<1, kDiagMaxBlocks, 0, st>>>(m->diag_partial, nblk, m->diag_dev);
    if (nb)
        diag_boundary_kernel<T><<<(unsigned)((nb + 255) / 256), 256, 0, st>>>(
            cur, (const V4<T>*)m->geoA, (const V4<T>*)m->geoB, (const V4<T>*)m->geoR, m->diag_slots, m->diag_groups,
            nb, m->bc, (T)m->cfg.g, (T)m->cfg.h_dry, m->cfg.flux == SWE_FLUX_HLL ? 1 : 0, dq);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->diag_dev + kDiagWords, m->small, kSmallWords * sizeof(double), cudaMemcpyDeviceToDevice,
                            st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->diag_host, m->diag_dev, (kDiagWords + kSmallWords + nb) * sizeof(double),
                            cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return dfail(e, "swe_diagnostics");
    const double *r = m->diag_host, *sm = r + kDiagWords, *q = sm + kSmallWords;
    std::memset(out, 0, sizeof *out);
    out->volume = r[0];
    out->dh_max = r[1];
    out->h_max = r[2];
    out->speed_max = r[3];
    out->n_wet = (int64_t)r[4];
    out->n_groups = m->n_groups;
    for (long long k = 0; k < nb; ++k) out->discharge[m->diag_edge_group[k]] += q[k];
    std::memcpy(&out->t, &sm[kSlotT], sizeof(double));
    if (m->nstep > 0) std::memcpy(&out->dt_last, &sm[kSlotDtLast], sizeof(double));
    return SWE_OK;
}

// The status block after the steps in flight, and the largest depth change of
// the last one.
int steady_check(swe_mesh* m, double* dh_max, unsigned long long status[kSmallWords]) {
    int rc = diag_workspace(m);
    if (rc) return rc;
    const int64_t n = m->hm.n_cells;
    cudaStream_t st = m->stream;
    const int nblk = (int)std::min<long long>(kDiagMaxBlocks, (n + kDiagBlock - 1) / kDiagBlock);
    cudaError_t e = cudaMemsetAsync(m->diag_dev + kDiagWords - 1, 0, sizeof(double), st);
    if (e == cudaSuccess) {
        const void *cur = m->state[m->nstep % 2], *prev = m->state[(m->nstep + 1) % 2];
        unsigned long long* out = (unsigned long long*)(m->diag_dev + kDiagWords - 1);   // beside the status block
        if (m->cfg.precision == SWE_FP32)
            diag_change_kernel<float><<<nblk, kDiagBlock, 0, st>>>((const V4<float>*)cur, (const V4<float>*)prev, n,
                                                                  out);
        else
            diag_change_kernel<double><<<nblk, kDiagBlock, 0, st>>>((const V4<double>*)cur, (const V4<double>*)prev, n,
                                                                   out);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->diag_dev + kDiagWords, m->small, kSmallWords * sizeof(double), cudaMemcpyDeviceToDevice,
                            st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->diag_host, m->diag_dev + kDiagWords - 1, (1 + kSmallWords) * sizeof(double),
                            cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return dfail(e, "swe_run_to_steady");
    *dh_max = m->diag_host[0];
    std::memcpy(status, m->diag_host + 1, kSmallWords * sizeof(unsigned long long));
    return SWE_OK;
}

}  // namespace

namespace swe {

void drop_diag_workspace(swe_mesh* m) {
    for (void* p : {(void*)m->diag_dev, (void*)m->diag_partial, (void*)m->diag_slots, (void*)m->diag_groups})
        if (p) cudaFree(p);
    if (m->diag_host) cudaFreeHost(m->diag_host);
    m->diag_dev = m->diag_partial = m->diag_host = nullptr;
    m->diag_slots = nullptr;
    m->diag_groups = nullptr;
    m->diag_edge_group.clear();
    m->diag_edge.clear();
    m->device_bytes -= m->diag_bytes;
    m->diag_bytes = 0;
}

}  // namespace swe

extern "C" {

int swe_diagnostics(swe_mesh* m, swe_diag* out) {
    if (!m || !out) { set_error("swe_diagnostics: bad arguments"); return SWE_EINVAL; }
    if (!m->have_state) { set_error("swe_diagnostics: no state set"); return SWE_EINVAL; }
    DiagDeviceGuard dg(m->cfg.device);
    int rc = flush_mesh_bc(m);
    if (rc) return rc;
    return m->cfg.precision == SWE_FP32 ? diagnostics_t<float>(m, out) : diagnostics_t<double>(m, out);
}

int swe_run_to_steady(swe_mesh* m, double cfl, double tol, int64_t check_every, int64_t max_steps,
                      int64_t* steps_done, int* converged, double* t_out) {
    NvtxRange nvtx_range("swe_run_to_steady");
    if (!m || !(tol > 0.0) || check_every < 1 || max_steps < 0) {
        set_error("swe_run_to_steady: bad arguments");
        return SWE_EINVAL;
    }
    int64_t done = 0;
    int conv = 0;
    DiagDeviceGuard dg(m->cfg.device);
    while (done < max_steps) {
        const int64_t k = std::min(check_every, max_steps - done);
        int rc = swe_step(m, k, cfl, nullptr);
        if (rc) return rc;
        // one wait for the steps' status and their last depth change
        double dh_max = 0.0, dt_last = 0.0;
        unsigned long long sm[kSmallWords];
        rc = steady_check(m, &dh_max, sm);
        if (rc) return rc;
        rc = status_code(sm[kSlotStatus]);
        if (rc) return rc;
        done += k;
        std::memcpy(&dt_last, &sm[kSlotDtLast], sizeof(double));
        if (dt_last > 0.0 && dh_max / dt_last < tol) { conv = 1; break; }
    }
    if (steps_done) *steps_done = done;
    if (converged) *converged = conv;
    if (t_out) {
        swe_info info;
        int rc = swe_get_info(m, &info);
        if (rc) return rc;
        *t_out = info.t;
    }
    return SWE_OK;
}

}  // extern "C"
