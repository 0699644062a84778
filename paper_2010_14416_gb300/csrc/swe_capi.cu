// swe_capi.cu -- the C ABI of libswe (declared in include/swe.h).
//
// Device layout of one mesh (n cells, precision T, internal locality order):
//   state[2]  V4<T>[n]   (h, hu, hv, z) ping-pong pair
//   geoA      V4<T>[n]   L n of edges 0 and 1 (FP64: n)
//   geoB      V4<T>[n]   L n of edge 2 (FP64: n), 1/|Omega|, inscribed radius
//   geoR      V4<T>[n]   FP64: L of the three edges
//   topo      int4[n]    neighbour codes
//   gm2       T[n]       g m^2
//   perm, inv u32[n]     internal -> caller index and back
//   small     u64[8]     dt slots 0..2 (double bits), t, status, clamp count
// Step n reads state[n % 2] and dt slot n % 3, writes state[(n+1) % 2] and
// slot (n+1) % 3, and clears slot (n+2) % 3, so a graph of a multiple of six
// steps replays from any step index that is a multiple of six.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "swe_internal.h"
#include "swe_loop.cuh"

namespace swe {

static thread_local std::string g_last_error;
void set_error(const std::string& msg) { g_last_error = msg; }

namespace {

constexpr int kDefaultGraphSteps = 48;
constexpr int64_t kListCells = 800000;   // FP32 activity steps over a list (list_activity)

struct DeviceGuard {
    int prev = -1;
    bool ok = true;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) ok = cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

int cuda_fail(cudaError_t e, const char* what) {
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return SWE_ECUDA;
}

__global__ void init_small_kernel(unsigned long long* small, double t) {
    if (threadIdx.x == 0) {
        small[0] = kInfBits; small[1] = kInfBits; small[2] = kInfBits;
        small[kSlotT] = (unsigned long long)__double_as_longlong(t);
        small[kSlotStatus] = 0ULL;
        small[kSlotClamp] = 0ULL;
        small[6] = 0ULL; small[7] = 0ULL;
        small[kSmallWords] = 0ULL;   // wet cells (set_state)
    }
}

}  // namespace
}  // namespace swe

using namespace swe;

int swe::status_code(unsigned long long st) {
    if (st & kStatusBadIndex) {
        set_error("swe_step: a neighbour index, edge index or boundary group out of range (debug checks)");
        return SWE_EMESH;
    }
    if (st & kStatusStall) { set_error("swe_step: the step loop gave up waiting for its blocks"); return SWE_ETIMEOUT; }
    if (st & kStatusNonFinite) { set_error("swe_step: non-finite state"); return SWE_ENONFINITE; }
    if (st & kStatusDry) { set_error("swe_step: every cell is dry, no CFL time step"); return SWE_EDRY; }
    return SWE_OK;
}

namespace {

int dev_alloc(swe_mesh* m, void** p, size_t bytes, const char* what) {
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
        *p = nullptr;
        set_error(std::string("device allocation failed for ") + what + ": " + cudaGetErrorString(e));
        return SWE_ENOMEM;
    }
    m->device_bytes += (int64_t)bytes;
    return SWE_OK;
}

void drop_graph(swe_mesh* m) {
    if (m->graph) cudaGraphExecDestroy(m->graph);
    m->graph = nullptr;
    m->graph_len = 0;
    m->graph_cfl = -1.0;
}

// topo[c] = (neighbour codes, and for FP32 the bits of g m^2 in .w)
std::vector<int4> make_topo(const swe_mesh* m) {
    const HostMesh& H = m->hm;
    const int64_t n = H.n_cells;
    std::vector<int4> topo(n);
    for (int64_t c = 0; c < n; ++c) {
        int w = 0;
        if (m->esz == 4) {
            const float gm2 = (float)(m->cfg.g * H.m[c] * H.m[c]);
            std::memcpy(&w, &gm2, sizeof w);
        }
        // static activity: an inflow or fixed-stage edge keeps the cell out of the quiet path
        bool fixed = false;
        for (int j = 0; j < 3; ++j) {
            const int32_t code = H.code[3 * c + j];
            if (code < 0) {
                const int kind = m->bc.kind[-1 - code];
                fixed = fixed || kind == kBcInflow || kind == kBcStage;
            }
        }
        if (fixed) w |= kStaticBit;
        topo[c] = make_int4(H.code[3 * c], H.code[3 * c + 1], H.code[3 * c + 2], w);
    }
    return topo;
}

template <typename T>
int upload_static(swe_mesh* m) {
    const HostMesh& H = m->hm;
    const int64_t n = H.n_cells;
    std::vector<V4<T>> A(n), B(n), R(sizeof(T) == 8 ? n : 0);
    std::vector<T> gm2(n), zt(n);
    std::vector<unsigned> perm(n), inv(n);
    const std::vector<int4> topo = make_topo(m);
    for (int64_t c = 0; c < n; ++c) {
        double ln[6];
        std::memcpy(ln, &H.ln[6 * c], sizeof ln);
        if (sizeof(T) == 8) {
            R[c].x = (T)host_unit_normal(ln[0], ln[1]);
            R[c].y = (T)host_unit_normal(ln[2], ln[3]);
            R[c].z = (T)host_unit_normal(ln[4], ln[5]);
            R[c].w = (T)0;
        }
        A[c].x = (T)ln[0]; A[c].y = (T)ln[1];
        A[c].z = (T)ln[2]; A[c].w = (T)ln[3];
        B[c].x = (T)ln[4]; B[c].y = (T)ln[5];
        B[c].z = (T)H.inv_area[c]; B[c].w = (T)H.rin[c];
        gm2[c] = (T)(m->cfg.g * H.m[c] * H.m[c]);
        zt[c] = (T)H.z[c];
        perm[c] = (unsigned)H.perm[c];
        inv[H.perm[c]] = (unsigned)c;
    }
    cudaError_t e;
    if ((e = cudaMemcpy(m->geoA, A.data(), n * sizeof(V4<T>), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(m->geoB, B.data(), n * sizeof(V4<T>), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (sizeof(T) == 8 &&
         (e = cudaMemcpy(m->geoR, R.data(), n * sizeof(V4<T>), cudaMemcpyHostToDevice)) != cudaSuccess) ||
        (e = cudaMemcpy(m->gm2, gm2.data(), n * sizeof(T), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(m->zdev, zt.data(), n * sizeof(T), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(m->topo, topo.data(), n * sizeof(int4), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(m->perm, perm.data(), n * sizeof(unsigned), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemcpy(m->inv, inv.data(), n * sizeof(unsigned), cudaMemcpyHostToDevice)) != cudaSuccess)
        return cuda_fail(e, "swe_mesh_create: upload");
    return SWE_OK;
}

int flush_topo(swe_mesh* m) {
    if (!m->topo_dirty) return SWE_OK;
    const int64_t n = m->hm.n_cells;
    const std::vector<int4> topo = make_topo(m);
    cudaError_t e = cudaMemcpyAsync(m->topo, topo.data(), n * sizeof(int4), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "swe_set_bc: upload");
    for (int gI = 0; gI < m->n_groups; ++gI) {
        if (m->bc.kind[gI] == kBcInflow)
            m->bc.value[gI] = m->group_len[gI] > 0.0 ? m->group_value[gI] / m->group_len[gI] : 0.0;
        else
            m->bc.value[gI] = m->group_value[gI];
    }
    m->topo_dirty = false;
    m->act_valid = false;   // static activity may have changed
    m->diag_groups_old = true;
    drop_graph(m);
    return SWE_OK;
}

template <typename T>
StepArgs<T> make_args(swe_mesh* m, int64_t step_index, double cfl) {
    StepArgs<T> a;
    const int p2 = (int)(step_index % 2), p3 = (int)(step_index % 3);
    a.s_in = (const V4<T>*)m->state[p2];
    a.s_out = (V4<T>*)m->state[1 - p2];
    a.geoA = (const V4<T>*)m->geoA;
    a.geoB = (const V4<T>*)m->geoB;
    a.geoR = (const V4<T>*)m->geoR;
    a.topo = m->topo;
    a.gm2 = (const T*)m->gm2;
    a.dt_read = (const double*)(m->small + p3);
    a.dt_write = m->small + (p3 + 1) % 3;
    a.dt_reset = m->small + (p3 + 2) % 3;
    a.t = (double*)(m->small + kSlotT);
    a.status = (unsigned*)(m->small + kSlotStatus);
    a.n_clamped = m->small + kSlotClamp;
    a.n_active = m->small + kSlotActive;
    a.n = m->hm.n_cells;
    a.grid = m->grid;
    a.cfl = cfl;
    a.hll = m->cfg.flux == SWE_FLUX_HLL ? 1 : 0;
    a.dt_fixed = nullptr;
    a.dt_log = (double*)(m->small + kSlotDtLast);  // size of the last step, for diagnostics
    a.ecells = nullptr;
    a.eln = nullptr;
    a.erl = (const T*)m->erl;
    a.eflux = nullptr;
    a.esrc = nullptr;
    a.eidx = nullptr;
    a.n_edges = 0;
    if (m->cfg.edge_pass && m->eflux) {
        a.ecells = m->ecells;
        a.eln = (const T*)m->eln;
        a.eflux = (V4<T>*)m->eflux;
        a.esrc = (T*)m->esrc;
        a.eidx = m->eidx;
        a.n_edges = m->n_edges;
    }
    a.act_in = nullptr;
    a.act_next = nullptr;
    a.act_clear = nullptr;
    a.span_in = nullptr;
    a.span_next = nullptr;
    a.span_clear = nullptr;
    a.span_first = m->span_first;
    a.span_adj = m->span_adj;
    a.act_list = m->act_by_list ? m->act_list : nullptr;
    a.act_count = m->act_count;
    if (m->cfg.activity && m->act[0]) {
        a.act_in = m->act[p3];
        a.act_next = m->act[(p3 + 1) % 3];
        a.act_clear = m->act[(p3 + 2) % 3];
        // the flags lie behind the bytes
        a.span_in = a.act_in + m->act_len;
        a.span_next = a.act_next + m->act_len;
        a.span_clear = a.act_clear + m->act_len;
    }
    a.g = (T)m->cfg.g;
    a.h_dry = (T)m->cfg.h_dry;
    a.bc = m->bc;
    a.debug = m->cfg.debug_checks;
    a.n_groups = m->n_groups;
    return a;
}

template <typename T>
cudaError_t launch_one(swe_mesh* m, int64_t step_index, double cfl, cudaStream_t st) {
    if (m->cfg.cell_pairs)
        return Launch<T>::step_pair(make_args<T>(m, step_index, cfl), m->cfg.block_size, m->cfg.min_blocks,
                                    m->cfg.geometry_early, m->cfg.stages, st);
    return Launch<T>::step(make_args<T>(m, step_index, cfl), m->cfg.block_size, m->cfg.min_blocks,
                           m->cfg.stages, m->cfg.geometry_early, st);
}

template <typename T>
int capture_graph(swe_mesh* m, int len, double cfl) {
    drop_graph(m);
    cudaError_t e = cudaStreamBeginCapture(m->cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(e, "swe_step: begin capture");
    cudaError_t le = cudaSuccess;
    for (int s = 0; s < len && le == cudaSuccess; ++s) le = launch_one<T>(m, s, cfl, m->cap_stream);
    cudaGraph_t gr = nullptr;
    e = cudaStreamEndCapture(m->cap_stream, &gr);
    if (le != cudaSuccess) { if (gr) cudaGraphDestroy(gr); return cuda_fail(le, "swe_step: capture launch"); }
    if (e != cudaSuccess) return cuda_fail(e, "swe_step: end capture");
    e = cudaGraphInstantiate(&m->graph, gr, 0);
    cudaGraphDestroy(gr);
    if (e != cudaSuccess) { m->graph = nullptr; return cuda_fail(e, "swe_step: instantiate"); }
    m->graph_len = len;
    m->graph_cfl = cfl;
    return SWE_OK;
}

static_assert(kLoopSlotT == kSlotT && kLoopSlotStatus == kSlotStatus && kLoopSlotClamp == kSlotClamp &&
                  kLoopSlotActive == kSlotActive && kLoopSlotDtLast == kSlotDtLast,
              "words of the status block");

// The edges that touch each block's cells, for the FP64 step loop.
int build_loop_edges(swe_mesh* m) {
    const HostMesh& H = m->hm;
    const int64_t n = H.n_cells, nb = (n + kLoopCells - 1) / kLoopCells;
    std::vector<int2> ecell(nb * kLoopEdges, make_int2(-1, -1));
    std::vector<double> egeo(nb * 2 * kLoopEdges, 0.0);
    std::vector<uchar4> eslot(n, make_uchar4(0, 0, 0, 0));
    auto slot = [&](int64_t c, int j) -> unsigned char& { return j == 0 ? eslot[c].x : (j == 1 ? eslot[c].y : eslot[c].z); };
    for (int64_t b = 0; b < nb; ++b) {
        const int64_t c0 = b * kLoopCells, c1 = std::min(n, c0 + kLoopCells);
        int ne = 0;
        for (int64_t c = c0; c < c1; ++c)
            for (int j = 0; j < 3; ++j) {
                const int32_t code = H.code[3 * c + j];
                if (code < 0) continue;
                const int64_t k = code & kNbrMask;
                if (k >= c0 && k < c) {   // listed from k already
                    for (int jk = 0; jk < 3; ++jk)
                        if (H.code[3 * k + jk] >= 0 && (H.code[3 * k + jk] & kNbrMask) == c) slot(c, j) = slot(k, jk);
                    continue;
                }
                const bool flip = (code & kFlipBit) != 0;
                double lx = H.ln[6 * c + 2 * j], ly = H.ln[6 * c + 2 * j + 1];
                (void)host_unit_normal(lx, ly);
                ecell[b * kLoopEdges + ne] = flip ? make_int2((int)k, (int)c) : make_int2((int)c, (int)k);
                double* g = &egeo[b * 2 * kLoopEdges + ne];
                g[0] = flip ? -lx : lx;
                g[kLoopEdges] = flip ? -ly : ly;
                slot(c, j) = (unsigned char)ne++;
            }
    }
    cudaError_t e = cudaMalloc((void**)&m->loop_ecell, ecell.size() * sizeof(int2));
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->loop_egeo, egeo.size() * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->loop_eslot, eslot.size() * sizeof(uchar4));
    if (e == cudaSuccess) e = cudaMemcpy(m->loop_ecell, ecell.data(), ecell.size() * sizeof(int2), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->loop_egeo, egeo.data(), egeo.size() * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->loop_eslot, eslot.data(), eslot.size() * sizeof(uchar4), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        for (void* p : {(void*)m->loop_ecell, (void*)m->loop_egeo, (void*)m->loop_eslot})
            if (p) cudaFree(p);
        m->loop_ecell = nullptr;
        m->loop_egeo = nullptr;
        m->loop_eslot = nullptr;
        return cuda_fail(e, "swe_step: step loop");
    }
    m->device_bytes += (int64_t)(ecell.size() * sizeof(int2) + egeo.size() * sizeof(double) + eslot.size() * sizeof(uchar4));
    return SWE_OK;
}

// Whether the next steps run as one loop launch: a small mesh, nothing chosen
// about its launches, no debug checks and no capture of the stream (a
// cooperative launch is not for every graph).  From 4 steps on: the loop's
// launch and first reads cost about what two step launches do.  FP32 meshes of
// more than four of the six blocks an SM holds take it for calls shorter than a
// graph only: more blocks meet more slowly, and a replayed graph has no gaps
// between its launches (us a step of a half wet canal, loop against graph: 60,000
// cells 4.4 and 4.7, 80,000 5.4 and 5.2, 112,000 6.7 and 5.5; of calls of 20
// steps, against single launches, 5.1 and 6.9, 5.7 and 6.9, 6.9 and 7.1).
template <typename T>
bool use_loop(swe_mesh* m, int64_t nsteps) {
    const bool graphs = nsteps >= m->cfg.graph_steps;
    const int tuned = graphs ? m->loop_long : m->loop_short;
    if (!m->loop_allowed || nsteps < 4 || tuned == 0) return false;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(m->stream, &cs) != cudaSuccess) { (void)cudaGetLastError(); return false; }
    if (cs != cudaStreamCaptureStatusNone) return false;
    if (m->loop_cells < 0) {
        long long cells = m->loop_cells_set;
        if (cells < 0 && Launch<T>::loop_capacity(m->cfg.device, &cells) != cudaSuccess) {
            (void)cudaGetLastError();
            cells = 0;
        }
        m->loop_cells = cells;
        if (m->hm.n_cells <= cells && !m->loop_barrier) {
            bool ok = cudaMalloc((void**)&m->loop_barrier, sizeof(unsigned)) == cudaSuccess;
            try {
                if (ok && sizeof(T) == 8) ok = build_loop_edges(m) == SWE_OK;
            } catch (const std::bad_alloc&) {
                ok = false;
            }
            if (ok) {
                m->device_bytes += sizeof(unsigned);
            } else {   // the steps are launched one by one, then
                (void)cudaGetLastError();
                if (m->loop_barrier) cudaFree(m->loop_barrier);
                m->loop_barrier = nullptr;
                m->loop_allowed = false;
                return false;
            }
        }
    }
    const bool fewer = sizeof(T) == 4 && graphs && tuned < 0;
    return m->hm.n_cells <= (fewer ? m->loop_cells / 3 * 2 : m->loop_cells);
}

// Runs nsteps steps in the loop; on return nsteps is what is left of them.  Where
// the launch is refused (fewer SMs open to the stream than the device has, as
// under a green context), this mesh goes on without the loop.
template <typename T>
void run_loop(swe_mesh* m, int64_t& nsteps, double cfl) {
    LoopArgs<T> a;
    a.state[0] = (V4<T>*)m->state[0];
    a.state[1] = (V4<T>*)m->state[1];
    a.geoA = (const V4<T>*)m->geoA;
    a.geoB = (const V4<T>*)m->geoB;
    a.geoR = (const V4<T>*)m->geoR;
    a.topo = m->topo;
    a.gm2 = (const T*)m->gm2;
    a.small = m->small;
    a.barrier = m->loop_barrier;
    a.n = m->hm.n_cells;
    a.cfl = cfl;
    a.g = (T)m->cfg.g;
    a.h_dry = (T)m->cfg.h_dry;
    a.hll = m->cfg.flux == SWE_FLUX_HLL ? 1 : 0;
    a.debug = 0;
    a.n_groups = m->n_groups;
    a.bc = m->bc;
    a.ecell = m->loop_ecell;
    a.egeo = m->loop_egeo;
    a.eslot = m->loop_eslot;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->cfg.device) != cudaSuccess) sms = 0;
    a.one_block_sms = a.n <= (long long)sms * kLoopCells;
    m->act_valid = false;   // steps without activity bytes do not maintain them
    while (nsteps > 0) {
        a.step0 = m->nstep;
        a.steps = (int)std::min<int64_t>(nsteps, 2000);   // some milliseconds a launch
        a.max_polls = m->loop_polls;
        if (Launch<T>::loop(a, m->stream) != cudaSuccess) {
            (void)cudaGetLastError();
            m->loop_allowed = false;
            return;
        }
        m->nstep += a.steps;
        m->loop_steps += a.steps;
        nsteps -= a.steps;
    }
}

// Whether the activity steps of m run over a list of the active cells (two
// launches) or, FP32, through all cells (one).  The list costs 5 us a step and
// 6 ps for each active cell more and saves 5 ps for each quiet one, more where
// the active cells lie unevenly among the blocks: of n cells with a share s
// active it pays from n (1 - 2.2 s) = 550,000 (a winding channel) to 1.3M (one
// wet end) on; the line is at 800,000 (a tenth less before a mesh on the list
// leaves it).  us a step, list and all cells: a half
// wet canal of 200,000 cells 11.7 and 6.9, of 1.2M 24.1 and 20.8; a canal 10 %
// wet of 1.2M 12.2 and 10.6, of 2.5M 19.5 and 22.3; a reach 6 % wet of 300,000
// 9.4 and 8.3, of 1.2M 10.4 and 15.4, of 6M 24.2 and 47.4; 6M cells 30 % wet 65.9
// and 70.6, 50 % 101.5 and 96.5, all wet 189.5 and 158.2.  The autotuner times
// the list's shapes (through all cells no shape came first), and a shape of
// them that it keeps stays on the list.
bool list_activity(const swe_mesh* m) {
    if (m->cfg.precision != SWE_FP32 || m->act_tuned || m->list_cells == 0) return true;
    return (double)m->hm.n_cells * (1.0 - 2.2 * m->act_share) > (double)m->list_cells * (m->act_by_list ? 0.9 : 1.0);
}

// The activity bytes for the next steps of m, rebuilt where they are not those
// of its state or where the other kernel is to maintain them.
int prepare_activity(swe_mesh* m) {
    if (list_activity(m) != m->act_by_list) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(m->stream, &cs) != cudaSuccess) (void)cudaGetLastError();
        if (cs == cudaStreamCaptureStatusNone) {
            m->act_by_list = !m->act_by_list;
            m->act_valid = false;
            drop_graph(m);
        }
    }
    return m->act_valid ? SWE_OK : init_activity(m);
}

template <typename T>
int run_steps(swe_mesh* m, int64_t nsteps, double cfl) {
    if (use_loop<T>(m, nsteps)) {
        run_loop<T>(m, nsteps, cfl);
        if (nsteps == 0) return SWE_OK;
    }
    if (m->cfg.activity) {
        const int rc = prepare_activity(m);
        if (rc) return rc;
    } else {
        m->act_valid = false;   // steps without activity bytes do not maintain them
    }
    int64_t left = nsteps;
    const int gsteps = m->cfg.graph_steps;
    // singles until the step index is a multiple of six
    while (left > 0 && (m->nstep % 6 != 0 || gsteps <= 0 || left < gsteps)) {
        cudaError_t e = launch_one<T>(m, m->nstep, cfl, m->stream);
        if (e != cudaSuccess) return cuda_fail(e, "swe_step: launch");
        ++m->nstep;
        --left;
        if (m->nstep % 6 == 0 && gsteps > 0 && left >= gsteps) break;
    }
    if (left >= gsteps && gsteps > 0) {
        if (!m->graph || m->graph_len != gsteps || m->graph_cfl != cfl) {
            int rc = capture_graph<T>(m, gsteps, cfl);
            if (rc) return rc;
        }
        while (left >= gsteps) {
            cudaError_t e = cudaGraphLaunch(m->graph, m->stream);
            if (e != cudaSuccess) return cuda_fail(e, "swe_step: graph launch");
            m->nstep += gsteps;
            left -= gsteps;
        }
    }
    while (left > 0) {
        cudaError_t e = launch_one<T>(m, m->nstep, cfl, m->stream);
        if (e != cudaSuccess) return cuda_fail(e, "swe_step: launch");
        ++m->nstep;
        --left;
    }
    return SWE_OK;
}

int read_small(swe_mesh* m, unsigned long long out[kSmallWords]) {
    cudaError_t e = cudaMemcpyAsync(out, m->small, sizeof(unsigned long long) * kSmallWords,
                                    cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "swe: reading the status block");
    if (m->nstep > m->act_seen_step && out[kSlotActive] >= m->act_seen)
        m->act_share = (double)(out[kSlotActive] - m->act_seen) /
                       ((double)(m->nstep - m->act_seen_step) * (double)m->hm.n_cells);
    m->act_seen = out[kSlotActive];
    m->act_seen_step = m->nstep;
    return SWE_OK;
}

double bits_to_double(unsigned long long b) {
    double d;
    std::memcpy(&d, &b, sizeof d);
    return d;
}

int ensure_stage(swe_mesh* m) {
    for (int k = 0; k < 3; ++k) {
        if (!m->stage[k]) {
            int rc = dev_alloc(m, &m->stage[k], m->hm.n_cells * m->esz, "staging");
            if (rc) return rc;
        }
    }
    return SWE_OK;
}

template <typename T>
int set_state_t(swe_mesh* m, const void* h, const void* hu, const void* hv, int where, double t) {
    const int64_t n = m->hm.n_cells;
    const T* src[3] = {(const T*)h, (const T*)hu, (const T*)hv};
    cudaError_t e;
    if (where == SWE_HOST) {
        int rc = ensure_stage(m);
        if (rc) return rc;
        for (int k = 0; k < 3; ++k) {
            e = cudaMemcpyAsync(m->stage[k], src[k], n * sizeof(T), cudaMemcpyHostToDevice, m->stream);
            if (e != cudaSuccess) return cuda_fail(e, "swe_set_state: copy");
            src[k] = (const T*)m->stage[k];
        }
    }
    // z rides in the state record (copied from the static z array)
    e = Launch<T>::pack(src[0], src[1], src[2], m->perm, (const T*)m->zdev, (V4<T>*)m->state[0], n, m->stream);
    // (the other buffer holds nothing that is read: a step writes every record,
    // with the activity bytes the first two after a set_state do)
    if (e == cudaSuccess) { init_small_kernel<<<1, 32, 0, m->stream>>>(m->small, t); e = cudaGetLastError(); }
    // list_activity asks how much of the mesh is wet
    unsigned long long wet = 0;
    unsigned long long* const n_wet =
        sizeof(T) == 4 && m->cfg.activity && n > m->list_cells ? m->small + kSmallWords : nullptr;
    if (e == cudaSuccess)
        e = Launch<T>::dt((const V4<T>*)m->state[0], (const V4<T>*)m->geoB, n, (T)m->cfg.g, (T)m->cfg.h_dry,
                          m->small + 0, n_wet, m->stream);
    if (e == cudaSuccess && n_wet) e = cudaMemcpyAsync(&wet, n_wet, sizeof wet, cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "swe_set_state");
    if (n_wet) m->act_share = (double)wet / (double)n;
    m->act_seen = 0;
    m->act_seen_step = 0;
    m->have_state = true;
    m->nstep = 0;
    m->act_valid = false;
    return SWE_OK;
}

template <typename T>
int get_state_t(swe_mesh* m, void* h, void* hu, void* hv, int where) {
    const int64_t n = m->hm.n_cells;
    const V4<T>* cur = (const V4<T>*)m->state[m->nstep % 2];
    cudaError_t e;
    if (where == SWE_DEVICE) {
        e = Launch<T>::unpack(cur, m->inv, (T*)h, (T*)hu, (T*)hv, n, m->stream);
        if (e != cudaSuccess) return cuda_fail(e, "swe_get_state");
        return SWE_OK;
    }
    int rc = ensure_stage(m);
    if (rc) return rc;
    e = Launch<T>::unpack(cur, m->inv, (T*)m->stage[0], (T*)m->stage[1], (T*)m->stage[2], n, m->stream);
    void* dst[3] = {h, hu, hv};
    for (int k = 0; k < 3 && e == cudaSuccess; ++k)
        e = cudaMemcpyAsync(dst[k], m->stage[k], n * sizeof(T), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "swe_get_state");
    return SWE_OK;
}

}  // namespace

namespace swe {

template <typename T>
cudaError_t launch_raw_t(swe_mesh* m, const void* in, void* out, unsigned long long* small, int64_t step_index,
                         double cfl, const double* dt_fixed, double* dt_log, cudaStream_t st, bool with_activity,
                         void* eflux_out, void* esrc_out) {
    StepArgs<T> a = make_args<T>(m, step_index, cfl);
    a.s_in = (const V4<T>*)in;
    a.s_out = (V4<T>*)out;
    const int p3 = (int)(step_index % 3);
    a.dt_read = (const double*)(small + p3);
    a.dt_write = small + (p3 + 1) % 3;
    a.dt_reset = small + (p3 + 2) % 3;
    a.t = (double*)(small + kSlotT);
    a.status = (unsigned*)(small + kSlotStatus);
    a.n_clamped = small + kSlotClamp;
    a.n_active = small + kSlotActive;
    a.dt_fixed = dt_fixed;
    a.dt_log = dt_log;
    if (with_activity && a.act_in)
        return Launch<T>::step(a, m->cfg.block_size, m->cfg.min_blocks, m->cfg.stages, m->cfg.geometry_early, st);
    a.act_in = nullptr;
    a.act_next = nullptr;
    a.act_clear = nullptr;
    const bool edges = m->plain.edges && m->eflux;
    a.ecells = edges ? m->ecells : nullptr;
    a.eln = edges ? (const T*)m->eln : nullptr;
    a.eflux = edges ? (V4<T>*)(eflux_out ? eflux_out : m->eflux) : nullptr;
    a.esrc = edges ? (T*)(esrc_out ? esrc_out : m->esrc) : nullptr;
    a.eidx = edges ? m->eidx : nullptr;
    a.n_edges = edges ? m->n_edges : 0;
    a.grid = m->plain.grid;
    if (m->plain.pairs)
        return Launch<T>::step_pair(a, m->plain.block, m->plain.min_blocks, m->plain.geo, m->plain.stages, st);
    return Launch<T>::step(a, m->plain.block, m->plain.min_blocks, m->plain.stages, m->plain.geo, st);
}

int advance(swe_mesh* m, int64_t nsteps, double cfl) {
    return m->cfg.precision == SWE_FP32 ? run_steps<float>(m, nsteps, cfl) : run_steps<double>(m, nsteps, cfl);
}

bool loop_possible(swe_mesh* m) {
    const int was = m->loop_short;
    m->loop_short = -1;
    const bool can = m->cfg.precision == SWE_FP32 ? use_loop<float>(m, 4) : use_loop<double>(m, 4);
    m->loop_short = was;
    return can;
}

// One step of mesh m from buffer `in` to buffer `out` with the given status
// block and step index (dt slot rotation), taking dt from *dt_fixed when set.
cudaError_t launch_step_raw(swe_mesh* m, const void* in, void* out, unsigned long long* small, int64_t step_index,
                            double cfl, const double* dt_fixed, double* dt_log, cudaStream_t st, bool with_activity,
                            void* eflux_out, void* esrc_out) {
    return m->cfg.precision == SWE_FP32
               ? launch_raw_t<float>(m, in, out, small, step_index, cfl, dt_fixed, dt_log, st, with_activity,
                                     eflux_out, esrc_out)
               : launch_raw_t<double>(m, in, out, small, step_index, cfl, dt_fixed, dt_log, st, with_activity,
                                      eflux_out, esrc_out);
}

double host_unit_normal(double& lx, double& ly) {
    const double l2 = std::fma(lx, lx, ly * ly);
    const double rl = 1.0 / std::sqrt(l2);
    lx *= rl;
    ly *= rl;
    return l2 * rl;
}

void append_edges(const HostMesh& H, int64_t base, std::vector<int2>& cells, std::vector<double>& ln, int4* eidx,
                  std::vector<double>* len) {
    const int64_t n = H.n_cells;
    for (int64_t c = 0; c < n; ++c) eidx[c] = make_int4(-1, -1, -1, 0);
    for (int64_t c = 0; c < n; ++c)
        for (int j = 0; j < 3; ++j) {
            const int32_t code = H.code[3 * c + j];
            if (code >= 0 && !(code & kFlipBit)) {
                const int e = (int)cells.size();
                const int k = code & kNbrMask;
                cells.push_back(make_int2((int)(base + c), (int)(base + k)));
                double lx = H.ln[6 * c + 2 * j], ly = H.ln[6 * c + 2 * j + 1];
                if (len) len->push_back(host_unit_normal(lx, ly));
                ln.push_back(lx);
                ln.push_back(ly);
                (j == 0 ? eidx[c].x : (j == 1 ? eidx[c].y : eidx[c].z)) = e;
                for (int jk = 0; jk < 3; ++jk)
                    if ((H.code[3 * k + jk] & kNbrMask) == (int32_t)c && H.code[3 * k + jk] >= 0)
                        (jk == 0 ? eidx[k].x : (jk == 1 ? eidx[k].y : eidx[k].z)) = e;
            }
        }
}

static int upload_edges(swe_mesh* m) {
    const HostMesh& H = m->hm;
    const int64_t n = H.n_cells;
    std::vector<int2> cells;
    std::vector<double> ln, rl;
    std::vector<int4> eidx(n);
    cells.reserve(3 * n / 2 + 1);
    ln.reserve(3 * n + 2);
    append_edges(H, 0, cells, ln, eidx.data(), m->esz == 8 ? &rl : nullptr);
    const int64_t E = (int64_t)cells.size();
    const size_t esz = m->esz;
    std::vector<char> lnt(2 * E * esz);
    for (int64_t q = 0; q < 2 * E; ++q) {
        if (esz == 4) { const float v = (float)ln[q]; std::memcpy(&lnt[q * 4], &v, 4); }
        else std::memcpy(&lnt[q * 8], &ln[q], 8);
    }
    const size_t Eb = (size_t)std::max<int64_t>(E, 1);
    cudaError_t e = cudaMalloc((void**)&m->ecells, Eb * sizeof(int2));
    if (e == cudaSuccess) e = cudaMalloc(&m->eln, 2 * Eb * esz);
    if (e == cudaSuccess) e = cudaMalloc(&m->eflux, Eb * 4 * esz);
    if (e == cudaSuccess) e = cudaMalloc(&m->esrc, Eb * esz);
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->eidx, (size_t)n * sizeof(int4));
    if (e == cudaSuccess && esz == 8) e = cudaMalloc(&m->erl, Eb * esz);
    if (e != cudaSuccess) {
        void* bufs[] = {m->ecells, m->eln, m->eflux, m->esrc, m->eidx, m->erl};
        for (void* b : bufs)
            if (b) cudaFree(b);
        m->ecells = nullptr; m->eln = nullptr; m->eflux = nullptr; m->esrc = nullptr; m->eidx = nullptr;
        m->erl = nullptr;
        set_error("edge pass: device allocation failed");
        return SWE_ENOMEM;
    }
    if (E) e = cudaMemcpy(m->ecells, cells.data(), E * sizeof(int2), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && E) e = cudaMemcpy(m->eln, lnt.data(), 2 * E * esz, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->eidx, eidx.data(), n * sizeof(int4), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && esz == 8 && E) e = cudaMemcpy(m->erl, rl.data(), E * sizeof(double), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "edge pass: upload");
    m->n_edges = E;
    m->device_bytes += (int64_t)(Eb * (sizeof(int2) + (esz == 8 ? 8 : 7) * esz) + n * sizeof(int4));
    return SWE_OK;
}

int build_edges(swe_mesh* m) {
    if (m->eflux) return SWE_OK;
    try {
        return upload_edges(m);
    } catch (const std::bad_alloc&) {   // before any device allocation
        set_error("edge pass: out of host memory");
        return SWE_ENOMEM;
    }
}

// The spans (2^kScanLog cells) beside each span: those with an edge in common,
// and itself.
static cudaError_t build_spans(swe_mesh* m) {
    const HostMesh& H = m->hm;
    const int64_t n = H.n_cells, ns = (n + (1 << kScanLog) - 1) >> kScanLog;
    std::vector<unsigned> first(ns + 1, 0u), adj, seen(ns, 0xFFFFFFFFu);
    for (int64_t sp = 0; sp < ns; ++sp) {
        first[sp] = (unsigned)adj.size();
        adj.push_back((unsigned)sp);
        seen[sp] = (unsigned)sp;
        const int64_t lo = sp << kScanLog, hi = std::min(n, (sp + 1) << kScanLog);
        for (int64_t k = 3 * lo; k < 3 * hi; ++k) {
            if (H.code[k] < 0) continue;
            const int64_t o = (H.code[k] & kNbrMask) >> kScanLog;
            if (seen[o] != (unsigned)sp) {
                seen[o] = (unsigned)sp;
                adj.push_back((unsigned)o);
            }
        }
    }
    first[ns] = (unsigned)adj.size();
    cudaError_t e = cudaMalloc((void**)&m->span_first, first.size() * sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->span_adj, adj.size() * sizeof(unsigned));
    if (e == cudaSuccess)
        e = cudaMemcpy(m->span_first, first.data(), first.size() * sizeof(unsigned), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->span_adj, adj.data(), adj.size() * sizeof(unsigned), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) m->device_bytes += (int64_t)((first.size() + adj.size()) * sizeof(unsigned));
    return e;
}

int init_activity(swe_mesh* m) {
    const int64_t n = m->hm.n_cells;
    cudaError_t e = cudaSuccess;
    if (!m->act[0]) {
        const int64_t len = (n + 31) / 32 * 32 + 32;   // bytes, then a flag per span
        const int64_t all = len + ((n + (1 << kScanLog) - 1) >> kScanLog);
        for (int k = 0; k < 3 && e == cudaSuccess; ++k) e = cudaMalloc((void**)&m->act[k], all);
        try {
            if (e == cudaSuccess) e = build_spans(m);
        } catch (const std::bad_alloc&) {
            e = cudaErrorMemoryAllocation;
        }
        if (e == cudaSuccess) e = cudaMalloc((void**)&m->act_list, n * sizeof(unsigned));
        if (e == cudaSuccess) e = cudaMalloc((void**)&m->act_count, 2 * sizeof(unsigned));
        if (e == cudaSuccess) e = cudaMemsetAsync(m->act_count, 0, 2 * sizeof(unsigned), m->stream);
        if (e != cudaSuccess) {
            for (void* p : {(void*)m->act[0], (void*)m->act[1], (void*)m->act[2], (void*)m->act_list,
                            (void*)m->act_count, (void*)m->span_first, (void*)m->span_adj})
                if (p) cudaFree(p);
            for (auto& p : m->act) p = nullptr;
            m->span_first = m->span_adj = nullptr;
            m->act_list = m->act_count = nullptr;
            set_error("activity bytes: allocation failed");
            return SWE_ENOMEM;
        }
        m->act_len = len;
        m->device_bytes += 3 * all + (int64_t)((n + 2) * sizeof(unsigned));
    }
    const int p3 = (int)(m->nstep % 3);
    const int64_t all = m->act_len + ((n + (1 << kScanLog) - 1) >> kScanLog);
    e = cudaMemsetAsync(m->act[p3], 2, all, m->stream);   // bit 1: rebuilt (act_init_kernel)
    if (e == cudaSuccess) e = cudaMemsetAsync(m->act[(p3 + 1) % 3], 0, all, m->stream);
    // the previous step's bytes: all 1, so the next step writes every cell's
    // state (its output buffer holds no step's result yet)
    if (e == cudaSuccess) e = cudaMemsetAsync(m->act[(p3 + 2) % 3], 1, all, m->stream);
    if (e == cudaSuccess)
        e = m->cfg.precision == SWE_FP32
                ? Launch<float>::act_init((const V4<float>*)m->state[m->nstep % 2], m->topo, n, (float)m->cfg.h_dry,
                                          m->act[p3], m->stream)
                : Launch<double>::act_init((const V4<double>*)m->state[m->nstep % 2], m->topo, n, m->cfg.h_dry,
                                           m->act[p3], m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "activity bytes: initialisation");
    m->act_valid = true;
    return SWE_OK;
}

int flush_mesh_bc(swe_mesh* m) { return flush_topo(m); }

void drop_mesh_graph(swe_mesh* m) { drop_graph(m); }

}  // namespace swe

extern "C" {

void swe_config_default(swe_config* cfg) {
    if (!cfg) return;
    cfg->precision = SWE_FP64;
    cfg->g = 9.81;
    cfg->h_dry = 1e-6;
    cfg->reorder = SWE_REORDER_HILBERT;
    cfg->block_size = 0;
    cfg->graph_steps = 0;
    cfg->device = 0;
    cfg->min_blocks = 0;
    cfg->stages = 0;
    cfg->geometry_early = 0;
    cfg->activity = 0;
    cfg->edge_pass = 0;
    cfg->grid = 0;
    cfg->debug_checks = 0;
    cfg->cell_pairs = 0;
    cfg->flux = SWE_FLUX_HLLC;
}

const char* swe_last_error(void) { return g_last_error.c_str(); }

int swe_debug_code_ok(int32_t code, int64_t n_cells, int n_groups) {
    return code_ok(code, (long long)n_cells, n_groups) ? 1 : 0;
}

int swe_debug_activity(swe_mesh* m, int64_t list_cells, int* listed) {
    if (!m) { set_error("swe_debug_activity: NULL mesh"); return SWE_EINVAL; }
    if (list_cells >= 0) m->list_cells = list_cells;
    if (listed) *listed = m->cfg.activity && m->act_valid && m->act_by_list ? 1 : 0;
    return SWE_OK;
}

int swe_debug_loop(swe_mesh* m, int64_t max_cells, int64_t max_polls, int64_t* steps) {
    if (!m || max_polls > (int64_t)0xFFFFFFFF) { set_error("swe_debug_loop: bad arguments"); return SWE_EINVAL; }
    if (max_cells >= 0) {
        m->loop_cells_set = max_cells;
        m->loop_cells = -1;
    }
    if (max_polls >= 0) m->loop_polls = (unsigned)max_polls;
    if (steps) *steps = m->loop_steps;
    return SWE_OK;
}

void swe_mesh_destroy(swe_mesh* m) {
    if (!m) return;
    DeviceGuard dg(m->cfg.device);
    if (m->stream) cudaStreamSynchronize(m->stream);
    drop_graph(m);
    drop_diag_workspace(m);
    drop_adjoint_workspace(m);
    void* bufs[] = {m->state[0], m->state[1], m->geoA, m->geoB, m->topo, m->gm2, m->zdev, m->perm, m->inv, m->loop_barrier, m->loop_ecell, m->loop_egeo, m->loop_eslot,
                    m->stage[0], m->stage[1], m->stage[2], m->small, m->act[0], m->act[1], m->act[2],
                    m->ecells, m->eln, m->eflux, m->esrc, m->eidx, m->geoR, m->erl, m->act_list, m->act_count, m->span_first, m->span_adj};
    for (void* b : bufs)
        if (b) cudaFree(b);
    if (m->cap_stream) cudaStreamDestroy(m->cap_stream);
    delete m;
}

int swe_mesh_create(const double* nodes, int64_t n_nodes, const int32_t* tris, int64_t n_tris,
                    const double* bathy, const double* manning, const swe_config* cfg, swe_mesh** out) {
    if (!out) { set_error("swe_mesh_create: out is NULL"); return SWE_EINVAL; }
    *out = nullptr;
    swe_config c;
    swe_config_default(&c);
    if (cfg) c = *cfg;
    if (c.precision != SWE_FP64 && c.precision != SWE_FP32) { set_error("swe_mesh_create: bad precision"); return SWE_EINVAL; }
    if (!(c.g > 0.0) || !(c.h_dry > 0.0) || !std::isfinite(c.g) || !std::isfinite(c.h_dry)) {
        set_error("swe_mesh_create: g and h_dry must be finite and > 0");
        return SWE_EINVAL;
    }
    if (c.h_dry < (double)FLT_MIN) {
        // a wet depth must stay a normal float: FP32 kernels hold it as one, and the
        // FP64 friction term starts its h^(-1/3) iteration from the float reciprocal cube root
        set_error("swe_mesh_create: h_dry must be at least FLT_MIN (1.18e-38)");
        return SWE_EINVAL;
    }
    if (c.flux != SWE_FLUX_HLLC && c.flux != SWE_FLUX_HLL) { set_error("swe_mesh_create: unknown flux"); return SWE_EINVAL; }
    if (c.geometry_early != 0 && c.geometry_early != 1) {
        set_error("swe_mesh_create: geometry_early must be 0 or 1");
        return SWE_EINVAL;
    }
    if (c.activity != 0 && c.activity != 1) {
        set_error("swe_mesh_create: activity must be 0 or 1");
        return SWE_EINVAL;
    }
    if (c.edge_pass != 0 && c.edge_pass != 1) {
        set_error("swe_mesh_create: edge_pass must be 0 or 1");
        return SWE_EINVAL;
    }
    if (c.grid < 0) {
        set_error("swe_mesh_create: grid must be >= 0");
        return SWE_EINVAL;
    }
    if (c.debug_checks != 0 && c.debug_checks != 1) {
        set_error("swe_mesh_create: debug_checks must be 0 or 1");
        return SWE_EINVAL;
    }

    if (c.cell_pairs != 0 && c.cell_pairs != 1) {
        set_error("swe_mesh_create: cell_pairs must be 0 or 1");
        return SWE_EINVAL;
    }
    if (c.cell_pairs && (c.precision != SWE_FP32 || c.activity || c.edge_pass)) {
        set_error("swe_mesh_create: cell_pairs needs FP32, without activity or edge_pass");
        return SWE_EINVAL;
    }
    if (c.edge_pass && c.activity) {
        set_error("swe_mesh_create: edge_pass and activity exclude each other");
        return SWE_EINVAL;
    }
    // FP64 with nothing chosen: the edge pass.  Its 1.5 evaluations a cell in
    // place of 3 halve the step's work (and 4,000 cells are one chain of
    // instructions a warp: 18.3 us a step without it); the results are the same.
    const bool implied_edges = c.precision == SWE_FP64 && c.block_size == 0 && c.min_blocks == 0 && c.stages == 0 &&
                               c.grid == 0 && !c.geometry_early && !c.activity;
    const bool nothing_chosen = c.block_size == 0 && c.min_blocks == 0 && c.stages == 0 && c.grid == 0 &&
                                !c.geometry_early && !c.activity && !c.edge_pass && !c.cell_pairs &&
                                c.graph_steps == 0;
    if (implied_edges) c.edge_pass = 1;
    if (c.block_size == 0) c.block_size = c.precision == SWE_FP32 ? 256 : 128;
    if (c.block_size != 128 && c.block_size != 256 && c.block_size != 512) {
        set_error("swe_mesh_create: block_size must be 128, 256 or 512");
        return SWE_EINVAL;
    }
    if (c.min_blocks == 0)
        c.min_blocks = c.precision == SWE_FP32 ? Launch<float>::default_min_blocks(c.block_size)
                                               : Launch<double>::default_min_blocks(c.block_size);
    if (c.stages == 0) c.stages = (c.precision == SWE_FP32 || c.activity) && !c.cell_pairs ? 3 : 1;
    if (c.graph_steps == 0) c.graph_steps = kDefaultGraphSteps;
    if (c.graph_steps > 0) c.graph_steps = std::max(6, (c.graph_steps / 6) * 6);
    if (c.activity && n_tris >= kActivityMaxCells) {
        set_error("swe_mesh_create: activity needs fewer than 2^29 cells");
        return SWE_EINVAL;
    }
    swe_mesh* m = new (std::nothrow) swe_mesh();
    if (!m) { set_error("swe_mesh_create: out of host memory"); return SWE_ENOMEM; }
    m->cfg = c;
    m->loop_allowed = nothing_chosen && !c.debug_checks;
    m->loop_polls = kMaxPolls;
    m->list_cells = kListCells;
    m->act_by_list = c.precision != SWE_FP32 || n_tris > kListCells;
    m->esz = c.precision == SWE_FP32 ? 4 : 8;
    std::string err;
    int rc;
    try {
        rc = build_host_mesh(nodes, n_nodes, tris, n_tris, bathy, manning, c.reorder, c.precision == SWE_FP32, m->hm,
                             err);
    } catch (const std::bad_alloc&) {
        rc = SWE_ENOMEM;
        err = "swe_mesh_create: out of host memory";
    }
    if (rc) { set_error(err); delete m; return rc; }
    DeviceGuard dg(c.device);
    if (!dg.ok) { set_error("swe_mesh_create: cannot select the device"); delete m; return SWE_ECUDA; }
    cudaError_t e = cudaStreamCreateWithFlags(&m->cap_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) { delete m; return cuda_fail(e, "swe_mesh_create: stream"); }
    const int64_t n = n_tris;
    const size_t v4 = 4 * m->esz;
    if ((rc = dev_alloc(m, &m->state[0], n * v4, "state")) || (rc = dev_alloc(m, &m->state[1], n * v4, "state")) ||
        (rc = dev_alloc(m, &m->geoA, n * v4, "geometry")) || (rc = dev_alloc(m, &m->geoB, n * v4, "geometry")) ||
        (c.precision == SWE_FP64 && (rc = dev_alloc(m, &m->geoR, n * v4, "geometry"))) ||
        (rc = dev_alloc(m, (void**)&m->topo, n * sizeof(int4), "topology")) ||
        (rc = dev_alloc(m, &m->gm2, n * m->esz, "manning")) ||
        (rc = dev_alloc(m, &m->zdev, n * m->esz, "bed")) ||
        (rc = dev_alloc(m, (void**)&m->perm, n * sizeof(unsigned), "permutation")) ||
        (rc = dev_alloc(m, (void**)&m->inv, n * sizeof(unsigned), "permutation")) ||
        (rc = dev_alloc(m, (void**)&m->small, (kSmallWords + 1) * sizeof(unsigned long long), "status"))) {
        swe_mesh_destroy(m);
        return rc;
    }
    rc = c.precision == SWE_FP32 ? upload_static<float>(m) : upload_static<double>(m);
    if (rc) { swe_mesh_destroy(m); return rc; }
    if (c.edge_pass) {
        rc = build_edges(m);
        if (rc == SWE_ENOMEM && implied_edges && !(cfg && cfg->edge_pass)) {   // without the edges' arrays, then
            (void)cudaGetLastError();
            c.edge_pass = m->cfg.edge_pass = 0;
            rc = SWE_OK;
        }
        if (rc) { swe_mesh_destroy(m); return rc; }
    }
    {
        int per_sm = 0, sms = 0;
        e = c.cell_pairs ? Launch<float>::pair_resident_blocks(c.block_size, c.min_blocks, c.geometry_early, c.stages,
                                                               &per_sm)
            : c.precision == SWE_FP32
                ? Launch<float>::resident_blocks(c.block_size, c.min_blocks, c.stages, c.geometry_early, c.activity,
                                                 c.edge_pass, &per_sm)
                : Launch<double>::resident_blocks(c.block_size, c.min_blocks, c.stages, c.geometry_early, c.activity,
                                                  c.edge_pass, &per_sm);
        if (e == cudaErrorInvalidValue) {
            swe_mesh_destroy(m);
            set_error("swe_mesh_create: no compiled step kernel for this block_size / min_blocks / stages / "
                      "geometry_early / activity / edge_pass / cell_pairs");
            return SWE_EINVAL;
        }
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c.device);
        if (e != cudaSuccess) { swe_mesh_destroy(m); return cuda_fail(e, "swe_mesh_create: occupancy"); }
        const long long units = c.cell_pairs ? (n + 1) / 2 : n;   // a thread's work item: a cell or a pair
        const long long need = (units + c.block_size - 1) / c.block_size;
        const long long wave = (long long)std::max(per_sm, 1) * std::max(sms, 1);
        m->grid = (unsigned)std::min(need, c.grid > 0 ? (long long)c.grid : wave);
        if (c.grid == 0 && c.precision == SWE_FP64 && !c.activity && n <= kSpreadCells) m->grid = spread_grid(n);
        // launches without activity bytes: the same shape, or the default one
        // when the configured shape exists only as an activity kernel
        m->plain = LaunchShape{c.block_size, c.min_blocks, c.stages, c.geometry_early, c.edge_pass, m->grid,
                               c.cell_pairs};
        if (c.activity) {
            LaunchShape d;
            d.block = c.precision == SWE_FP32 ? 256 : 128;
            d.min_blocks = c.precision == SWE_FP32 ? Launch<float>::default_min_blocks(d.block)
                                                   : Launch<double>::default_min_blocks(d.block);
            d.stages = c.precision == SWE_FP32 ? 3 : 1;
            d.geo = 0;
            int pb = 0;
            e = c.precision == SWE_FP32
                    ? Launch<float>::resident_blocks(d.block, d.min_blocks, d.stages, 0, 0, 0, &pb)
                    : Launch<double>::resident_blocks(d.block, d.min_blocks, d.stages, 0, 0, 0, &pb);
            if (e != cudaSuccess) { swe_mesh_destroy(m); return cuda_fail(e, "swe_mesh_create: occupancy"); }
            d.grid = (unsigned)std::min((long long)((n + d.block - 1) / d.block), (long long)std::max(pb, 1) * std::max(sms, 1));
            if (c.precision == SWE_FP64 && n <= kSpreadCells) d.grid = spread_grid(n);
            m->plain = d;
        }
    }
    m->bc.kind[0] = kBcWall;
    m->bc.value[0] = 0.0;
    m->group_len.assign(1, 0.0);
    m->group_value.assign(1, 0.0);
    for (int64_t s = 0; s < 3 * n; ++s)
        if (m->hm.code[s] < 0) m->group_len[0] += m->hm.len[s];
    *out = m;
    return SWE_OK;
}

int swe_set_bc(swe_mesh* m, const int32_t* pairs, int64_t n, int kind, double value) {
    if (!m || (!pairs && n > 0) || n < 0) { set_error("swe_set_bc: bad arguments"); return SWE_EINVAL; }
    if (kind < SWE_BC_WALL || kind > SWE_BC_STAGE) { set_error("swe_set_bc: unknown kind"); return SWE_EINVAL; }
    if (m->n_groups >= kMaxGroups - 1) { set_error("swe_set_bc: too many boundary groups"); return SWE_EINVAL; }
    if (!std::isfinite(value)) { set_error("swe_set_bc: non-finite value"); return SWE_EINVAL; }
    HostMesh& H = m->hm;
    const int grp = m->n_groups;
    std::vector<int64_t> slots;
    slots.reserve(n);
    for (int64_t e = 0; e < n; ++e) {
        const int32_t a = pairs[2 * e], b = pairs[2 * e + 1];
        const uint64_t key = ((uint64_t)std::min(a, b) << 32) | (uint64_t)std::max(a, b);
        auto it = std::lower_bound(H.bkey.begin(), H.bkey.end(), key);
        if (it == H.bkey.end() || *it != key) {
            set_error("swe_set_bc: node pair " + std::to_string(a) + "," + std::to_string(b) +
                      " is not a boundary edge");
            return SWE_EINVAL;
        }
        slots.push_back(H.bslot[it - H.bkey.begin()]);
    }
    double total = 0.0;
    for (int64_t s : slots) {
        const int old = -1 - H.code[s];
        if (old == grp) continue;
        m->group_len[old] -= H.len[s];
        total += H.len[s];
        H.code[s] = -1 - grp;
    }
    m->group_len.push_back(total);
    m->group_value.push_back(value);
    m->bc.kind[grp] = kind;
    m->n_groups = grp + 1;
    m->topo_dirty = true;
    DeviceGuard dg(m->cfg.device);
    return flush_topo(m);
}

int swe_set_stream(swe_mesh* m, void* stream) {
    if (!m) { set_error("swe_set_stream: NULL mesh"); return SWE_EINVAL; }
    m->stream = (cudaStream_t)stream;
    return SWE_OK;
}

int swe_set_state(swe_mesh* m, const void* h, const void* hu, const void* hv, int where, double t) {
    if (!m || !h || !hu || !hv || (where != SWE_HOST && where != SWE_DEVICE) || !std::isfinite(t)) {
        set_error("swe_set_state: bad arguments");
        return SWE_EINVAL;
    }
    DeviceGuard dg(m->cfg.device);
    int rc = flush_topo(m);
    if (rc) return rc;
    return m->cfg.precision == SWE_FP32 ? set_state_t<float>(m, h, hu, hv, where, t)
                                        : set_state_t<double>(m, h, hu, hv, where, t);
}

int swe_step(swe_mesh* m, int64_t nsteps, double cfl, double* t_out) {
    NvtxRange nvtx_range("swe_step");
    if (!m || nsteps < 0 || !(cfl > 0.0) || !std::isfinite(cfl)) { set_error("swe_step: bad arguments"); return SWE_EINVAL; }
    if (!m->have_state) { set_error("swe_step: no state set"); return SWE_EINVAL; }
    DeviceGuard dg(m->cfg.device);
    int rc = flush_topo(m);
    if (rc) return rc;
    rc = advance(m, nsteps, cfl);
    if (rc) return rc;
    if (t_out) {
        unsigned long long s[kSmallWords];
        rc = read_small(m, s);
        if (rc) return rc;
        *t_out = bits_to_double(s[kSlotT]);
        return status_code(s[kSlotStatus]);
    }
    return SWE_OK;
}

int swe_get_state(swe_mesh* m, void* h, void* hu, void* hv, int where) {
    if (!m || !h || !hu || !hv || (where != SWE_HOST && where != SWE_DEVICE)) {
        set_error("swe_get_state: bad arguments");
        return SWE_EINVAL;
    }
    if (!m->have_state) { set_error("swe_get_state: no state set"); return SWE_EINVAL; }
    DeviceGuard dg(m->cfg.device);
    return m->cfg.precision == SWE_FP32 ? get_state_t<float>(m, h, hu, hv, where)
                                        : get_state_t<double>(m, h, hu, hv, where);
}

int swe_synchronize(swe_mesh* m) {
    if (!m) { set_error("swe_synchronize: NULL mesh"); return SWE_EINVAL; }
    DeviceGuard dg(m->cfg.device);
    unsigned long long s[kSmallWords];
    int rc = read_small(m, s);
    if (rc) return rc;
    return status_code(s[kSlotStatus]);
}

int swe_get_info(swe_mesh* m, swe_info* info) {
    if (!m || !info) { set_error("swe_get_info: bad arguments"); return SWE_EINVAL; }
    DeviceGuard dg(m->cfg.device);
    std::memset(info, 0, sizeof *info);
    info->n_cells = m->hm.n_cells;
    info->precision = m->cfg.precision;
    info->device_bytes = m->device_bytes;
    info->n_steps = m->nstep;
    if (!m->have_state) {
        info->dt_next = INFINITY;
        return SWE_OK;
    }
    unsigned long long s[kSmallWords];
    int rc = read_small(m, s);
    if (rc) return rc;
    info->t = bits_to_double(s[kSlotT]);
    // the slot holds min_i R_i / (c_i + |u_i|); the CFL number of the next
    // swe_step call multiplies it
    info->dt_next = bits_to_double(s[m->nstep % 3]);
    info->n_clamped = (int64_t)s[kSlotClamp];
    info->n_active = (int64_t)s[kSlotActive];
    info->status = s[kSlotStatus] & kStatusBadIndex    ? SWE_EMESH
                   : s[kSlotStatus] & kStatusStall     ? SWE_ETIMEOUT
                   : s[kSlotStatus] & kStatusNonFinite ? SWE_ENONFINITE
                   : (s[kSlotStatus] & kStatusDry ? SWE_EDRY : SWE_OK);
    return SWE_OK;
}

int swe_get_permutation(swe_mesh* m, int64_t* perm) {
    if (!m || !perm) { set_error("swe_get_permutation: bad arguments"); return SWE_EINVAL; }
    std::memcpy(perm, m->hm.perm.data(), sizeof(int64_t) * m->hm.n_cells);
    return SWE_OK;
}

int swe_mesh_preprocess(const double* nodes, int64_t n_nodes, const int32_t* tris, int64_t n_tris, int reorder,
                        int precision, int64_t* perm, int32_t* code, double* ln, double* inv_area, double* rin) {
    if (n_tris < 1) { set_error("swe_mesh_preprocess: empty mesh"); return SWE_EINVAL; }
    if (precision != SWE_FP32 && precision != SWE_FP64) { set_error("swe_mesh_preprocess: bad precision"); return SWE_EINVAL; }
    HostMesh H;
    std::string err;
    int rc;
    try {
        std::vector<double> zeros((size_t)n_tris, 0.0);
        rc = build_host_mesh(nodes, n_nodes, tris, n_tris, zeros.data(), zeros.data(), reorder, precision == SWE_FP32, H,
                             err);
    } catch (const std::bad_alloc&) {
        rc = SWE_ENOMEM;
        err = "swe_mesh_preprocess: out of host memory";
    }
    if (rc) { set_error(err); return rc; }
    const size_t n = (size_t)n_tris;
    if (perm) std::memcpy(perm, H.perm.data(), n * sizeof(int64_t));
    if (code) std::memcpy(code, H.code.data(), 3 * n * sizeof(int32_t));
    if (ln) std::memcpy(ln, H.ln.data(), 6 * n * sizeof(double));
    if (inv_area) std::memcpy(inv_area, H.inv_area.data(), n * sizeof(double));
    if (rin) std::memcpy(rin, H.rin.data(), n * sizeof(double));
    return SWE_OK;
}

int swe_riemann_flux(int precision, int64_t n, const void* hL, const void* unL, const void* utL,
                     const void* hR, const void* unR, const void* utR, double g, double h_dry, void* G1,
                     void* G2, void* G3, void* S, void* stream) {
    return swe_riemann_flux_kind(precision, SWE_FLUX_HLLC, n, hL, unL, utL, hR, unR, utR, g, h_dry, G1, G2, G3, S,
                                 stream);
}

int swe_riemann_flux_kind(int precision, int flux, int64_t n, const void* hL, const void* unL, const void* utL,
                          const void* hR, const void* unR, const void* utR, double g, double h_dry, void* G1,
                          void* G2, void* G3, void* S, void* stream) {
    if (flux != SWE_FLUX_HLLC && flux != SWE_FLUX_HLL) { set_error("swe_riemann_flux: unknown flux"); return SWE_EINVAL; }
    const int hll = flux == SWE_FLUX_HLL ? 1 : 0;
    if (n < 0 || (n > 0 && (!hL || !unL || !utL || !hR || !unR || !utR || !G1 || !G2 || !G3))) {
        set_error("swe_riemann_flux: bad arguments");
        return SWE_EINVAL;
    }
    cudaError_t e;
    if (precision == SWE_FP32)
        e = Launch<float>::riemann(n, (const float*)hL, (const float*)unL, (const float*)utL, (const float*)hR,
                                   (const float*)unR, (const float*)utR, (float)g, (float)h_dry, (float*)G1,
                                   (float*)G2, (float*)G3, (float*)S, hll, (cudaStream_t)stream);
    else if (precision == SWE_FP64)
        e = Launch<double>::riemann(n, (const double*)hL, (const double*)unL, (const double*)utL,
                                    (const double*)hR, (const double*)unR, (const double*)utR, g, h_dry,
                                    (double*)G1, (double*)G2, (double*)G3, (double*)S, hll, (cudaStream_t)stream);
    else {
        set_error("swe_riemann_flux: bad precision");
        return SWE_EINVAL;
    }
    if (e != cudaSuccess) return cuda_fail(e, "swe_riemann_flux");
    return SWE_OK;
}

}  // extern "C"
