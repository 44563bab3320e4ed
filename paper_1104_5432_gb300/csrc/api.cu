// api.cu -- the C ABI (include/su2.h): handles, binding of caller-owned
// device memory, sweep orchestration through a replayed CUDA graph, host /
// device output handling, checkpoints and statistics.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "su2_testing.h"
#include "su2_internal.h"
#include "su2_math.cuh"
#include "su2_fixed.cuh"

using namespace su2;

static_assert(SU2_NUM_LAUNCH_CONFIGS == NUM_LAUNCH_CFG, "shape count of the header");
static_assert(SU2_LAUNCH_CLUSTER == CFG_CLUSTER, "cluster launch index of the header");

namespace {

thread_local std::string g_err;

int fail(int code, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

int cuda_fail(cudaError_t e, const char* what)
{
    return fail(SU2_E_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define SU2_CUDA(call)                                   \
    do {                                                 \
        cudaError_t e_ = (call);                         \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
uint32_t blocks_of(uint64_t n) { return (uint32_t)((n + TPB - 1) / TPB); }

struct DeviceGuard {
    int prev = -1;
    bool changed = false;
    explicit DeviceGuard(int dev)
    {
        if (dev < 0) return;
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) {
            changed = cudaSetDevice(dev) == cudaSuccess;
        }
    }
    ~DeviceGuard()
    {
        if (changed) cudaSetDevice(prev);
    }
};

__global__ void put_u64_kernel(uint64_t* dst, uint64_t v) { *dst = v; }

// NVTX range over one library call (visible in Nsight Systems timelines;
// free when no tool is attached)
struct Range {
    explicit Range(const char* name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
};

}  // namespace

struct su2_lattice {
    int n = 0;
    int dtype = 0;
    int row = 0;                    // shape-table row: FP32, FP64 or FP32 site pairs
    std::vector<int> Ns, Nt;
    std::vector<uint64_t> V, Vs, link_off, field_off;
    std::vector<uint32_t> site_start, spat_start;
    uint32_t site_blocks = 0, spat_blocks = 0;
    // per launch shape of the phase kernel: first block of each lattice,
    // total blocks, sweep-end chunks
    std::vector<uint32_t> phase_start[NUM_LAUNCH_CFG];
    uint32_t phase_blocks[NUM_LAUNCH_CFG] = {};
    uint32_t cfg_chunks[NUM_LAUNCH_CFG] = {};
    size_t off_pstart_cfg[NUM_LAUNCH_CFG] = {};
    uint32_t max_phase_blocks = 0;
    // the launch index selected or tuned: sweeps without measurements
    int chosen = 0;
    // sweeps replayed from a graph (with measurements, under the Creutz
    // sampler, and wherever the chosen index has no one-launch chain): the
    // cluster sweep (index CFG_CLUSTER) or the shape cfg, which single phases
    // take too.  Tuning sets them apart from `chosen`, since the chain is the
    // fastest on lattices whose phase launches in the same shape are not; and
    // the measured sweeps apart from the others, since their measurements run
    // beside phase launches and before a cluster sweep (8^4 FP32: 31 us a
    // measured sweep against 37, 29 and 23 without).
    int cfg = 0;
    bool cluster = false, cluster_measured = false;
    // cluster geometry (cluster_ok: -1 not yet known, 0 / 1)
    int cluster_ok = -1;
    ClusterGeom cgeom{};
    // all sweeps of a call in one cluster launch: index CFG_CLUSTER where a
    // CTA's share is small enough, and shape 0 on the smallest lattices
    // (chain0_ok as cluster_ok)
    bool cluster_chain = false;
    int chain0_ok = -1;
    ChainGeom chain_geom{}, chain0_geom{};
    std::string tune_key;
    std::vector<int> ysplit;        // y slabs per lattice (slab launch shapes)
    bool hybrid = false;            // Creutz/Kennedy-Pendleton sampler variant in use
    // last uniform parameters written by su2_heatbath_phase (beta, seed)
    bool phase_params_valid = false;
    double phase_beta = 0.0;
    uint64_t phase_seed = 0;
    int rmax_limit = 0;             // rmax <= min_l Ns_l / 2
    size_t link_bytes = 0, work_bytes = 0;
    size_t off_status = 0, off_desc = 0, off_sstart = 0, off_spstart = 0;
    size_t off_plaq = 0, off_obs = 0, off_field = 0, off_ring = 0, off_res = 0, off_stage = 0;
    size_t off_chunks = 0, off_tickets = 0, off_acc = 0, off_tslots = 0, off_fp64tab = 0, off_fixtab = 0, off_mirror = 0, off_oflag = 0;
    bool wide = false;              // some lattice of more than 2 OFF32_MAX_VH sites
    bool mirror = false;            // FP64: the work buffer holds a fixed-point copy of the links
    uint32_t max_chunks = 1;
    size_t res_doubles = 0;
    // bound state
    void* links = nullptr;
    char* work = nullptr;
    int device = -1;
    cudaStream_t stream = 0;
    cudaStream_t capture = nullptr;
    cudaStream_t capture_side = nullptr;    // the measurement branch while capturing
    cudaEvent_t fork_ev = nullptr, join_ev = nullptr;
    // replayable sweeps per launch shape and fused-plaquette flag
    cudaGraphExec_t sweep_graph[NUM_LAUNCH_CFG][2] = {};
    int measure_rmax = -1;                  // rmax baked into the measurement graphs
    // a sweep with the measurement of the previous sweep's result on a
    // parallel branch, and the measurement alone (after the last sweep)
    cudaGraphExec_t measure_graph[NUM_LAUNCH_CFG][2] = {};
    cudaGraphExec_t measure_tail = nullptr;
    // the same two for the cluster sweep
    cudaGraphExec_t cluster_graph[2] = {}, cluster_measure_graph[2] = {};
    Ctx ctx{};                      // non-phase kernels
    Ctx cfg_ctx[NUM_LAUNCH_CFG]{};  // phase kernels and sweep end, per launch shape

    bool bound() const { return links != nullptr && work != nullptr; }
    LatDesc* desc_dev(int l) const
    {
        return reinterpret_cast<LatDesc*>(work + off_desc) + l;
    }
    uint32_t* status_dev() const { return reinterpret_cast<uint32_t*>(work + off_status); }
    double* res_dev() const { return reinterpret_cast<double*>(work + off_res); }
    double* ring_dev() const { return reinterpret_cast<double*>(work + off_ring); }
    double* stage_dev() const { return reinterpret_cast<double*>(work + off_stage); }

    double* acc_dev() const { return reinterpret_cast<double*>(work + off_acc); }

    static void drop(cudaGraphExec_t (&gs)[NUM_LAUNCH_CFG][2])
    {
        for (auto& row : gs)
            for (auto& g : row)
                if (g) {
                    cudaGraphExecDestroy(g);
                    g = nullptr;
                }
    }

    static void drop2(cudaGraphExec_t (&gs)[2])
    {
        for (auto& g : gs)
            if (g) {
                cudaGraphExecDestroy(g);
                g = nullptr;
            }
    }

    void drop_measure_graphs()
    {
        drop(measure_graph);
        drop2(cluster_measure_graph);
        if (measure_tail) {
            cudaGraphExecDestroy(measure_tail);
            measure_tail = nullptr;
        }
    }

    void drop_graphs()
    {
        drop(sweep_graph);
        drop2(cluster_graph);
        drop_measure_graphs();
        measure_rmax = -1;
    }
};

namespace {

int check_handle(const su2_lattice* lat, bool need_bound = true)
{
    if (!lat) return fail(SU2_E_INVAL, "null handle");
    if (need_bound && !lat->bound()) return fail(SU2_E_INVAL, "no device memory bound");
    return SU2_OK;
}

// true when p is device (or managed) memory of some device
// the device address of page-locked (pinned or registered) host memory,
// which kernels read and write directly under unified addressing; null for
// anything else
const void* mapped_host_ptr(const void* p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return a.type == cudaMemoryTypeHost ? a.devicePointer : nullptr;
}

bool is_device_ptr(const void* p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// links one block of launch shape k updates per phase (a site-pair shape's
// rounds count pairs; FP64 shapes 10 and 11 give each link `group` threads)
uint64_t links_per_block(const su2_lattice* L, int k)
{
    const LaunchCfg& c = LAUNCH_CFG[L->row][k];
    return (uint64_t)c.threads * (uint64_t)c.rounds * (L->row == ROW_F32_PAIRS ? 2u : 1u) /
           (uint64_t)c.group;
}

int layout(su2_lattice* L)
{
    const int n = L->n;
    L->V.resize(n);
    L->Vs.resize(n);
    L->link_off.resize(n);
    L->field_off.resize(n);
    for (int k = 0; k < NUM_LAUNCH_CFG; ++k) L->phase_start[k].assign(n + 1, 0);
    L->site_start.assign(n + 1, 0);
    L->spat_start.assign(n + 1, 0);
    size_t lb = 0;
    uint64_t fo = 0;
    int rlim = 1 << 30;
    const size_t link_size = L->dtype == SU2_F32 ? 16 : 32;
    for (int l = 0; l < n; ++l) {
        const uint64_t Ns = (uint64_t)L->Ns[l], Nt = (uint64_t)L->Nt[l];
        L->Vs[l] = Ns * Ns * Ns;
        L->V[l] = L->Vs[l] * Nt;
        L->wide = L->wide || L->V[l] / 2 > OFF32_MAX_VH;
        L->link_off[l] = lb;
        lb += align256(4 * L->V[l] * link_size);
        L->field_off[l] = fo;
        fo += (L->Vs[l] + 31) & ~uint64_t(31);
        for (int k = 0; k < NUM_LAUNCH_CFG; ++k) {
            // links per block: threads x rounds
            const uint64_t nt = links_per_block(L, k);
            L->phase_start[k][l + 1] = L->phase_start[k][l] + (uint32_t)((L->V[l] / 2 + nt - 1) / nt);
        }
        L->site_start[l + 1] = L->site_start[l] + blocks_of(L->V[l]);
        L->spat_start[l + 1] = L->spat_start[l] + blocks_of(L->Vs[l]);
        rlim = std::min(rlim, L->Ns[l] / 2);
    }
    L->max_chunks = 1;
    L->max_phase_blocks = 0;
    for (int k = 0; k < NUM_LAUNCH_CFG; ++k) {
        L->phase_blocks[k] = L->phase_start[k][n];
        const uint32_t wpb = (uint32_t)LAUNCH_CFG[L->row][k].threads / 32;
        L->max_phase_blocks = std::max(L->max_phase_blocks, L->phase_blocks[k] * wpb);
        L->cfg_chunks[k] = 1;
        for (int l = 0; l < n; ++l) {
            const uint32_t nb = (L->phase_start[k][l + 1] - L->phase_start[k][l]) * wpb;
            L->cfg_chunks[k] = std::max<uint32_t>(L->cfg_chunks[k], (3 * nb + SWEEP_CHUNK - 1) / SWEEP_CHUNK);
        }
        L->max_chunks = std::max(L->max_chunks, L->cfg_chunks[k]);
    }
    L->site_blocks = L->site_start[n];
    L->spat_blocks = L->spat_start[n];
    L->rmax_limit = std::min(rlim, MAX_RMAX);
    L->link_bytes = lb;

    size_t w = 0;
    auto take = [&](size_t bytes) {
        const size_t o = w;
        w += align256(bytes);
        return o;
    };
    // the status word, the results and the plaquette ring lie together: one
    // copy brings a call's results and its status to the host
    L->res_doubles = (size_t)n * (L->rmax_limit + 1) + 2 * (size_t)n;
    L->off_status = take(256);
    L->off_res = take(8 * L->res_doubles);
    L->off_ring = take(8 * (size_t)PLAQ_RING * n);
    L->off_desc = take(sizeof(LatDesc) * n);
    for (int k = 0; k < NUM_LAUNCH_CFG; ++k) L->off_pstart_cfg[k] = take(4 * (n + 1));
    L->off_sstart = take(4 * (n + 1));
    L->off_spstart = take(4 * (n + 1));
    L->off_plaq = take(8 * 3 * (size_t)L->max_phase_blocks);
    const size_t obs_rows = std::max<size_t>(L->site_blocks,
                                             (size_t)L->spat_blocks * (size_t)(L->rmax_limit + 1));
    L->off_obs = take(8 * obs_rows);
    L->off_field = take(8 * fo);
    L->off_chunks = take(8 * (size_t)L->max_chunks * n);
    L->off_tickets = take(4 * (size_t)n);
    L->off_tslots = take(8 * (size_t)TRIAL_SLOTS * n);
    L->off_oflag = take(4 * (size_t)n);
    L->off_acc = take(8 * L->res_doubles);
    L->off_stage = take(STAGE_BYTES);
    L->off_fp64tab = take(sizeof(double2) * FP64_TABLE_ENTRIES);
    L->off_fixtab = take(sizeof(FixTables));
    L->mirror = L->dtype == SU2_F64 && L->link_bytes <= MIRROR_MAX;
    L->off_mirror = take(L->mirror ? L->link_bytes : 0);
    L->work_bytes = w;
    return SU2_OK;
}

int create(int n, const int* Ns, const int* Nt, int dtype, su2_lattice** out)
{
    if (!out) return fail(SU2_E_INVAL, "out is null");
    *out = nullptr;
    if (n < 1 || n > 4096) return fail(SU2_E_INVAL, "n must be in 1..4096 (got %d)", n);
    if (!Ns || !Nt) return fail(SU2_E_INVAL, "null shape array");
    if (dtype != SU2_F32 && dtype != SU2_F64) return fail(SU2_E_INVAL, "bad dtype %d", dtype);
    for (int l = 0; l < n; ++l) {
        if (Ns[l] < 2 || Nt[l] < 2 || (Ns[l] & 1) || (Nt[l] & 1))
            return fail(SU2_E_INVAL, "lattice %d: Ns=%d Nt=%d must be even and >= 2", l, Ns[l],
                        Nt[l]);
        // extents bounded first, so the volume product cannot wrap
        if (Ns[l] > 1024 || Nt[l] > (1 << 30))
            return fail(SU2_E_INVAL, "lattice %d: Ns=%d Nt=%d, volume above 2^30", l, Ns[l],
                        Nt[l]);
        const uint64_t V = (uint64_t)Ns[l] * (uint64_t)Ns[l] * (uint64_t)Ns[l] * (uint64_t)Nt[l];
        if (V > (uint64_t(1) << 30))
            return fail(SU2_E_INVAL, "lattice %d: volume %llu above 2^30", l,
                        (unsigned long long)V);
    }
    su2_lattice* L = new su2_lattice;
    L->n = n;
    L->dtype = dtype;
    // the plain layout by default; site pairs only on request
    // (su2_set_link_layout), being slower on every lattice measured
    L->row = dtype == SU2_F64 ? ROW_F64 : ROW_F32;
    L->Ns.assign(Ns, Ns + n);
    L->Nt.assign(Nt, Nt + n);
    layout(L);
    *out = L;
    return SU2_OK;
}

// y slabs for the large-lattice traversal: the smallest power of two
// dividing Ns that keeps the t-neighbour window Nh (Ns/S) Ns sites (records
// of site pairs) x 7 link loads within SLAB_WINDOW_BYTES (FP32 only; 1 =
// plain order)
int slab_rule(const su2_lattice* L, int l)
{
    if (L->dtype != SU2_F32) return 1;
    const double link = L->row == ROW_F32_PAIRS ? 32.0 : 16.0;
    const double Ns = L->Ns[l];
    int S = 1;
    while ((L->Ns[l] % (2 * S)) == 0 &&
           (Ns / 2) * (Ns / S) * Ns * 7.0 * link > SLAB_WINDOW_BYTES)
        S *= 2;
    return S;
}

void set_slabs(LatDesc& D, int S)
{
    D.ysplit = S;
    D.Ny = D.Ns / S;
    D.div_ny = make_fastdiv((uint32_t)D.Ny);
    D.div_nt = make_fastdiv((uint32_t)D.Nt);
}

// per-lattice parameters for the next sweeps; plaq_out[l] may be null
int set_params(su2_lattice* L, const double* betas, double beta, const uint64_t* seeds,
               uint64_t seed, double* plaq_dev, int nsweeps)
{
    L->phase_params_valid = false;
    for (int first = 0; first < L->n; first += PARAM_CHUNK) {
        ParamChunk pc{};
        pc.first = first;
        pc.count = std::min(PARAM_CHUNK, L->n - first);
        for (int j = 0; j < pc.count; ++j) {
            const int l = first + j;
            pc.beta[j] = betas ? betas[l] : beta;
            pc.seed[j] = seeds ? seeds[l] : seed + (uint64_t)l;
            pc.plaq_out[j] = plaq_dev ? plaq_dev + (size_t)l * nsweeps : nullptr;
        }
        SU2_CUDA(launch_set_params(L->ctx, pc, L->stream));
    }
    return SU2_OK;
}

// one sweep: 8 phases + sweep end; with rmax >= 0 also the Polyakov loop
// and the correlator, added into the handle's accumulators
// the Polyakov loop and correlator of the current links, summed into the
// accumulators (they read only the mu = 3 links and the Polyakov field)
int record_measure(su2_lattice* L, int rmax, cudaStream_t s)
{
    double* acc = L->acc_dev();
    SU2_CUDA(launch_polyakov(L->ctx, L->row, acc, acc + L->n, 1, s));
    SU2_CUDA(launch_correlator(L->ctx, L->dtype, rmax, acc + 2 * L->n, 1, s));
    return SU2_OK;
}

// One sweep.  With rmax >= 0 the links present at the START of the sweep
// (the previous sweep's result) are measured on a parallel branch: the
// measurement reads only the mu = 3 links, which the phases mu = 0, 1, 2
// leave alone, so it overlaps them and joins before phase (3, 0).
int record_sweep(su2_lattice* L, bool plaq, int rmax, cudaStream_t s)
{
    if (rmax >= 0 ? L->cluster_measured : L->cluster) {
        // the cluster kernel holds all links for the whole sweep: the
        // previous sweep's result is measured before it, not beside it
        if (rmax >= 0)
            if (int rc = record_measure(L, rmax, s)) return rc;
        SU2_CUDA(launch_cluster_sweep(L->cfg_ctx[L->cfg], L->cgeom, plaq, L->hybrid, s));
        return SU2_OK;
    }
    const bool branch = rmax >= 0;
    if (branch) {
        SU2_CUDA(cudaEventRecord(L->fork_ev, s));
        SU2_CUDA(cudaStreamWaitEvent(L->capture_side, L->fork_ev, 0));
        if (int rc = record_measure(L, rmax, L->capture_side)) return rc;
        SU2_CUDA(cudaEventRecord(L->join_ev, L->capture_side));
    }
    for (int mu = 0; mu < 4; ++mu) {
        if (branch && mu == 3) SU2_CUDA(cudaStreamWaitEvent(s, L->join_ev, 0));
        for (int p = 0; p < 2; ++p)
            SU2_CUDA(launch_phase(L->cfg_ctx[L->cfg], L->row, L->cfg, mu, p, plaq, nullptr,
                                  L->hybrid, false, s));
    }
    SU2_CUDA(launch_sweep_end(L->cfg_ctx[L->cfg], L->row == ROW_F64, plaq, s));
    return SU2_OK;
}

// capture what `record` enqueues into an executable graph
template <typename F>
int capture_graph(su2_lattice* L, F record, cudaGraphExec_t* g)
{
    if (!L->capture) SU2_CUDA(cudaStreamCreateWithFlags(&L->capture, cudaStreamNonBlocking));
    if (!L->capture_side)
        SU2_CUDA(cudaStreamCreateWithFlags(&L->capture_side, cudaStreamNonBlocking));
    if (!L->fork_ev) SU2_CUDA(cudaEventCreateWithFlags(&L->fork_ev, cudaEventDisableTiming));
    if (!L->join_ev) SU2_CUDA(cudaEventCreateWithFlags(&L->join_ev, cudaEventDisableTiming));
    SU2_CUDA(cudaStreamBeginCapture(L->capture, cudaStreamCaptureModeThreadLocal));
    const int rc = record(L->capture);
    cudaGraph_t graph = nullptr;
    const cudaError_t e = cudaStreamEndCapture(L->capture, &graph);
    if (rc != SU2_OK) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
    const cudaError_t ei = cudaGraphInstantiate(g, graph, 0);
    cudaGraphDestroy(graph);
    if (ei != cudaSuccess) {
        *g = nullptr;
        return cuda_fail(ei, "cudaGraphInstantiate");
    }
    return SU2_OK;
}

void set_measure_rmax(su2_lattice* L, int rmax)
{
    if (rmax != L->measure_rmax) {
        L->drop_measure_graphs();
        L->measure_rmax = rmax;
    }
}

// one sweep as a graph of kernels, built once per handle, binding and rmax
// (rmax >= 0: with the measurement branch of the previous sweep's result)
int sweep_graph(su2_lattice* L, bool plaq, int rmax, cudaGraphExec_t* exec)
{
    if (rmax >= 0) set_measure_rmax(L, rmax);
    const int pl = plaq ? 1 : 0;
    cudaGraphExec_t& g =
        rmax >= 0 ? (L->cluster_measured ? L->cluster_measure_graph[pl] : L->measure_graph[L->cfg][pl])
                  : (L->cluster ? L->cluster_graph[pl] : L->sweep_graph[L->cfg][pl]);
    if (!g) {
        if (int rc = capture_graph(
                L, [&](cudaStream_t s) { return record_sweep(L, plaq, rmax, s); }, &g))
            return rc;
    }
    *exec = g;
    return SU2_OK;
}

// the measurement alone, for the result of the last sweep of a call
int measure_tail_graph(su2_lattice* L, int rmax, cudaGraphExec_t* exec)
{
    set_measure_rmax(L, rmax);
    if (!L->measure_tail) {
        if (int rc = capture_graph(
                L, [&](cudaStream_t s) { return record_measure(L, rmax, s); }, &L->measure_tail))
            return rc;
    }
    *exec = L->measure_tail;
    return SU2_OK;
}

// turn a latched status word (fetched to the host) into its error, once
int report_status(su2_lattice* L, uint32_t st)
{
    if (st) {
        SU2_CUDA(cudaMemset(L->status_dev(), 0, sizeof st));
        if (st & STATUS_BOUNDS)
            return fail(SU2_E_BOUNDS, "link index out of bounds (bounds-checked build)");
        if (st & STATUS_STAGE)
            return fail(SU2_E_CUDA, "bulk copy of neighbour rows did not complete; phase abandoned");
        if (st & STATUS_CAP_HIT)
            return fail(SU2_E_TRIALS, "Kennedy-Pendleton trial cap (%d) hit; links kept", KP_CAP);
    }
    return SU2_OK;
}

// synchronise and turn a latched cap hit into SU2_E_TRIALS
int sync_status(su2_lattice* L)
{
    uint32_t st = 0;
    SU2_CUDA(cudaMemcpyAsync(&st, L->status_dev(), sizeof st, cudaMemcpyDeviceToHost, L->stream));
    SU2_CUDA(cudaStreamSynchronize(L->stream));
    return report_status(L, st);
}

// As sync_status, and the work buffer's bytes between the status word and
// src + count come with it in the same copy (each copy to pageable memory and
// its wait take ~10 us): the `count` values at src go to out, and n2 more that
// follow to out2.
int fetch_status(su2_lattice* L, const double* src, size_t count, double* out, size_t n2 = 0,
                 double* out2 = nullptr)
{
    const size_t at = (size_t)(reinterpret_cast<const char*>(src) - (L->work + L->off_status));
    const size_t bytes = at + sizeof(double) * (count + n2);
    const std::unique_ptr<char[]> buf(new (std::nothrow) char[bytes]);
    if (!buf) return fail(SU2_E_NOMEM, "no host memory for the results");
    SU2_CUDA(cudaMemcpyAsync(buf.get(), L->work + L->off_status, bytes, cudaMemcpyDeviceToHost,
                             L->stream));
    SU2_CUDA(cudaStreamSynchronize(L->stream));
    uint32_t st = 0;
    memcpy(&st, buf.get(), sizeof st);
    memcpy(out, buf.get() + at, sizeof(double) * count);
    if (out2) memcpy(out2, buf.get() + at + sizeof(double) * count, sizeof(double) * n2);
    return report_status(L, st);
}

// Whether the whole-sweep cluster kernel applies to this handle: one FP32
// lattice in the plain layout whose links fit the shared memory of one
// cluster that the GPU can hold (decided once per binding and layout).
bool cluster_available(su2_lattice* L)
{
    if (L->cluster_ok < 0) {
        L->cluster_ok = 0;
        if (L->row == ROW_F32 && L->n == 1 && L->device >= 0) {
            DeviceGuard dg(L->device);
            ClusterGeom g;
            if (cluster_geometry((uint32_t)(L->V[0] / 2), L->dtype == SU2_F32, L->n, &g) &&
                cluster_launchable(g)) {
                L->cgeom = g;
                L->cluster_ok = 1;
                L->cluster_chain = chain_geometry((uint32_t)(L->V[0] / 2), g.S, &L->chain_geom) &&
                                   chain_launchable(L->chain_geom);
            }
        }
    }
    return L->cluster_ok == 1;
}

// The geometry of the one-launch chain when the handle's sweeps run in it
// (without measurements, Kennedy-Pendleton only), or null.  Launch shape 0 takes
// it on lattices of at most CHAIN0_MAX_SITES sites (the most that fit: 512
// links of a phase on each of 16 SMs), where it is the faster (12^3 x 8: 23.1
// us a sweep against 28.9; 8^4: 12.2 against 28.7) and gives the same links
// and plaquettes bit by bit.
// FP64: at most 4096 sites (128 links of a phase on each SM).
constexpr uint64_t CHAIN0_MAX_SITES = 16384, CHAIN0_MAX_SITES_F64 = 4096;
const ChainGeom* chain_of(su2_lattice* L)
{
    if (L->hybrid || L->row == ROW_F32_PAIRS || L->n != 1) return nullptr;
    if (L->chosen == CFG_CLUSTER) return L->cluster_chain ? &L->chain_geom : nullptr;
    const bool f64 = L->row == ROW_F64;
    if (L->chosen != 0 || L->V[0] > (f64 ? CHAIN0_MAX_SITES_F64 : CHAIN0_MAX_SITES)) return nullptr;
    if (L->chain0_ok < 0) {
        DeviceGuard dg(L->device);
        const uint32_t Vh = (uint32_t)(L->V[0] / 2);
        ChainGeom& g = L->chain0_geom;
        L->chain0_ok = f64 ? chain64_geometry(Vh, &g) && chain64_launchable(g)
                           : chain_geometry(Vh, CLUSTER_MAX, &g) && chain_launchable(g);
    }
    return L->chain0_ok ? &L->chain0_geom : nullptr;
}
cudaError_t run_chain(su2_lattice* L, const ChainGeom& g, bool plaq, int nsweeps)
{
    return L->row == ROW_F64 ? launch_chain64(L->ctx, g, plaq, nsweeps, L->stream)
                             : launch_chain(L->ctx, g, plaq, nsweeps, L->stream);
}

// Launch indices (0 .. NUM_LAUNCH_CFG - 1, or CFG_CLUSTER): the one selected,
// and those of the sweeps replayed from a graph without and with measurements
// (a shape in both places is the same one).
struct Choice {
    int cfg = -1, replay = -1, measured = -1;
    Choice() = default;
    explicit Choice(int c) : cfg(c), replay(c), measured(c) {}
};
// false, and nothing changed, when one is not available
bool select_cfg(su2_lattice* L, const Choice& c)
{
    for (int k : {c.cfg, c.replay, c.measured})
        if (k < 0 || k > CFG_CLUSTER || (k == CFG_CLUSTER && !cluster_available(L))) return false;
    L->chosen = c.cfg;
    L->cluster = c.replay == CFG_CLUSTER;
    L->cluster_measured = c.measured == CFG_CLUSTER;
    // (where both are the cluster sweep cfg stays, for single phases)
    if (!L->cluster) L->cfg = c.replay;
    else if (!L->cluster_measured) L->cfg = c.measured;
    return true;
}

int heatbath_impl(su2_lattice* L, const double* betas, double beta, int nsweeps,
                  const uint64_t* seeds, uint64_t seed, double* plaq, int rmax = -1,
                  double* poly_sum = nullptr, double* corr_sum = nullptr)
{
    Range range(rmax >= 0 ? "su2_heatbath_measure" : "su2_heatbath");
    if (int rc = check_handle(L)) return rc;
    if (nsweeps < 0) return fail(SU2_E_INVAL, "nsweeps < 0");
    if (rmax >= 0) {
        if (rmax > L->rmax_limit)
            return fail(SU2_E_INVAL, "rmax %d outside 0..%d", rmax, L->rmax_limit);
        if (!poly_sum || !corr_sum) return fail(SU2_E_INVAL, "null measurement output");
    }
    for (int l = 0; l < L->n; ++l) {
        const double b = betas ? betas[l] : beta;
        if (!(b >= 0.0) || !std::isfinite(b)) return fail(SU2_E_INVAL, "beta must be finite and >= 0");
    }
    DeviceGuard dg(L->device);
    const bool want = plaq != nullptr;
    const bool dev_out = want && is_device_ptr(plaq);
    // Measured runs: the first sweep is a plain one; every later sweep
    // measures its predecessor's result on a parallel branch, and the tail
    // graph measures the last one, so each of the nsweeps results is
    // measured exactly once.
    cudaGraphExec_t g = nullptr, g_first = nullptr, g_tail = nullptr;
    if (rmax >= 0) {
        if (int rc = sweep_graph(L, want, -1, &g_first)) return rc;
        if (int rc = measure_tail_graph(L, rmax, &g_tail)) return rc;
    }
    const ChainGeom* chain = rmax < 0 ? chain_of(L) : nullptr;
    if (!chain)
        if (int rc = sweep_graph(L, want, rmax, &g)) return rc;
    const size_t acc_count = rmax >= 0 ? 2 * (size_t)L->n + (size_t)L->n * (rmax + 1) : 0;
    if (rmax >= 0)
        SU2_CUDA(cudaMemsetAsync(L->acc_dev(), 0, sizeof(double) * acc_count, L->stream));
    int done = 0;
    while (done < nsweeps) {
        const int chunk = (want && !dev_out) ? std::min(PLAQ_RING, nsweeps - done) : nsweeps;
        if (int rc = set_params(L, betas, beta, seeds, seed, dev_out ? plaq : nullptr, nsweeps))
            return rc;
        if (L->row == ROW_F64) SU2_CUDA(launch_unit_check(L->ctx, !chain, L->stream));
        if (chain) {
            for (int s = 0; s < chunk; s += PLAQ_RING)
                SU2_CUDA(run_chain(L, *chain, want, std::min(PLAQ_RING, chunk - s)));
        } else {
            for (int s = 0; s < chunk; ++s)
                SU2_CUDA(cudaGraphLaunch(g_first && done + s == 0 ? g_first : g, L->stream));
        }
        if (want && !dev_out) {
            if (L->n == 1 && rmax < 0 && done + chunk == nsweeps)
                return fetch_status(L, L->ring_dev(), (size_t)chunk, plaq + done);
            // one pitched copy when its rows fill the caller's buffer; a pitched
            // copy of part of the sweeps would span a whole pitch past its last
            // row, beyond the buffer's end
            if (chunk == nsweeps) {
                SU2_CUDA(cudaMemcpy2DAsync(plaq, sizeof(double) * nsweeps, L->ring_dev(),
                                           sizeof(double) * PLAQ_RING, sizeof(double) * chunk, L->n,
                                           cudaMemcpyDeviceToHost, L->stream));
            } else {
                for (int l = 0; l < L->n; ++l)
                    SU2_CUDA(cudaMemcpyAsync(plaq + (size_t)l * nsweeps + done,
                                             L->ring_dev() + (size_t)l * PLAQ_RING,
                                             sizeof(double) * chunk, cudaMemcpyDeviceToHost,
                                             L->stream));
            }
        }
        done += chunk;
    }
    if (rmax >= 0) {
        if (nsweeps > 0) SU2_CUDA(cudaGraphLaunch(g_tail, L->stream));
        const bool pdev = is_device_ptr(poly_sum), cdev = is_device_ptr(corr_sum);
        const double* acc = L->acc_dev();
        SU2_CUDA(cudaMemcpyAsync(poly_sum, acc, sizeof(double) * 2 * L->n,
                                 pdev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                                 L->stream));
        SU2_CUDA(cudaMemcpyAsync(corr_sum, acc + 2 * L->n,
                                 sizeof(double) * (size_t)L->n * (rmax + 1),
                                 cdev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                                 L->stream));
        if (!pdev || !cdev) return sync_status(L);
    }
    if (want && !dev_out) return sync_status(L);
    SU2_CUDA(cudaGetLastError());
    return SU2_OK;
}

int init_impl(su2_lattice* L, int start, const uint64_t* seeds, uint64_t seed)
{
    Range range("su2_init");
    if (int rc = check_handle(L)) return rc;
    if (start != SU2_COLD && start != SU2_HOT) return fail(SU2_E_INVAL, "bad start %d", start);
    DeviceGuard dg(L->device);
    for (int l = 0; l < L->n; ++l)
        SU2_CUDA(launch_init(L->ctx, L->dtype, l, (uint32_t)L->V[l], start,
                             seeds ? seeds[l] : seed + (uint64_t)l, L->stream));
    return SU2_OK;
}

}  // namespace

// ---------------------------------------------------------------------------
// launch-shape autotuning: key, cache file, measurement
// ---------------------------------------------------------------------------
namespace {

// Coupling band of a tuning: the mean beta of the lattices in steps of a
// factor sqrt 2 (the retry queue's share of the work follows the
// Kennedy-Pendleton acceptance, which grows with alpha = beta k).
int beta_band(const su2_lattice* L, const double* betas, double beta)
{
    double m = 0.0;
    for (int l = 0; l < L->n; ++l) m += betas ? betas[l] : beta;
    m /= L->n;
    if (!(m > 0.0)) return -99;
    return (int)std::floor(2.0 * std::log2(m));
}

constexpr double TUNE_BETA = 2.4;  // coupling of su2_autotune without betas

// Raised when another kernel comes to stand behind a launch index, so that no
// choice timed with the old one is taken from a cache file.
constexpr int KERNEL_VERSION = 1;

// FNV-1a over the lattice shapes, with the GPU name and precision in clear,
// and the coupling band
std::string tune_key(const su2_lattice* L, int dev, int band)
{
    cudaDeviceProp prop;
    std::string name = "unknown-gpu";
    if (cudaGetDeviceProperties(&prop, dev) == cudaSuccess) name = prop.name;
    else cudaGetLastError();
    for (auto& ch : name)
        if (ch == ' ' || ch == '\t') ch = '_';
    uint64_t h = 1469598103934665603ull;
    for (int l = 0; l < L->n; ++l)
        for (int v : {L->Ns[l], L->Nt[l]}) {
            h ^= (uint64_t)v;
            h *= 1099511628211ull;
        }
    // the launch-shape table of this precision, the kernels behind it and the
    // sampler: a cached index names the kernel that was timed only with these
    uint32_t th = 2166136261u;
    auto hash = [&](int v) {
        th ^= (uint32_t)v;
        th *= 16777619u;
    };
    for (const LaunchCfg& c : LAUNCH_CFG[L->row])
        for (int v : {c.threads, c.min_blocks, (int)c.slab, c.rounds, (int)c.persistent, c.group,
                      (int)c.stage})
            hash(v);
    hash(KERNEL_VERSION);
    hash(L->hybrid ? 1 : 0);
    char buf[256];
    static const char* const rows[NUM_ROWS] = {"f32", "f64", "f32pairs"};
    snprintf(buf, sizeof buf, "%s|%s|n%d|V%llu|%016llx|t%08x|b%d", name.c_str(), rows[L->row],
             L->n, (unsigned long long)[&] {
                 uint64_t t = 0;
                 for (uint64_t v : L->V) t += v;
                 return t;
             }(), (unsigned long long)h, th, band);
    return buf;
}

// Cache file: one line per key, "key cfg ms_per_sweep [replay measured]"; later
// lines win.  The last two (Choice) are cfg where absent.
bool cache_lookup(const char* path, const std::string& key, Choice* out)
{
    FILE* f = fopen(path, "r");
    if (!f) return false;
    char line[512];
    bool found = false;
    while (fgets(line, sizeof line, f)) {
        char k[400];
        Choice c;
        double ms = 0;
        const int got = sscanf(line, "%399s %d %lf %d %d", k, &c.cfg, &ms, &c.replay, &c.measured);
        if (got >= 2 && key == k) {
            *out = got == 5 ? c : Choice(c.cfg);
            found = true;
        }
    }
    fclose(f);
    return found;
}

bool cache_store(const char* path, const std::string& key, const Choice& c, double ms)
{
    FILE* f = fopen(path, "a");
    if (!f) return false;
    const bool ok = fprintf(f, "%s %d %.6f %d %d\n", key.c_str(), c.cfg, ms, c.replay, c.measured) > 0;
    return fclose(f) == 0 && ok;
}

}  // namespace

void su2::record_error(const char* msg) { g_err = msg; }

// The FP64 path's tables (su2_math.cuh).  ln_u01_tab: for each of the 256
// intervals of the mantissa
// M in [1, 2) (m = M / 2 from M = 1.5 on), g = 1 / c rounded, c the
// interval's centre, and -ln g from the long double logarithm; the last
// interval (m just below 1) takes c = 1, so that r = m - 1 is exact and
// ln u near 1 keeps its relative accuracy (no cancellation between -ln g
// and ln(1 + r)); then ln 2 = hi + lo with hi cut to 32 significant bits
// (n hi exact for |n| < 2^21).  sincospi_tab: cos and sin of pi j / 128
// from the long double functions.
void su2::fill_fp64_table(double2* tab)
{
    for (int t = 0; t < 256; ++t) {
        const double cM = 1.0 + (t + 0.5) / 256.0;  // exact
        const double g = t == 255 ? 1.0 : 1.0 / (t >= 128 ? 0.5 * cM : cM);
        tab[TAB_LN + t] = make_double2(g, t == 255 ? 0.0 : (double)(-logl((long double)g)));
    }
    const long double l2 = logl(2.0L);
    double hi = (double)l2;
    uint64_t b = 0;
    memcpy(&b, &hi, sizeof b);
    b &= ~((uint64_t(1) << 21) - 1);
    memcpy(&hi, &b, sizeof hi);
    tab[TAB_LN2] = make_double2(hi, (double)(l2 - (long double)hi));
    const long double pi = acosl(-1.0L);
    for (int j = 0; j < 256; ++j) {
        const long double a = pi * (long double)j / 128.0L;
        tab[TAB_TRIG + j] = make_double2((double)cosl(a), (double)sinl(a));
    }
}

// --------------------------------------------------------------------------
// exported
// --------------------------------------------------------------------------
namespace {

// The FP64 path's tables, computed once per process (2 ms in extended
// precision on the Arm host).
struct HostTables {
    double2 fp64[FP64_TABLE_ENTRIES];
    FixTables fix;
};
const HostTables& host_tables()
{
    static const HostTables t = [] {
        HostTables h;
        fill_fp64_table(h.fp64);
        fill_fix_tables(&h.fix);
        return h;
    }();
    return t;
}

// Links of lattice l to / from the canonical layout with values of type C
// (double or float): device buffers and page-locked host memory go through
// the conversion kernel directly, pageable host memory through the staging
// area in 32 MiB pieces.
template <typename C>
int get_links_impl(su2_lattice* lat, int l, C* dst)
{
    constexpr int cd = sizeof(C) == 8 ? 1 : 0;
    if (int rc = check_handle(lat)) return rc;
    if (!dst || l < 0 || l >= lat->n) return fail(SU2_E_INVAL, "bad lattice index or buffer");
    DeviceGuard dg(lat->device);
    const uint32_t V = (uint32_t)lat->V[l];
    const bool pw = lat->row == ROW_F32_PAIRS;  // whole lattice record by record
    if (is_device_ptr(dst)) {
        if ((uintptr_t)dst & 15) return fail(SU2_E_INVAL, "device buffer must be 16-byte aligned");
        SU2_CUDA(launch_links_to_canonical(lat->ctx, lat->dtype, l, 0, V, dst, cd, lat->stream, pw));
        return SU2_OK;
    }
    if (void* hd = const_cast<void*>(mapped_host_ptr(dst))) {
        if ((uintptr_t)hd & 15) return fail(SU2_E_INVAL, "host buffer must be 16-byte aligned");
        // page-locked host memory: written directly by the conversion kernel
        SU2_CUDA(launch_links_to_canonical(lat->ctx, lat->dtype, l, 0, V, hd, cd, lat->stream, pw));
        SU2_CUDA(cudaStreamSynchronize(lat->stream));
        return sync_status(lat);
    }
    const uint32_t per = (uint32_t)(STAGE_BYTES / (16 * sizeof(C)));
    for (uint32_t lex0 = 0; lex0 < V; lex0 += per) {
        const uint32_t cnt = std::min(per, V - lex0);
        SU2_CUDA(launch_links_to_canonical(lat->ctx, lat->dtype, l, lex0, cnt, lat->stage_dev(),
                                           cd, lat->stream));
        SU2_CUDA(cudaMemcpyAsync(dst + (size_t)lex0 * 16, lat->stage_dev(),
                                 sizeof(C) * 16 * cnt, cudaMemcpyDeviceToHost, lat->stream));
        SU2_CUDA(cudaStreamSynchronize(lat->stream));
    }
    return sync_status(lat);
}

template <typename C>
int set_links_impl(su2_lattice* lat, int l, const C* src)
{
    constexpr int cd = sizeof(C) == 8 ? 1 : 0;
    if (int rc = check_handle(lat)) return rc;
    if (!src || l < 0 || l >= lat->n) return fail(SU2_E_INVAL, "bad lattice index or buffer");
    DeviceGuard dg(lat->device);
    const uint32_t V = (uint32_t)lat->V[l];
    const bool pw = lat->row == ROW_F32_PAIRS;  // whole lattice record by record
    if (is_device_ptr(src)) {
        if ((uintptr_t)src & 15) return fail(SU2_E_INVAL, "device buffer must be 16-byte aligned");
        SU2_CUDA(launch_links_from_canonical(lat->ctx, lat->dtype, l, 0, V, src, cd, lat->stream, pw));
        return SU2_OK;
    }
    if (const void* hd = mapped_host_ptr(src)) {
        if ((uintptr_t)hd & 15) return fail(SU2_E_INVAL, "host buffer must be 16-byte aligned");
        // page-locked host memory: read directly by the conversion kernel
        SU2_CUDA(launch_links_from_canonical(lat->ctx, lat->dtype, l, 0, V, hd, cd, lat->stream, pw));
        SU2_CUDA(cudaStreamSynchronize(lat->stream));
        return SU2_OK;
    }
    const uint32_t per = (uint32_t)(STAGE_BYTES / (16 * sizeof(C)));
    for (uint32_t lex0 = 0; lex0 < V; lex0 += per) {
        const uint32_t cnt = std::min(per, V - lex0);
        SU2_CUDA(cudaMemcpyAsync(lat->stage_dev(), src + (size_t)lex0 * 16,
                                 sizeof(C) * 16 * cnt, cudaMemcpyHostToDevice, lat->stream));
        SU2_CUDA(launch_links_from_canonical(lat->ctx, lat->dtype, l, lex0, cnt, lat->stage_dev(),
                                             cd, lat->stream));
    }
    SU2_CUDA(cudaStreamSynchronize(lat->stream));
    return SU2_OK;
}

}  // namespace

extern "C" {

int su2_lattice_create(int Ns, int Nt, int dtype, su2_lattice** out)
{
    return create(1, &Ns, &Nt, dtype, out);
}

int su2_batch_create(int n, const int* Ns, const int* Nt, int dtype, su2_lattice** out)
{
    return create(n, Ns, Nt, dtype, out);
}

int su2_lattice_destroy(su2_lattice* lat)
{
    if (!lat) return SU2_OK;
    {
        DeviceGuard dg(lat->device);
        lat->drop_graphs();
        if (lat->capture) cudaStreamDestroy(lat->capture);
        if (lat->capture_side) cudaStreamDestroy(lat->capture_side);
        if (lat->fork_ev) cudaEventDestroy(lat->fork_ev);
        if (lat->join_ev) cudaEventDestroy(lat->join_ev);
    }
    delete lat;
    return SU2_OK;
}

int su2_lattice_count(const su2_lattice* lat, int* n)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (!n) return fail(SU2_E_INVAL, "null output");
    *n = lat->n;
    return SU2_OK;
}

int su2_lattice_volume(const su2_lattice* lat, int l, uint64_t* V)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (!V || l < 0 || l >= lat->n) return fail(SU2_E_INVAL, "bad lattice index or output");
    *V = lat->V[l];
    return SU2_OK;
}

int su2_memory_requirements(const su2_lattice* lat, size_t* link_bytes, size_t* work_bytes)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (link_bytes) *link_bytes = lat->link_bytes;
    if (work_bytes) *work_bytes = lat->work_bytes;
    return SU2_OK;
}

int su2_bind_memory(su2_lattice* lat, void* links, size_t link_bytes, void* work, size_t work_bytes)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (!links || !work) return fail(SU2_E_INVAL, "null buffer");
    if (((uintptr_t)links & 255) || ((uintptr_t)work & 255))
        return fail(SU2_E_INVAL, "buffers must be 256-byte aligned");
    if (link_bytes < lat->link_bytes || work_bytes < lat->work_bytes)
        return fail(SU2_E_NOMEM, "buffers too small: need %zu + %zu bytes, got %zu + %zu",
                    lat->link_bytes, lat->work_bytes, link_bytes, work_bytes);
    if (!is_device_ptr(links) || !is_device_ptr(work))
        return fail(SU2_E_INVAL, "buffers must be device memory");
    int dev = 0;
    SU2_CUDA(cudaGetDevice(&dev));
    lat->drop_graphs();
    lat->links = links;
    lat->work = static_cast<char*>(work);
    lat->device = dev;

    std::vector<LatDesc> d(lat->n);
    lat->ysplit.assign(lat->n, 1);
    for (int l = 0; l < lat->n; ++l) {
        LatDesc& D = d[l];
        memset(&D, 0, sizeof D);
        D.Ns = lat->Ns[l];
        D.Nt = lat->Nt[l];
        D.Nh = lat->Ns[l] / 2;
        D.Vs = (int32_t)lat->Vs[l];
        D.V = (uint32_t)lat->V[l];
        D.Vh = (uint32_t)(lat->V[l] / 2);
        D.div_nh = make_fastdiv((uint32_t)D.Nh);
        D.div_ns = make_fastdiv((uint32_t)D.Ns);
        D.paired = lat->row == ROW_F32_PAIRS ? 1 : 0;
        D.Vq = (uint32_t)(lat->V[l] / 4);
        D.div_nt2 = make_fastdiv((uint32_t)std::max(1, D.Nt / 2));
        set_slabs(D, slab_rule(lat, l));
        lat->ysplit[l] = D.ysplit;
        D.link_off = lat->link_off[l];
        D.field_off = lat->field_off[l];
        D.fp64_table = reinterpret_cast<const double2*>(lat->work + lat->off_fp64tab);
        D.fix_table = reinterpret_cast<const FixTables*>(lat->work + lat->off_fixtab);
    }
    char* w = lat->work;
    if (lat->dtype == SU2_F64) {
        const HostTables& t = host_tables();
        SU2_CUDA(cudaMemcpy(w + lat->off_fp64tab, t.fp64, sizeof t.fp64, cudaMemcpyHostToDevice));
        SU2_CUDA(cudaMemcpy(w + lat->off_fixtab, &t.fix, sizeof t.fix, cudaMemcpyHostToDevice));
    }
    SU2_CUDA(cudaMemset(w + lat->off_status, 0, 256));
    SU2_CUDA(cudaMemcpy(w + lat->off_desc, d.data(), sizeof(LatDesc) * lat->n,
                        cudaMemcpyHostToDevice));
    lat->phase_params_valid = false;
    // persistent shapes on a single lattice: as many blocks as fit at once
    // (each walks several tiles); on a batch they launch one block per tile
    int sms = 1;
    SU2_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    for (int k = 0; k < NUM_LAUNCH_CFG; ++k) {
        const LaunchCfg& cf = LAUNCH_CFG[lat->row][k];
        if (!cf.persistent || lat->n != 1) continue;
        const uint64_t per = links_per_block(lat, k);
        const uint32_t tiles = (uint32_t)((lat->V[0] / 2 + per - 1) / per);
        const uint32_t nb = std::min<uint32_t>(tiles, (uint32_t)(sms * cf.min_blocks));
        lat->phase_start[k][1] = nb;
        lat->phase_blocks[k] = nb;
        const uint32_t wpb = (uint32_t)cf.threads / 32;
        lat->cfg_chunks[k] = std::max<uint32_t>(1, (3 * nb * wpb + SWEEP_CHUNK - 1) / SWEEP_CHUNK);
    }
    for (int k = 0; k < NUM_LAUNCH_CFG; ++k)
        SU2_CUDA(cudaMemcpy(w + lat->off_pstart_cfg[k], lat->phase_start[k].data(),
                            4 * (lat->n + 1), cudaMemcpyHostToDevice));
    SU2_CUDA(cudaMemcpy(w + lat->off_sstart, lat->site_start.data(), 4 * (lat->n + 1),
                        cudaMemcpyHostToDevice));
    SU2_CUDA(cudaMemcpy(w + lat->off_spstart, lat->spat_start.data(), 4 * (lat->n + 1),
                        cudaMemcpyHostToDevice));
    SU2_CUDA(cudaMemset(w + lat->off_ring, 0, 8 * (size_t)PLAQ_RING * lat->n));
    SU2_CUDA(cudaMemset(w + lat->off_tickets, 0, 4 * (size_t)lat->n));
    SU2_CUDA(cudaMemset(w + lat->off_oflag, 0, 4 * (size_t)lat->n));
    SU2_CUDA(cudaMemset(w + lat->off_tslots, 0, 8 * (size_t)TRIAL_SLOTS * lat->n));

    Ctx& c = lat->ctx;
    c.links = links;
    c.mirror = lat->mirror ? reinterpret_cast<int4*>(w + lat->off_mirror) : nullptr;
    c.desc = reinterpret_cast<LatDesc*>(w + lat->off_desc);
    c.phase_start = reinterpret_cast<const uint32_t*>(w + lat->off_pstart_cfg[0]);
    c.site_start = reinterpret_cast<const uint32_t*>(w + lat->off_sstart);
    c.spat_start = reinterpret_cast<const uint32_t*>(w + lat->off_spstart);
    c.plaq_partial = reinterpret_cast<double*>(w + lat->off_plaq);
    c.obs_partial = reinterpret_cast<double*>(w + lat->off_obs);
    c.field = reinterpret_cast<double*>(w + lat->off_field);
    c.ring = reinterpret_cast<double*>(w + lat->off_ring);
    c.chunk_partial = reinterpret_cast<double*>(w + lat->off_chunks);
    c.chunk_count = reinterpret_cast<uint32_t*>(w + lat->off_tickets);
    c.trial_slots = reinterpret_cast<unsigned long long*>(w + lat->off_tslots);
    c.max_chunks = lat->cfg_chunks[0];
    c.phase_wpb = (uint32_t)LAUNCH_CFG[lat->row][0].threads / 32;
    c.status = reinterpret_cast<uint32_t*>(w + lat->off_status);
    c.obs_flag = reinterpret_cast<uint32_t*>(w + lat->off_oflag);
    c.n = lat->n;
    c.wide = lat->wide;
    c.phase_blocks = lat->phase_blocks[0];
    c.site_blocks = lat->site_blocks;
    c.spat_blocks = lat->spat_blocks;
    for (int k = 0; k < NUM_LAUNCH_CFG; ++k) {
        lat->cfg_ctx[k] = c;
        lat->cfg_ctx[k].phase_start = reinterpret_cast<const uint32_t*>(w + lat->off_pstart_cfg[k]);
        lat->cfg_ctx[k].phase_blocks = lat->phase_blocks[k];
        lat->cfg_ctx[k].max_chunks = lat->cfg_chunks[k];
        lat->cfg_ctx[k].phase_wpb = (uint32_t)LAUNCH_CFG[lat->row][k].threads / 32;
    }
    // a launch shape tuned earlier for these shapes on this GPU, if cached
    // (at the default tuning coupling)
    lat->tune_key = tune_key(lat, dev, beta_band(lat, nullptr, TUNE_BETA));
    lat->cluster_ok = lat->chain0_ok = -1;
    select_cfg(lat, Choice(0));
    if (const char* path = getenv("SU2_AUTOTUNE_CACHE")) {
        Choice cached;
        if (cache_lookup(path, lat->tune_key, &cached)) select_cfg(lat, cached);
    }
    return SU2_OK;
}

int su2_set_link_layout(su2_lattice* lat, int layout_code)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (lat->bound()) return fail(SU2_E_INVAL, "the link layout is fixed once memory is bound");
    if (layout_code == SU2_LAYOUT_PLAIN) {
        if (lat->dtype == SU2_F32) lat->row = ROW_F32;
    } else if (layout_code == SU2_LAYOUT_PAIRS) {
        if (lat->dtype != SU2_F32) return fail(SU2_E_INVAL, "site pairs are an FP32 layout");
        for (int l = 0; l < lat->n; ++l)
            if (lat->Nt[l] % 4)
                return fail(SU2_E_INVAL, "lattice %d: site pairs need Nt a multiple of 4 (Nt=%d)",
                            l, lat->Nt[l]);
        lat->row = ROW_F32_PAIRS;
    } else {
        return fail(SU2_E_INVAL, "bad link layout %d", layout_code);
    }
    lat->cluster_ok = lat->chain0_ok = -1;
    select_cfg(lat, Choice(0));
    return layout(lat);
}

int su2_get_link_layout(const su2_lattice* lat, int* layout_code)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (!layout_code) return fail(SU2_E_INVAL, "null output");
    *layout_code = lat->row == ROW_F32_PAIRS ? SU2_LAYOUT_PAIRS : SU2_LAYOUT_PLAIN;
    return SU2_OK;
}

int su2_set_stream(su2_lattice* lat, void* stream)
{
    if (int rc = check_handle(lat, false)) return rc;
    lat->stream = static_cast<cudaStream_t>(stream);
    return SU2_OK;
}

int su2_init(su2_lattice* lat, int start, uint64_t seed)
{
    return init_impl(lat, start, nullptr, seed);
}

int su2_batch_init(su2_lattice* lat, int start, const uint64_t* seeds)
{
    if (!seeds) return fail(SU2_E_INVAL, "null seeds");
    return init_impl(lat, start, seeds, 0);
}

int su2_heatbath(su2_lattice* lat, double beta, int nsweeps, uint64_t seed, double* plaq)
{
    return heatbath_impl(lat, nullptr, beta, nsweeps, nullptr, seed, plaq);
}

int su2_batch_heatbath(su2_lattice* lat, const double* betas, int nsweeps, const uint64_t* seeds,
                       double* plaq)
{
    if (!betas || !seeds) return fail(SU2_E_INVAL, "null betas or seeds");
    return heatbath_impl(lat, betas, 0.0, nsweeps, seeds, 0, plaq);
}

int su2_batch_heatbath_measure(su2_lattice* lat, const double* betas, int nsweeps,
                               const uint64_t* seeds, double* plaq, int rmax, double* poly_sum,
                               double* corr_sum)
{
    if (!betas || !seeds) return fail(SU2_E_INVAL, "null betas or seeds");
    if (rmax < 0) return fail(SU2_E_INVAL, "rmax < 0");
    return heatbath_impl(lat, betas, 0.0, nsweeps, seeds, 0, plaq, rmax, poly_sum, corr_sum);
}

int su2_heatbath_phase(su2_lattice* lat, double beta, int mu, int parity, uint64_t seed,
                       int32_t* trials)
{
    if (int rc = check_handle(lat)) return rc;
    if (mu < 0 || mu > 3 || (parity != 0 && parity != 1))
        return fail(SU2_E_INVAL, "bad phase (mu=%d parity=%d)", mu, parity);
    if (!(beta >= 0.0) || !std::isfinite(beta)) return fail(SU2_E_INVAL, "bad beta");
    if (trials && lat->n != 1) return fail(SU2_E_INVAL, "trials output needs n == 1");
    if (trials && !is_device_ptr(trials)) return fail(SU2_E_INVAL, "trials must be device memory");
    DeviceGuard dg(lat->device);
    // consecutive phases with the same beta and seed reuse the parameters
    // already on the device (no parameter kernel between the phases)
    if (!(lat->phase_params_valid && lat->phase_beta == beta && lat->phase_seed == seed)) {
        if (int rc = set_params(lat, nullptr, beta, nullptr, seed, nullptr, 0)) return rc;
        lat->phase_params_valid = true;
        lat->phase_beta = beta;
        lat->phase_seed = seed;
    }
    SU2_CUDA(launch_phase(lat->cfg_ctx[lat->cfg], lat->row, lat->cfg, mu, parity, false, trials,
                          lat->hybrid, true, lat->stream));
    return SU2_OK;
}

int su2_plaquette(su2_lattice* lat, double* out)
{
    if (int rc = check_handle(lat)) return rc;
    if (!out) return fail(SU2_E_INVAL, "null output");
    DeviceGuard dg(lat->device);
    const bool dev = is_device_ptr(out);
    double* tgt = dev ? out : lat->res_dev();
    SU2_CUDA(launch_plaquette(lat->ctx, lat->row, tgt, lat->stream));
    if (!dev) return fetch_status(lat, tgt, lat->n, out);
    return SU2_OK;
}

int su2_polyakov_loop(su2_lattice* lat, double* out_signed, double* out_abs)
{
    if (int rc = check_handle(lat)) return rc;
    if (!out_signed) return fail(SU2_E_INVAL, "null output");
    DeviceGuard dg(lat->device);
    const bool dev = is_device_ptr(out_signed);
    if (out_abs && is_device_ptr(out_abs) != dev)
        return fail(SU2_E_INVAL, "out_signed and out_abs must both be host or both device");
    double* ts = dev ? out_signed : lat->res_dev();
    double* ta = out_abs ? (dev ? out_abs : lat->res_dev() + lat->n) : nullptr;
    SU2_CUDA(launch_polyakov(lat->ctx, lat->row, ts, ta, 0, lat->stream));
    if (!dev) return fetch_status(lat, ts, lat->n, out_signed, out_abs ? lat->n : 0, out_abs);
    return SU2_OK;
}

int su2_polyakov_correlator(su2_lattice* lat, int rmax, double* out, int accumulate)
{
    if (int rc = check_handle(lat)) return rc;
    if (!out) return fail(SU2_E_INVAL, "null output");
    if (rmax < 0 || rmax > lat->rmax_limit)
        return fail(SU2_E_INVAL, "rmax %d outside 0..%d", rmax, lat->rmax_limit);
    DeviceGuard dg(lat->device);
    const bool dev = is_device_ptr(out);
    const size_t cnt = (size_t)lat->n * (rmax + 1);
    double* scratch = lat->res_dev();  // [2n] Polyakov means, then correlator rows
    double* tgt = dev ? out : scratch + 2 * lat->n;
    SU2_CUDA(launch_polyakov(lat->ctx, lat->row, nullptr, nullptr, 0, lat->stream));
    if (!dev && accumulate)
        SU2_CUDA(cudaMemcpyAsync(tgt, out, sizeof(double) * cnt, cudaMemcpyHostToDevice,
                                 lat->stream));
    SU2_CUDA(launch_correlator(lat->ctx, lat->dtype, rmax, tgt, accumulate, lat->stream));
    if (!dev) return fetch_status(lat, tgt, cnt, out);
    return SU2_OK;
}

int su2_get_links(su2_lattice* lat, int l, double* dst) { return get_links_impl(lat, l, dst); }
int su2_set_links(su2_lattice* lat, int l, const double* src) { return set_links_impl(lat, l, src); }
int su2_get_links_f32(su2_lattice* lat, int l, float* dst) { return get_links_impl(lat, l, dst); }
int su2_set_links_f32(su2_lattice* lat, int l, const float* src)
{
    return set_links_impl(lat, l, src);
}

int su2_gauge_transform(su2_lattice* lat, int l, uint64_t seed)
{
    if (int rc = check_handle(lat)) return rc;
    if (l < 0 || l >= lat->n) return fail(SU2_E_INVAL, "bad lattice index");
    DeviceGuard dg(lat->device);
    SU2_CUDA(launch_gauge(lat->ctx, lat->dtype, l, (uint32_t)lat->V[l], seed, lat->stream));
    return SU2_OK;
}

int su2_stats(su2_lattice* lat, int l, uint64_t out[3])
{
    if (int rc = check_handle(lat)) return rc;
    if (!out || l < 0 || l >= lat->n) return fail(SU2_E_INVAL, "bad lattice index or output");
    DeviceGuard dg(lat->device);
    SU2_CUDA(cudaStreamSynchronize(lat->stream));
    LatDesc d;
    SU2_CUDA(cudaMemcpy(&d, lat->desc_dev(l), sizeof d, cudaMemcpyDeviceToHost));
    unsigned long long slots[TRIAL_SLOTS];
    SU2_CUDA(cudaMemcpy(slots, lat->ctx.trial_slots + (size_t)l * TRIAL_SLOTS, sizeof slots,
                        cudaMemcpyDeviceToHost));
    out[0] = d.trials;
    for (unsigned long long v : slots) out[0] += v;
    out[1] = d.updates;
    out[2] = d.caps;
    return SU2_OK;
}

int su2_get_sweep(su2_lattice* lat, int l, uint64_t* sweep)
{
    if (int rc = check_handle(lat)) return rc;
    if (!sweep || l < 0 || l >= lat->n) return fail(SU2_E_INVAL, "bad lattice index or output");
    DeviceGuard dg(lat->device);
    SU2_CUDA(cudaStreamSynchronize(lat->stream));
    SU2_CUDA(cudaMemcpy(sweep, &lat->desc_dev(l)->sweep, sizeof *sweep, cudaMemcpyDeviceToHost));
    return SU2_OK;
}

int su2_set_sweep(su2_lattice* lat, int l, uint64_t sweep)
{
    if (int rc = check_handle(lat)) return rc;
    if (l < 0 || l >= lat->n) return fail(SU2_E_INVAL, "bad lattice index");
    DeviceGuard dg(lat->device);
    put_u64_kernel<<<1, 1, 0, lat->stream>>>(&lat->desc_dev(l)->sweep, sweep);
    SU2_CUDA(cudaGetLastError());
    return SU2_OK;
}

int su2_sync(su2_lattice* lat)
{
    if (int rc = check_handle(lat)) return rc;
    DeviceGuard dg(lat->device);
    return sync_status(lat);
}

int su2_autotune(su2_lattice* lat, int* chosen) { return su2_autotune_beta(lat, nullptr, chosen); }

int su2_autotune_beta(su2_lattice* lat, const double* betas, int* chosen)
{
    Range range("su2_autotune");
    if (int rc = check_handle(lat)) return rc;
    if (betas)
        for (int l = 0; l < lat->n; ++l)
            if (!(betas[l] >= 0.0) || !std::isfinite(betas[l]))
                return fail(SU2_E_INVAL, "beta must be finite and >= 0");
    DeviceGuard dg(lat->device);
    cudaStream_t s = lat->stream;
    const uint64_t tune_seed = 0x5EEDull;
    const int band = beta_band(lat, betas, TUNE_BETA);
    lat->tune_key = tune_key(lat, lat->device, band);
    for (int l = 0; l < lat->n; ++l)
        SU2_CUDA(launch_init(lat->ctx, lat->dtype, l, (uint32_t)lat->V[l], SU2_HOT, tune_seed + l, s));
    // a choice cached for this GPU, shapes and coupling band: no timing
    if (const char* path = getenv("SU2_AUTOTUNE_CACHE")) {
        Choice cached;
        if (cache_lookup(path, lat->tune_key, &cached) && select_cfg(lat, cached)) {
            if (int r2 = sync_status(lat)) return r2;
            if (chosen) *chosen = cached.cfg;
            return SU2_OK;
        }
    }
    if (int rc = set_params(lat, betas, TUNE_BETA, nullptr, tune_seed, nullptr, 0)) return rc;
    if (lat->row == ROW_F64) SU2_CUDA(launch_unit_check(lat->ctx, true, s));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    SU2_CUDA(cudaEventCreate(&e0));
    SU2_CUDA(cudaEventCreate(&e1));
    const int saved_chosen = lat->chosen, saved = lat->cfg;
    const bool saved_cluster = lat->cluster, saved_measured = lat->cluster_measured;
    // the shapes and the cluster sweep replayed from a graph, then the two
    // one-launch chains (of shape 0 and of the cluster index) where they apply
    constexpr int NI = NUM_LAUNCH_CFG + 1, NC = NI + 2;
    auto index_of = [](int k) { return k < NI ? k : (k == NI ? 0 : CFG_CLUSTER); };
    int rmax = -1;  // the measured sweeps' once those are timed
    double best_ms[NC];
    int reps[NC];
    int rc = SU2_OK;
    // Time what production runs: whole sweeps (graph replay or chain, fused
    // plaquette), candidates interleaved over three rounds, best round kept.
    auto time_sweeps = [&](int k, int n, float* ms) -> int {
        lat->chosen = index_of(k);
        lat->cluster = lat->cluster_measured = k == CFG_CLUSTER;
        if (k < NUM_LAUNCH_CFG) lat->cfg = k;
        const ChainGeom* chain = k < NI ? nullptr : chain_of(lat);
        cudaGraphExec_t g = nullptr;
        if (!chain)
            if (int r = sweep_graph(lat, true, rmax, &g)) return r;
        cudaError_t e = cudaEventRecord(e0, s);
        if (chain && e == cudaSuccess) e = run_chain(lat, *chain, true, n);
        for (int i = 0; i < n && !chain && e == cudaSuccess; ++i) e = cudaGraphLaunch(g, s);
        if (e == cudaSuccess) e = cudaEventRecord(e1, s);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
        return e == cudaSuccess ? SU2_OK : cuda_fail(e, "autotune timing");
    };
    // slab shapes only matter when some lattice is walked in slabs
    bool any_slab = false;
    for (int l = 0; l < lat->n; ++l) any_slab = any_slab || lat->ysplit[l] > 1;
    bool cand[NC];
    for (int k = 0; k < NUM_LAUNCH_CFG; ++k) cand[k] = any_slab || !LAUNCH_CFG[lat->row][k].slab;
    cand[CFG_CLUSTER] = cluster_available(lat);
    for (int k = NI; k < NC; ++k) {
        lat->chosen = index_of(k);
        cand[k] = cand[index_of(k)] && chain_of(lat) != nullptr;
    }
    auto time_candidates = [&]() {
        for (int k = 0; k < NC && rc == SU2_OK; ++k) {
            if (!cand[k]) continue;
            float ms = 0.f;
            rc = time_sweeps(k, 1, &ms);  // builds the graph, warms up
            if (rc == SU2_OK) rc = time_sweeps(k, 1, &ms);
            // about 20 ms of sweeps per round, between 1 and 50
            reps[k] = std::max(1, std::min(50, (int)(20.0 / std::max(ms, 1e-3f))));
            best_ms[k] = 1e300;
        }
        for (int round = 0; round < 3 && rc == SU2_OK; ++round)
            for (int k = 0; k < NC && rc == SU2_OK; ++k) {
                if (!cand[k]) continue;
                float ms = 0.f;
                rc = time_sweeps(k, reps[k], &ms);
                best_ms[k] = std::min(best_ms[k], (double)ms / reps[k]);
            }
    };
    // the best candidate below n
    auto best_of = [&](int n, bool chains) {
        int best = -1;
        for (int k = 0; k < n; ++k) {
            // an index whose chain applies runs as the chain
            if (!cand[k] || (chains && ((k == 0 && cand[NI]) || (k == CFG_CLUSTER && cand[NI + 1]))))
                continue;
            if (best < 0 || best_ms[k] < best_ms[best]) best = k;
        }
        return best;
    };
    time_candidates();
    Choice pick;
    double ms_chosen = 0.0;
    if (rc == SU2_OK) {
        const int best = best_of(NC, true), shape = best_of(NUM_LAUNCH_CFG, false);
        ms_chosen = best_ms[best];
        pick = Choice(index_of(best));
        // no chain: every sweep is a replayed one
        pick.replay = pick.measured = best < NI ? best : best_of(NI, false);
        if (pick.replay == CFG_CLUSTER) {
            // the measured sweeps: the cluster sweep or the best shape
            for (int k = 0; k < NC; ++k) cand[k] = k == shape || k == CFG_CLUSTER;
            rmax = lat->rmax_limit;
            time_candidates();
            if (rc == SU2_OK) pick.measured = best_of(NI, false);
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    lat->chosen = saved_chosen;
    lat->cfg = saved;
    lat->cluster = saved_cluster;
    lat->cluster_measured = saved_measured;
    if (rc != SU2_OK) return rc;
    // leave the handle as su2_init(SU2_HOT) with the tuning seed would; trial
    // caps hit by the tuning sweeps (small couplings under Kennedy-Pendleton
    // alone) belong to no run of the caller and are not reported
    SU2_CUDA(cudaMemsetAsync(lat->status_dev(), 0, sizeof(uint32_t), s));
    for (int l = 0; l < lat->n; ++l)
        SU2_CUDA(launch_init(lat->ctx, lat->dtype, l, (uint32_t)lat->V[l], SU2_HOT, tune_seed + l, s));
    if (int r2 = sync_status(lat)) return r2;
    select_cfg(lat, pick);
    if (const char* path = getenv("SU2_AUTOTUNE_CACHE"))
        if (!cache_store(path, lat->tune_key, pick, ms_chosen))
            return fail(SU2_E_INVAL, "cannot append to autotune cache %s", path);
    if (chosen) *chosen = pick.cfg;
    return SU2_OK;
}

int su2_set_launch_config(su2_lattice* lat, int cfg)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (cfg == CFG_CLUSTER && !lat->bound())
        return fail(SU2_E_INVAL, "the cluster sweep is chosen once memory is bound");
    if (!select_cfg(lat, Choice(cfg))) {  // graphs are kept per launch shape
        if (cfg == CFG_CLUSTER)
            return fail(SU2_E_INVAL, "the cluster sweep needs one FP32 lattice in the plain "
                                     "layout whose links fit one thread-block cluster");
        return fail(SU2_E_INVAL, "launch config %d outside 0..%d", cfg, CFG_CLUSTER);
    }
    return SU2_OK;
}

int su2_get_launch_config(const su2_lattice* lat, int* cfg, int* threads, int* min_blocks)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (lat->chosen == CFG_CLUSTER) {
        if (cfg) *cfg = CFG_CLUSTER;
        const bool chain = lat->cluster_chain && !lat->hybrid;
        if (threads) *threads = chain ? lat->chain_geom.updaters : lat->cgeom.threads;
        if (min_blocks) *min_blocks = lat->cgeom.S;
        return SU2_OK;
    }
    if (cfg) *cfg = lat->chosen;
    if (threads) *threads = LAUNCH_CFG[lat->row][lat->chosen].threads;
    if (min_blocks) *min_blocks = LAUNCH_CFG[lat->row][lat->chosen].min_blocks;
    return SU2_OK;
}

int su2_set_sampler(su2_lattice* lat, double creutz_below)
{
    if (int rc = check_handle(lat)) return rc;
    if (!(creutz_below >= 0.0) || !std::isfinite(creutz_below))
        return fail(SU2_E_INVAL, "creutz_below must be finite and >= 0");
    DeviceGuard dg(lat->device);
    SU2_CUDA(cudaStreamSynchronize(lat->stream));
    struct {
        double d;
        float f;
    } v{creutz_below, (float)creutz_below};
    static_assert(offsetof(LatDesc, creutz_below_f) == offsetof(LatDesc, creutz_below) + 8,
                  "sampler fields are adjacent");
    for (int l = 0; l < lat->n; ++l)
        SU2_CUDA(cudaMemcpy(reinterpret_cast<char*>(lat->desc_dev(l)) +
                                offsetof(LatDesc, creutz_below),
                            &v, 12, cudaMemcpyHostToDevice));
    const bool hyb = creutz_below > 0.0;
    if (hyb != lat->hybrid) {
        lat->hybrid = hyb;
        lat->drop_graphs();  // graphs bake in the sampler variant
    }
    return SU2_OK;
}

int su2_set_slabs(su2_lattice* lat, int S)
{
    if (int rc = check_handle(lat)) return rc;
    if (S < 1) return fail(SU2_E_INVAL, "slab count must be >= 1");
    for (int l = 0; l < lat->n; ++l)
        if (lat->Ns[l] % S) return fail(SU2_E_INVAL, "lattice %d: Ns=%d not divisible by %d", l,
                                        lat->Ns[l], S);
    DeviceGuard dg(lat->device);
    SU2_CUDA(cudaStreamSynchronize(lat->stream));
    for (int l = 0; l < lat->n; ++l) {
        LatDesc D;
        SU2_CUDA(cudaMemcpy(&D, lat->desc_dev(l), sizeof D, cudaMemcpyDeviceToHost));
        set_slabs(D, S);
        const size_t off = offsetof(LatDesc, ysplit);
        const size_t len = offsetof(LatDesc, div_nt) + sizeof(FastDiv) - off;
        SU2_CUDA(cudaMemcpy(reinterpret_cast<char*>(lat->desc_dev(l)) + off,
                            reinterpret_cast<const char*>(&D) + off, len, cudaMemcpyHostToDevice));
        lat->ysplit[l] = S;
    }
    return SU2_OK;
}

int su2_tune_key(const su2_lattice* lat, char* buf, size_t len)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (!buf || len == 0) return fail(SU2_E_INVAL, "null buffer");
    int dev = lat->device;
    if (dev < 0 && cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        dev = 0;
    }
    const std::string k = tune_key(lat, dev, beta_band(lat, nullptr, TUNE_BETA));
    if (k.size() + 1 > len) return fail(SU2_E_INVAL, "buffer too small");
    memcpy(buf, k.c_str(), k.size() + 1);
    return SU2_OK;
}

int su2_tune_cache_lookup(const char* path, const char* key, int* cfg)
{
    if (!path || !key || !cfg) return fail(SU2_E_INVAL, "null argument");
    Choice c;
    if (!cache_lookup(path, key, &c)) return 0;
    *cfg = c.cfg;
    return 1;
}

int su2_tune_cache_store(const char* path, const char* key, int cfg, double ms)
{
    if (!path || !key) return fail(SU2_E_INVAL, "null argument");
    if (cfg < 0 || cfg > CFG_CLUSTER) return fail(SU2_E_INVAL, "bad config");
    return cache_store(path, key, Choice(cfg), ms) ? SU2_OK : fail(SU2_E_INVAL, "cannot write %s", path);
}

int su2_one_launch(su2_lattice* lat, int* on)
{
    if (int rc = check_handle(lat)) return rc;
    if (!on) return fail(SU2_E_INVAL, "null output");
    *on = chain_of(lat) != nullptr;
    return SU2_OK;
}

int su2_replay_config(const su2_lattice* lat, int* plain, int* measured)
{
    if (int rc = check_handle(lat, false)) return rc;
    if (!plain || !measured) return fail(SU2_E_INVAL, "null output");
    *plain = lat->cluster ? CFG_CLUSTER : lat->cfg;
    *measured = lat->cluster_measured ? CFG_CLUSTER : lat->cfg;
    return SU2_OK;
}

const char* su2_last_error(void) { return g_err.c_str(); }

uint64_t su2_selftest_fastdiv(uint32_t dmax, uint32_t limit)
{
    uint64_t bad = 0;
    for (uint32_t d = 1; d <= dmax; ++d) {
        const FastDiv f = make_fastdiv(d);
        for (uint32_t n = 0; n < limit; ++n)
            if (fdiv(n, f) != n / d) ++bad;
        // the top of the supported range
        for (uint32_t n = (1u << 31) - 4096; n < (1u << 31); ++n)
            if (fdiv(n, f) != n / d) ++bad;
    }
    return bad;
}

}  // extern "C"
