// heatbath.cu -- sweep orchestration kernels of the SU(2) heat bath: the
// end-of-sweep reduction of the fused plaquette, the per-call parameter
// kernel and the dispatch of the phase kernels (heatbath_kernel.cuh,
// instantiated per pair of launch shapes and precision by
// heatbath_shapes.cu).
#include <algorithm>

#include "su2_internal.h"
#include "su2_mirror.cuh"
#include "su2_reduce.cuh"

namespace su2 {

// whether the links eo of the eight (mu, parity) planes of an FP64 lattice
// are unit quaternions; mirror: their fixed-point copies are written too
__device__ __forceinline__ bool unit_links_at(const Ctx& ctx, const LatDesc& D, uint32_t eo, bool mirror)
{
    const double2* U = reinterpret_cast<const double2*>(static_cast<const char*>(ctx.links) + D.link_off);
    bool ok = true;
#pragma unroll
    for (int mp = 0; mp < 8; ++mp) {
        const double2 lo = U[(size_t)(2 * mp) * D.Vh + eo], hi = U[(size_t)(2 * mp + 1) * D.Vh + eo];
        ok = ok && unit_link(lo, hi);
        if (mirror) {
            const FixMirror M(ctx, D);
            M.store(mp >> 1, mp & 1, eo, {lo.x, lo.y, hi.x, hi.y});
        }
    }
    return ok;
}

// One thread per two sites.  Bound by HBM: one read of the links (64^4: 2.1
// GB) and one write of their copies per call of any number of sweeps.
__global__ void __launch_bounds__(TPB) unit_check_kernel(Ctx ctx, bool mirror)
{
    const int l = lattice_of_block(ctx.site_start, ctx.n, blockIdx.x);
    LatDesc* D = ctx.desc + l;
    const uint32_t eo = (blockIdx.x - first_block(ctx.site_start, l)) * TPB + threadIdx.x;
    if (D->general & GENERAL_BETA) return;
    if (eo < D->Vh && !unit_links_at(ctx, *D, eo, mirror)) D->general = GENERAL_LINKS;
}

// The same by `nb` blocks after a sweep of a lattice that failed the check:
// once every link has been updated the lattice takes the fixed-point path.  The
// last block to finish (the counter D->recheck) clears the lattice's flag, so
// every block has read it by then.  (By one block a sweep of 64^4 with one bad
// link took 254 ms in all, by 32 62, by 304 56.)
constexpr unsigned RECHECK_BLOCKS = 32;  // over all lattices (200 idle ones took 0.9 us a sweep)
__device__ void unit_recheck(const Ctx& ctx, LatDesc* D, uint32_t block, uint32_t nb)
{
    bool ok = true;
    for (uint32_t eo = block * TPB + threadIdx.x; eo < D->Vh; eo += nb * TPB)
        if (!unit_links_at(ctx, *D, eo, ctx.mirror != nullptr)) ok = false;
    ok = __syncthreads_and(ok);
    if (threadIdx.x == 0) {
        const uint32_t mine = ok ? 1u : 0x10001u, sum = atomicAdd(&D->recheck, mine) + mine;
        if ((sum & 0xFFFFu) == nb) {
            D->recheck = 0u;
            if (sum >> 16 == 0u) D->general = 0u;
        }
    }
}

// Finishes a sweep: the fixed-order sum of the fused plaquette partials and
// the lattice's sweep counter.  Grid (chunks, lattices); each block sums
// SWEEP_CHUNK partials of its lattice, the last block of a lattice to finish
// (ticket counter) adds the chunk sums in chunk order.
// F64: nrecheck further blocks per lattice look again at the links of one that
// has non-unit ones (without the plaquette the first nrecheck blocks do).
template <bool PLAQ, bool F64>
__global__ void __launch_bounds__(TPB) sweep_end_kernel(Ctx ctx, uint32_t nrecheck)
{
    __shared__ double sred[TPB / 32];
    __shared__ int s_last;
    const int l = blockIdx.y;
    LatDesc* D = ctx.desc + l;
    if (!PLAQ && blockIdx.x == 0 && threadIdx.x == 0) D->sweep += 1;
    if (!PLAQ || (F64 && blockIdx.x >= ctx.max_chunks)) {
        if (F64 && D->general == GENERAL_LINKS)
            unit_recheck(ctx, D, PLAQ ? blockIdx.x - ctx.max_chunks : blockIdx.x, nrecheck);
        return;
    }
    // partials are per warp: lattice l owns warps [b0, b0 + nb) of each slot
    const uint32_t b0 = ctx.phase_start[l] * ctx.phase_wpb;
    const uint32_t nb = ctx.phase_start[l + 1] * ctx.phase_wpb - b0;
    const uint32_t stride = ctx.phase_blocks * ctx.phase_wpb;
    const uint32_t total = 3 * nb;
    const uint32_t nchunk = (total + SWEEP_CHUNK - 1) / SWEEP_CHUNK;
    if (blockIdx.x >= nchunk) return;

    const uint32_t e0 = blockIdx.x * SWEEP_CHUNK;
    const uint32_t e1 = min(e0 + (uint32_t)SWEEP_CHUNK, total);
    double acc = 0.0;
    for (uint32_t e = e0 + threadIdx.x; e < e1; e += TPB) {
        const uint32_t slot = (e >= nb) + (e >= 2 * nb);
        acc += ctx.plaq_partial[(size_t)slot * stride + b0 + (e - slot * nb)];
    }
    const double part = block_sum<TPB>(acc, sred);
    double* chunks = ctx.chunk_partial + (size_t)l * ctx.max_chunks;
    if (threadIdx.x == 0) {
        chunks[blockIdx.x] = part;
        __threadfence();
        const uint32_t ticket = atomicAdd(ctx.chunk_count + l, 1u);
        s_last = ticket == nchunk - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double c = 0.0;
    for (uint32_t k = threadIdx.x; k < nchunk; k += TPB) c += __ldcg(chunks + k);
    const double tot = block_sum<TPB>(c, sred);
    if (threadIdx.x == 0) {
        ctx.chunk_count[l] = 0;
        const double P = tot / (6.0 * (double)D->V);
        const uint64_t k = D->sweep - D->sweep_base;
        ctx.ring[(size_t)l * PLAQ_RING + (k % PLAQ_RING)] = P;
        if (D->plaq_out) D->plaq_out[k] = P;
        D->sweep += 1;
    }
}

// Per-call parameters go in by value (no host-to-device copy); the
// plaquette index origin is the lattice's own sweep counter at call time.
__global__ void set_params_kernel(Ctx ctx, ParamChunk pc)
{
    const int j = threadIdx.x;
    if (j >= pc.count) return;
    LatDesc* D = ctx.desc + pc.first + j;
    D->beta = pc.beta[j];
    D->beta_f = (float)pc.beta[j];
    D->half_inv_beta_f = (float)(0.5 / pc.beta[j]);
    D->half_inv_beta = 0.5 / pc.beta[j];  // inf at beta = 0, where the Haar draw applies
    D->seed = pc.seed[j];
    D->plaq_out = pc.plaq_out[j];
    D->general = pc.beta[j] > FIX_BETA_MAX ? GENERAL_BETA : 0u;
    D->sweep_base = D->sweep;
}

// one pair of FP32 launch shapes per instantiation of heatbath_shapes.cu, one
// FP64 kernel and sampler per instantiation of heatbath_fp64.cu
template <int ROW, int FIRST, bool WIDE>
cudaError_t launch_phase_pair(const Ctx& c, int cfg, int mu, int parity, bool plaq, int32_t* dbg,
                              bool hyb, cudaStream_t s);
template <int KIND, bool HYB>
cudaError_t launch_fix_kind(const Ctx& c, const LaunchCfg& f, int mu, int parity, bool plaq,
                            int32_t* dbg, bool mirror, cudaStream_t s);

cudaError_t launch_phase(const Ctx& c, int row, int cfg, int mu, int parity, bool plaq,
                         int32_t* dbg_trials, bool hybrid, bool single, cudaStream_t s)
{
    if (row < 0 || row >= NUM_ROWS || cfg < 0 || cfg >= NUM_LAUNCH_CFG) return cudaErrorInvalidValue;
    if (row == ROW_F64) {
        using Fn = cudaError_t (*)(const Ctx&, const LaunchCfg&, int, int, bool, int32_t*, bool,
                                   cudaStream_t);
        static_assert(NUM_FIX_KINDS == 6, "one entry per kernel below");
        static const Fn kinds[NUM_FIX_KINDS][2] = {
            {launch_fix_kind<0, false>, launch_fix_kind<0, true>},
            {launch_fix_kind<1, false>, launch_fix_kind<1, true>},
            {launch_fix_kind<2, false>, launch_fix_kind<2, true>},
            {launch_fix_kind<3, false>, launch_fix_kind<3, true>},
            {launch_fix_kind<4, false>, launch_fix_kind<4, true>},
            {launch_fix_kind<5, false>, launch_fix_kind<5, true>},
        };
        const LaunchCfg& f = LAUNCH_CFG[ROW_F64][cfg];
        Ctx cc = c;
        cc.look = single;
        return kinds[fix_kind(f)][hybrid](cc, f, mu, parity, plaq && !single, dbg_trials,
                                          !single && c.mirror, s);
    }
    using Fn = cudaError_t (*)(const Ctx&, int, int, int, bool, int32_t*, bool, cudaStream_t);
    static_assert(NUM_LAUNCH_CFG == 14 && NUM_ROWS == 3, "one entry per pair of shapes below");
    static const Fn pairs[3][NUM_LAUNCH_CFG / 2] = {
        {launch_phase_pair<0, 0, false>, launch_phase_pair<0, 2, false>, launch_phase_pair<0, 4, false>,
         launch_phase_pair<0, 6, false>, launch_phase_pair<0, 8, false>, launch_phase_pair<0, 10, false>,
         launch_phase_pair<0, 12, false>},
        {launch_phase_pair<2, 0, false>, launch_phase_pair<2, 2, false>, launch_phase_pair<2, 4, false>,
         launch_phase_pair<2, 6, false>, launch_phase_pair<2, 8, false>, launch_phase_pair<2, 10, false>,
         launch_phase_pair<2, 12, false>},
        {launch_phase_pair<0, 0, true>, launch_phase_pair<0, 2, true>, launch_phase_pair<0, 4, true>,
         launch_phase_pair<0, 6, true>, launch_phase_pair<0, 8, true>, launch_phase_pair<0, 10, true>,
         launch_phase_pair<0, 12, true>},
    };
    const int table = row == ROW_F32_PAIRS ? 1 : (c.wide ? 2 : 0);
    return pairs[table][cfg >> 1](c, cfg, mu, parity, plaq, dbg_trials, hybrid, s);
}

cudaError_t launch_sweep_end(const Ctx& c, bool fp64, bool plaq, cudaStream_t s)
{
    // a block for each TPB of an average lattice's Vh (site_blocks count V)
    const unsigned n = (unsigned)c.n, most = std::max(1u, RECHECK_BLOCKS / n);
    const unsigned nrecheck = fp64 ? std::min(most, std::max(1u, c.site_blocks / (2 * n))) : 0u;
    const dim3 grid(plaq ? c.max_chunks + nrecheck : std::max(1u, nrecheck), n);
    const unsigned nt = plaq || fp64 ? TPB : 32;
    if (fp64 && plaq) sweep_end_kernel<true, true><<<grid, nt, 0, s>>>(c, nrecheck);
    else if (fp64) sweep_end_kernel<false, true><<<grid, nt, 0, s>>>(c, nrecheck);
    else if (plaq) sweep_end_kernel<true, false><<<grid, nt, 0, s>>>(c, nrecheck);
    else sweep_end_kernel<false, false><<<grid, nt, 0, s>>>(c, nrecheck);
    return cudaGetLastError();
}

cudaError_t launch_unit_check(const Ctx& c, bool mirror, cudaStream_t s)
{
    unit_check_kernel<<<c.site_blocks, TPB, 0, s>>>(c, mirror && c.mirror);
    return cudaGetLastError();
}

cudaError_t launch_set_params(const Ctx& c, const ParamChunk& pc, cudaStream_t s)
{
    set_params_kernel<<<1, PARAM_CHUNK, 0, s>>>(c, pc);
    return cudaGetLastError();
}

}  // namespace su2
