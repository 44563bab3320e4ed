// heatbath_fp64.cu -- the FP64 row of the launch-shape table: its 14 shapes run
// six kernels (heatbath_fixed.cuh).  The build compiles this file once per
// kernel and sampler, with SU2_KIND = 0 .. 5 and SU2_HYB = 0 or 1, so that
// they compile in parallel.
#include "heatbath_fixed.cuh"

#if !defined(SU2_KIND) || !defined(SU2_HYB)
#error "compile with -DSU2_KIND=<0..5> -DSU2_HYB=<0|1>"
#endif

namespace su2 {

template <int KIND, bool HYB, bool MIR, int MU, bool PLAQ>
static void launch_fix_k(const Ctx& c, const LaunchCfg& f, int parity, int32_t* dbg, cudaStream_t s)
{
    const dim3 grid(c.phase_blocks), block(f.threads);
    if constexpr (KIND == FIX_LINK_255)
        fix_phase_kernel<MU, PLAQ, HYB, MIR, 256, FIX_THREADS[FIX_LINK_255] / 256><<<grid, block, 0, s>>>(c, parity, dbg);
    else if constexpr (KIND == FIX_LINK_96)
        fix_phase_kernel<MU, PLAQ, HYB, MIR, 128, FIX_THREADS[FIX_LINK_96] / 128><<<grid, block, 0, s>>>(c, parity, dbg);
    else if constexpr (KIND == FIX_QUAD_128)
        fix_quad_kernel<MU, PLAQ, HYB, MIR, FIX_THREADS[FIX_QUAD_128] / 128><<<grid, block, 0, s>>>(c, parity, dbg);
    else if constexpr (KIND == FIX_QUAD_72)
        fix_quad_kernel<MU, PLAQ, HYB, MIR, FIX_THREADS[FIX_QUAD_72] / 128><<<grid, block, 0, s>>>(c, parity, dbg);
    else
        fix_queue_kernel<MU, PLAQ, HYB, MIR, KIND == FIX_PERSIST>
            <<<grid, block, 0, s>>>(c, parity, f.rounds, dbg);
}
template <int KIND, bool HYB, int MU, bool PLAQ>
static void launch_fix_mu(const Ctx& c, const LaunchCfg& f, int parity, int32_t* dbg, bool mirror,
                          cudaStream_t s)
{
    if (mirror) launch_fix_k<KIND, HYB, true, MU, PLAQ>(c, f, parity, dbg, s);
    else launch_fix_k<KIND, HYB, false, MU, PLAQ>(c, f, parity, dbg, s);
}

template <int KIND, bool HYB>
cudaError_t launch_fix_kind(const Ctx& c, const LaunchCfg& f, int mu, int parity, bool plaq,
                            int32_t* dbg, bool mirror, cudaStream_t s)
{
    // the fused plaquette exists only in the odd phases with mu >= 1
    const bool pl = plaq && parity == 1 && mu >= 1 && !dbg;
    switch (mu) {
    case 0: launch_fix_mu<KIND, HYB, 0, false>(c, f, parity, dbg, mirror, s); break;
    case 1:
        if (pl) launch_fix_mu<KIND, HYB, 1, true>(c, f, parity, dbg, mirror, s);
        else launch_fix_mu<KIND, HYB, 1, false>(c, f, parity, dbg, mirror, s);
        break;
    case 2:
        if (pl) launch_fix_mu<KIND, HYB, 2, true>(c, f, parity, dbg, mirror, s);
        else launch_fix_mu<KIND, HYB, 2, false>(c, f, parity, dbg, mirror, s);
        break;
    default:
        if (pl) launch_fix_mu<KIND, HYB, 3, true>(c, f, parity, dbg, mirror, s);
        else launch_fix_mu<KIND, HYB, 3, false>(c, f, parity, dbg, mirror, s);
        break;
    }
    return cudaGetLastError();
}

template cudaError_t launch_fix_kind<SU2_KIND, (SU2_HYB != 0)>(const Ctx&, const LaunchCfg&, int, int,
                                                               bool, int32_t*, bool, cudaStream_t);

}  // namespace su2
