// cluster.cuh -- pieces of the kernels that hold a small lattice in the
// distributed shared memory of one thread-block cluster.
#pragma once
#include "su2_internal.h"
#include "su2_links.cuh"
#include "su2_reduce.cuh"

namespace su2 {

// all threads of all CTAs of the cluster; the release/acquire pair orders
// every shared-memory write before it with every read after it
__device__ __forceinline__ void cluster_sync()
{
    __syncwarp();  // .aligned: the warp arrives together
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Lets kernel k run in clusters of 16 CTAs of up to max_smem bytes of dynamic
// shared memory.  The limits belong to the kernel, not to a launch: max_smem
// is the most any lattice asks of k, one value for all of them, so that a
// host thread of another lattice never lowers the limit under a launch.
inline cudaError_t allow_cluster(const void* k, size_t max_smem)
{
    if (max_smem == 0) return cudaErrorInvalidDevice;  // (cluster_room: the device did not answer)
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e != cudaSuccess
               ? e
               : cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem);
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// The shared-memory addresses of the 20 neighbour sites of site i of parity p,
// for links stored 16 bytes apart from `base` on, C sites per CTA: plus hops
// 0..3, minus hops 4..7, then 8 + 3 mu + k: x + mu - nu, nu the k-th
// direction other than mu.  ad: entry 0 of this site, entries C apart.
__device__ __forceinline__ void chain_addresses(const LatDesc& D, uint32_t i, int p, uint32_t C,
                                                const FastDiv& div_c, uint32_t base,
                                                const LinkCheck& chk, uint32_t* ad)
{
    const EoSite s(D, i, p);
    uint32_t hp[4], hm[4];
    s.hops(hp, hm);
    auto put = [&](int slot, uint32_t e) {
        if (!chk.ok(0, 0, e)) e = 0;
        const uint32_t r = fdiv(e, div_c);
        uint32_t ra;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(base + ((e - r * C) << 4)), "r"(r));
        ad[slot * C] = ra;
    };
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        put(m, i + hp[m]);
        put(4 + m, i + hm[m]);
        for (int k = 0; k < 3; ++k) put(8 + 3 * m + k, i + hp[m] + hm[k + (k >= m ? 1 : 0)]);
    }
}

// a warp's plaquette partial into the same place of CTA 0's shared memory
__device__ __forceinline__ void chain_put_partial(double* slot, double v)
{
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(ra) : "r"((uint32_t)__cvta_generic_to_shared(slot)), "r"(0u));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}
// sweep_end_kernel's sum of a sweep's 3 npart partials (one chunk of 256
// threads) in two steps a barrier apart: nw warps stand in for its eight, then
// one thread adds the warps in order and writes the plaquette of sweep sw
__device__ __forceinline__ void chain_sum_warps(const double* part, uint32_t npart, int w, int nw,
                                                double* scratch)
{
    const int lane = threadIdx.x & 31;
    for (int vw = w; vw < 8; vw += nw) {
        double acc = 0.0;
        for (uint32_t e = vw * 32 + lane; e < 3 * npart; e += 256) acc += part[e];
        acc = warp_sum(acc);
        if (lane == 0) scratch[vw] = acc;
    }
}
__device__ __forceinline__ void chain_finish_sum(const Ctx& ctx, const LatDesc& D,
                                                 const double* scratch, uint64_t sw)
{
    double tot = 0.0;
    for (int vw = 0; vw < 8; ++vw) tot += scratch[vw];
    const double P = tot / (6.0 * (double)D.V);
    const uint64_t at = sw - D.sweep_base;
    ctx.ring[at % PLAQ_RING] = P;
    if (D.plaq_out) D.plaq_out[at] = P;
}

}  // namespace su2
