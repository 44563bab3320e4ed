// cluster.cu -- one heat-bath sweep of a small FP32 lattice in one launch,
// the whole lattice held in the distributed shared memory of one
// thread-block cluster.
//
// A small lattice (8^4: 2048 link updates per phase) spends most of a sweep
// in launch gaps and in the dependent chain of one update, not in memory
// traffic.  Here the CTAs of one cluster (up to 16 SMs) copy the lattice's
// links from global memory into their shared memory, run the eight
// checkerboard phases with the hardware cluster barrier between them (no
// global-memory flag, no spin), finish the sweep (the fused plaquette in a
// fixed order, the sweep counter) and copy the links back: one launch per
// sweep instead of nine.  Every link is updated by update_link, the body of
// the one-link-per-thread kernel, on the same random streams, so the links
// are bit-identical to every other FP32 launch shape.
//
// Layout: CTA r of a cluster of S holds, for each (mu, parity), the links
// eo in [r C, (r + 1) C), C = Vh / S, as float4s at shared-memory offset
// (mu 2 + parity) C + (eo - r C).  A neighbour link of another CTA is read
// with mapa + ld.shared::cluster; a CTA writes only its own links.
#include "cluster.cuh"
#include "heatbath_kernel.cuh"

namespace su2 {

// the links of the cluster, read where they live; written by their owner
struct ClusterLinks {
    uint32_t base;  // shared-window address of this CTA's links
    uint32_t C;     // links per (mu, parity) per CTA
    FastDiv div_c;
    LinkCheck chk;  // bounds-checked builds: a bad index is recorded, link 0 read
    static constexpr int UNIT = 1;
    __device__ __forceinline__ Quat<float> load_at(int mu, int p, uint32_t eo) const
    {
        if (!chk.ok(mu, p, eo)) eo = 0;
        const uint32_t r = fdiv(eo, div_c);
        const uint32_t a = base + (((uint32_t)(mu * 2 + p) * C + (eo - r * C)) << 4);
        uint32_t ra;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(r));
        float4 v;
        // volatile: never moved across the cluster barriers
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"(ra));
        return {v.x, v.y, v.z, v.w};
    }
};

// One phase (MU, p) on this CTA's links: thread t updates eo = r C + t,
// r C + t + NT, ...; the plaquette part of the staple (PLAQ) goes into the
// warp's FP64 partial, lane 0.
template <int MU, bool PLAQ, bool HYB, int NT>
__device__ __forceinline__ void cluster_phase(const LatDesc& D, const ClusterLinks& CU, float4* own,
                                              uint32_t rank, int p, uint64_t sw, double& wplaq,
                                              uint32_t& ntrial, uint32_t& ncap)
{
    const uint32_t C = CU.C;
    float plaq = 0.0f;
    for (uint32_t o = threadIdx.x; o < C; o += NT) {
        const uint32_t i = rank * C + o;
        const EoSite s(D, i, p);
        Quat<float> un, P;
        const int32_t tr = update_link<float, MU, PLAQ, HYB>(CU, D, s, i, p, sw, &un, &P);
        float4& slot = own[(uint32_t)(MU * 2 + p) * C + o];
        if (tr >= 0) {
            slot = make_float4(un.a0, un.a1, un.a2, un.a3);
        } else {
            ++ncap;
            if (PLAQ) un = {slot.x, slot.y, slot.z, slot.w};
        }
        ntrial += tr > 0 ? (uint32_t)tr : (tr < 0 ? (uint32_t)KP_CAP : 0u);
        if (PLAQ) plaq = add_(plaq, qretr(un, P));
    }
    if (PLAQ) {
        const float wp = warp_sum_t(plaq);
        if ((threadIdx.x & 31) == 0) wplaq += (double)wp;
    }
}

template <int MU, bool HYB, int NT>
__device__ __forceinline__ void cluster_mu(const LatDesc& D, const ClusterLinks& CU, float4* own,
                                           uint32_t rank, uint64_t sw, bool pl, double& wplaq,
                                           uint32_t& ntrial, uint32_t& ncap)
{
    cluster_phase<MU, false, HYB, NT>(D, CU, own, rank, 0, sw, wplaq, ntrial, ncap);
    cluster_sync();
    if (MU >= 1 && pl)
        cluster_phase<MU, (MU >= 1), HYB, NT>(D, CU, own, rank, 1, sw, wplaq, ntrial, ncap);
    else
        cluster_phase<MU, false, HYB, NT>(D, CU, own, rank, 1, sw, wplaq, ntrial, ncap);
    cluster_sync();
}

// One sweep of lattice 0 of a single-lattice handle.  Grid: one cluster of
// S CTAs of NT threads, 8 C float4s of dynamic shared memory per CTA.
template <bool HYB, int NT>
__global__ void __launch_bounds__(NT, 1)
hb_cluster_kernel(Ctx ctx, uint32_t C, FastDiv div_c, int pl)
{
    extern __shared__ float4 own[];
    __shared__ double wsum[NT / 32];
    __shared__ double cta_part[CLUSTER_MAX];
    LatDesc* const Dw = ctx.desc;
    // a register copy: the barriers' memory clobbers would otherwise reload
    // the geometry and the coupling from global memory in every phase
    const LatDesc D = *Dw;
    const uint32_t rank = cluster_rank();
    const uint32_t S = gridDim.x;
    const uint32_t Vh = D.Vh;
    const uint64_t sw = D.sweep;
    float4* const glob = reinterpret_cast<float4*>(static_cast<char*>(ctx.links) + D.link_off);

    for (uint32_t k = threadIdx.x; k < 8 * C; k += NT) {
        const uint32_t mp = k / C;
        own[k] = glob[(size_t)mp * Vh + rank * C + (k - mp * C)];
    }
    cluster_sync();  // every CTA's links are in place

    ClusterLinks CU{(uint32_t)__cvta_generic_to_shared(own), C, div_c, {}};
#ifdef SU2_CHECK_BOUNDS
    CU.chk = {ctx.status, Vh};
#endif
    double wplaq = 0.0;
    uint32_t ntrial = 0, ncap = 0;
    const bool plq = pl != 0;
    cluster_mu<0, HYB, NT>(D, CU, own, rank, sw, plq, wplaq, ntrial, ncap);
    cluster_mu<1, HYB, NT>(D, CU, own, rank, sw, plq, wplaq, ntrial, ncap);
    cluster_mu<2, HYB, NT>(D, CU, own, rank, sw, plq, wplaq, ntrial, ncap);
    cluster_mu<3, HYB, NT>(D, CU, own, rank, sw, plq, wplaq, ntrial, ncap);

    // links back to global memory (own links only: no remote reads left)
    for (uint32_t k = threadIdx.x; k < 8 * C; k += NT) {
        const uint32_t mp = k / C;
        glob[(size_t)mp * Vh + rank * C + (k - mp * C)] = own[k];
    }
    // trial counts and cap hits, as the phase kernels count them
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t wt = __reduce_add_sync(0xffffffffu, ntrial);
    const uint32_t wc = __reduce_add_sync(0xffffffffu, ncap);
    if (lane == 0) {
        const uint32_t gw = rank * (NT / 32) + w;
        atomicAdd(ctx.trial_slots + (gw % TRIAL_SLOTS), (unsigned long long)wt);
        if (wc) {
            atomicAdd(&Dw->caps, (unsigned long long)wc);
            atomicOr(ctx.status, STATUS_CAP_HIT);
        }
    }
    // the fused plaquette: warps in order, then CTAs in order on CTA 0
    if (plq) {
        if (lane == 0) wsum[w] = wplaq;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int k = 0; k < NT / 32; ++k) t += wsum[k];
            const uint32_t a = (uint32_t)__cvta_generic_to_shared(&cta_part[rank]);
            uint32_t ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(0u));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(t) : "memory");
        }
    }
    cluster_sync();  // the CTAs' sums are on CTA 0; nobody reads remote memory after this
    if (rank == 0 && threadIdx.x == 0) {
        atomicAdd(&Dw->updates, 8ull * (unsigned long long)Vh);
        if (plq) {
            double tot = 0.0;
            for (uint32_t r = 0; r < S; ++r) tot += cta_part[r];
            const double P = tot / (6.0 * (double)D.V);
            const uint64_t k = sw - D.sweep_base;
            ctx.ring[k % PLAQ_RING] = P;
            if (D.plaq_out) D.plaq_out[k] = P;
        }
        Dw->sweep = sw + 1;
    }
}

// ---------------------------------------------------------------------------
// all sweeps of a call in one launch, draws computed ahead
// ---------------------------------------------------------------------------
// The chain kernel runs every sweep of a call on a lattice whose share per CTA
// is at most 512 links of each (mu, parity).  A phase of a small lattice lasts
// as long as one link's chain of instructions, so the chain is cut:
//   * half the threads (the updaters, one link each) form the staple, decide
//     and store; the other half (the drawers) compute the next phase's first
//     trials in the meantime -- Philox, both logarithms, the cosine, the
//     direction, everything that does not depend on the links -- and leave
//     them in shared memory;
//   * the shared-memory addresses of a link's 20 neighbour sites of either
//     parity are computed once per launch (a neighbour of another CTA is one
//     mapa away) and read from a table;
//   * the cluster barrier between the phases is the only synchronisation.
// The FP32 operations are those of staple_sum and draw_link, in their order, so
// the links are the other kernels' bit by bit.  C is a multiple of 32: the
// warps hold the same 32 links as launch shape 0's, and the plaquette
// partials are summed in that shape's order (sweep_end_kernel's), so its
// plaquettes are reproduced bit by bit too.
// Measured per sweep with the plaquette (beta = 2.4): 8^4 12.2 us (28.7 in
// launch shape 0's phase launches, 22.6 in the whole-sweep kernel above),
// 10^3 x 6 13.8 (28.7), 12^3 x 8 23.1 (28.8), 4^4 9.5.  A phase takes 1.2 us at
// 4^4, one update's remaining chain and the barrier, and grows with the links
// a CTA updates: 1.5 us at 128 (8^4), 1.7 at 192, 2.9 at 448.  (With only the
// first trial drawn ahead 8^4 took 13.0: some link rejects it in every phase,
// and all wait.)
struct ChainShared {
    float4* own;       // [8][C] links
    float4* tdir;      // [2][C] (t, r4^2, cos theta, sin theta) of the coming phase
    float2* phi;       // [2][C] (sin phi, cos phi)
    float2* second;    // [2][C] (t, r4^2) of the second trial
    uint32_t* addr;    // [2][20][C] site addresses: plus 0..3, minus 4..7, 8 + 3 mu + k:
                       // x + mu - nu, nu the k-th direction other than mu
    double* part;      // CTA 0: [2][3 npart] plaquette partials
    __device__ __forceinline__ ChainShared(char* base, uint32_t C)
        : own(reinterpret_cast<float4*>(base)), tdir(own + 8 * C),
          phi(reinterpret_cast<float2*>(tdir + 2 * C)), second(phi + 2 * C),
          addr(reinterpret_cast<uint32_t*>(second + 2 * C)),
          part(reinterpret_cast<double*>(addr + 40 * C))
    {
    }
};
constexpr size_t chain_smem(uint32_t C, uint32_t npart)
{
    return (size_t)C * (8 * 16 + 2 * 16 + 4 * 8 + 40 * 4) + 2 * 3 * (size_t)npart * 8;
}

__device__ __forceinline__ Quat<float> ld_cluster(uint32_t a)
{
    float4 v;
    // volatile: never moved across the cluster barriers
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a));
    return {v.x, v.y, v.z, v.w};
}

// The first two trials of a link as far as they go without the staple:
// kp_eval's lambda^2 = t / (2 alpha), accepted iff r4^2 <= 1 - lambda^2
__device__ __forceinline__ float2 trial_ahead(const U4& w)
{
    const float t = neg_(fma_(Math<float>::cos2pi_sq(u01<float>(w.y)), Math<float>::ln_u01(u01<float>(w.z)),
                              Math<float>::ln_u01(u01<float>(w.x))));
    const float r4 = u01<float>(w.w);
    return make_float2(t, mul_(r4, r4));
}
__device__ __forceinline__ void draw_ahead(const Stream& st, float4* tdir, float2* phi, float2* second)
{
    const U4 w = st.draw(TAG_TRIAL, 0u);
    const float2 t = trial_ahead(w);
    // new_link_u, new_link_dir: the direction
    const float cth = fma_(2.0f, u18<float>(spare_bits_1(w)), -1.0f);
    const float sth = Math<float>::sqrt_pos(mul_(add_(1.0f, neg_(cth)), add_(1.0f, cth)));
    float sph, cph;
    Math<float>::sincos2pi(u18<float>(spare_bits_2(w)), &sph, &cph);
    *tdir = make_float4(t.x, t.y, cth, sth);
    *phi = make_float2(sph, cph);
    *second = trial_ahead(st.draw(TAG_TRIAL, 1u));
}

// phase (MU, p) on this thread's link o
template <int MU>
__device__ __forceinline__ void chain_phase(const ChainShared& sh, const LatDesc& D, uint32_t C,
                                            uint32_t o, int p, uint32_t key, uint64_t sw,
                                            const float4& td, const float2& ph, Quat<float>& P,
                                            Quat<float>& un, uint32_t& ntrial, uint32_t& ncap)
{
    const int q = p ^ 1;
    const uint32_t* ad = sh.addr + (size_t)p * 20 * C + o;
    const uint32_t plane = C * 16;  // bytes from one (mu, parity) to the next
    const uint32_t e_pmu = ad[MU * C];
    Quat<float> A = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int nu = nu_of<MU>(k);
        const uint32_t e_pnu = ad[nu * C], e_mnu = ad[(4 + nu) * C];
        const uint32_t e_pmu_mnu = ad[(8 + 3 * MU + k) * C];
        const float4 cc = sh.own[(nu * 2 + p) * C + o];
        const Quat<float> a = ld_cluster(e_pmu + (nu * 2 + q) * plane);      // U_nu(x+mu)
        const Quat<float> b = ld_cluster(e_pnu + (MU * 2 + q) * plane);      // U_mu(x+nu)
        const Quat<float> c = {cc.x, cc.y, cc.z, cc.w};                      // U_nu(x)
        const Quat<float> d = ld_cluster(e_pmu_mnu + (nu * 2 + p) * plane);  // U_nu(x+mu-nu)
        const Quat<float> e = ld_cluster(e_mnu + (MU * 2 + q) * plane);      // U_mu(x-nu)
        const Quat<float> f = ld_cluster(e_mnu + (nu * 2 + q) * plane);      // U_nu(x-nu)
        A = qmul_dn_acc(qmul(e, d), f, qmul_nd_acc(qmul_nd(a, b), c, A));
        if (nu == MU - 1) P = A;
    }
    // draw_link on the values drawn ahead
    const float k2 = qnorm2(A);
    const float rk = Math<float>::rsqrt(k2);
    const float alpha = mul_(mul_(D.beta_f, k2), rk);
    const Stream st{(uint32_t)D.seed, (uint32_t)(D.seed >> 32), key, (uint32_t)sw, (uint32_t)(sw >> 32)};
    float4& slot = sh.own[(MU * 2 + p) * C + o];
    if (!(alpha >= alpha_haar<float>())) {
        un = haar_from<float>(st.draw(TAG_DIRECTION, 0));
        slot = make_float4(un.a0, un.a1, un.a2, un.a3);
        return;
    }
    const float inv2a = mul_(rk, D.half_inv_beta_f);
    const float lam2 = mul_(td.x, inv2a);
    float delta = add_(lam2, lam2);
    uint32_t tr = 1;
    if (!(td.y <= add_(1.0f, neg_(lam2)))) {
        const float2 t2 = sh.second[p * C + o];
        const float l2 = mul_(t2.x, inv2a);
        delta = add_(l2, l2);
        tr = t2.y <= add_(1.0f, neg_(l2)) ? 2 : 0;
        for (uint32_t t = 2; tr == 0 && t < (uint32_t)KP_CAP; ++t)
            if (kp_try(st.draw(TAG_TRIAL, t), inv2a, &delta)) tr = t + 1;
    }
    if (tr == 0) {  // cap hit: the link keeps its value
        un = {slot.x, slot.y, slot.z, slot.w};
        ncap += 1;
        ntrial += (uint32_t)KP_CAP;
        return;
    }
    ntrial += tr;
    const float vl = Math<float>::sqrt_pos(mul_(delta, add_(2.0f, neg_(delta))));
    const float vs = mul_(vl, td.w);
    const Quat<float> X = {add_(1.0f, neg_(delta)), mul_(vs, ph.y), mul_(vs, ph.x), mul_(vl, td.z)};
    un = qnormalise(qmul_nd(X, A));
    slot = make_float4(un.a0, un.a1, un.a2, un.a3);
}

// nsweeps sweeps of a single-lattice handle.  Grid: one cluster of CTAs of NU
// updaters and NU drawers (NU >= C); npart: launch shape 0's warps per phase.
template <int NU>
__global__ void __launch_bounds__(2 * NU, 1)
hb_chain_kernel(Ctx ctx, uint32_t C, FastDiv div_c, uint32_t npart, int pl, int nsweeps)
{
    extern __shared__ float4 chain_mem[];
    __shared__ double scratch[8];
    LatDesc* const Dw = ctx.desc;
    const LatDesc D = *Dw;  // a register copy (the barriers clobber memory)
    const ChainShared sh(reinterpret_cast<char*>(chain_mem), C);
    const uint32_t rank = cluster_rank(), Vh = D.Vh;
    const bool updater = threadIdx.x < NU;
    const uint32_t o = updater ? threadIdx.x : threadIdx.x - NU;
    const uint32_t i = rank * C + o;
    const bool act = o < C && i < Vh;
    const int lane = threadIdx.x & 31, w = (int)(o >> 5);
    const uint64_t sw0 = D.sweep;
    float4* const glob = reinterpret_cast<float4*>(static_cast<char*>(ctx.links) + D.link_off);
    LinkCheck chk;
#ifdef SU2_CHECK_BOUNDS
    chk = {ctx.status, Vh};
#endif

    // the links; each half of the threads fills one parity's address table
    if (act && updater)
        for (int mp = 0; mp < 8; ++mp) sh.own[mp * C + o] = glob[(size_t)mp * Vh + i];
    uint32_t lex[2] = {0, 0};
    if (act) {
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(sh.own);
        lex[0] = EoSite(D, i, 0).lex();
        lex[1] = EoSite(D, i, 1).lex();
        const int p = updater ? 0 : 1;
        chain_addresses(D, i, p, C, div_c, base, chk, sh.addr + (size_t)p * 20 * C + o);
    }
    if (pl && rank == 0)
        for (uint32_t k = threadIdx.x; k < 2 * 3 * npart; k += 2 * NU) sh.part[k] = 0.0;
    auto stream = [&](int mu, int p, uint64_t sw) {
        return Stream{(uint32_t)D.seed, (uint32_t)(D.seed >> 32), lex[p] * 4u + (uint32_t)mu,
                      (uint32_t)sw, (uint32_t)(sw >> 32)};
    };
    if (act && !updater) draw_ahead(stream(0, 0, sw0), sh.tdir + o, sh.phi + o, sh.second + o);
    cluster_sync();

    uint32_t ntrial = 0, ncap = 0;
    auto sum_warps = [&](int k) {
        chain_sum_warps(sh.part + (size_t)(k & 1) * 3 * npart, npart, w, NU / 32, scratch);
    };
    auto finish_sum = [&](int k) { chain_finish_sum(ctx, D, scratch, sw0 + (uint64_t)k); };
    for (int k = 0; k < nsweeps; ++k) {
        const uint64_t sw = sw0 + (uint64_t)k;
#pragma unroll 1
        for (int ph8 = 0; ph8 < 8; ++ph8) {
            const int mu = ph8 >> 1, p = ph8 & 1;
            if (updater) {
                Quat<float> P = {0.f, 0.f, 0.f, 0.f}, un = P;
                if (act) {
                    const float4 td = sh.tdir[p * C + o];
                    const float2 ph = sh.phi[p * C + o];
                    const uint32_t key = lex[p] * 4u + (uint32_t)mu;
                    switch (mu) {
                    case 0: chain_phase<0>(sh, D, C, o, p, key, sw, td, ph, P, un, ntrial, ncap); break;
                    case 1: chain_phase<1>(sh, D, C, o, p, key, sw, td, ph, P, un, ntrial, ncap); break;
                    case 2: chain_phase<2>(sh, D, C, o, p, key, sw, td, ph, P, un, ntrial, ncap); break;
                    default: chain_phase<3>(sh, D, C, o, p, key, sw, td, ph, P, un, ntrial, ncap); break;
                    }
                }
                if (pl && p == 1 && mu >= 1) {
                    const float wp = warp_sum_t(act ? qretr(un, P) : 0.0f);
                    const uint32_t gw = rank * (C >> 5) + (uint32_t)w;
                    if (lane == 0 && gw < npart && o < C)
                        chain_put_partial(sh.part + (size_t)((k & 1) * 3 + mu - 1) * npart + gw,
                                          (double)wp);
                }
            } else {
                if (act && !(ph8 == 7 && k + 1 == nsweeps)) {
                    const int np = p ^ 1, nmu = (mu + p) & 3;
                    draw_ahead(stream(nmu, np, ph8 == 7 ? sw + 1 : sw), sh.tdir + np * C + o,
                               sh.phi + np * C + o, sh.second + np * C + o);
                }
                if (pl && rank == 0 && k > 0) {
                    if (ph8 == 0) sum_warps(k - 1);
                    else if (ph8 == 1 && threadIdx.x == NU) finish_sum(k - 1);
                }
            }
            cluster_sync();
        }
    }

    // links back to global memory (no remote accesses after the last barrier)
    if (act && updater)
        for (int mp = 0; mp < 8; ++mp) glob[(size_t)mp * Vh + i] = sh.own[mp * C + o];
    if (updater) {
        const uint32_t wt = __reduce_add_sync(0xffffffffu, ntrial);
        const uint32_t wc = __reduce_add_sync(0xffffffffu, ncap);
        if (lane == 0) {
            const uint32_t gw = rank * (NU / 32) + (uint32_t)w;
            atomicAdd(ctx.trial_slots + (gw % TRIAL_SLOTS), (unsigned long long)wt);
            if (wc) {
                atomicAdd(&Dw->caps, (unsigned long long)wc);
                atomicOr(ctx.status, STATUS_CAP_HIT);
            }
        }
    }
    if (rank == 0) {
        if (pl) {
            if (!updater) sum_warps(nsweeps - 1);
            __syncthreads();
        }
        if (threadIdx.x == NU) {
            if (pl) finish_sum(nsweeps - 1);
            atomicAdd(&Dw->updates, 8ull * (unsigned long long)Vh * (unsigned long long)nsweeps);
            Dw->sweep = sw0 + (uint64_t)nsweeps;
        }
    }
}

bool chain_geometry(uint32_t Vh, int S, ChainGeom* g)
{
    const uint32_t C = ((Vh + (uint32_t)S - 1) / (uint32_t)S + 31) & ~31u;
    if (C > 512) return false;
    g->S = S;
    g->C = C;
    g->div_c = make_fastdiv(C);
    g->updaters = C <= 128 ? 128 : (C <= 256 ? 256 : 512);
    g->npart = (Vh + 255) / 256 * 8;  // launch shape 0: blocks of 256 threads
    g->smem = chain_smem(C, g->npart);
    return 3 * g->npart <= (uint32_t)SWEEP_CHUNK;
}

static_assert(chain_smem(512, SWEEP_CHUNK / 3) + 64 <= 227 * 1024, "the largest geometry fits an SM");

static const void* chain_kernel(const ChainGeom& g)
{
    return g.updaters == 128   ? (const void*)hb_chain_kernel<128>
           : g.updaters == 256 ? (const void*)hb_chain_kernel<256>
                               : (const void*)hb_chain_kernel<512>;
}
static cudaError_t chain_config(const ChainGeom& g, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at)
{
    const cudaError_t e = allow_cluster(
        chain_kernel(g), chain_smem((uint32_t)g.updaters, (uint32_t)SWEEP_CHUNK / 3));
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3((unsigned)g.S);
    cfg->blockDim = dim3((unsigned)(2 * g.updaters));
    cfg->dynamicSmemBytes = g.smem;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)g.S;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return e;
}

bool chain_launchable(const ChainGeom& g)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    int n = 0;
    if (chain_config(g, &cfg, at) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, chain_kernel(g), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n >= 1;
}

cudaError_t launch_chain(const Ctx& c, const ChainGeom& g, bool plaq, int nsweeps, cudaStream_t s)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    if (cudaError_t e = chain_config(g, &cfg, at)) return e;
    cfg.stream = s;
    const int pl = plaq ? 1 : 0;
    if (g.updaters == 128)
        return cudaLaunchKernelEx(&cfg, hb_chain_kernel<128>, c, g.C, g.div_c, g.npart, pl, nsweeps);
    if (g.updaters == 256)
        return cudaLaunchKernelEx(&cfg, hb_chain_kernel<256>, c, g.C, g.div_c, g.npart, pl, nsweeps);
    return cudaLaunchKernelEx(&cfg, hb_chain_kernel<512>, c, g.C, g.div_c, g.npart, pl, nsweeps);
}

// dynamic shared memory of a CTA of the current device beside the whole-sweep
// kernel's static part (warp and CTA partials); 0 if unknown
static size_t cluster_room()
{
    int max_smem = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
            cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return (size_t)max_smem - 8 * (1024 / 32) - 8 * CLUSTER_MAX;
}

// cluster size and shared memory for lattice 0, or false when the lattice
// does not fit: the largest S in {16, 8, 4, 2} dividing Vh whose share of
// the links fits a CTA
bool cluster_geometry(uint32_t Vh, int dtype_f32, int n, ClusterGeom* g)
{
    if (!dtype_f32 || n != 1) return false;
    const size_t room = cluster_room();
    for (int S = CLUSTER_MAX; S >= 2; S /= 2) {
        if (Vh % (uint32_t)S) continue;
        const uint32_t C = Vh / (uint32_t)S;
        if ((size_t)8 * C * sizeof(float4) > room) continue;
        g->S = S;
        g->C = C;
        g->div_c = make_fastdiv(C);
        g->threads = C <= 128 ? 128 : 1024;
        g->smem = (size_t)8 * C * sizeof(float4);
        return true;
    }
    return false;
}

template <bool HYB, int NT>
static cudaError_t launch_cluster_nt(const Ctx& c, const ClusterGeom& g, bool plaq, cudaStream_t s)
{
    auto k = hb_cluster_kernel<HYB, NT>;
    if (cudaError_t e = allow_cluster((const void*)k, cluster_room())) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.S);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)g.S;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, c, g.C, g.div_c, plaq ? 1 : 0);
}

cudaError_t launch_cluster_sweep(const Ctx& c, const ClusterGeom& g, bool plaq, bool hyb,
                                 cudaStream_t s)
{
    if (g.threads == 128)
        return hyb ? launch_cluster_nt<true, 128>(c, g, plaq, s)
                   : launch_cluster_nt<false, 128>(c, g, plaq, s);
    return hyb ? launch_cluster_nt<true, 1024>(c, g, plaq, s)
               : launch_cluster_nt<false, 1024>(c, g, plaq, s);
}

// whether one cluster of g.S CTAs with this shared memory can be resident
bool cluster_launchable(const ClusterGeom& g)
{
    auto k = g.threads == 128 ? hb_cluster_kernel<false, 128> : hb_cluster_kernel<false, 1024>;
    if (allow_cluster((const void*)k, cluster_room()) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.S);
    cfg.blockDim = dim3((unsigned)g.threads);
    cfg.dynamicSmemBytes = g.smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)g.S;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nclusters = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&nclusters, k, &cfg);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return nclusters >= 1;
}

}  // namespace su2
