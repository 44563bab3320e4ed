// cluster64.cu -- all sweeps of a call on a small FP64 lattice in one launch of
// one thread-block cluster (the FP64 counterpart of hb_chain_kernel).
//
// A phase of a small FP64 lattice is one link's chain of ~2,700 integer
// instructions and a launch.  Here the lattice's links live in the distributed
// shared memory of 16 CTAs as limbs (su2_mirror.cuh's form), and each link
// has four threads, one in each quarter of the block: three form the staple
// terms of one plane each (exact integer sums, so any order gives the same
// bits), the first of them then adds the three, decides and stores; the
// fourth computes the next phase's first trials -- Philox, logarithms,
// cosines, the direction -- in the meantime.  Some of 2048 links reject a
// trial or two in every phase and all wait for them, so two more trials per
// link are drawn ahead, by the two idle plane threads (8^4, beta = 2.3, us a
// sweep with 1, 2, 3, 4 trials ahead: 39.4, 37.4, 36.0, 37.2; phase
// launches of four threads per link: 44.0).  Bound by the integer pipes of 16 SMs:
// ~2,900 instructions per 32 links on 64 sub-partitions.  The stored doubles go straight
// to global memory.  Every value comes from the functions of su2_fixed.cuh,
// and the plaquette partials are summed in launch shape 0's order: links and
// plaquettes are those of the phase launches bit by bit.
//
// A lattice with non-unit links (D.general) runs its sweeps in the FP64
// sequence here, through L2, until all links are unit quaternions; one at a
// coupling above FIX_BETA_MAX runs all of them so.
#include "cluster.cuh"
#include "heatbath_fixed.cuh"

namespace su2 {

constexpr int C64_LINKS = 128;  // threads per quarter: links of a phase per CTA, at most

// drawn ahead for one link: its direction (trial 0's spare bits) and trials
// 0 .. AHEAD - 1 (KpSum, and the word the accept test takes)
constexpr int AHEAD = 3;
struct Chain64Shared {
    int4* own;        // [8][2][C] limbs of the links
    longlong2* sums;  // [3][2][C] staple sums of the three planes
    Trial64* trial;   // [2][AHEAD][C]
    Dir64* dir;       // [2][C]
    uint32_t* addr;   // [2][20][C]
    double* part;     // CTA 0: [2][3 npart]
    __device__ __forceinline__ Chain64Shared(char* base, uint32_t C)
        : own(reinterpret_cast<int4*>(base)), sums(reinterpret_cast<longlong2*>(own + 16 * C)),
          trial(reinterpret_cast<Trial64*>(sums + 6 * C)),
          dir(reinterpret_cast<Dir64*>(trial + 2 * AHEAD * C)),
          addr(reinterpret_cast<uint32_t*>(dir + 2 * C)),
          part(reinterpret_cast<double*>(addr + 40 * C))
    {
    }
};
constexpr size_t chain64_smem(uint32_t C, uint32_t npart)
{
    return (size_t)C * (16 * 16 + 6 * 16 + 2 * AHEAD * 16 + 2 * 32 + 40 * 4) + 2 * 3 * (size_t)npart * 8;
}

// the link whose first half lies at a, C sites per CTA
__device__ __forceinline__ FQuat ld_cluster_fix(uint32_t a, uint32_t C)
{
    int4 u, v;
    // volatile: never moved across the cluster barriers
    asm volatile("ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w) : "r"(a));
    asm volatile("ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a + 16 * C));
    return {{u.x, u.y}, {u.z, u.w}, {v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ void put_fix(int4* a, uint32_t C, const Quat<double>& q)
{
    const FQuat f = fq_link(q);
    a[0] = make_int4(f.a0.h, f.a0.l, f.a1.h, f.a1.l);
    a[C] = make_int4(f.a2.h, f.a2.l, f.a3.h, f.a3.l);
}

// what thread `role` of a link draws for its next update: trial role (roles 1
// and 2), or trial 0 and the direction (role 3)
__device__ __forceinline__ void draw_ahead64(const FixCall& F, const Stream& st, int role, uint32_t C,
                                             Trial64* trial, Dir64* dir)
{
#pragma unroll 1
    for (int t = role == 3 ? 0 : role; t < AHEAD; t += 3) {
        const U4 w = st.draw(TAG_TRIAL, (uint32_t)t);
        const KpSum k = kp_sum(w.x, w.y, w.z, F.tab);
        trial[(size_t)t * C] = {k.t, k.e, w.w};
        if (t == 0) {
            const FixDir d = direction_fix(spare_bits_1(w), spare_bits_2(w), F.tab);
            *dir = {d.sth, d.cph, d.sph, d.cth, 0};
        }
    }
}

// links read through L2 (other SMs write them during the launch)
struct L2Links : Links<double> {
    __device__ __forceinline__ L2Links(void* links, const LatDesc& d, uint32_t* status)
        : Links<double>(links, d, status) {}
    __device__ __forceinline__ Quat<double> load(int mu, int p, uint32_t eo) const
    {
        const double2 lo = __ldcg(base + idx(mu, p, 0, eo)), hi = __ldcg(base + idx(mu, p, 1, eo));
        return {lo.x, lo.y, hi.x, hi.y};
    }
    __device__ __forceinline__ Quat<double> load_rw(int mu, int p, uint32_t eo) const
    {
        return load(mu, p, eo);
    }
};

__global__ void __launch_bounds__(4 * C64_LINKS, 1)
fix_chain_kernel(Ctx ctx, uint32_t C, FastDiv div_c, uint32_t npart, int pl, int nsweeps)
{
    extern __shared__ int4 chain64_mem[];
    __shared__ double scratch[8];
    __shared__ uint32_t bad[CLUSTER_MAX];  // CTA 0: CTAs that saw non-unit links
    constexpr int NL = C64_LINKS;
    LatDesc* const Dw = ctx.desc;
    const LatDesc D = *Dw;  // a register copy (the barriers clobber memory)
    const Chain64Shared sh(reinterpret_cast<char*>(chain64_mem), C);
    const FixCall F(D);
    const uint32_t rank = cluster_rank(), S = gridDim.x, Vh = D.Vh;
    const int role = threadIdx.x / NL;  // 0, 1, 2: plane of the staple (0 finishes); 3: draws ahead
    const uint32_t o = threadIdx.x % NL;
    const uint32_t i = rank * C + o;
    const bool act = o < C && i < Vh;
    const int lane = threadIdx.x & 31, w = (int)(o >> 5);
    const uint64_t sw0 = D.sweep;
    const Links<double> G(ctx.links, D, ctx.status);
    LinkCheck chk;
#ifdef SU2_CHECK_BOUNDS
    chk = {ctx.status, Vh};
#endif
    uint32_t lex[2] = {0, 0};
    if (act) {
        lex[0] = EoSite(D, i, 0).lex();
        lex[1] = EoSite(D, i, 1).lex();
    }
    if (pl && rank == 0)
        for (uint32_t k = threadIdx.x; k < 2 * 3 * npart; k += 4 * NL) sh.part[k] = 0.0;
    cluster_sync();

    uint32_t ntrial = 0, ncap = 0;
    const uint32_t gw = rank * (C >> 5) + (uint32_t)w;
    auto put_partial = [&](int k, int mu, double v) {
        if (lane == 0 && gw < npart && o < C)
            chain_put_partial(sh.part + (size_t)((k & 1) * 3 + mu - 1) * npart + gw, v);
    };
    auto sum_warps = [&](int k) {
        chain_sum_warps(sh.part + (size_t)(k & 1) * 3 * npart, npart, w, NL / 32, scratch);
    };
    auto finish_sum = [&](int k) { chain_finish_sum(ctx, D, scratch, sw0 + (uint64_t)k); };

    // sweeps in the FP64 sequence while some link is not a unit quaternion
    int k = 0;
    for (bool general = D.general != 0; general && k < nsweeps; ++k) {
        LatDesc Dk = D;
        Dk.sweep = sw0 + (uint64_t)k;
        for (int ph = 0; ph < 8; ++ph) {
            const int mu = ph >> 1, p = ph & 1;
            if (role == 0) {
                double plaq = 0.0;
                uint32_t lx;
                if (act) {
                    const int32_t tr = general_link<L2Links>(ctx, Dk, i, mu, p, false, &plaq, &lx);
                    ncap += tr < 0;
                    ntrial += tr < 0 ? (uint32_t)KP_CAP : (uint32_t)tr;
                }
                __syncwarp();
                if (pl && p == 1 && mu >= 1) put_partial(k, mu, warp_sum(plaq));
            }
            __threadfence();
            cluster_sync();
        }
        bool ok = (D.general & GENERAL_BETA) == 0;
        if (ok && role == 0 && act)
            for (int mp = 0; mp < 8; ++mp) {
                const Quat<double> q = G.load_rw(mp >> 1, mp & 1, i);  // this thread's own stores
                if (!unit_link(make_double2(q.a0, q.a1), make_double2(q.a2, q.a3))) ok = false;
            }
        ok = __syncthreads_and(ok);
        if (pl && rank == 0 && role == 3) sum_warps(k);
        if (threadIdx.x < S) {  // every CTA's verdict to every CTA
            uint32_t ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                         : "=r"(ra)
                         : "r"((uint32_t)__cvta_generic_to_shared(&bad[rank])), "r"(threadIdx.x));
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(ra), "r"(ok ? 0u : 1u) : "memory");
        }
        cluster_sync();
        if (pl && rank == 0 && threadIdx.x == 0) finish_sum(k);
        general = false;
        for (uint32_t r = 0; r < S; ++r) general = general || bad[r] != 0;
        cluster_sync();  // bad[] and scratch may be written again
        if (!general && rank == 0 && threadIdx.x == 0) Dw->general = 0u;
    }

    const int k0 = k;  // sweeps k0 .. nsweeps - 1 in fixed point
    if (k0 < nsweeps) {
        if (act) {
            if (role < 2)
                for (int mp = role; mp < 8; mp += 2)
                    put_fix(sh.own + (size_t)(mp * 2) * C + o, C, L2Links(ctx.links, D, ctx.status)
                                                                     .load(mp >> 1, mp & 1, i));
            else
                chain_addresses(D, i, role - 2, C, div_c, (uint32_t)__cvta_generic_to_shared(sh.own),
                                chk, sh.addr + (size_t)(role - 2) * 20 * C + o);
        }
        auto stream = [&](int mu, int p, uint64_t sw) {
            return Stream{F.k0, F.k1, lex[p] * 4u + (uint32_t)mu, (uint32_t)sw, (uint32_t)(sw >> 32)};
        };
        // the draws of the phase (mu, p) of sweep sw
        auto draw = [&](int mu, int p, uint64_t sw) {
            draw_ahead64(F, stream(mu, p, sw), role, C, sh.trial + (size_t)p * AHEAD * C + o,
                         sh.dir + (size_t)p * C + o);
        };
        if (act && role > 0) draw(0, 0, sw0 + (uint64_t)k0);
        cluster_sync();
        for (; k < nsweeps; ++k) {
            const uint64_t sw = sw0 + (uint64_t)k;
#pragma unroll 1
            for (int ph = 0; ph < 8; ++ph) {
                const int mu = ph >> 1, p = ph & 1, q = p ^ 1;
                if (role < 3) {
                    int64_t A[4] = {0, 0, 0, 0};
                    if (act) {
                        const int nu = role + (role >= mu ? 1 : 0);
                        const uint32_t* ad = sh.addr + (size_t)p * 20 * C + o;
                        const uint32_t plane = 32 * C;  // bytes of one (mu, parity)
                        const uint32_t e_pmu = ad[mu * C], e_pnu = ad[nu * C], e_mnu = ad[(4 + nu) * C];
                        const uint32_t e_pmu_mnu = ad[(8 + 3 * mu + role) * C];
                        const int4* c0 = sh.own + (size_t)((nu * 2 + p) * 2) * C + o;
                        const int4 cl = c0[0], ch = c0[C];
                        fq_staple(ld_cluster_fix(e_pmu + (nu * 2 + q) * plane, C),
                                  ld_cluster_fix(e_pnu + (mu * 2 + q) * plane, C),
                                  {{cl.x, cl.y}, {cl.z, cl.w}, {ch.x, ch.y}, {ch.z, ch.w}}, false, A);
                        fq_staple(ld_cluster_fix(e_mnu + (mu * 2 + q) * plane, C),
                                  ld_cluster_fix(e_pmu_mnu + (nu * 2 + p) * plane, C),
                                  ld_cluster_fix(e_mnu + (nu * 2 + q) * plane, C), true, A);
                        if (role > 0) {
                            longlong2* s = sh.sums + (size_t)(role * 2) * C + o;
                            s[0] = make_longlong2(A[0], A[1]);
                            s[C] = make_longlong2(A[2], A[3]);
                        }
                    }
                    __syncwarp();
                    asm volatile("bar.sync 1, %0;" ::"n"(3 * C64_LINKS) : "memory");
                    if (role == 0) {
                        int64_t P[4] = {A[0], A[1], A[2], A[3]}, un[4] = {0, 0, 0, 0};
                        if (act) {
#pragma unroll
                            for (int r = 1; r < 3; ++r) {
                                const longlong2* s = sh.sums + (size_t)(r * 2) * C + o;
                                const longlong2 lo = s[0], hi = s[C];
                                A[0] += lo.x;
                                A[1] += lo.y;
                                A[2] += hi.x;
                                A[3] += hi.y;
                                if (r < mu)
#pragma unroll
                                    for (int c = 0; c < 4; ++c) P[c] = A[c];
                            }
                            const Stream st = stream(mu, p, sw);
                            int4* slot = sh.own + (size_t)((mu * 2 + p) * 2) * C + o;
                            Drawn d;
                            double qc;
                            if (!fix_prepare<false>(F, A, &d, &qc)) {
                                const Quat<double> h = haar_link(st, F.tab);
                                G.store(mu, p, i, h);
                                put_fix(slot, C, h);
                                if (pl) fix_from_link(h, un);
                            } else {
                                Lambda L;
                                uint32_t tr = 0;
#pragma unroll 1
                                for (uint32_t t = 0; t < (uint32_t)AHEAD; ++t) {
                                    const Trial64 a = sh.trial[((size_t)p * AHEAD + t) * C + o];
                                    L = kp_lambda(KpSum{a.t, a.e}, d.inv, d.ei);
                                    if (kp_accept(L, a.w3)) {
                                        tr = t + 1;
                                        break;
                                    }
                                }
                                for (uint32_t t = AHEAD; tr == 0 && t < (uint32_t)KP_CAP; ++t)
                                    if (fix_try<false>(F, st.draw(TAG_TRIAL, t), d.inv, d.ei, 0.0, &L))
                                        tr = t + 1;
                                if (tr) {
                                    const Dir64 dr = sh.dir[(size_t)p * C + o];
                                    new_link_dir_fix(L, {dr.cth, dr.sth, dr.cph, dr.sph}, d.V, un);
                                    const Quat<double> u = dq_link(un);
                                    G.store(mu, p, i, u);
                                    put_fix(slot, C, u);
                                    ntrial += tr;
                                } else {  // cap hit: the link keeps its value
                                    ncap += 1;
                                    ntrial += (uint32_t)KP_CAP;
                                    if (pl) fix_from_link(L2Links(ctx.links, D, ctx.status).load(mu, p, i), un);
                                }
                            }
                        }
                        if (pl && p == 1 && mu >= 1)
                            put_partial(k, mu, plaq_double(warp_sum64(act ? retr_fix(un, P) : 0)));
                    }
                }
                if (role > 0) {
                    if (act && !(ph == 7 && k + 1 == nsweeps))
                        draw((mu + p) & 3, q, ph == 7 ? sw + 1 : sw);
                    if (pl && rank == 0 && role == 3 && k > k0) {
                        if (ph == 0) sum_warps(k - 1);
                        else if (ph == 1 && o == 0) finish_sum(k - 1);
                    }
                }
                cluster_sync();
            }
        }
    }

    if (role == 0) {
        const uint32_t wt = __reduce_add_sync(0xffffffffu, ntrial);
        const uint32_t wc = __reduce_add_sync(0xffffffffu, ncap);
        if (lane == 0) {
            atomicAdd(ctx.trial_slots + ((rank * (NL / 32) + (uint32_t)w) % TRIAL_SLOTS),
                      (unsigned long long)wt);
            if (wc) {
                atomicAdd(&Dw->caps, (unsigned long long)wc);
                atomicOr(ctx.status, STATUS_CAP_HIT);
            }
        }
    }
    if (rank == 0) {
        const bool last = pl && k0 < nsweeps;
        if (last) {
            if (role == 3) sum_warps(nsweeps - 1);
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            if (last) finish_sum(nsweeps - 1);
            atomicAdd(&Dw->updates, 8ull * (unsigned long long)Vh * (unsigned long long)nsweeps);
            Dw->sweep = sw0 + (uint64_t)nsweeps;
        }
    }
}

bool chain64_geometry(uint32_t Vh, ChainGeom* g)
{
    const uint32_t C = ((Vh + CLUSTER_MAX - 1) / CLUSTER_MAX + 31) & ~31u;
    if (C > (uint32_t)C64_LINKS) return false;
    g->S = CLUSTER_MAX;
    g->C = C;
    g->div_c = make_fastdiv(C);
    g->updaters = C64_LINKS;
    g->npart = (Vh + 255) / 256 * 8;  // launch shape 0: blocks of 256 threads
    g->smem = chain64_smem(C, g->npart);
    return 3 * g->npart <= (uint32_t)SWEEP_CHUNK;
}

static_assert(chain64_smem(C64_LINKS, SWEEP_CHUNK / 3) + 128 <= 227 * 1024, "the largest geometry fits an SM");

static cudaError_t chain64_config(const ChainGeom& g, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at)
{
    const cudaError_t e =
        allow_cluster((const void*)fix_chain_kernel,
                      chain64_smem((uint32_t)C64_LINKS, (uint32_t)SWEEP_CHUNK / 3));
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3((unsigned)g.S);
    cfg->blockDim = dim3((unsigned)(4 * C64_LINKS));
    cfg->dynamicSmemBytes = g.smem;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)g.S;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return e;
}
bool chain64_launchable(const ChainGeom& g)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    int n = 0;
    if (chain64_config(g, &cfg, at) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, fix_chain_kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n >= 1;
}
cudaError_t launch_chain64(const Ctx& c, const ChainGeom& g, bool plaq, int nsweeps, cudaStream_t s)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    if (cudaError_t e = chain64_config(g, &cfg, at)) return e;
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, fix_chain_kernel, c, g.C, g.div_c, g.npart, plaq ? 1 : 0, nsweeps);
}

}  // namespace su2
