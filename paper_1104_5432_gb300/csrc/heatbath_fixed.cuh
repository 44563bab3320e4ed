// heatbath_fixed.cuh -- the FP64 phase kernels: links stored as doubles,
// updated in 64-bit fixed point (su2_fixed.cuh), in the three forms of the
// launch-shape table: one link per thread, R links per thread with a
// per-warp retry queue, four threads per link.
//
// An FP64 warp instruction holds its SM sub-partition for ~76 clocks on
// GB300, an IMAD.WIDE or a logic operation for 2, so the FP64 sequence
// (general_link: ~270 FP64 instructions, 20,600 clocks per warp) was
// bound by the FP64 unit alone: 1.66 G link updates/s at 64^4, beta = 2.5,
// whatever the shape.  The integer update issues ~2,730 instructions per
// 32 links, 1,360 to 1,490 of them on the multiply pipe, which is busy 2.8 to
// 3.2 clocks for each (32^4, by its counters: a product takes 2, one with a
// 64-bit addend more), i.e. ~4,500 clocks of it, and ~1,090 on the ALU pipe.
// With that pipe 79 to 82% busy it runs at 7.16 G/s at 64^4 (R = 8 or 16, 24
// blocks a SM; 6.76 with 16) and 6.3 G/s at 32^4, beta = 6.0 (one link per
// thread, from 1.57); without the fixed-point copy of the links 5.76 and 5.22.  All forms call the same
// functions on integers, so links and trial counts are bit-identical between
// them.
//
// The fixed-point ranges hold for unit links.  unit_check_kernel looks at
// every link before the sweeps of a call and sweep_end_kernel again after
// each sweep of a lattice that failed; such a lattice, and one at a coupling
// above FIX_BETA_MAX (D.general), takes the FP64 sequence, one link per
// thread, in the same kernels.  A single phase is launched without that look
// (a pass over all links and the parameters' launch before it: 8^4 15.5 us a
// phase, 16^4 22.7, 64^4 1652): each update looks at the 18 links it reads, and
// a link with a neighbour that fails takes the FP64 sequence by itself (7.4,
// 13.6, 1480).
#pragma once
#include "heatbath_kernel.cuh"
#include "su2_mirror.cuh"

namespace su2 {

// An FP64 lattice's links: neighbours read as limbs, from the fixed-point copy
// (MIR) or from the doubles; the stored values are doubles.
template <bool MIR> struct FixLinks;
template <> struct FixLinks<false> : Links<double> {
    bool look;
    mutable bool all_unit = true;  // (look) every link read so far is a unit quaternion
    __device__ __forceinline__ FixLinks(const Ctx& c, const LatDesc& d)
        : Links<double>(c.links, d, c.status), look(c.look != 0) {}
    __device__ __forceinline__ FQuat fix(int mu, int p, uint32_t eo) const
    {
        const Quat<double> q = load(mu, p, eo);
        const FQuat f = fq_link(q);
        if (look && !unit_limbs(q, f)) all_unit = false;
        return f;
    }
};
template <> struct FixLinks<true> : Links<double> {
    FixMirror m;
    static constexpr bool all_unit = true;
    __device__ __forceinline__ FixLinks(const Ctx& c, const LatDesc& d)
        : Links<double>(c.links, d, c.status), m(c, d) {}
    __device__ __forceinline__ FQuat fix(int mu, int p, uint32_t eo) const { return m.load(mu, p, eo); }
    __device__ __forceinline__ void store(int mu, int p, uint32_t eo, const Quat<double>& q) const
    {
        Links<double>::store(mu, p, eo, q);
        m.store(mu, p, eo, q);
    }
};

// a stored link at 2^60
__device__ __forceinline__ void fix_from_link(const Quat<double>& q, int64_t* U)
{
    const FQuat f = fq_link(q);
    const Fx* c[4] = {&f.a0, &f.a1, &f.a2, &f.a3};
#pragma unroll
    for (int k = 0; k < 4; ++k) U[k] = (((int64_t)c[k]->h << 32) + c[k]->l) >> 1;
}

// one staple term of U_mu(x) in the plane (nu, mu), added to A (fq_staple)
template <typename LT>
__device__ __forceinline__ void fix_term(const LT& U, int mu, int nu, int p, uint32_t i, uint32_t hpm,
                                         uint32_t hpn, uint32_t hmn, bool lower, int64_t* A)
{
    const int q = p ^ 1;
    const FQuat x = U.fix(lower ? mu : nu, q, i + (lower ? hmn : hpm));
    const FQuat y = U.fix(lower ? nu : mu, lower ? p : q, i + (lower ? hpm + hmn : hpn));
    const FQuat z = U.fix(nu, lower ? q : p, lower ? i + hmn : i);
    fq_staple(x, y, z, lower, A);
}

// staple_sum: A, and (PLAQ) its part P over nu < mu.  The three planes are one
// loop body: the update's code has to fit the instruction caches (fully
// unrolled and with the draw inlined twice, 43% of the stalls waited for
// instructions and 64^4 ran at 3.7 G updates/s).
template <int MU, bool PLAQ, typename LT>
__device__ __forceinline__ void fix_staple_sum(const LT& U, const EoSite& s, uint32_t i,
                                               int p, int64_t* A, int64_t* P)
{
    uint32_t hp[4], hm[4];
    s.hops(hp, hm);
    A[0] = A[1] = A[2] = A[3] = 0;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        constexpr int n0 = nu_of<MU>(0), n1 = nu_of<MU>(1), n2 = nu_of<MU>(2);
        const int nu = k == 0 ? n0 : (k == 1 ? n1 : n2);
        const uint32_t hpn = k == 0 ? hp[n0] : (k == 1 ? hp[n1] : hp[n2]);
        const uint32_t hmn = k == 0 ? hm[n0] : (k == 1 ? hm[n1] : hm[n2]);
        fix_term(U, MU, nu, p, i, hp[MU], hpn, hmn, false, A);
        fix_term(U, MU, nu, p, i, hp[MU], hpn, hmn, true, A);
        if (PLAQ && k == MU - 1) {
#pragma unroll
            for (int c = 0; c < 4; ++c) P[c] = A[c];
        }
    }
}

// Per-lattice values of a call, in registers.
struct FixCall {
    HalfInvBeta hb;
    double beta, creutz;
    float beta_f;
    const FixTables* tab;
    uint32_t k0, k1, slo, shi;
    __device__ __forceinline__ explicit FixCall(const LatDesc& D)
    {
        const double h = D.half_inv_beta;
        hb = half_inv_beta_fix((uint64_t)__double_as_longlong(h));
        beta = D.beta;
        creutz = D.creutz_below;
        beta_f = D.beta_f;
        tab = D.fix_table;
        k0 = (uint32_t)D.seed;
        k1 = (uint32_t)(D.seed >> 32);
        slo = (uint32_t)D.sweep;
        shi = (uint32_t)(D.sweep >> 32);
    }
    __device__ __forceinline__ Stream stream(uint32_t key) const { return {k0, k1, key, slo, shi}; }
};

// alpha -> 0 limit of the conditional law (rare: kept out of the loops' code)
static __device__ __noinline__ Quat<double> haar_link(Stream st, const FixTables* tab)
{
    return haar_double(st.draw(TAG_DIRECTION, 0), tab);
}

// The draw's inputs from the staple sum: false for the Haar branch
// (alpha = beta |A| below its threshold).  HYB: *qc = 1 - exp(-2 alpha) of a
// link that takes Creutz's draw, 0 otherwise.
template <bool HYB>
__device__ __forceinline__ bool fix_prepare(const FixCall& C, const int64_t* A, Drawn* d, double* qc)
{
    uint64_t K;
    int n;
    *qc = 0.0;
    if (!unit_staple(A, C.hb, d, &K, &n)) return false;
    // |A| = sqrt(K 2^-60) 2^(7 - n); in single precision away from the threshold
    const float kf = __fsqrt_rn((float)(uint32_t)(K >> 29)) * exp2f((float)(7 - n) - 15.5f);
    double alpha = 0.0;
    if (HYB || !(C.beta_f * kf > 2e-12f)) {
        alpha = C.beta * ldexp(sqrt((double)K), 7 - n - 30);
        if (!(alpha >= alpha_haar<double>())) return false;
    }
    if (HYB && alpha < C.creutz) *qc = creutz_qc(alpha);
    return true;
}

// one trial; true when accepted
template <bool HYB>
__device__ __forceinline__ bool fix_try(const FixCall& C, const U4& w, int64_t inv, int ei, double qc,
                                        Lambda* L)
{
    if (HYB && qc > 0.0) {
        double delta;
        const double inv2a = __longlong_as_double((long long)double_bits(inv, ei));
        const bool ok = creutz_try(w, qc, inv2a, &delta);
        *L = lambda_from_delta((uint64_t)__double_as_longlong(delta));
        return ok;
    }
    *L = kp_lambda(kp_sum(w.x, w.y, w.z, C.tab), inv, ei);
    return kp_accept(*L, w.w);
}

// warp sum of 64-bit integers
__device__ __forceinline__ int64_t warp_sum64(int64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += (int64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)v, o);
    return v;
}

// warp_totals with the plaquette already summed over the warp
template <int MU, bool PLAQ>
__device__ __forceinline__ void fix_totals(const Ctx& ctx, int l, uint32_t blk0, uint32_t Vh,
                                           double wp, uint32_t ntrial, uint32_t ncap)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t wt = __reduce_add_sync(0xffffffffu, ntrial);
    const uint32_t wc = __reduce_add_sync(0xffffffffu, ncap);
    if (lane == 0) add_warp_totals<MU, PLAQ>(ctx, ctx.phase_wpb, l, blk0, Vh, wp, w, wt, wc);
}
__device__ __forceinline__ double plaq_double(int64_t v)  // v 2^-51
{
    return __longlong_as_double((long long)double_bits(v, -51));
}

// ---------------------------------------------------------------------------
// lattices with non-unit links or a large coupling: the FP64 sequence
// ---------------------------------------------------------------------------
// the draw and the new link from the staple sum A and its plaquette part P
template <typename LT>
__device__ __forceinline__ int32_t general_draw(const LT& U, const LatDesc& D, uint32_t i, int mu, int p,
                                                bool hyb, const Quat<double>& A, const Quat<double>& P,
                                                uint32_t lex, double* plaq)
{
    Quat<double> un;
    const int32_t tr = draw_link<double>(D, hyb, A, lex * 4u + (uint32_t)mu, D.sweep, &un);
    if (tr >= 0) U.store(mu, p, i, un);
    else un = U.load_rw(mu, p, i);
    *plaq += qretr(un, P);
    return tr;
}
// Staple sum by the tree s_k = up_k + lo_k for the k-th nu != mu,
// A = (s_0 + s_1) + s_2 (P = its prefix over nu < mu), FP64 draw, new link.
// Returns what update_link returns; *un is the link's final value.
template <typename LT>
__device__ __noinline__ int32_t general_link(const Ctx& ctx, const LatDesc& D, uint32_t i, int mu,
                                             int p, bool hyb, double* plaq, uint32_t* lex)
{
    const LT U(ctx.links, D, ctx.status);
    const EoSite s(D, i, p);
    uint32_t hp[4], hm[4];
    s.hops(hp, hm);
    Quat<double> A = {0, 0, 0, 0}, P = A;
    for (int nu = 0, k = 0; nu < 4; ++nu) {
        if (nu == mu) continue;
        const Quat<double> sk = qadd(staple_term<double>(U, mu, nu, p, i, hp, hm, false),
                                     staple_term<double>(U, mu, nu, p, i, hp, hm, true));
        A = k++ == 0 ? sk : qadd(A, sk);
        if (nu == mu - 1) P = A;
    }
    *lex = s.lex();
    return general_draw(U, D, i, mu, p, hyb, A, P, s.lex(), plaq);
}
template <typename LT>
__device__ __forceinline__ int32_t general_link(const Ctx& ctx, const LatDesc& D, uint32_t i, int mu,
                                                int p, bool hyb)
{
    double plaq = 0.0;
    uint32_t lex;
    return general_link<LT>(ctx, D, i, mu, p, hyb, &plaq, &lex);
}
// the links i0, i0 + step, ... below end of one thread, then the warp totals
template <int MU, bool PLAQ>
__device__ __noinline__ void general_links(const Ctx& ctx, int l, uint32_t blk0, uint32_t i0,
                                           uint32_t step, uint32_t end, int p, bool hyb, int32_t* dbg)
{
    const LatDesc& D = ctx.desc[l];
    double plaq = 0.0;
    uint32_t ntrial = 0, ncap = 0, lex;
    for (uint32_t i = i0; i < end; i += step) {
        const int32_t tr = general_link<Links<double>>(ctx, D, i, MU, p, hyb, &plaq, &lex);
        ncap += tr < 0;
        ntrial += tr < 0 ? (uint32_t)KP_CAP : (uint32_t)tr;
        if (dbg) dbg[lex] = tr;
    }
    __syncwarp();
    fix_totals<MU, PLAQ>(ctx, l, blk0, D.Vh, PLAQ ? warp_sum_t(plaq) : 0.0, ntrial, ncap);
}

// ---------------------------------------------------------------------------
// one link per thread
// ---------------------------------------------------------------------------
// NT, MINB bound the registers (255 or 96 a thread: 16^4 runs 95 us a sweep
// with many registers and 98 with 96, 32^4 674 with 128 and 663 with 96);
// smaller blocks of the same register count run the same kernel.
template <int MU, bool PLAQ, bool HYB, bool MIR, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
fix_phase_kernel(Ctx ctx, int p, int32_t* __restrict__ dbg)
{
    const int l = lattice_of_block(ctx.phase_start, ctx.n, blockIdx.x);
    const LatDesc& D = ctx.desc[l];
    const uint32_t Vh = D.Vh;
    const uint32_t blk0 = first_block(ctx.phase_start, l);
    const uint32_t i = (blockIdx.x - blk0) * blockDim.x + threadIdx.x;
    if (D.general) {
        general_links<MU, PLAQ>(ctx, l, blk0, i, 1u, i < Vh ? i + 1 : i, p, HYB, dbg);
        return;
    }
    const FixLinks<MIR> U(ctx, D);
    const FixCall C(D);
    int64_t plaq = 0;
    uint32_t ntrial = 0, ncap = 0;
    if (i < Vh) {
        const EoSite s(D, i, p);
        int64_t A[4], P[4], un[4];
        fix_staple_sum<MU, PLAQ>(U, s, i, p, A, P);
        const Stream st = C.stream(s.lex() * 4u + MU);
        Drawn d;
        double qc;
        int32_t tr = -1;
        if (!PLAQ && !U.all_unit) {
            tr = general_link<Links<double>>(ctx, D, i, MU, p, HYB);
            ncap = tr < 0;
        } else if (!fix_prepare<HYB>(C, A, &d, &qc)) {
            const Quat<double> h = haar_link(st, C.tab);
            U.store(MU, p, i, h);
            if (PLAQ) fix_from_link(h, un);
            tr = 0;
        } else {
            // trial 0 also carries the direction in the low 9 bits of its words
            U4 w = st.draw(TAG_TRIAL, 0u);
            const uint32_t kd1 = spare_bits_1(w), kd2 = spare_bits_2(w);
            Lambda L;
            for (int t = 0;;) {
                if (fix_try<HYB>(C, w, d.inv, d.ei, qc, &L)) {
                    tr = t + 1;
                    break;
                }
                if (++t == KP_CAP) break;
                w = st.draw(TAG_TRIAL, (uint32_t)t);
            }
            if (tr > 0) {
                new_link_fix(L, kd1, kd2, d.V, C.tab, un);
                U.store(MU, p, i, dq_link(un));
            } else {
                ncap = 1;
                if (PLAQ) fix_from_link(U.load_rw(MU, p, i), un);
            }
        }
        ntrial = tr < 0 ? (uint32_t)KP_CAP : (uint32_t)tr;
        if (dbg) dbg[s.lex()] = tr;
        if (PLAQ) plaq = retr_fix(un, P);
    }
    fix_totals<MU, PLAQ>(ctx, l, blk0, Vh, PLAQ ? plaq_double(warp_sum64(plaq)) : 0.0, ntrial,
                             ncap);
}

// ---------------------------------------------------------------------------
// R links per thread with a per-warp retry queue
// ---------------------------------------------------------------------------
// The warp alternates between two steps.  Step 1 takes 32 links: each lane
// forms its link's staple sum and puts the draw's inputs (unit staple,
// 1 / (2 alpha), counter word, trial index, storage index) into a queue in
// shared memory.  Step 2 takes the last 32 of the queue, one trial a lane:
// an accepted link is finished, a rejected one goes back with its next
// trial.  Step 1 runs while fewer than 32 links wait, so nearly every trial
// runs with all lanes, each step has one copy of its code, and the registers
// of the staple sum and of the draw are not held together.
template <bool PLAQ, bool HYB>
struct FixQueue {
    static constexpr int CAP = 64;  // < 32 held before a push of at most 32
    int64_t pl[PLAQ ? 4 : 1][PLAQ ? CAP : 1];
    int64_t inv[CAP];
    double qc[HYB ? CAP : 1];
    Fx v[4][CAP];
    int32_t ei[CAP];
    uint32_t key[CAP];
    uint32_t tk[CAP];    // next trial | first 18-bit direction word << 13
    uint32_t kd2[CAP];   // second 18-bit direction word (both set by trial 0)
    uint32_t site[CAP];  // storage index
};

// R <= FIX_MAX_ROUNDS: the warp's plaquette sum (6 * 2^51 a link, 32 R
// links) stays below 2^63.
constexpr int FIX_MAX_ROUNDS = 16;
template <int MU, bool PLAQ, bool HYB, bool MIR, bool PERSIST>
__global__ void __launch_bounds__(32, FIX_THREADS[PERSIST ? FIX_PERSIST : FIX_QUEUE] / 32)
fix_queue_kernel(Ctx ctx, int p, int R, int32_t* __restrict__ dbg)
{
    static_assert(KP_CAP <= (1 << 13), "trial index must fit 13 bits");
    constexpr uint32_t NT = 32;
    using Queue = FixQueue<PLAQ, HYB>;
    __shared__ Queue Q;

    const int l = lattice_of_block(ctx.phase_start, ctx.n, blockIdx.x);
    const LatDesc& D = ctx.desc[l];
    const uint32_t Vh = D.Vh;
    const uint32_t blk0 = first_block(ctx.phase_start, l);
    // tiles of 32 R positions; a persistent block takes every nb-th
    const uint32_t nb = PERSIST ? __ldg(ctx.phase_start + l + 1) - blk0 : 0u;
    const uint32_t tile0 = blockIdx.x - blk0;
    if (D.general) {
        if (PERSIST) {
            general_links<MU, PLAQ>(ctx, l, blk0, tile0 * NT + threadIdx.x, nb * NT, Vh, p, HYB, dbg);
        } else {
            const uint32_t i0 = tile0 * (NT * R) + threadIdx.x;
            general_links<MU, PLAQ>(ctx, l, blk0, i0, NT, min(Vh, (tile0 + 1) * (NT * R)), p, HYB, dbg);
        }
        return;
    }
    const FixLinks<MIR> U(ctx, D);
    const FixCall C(D);
    const int lane = threadIdx.x;
    const uint32_t below = (1u << lane) - 1u;

    int64_t plaq = 0, plaq_hi = 0;  // at 2^51, and (persistent) 2^31
    uint32_t ntrial = 0, ncap = 0;
    int cnt = 0;                    // queued links (warp-uniform)
    uint32_t base = tile0 * (NT * R), left = R;  // next 32 positions, rounds left in the tile

    while (true) {
        bool pend = false;
        Drawn d;
        int64_t P[4];
        double qc = 0.0;
        uint32_t key = 0, tk = 0, kd2 = 0, i;
        if (cnt < 32 && base < Vh) {
            // step 1
            i = base + lane;
            if (i < Vh) {
                const EoSite s(D, i, p);
                int64_t A[4];
                fix_staple_sum<MU, PLAQ>(U, s, i, p, A, P);
                key = s.lex() * 4u + MU;
                if (!PLAQ && !U.all_unit) {
                    const int32_t tr = general_link<Links<double>>(ctx, D, i, MU, p, HYB);
                    ncap += tr < 0;
                    ntrial += tr < 0 ? (uint32_t)KP_CAP : (uint32_t)tr;
                    if (dbg) dbg[key >> 2] = tr;
                    if constexpr (!MIR) U.all_unit = true;
                } else if (!(pend = fix_prepare<HYB>(C, A, &d, &qc))) {
                    const Quat<double> h = haar_link(C.stream(key), C.tab);
                    U.store(MU, p, i, h);
                    if (PLAQ) {
                        int64_t un[4];
                        fix_from_link(h, un);
                        plaq += retr_fix(un, P);
                    }
                    if (dbg) dbg[key >> 2] = 0;
                }
            }
            base += NT;
            if (--left == 0) {
                left = R;
                base = PERSIST ? base + (nb - 1) * (NT * R) : Vh;
                if (PLAQ && PERSIST) {
                    plaq_hi += plaq >> 20;
                    plaq &= (int64_t(1) << 20) - 1;
                }
            }
        } else if (cnt > 0) {
            // step 2
            const int n = cnt < 32 ? cnt : 32;
            const bool have = lane < n;
            const int e = have ? cnt - n + lane : 0;
            d.V = {Q.v[0][e], Q.v[1][e], Q.v[2][e], Q.v[3][e]};
            d.inv = Q.inv[e];
            d.ei = Q.ei[e];
            if (PLAQ) { P[0] = Q.pl[0][e]; P[1] = Q.pl[1][e]; P[2] = Q.pl[2][e]; P[3] = Q.pl[3][e]; }
            if (HYB) qc = Q.qc[e];
            key = Q.key[e];
            tk = Q.tk[e];
            kd2 = Q.kd2[e];
            i = Q.site[e];
            __syncwarp();
            cnt -= n;
            if (have) {
                const uint32_t t = tk & 0x1FFFu;
                const U4 w = C.stream(key).draw(TAG_TRIAL, t);
                // trial 0 also carries the direction in the low 9 bits of its words
                if (t == 0) {
                    tk = spare_bits_1(w) << 13;
                    kd2 = spare_bits_2(w);
                }
                Lambda L;
                int64_t un[4];
                if (fix_try<HYB>(C, w, d.inv, d.ei, qc, &L)) {
                    new_link_fix(L, tk >> 13, kd2, d.V, C.tab, un);
                    U.store(MU, p, i, dq_link(un));
                    if (PLAQ) plaq += retr_fix(un, P);
                    ntrial += t + 1;
                    if (dbg) dbg[key >> 2] = (int32_t)t + 1;
                } else if (t + 1 >= (uint32_t)KP_CAP) {
                    // cap hit: the link keeps its value
                    ncap += 1;
                    ntrial += (uint32_t)KP_CAP;
                    if (PLAQ) {
                        fix_from_link(U.load_rw(MU, p, i), un);
                        plaq += retr_fix(un, P);
                    }
                    if (dbg) dbg[key >> 2] = -1;
                } else {
                    pend = true;
                    ++tk;
                }
            }
        } else {
            break;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, pend);
        if (pend) {
            const int e = cnt + __popc(m & below);
            Q.v[0][e] = d.V.a0; Q.v[1][e] = d.V.a1; Q.v[2][e] = d.V.a2; Q.v[3][e] = d.V.a3;
            if (PLAQ) { Q.pl[0][e] = P[0]; Q.pl[1][e] = P[1]; Q.pl[2][e] = P[2]; Q.pl[3][e] = P[3]; }
            Q.inv[e] = d.inv;
            Q.ei[e] = d.ei;
            if (HYB) Q.qc[e] = qc;
            Q.key[e] = key;
            Q.tk[e] = tk;
            Q.kd2[e] = kd2;
            Q.site[e] = i;
        }
        cnt += __popc(m);
        __syncwarp();
    }
    double wp = 0.0;
    if (PLAQ) {
        wp = plaq_double(warp_sum64(plaq));
        if (PERSIST) wp += __longlong_as_double((long long)double_bits(warp_sum64(plaq_hi), -31));
    }
    fix_totals<MU, PLAQ>(ctx, l, blk0, Vh, wp, ntrial, ncap);
}

// ---------------------------------------------------------------------------
// four threads per link: small lattices
// ---------------------------------------------------------------------------
// A lattice that gives each SM sub-partition a warp or two of one link per
// thread (16^4: 1024 warps per phase) spends a phase in one link's chain of
// ~2,700 instructions.  Here four warps share 32 links: three form the staple
// terms of one plane each (exact integer sums: any order gives the same bits),
// the fourth draws the first trial and the direction meanwhile.  The first
// warp then adds the sums, decides and stores; among 32 links some nearly
// always reject, so the others draw the next trials while it does.  Links
// still waiting get four trials at a time, one from each warp, and take the
// first accepted one of their own sequence.  us a sweep at beta = 2.3, the
// best one link per thread / eight lanes per link (which this replaced) /
// here with 128 registers / with 72, which hold 7 blocks an SM instead of 4:
//   8^4  74.5 / 47.2 / 44.0 / 47.7    12^4  78.3 / 87.9 / 53.3 / 56.4
//   16^4 95.1 / 184.5 / 88.3 / 79.1   20^4 164 / 391 / 178 / 148
//   24^4 266 against 349 in an earlier form: one link per thread takes over.
// Trials drawn ahead: with 128 registers 2 or 3 give 53.7, 53.3 at 12^4; with
// 72, where the SM is full, 79.1, 80.0 at 16^4 and 148, 152 at 20^4.
struct Trial64 {
    int64_t t;
    int32_t e;
    uint32_t w3;  // the word of the accept test
};
struct Dir64 {
    int64_t sth, cph, sph;
    int32_t cth, pad;
};
static_assert(sizeof(Trial64) == 16 && sizeof(Dir64) == 32, "16-byte accesses");
static_assert(KP_CAP % 4 == 0, "whole rounds of four trials");

// general_link's sum of 32 links by their four warps: a warp forms s_k of one
// plane (planes 1 and 2 through `sums`), the first adds them and draws.  The
// other three give the FP64 unit of their sub-partition a third of the staple
// each: 8^4 at beta = 1000 92 us a sweep, 126 with one link per thread in one
// cluster launch.
template <int MU, bool PLAQ, bool HYB>
__device__ __noinline__ void general_quad(const Ctx& ctx, int l, uint32_t blk0, uint32_t i, int p,
                                          double2 (*sums)[2][32], int32_t* dbg)
{
    const LatDesc& D = ctx.desc[l];
    const Links<double> U(ctx.links, D, ctx.status);
    const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
    const bool act = i < D.Vh;
    Quat<double> s0 = {0, 0, 0, 0};
    uint32_t lex = 0;
    if (act && role < 3) {
        const EoSite s(D, i, p);
        lex = s.lex();
        uint32_t hp[4], hm[4];
        s.hops(hp, hm);
        const int nu = nu_of<MU>(role);
        s0 = qadd(staple_term<double>(U, MU, nu, p, i, hp, hm, false),
                  staple_term<double>(U, MU, nu, p, i, hp, hm, true));
        if (role > 0) {
            sums[role - 1][0][lane] = make_double2(s0.a0, s0.a1);
            sums[role - 1][1][lane] = make_double2(s0.a2, s0.a3);
        }
    }
    __syncthreads();
    double plaq = 0.0;
    uint32_t ntrial = 0, ncap = 0;
    if (act && role == 0) {
        auto plane = [&](int k) -> Quat<double> {
            const double2 lo = sums[k - 1][0][lane], hi = sums[k - 1][1][lane];
            return {lo.x, lo.y, hi.x, hi.y};
        };
        const Quat<double> s01 = qadd(s0, plane(1));
        const Quat<double> A = qadd(s01, plane(2));
        const Quat<double> P = MU == 1 ? s0 : (MU == 2 ? s01 : A);
        const int32_t tr = general_draw(U, D, i, MU, p, HYB, A, P, lex, &plaq);
        ncap = tr < 0;
        ntrial = tr < 0 ? (uint32_t)KP_CAP : (uint32_t)tr;
        if (dbg) dbg[lex] = tr;
    }
    __syncwarp();
    fix_totals<MU, PLAQ>(ctx, l, blk0, D.Vh, PLAQ ? warp_sum_t(plaq) : 0.0, ntrial, ncap);
}

template <int MU, bool PLAQ, bool HYB, bool MIR, int MINB>
__global__ void __launch_bounds__(128, MINB)
fix_quad_kernel(Ctx ctx, int p, int32_t* __restrict__ dbg)
{
    struct Group {
        longlong2 sums[2][2][32];  // planes 1 and 2 (general_quad: as double2)
        Trial64 trial[4][32];  // HYB: lambda^2 of a trial, and whether it was accepted
        Dir64 dir[32];
        struct Hyb {  // a link's inputs to its trials
            int64_t inv[HYB ? 32 : 1];
            double qc[HYB ? 32 : 1];
            int32_t ei[HYB ? 32 : 1];
        } hyb;
        uint32_t pend;
        uint32_t bad[3];  // links with a neighbour that is not a unit quaternion, by plane
    };
    constexpr int SPEC = MINB > 4 ? 2 : 3;  // trials drawn ahead besides the first
    // HYB: Creutz's logarithm runs on the FP64 unit (~2,500 clocks a warp), so
    // with few blocks an SM each of the four sub-partitions takes a trial of
    // the waiting links (8^4, beta = 0.9, Creutz's draw below alpha = 1.7: 128 ->
    // 88 us a sweep); where the SM is full the trials after an accepted one
    // would cost others their turn (16^4 189 us one by one, 223 so)
    constexpr bool SPREAD = MINB <= 4;
    __shared__ Group G;
    const int l = lattice_of_block(ctx.phase_start, ctx.n, blockIdx.x);
    const LatDesc& D = ctx.desc[l];
    const uint32_t Vh = D.Vh;
    const uint32_t blk0 = first_block(ctx.phase_start, l);
    const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
    const uint32_t i = (blockIdx.x - blk0) * 32u + (uint32_t)lane;
    const bool act = i < Vh;
    if (D.general) {
        // (with few registers the call costs the fixed-point path 1.5% at 18^4)
        if constexpr (MINB > 4)
            general_links<MU, PLAQ>(ctx, l, blk0, i, 1u, act && role == 0 ? i + 1 : i, p, HYB, dbg);
        else
            general_quad<MU, PLAQ, HYB>(ctx, l, blk0, i, p, reinterpret_cast<double2(*)[2][32]>(G.sums),
                                        dbg);
        return;
    }
    const FixLinks<MIR> U(ctx, D);
    const FixCall C(D);
    auto draw = [&](const Stream& st, int t, int slot) {
        const U4 w = st.draw(TAG_TRIAL, (uint32_t)t);
        if (!HYB) {
            const KpSum k = kp_sum(w.x, w.y, w.z, C.tab);
            G.trial[slot][lane] = {k.t, k.e, w.w};
        }
        if (t == 0) {
            const FixDir f = direction_fix(spare_bits_1(w), spare_bits_2(w), C.tab);
            G.dir[lane] = {f.sth, f.cph, f.sph, f.cth, 0};
        }
    };

    int64_t A[4] = {0, 0, 0, 0}, P[4];
    uint32_t lex = 0;
    if (act) {
        const EoSite s(D, i, p);
        lex = s.lex();
        if (role < 3) {
            uint32_t hp[4], hm[4];
            s.hops(hp, hm);
            const int nu = nu_of<MU>(role);
            const uint32_t hpn = nu == 0 ? hp[0] : (nu == 1 ? hp[1] : (nu == 2 ? hp[2] : hp[3]));
            const uint32_t hmn = nu == 0 ? hm[0] : (nu == 1 ? hm[1] : (nu == 2 ? hm[2] : hm[3]));
            fix_term(U, MU, nu, p, i, hp[MU], hpn, hmn, false, A);
            fix_term(U, MU, nu, p, i, hp[MU], hpn, hmn, true, A);
            if (role > 0) {
                G.sums[role - 1][0][lane] = make_longlong2(A[0], A[1]);
                G.sums[role - 1][1][lane] = make_longlong2(A[2], A[3]);
            }
        } else {
            draw(C.stream(lex * 4u + MU), 0, 0);
        }
    }
    if (!MIR && !PLAQ) {
        const uint32_t m = __ballot_sync(0xffffffffu, !U.all_unit);
        if (lane == 0 && role < 3) G.bad[role] = m;
    }
    __syncthreads();
    const Stream st = C.stream(lex * 4u + MU);
    Drawn d;
    double qc = 0.0;
    Lambda L = {0, 0, 0};
    int32_t tr = -1;
    bool haar = false, wait = false, general = false;
    if (!MIR && !PLAQ && role == 0 && act) general = ((G.bad[0] | G.bad[1] | G.bad[2]) >> lane) & 1u;
    if (general) {
        tr = general_link<Links<double>>(ctx, D, i, MU, p, HYB);
    } else if (role == 0 && act) {
#pragma unroll
        for (int c = 0; c < 4; ++c) P[c] = A[c];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const longlong2 lo = G.sums[r][0][lane], hi = G.sums[r][1][lane];
            A[0] += lo.x;
            A[1] += lo.y;
            A[2] += hi.x;
            A[3] += hi.y;
            if (PLAQ && r + 1 < MU) {
#pragma unroll
                for (int c = 0; c < 4; ++c) P[c] = A[c];
            }
        }
        haar = !fix_prepare<HYB>(C, A, &d, &qc);
        if (haar) {
            tr = 0;
        } else if (HYB && !SPREAD) {
            for (int t = 0; t < KP_CAP && tr < 0; ++t)
                if (fix_try<HYB>(C, st.draw(TAG_TRIAL, (uint32_t)t), d.inv, d.ei, qc, &L)) tr = t + 1;
        } else if (HYB) {
            wait = true;
            G.hyb.inv[lane] = d.inv;
            G.hyb.qc[lane] = qc;
            G.hyb.ei[lane] = d.ei;
        } else {
            const Trial64 a = G.trial[0][lane];
            L = kp_lambda(KpSum{a.t, a.e}, d.inv, d.ei);
            if (kp_accept(L, a.w3)) tr = 1;
            else wait = true;
        }
    }
    if (HYB && SPREAD) {
        for (int t0 = 0; t0 < KP_CAP; t0 += 4) {
            if (role == 0) {
                const uint32_t m = __ballot_sync(0xffffffffu, wait);
                if (lane == 0) G.pend = m;
            }
            __syncthreads();
            const uint32_t m = G.pend;
            if (m == 0) break;
            if ((m >> lane) & 1u) {
                const U4 w = st.draw(TAG_TRIAL, (uint32_t)(t0 + role));
                Lambda t;
                const bool ok = fix_try<HYB>(C, w, G.hyb.inv[lane], G.hyb.ei[lane], G.hyb.qc[lane], &t);
                G.trial[role][lane] = {t.P, t.qe, ok ? 1u : 0u};
            }
            __syncthreads();
            for (int k = 0; k < 4 && wait; ++k) {
                const Trial64 a = G.trial[k][lane];
                if (a.w3) {
                    L = lambda_of(a.t, a.e);
                    tr = t0 + k + 1;
                    wait = false;
                }
            }
        }
    } else if (!HYB) {
        // tests trials t0 .. t0 + n - 1 (slots t & 3) of the waiting links
        auto pick = [&](int t0, int n) {
            for (int k = 0; k < n && wait; ++k) {
                const Trial64 a = G.trial[(t0 + k) & 3][lane];
                L = kp_lambda(KpSum{a.t, a.e}, d.inv, d.ei);
                if (kp_accept(L, a.w3)) {
                    tr = t0 + k + 1;
                    wait = false;
                }
            }
        };
        if (act && role > 0 && role <= SPEC) draw(st, role, role);
        __syncthreads();
        pick(1, SPEC);
        for (int t0 = 1 + SPEC; t0 < KP_CAP; t0 += 4) {
            if (role == 0) {
                const uint32_t m = __ballot_sync(0xffffffffu, wait);
                if (lane == 0) G.pend = m;
            }
            __syncthreads();
            const uint32_t m = G.pend;
            if (m == 0) break;
            if (((m >> lane) & 1u) && t0 + role < KP_CAP) draw(st, t0 + role, (t0 + role) & 3);
            __syncthreads();
            pick(t0, KP_CAP - t0 < 4 ? KP_CAP - t0 : 4);
        }
    }
    if (role != 0) {
        // one partial per warp: only the first of a group has plaquettes
        if (PLAQ && lane == 0)
            ctx.plaq_partial[((size_t)(MU - 1) * ctx.phase_blocks + blockIdx.x) * ctx.phase_wpb +
                             (threadIdx.x >> 5)] = 0.0;
        return;
    }
    int64_t plaq = 0;
    uint32_t ntrial = 0, ncap = 0;
    if (act) {
        int64_t un[4];
        if (general) {
            ncap = tr < 0;  // general_link stored it
        } else if (haar) {
            const Quat<double> h = haar_link(st, C.tab);
            U.store(MU, p, i, h);
            if (PLAQ) fix_from_link(h, un);
        } else if (tr > 0) {
            const Dir64 f = G.dir[lane];
            new_link_dir_fix(L, {f.cth, f.sth, f.cph, f.sph}, d.V, un);
            U.store(MU, p, i, dq_link(un));
        } else {
            ncap = 1;
            if (PLAQ) fix_from_link(U.load_rw(MU, p, i), un);
        }
        ntrial = tr < 0 ? (uint32_t)KP_CAP : (uint32_t)tr;
        if (dbg) dbg[lex] = tr;
        if (PLAQ) plaq = retr_fix(un, P);
    }
    __syncwarp();
    fix_totals<MU, PLAQ>(ctx, l, blk0, Vh, PLAQ ? plaq_double(warp_sum64(plaq)) : 0.0, ntrial, ncap);
}

}  // namespace su2
