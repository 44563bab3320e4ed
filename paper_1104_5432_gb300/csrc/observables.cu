// observables.cu -- stand-alone measurements on the links:
//   mean plaquette (Sec. 2.1: "mean average plaquette"),
//   Polyakov loop L(x) = 1/2 Tr prod_t U_t(x,t) and its volume mean
//   (Sec. 2.2, Eq. 1), and the Polyakov-loop correlator
//   C(r) = <L(x) L(x + r e_i)> over x and the three spatial axes
//   (Sec. 2.2, Eq. 3: for SU(2) the traces are real, so 1/4 Tr L Tr L^+ is
//   the product of the normalised loops).
// Products and warp partial sums are taken in the link precision; block,
// lattice and over-sweep sums in FP64, each in a fixed order (per-block
// partials, then one block per (lattice, row)).
#include "su2_internal.h"
#include "su2_links.cuh"
#include "su2_mirror.cuh"
#include "su2_reduce.cuh"

namespace su2 {

template <typename T>
__device__ __forceinline__ T warp_total(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// block total of one value per thread: warp sums in T, block sum in FP64
// (valid in thread 0)
template <typename T>
__device__ __forceinline__ double block_total(T v, T* s_warp)
{
    v = warp_total(v);
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 0; w < TPB / 32; ++w) s += (double)s_warp[w];
    }
    return s;
}

// LT: the links in the handle's layout (a choice per load would keep the
// loads from being issued together: 64^4 FP32 607 -> 424 us with the final sum).
// GENERAL (FP64): only lattices whose fixed-point result is not valid.
template <typename T, typename LT, bool GENERAL>
__global__ void __launch_bounds__(TPB) plaquette_kernel(Ctx ctx)
{
    __shared__ T s_warp[TPB / 32];
    const int l = lattice_of_block(ctx.site_start, ctx.n, blockIdx.x);
    if (GENERAL && ctx.obs_flag[l] == 0) return;
    const LatDesc& D = ctx.desc[l];
    const uint32_t lex = (blockIdx.x - first_block(ctx.site_start, l)) * TPB + threadIdx.x;
    T acc = T(0);
    if (lex < D.V) {
        const LT U(ctx.links, D, ctx.status);
        int p;
        const EoSite s = EoSite::from_lex(D, lex, &p);
        uint32_t hp[4], hm[4];
        s.hops(hp, hm, LT::UNIT);
        const uint32_t o = (lex >> 1) * (uint32_t)LT::UNIT;
        const int q = p ^ 1;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const Quat<T> umu = U.load_at(mu, p, o);
            const uint32_t e_pmu = o + hp[mu];
#pragma unroll
            for (int nu = mu + 1; nu < 4; ++nu) {
                // 1/2 Tr U_mu(x) U_nu(x+mu) [U_nu(x) U_mu(x+nu)]^+
                const Quat<T> left = qmul(umu, U.load_at(nu, q, e_pmu));
                const Quat<T> right = qmul(U.load_at(nu, p, o), U.load_at(mu, q, o + hp[nu]));
                acc += qretr(left, qdag(right));
            }
        }
    }
    const double b = block_total(acc, s_warp);
    if (threadIdx.x == 0) ctx.obs_partial[blockIdx.x] = b;
}

// The FP64 plaquette in fixed point (su2_fixed.cuh: ~12 times the rate of the
// FP64 unit's ~220 multiply-adds per site; 64^4 6.52 -> 2.19 ms): the
// six traces are exact integer dot products of 2^58 quaternions, kept at
// 2^60 and summed over a warp at 2^52.  Each thread looks at the norms of its
// own four links; where one is not a unit quaternion the ranges do not hold,
// and the lattice's flag makes the FP64 kernel above compute it again.
__global__ void __launch_bounds__(TPB) plaquette_fix_kernel(Ctx ctx)
{
    __shared__ double s_warp[TPB / 32];
    const int l = lattice_of_block(ctx.site_start, ctx.n, blockIdx.x);
    const LatDesc& D = ctx.desc[l];
    const uint32_t lex = (blockIdx.x - first_block(ctx.site_start, l)) * TPB + threadIdx.x;
    int64_t acc = 0;
    if (lex < D.V) {
        const Links<double> U(ctx.links, D, ctx.status);
        int p;
        const EoSite s = EoSite::from_lex(D, lex, &p);
        uint32_t hp[4], hm[4];
        s.hops(hp, hm);
        const uint32_t eo = lex >> 1;
        const int q = p ^ 1;
        FQuat own[4];
        bool ok = true;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const Quat<double> u = U.load(mu, p, eo);
            ok = ok && unit_link(make_double2(u.a0, u.a1), make_double2(u.a2, u.a3));
            own[mu] = fq_link(u);
        }
        if (!ok) ctx.obs_flag[l] = 1u;
        auto product = [](const FQuat& a, const FQuat& b) {
            return fq_mul_nd(a, {b.a0, neg(b.a1), neg(b.a2), neg(b.a3)});
        };
#pragma unroll
        for (int mu = 0; mu < 4; ++mu)
#pragma unroll
            for (int nu = mu + 1; nu < 4; ++nu) {
                const FQuat a = product(own[mu], fq_link(U.load(nu, q, eo + hp[mu])));
                const FQuat b = product(own[nu], fq_link(U.load(mu, q, eo + hp[nu])));
                acc += dot4_k<8>(a.a0, b.a0, a.a1, b.a1, a.a2, b.a2, a.a3, b.a3);
            }
        acc = (acc + 128) >> 8;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        acc += (int64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)acc, o);
    if ((threadIdx.x & 31) == 0)
        s_warp[threadIdx.x >> 5] = __longlong_as_double((long long)double_bits(acc, -52));
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < TPB / 32; ++w) t += s_warp[w];
        ctx.obs_partial[blockIdx.x] = t;
    }
}

// L(x) for every spatial site into the field (link precision) and the
// per-block partial sums of L.  Bound by the latency of the links' loads: four
// time slices are loaded together.
template <typename T, typename LT>
__global__ void __launch_bounds__(TPB) polyakov_kernel(Ctx ctx)
{
    __shared__ T s_warp[TPB / 32];
    const int l = lattice_of_block(ctx.spat_start, ctx.n, blockIdx.x);
    const LatDesc& D = ctx.desc[l];
    const uint32_t sidx = (blockIdx.x - first_block(ctx.spat_start, l)) * TPB + threadIdx.x;
    T L = T(0);
    if (sidx < (uint32_t)D.Vs) {
        const LT U(ctx.links, D, ctx.status);
        const uint32_t r = fdiv(sidx, D.div_ns);
        const uint32_t x = sidx - r * (uint32_t)D.Ns;
        const uint32_t z = fdiv(r, D.div_ns);
        const uint32_t y = r - z * (uint32_t)D.Ns;
        const int p0 = (int)((x + y + z) & 1u);
        Quat<T> P = {T(1), T(0), T(0), T(0)};
        // the site at t is eo = sidx / 2 + (Vs / 2) t (Vs is even), of parity p0 + t
        uint32_t o = (sidx >> 1) * (uint32_t)LT::UNIT;
        const uint32_t step = ((uint32_t)D.Vs >> 1) * (uint32_t)LT::UNIT;
        int t = 0;
        for (; t + 4 <= D.Nt; t += 4, o += 4 * step) {
            const Quat<T> u0 = U.load_at(3, p0, o), u1 = U.load_at(3, p0 ^ 1, o + step);
            const Quat<T> u2 = U.load_at(3, p0, o + 2 * step), u3 = U.load_at(3, p0 ^ 1, o + 3 * step);
            P = qmul(qmul(qmul(qmul(P, u0), u1), u2), u3);
        }
        for (; t < D.Nt; ++t, o += step) P = qmul(P, U.load_at(3, p0 ^ (t & 1), o));
        L = P.a0;
        reinterpret_cast<T*>(ctx.field)[D.field_off + sidx] = L;
    }
    const double b = block_total(L, s_warp);
    if (threadIdx.x == 0) ctx.obs_partial[blockIdx.x] = b;
}

// rows r = 0..rmax of partials, from the Polyakov field of the last
// polyakov_kernel launch; one barrier for all rows.  Bound by the FP64 unit in
// double (~76 clocks an addition), where eight rows share warp_total's tree:
// four additions per row and lane in place of eight, the same sums; by the
// field's loads in float, one row at a time (eight: 0.149 against 0.147 ms).
// 21 lattices 48^3, r <= 24, with the Polyakov loops before it: FP64 1.21 -> 0.90
// ms, a measured sweep at Nt = 4 6.19 -> 5.91.
template <typename T>
__global__ void __launch_bounds__(TPB) correlator_kernel(Ctx ctx, int rmax)
{
    __shared__ T s_rows[MAX_RMAX + 1][TPB / 32];
    const int l = lattice_of_block(ctx.spat_start, ctx.n, blockIdx.x);
    const LatDesc& D = ctx.desc[l];
    const uint32_t sidx = (blockIdx.x - first_block(ctx.spat_start, l)) * TPB + threadIdx.x;
    const bool act = sidx < (uint32_t)D.Vs;
    const T* F = reinterpret_cast<const T*>(ctx.field) + D.field_off;
    uint32_t x = 0, y = 0, z = 0;
    T L0 = T(0);
    const uint32_t Ns = (uint32_t)D.Ns;
    if (act) {
        const uint32_t r = fdiv(sidx, D.div_ns);
        x = sidx - r * Ns;
        z = fdiv(r, D.div_ns);
        y = r - z * Ns;
        L0 = F[sidx];
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // indices of x + r in the three directions, and where each wraps
    const uint32_t dz = Ns * Ns;
    uint32_t ox = sidx, oy = sidx, oz = sidx;
    const uint32_t ex = ox + (Ns - x), ey = oy + (Ns - y) * Ns, ez = oz + (Ns - z) * dz;
    constexpr int G = sizeof(T) == 8 ? 8 : 1;  // rows at a time
    for (int r0 = 0; r0 <= rmax; r0 += G) {
        T v[G];
#pragma unroll
        for (int k = 0; k < G; ++k) {
            v[k] = T(0);
            if (act && r0 + k <= rmax) v[k] = L0 * (F[ox] + F[oy] + F[oz]);
            ox += 1;
            oy += Ns;
            oz += dz;
            if (ox == ex) ox -= Ns;
            if (oy == ey) oy -= dz;
            if (oz == ez) oz -= Ns * dz;
        }
        // in the tree's first levels a lane keeps half of its rows and adds the
        // partner's
#pragma unroll
        for (int h = G / 2; h > 0; h >>= 1) {
            const bool up = lane & (32 / G * h);
#pragma unroll
            for (int k = 0; k < h; ++k) {
                const T give = up ? v[k] : v[k + h];
                v[k] = (up ? v[k + h] : v[k]) + __shfl_xor_sync(0xffffffffu, give, 32 / G * h);
            }
        }
#pragma unroll
        for (int o = 16 / G; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        const int row = r0 + lane / (32 / G);  // the lane's upper bits chose the halves
        if (lane % (32 / G) == 0 && row <= rmax) s_rows[row][w] = v[0];
    }
    __syncthreads();
    if ((int)threadIdx.x <= rmax) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < TPB / 32; ++k) s += (double)s_rows[threadIdx.x][k];
        ctx.obs_partial[(size_t)threadIdx.x * ctx.spat_blocks + blockIdx.x] = s;
    }
}

// out[l*rows + row] (=|+=) scale_l * sum of the lattice's partials in row
// `row`; mode 0: scale 1/(6V) (plaquette), 1: 1/Vs (Polyakov), 2: 1/(3Vs)
// (correlator).  abs_out (nullable, mode 1) gets |mean|.
__global__ void __launch_bounds__(TPB)
finalize_kernel(Ctx ctx, const uint32_t* __restrict__ start, uint32_t stride, int rows, int mode,
                double* out, double* abs_out, int accumulate)
{
    __shared__ double sred[TPB / 32];
    const int l = blockIdx.x, row = blockIdx.y;
    const LatDesc& D = ctx.desc[l];
    const uint32_t b0 = start[l], b1 = start[l + 1];
    double acc = 0.0;
    for (uint32_t b = b0 + threadIdx.x; b < b1; b += TPB)
        acc += ctx.obs_partial[(size_t)row * stride + b];
    const double tot = block_sum<TPB>(acc, sred);
    if (threadIdx.x == 0) {
        const double scale = mode == 0 ? 1.0 / (6.0 * (double)D.V)
                           : mode == 1 ? 1.0 / (double)D.Vs
                                       : 1.0 / (3.0 * (double)D.Vs);
        const double v = tot * scale;
        double* o = out + (size_t)l * rows + row;
        *o = accumulate ? *o + v : v;
        if (abs_out) {
            double* a = abs_out + l;
            *a = accumulate ? *a + fabs(v) : fabs(v);
        }
        if (mode == 0) ctx.obs_flag[l] = 0u;  // for the next plaquette
    }
}

cudaError_t launch_plaquette(const Ctx& c, int row, double* out_dev, cudaStream_t s)
{
    const unsigned g = c.site_blocks;
    if (row == ROW_F64) {
        plaquette_fix_kernel<<<g, TPB, 0, s>>>(c);
        plaquette_kernel<double, Links<double>, true><<<g, TPB, 0, s>>>(c);
    } else if (row == ROW_F32_PAIRS) {
        plaquette_kernel<float, PairLinks, false><<<g, TPB, 0, s>>>(c);
    } else if (c.wide) {
        plaquette_kernel<float, WideLinks, false><<<g, TPB, 0, s>>>(c);
    } else {
        plaquette_kernel<float, Links<float>, false><<<g, TPB, 0, s>>>(c);
    }
    finalize_kernel<<<dim3(c.n, 1), TPB, 0, s>>>(c, c.site_start, c.site_blocks, 1, 0, out_dev,
                                                 nullptr, 0);
    return cudaGetLastError();
}

cudaError_t launch_polyakov(const Ctx& c, int row, double* out_signed_dev, double* out_abs_dev,
                            int accumulate, cudaStream_t s)
{
    const unsigned g = c.spat_blocks;
    if (row == ROW_F64) polyakov_kernel<double, Links<double>><<<g, TPB, 0, s>>>(c);
    else if (row == ROW_F32_PAIRS) polyakov_kernel<float, PairLinks><<<g, TPB, 0, s>>>(c);
    else if (c.wide) polyakov_kernel<float, WideLinks><<<g, TPB, 0, s>>>(c);
    else polyakov_kernel<float, Links<float>><<<g, TPB, 0, s>>>(c);
    if (out_signed_dev)
        finalize_kernel<<<dim3(c.n, 1), TPB, 0, s>>>(c, c.spat_start, c.spat_blocks, 1, 1,
                                                     out_signed_dev, out_abs_dev, accumulate);
    return cudaGetLastError();
}

cudaError_t launch_correlator(const Ctx& c, int dtype, int rmax, double* out_dev, int accumulate,
                              cudaStream_t s)
{
    if (dtype == 0) correlator_kernel<float><<<c.spat_blocks, TPB, 0, s>>>(c, rmax);
    else correlator_kernel<double><<<c.spat_blocks, TPB, 0, s>>>(c, rmax);
    finalize_kernel<<<dim3(c.n, rmax + 1), TPB, 0, s>>>(c, c.spat_start, c.spat_blocks, rmax + 1,
                                                        2, out_dev, nullptr, accumulate);
    return cudaGetLastError();
}

}  // namespace su2
