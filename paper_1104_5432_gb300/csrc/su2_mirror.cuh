// su2_mirror.cuh -- the fixed-point copy of an FP64 handle's links.
//
// A link is read 18 times for each time it is written, and turning its double
// components into limbs takes ~11 instructions each, a fifth of an update.
// So the sweeps of a call read a copy of the links in limbs, written before
// the first sweep (with the look at the links' norms) and kept in step by
// the updates, which store both: int4 M[mu][parity][plane][eo], plane 0 =
// the limbs of (a0, a1), plane 1 = (a2, a3), the doubles' layout and size.
// The copy is exactly fx_link of the stored double, so a kernel that reads the
// doubles gives the same bits.  Measured at 64^4, beta = 2.5: 5.76 -> 6.76 G
// link updates/s, for 0.7 ms of copying per call.
#pragma once
#include "su2_fixed.cuh"
#include "su2_links.cuh"

namespace su2 {

__device__ __forceinline__ FQuat fq_link(const Quat<double>& q)
{
    auto f = [](double x) {
        return fx_link((uint32_t)__double2hiint(x), (uint32_t)__double2loint(x));
    };
    return {f(q.a0), f(q.a1), f(q.a2), f(q.a3)};
}

// A link component as a float (0 below 2^-126, at least 2 for |x| >= 2, an
// infinity or a NaN), from its words: conversion instructions run on the
// slow FP64 unit.
__device__ __forceinline__ float narrow(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7FFu;
    if (e > 1023u) return 2.0f;
    if (e < 897u) return 0.0f;
    return __uint_as_float((((hi & 0x7FFFFFFFu) << 3) | (lo >> 29)) - (896u << 23));
}
__device__ __forceinline__ bool unit_link(const double2& lo, const double2& hi)
{
    const float a = narrow(lo.x), b = narrow(lo.y), c = narrow(hi.x), d = narrow(hi.y);
    return fabsf(a * a + b * b + c * c + d * d - 1.0f) <= (float)UNIT_TOLERANCE;
}
// The same from the link's limbs f = fq_link(q) (a third of the instructions:
// 18 links of an update, 64^4 1790 -> 1480 us a single phase): no component of
// magnitude 2 or more, an infinity or a NaN among them, and sum h^2 2^-58
// within 2^-10 of 1.
__device__ __forceinline__ bool unit_limbs(const Quat<double>& q, const FQuat& f)
{
    const int hi = __double2hiint(q.a0) | __double2hiint(q.a1) | __double2hiint(q.a2) | __double2hiint(q.a3);
    const int64_t n = mulw(f.a0.h, f.a0.h) + mulw(f.a1.h, f.a1.h) + mulw(f.a2.h, f.a2.h) +
                      mulw(f.a3.h, f.a3.h);
    constexpr uint32_t ONE = 1u << 26, TOL = 1u << 16;  // at 2^26
    static_assert(UNIT_TOLERANCE * ONE == TOL, "the same bound");
    return (hi & 0x40000000) == 0 && (uint32_t)hi32(n) - (ONE - TOL) <= 2 * TOL;
}
// a quaternion at 2^60 as doubles
__device__ __forceinline__ Quat<double> dq_link(const int64_t* U)
{
    auto f = [](int64_t v) { return __longlong_as_double((long long)double_bits(v, -60)); };
    return {f(U[0]), f(U[1]), f(U[2]), f(U[3])};
}
__device__ __forceinline__ Quat<double> haar_double(const U4& w, const FixTables* tab)
{
    int64_t U[4];
    haar_fix(w.x, w.y, w.z, w.w, tab, U);
    return dq_link(U);
}

struct FixMirror {
    int4* base;
    uint32_t Vh;
    LinkCheck chk;
    __device__ __forceinline__ FixMirror(const Ctx& c, const LatDesc& d)
        : base(reinterpret_cast<int4*>(reinterpret_cast<char*>(c.mirror) + d.link_off)), Vh(d.Vh)
    {
#ifdef SU2_CHECK_BOUNDS
        chk = {c.status, d.Vh};
#endif
    }
    __device__ __forceinline__ size_t idx(int mu, int p, uint32_t eo) const
    {
        return chk.ok(mu, p, eo) ? size_t((mu * 2 + p) * 2) * Vh + eo : 0;
    }
    __device__ __forceinline__ FQuat load(int mu, int p, uint32_t eo) const
    {
        const int4* a = base + idx(mu, p, eo);
        const int4 lo = __ldg(a), hi = __ldg(a + Vh);
        return {{lo.x, lo.y}, {lo.z, lo.w}, {hi.x, hi.y}, {hi.z, hi.w}};
    }
    __device__ __forceinline__ void store(int mu, int p, uint32_t eo, const Quat<double>& q) const
    {
        if (!chk.ok(mu, p, eo)) return;
        int4* a = base + size_t((mu * 2 + p) * 2) * Vh + eo;
        const FQuat f = fq_link(q);
        a[0] = make_int4(f.a0.h, f.a0.l, f.a1.h, f.a1.l);
        a[Vh] = make_int4(f.a2.h, f.a2.l, f.a3.h, f.a3.l);
    }
};

}  // namespace su2
