// su2_fixed.cuh -- the FP64 link update in 64-bit fixed point.
//
// GB300 issues an FP64 instruction every ~76 clocks per SM sub-partition and
// a 32 x 32 + 64-bit integer multiply-add (IMAD.WIDE) every 2 (both measured
// with independent chains, 8 warps per sub-partition).  The components of
// SU(2) links lie in [-1, 1], so the staple products, the
// Kennedy-Pendleton draw and the new link are computed here on 64-bit
// integers with a fixed binary point, each held as two signed 32-bit limbs
//   v = h 2^32 + l,  -2^31 <= l < 2^31,
// a product keeping h h' and the cross terms h l' + l h' (l l' is below the
// last place kept).  A quaternion product component is then 4 + 8 IMAD.WIDE
// (24 clocks) in place of 4 DFMA (~300).
//
// Precision: the links enter at 2^-61, the staple sum is kept at 2^-55 (an
// FP64 sum of the same size rounds to 2^-51) with one rounding per staple,
// the unit staple and the draw at 2^-57 .. 2^-62, the new link at 2^-60, and
// it is rounded once, to nearest, to the double that is stored.  The errors
// against 128-bit arithmetic are below those of the FP64 sequence
// (tests/test_fixed_point.py).
//
// Range: |sum of four h l'| <= |h|_1 2^31, and |h|_1 <= 2 |h|_2 for four
// components, so with unit quaternions at 2^61 (h <= 2^29) the two cross
// sums stay below 2 * 2^30 * 2^31 = 2^62.  Every bound is stated where it
// is used; they hold for links with | |U|^2 - 1 | <= 2^-10
// (UNIT_TOLERANCE), which a check before the sweeps establishes; a lattice
// with other links takes the FP64 sequence (general_link).
//
// Everything below is integer arithmetic but for one hardware reciprocal
// square root that seeds an exact refinement, so all kernels that call it
// give the same bits.  The functions are host functions too, for the tests.
#pragma once
#include <cmath>
#include <cstdint>
#ifdef __CUDACC__
#include <cuda_runtime.h>
#define SU2_HD __host__ __device__ __forceinline__
#else
#define SU2_HD inline
#endif

namespace su2 {

constexpr double UNIT_TOLERANCE = 1.0 / 1024.0;

// the tables (filled on the host): 512 intervals of the logarithm's argument
// and 1024 points of the circle, 16 bytes each
struct LnEntry {
    uint32_t g, pad;  // round(2^32 / c), c the centre of the interval of m in [1, 2)
    int64_t lng;      // ln(2 g 2^-32) at 2^61
};
struct TrigEntry {
    int64_t c, s;  // cos and sin of 2 pi j / 1024 at 2^62
};
constexpr int FIX_LN = 512, FIX_TRIG = 1024;
struct FixTables {
    LnEntry ln[FIX_LN];
    TrigEntry trig[FIX_TRIG];
};

// (long double: rounded once to the integers stored)
inline void fill_fix_tables(FixTables* t)
{
    for (int k = 0; k < FIX_LN; ++k) {
        const double c = 1.0 + (k + 0.5) / FIX_LN;
        const uint32_t g = (uint32_t)(4294967296.0 / c + 0.5);
        const long double l = logl((long double)g / 2147483648.0L);
        t->ln[k] = {g, 0u, (int64_t)llrintl(ldexpl(l, 61))};
    }
    const long double pi = acosl(-1.0L);
    for (int j = 0; j < FIX_TRIG; ++j) {
        const long double a = 2.0L * pi * (long double)j / (long double)FIX_TRIG;
        t->trig[j] = {(int64_t)llrintl(ldexpl(cosl(a), 62)), (int64_t)llrintl(ldexpl(sinl(a), 62))};
    }
}

// --------------------------------------------------------------------------
// integer pieces
// --------------------------------------------------------------------------
SU2_HD int clz64(uint64_t x)  // 64 for 0
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}
SU2_HD uint32_t mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
// a b + c in one instruction (written out on the device: the compiler would
// re-associate the integer sums into separate products and additions)
SU2_HD int64_t wide(int32_t a, int32_t b, int64_t c)
{
#ifdef __CUDA_ARCH__
    int64_t d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (int64_t)a * b + c;
#endif
}
// v >> n, 0 for n >= 64
SU2_HD uint64_t shr64(uint64_t v, uint32_t n)
{
#ifdef __CUDA_ARCH__
    uint64_t d;
    asm("shr.u64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(n));
    return d;
#else
    return n < 64 ? v >> n : 0;
#endif
}
SU2_HD int64_t shl64(int64_t v, int n) { return (int64_t)((uint64_t)v << n); }
SU2_HD int32_t hi32(int64_t v) { return (int32_t)(v >> 32); }

// v = h 2^32 + l
struct Fx {
    int32_t h, l;
};
SU2_HD Fx limbs(int64_t v)
{
    const int32_t l = (int32_t)v;
    // h = (v - l) / 2^32: the upper word plus bit 31 of the lower one
    return {(int32_t)((uint32_t)hi32(v) + ((uint32_t)l >> 31)), l};
}
// -v - 1 unit of the last place (the complement: -(-2^31) has no limb)
SU2_HD Fx neg(const Fx& a) { return {-a.h, ~a.l}; }

struct FQuat {
    Fx a0, a1, a2, a3;
};

// sums of h h' (units 2^64) and of the cross terms (units 2^32); the cross
// sum starts at the half that rounds the bits cut off it
constexpr int64_t HALF32 = int64_t(1) << 31;
struct Dot {
    int64_t hh, cr;
    SU2_HD void mac(const Fx& a, const Fx& b)
    {
        hh = wide(a.h, b.h, hh);
        cr = wide(a.h, b.l, cr);
        cr = wide(a.l, b.h, cr);
    }
    // the sum >> 64 and >> (64 - K), K < 32
    SU2_HD int64_t top() const { return wide(hi32(cr), 1, hh); }
    template <int K>
    SU2_HD int64_t top_k() const
    {
        return shl64(hh, K) + (cr >> (32 - K));
    }
};
// (a b) >> 64 and (a b) >> (64 - K)
SU2_HD int64_t mul64(const Fx& a, const Fx& b)
{
    Dot d{0, HALF32};
    d.mac(a, b);
    return d.top();
}
template <int K>
SU2_HD int64_t mulk(const Fx& a, const Fx& b)
{
    Dot d{0, HALF32 >> K};
    d.mac(a, b);
    return d.template top_k<K>();
}

// --------------------------------------------------------------------------
// doubles in and out
// --------------------------------------------------------------------------
// A link component |x| < 2 at 2^61 from the words of the double: the 53-bit
// mantissa shifted into place by its exponent, the sign by complement (one
// unit of 2^-61 off for negative values).  flip: the sign bit of -1 for
// the conjugate's vector part.
SU2_HD Fx fx_link(uint32_t hi, uint32_t lo, bool flip)
{
    const uint32_t n = ~(hi >> 20) & 0x3FFu;  // 1023 - exponent
    const uint32_t w1 = (((hi << 9) | (lo >> 23)) & 0x1FFFFFFFu) | 0x20000000u;
    const uint64_t w = ((uint64_t)w1 << 32) | (uint64_t)(lo << 9);
    const uint64_t v = shr64(w, n);
    const uint32_t sm = flip ? ~(uint32_t)((int32_t)hi >> 31) : (uint32_t)((int32_t)hi >> 31);
    const uint32_t vl = (uint32_t)v ^ sm, vh = (uint32_t)(v >> 32) ^ sm;
    return {(int32_t)(vh + (vl >> 31)), (int32_t)vl};
}
// v 2^e as the nearest double's bits (e such that the result is normal)
SU2_HD uint64_t double_bits(int64_t v, int e)
{
    const uint64_t sg = (uint64_t)v & 0x8000000000000000ull;
    const uint64_t a = v < 0 ? 0 - (uint64_t)v : (uint64_t)v;
    if (a == 0) return 0;
    const int z = clz64(a);
    const uint64_t m = a << z;  // bit 63 set
    // 53 bits, to nearest (ties up in magnitude): the rounding carry runs
    // on into the exponent
    const uint64_t r = (m >> 11) + ((m >> 10) & 1u);
    return sg | (((uint64_t)(uint32_t)(1023 + 63 - z + e - 1) << 52) + r);
}

// --------------------------------------------------------------------------
// products
// --------------------------------------------------------------------------
// p q^dagger: (p0 q0 + p.q, q0 p - p0 q + p x q)
template <typename F>
SU2_HD void nd_components(const FQuat& p, const FQuat& q, F f)
{
    const Fx n1 = neg(q.a1), n2 = neg(q.a2), n3 = neg(q.a3);
    f(0, p.a0, q.a0, p.a1, q.a1, p.a2, q.a2, p.a3, q.a3);
    f(1, p.a1, q.a0, p.a0, n1, p.a3, n2, p.a2, q.a3);
    f(2, p.a2, q.a0, p.a0, n2, p.a3, q.a1, p.a1, n3);
    f(3, p.a3, q.a0, p.a0, n3, p.a2, n1, p.a1, q.a2);
}

// links at 2^61 in, 2^58 out; |cross sum| <= 2 * 2^30 * 2^31
SU2_HD FQuat fq_mul_nd(const FQuat& p, const FQuat& q)
{
    int64_t r[4];
    nd_components(p, q, [&](int c, const Fx& x0, const Fx& y0, const Fx& x1, const Fx& y1,
                            const Fx& x2, const Fx& y2, const Fx& x3, const Fx& y3) {
        Dot d{0, HALF32};
        d.mac(x0, y0);
        d.mac(x1, y1);
        d.mac(x2, y2);
        d.mac(x3, y3);
        r[c] = d.top();
    });
    return {limbs(r[0]), limbs(r[1]), limbs(r[2]), limbs(r[3])};
}
// A += p q^dagger, p at 2^58, q a link at 2^61, A at 2^55 (six terms:
// |A| <= 6 * 2^55)
SU2_HD void fq_mul_nd_acc(const FQuat& p, const FQuat& q, int64_t* A)
{
    nd_components(p, q, [&](int c, const Fx& x0, const Fx& y0, const Fx& x1, const Fx& y1,
                            const Fx& x2, const Fx& y2, const Fx& x3, const Fx& y3) {
        Dot d{A[c], HALF32};
        d.mac(x0, y0);
        d.mac(x1, y1);
        d.mac(x2, y2);
        d.mac(x3, y3);
        A[c] = d.top();
    });
}

// --------------------------------------------------------------------------
// reciprocal square root
// --------------------------------------------------------------------------
// Y = 2^60 / sqrt(x), x = K 2^-60 in [2^-4, 1]: a hardware seed y0 of 22
// bits, its residual r = 1 - x y0^2 exactly modulo 2^64, and the third-order
// series y0 (1 + r/2 + 3 r^2/8) (|r| < 2^-20: the next term is 2^-62).
SU2_HD int64_t rsqrt_fix(uint64_t K)
{
    const float kf = (float)(int32_t)(K >> 30);  // x 2^30
#ifdef __CUDA_ARCH__
    const uint32_t y0 = (uint32_t)__float2int_rn(rsqrtf(kf) * 137438953472.0f);  // 2^37
#else
    const uint32_t y0 = (uint32_t)(1.0 / std::sqrt((double)kf) * 137438953472.0 + 0.5);
#endif
    // y0 = y 2^22 < 2^24.1, S = y0^2
    const uint64_t S = (uint64_t)y0 * y0;
    const uint32_t kh = (uint32_t)(K >> 32), kl = (uint32_t)K;
    const uint32_t sh = (uint32_t)(S >> 32), sl = (uint32_t)S;
    const uint64_t p0 = (uint64_t)kl * sl;
    const uint64_t p1 = (uint64_t)kh * sl + (p0 >> 32);
    const uint64_t p2 = (uint64_t)kl * sh + p1;  // < 2^62
    const uint64_t p3 = (uint64_t)kh * sh + (p2 >> 32);
    // K S at 2^104 = x y^2; bits 40 .. 103 of it, from 1 = 2^104
    const int64_t r = (int64_t)(0 - ((p3 << 24) | ((uint32_t)p2 >> 8)));  // at 2^64
    const int32_t rs = (int32_t)(r >> 16);  // at 2^48
    const int64_t r2 = wide(rs, rs, 0) >> 32;  // r^2 at 2^64
    const int64_t c = (r >> 1) + ((3 * r2) >> 3);
    // y0 c 2^-22 at 2^60 : y0 c >> 26
    const int64_t yc = shl64((int64_t)(int32_t)y0 * (c >> 32), 6) +
                       (int64_t)(((uint64_t)y0 * (uint32_t)c) >> 26);
    return ((int64_t)y0 << 38) + yc;
}

// --------------------------------------------------------------------------
// logarithm and circle of the random grids
// --------------------------------------------------------------------------
// -ln u = n' ln 2 + f, u = a 2^-24, a odd and below 2^24 (table-driven after
// Tang, ACM TOMS 15 (1989) 144): u = 2^-(n' + 1) m, m in [1, 2), r = m g - 1
// exactly with the 32-bit g of m's interval (|r| <= 2^-10), and
// f = ln 2 + ln g - ln(1 + r) in (0, ln 2] at 2^61,
// ln(1 + r) = r - r^2/2 + r^3 (1/3 - r (1/4 - r (1/5 - r/6))).
struct NegLn {
    int64_t f;
    int n;  // n'
};
SU2_HD NegLn neg_ln(uint32_t a, const FixTables* __restrict__ tab)
{
#ifdef __CUDA_ARCH__
    const int z = __clz((int)a);
#else
    const int z = __builtin_clz(a);
#endif
    const uint32_t m = a << z;  // m 2^31
    const LnEntry* e = &tab->ln[(m >> 22) & (FIX_LN - 1)];
#ifdef __CUDA_ARCH__
    const uint4 ev = __ldg(reinterpret_cast<const uint4*>(e));
    const uint32_t g = ev.x;
    const int64_t lng = (int64_t)(((uint64_t)ev.w << 32) | ev.z);
#else
    const uint32_t g = e->g;
    const int64_t lng = e->lng;
#endif
    const int64_t r = (int64_t)((uint64_t)m * g - (uint64_t(1) << 63));  // at 2^63
    const int32_t rh = (int32_t)(r >> 22);                               // at 2^41
    const int32_t rl = (int32_t)((uint32_t)r & 0x3FFFFFu);
    const int64_t r2 = wide(rh, rh, wide(rh, rl, 0) >> 21);              // at 2^82
    const int32_t r3 = hi32(wide((int32_t)(r2 >> 31), rh, 0));           // at 2^60
    const int32_t w2 = 429496730 - hi32(wide(rh, 699051, 0));            // 1/5 - r/6 at 2^31
    const int32_t w1 = 536870912 - (hi32(wide(rh, w2, 0)) >> 9);
    const int32_t w0 = 715827883 - (hi32(wide(rh, w1, 0)) >> 9);
    const int64_t ln1 = (r >> 2) - (r2 >> 22) + (wide(r3, w0, 0) >> 30);
    return {lng - ln1, z - 8};
}
// n' ln 2 + f at 2^57 (s = 4) or, for n' = 0, f itself at 2^61 (s = 0)
SU2_HD int64_t neg_ln_at(const NegLn& L, int s)
{
    constexpr int64_t LN2 = 99893036290645747ll;  // ln 2 at 2^57
    constexpr int32_t LN2_LO = 1469302631;        // and its rest at 2^89
    return (L.f >> s) + (int64_t)L.n * LN2 + (int64_t)((L.n * (int64_t)LN2_LO) >> 32);
}

// cos and sin of num 2^-23 turns at 2^62, num < 2^23 (any multiple of 2^23
// more is the same): the nearest of 1024 table points (C, S) and the rest b,
// |b| <= 2 pi / 2048:
//   cos = C + C (cos b - 1) - S sin b, sin = S + S (cos b - 1) + C sin b,
// cos b - 1 = -b^2/2 + b^4/24 - b^6/720, sin b = b - b^3 (1/6 - b^2/120).
struct Arc {
    Fx C, S, cm1, sb;
    int64_t c, s;
};
SU2_HD Arc arc_at(uint32_t num, const FixTables* __restrict__ tab)
{
    const uint32_t j = (num + 4096u) >> 13;
    const int32_t res = (int32_t)(num - (j << 13));
    const TrigEntry* e = &tab->trig[j & (FIX_TRIG - 1)];
    Arc A;
#ifdef __CUDA_ARCH__
    const uint4 ev = __ldg(reinterpret_cast<const uint4*>(e));
    A.c = (int64_t)(((uint64_t)ev.y << 32) | ev.x);
    A.s = (int64_t)(((uint64_t)ev.w << 32) | ev.z);
#else
    A.c = e->c;
    A.s = e->s;
#endif
    constexpr int64_t TWO_PI = 1768559438007110ll;  // 2 pi at 2^48
    const int64_t b71 = (int64_t)res * TWO_PI;      // b at 2^71, below 2^62.7
    const Fx b = limbs(b71);                        // b.h: b at 2^39
    const int64_t b2 = wide(b.h, b.h, wide(b.h, b.l, 0) >> 31);  // b^2 at 2^78
    const uint32_t q = (uint32_t)(b2 >> 30);                     // at 2^48
    const uint32_t b4 = mulhi32(q, q);                           // at 2^64
    const uint32_t b6 = mulhi32(b4, q);                          // at 2^80
    A.cm1 = limbs((int64_t)(mulhi32(b4, 44739243u) - mulhi32(b6, 23u)) - (b2 >> 17));
    const int64_t b3 = wide(b.h, (int32_t)(q >> 1), 0);          // b^3 at 2^86
    const int32_t w = 1431655765 - (int32_t)mulhi32(q, 1092u);   // 1/6 - b^2/120 at 2^33
    A.sb = limbs((b71 >> 9) - (wide((int32_t)(b3 >> 30), w, 0) >> 27));
    A.C = limbs(A.c);
    A.S = limbs(A.s);
    return A;
}
SU2_HD int64_t arc_cos(const Arc& A)
{
    Dot d{0, HALF32 >> 2};
    d.mac(A.C, A.cm1);
    d.mac(neg(A.S), A.sb);
    return A.c + d.top_k<2>();
}
SU2_HD int64_t arc_sin(const Arc& A)
{
    Dot d{0, HALF32 >> 2};
    d.mac(A.S, A.cm1);
    d.mac(A.C, A.sb);
    return A.s + d.top_k<2>();
}

// --------------------------------------------------------------------------
// the draw
// --------------------------------------------------------------------------
// What a link's draw needs of its staple sum A: the unit quaternion
// V = A / |A| at 2^58, and 1 / (2 alpha) = inv 2^ei, inv in [2^61, 2^62).
struct Drawn {
    FQuat V;
    int64_t inv;
    int ei;
};

// 1 / (2 beta) as a mantissa in [2^61, 2^62) and an exponent
struct HalfInvBeta {
    Fx g;
    int e;
};
SU2_HD HalfInvBeta half_inv_beta_fix(uint64_t bits)
{
    const int64_t m = (int64_t)(((bits & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 9);
    return {limbs(m), (int)((bits >> 52) & 0x7FFu) - 1084};
}

// false for a zero staple.  *root = |A| 2^62 2^(n - 7), the caller's alpha.
SU2_HD bool unit_staple(const int64_t* A, const HalfInvBeta& hb, Drawn* D, uint64_t* K2, int* sc)
{
    uint64_t m = 0;
    for (int c = 0; c < 4; ++c) m |= (uint64_t)(A[c] ^ (A[c] >> 63));
    // the largest component in [2^60, 2^61) (a negative power of two may
    // reach 2^61): h <= 2^29, |cross sum| <= 4 * 2^29 * 2^31
    const int n = clz64(m) - 3;
    if (n > 60) return false;
    Fx B[4];
    Dot d{0, HALF32 >> 1};
    for (int c = 0; c < 4; ++c) {
        B[c] = limbs(shl64(A[c], n));
        d.hh = wide(B[c].h, B[c].h, d.hh);
        d.cr = wide(B[c].h, B[c].l, d.cr);
    }
    const uint64_t K = (uint64_t)(d.hh + (d.cr >> 31));  // |B|^2 2^-64, in [2^56, 2^60]
    const int64_t Y = rsqrt_fix(K);                      // |A| = 2^60 / Y * 2^(7 - n)
    const Fx y = limbs(Y);
    D->V = {limbs(mul64(B[0], y)), limbs(mul64(B[1], y)), limbs(mul64(B[2], y)),
            limbs(mul64(B[3], y))};
    const int64_t J = mulk<2>(y, hb.g);  // in [2^59, 2^62)
    const int s = clz64((uint64_t)J) - 2;
    D->inv = shl64(J, s);
    D->ei = hb.e + n - 5 - s;
    *K2 = K;
    *sc = n;
    return true;
}

// lambda^2 of one Kennedy-Pendleton trial as P 2^qe, P in [2^60, 2^62), and
// at 2^61 where it is below 2 (lam < 0 otherwise)
struct Lambda {
    int64_t P, lam;
    int qe;
};
SU2_HD Lambda lambda_of(int64_t P, int qe)
{
    const int s = -(qe + 61);
    return {P, s < 0 ? int64_t(-1) : (int64_t)shr64((uint64_t)P, (uint32_t)s), qe};
}
SU2_HD Lambda kp_lambda(uint32_t w0, uint32_t w1, uint32_t w2, int64_t inv, int ei,
                        const FixTables* __restrict__ tab)
{
    const NegLn l1 = neg_ln(2u * (w0 >> 9) + 1u, tab), l3 = neg_ln(2u * (w2 >> 9) + 1u, tab);
    // the logarithms at 2^57 (up to 16.64), or at 2^61 where both uniforms
    // are above 1/2, so that a small sum keeps its accuracy
    const int s = (l1.n | l3.n) == 0 ? 0 : 4;
    const int64_t L1 = neg_ln_at(l1, s), L3 = neg_ln_at(l3, s);
    // cos^2(2 pi r2) = (1 + cos(4 pi r2)) / 2, 2 r2 = (2k + 1) 2^-23 turns
    const Arc a = arc_at((2u * (w1 >> 9) + 1u) & 0x7FFFFFu, tab);
    const int64_t c2 = ((int64_t(1) << 62) + arc_cos(a)) >> 1;
    const uint64_t T = (uint64_t)(L1 + mulk<2>(limbs(c2), limbs(L3)));  // below 2^62.1
    const int z = clz64(T);
    const int64_t t = (int64_t)((T << z) >> 2);  // in [2^61, 2^62)
    return lambda_of(mulk<2>(limbs(t), limbs(inv)), 3 + s - z + ei);
}
// accepted iff r4^2 <= 1 - lambda^2
SU2_HD bool kp_accept(const Lambda& L, uint32_t w3)
{
    const uint32_t a = 2u * (w3 >> 9) + 1u;
    return L.lam >= 0 && (int64_t)(((uint64_t)a * a) << 13) <= (int64_t(1) << 61) - L.lam;
}
// lambda^2 = delta / 2 from the bits of a double 0 < delta <= 2
SU2_HD Lambda lambda_from_delta(uint64_t bits)
{
    const int64_t m = (int64_t)(((bits & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 9);
    const int e = (int)((bits >> 52) & 0x7FFu);
    return e == 0 ? Lambda{int64_t(1) << 61, 0, -1100} : lambda_of(m, e - 1085);
}

// sqrt(v 2^e) at 2^62 for v in [2^58, 2^63), v 2^e <= 1
SU2_HD int64_t sqrt_fix(uint64_t v, int e)
{
    const int z = clz64(v);
    v = z >= 2 ? v << (z - 2) : v >> 1;
    e -= z - 2;
    const int sh = 2 + (e & 1);
    const uint64_t K = v >> sh;  // in [2^58, 2^60)
    const Fx y = limbs(rsqrt_fix(K)), k = limbs((int64_t)K);
    // sqrt(x) = x / sqrt(x) at 2^63, x = K 2^-60 in [1/4, 1)
    const uint64_t r = (uint64_t)mulk<7>(k, y);
    const int s = -(29 + (e + sh) / 2);  // right shift to 2^62, >= 0
    return (int64_t)shr64(r, (uint32_t)s);
}

// The new link X V^dagger at 2^60, X = (1 - delta, |x| n): |x|^2 =
// delta (2 - delta) = 4 lambda^2 (1 - lambda^2), the direction n from the two
// 18-bit integers of the first trial.  X and V are unit to 2^-57, so the
// product needs no normalisation.
SU2_HD void new_link_fix(const Lambda& L, uint32_t kd1, uint32_t kd2, const FQuat& V,
                         const FixTables* __restrict__ tab, int64_t* U)
{
    const int64_t W = (int64_t(1) << 61) - L.lam;  // 1 - lambda^2 >= 0
    const int nw = clz64((uint64_t)W | 1u) - 2;
    const int64_t Q = mulk<2>(limbs(L.P), limbs(shl64(W, nw)));  // in [2^59, 2^62)
    // |x|^2 / 4 = Q 2^(qe - nw + 1): |x| = sqrt(Q 2^(qe - nw + 3))
    const int64_t vl = W == 0 ? 0 : sqrt_fix((uint64_t)Q, L.qe - nw + 3);
    const int32_t cth = (int32_t)(2u * kd1 + 1u) - (1 << 18);  // at 2^18
    const uint64_t N = (uint64_t(1) << 36) - (uint64_t)((int64_t)cth * cth);
    const int zn = (clz64(N) - 4) & ~1;
    const int64_t sth = sqrt_fix(N << zn, -36 - zn);
    const Fx v = limbs(vl);
    const Fx vs = limbs(mulk<2>(v, limbs(sth)));
    const Arc a = arc_at((2u * kd2 + 1u) << 4, tab);
    FQuat X;
    X.a0 = limbs((int64_t(1) << 62) - shl64(L.lam, 2));
    X.a1 = limbs(mulk<2>(vs, limbs(arc_cos(a))));
    X.a2 = limbs(mulk<2>(vs, limbs(arc_sin(a))));
    X.a3 = limbs(shl64((int64_t)v.h * cth, 14) + (((int64_t)v.l * cth) >> 18));
    // |cross sum| <= 2 * 2^30 * 2^31 + 2 * 2^26 * 2^31
    nd_components(X, V, [&](int c, const Fx& x0, const Fx& y0, const Fx& x1, const Fx& y1,
                            const Fx& x2, const Fx& y2, const Fx& x3, const Fx& y3) {
        Dot d{0, HALF32 >> 4};
        d.mac(x0, y0);
        d.mac(x1, y1);
        d.mac(x2, y2);
        d.mac(x3, y3);
        U[c] = d.top_k<4>();
    });
}

// 1/2 Tr(U P) at 2^51, U at 2^60, P (a part of A) at 2^55
SU2_HD int64_t retr_fix(const int64_t* U, const int64_t* P)
{
    Dot d{0, HALF32};
    d.mac(limbs(U[0]), limbs(P[0]));
    for (int c = 1; c < 4; ++c) d.mac(neg(limbs(U[c])), limbs(P[c]));
    return d.top();
}

}  // namespace su2
