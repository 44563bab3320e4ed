// su2_fixed.cuh -- the FP64 link update in 64-bit fixed point.
//
// GB300 issues an FP64 instruction every ~62-76 clocks per SM sub-partition, a
// 32 x 32 -> 64-bit integer product every 2 and a 32-bit addition every clock
// (a multiply-add with a 64-bit addend is a product and a 64-bit addition and
// took 6: measured with independent chains, 8 warps per sub-partition).  The
// components of SU(2) links lie in [-1, 1], so the staple products, the
// Kennedy-Pendleton draw and the new link are computed here on 64-bit
// integers with a fixed binary point, each held as two signed 32-bit limbs
//   v = h 2^32 + l,  -2^31 <= l < 2^31,
// a product keeping h h' and the upper words of the cross terms h l', l h'
// (l l' is below the last place kept).  A quaternion product component is
// then 4 + 8 products and ten additions (~24 clocks) in place of 4 DFMA
// (~300).
//
// Precision: the links enter at 2^-61, the staple sum is kept at 2^-55 (an
// FP64 sum of the same size rounds to 2^-51) with one rounding per staple,
// the unit staple and the draw at 2^-57 .. 2^-62, the new link at 2^-60, and
// it is rounded once, to nearest, to the double that is stored.  These are
// absolute errors, where a double's shrink with its value, and the vector part
// of a link at coupling beta is of the size of beta^-1/2: its rms error
// against extended precision is 0.2 of the FP64 sequence's at beta = 2.3, 0.36
// to 0.49 at 64, the same from about 300 on and 12 to 15 times larger at 10^5
// (tests/test_fixed_point.py).  So lattices at couplings above FIX_BETA_MAX
// take the FP64 sequence (general_link), at its speed: beta = 1000, us a
// sweep, 8^4 92, 16^4 217, 32^4 2557, 64^4 39800 (fixed point 36, 80, 594, 8654).
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
constexpr double FIX_BETA_MAX = 64.0;

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
// a b, one instruction (written out on the device: the compiler takes limbs
// cut out of 64-bit values for 64-bit factors)
SU2_HD int64_t mulw(int32_t a, int32_t b)
{
#ifdef __CUDA_ARCH__
    int64_t d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (int64_t)a * b;
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
// -v; for limbs with l != -2^31 (links and unit staples have odd l)
SU2_HD Fx neg(const Fx& a) { return {-a.h, -a.l}; }
SU2_HD Fx neg_if(const Fx& a, bool n) { return n ? neg(a) : a; }
// limbs of v with its last bit set: odd l
SU2_HD Fx limbs_odd(int64_t v) { return limbs(v | 1); }

struct FQuat {
    Fx a0, a1, a2, a3;
};

// (sum of four a b) >> 64, of the eight cross terms the upper words only
// (|their sum| < 2^31 where it is used; + 4: half a unit for each word cut
// off, at most 4 units wrong where the low words vanish)
SU2_HD int64_t dot4(const Fx& x0, const Fx& y0, const Fx& x1, const Fx& y1, const Fx& x2, const Fx& y2,
                    const Fx& x3, const Fx& y3)
{
    const int32_t c0 = hi32(mulw(x0.h, y0.l)) + hi32(mulw(x0.l, y0.h)) + 4;
    const int32_t c1 = hi32(mulw(x1.h, y1.l)) + hi32(mulw(x1.l, y1.h)) + c0;
    const int32_t c2 = hi32(mulw(x2.h, y2.l)) + hi32(mulw(x2.l, y2.h)) + c1;
    const int32_t c3 = hi32(mulw(x3.h, y3.l)) + hi32(mulw(x3.l, y3.h)) + c2;
    const int64_t hh = mulw(x0.h, y0.h) + mulw(x1.h, y1.h) + (int64_t)c3;
    return hh + mulw(x2.h, y2.h) + mulw(x3.h, y3.h);
}
// the cross terms in 64 bits, and the h h' products added to acc
SU2_HD int64_t cross4(int64_t cr, const Fx& x0, const Fx& y0, const Fx& x1, const Fx& y1,
                      const Fx& x2, const Fx& y2, const Fx& x3, const Fx& y3)
{
    cr = cr + mulw(x0.h, y0.l) + mulw(x0.l, y0.h);
    cr = cr + mulw(x1.h, y1.l) + mulw(x1.l, y1.h);
    cr = cr + mulw(x2.h, y2.l) + mulw(x2.l, y2.h);
    return cr + mulw(x3.h, y3.l) + mulw(x3.l, y3.h);
}
SU2_HD int64_t high4(int64_t acc, const Fx& x0, const Fx& y0, const Fx& x1, const Fx& y1,
                     const Fx& x2, const Fx& y2, const Fx& x3, const Fx& y3)
{
    acc = acc + mulw(x0.h, y0.h) + mulw(x1.h, y1.h);
    return acc + mulw(x2.h, y2.h) + mulw(x3.h, y3.h);
}
// acc + (sum of four a b) >> 64, rounded once
SU2_HD int64_t dot4_acc(int64_t acc, const Fx& x0, const Fx& y0, const Fx& x1, const Fx& y1,
                        const Fx& x2, const Fx& y2, const Fx& x3, const Fx& y3)
{
    const int64_t cr = cross4(int64_t(1) << 31, x0, y0, x1, y1, x2, y2, x3, y3);
    return high4(acc + (int64_t)hi32(cr), x0, y0, x1, y1, x2, y2, x3, y3);
}
// (sum of four a b) >> (64 - K), rounded
template <int K>
SU2_HD int64_t dot4_k(const Fx& x0, const Fx& y0, const Fx& x1, const Fx& y1, const Fx& x2, const Fx& y2,
                      const Fx& x3, const Fx& y3)
{
    const int64_t cr = cross4(int64_t(1) << (31 - K), x0, y0, x1, y1, x2, y2, x3, y3);
    return shl64(high4(0, x0, y0, x1, y1, x2, y2, x3, y3), K) + (cr >> (32 - K));
}
// (a b) >> 64
SU2_HD int64_t mul64(const Fx& a, const Fx& b)
{
    return mulw(a.h, b.h) + (int64_t)(hi32(mulw(a.h, b.l)) + hi32(mulw(a.l, b.h)) + 1);
}
// (a b + c d) >> (64 - K) and (a b) >> (64 - K), 0 < K < 32, rounded; the
// terms l l' left out are below 2^(K-2) each
template <int K>
SU2_HD int64_t mulk2(const Fx& a, const Fx& b, const Fx& c, const Fx& d)
{
    const int64_t hh = mulw(a.h, b.h) + mulw(c.h, d.h);
    const int64_t cr = mulw(a.h, b.l) + mulw(a.l, b.h) + (int64_t(1) << (31 - K));
    return shl64(hh, K) + ((cr + mulw(c.h, d.l) + mulw(c.l, d.h)) >> (32 - K));
}
template <int K>
SU2_HD int64_t mulk(const Fx& a, const Fx& b)
{
    const int64_t cr = mulw(a.h, b.l) + mulw(a.l, b.h) + (int64_t(1) << (31 - K));
    return shl64(mulw(a.h, b.h), K) + (cr >> (32 - K));
}

// --------------------------------------------------------------------------
// doubles in and out
// --------------------------------------------------------------------------
// A link component |x| < 2 at 2^61 from the words of the double: the 53-bit
// mantissa shifted into place by its exponent, the sign by complement, the
// last bit set (l odd; the value within one unit of 2^-61).
SU2_HD Fx fx_link(uint32_t hi, uint32_t lo)
{
    const uint32_t n = ~(hi >> 20) & 0x3FFu;  // 1023 - exponent
    const uint32_t w1 = (((hi << 9) | (lo >> 23)) & 0x1FFFFFFFu) | 0x20000000u;
    const uint64_t v = shr64(((uint64_t)w1 << 32) | (uint64_t)(lo << 9), n);
    const uint32_t sm = (uint32_t)((int32_t)hi >> 31);
    const uint32_t vl = ((uint32_t)v ^ sm) | 1u, vh = (uint32_t)(v >> 32) ^ sm;
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
// x y^dagger = (x0 y0 + x.y, y0 x - x0 y + x cross y), links at 2^61 in, 2^58
// out; |sum of the cross words| <= 2 * 2 * 2^29 / 2 = 2^30
SU2_HD FQuat fq_mul_nd(const FQuat& x, const FQuat& y)
{
    const Fx n1 = neg(y.a1), n2 = neg(y.a2), n3 = neg(y.a3);
    return {limbs(dot4(x.a0, y.a0, x.a1, y.a1, x.a2, y.a2, x.a3, y.a3)),
            limbs(dot4(x.a1, y.a0, x.a0, n1, x.a3, n2, x.a2, y.a3)),
            limbs(dot4(x.a2, y.a0, x.a0, n2, x.a3, y.a1, x.a1, n3)),
            limbs(dot4(x.a3, y.a0, x.a0, n3, x.a2, n1, x.a1, y.a2))};
}
// A += g z^dagger, or with `lower` g^dagger z: (g0 z0 + g.z, +-(z0 g - g0 z) +
// g cross z).  g at 2^58, z a link at 2^61, A at 2^55 (six terms: |A| <= 6 *
// 2^55); |sum of the cross terms| <= 2 * 2^30 * 2^31
SU2_HD void fq_acc(const FQuat& g, const FQuat& z, bool lower, int64_t* A)
{
    const Fx n1 = neg(z.a1), n2 = neg(z.a2), n3 = neg(z.a3);
    const Fx s0 = neg_if(z.a0, lower);
    const Fx &t1 = lower ? z.a1 : n1, &t2 = lower ? z.a2 : n2, &t3 = lower ? z.a3 : n3;
    A[0] = dot4_acc(A[0], g.a0, z.a0, g.a1, z.a1, g.a2, z.a2, g.a3, z.a3);
    A[1] = dot4_acc(A[1], g.a1, s0, g.a0, t1, g.a3, n2, g.a2, z.a3);
    A[2] = dot4_acc(A[2], g.a2, s0, g.a0, t2, g.a3, z.a1, g.a1, n3);
    A[3] = dot4_acc(A[3], g.a3, s0, g.a0, t3, g.a2, n1, g.a1, z.a2);
}
// One staple term: the upper x y^dagger z^dagger with (x, y, z) = (U_nu(x+mu),
// U_mu(x+nu), U_nu(x)), or the lower (x y)^dagger z with (U_mu(x-nu),
// U_nu(x+mu-nu), U_nu(x-nu)), added to A.
SU2_HD void fq_staple(const FQuat& x, const FQuat& y, const FQuat& z, bool lower, int64_t* A)
{
    const FQuat yc = {y.a0, neg_if(y.a1, lower), neg_if(y.a2, lower), neg_if(y.a3, lower)};
    fq_acc(fq_mul_nd(x, yc), z, lower, A);
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
    const int64_t r2 = mulw(rs, rs) >> 32;  // r^2 at 2^64
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
    const int64_t r2 = mulw(rh, rh) + (mulw(rh, rl) >> 21);              // at 2^82
    const int32_t r3 = hi32(mulw((int32_t)(r2 >> 31), rh));           // at 2^60
    const int32_t w2 = 429496730 - hi32(mulw(rh, 699051));            // 1/5 - r/6 at 2^31
    const int32_t w1 = 536870912 - (hi32(mulw(rh, w2)) >> 9);
    const int32_t w0 = 715827883 - (hi32(mulw(rh, w1)) >> 9);
    const int64_t ln1 = (r >> 2) - (r2 >> 22) + (mulw(r3, w0) >> 30);
    return {lng - ln1, z - 8};
}
// n' ln 2 + f at 2^57 (s = 4) or, for n' = 0, f itself at 2^61 (s = 0)
SU2_HD int64_t neg_ln_at(const NegLn& L, int s)
{
    constexpr int64_t LN2 = 99893036290645747ll;  // ln 2 at 2^57
    constexpr int32_t LN2_LO = 1469302631;        // and its rest at 2^89
    return (L.f >> s) + (int64_t)L.n * LN2 + (int64_t)hi32(mulw(L.n, LN2_LO));
}

// cos and sin of num 2^-24 turns at 2^62, num < 2^24 (any multiple of 2^24
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
    const uint32_t j = (num + 8192u) >> 14;
    const int32_t res = (int32_t)(num - (j << 14));
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
    constexpr int64_t TWO_PI = 884279719003555ll;   // 2 pi at 2^47
    const int64_t b71 = (int64_t)res * TWO_PI;      // b at 2^71, below 2^62.7
    const Fx b = limbs(b71);                        // b.h: b at 2^39
    const int64_t b2 = mulw(b.h, b.h) + (mulw(b.h, b.l) >> 31);  // b^2 at 2^78
    const uint32_t q = (uint32_t)(b2 >> 30);                     // at 2^48
    const uint32_t b4 = mulhi32(q, q);                           // at 2^64
    const uint32_t b6 = mulhi32(b4, q);                          // at 2^80
    A.cm1 = limbs((int64_t)(mulhi32(b4, 44739243u) - mulhi32(b6, 23u)) - (b2 >> 17));
    const int64_t b3 = mulw(b.h, (int32_t)(q >> 1));          // b^3 at 2^86
    const int32_t w = 1431655765 - (int32_t)mulhi32(q, 1092u);   // 1/6 - b^2/120 at 2^33
    A.sb = limbs((b71 >> 9) - (mulw((int32_t)(b3 >> 30), w) >> 27));
    A.C = limbs(A.c);
    A.S = limbs(A.s);
    return A;
}
SU2_HD int64_t arc_cos(const Arc& A)
{
    return A.c + mulk2<2>(A.C, A.cm1, limbs(-A.s), A.sb);
}
SU2_HD int64_t arc_sin(const Arc& A) { return A.s + mulk2<2>(A.S, A.cm1, A.C, A.sb); }

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
    const Fx B[4] = {limbs(shl64(A[0], n)), limbs(shl64(A[1], n)), limbs(shl64(A[2], n)),
                     limbs(shl64(A[3], n))};
    int64_t hh = mulw(B[0].h, B[0].h) + mulw(B[1].h, B[1].h);
    hh = hh + mulw(B[2].h, B[2].h) + mulw(B[3].h, B[3].h);
    int64_t cr = mulw(B[0].h, B[0].l) + mulw(B[1].h, B[1].l) + (int64_t(1) << 30);
    cr = cr + mulw(B[2].h, B[2].l) + mulw(B[3].h, B[3].l);
    const uint64_t K = (uint64_t)(hh + (cr >> 31));  // |B|^2 2^-64, in [2^56, 2^60]
    const int64_t Y = rsqrt_fix(K);                  // |A| = 2^60 / Y * 2^(7 - n)
    const Fx y = limbs(Y);
    D->V = {limbs_odd(mul64(B[0], y)), limbs_odd(mul64(B[1], y)), limbs_odd(mul64(B[2], y)),
            limbs_odd(mul64(B[3], y))};
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
// -(ln r1 + cos^2(2 pi r2) ln r3) = t 2^e, t in [2^61, 2^62): lambda^2 times
// 2 alpha, which needs no staple
struct KpSum {
    int64_t t;
    int e;
};
SU2_HD KpSum kp_sum(uint32_t w0, uint32_t w1, uint32_t w2, const FixTables* __restrict__ tab)
{
    const NegLn l1 = neg_ln(2u * (w0 >> 9) + 1u, tab), l3 = neg_ln(2u * (w2 >> 9) + 1u, tab);
    // the logarithms at 2^57 (up to 16.64), or at 2^61 where both uniforms
    // are above 1/2, so that a small sum keeps its accuracy
    const int s = (l1.n | l3.n) == 0 ? 0 : 4;
    const int64_t L1 = neg_ln_at(l1, s), L3 = neg_ln_at(l3, s);
    // cos^2(2 pi r2) = (1 + cos(4 pi r2)) / 2, 2 r2 = 2 (2k + 1) 2^-24 turns
    const Arc a = arc_at((4u * (w1 >> 9) + 2u) & 0xFFFFFFu, tab);
    const int64_t c2 = ((int64_t(1) << 62) + arc_cos(a)) >> 1;
    const uint64_t T = (uint64_t)(L1 + mulk<2>(limbs(c2), limbs(L3)));  // below 2^62.1
    const int z = clz64(T);
    return {(int64_t)((T << z) >> 2), s - z - 59};
}
SU2_HD Lambda kp_lambda(const KpSum& k, int64_t inv, int ei)
{
    return lambda_of(mulk<2>(limbs(k.t), limbs(inv)), 62 + k.e + ei);
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

// sqrt(v 2^e) at 2^62 for 0 < v < 2^63, v 2^e <= 1
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
// the direction: cos theta at 2^18, the rest at 2^62
struct FixDir {
    int32_t cth;
    int64_t sth, cph, sph;
};
SU2_HD FixDir direction_fix(uint32_t kd1, uint32_t kd2, const FixTables* __restrict__ tab)
{
    FixDir d;
    d.cth = (int32_t)(2u * kd1 + 1u) - (1 << 18);
    const uint64_t N = (uint64_t(1) << 36) - (uint64_t)((int64_t)d.cth * d.cth);
    const int zn = (clz64(N) - 4) & ~1;
    d.sth = sqrt_fix(N << zn, -36 - zn);
    const Arc a = arc_at((2u * kd2 + 1u) << 5, tab);
    d.cph = arc_cos(a);
    d.sph = arc_sin(a);
    return d;
}
SU2_HD void new_link_dir_fix(const Lambda& L, const FixDir& d, const FQuat& V, int64_t* U)
{
    const int64_t W = (int64_t(1) << 61) - L.lam;  // 1 - lambda^2 >= 0
    const int nw = clz64((uint64_t)W | 1u) - 2;
    const int64_t Q = mulk<2>(limbs(L.P), limbs(shl64(W, nw)));  // in [2^59, 2^62)
    // |x|^2 / 4 = Q 2^(qe - nw + 1): |x| = sqrt(Q 2^(qe - nw + 3))
    const int64_t vl = W == 0 ? 0 : sqrt_fix((uint64_t)Q, L.qe - nw + 3);
    const Fx v = limbs(vl);
    const Fx vs = limbs(mulk<2>(v, limbs(d.sth)));
    FQuat X;
    X.a0 = limbs((int64_t(1) << 62) - shl64(L.lam, 2));
    X.a1 = limbs(mulk<2>(vs, limbs(d.cph)));
    X.a2 = limbs(mulk<2>(vs, limbs(d.sph)));
    X.a3 = limbs(shl64((int64_t)v.h * d.cth, 14) + (((int64_t)v.l * d.cth) >> 18));
    // |sum of the cross terms| <= 2 * 2^30 * 2^31 + 2 * 2^26 * 2^31
    const Fx n1 = neg(V.a1), n2 = neg(V.a2), n3 = neg(V.a3);
    U[0] = dot4_k<4>(X.a0, V.a0, X.a1, V.a1, X.a2, V.a2, X.a3, V.a3);
    U[1] = dot4_k<4>(X.a1, V.a0, X.a0, n1, X.a3, n2, X.a2, V.a3);
    U[2] = dot4_k<4>(X.a2, V.a0, X.a0, n2, X.a3, V.a1, X.a1, n3);
    U[3] = dot4_k<4>(X.a3, V.a0, X.a0, n3, X.a2, n1, X.a1, V.a2);
}
SU2_HD void new_link_fix(const Lambda& L, uint32_t kd1, uint32_t kd2, const FQuat& V,
                         const FixTables* __restrict__ tab, int64_t* U)
{
    new_link_dir_fix(L, direction_fix(kd1, kd2, tab), V, U);
}

// Haar element of SU(2) at 2^60 from one Philox block: Box-Muller on (w0, w1)
// and (w2, w3), normalised.  With L = -ln u the four normals are sqrt(2 L0)
// (cos, sin)(2 pi u1) and sqrt(2 L2) (cos, sin)(2 pi u3), so their lengths
// over the norm are sqrt(L0 / (L0 + L2)) and sqrt(L2 / (L0 + L2)).
// Within 2^-12 of 1 a logarithm is taken at 2^73, so that a small one keeps
// its accuracy: -ln(1 - v) = v + v^2/2 + v^3/3 + v^4/4, v = j 2^-24, j < 4096.
SU2_HD int64_t small_neg_ln(uint32_t j)
{
    const uint64_t j2 = (uint64_t)j * j;
    return (int64_t)(((uint64_t)j << 49) + (j2 << 24) + 2 * j * j2 / 3 + ((j2 * j2) >> 25));
}
SU2_HD void haar_fix(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3,
                     const FixTables* __restrict__ tab, int64_t* U)
{
    const uint32_t a0 = 2u * (w0 >> 9) + 1u, a2 = 2u * (w2 >> 9) + 1u;
    const uint32_t j0 = (1u << 24) - a0, j2 = (1u << 24) - a2;
    const NegLn l0 = neg_ln(a0, tab), l2 = neg_ln(a2, tab);
    const int s = (l0.n | l2.n) == 0 ? 0 : 4;
    int64_t L0 = neg_ln_at(l0, s), L2 = neg_ln_at(l2, s);
    int sc = 61 - s, sc0 = sc, sc2 = sc;
    int64_t S = L0 + L2;
    if (j0 < 4096u || j2 < 4096u) {
        if (j0 < 4096u) L0 = small_neg_ln(j0), sc0 = 73;
        if (j2 < 4096u) L2 = small_neg_ln(j2), sc2 = 73;
        if (sc0 == sc2) S = L0 + L2, sc = 73;
    }
    const int z = clz64((uint64_t)S);
    // x = (L0 + L2) 2^c in [1/2, 1)
    const Fx y = limbs(rsqrt_fix(((uint64_t)S << z) >> 4));
    const int c = sc + z - 64;
    const Fx r0 = limbs(mulk<4>(limbs(sqrt_fix((uint64_t)L0, c - sc0)), y));
    const Fx r1 = limbs(mulk<4>(limbs(sqrt_fix((uint64_t)L2, c - sc2)), y));
    const Arc p0 = arc_at(2u * (w1 >> 9) + 1u, tab), p1 = arc_at(2u * (w3 >> 9) + 1u, tab);
    U[0] = mul64(r0, limbs(arc_cos(p0)));
    U[1] = mul64(r0, limbs(arc_sin(p0)));
    U[2] = mul64(r1, limbs(arc_cos(p1)));
    U[3] = mul64(r1, limbs(arc_sin(p1)));
}

// 1/2 Tr(U P) at 2^51, U at 2^60, P (a part of A) at 2^55
SU2_HD int64_t retr_fix(const int64_t* U, const int64_t* P)
{
    return dot4(limbs(U[0]), limbs(P[0]), limbs(-U[1]), limbs(P[1]), limbs(-U[2]), limbs(P[2]),
                limbs(-U[3]), limbs(P[3]));
}

}  // namespace su2
