// Errors of the fixed-point link update (csrc/su2_fixed.cuh, host build) and of
// the same update in doubles against long double, as lines of numbers read
// by test_fixed_point.py.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#define __restrict__ __restrict
#include "su2_fixed.cuh"

using namespace su2;
typedef long double LD;

static FixTables T;
static uint64_t bits(double d) { uint64_t b; memcpy(&b, &d, 8); return b; }
static double from_bits(uint64_t b) { double d; memcpy(&d, &b, 8); return d; }
static double err(LD a, LD b) { return (double)std::fabs(a - b); }

template <typename F> struct Q { F c[4]; };
template <typename F> Q<F> nd(const Q<F>& p, const Q<F>& q)
{
    const F *a = p.c, *b = q.c;
    return {{a[0] * b[0] + a[1] * b[1] + a[2] * b[2] + a[3] * b[3],
             a[1] * b[0] - a[0] * b[1] - a[3] * b[2] + a[2] * b[3],
             a[2] * b[0] - a[0] * b[2] + a[3] * b[1] - a[1] * b[3],
             a[3] * b[0] - a[0] * b[3] - a[2] * b[1] + a[1] * b[2]}};
}
template <typename F> Q<F> dag(const Q<F>& p) { return {{p.c[0], -p.c[1], -p.c[2], -p.c[3]}}; }

// one trial of one link from its 18 neighbours (x, y, z of the six terms) in F
template <typename F>
void update(const Q<double>* L, double beta, const uint32_t* w, F* lam2, bool* ok, Q<F>* U)
{
    Q<F> A = {{0, 0, 0, 0}};
    for (int i = 0; i < 6; ++i) {
        Q<F> x[3];
        for (int k = 0; k < 3; ++k)
            for (int c = 0; c < 4; ++c) x[k].c[c] = L[3 * i + k].c[c];
        const Q<F> t = i & 1 ? nd(dag(nd(x[0], dag(x[1]))), dag(x[2])) : nd(nd(x[0], x[1]), x[2]);
        for (int c = 0; c < 4; ++c) A.c[c] += t.c[c];
    }
    F k = 0;
    for (F c : A.c) k += c * c;
    k = std::sqrt(k);
    const F pi = std::acos((F)-1);
    auto u = [&](uint32_t v) { return ((F)(v >> 9) + (F)0.5) / (F)8388608; };
    const F cs = std::cos(2 * pi * u(w[1]));
    *lam2 = -(std::log(u(w[0])) + cs * cs * std::log(u(w[2]))) * ((F)(0.5 / beta) / k);
    *ok = u(w[3]) * u(w[3]) <= 1 - *lam2;
    const uint32_t k1 = ((w[0] & 511) << 9) | (w[1] & 511), k2 = ((w[2] & 511) << 9) | (w[3] & 511);
    const F cth = 2 * ((F)k1 + (F)0.5) / 262144 - 1, phi = 2 * pi * ((F)k2 + (F)0.5) / 262144;
    const F sth = std::sqrt((1 - cth) * (1 + cth)), d = 2 * *lam2, v = std::sqrt(d * (2 - d));
    *U = nd(Q<F>{{1 - d, v * sth * std::cos(phi), v * sth * std::sin(phi), v * cth}}, A);
    F n = 0;
    for (F c : U->c) n += c * c;
    for (F& c : U->c) c /= std::sqrt(n);
}

// errors of accepted new links in fixed point (f) and in doubles (d)
struct Errors {
    double mf = 0, md = 0, sf = 0, sd = 0;
    long n = 0, flips = 0, values = 0;
    void print(const char* name, double beta, double spread) const
    {
        printf("%s %g %g %ld %ld %.3e %.3e %.3e %.3e\n", name, beta, spread, n, flips, mf, md,
               std::sqrt(sf / values), std::sqrt(sd / values));
    }
};
// components c0 .. 3 of new links among random neighbours of spread `spread`
// around the identity (negative: any); in every near1-th draw (0: none) both
// logarithms are near zero
bool new_links(double beta, double spread, int iters, int near1, int c0, std::mt19937_64& g,
               std::normal_distribution<double>& N, Errors* e)
{
    for (int it = 0; it < iters; ++it) {
        Q<double> L[18];
        for (auto& q : L) {
            double s = 0;
            for (int c = 0; c < 4; ++c) {
                q.c[c] = N(g);
                if (spread >= 0) q.c[c] = c == 0 ? 1 : spread * q.c[c];
                s += q.c[c] * q.c[c];
            }
            for (double& c : q.c) c /= std::sqrt(s);
        }
        uint32_t w[4];
        for (uint32_t& x : w) x = (uint32_t)g();
        if (near1 && it % near1 == 0) {
            w[0] |= 0xFFFF0000u;
            w[2] |= 0xFFF00000u;
        }
        LD lam;
        double lamd;
        bool ok, okd;
        Q<LD> U;
        Q<double> Ud;
        update<LD>(L, beta, w, &lam, &ok, &U);
        update<double>(L, beta, w, &lamd, &okd, &Ud);
        int64_t A[4] = {0, 0, 0, 0};
        for (int i = 0; i < 6; ++i) {
            auto conv = [&](const Q<double>& q) {
                auto f = [&](int c) {
                    return fx_link((uint32_t)(bits(q.c[c]) >> 32), (uint32_t)bits(q.c[c]));
                };
                return FQuat{f(0), f(1), f(2), f(3)};
            };
            fq_staple(conv(L[3 * i]), conv(L[3 * i + 1]), conv(L[3 * i + 2]), i & 1, A);
        }
        Drawn D;
        uint64_t K;
        int sc;
        if (!unit_staple(A, half_inv_beta_fix(bits(0.5 / beta)), &D, &K, &sc)) return false;
        const Lambda l = kp_lambda(kp_sum(w[0], w[1], w[2], &T), D.inv, D.ei);
        const bool okf = kp_accept(l, w[3]);
        e->flips += okf != ok;
        if (!ok || !okf) continue;
        int64_t u[4];
        new_link_fix(l, ((w[0] & 511) << 9) | (w[1] & 511), ((w[2] & 511) << 9) | (w[3] & 511), D.V, &T, u);
        for (int c = c0; c < 4; ++c) {
            const double ef = err(from_bits(double_bits(u[c], -60)), U.c[c]);
            const double ed = err(Ud.c[c], U.c[c]);
            e->mf = std::max(e->mf, ef);
            e->md = std::max(e->md, ed);
            e->sf += ef * ef;
            e->sd += ed * ed;
            ++e->values;
        }
        ++e->n;
    }
    return true;
}

int main()
{
    fill_fix_tables(&T);
    std::mt19937_64 g(5);
    std::normal_distribution<double> N;
    double e0 = 0, e1 = 0;
    for (uint32_t k = 0; k < (1u << 23); k += (k < 4096 || k > (1u << 23) - 4096) ? 1 : 5) {
        const LD r = -std::log((LD)(2 * k + 1) / 16777216.0L);
        const NegLn l = neg_ln(2 * k + 1, &T);
        if (l.n == 0) e0 = std::max(e0, err(r, std::ldexp((LD)neg_ln_at(l, 0), -61)));
        else e1 = std::max(e1, err(r, std::ldexp((LD)neg_ln_at(l, 4), -57)));
    }
    printf("ln %.3e %.3e\n", e0, e1);
    e0 = e1 = 0;
    for (uint32_t k = 0; k < (1u << 24); k += 9) {
        const Arc a = arc_at(k, &T);
        const LD x = 2 * std::acos(-1.0L) * (LD)k / 16777216.0L;
        e0 = std::max(e0, err(std::cos(x), std::ldexp((LD)arc_cos(a), -62)));
        e1 = std::max(e1, err(std::sin(x), std::ldexp((LD)arc_sin(a), -62)));
    }
    printf("arc %.3e %.3e\n", e0, e1);
    e0 = e1 = 0;
    for (int i = 0; i < 1000000; ++i) {
        const uint64_t K = i < 8 ? (uint64_t(1) << (56 + i / 2)) + (i & 1)
                                 : (uint64_t(1) << 56) + g() % (uint64_t(15) << 56);
        e0 = std::max(e0, (double)std::fabs(std::ldexp((LD)rsqrt_fix(K), -60) *
                                            std::sqrt(std::ldexp((LD)K, -60)) - 1));
        const uint64_t v = (uint64_t(1) << 58) + g() % (uint64_t(31) << 58);
        int e = -60 - (int)(g() % 24);
        if (std::ldexp((LD)v, e) > 1) e -= 3;
        e1 = std::max(e1, err(std::sqrt(std::ldexp((LD)v, e)), std::ldexp((LD)sqrt_fix(v, e), -62)));
    }
    printf("root %.3e %.3e\n", e0, e1);
    e0 = e1 = 0;
    for (int i = 0; i < 1000000; ++i) {
        double x = (double)(int64_t)g() * 0x1p-63;
        if (i < 4) x = i == 0 ? 0.0 : (i == 1 ? 1.0 : (i == 2 ? -1.0 : -0x1p-30));
        else if (i % 3 == 0) x = std::ldexp(x, -(int)(g() % 80));
        const Fx f = fx_link((uint32_t)(bits(x) >> 32), (uint32_t)bits(x));
        const LD v = std::ldexp((LD)f.h, -29) + std::ldexp((LD)f.l, -61);
        e0 = std::max(e0, err(v, x));
        const int64_t m = (int64_t)g() >> (3 + g() % 60);
        const LD y = std::ldexp((LD)m, -60);
        const double d = from_bits(double_bits(m, -60));
        if (m) e1 = std::max(e1, (double)std::fabs((d - y) / y));
        else if (d != 0) e1 = 1;
    }
    printf("convert %.3e %.3e\n", e0, e1);
    // Haar elements: Box-Muller and normalisation in long double and in doubles
    double h0 = 0, h1 = 0, s0 = 0, s1 = 0;
    for (int i = 0; i < 400000; ++i) {
        uint32_t w[4];
        for (uint32_t& x : w) x = (uint32_t)g();
        if (i % 4 == 1) w[0] |= 0xFFFFFFFFu << (9 + g() % 20);  // u0 near 1
        if (i % 4 == 2) w[0] >>= g() % 24;                      // u0 near 0
        if (i % 8 == 3) w[0] |= 0xFFFF0000u, w[2] |= 0xFFFFF000u;
        int64_t U[4];
        haar_fix(w[0], w[1], w[2], w[3], &T, U);
        auto haar = [&](auto one) {
            using F = decltype(one);
            Q<F> q;
            F n = 0;
            for (int k = 0; k < 2; ++k) {
                const F r = std::sqrt(-2 * std::log(((F)(w[2 * k] >> 9) + (F)0.5) / 8388608));
                const F x = 2 * std::acos((F)-1) * (((F)(w[2 * k + 1] >> 9) + (F)0.5) / 8388608);
                q.c[2 * k] = r * std::cos(x);
                q.c[2 * k + 1] = r * std::sin(x);
            }
            for (F c : q.c) n += c * c;
            for (F& c : q.c) c /= std::sqrt(n);
            return q;
        };
        const Q<LD> ref = haar((LD)1);
        const Q<double> dbl = haar(1.0);
        for (int c = 0; c < 4; ++c) {
            const double f = err(from_bits(double_bits(U[c], -60)), ref.c[c]), d = err(dbl.c[c], ref.c[c]);
            h0 = std::max(h0, f);
            h1 = std::max(h1, d);
            s0 += f * f;
            s1 += d * d;
        }
    }
    printf("haar %.3e %.3e %.3e %.3e\n", h0, h1, std::sqrt(s0), std::sqrt(s1));
    const double betas[] = {0.1, 0.7, 2.3, 6.0, 50.0, 1e5};
    for (double beta : betas)
        for (double spread : {0.0, 0.3, -1.0}) {  // -1: random links
            Errors e;
            if (!new_links(beta, spread, 60000, 4, 0, g, N, &e)) return 1;
            e.print("link", beta, spread);
        }
    // the vector parts apart: their size, and with it a double's error, shrinks
    // as beta^-1/2, the fixed point's does not
    printf("limit %g\n", FIX_BETA_MAX);
    for (double beta : {2.3, FIX_BETA_MAX, 1e5})
        for (double spread : {1e-4, 0.5 / std::sqrt(beta)}) {
            Errors e;
            if (!new_links(beta, spread, 60000, 0, 1, g, N, &e)) return 1;
            e.print("vector", beta, spread);
        }
    return 0;
}
