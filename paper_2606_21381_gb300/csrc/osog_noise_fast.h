// The sensor noise draw on the FP32 pipes, with the decisions and the
// rounded result of the double-precision draw.
//
// GB300 issues FP64 at 1/64 of its FP32 rate, and the double-precision draw
// (two logarithms, a cosine, two square roots, a log-gamma) is all FP64.  Its
// results are one integer decision per comparison and one float, so each
// quantity here is computed with just enough precision to settle almost every
// decision, together with a bound on its error: float where a comparison has
// room (the squeeze and the acceptance test of the rejection, the inversion's
// cumulative sums), float-float where the value itself is needed (the normal,
// the candidate count, the quotient by the gain).  A comparison closer than its
// bound, or a quotient whose float rounding the bound leaves open, is reported
// as undecided and the caller draws that element in double precision.
//
// Header of plain float operations, so that the host can check the same code
// against double precision (built with -ffp-contract=off).
#pragma once

#include <stdint.h>

#include "osog_ff.h"

namespace osog {
namespace noise {

#if defined(__CUDA_ARCH__)
// (the plain approximations: no scaling of denormals, which do not occur here)
OSOG_HD float fast_rcp(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
OSOG_HD float fast_rsqrt(float a) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
OSOG_HD float fast_log(float a) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r * 0.693147181f;
}
OSOG_HD int count_lz(uint32_t x) { return __clz((int)x); }
#else
OSOG_HD float fast_rcp(float a) { return 1.0f / a; }
OSOG_HD float fast_rsqrt(float a) { return 1.0f / sqrtf(a); }
OSOG_HD float fast_log(float a) { return logf(a); }
OSOG_HD int count_lz(uint32_t x) { return x ? __builtin_clz(x) : 32; }
#endif

OSOG_HD ff split(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}
// Float-float product without the final renormalisation (|l| stays within a
// few ulp(h)), and c + p of a constant c at least as large as p.
OSOG_HD ff mul_lazy(ff a, ff b) {
    const float p = f_mul(a.h, b.h);
    float e = f_fma(a.h, b.h, -p);
    e = f_fma(a.h, b.l, e);
    return {p, f_fma(a.l, b.h, e)};
}
OSOG_HD ff add_small(ff c, ff p) {
    const ff s = fast_two_sum(c.h, p.h);
    return {s.h, f_add(s.l, f_add(c.l, p.l))};
}
OSOG_HD ff fast_root(ff a) {  // sqrt(a), a.h > 0, to about 2^-44
    const float r = fast_rsqrt(a.h);
    const float s = f_mul(a.h, r);
    const float e = f_add(f_fma(-s, s, a.h), a.l);
    return fast_two_sum(s, f_mul(e, f_mul(0.5f, r)));
}

// Constants as float-float, split by the compiler from double.
#define OSOG_FF_CONST(name, value)            \
    struct name {                             \
        static constexpr double v = (value);  \
        static constexpr float h = (float)v;  \
        static constexpr float l = (float)(v - (double)h); \
    }
OSOG_FF_CONST(Third, 1.0 / 3.0);
OSOG_FF_CONST(Fifth, 1.0 / 5.0);
OSOG_FF_CONST(PiScaled, 3.14159265358979323846 / 4294967296.0);  // pi 2^-32
OSOG_FF_CONST(PtrsB0, 0.931);
OSOG_FF_CONST(PtrsB1, 2.53);
OSOG_FF_CONST(PtrsA0, -0.059);
OSOG_FF_CONST(PtrsA1, 0.02483);
OSOG_FF_CONST(PtrsShift, 0.43);
#undef OSOG_FF_CONST
// ln 2 as a 16-bit head (its product with a small integer is exact) and the
// remaining float-float digits
constexpr double kLn2 = 0.693147180559945309417;
constexpr float kLn2Head = 0.693145751953125f;  // 45426 / 65536
constexpr float kLn2Tail = (float)(kLn2 - (double)kLn2Head);
constexpr float kLn2Rest = (float)(kLn2 - (double)kLn2Head - (double)kLn2Tail);

// sqrt(-2 ln u0) cos(2 pi u1) of u = (x + 1/2) 2^-32, relative error below
// kNormalErr; x0 = 0 (m = 1/2 below) is outside the series' range and left to
// the caller.
constexpr float kNormalErr = 7.3e-12f;  // 2^-37
OSOG_HD ff normal_ff(uint32_t x0, uint32_t x1) {
    // N = 2 x0 + 1 = m 2^e, m in [1, 2) from its top 24 bits and the rest
    int lz = count_lz(x0);
    lz = lz > 31 ? 31 : lz;
    const uint32_t X = x0 << lz;
    const float hi = (float)(X & 0xFFFFFF00u);                 // exact: 24 bits
    const float lo = (float)(2u * (X & 0xFFu) + (1u << lz));   // exact
    ff m = fast_two_sum(f_mul(hi, 4.656612873077393e-10f), f_mul(lo, 2.3283064365386963e-10f));
    float n = (float)(lz + 1);  // 33 - e
    if (m.h > 1.41421354f) {
        m.h = f_mul(m.h, 0.5f);
        m.l = f_mul(m.l, 0.5f);
        n = f_sub(n, 1.0f);
    }
    // ln m = 2 s (1 + t/3 + t^2/5 + ...), s = (m - 1) / (m + 1), t = s^2
    const ff f = two_sum(f_sub(m.h, 1.0f), m.l);
    ff d = fast_two_sum(m.h > 1.0f ? m.h : 1.0f, m.h > 1.0f ? 1.0f : m.h);
    d.l = f_add(d.l, m.l);
    const float r = fast_rcp(d.h);
    const float q = f_mul(f.h, r);
    const float rem = f_add(f_fma(-q, d.h, f.h), f_fma(-q, d.l, f.l));
    const ff s = fast_two_sum(q, f_mul(rem, r));
    const ff t = mul_lazy(s, s);
    float g = f_fma(t.h, 1.0f / 15.0f, 1.0f / 13.0f);
    g = f_fma(t.h, g, 1.0f / 11.0f);
    g = f_fma(t.h, g, 1.0f / 9.0f);
    g = f_fma(t.h, g, 1.0f / 7.0f);
    ff y = add_small(ff{Fifth::h, Fifth::l}, ff{f_mul(t.h, g), 0.0f});
    y = add_small(ff{Third::h, Third::l}, mul_lazy(t, y));
    y = add_small(ff{1.0f, 0.0f}, mul_lazy(t, y));
    const ff lm = mul_lazy(s, y);  // ln(m) / 2
    // -2 ln u0 = 2 n ln 2 - 2 ln m
    const float two_n = f_add(n, n);
    const ff w = two_sum(f_mul(two_n, kLn2Head), f_mul(-4.0f, lm.h));
    float wl = f_fma(-4.0f, lm.l, w.l);
    wl = f_fma(two_n, kLn2Rest, wl);
    const ff tail = two_prod(two_n, kLn2Tail);
    ff R = two_sum(w.h, tail.h);
    R = fast_two_sum(R.h, f_add(R.l, f_add(wl, tail.l)));
    const ff root = fast_root(R);
    // 2 pi u1 = quarter pi/2 + th, |th| <= pi/4
    const uint32_t quarter = ((x1 + 0x20000000u) >> 30) & 3u;
    const int32_t left = (int32_t)(2u * x1 + 1u - (quarter << 31));
    const int32_t head = left & ~0x7F;
    const ff th = mul_lazy(fast_two_sum((float)head, (float)(left - head)),
                           ff{PiScaled::h, PiScaled::l});
    const ff u = mul_lazy(th, th);
    const bool odd = quarter & 1u;  // -+ sin th, else +- cos th
    float c = odd ? (float)InvFact<13, 1>::v : (float)InvFact<12, 1>::v;
    c = f_fma(u.h, c, odd ? (float)InvFact<11, -1>::v : (float)InvFact<10, -1>::v);
    c = f_fma(u.h, c, odd ? (float)InvFact<9, 1>::v : (float)InvFact<8, 1>::v);
    ff p = add_small(odd ? ff{InvFact<7, -1>::h, InvFact<7, -1>::l}
                         : ff{InvFact<6, -1>::h, InvFact<6, -1>::l}, ff{f_mul(u.h, c), 0.0f});
    p = add_small(odd ? ff{InvFact<5, 1>::h, InvFact<5, 1>::l}
                      : ff{InvFact<4, 1>::h, InvFact<4, 1>::l}, mul_lazy(u, p));
    p = add_small(odd ? ff{InvFact<3, -1>::h, InvFact<3, -1>::l}
                      : ff{InvFact<2, -1>::h, InvFact<2, -1>::l}, mul_lazy(u, p));
    p = add_small(ff{1.0f, 0.0f}, mul_lazy(u, p));
    if (odd) p = mul_lazy(p, th);
    p = mul_lazy(p, root);
    const float sign = quarter == 1u || quarter == 2u ? -1.0f : 1.0f;
    return fast_two_sum(f_mul(sign, p.h), f_mul(sign, p.l));
}

// Outcome of a decision.
enum { kNo = 0, kYes = 1, kUndecided = 2 };

// Inversion by sequential search for a rate 0 <= lam < 10 and u2 = (x +
// 1/2) 2^-32: the smallest k with u <= F(k), sums in float.  A rounding error
// of about 2^-23 per step stays below lam 2^-22 < 3e-6 in F.
OSOG_HD int poisson_small(float lam, uint32_t x, float *k_out) {
    const float u = f_mul((float)(x >> 8) + (float)(x & 0xFFu) * 0.00390625f + 0.001953125f,
                          5.9604644775390625e-08f);
    float p = expf(-lam), F = p, k = 0.0f;
    for (int it = 0; it < 200; ++it) {
        const float d = f_sub(u, F);
        if (fabsf(d) < 6e-6f) return kUndecided;
        if (d < 0.0f) {
            *k_out = k;
            return kYes;
        }
        k = f_add(k, 1.0f);
        p = f_mul(p, f_mul(lam, fast_rcp(k)));
        F = f_add(F, p);
    }
    return kUndecided;
}

// Constants of the transformed rejection (PTRS, Hormann 1993) for one rate.
struct Ptrs {
    ff lam, a2, b;          // the rate, 2 a, b
    float inv_alpha, vr;    // squeeze and acceptance constants
};
OSOG_HD Ptrs ptrs_of(ff lam) {
    Ptrs c;
    c.lam = lam;
    const ff s = fast_root(lam);
    ff b = mul_lazy(s, ff{PtrsB1::h, PtrsB1::l});
    c.b = add_small(b, ff{PtrsB0::h, PtrsB0::l});  // 2.53 s >= 8
    const ff a = add_small(mul_lazy(c.b, ff{PtrsA1::h, PtrsA1::l}), ff{PtrsA0::h, PtrsA0::l});
    c.a2 = ff{f_add(a.h, a.h), f_add(a.l, a.l)};
    c.inv_alpha = f_fma(1.1328f, fast_rcp(f_sub(c.b.h, 3.4f)), 1.1239f);
    c.vr = f_fma(-3.6224f, fast_rcp(f_sub(c.b.h, 2.0f)), 0.9277f);
    return c;
}

// log of the ratio of the Poisson density at k to lam^lam-free form:
// -lam + k ln lam - ln k!, without the cancellation of its large terms:
// -(k ln(k / lam) - k + lam) - ln(2 pi k) / 2 - (Stirling's correction), the
// first bracket by Loader's deviance series in v = (k - lam) / (k + lam) (C.
// Loader, "Fast and accurate computation of binomial probabilities", 2000).
OSOG_HD float log_density(ff lam, float k) {
    if (k < 2.5f) {  // k! = 1, 1, 2
        const float ll = fast_log(lam.h);
        return f_sub(f_mul(k, ll), lam.h) - (k > 1.5f ? 0.693147181f : 0.0f);
    }
    const float diff = f_sub(f_sub(k, lam.h), lam.l);
    const float v = f_mul(diff, fast_rcp(f_add(k, lam.h)));
    float dev;
    if (fabsf(v) < 0.3f) {
        const float v2 = f_mul(v, v);
        float s = f_fma(v2, 1.0f / 17.0f, 1.0f / 15.0f);
        s = f_fma(v2, s, 1.0f / 13.0f);
        s = f_fma(v2, s, 1.0f / 11.0f);
        s = f_fma(v2, s, 1.0f / 9.0f);
        s = f_fma(v2, s, 1.0f / 7.0f);
        s = f_fma(v2, s, 1.0f / 5.0f);
        s = f_fma(v2, s, 1.0f / 3.0f);
        dev = f_fma(diff, v, f_mul(f_mul(2.0f * k, v), f_mul(v2, s)));
    } else {
        dev = f_fma(k, fast_log(f_mul(k, fast_rcp(lam.h))), -diff);
    }
    const float ik = fast_rcp(k), ik2 = f_mul(ik, ik);
    const float corr = f_mul(ik, f_fma(ik2, f_fma(ik2, 1.0f / 1260.0f, -1.0f / 360.0f),
                                       1.0f / 12.0f));
    return -dev - f_mul(0.5f, fast_log(f_mul(6.28318531f, k))) - corr;
}

// us >= 0.07 and us < 0.013 as integers: us = n 2^-33, n odd.
constexpr uint32_t kUs007 = 601295422u;   // smallest n with n 2^-33 >= 0.07
constexpr uint32_t kUs0013 = 111669150u;  // smallest n with n 2^-33 >= 0.013

// The candidate of one attempt of PTRS from the word of U (xv, the word of V,
// settles the rejection of slim tails): kYes with k = floor((2 a / us + b) U +
// lam + 0.43) and us = n 2^-33, kNo (rejected whatever k is) or kUndecided.
OSOG_HD int ptrs_candidate(const Ptrs &c, uint32_t xu, uint32_t xv, float *k_out, uint32_t *n_out) {
    // U = -+ m 2^-33, us = 1/2 - |U| = n 2^-33, m = 2^32 - n
    const bool neg = xu < 0x80000000u;
    const uint32_t n = neg ? 2u * xu + 1u : 0u - (2u * xu + 1u);
    const uint32_t m = 0u - n;
    // us < 0.013 and V > us: rejected (the quick acceptance needs us >= 0.07;
    // k < 0 is rejected too, so k is not needed)
    if (n < kUs0013 && xv > (n >> 1)) return kNo;
    const ff nf = {(float)(n & 0xFFFFFF00u), (float)(n & 0xFFu)};
    const ff mf = {(float)(m & 0xFFFFFF00u), (float)(m & 0xFFu)};
    // X = -+ (2 a m / n + b m 2^-33) + lam + 0.43
    const float r = fast_rcp(f_add(nf.h, nf.l));
    const float q0 = f_mul(f_add(mf.h, mf.l), r);
    float rem = f_fma(-q0, nf.h, mf.h);
    rem = f_add(rem, f_fma(-q0, nf.l, mf.l));
    const ff quot = fast_two_sum(q0, f_mul(rem, r));  // m / n
    const ff t1 = mul_lazy(c.a2, quot);
    const ff mu = fast_two_sum(f_mul(mf.h, 1.1641532182693481e-10f),
                               f_mul(mf.l, 1.1641532182693481e-10f));
    const ff t2 = mul_lazy(c.b, mu);
    const float sg = neg ? -1.0f : 1.0f;
    ff t = two_sum(t1.h, t2.h);
    t.l = f_add(t.l, f_add(t1.l, t2.l));
    const ff base = add_small(c.lam, ff{PtrsShift::h, PtrsShift::l});
    ff X = two_sum(f_mul(sg, t.h), base.h);
    X.l = f_add(X.l, f_fma(sg, t.l, base.l));  // |X.l| stays within a few ulps
    // 2^-39 of the largest term bounds the error of X
    const float err = f_mul(f_add(f_add(t.h, c.lam.h), 1.0f), 1.8189894035458565e-12f);
    if (X.h < -1.0f) return kNo;      // k < 0 (us is below 0.07 then)
    if (!(X.h < 4194304.0f)) return kUndecided;
    float k = floorf(X.h);
    float fr = f_add(f_sub(X.h, k), X.l);
    const float carry = fr < 0.0f ? -1.0f : fr >= 1.0f ? 1.0f : 0.0f;
    k = f_add(k, carry);
    fr = f_sub(fr, carry);
    if (fr < err || fr > f_sub(1.0f, err) - 1.2e-7f) return kUndecided;
    *k_out = k;
    *n_out = n;
    return kYes;
}

OSOG_HD float ptrs_v(uint32_t xv) {  // V = (xv + 1/2) 2^-32
    return f_mul((float)(xv >> 8) + (float)(xv & 0xFFu) * 0.00390625f + 0.001953125f,
                 5.9604644775390625e-08f);
}

// The quick acceptance of a candidate: kYes, kUndecided, or kNo: not accepted by
// it (ptrs_accept decides).
OSOG_HD int ptrs_quick(const Ptrs &c, uint32_t n, uint32_t xv) {
    const float dv = f_sub(c.vr, ptrs_v(xv));
    if (n < kUs007 || dv < -2e-6f) return kNo;
    return dv < 2e-6f ? kUndecided : kYes;
}

// The acceptance test of a candidate k that the quick one left: b and a2 of the
// rate in float are enough.
OSOG_HD int ptrs_accept(ff lam, float b, float a2, float inv_alpha, float k, uint32_t n, uint32_t xv) {
    if (k < 0.0f) return kNo;
    const float us = f_mul((float)n, 1.1641532182693481e-10f);
    const float lhs = fast_log(f_mul(f_mul(ptrs_v(xv), inv_alpha),
                                     fast_rcp(f_fma(f_mul(0.5f, a2), fast_rcp(f_mul(us, us)), b))));
    const float rhs = log_density(lam, k);
    const float gap = f_sub(rhs, lhs);
    const float tol = f_fma(fabsf(rhs), 1e-5f, 4e-5f);
    if (!(fabsf(gap) >= tol)) return kUndecided;
    return gap > 0.0f ? kYes : kNo;
}

// ptrs_accept with the constants of the rate taken in float (b to a few 1e-7
// relative, well inside its tolerance).
OSOG_HD int ptrs_accept_float(ff lam, float k, uint32_t n, uint32_t xv) {
    const float b = f_fma(2.53f, f_mul(lam.h, fast_rsqrt(lam.h)), 0.931f);
    const float a2 = 2.0f * f_fma(0.02483f, b, -0.059f);
    return ptrs_accept(lam, b, a2, f_fma(1.1328f, fast_rcp(f_sub(b, 3.4f)), 1.1239f), k, n, xv);
}

// One attempt of PTRS from the words of U and V: kYes with *k_out, kNo
// (rejected) or kUndecided.
OSOG_HD int ptrs_attempt(const Ptrs &c, uint32_t xu, uint32_t xv, float *k_out) {
    uint32_t n;
    float k;
    int s = ptrs_candidate(c, xu, xv, &k, &n);
    if (s != kYes) return s;
    *k_out = k;
    s = ptrs_quick(c, n, xv);
    return s != kNo ? s : ptrs_accept(c.lam, c.b.h, c.a2.h, c.inv_alpha, k, n, xv);
}

// (k + sigma z) / g rounded to float: true with *out when the error bounds of
// the parts decide the rounding.  sz = sigma z and inv_g = 1 / g as float-float.
OSOG_HD bool noisy_value(float k, ff sz, ff inv_g, float *out) {
    ff T = two_sum(k, sz.h);
    T = fast_two_sum(T.h, f_add(T.l, sz.l));
    const ff y = ff_mul(T, inv_g);
    const float e = f_mul(inv_g.h, f_fma(fabsf(sz.h), kNormalErr,
                                         f_mul(fabsf(T.h), 2.8421709430404007e-14f)));  // 2^-45
    *out = y.h;
    return f_add(y.h, f_add(y.l, e)) == y.h && f_add(y.h, f_sub(y.l, e)) == y.h;
}

}  // namespace noise
}  // namespace osog
