// The transcendental pieces of the canonical fp32 order -- feature
// standardisation, softplus, sigmoid -- each defined as a double-precision
// value rounded to float once, evaluated here in two-float arithmetic.
//
// Why: this GPU executes a double-precision instruction for a warp in 16 SM
// cycles, with 64 cycles of latency, so softplus in double takes 2,893 cycles
// on its own and 780 cycles of an SM's throughput per warp; layer 2 of one
// pair costs 128 cycles of an SM at H = 128, its two softplus heads in double
// another 49.  A value is instead carried as the unevaluated sum of two floats
// (Dekker's and Knuth's error-free sums and products, Shewchuk's expansions),
// good to about 2^-41, and rounded to float with Ziv's test: if adding and
// subtracting a bound on its error rounds to the same float, that float is the
// rounding of the exact value, and of the double-precision evaluation too
// (whose own error is 2^-51).  Otherwise, about once in 2^15 softplus values
// (1,451 of 2^26), and for arguments outside the ranges below, the
// double-precision evaluation runs.  The result is the same float for every
// argument: the tests check softplus and sigmoid for all 2^32 of them,
// standardisation for all 2^32 under several constants and for random
// constants on a sample.
//
// Series: exp by its Taylor polynomial after a reduction by multiples of ln 2
// (held in three parts, so that the reduction is exact); log(m) =
// 2 atanh((m - 1) / (m + 1)) with m in [sqrt(1/2), sqrt(2)].  Compiled with
// --fmad=false: every fused step is written out.
#pragma once

#include <stdint.h>

namespace hwr {

struct ff {
    float h, l;   // the value h + l, |l| at most a few units in h's last place
};

__device__ __forceinline__ ff two_sum(float a, float b) {
    const float s = a + b, t = s - a;
    return ff{s, (a - (s - t)) + (b - t)};
}

// |a| >= |b|, or a = 0
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
    const float s = a + b;
    return ff{s, b - (s - a)};
}

// c + x y (cl: low part of c); |c| >= |x y|
__device__ __forceinline__ ff ff_step(float c, float cl, ff x, ff y) {
    const float p = x.h * y.h;
    float e = __fmaf_rn(x.h, y.h, -p);
    e = __fmaf_rn(x.h, y.l, e);
    e = __fmaf_rn(x.l, y.h, e);
    const ff s = fast_two_sum(c, p);
    return ff{s.h, s.l + (e + cl)};
}

// the same for a single y whose own rounding does not matter
__device__ __forceinline__ ff ff_step1(float c, float cl, ff x, float y) {
    const float p = x.h * y;
    const ff s = fast_two_sum(c, p);
    return ff{s.h, s.l + cl};
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ ff ff_div(ff n, ff d) {
    const float rc = rcp_approx(d.h), q = n.h * rc;
    const float r = __fmaf_rn(-q, d.h, n.h) + __fmaf_rn(-q, d.l, n.l);
    return ff{q, r * rc};
}

// ln 2 in three parts: 17 bits, 17 bits (products with |n| < 128 are exact)
// and the rest
constexpr float LN2_A = 0x1.62e4p-1f, LN2_B = 0x1.7f7d0p-20f, LN2_C = 0x1.cf79acp-40f;

// exp(-a), 0 <= a <= 60
__device__ __forceinline__ ff ff_exp_neg(float a) {
    const float n = rintf(a * 0x1.715476p0f);
    const float r0 = __fmaf_rn(n, LN2_A, -a);           // exact
    ff r = two_sum(r0, n * LN2_B);
    r.l = __fmaf_rn(n, LN2_C, r.l);
    // sum of r^k / k!: k = 6 .. 11 in single, the rest in two floats
    float t = 0x1.ae6456p-26f;                          // 1 / 11!
    t = __fmaf_rn(t, r.h, 0x1.27e4fcp-22f);             // 1 / 10!
    t = __fmaf_rn(t, r.h, 0x1.71de3ap-19f);             // 1 / 9!
    t = __fmaf_rn(t, r.h, 0x1.a01a02p-16f);             // 1 / 8!
    t = __fmaf_rn(t, r.h, 0x1.a01a02p-13f);             // 1 / 7!
    t = __fmaf_rn(t, r.h, 0x1.6c16c2p-10f);             // 1 / 6!
    ff q = ff_step1(0x1.111112p-7f, -0x1.dddddep-32f, r, t);     // 1 / 5!
    q = ff_step(0x1.555556p-5f, -0x1.555556p-30f, r, q);         // 1 / 4!
    q = ff_step(0x1.555556p-3f, -0x1.555556p-28f, r, q);         // 1 / 3!
    q = ff_step(0.5f, 0.f, r, q);
    q = ff_step(1.f, 0.f, r, q);
    q = ff_step(1.f, 0.f, r, q);
    const float s = __int_as_float((127 - (int)n) << 23);
    return ff{q.h * s, q.l * s};
}

// 2 atanh(n / d), |n / d| <= 0.1716
__device__ __forceinline__ ff ff_atanh2(ff n, ff d) {
    const ff t = ff_div(n, d);
    ff z;
    z.h = t.h * t.h;
    z.l = __fmaf_rn(t.h, t.h, -z.h) + 2.f * t.h * t.l;
    // sum of z^k / (2 k + 1): k = 4 .. 8 in single, the rest in two floats
    float p = 0x1.e1e1e2p-5f;                           // 1 / 17
    p = __fmaf_rn(p, z.h, 0x1.111112p-4f);              // 1 / 15
    p = __fmaf_rn(p, z.h, 0x1.3b13b2p-4f);              // 1 / 13
    p = __fmaf_rn(p, z.h, 0x1.745d18p-4f);              // 1 / 11
    p = __fmaf_rn(p, z.h, 0x1.c71c72p-4f);              // 1 / 9
    ff q = ff_step1(0x1.24924ap-3f, -0x1.b6db6ep-28f, z, p);     // 1 / 7
    q = ff_step(0x1.99999ap-3f, -0x1.99999ap-29f, z, q);         // 1 / 5
    q = ff_step(0x1.555556p-2f, -0x1.555556p-27f, z, q);         // 1 / 3
    q = ff_step(1.f, 0.f, z, q);
    const float t2 = 2.f * t.h, h = t2 * q.h;
    float l = __fmaf_rn(t2, q.h, -h);
    l = __fmaf_rn(t2, q.l, l);
    l = __fmaf_rn(2.f * t.l, q.h, l);
    return ff{h, l};
}

// log(w), 2^-64 <= w.h <= 2^64
__device__ __forceinline__ ff ff_log(ff w) {
    const int n = (__float_as_int(w.h) - 0x3f3504f3) >> 23;      // w 2^-n in [0.707, 1.414]
    const float s = __int_as_float((127 - n) << 23), fn = (float)n;
    const float m = w.h * s, ml = w.l * s;
    const float d = m + 1.f;
    const ff a = ff_atanh2(ff{m - 1.f, ml}, ff{d, (m - (d - 1.f)) + ml});
    ff c = fast_two_sum(fn * LN2_A, fn * LN2_B);
    c.l = __fmaf_rn(fn, LN2_C, c.l);
    const ff r = two_sum(c.h, a.h);
    return ff{r.h, r.l + (c.l + a.l)};
}

// Ziv's test: the rounding of h + l, if no value within err of it rounds
// differently (never for NaN).
__device__ __forceinline__ bool ff_round(ff x, float err, float *r) {
    const float up = x.h + (x.l + err), dn = x.h + (x.l - err);
    *r = up;
    return up == dn;
}

// ---- the double-precision evaluations ------------------------------------------

static __device__ __noinline__ float standardise_dp(uint8_t code, float rh, float rl, float mu,
                                                    float sd) {
    const double raw = rl == 0.f ? (double)rh : (double)rh + (double)rl;   // keeps -0
    double t = raw;
    if (code == 1) t = log1p(raw);
    else if (code == 2) t = log(raw);
    return (float)((t - (double)mu) / (double)sd);
}

static __device__ __noinline__ float softplus_dp(float z) {
    const double zd = (double)z;
    return (float)(fmax(zd, 0.0) + log1p(exp(-fabs(zd))));
}

static __device__ __noinline__ float sigmoid_dp(float s) {
    return (float)(1.0 / (1.0 + exp(-(double)s)));
}

// ---- canonical functions -------------------------------------------------------

// Relative error bounds of the two-float values.  Largest errors seen over 2^26
// arguments in [-12, 12]: exp and softplus 2^-41.1, log 2^-44.1.
constexpr float FF_ERR = 0x1p-40f, FF_LOG_ERR = 0x1p-42f;

// (t - mu) / sd as q + l, and a bound on the error of rounding q + l +- err (t is
// off by terr at most).  With u = 2^-24 and r the remainder d - q sd: q is off
// by u from its product and 2 u from the reciprocal, so |r / sd| <= 3 u |q|; l
// takes one rounding of r and of d.l + t.l each, of their sum and of the
// product, and the reciprocal's 2 u, in all at most 5 u |l| + 6 u^2 |q|; adding
// err to l rounds once more, u |l|.  6 u |l| + 6 u^2 |q| is under 2^-21 |l| +
// 2^-43 |q|.  (2^-42 |q| alone does not always bracket the value where |l| comes
// near 2^-20 |q|, which only counts past 2^24 reach.)
__device__ __forceinline__ ff ff_standard(ff t, float terr, float mu, float sd, float *err) {
    const ff d = two_sum(t.h, -mu);
    const float rc = rcp_approx(sd), q = d.h * rc;
    const ff x{q, (__fmaf_rn(-q, sd, d.h) + (d.l + t.l)) * rc};
    *err = terr * fabsf(rc) + __fmaf_rn(0x1p-21f, fabsf(x.l), 0x1p-43f * fabsf(q));
    return x;
}

// (t(raw) - mu) / sd with the slot transform t: 0 identity, 1 log1p, 2 log.
// raw = rh + rl exactly (rl is non-zero for integers past 2^24 only).
__device__ __forceinline__ float standardise(uint8_t code, ff raw, float mu, float sd) {
    ff t = raw;
    float terr = 0.f;
    bool ok = true;
    if (code) {
        ff w = raw;
        if (code == 1) {
            w = two_sum(raw.h, 1.f);
            w.l += raw.l;                    // exact: raw.l is a small integer or 0
            ok = raw.l == 0.f || w.l == raw.l;
        }
        ok = ok && w.h >= 0x1p-40f && w.h <= 0x1p40f;
        t = ff_log(w);
        terr = FF_LOG_ERR * fabsf(t.h) + 0x1p-48f;
    }
    float err;
    const ff x = ff_standard(t, terr, mu, sd, &err);
    const float q = x.h;
    ok = ok && fabsf(sd) >= 0x1p-40f && fabsf(sd) <= 0x1p40f;
    // an exact zero: the quotient is a zero of the right sign
    if (ok && t.h == mu && x.l == 0.f && terr == 0.f) return q;
    // the quotient far from the ends of the float range, its low part small
    // (it is computed in single)
    ok = ok && fabsf(q) >= 0x1p-40f && fabsf(q) <= 0x1p60f && fabsf(x.l) <= 0x1p-20f * fabsf(q);
    float r;
    if (ok && ff_round(x, err, &r)) return r;
    return standardise_dp(code, raw.h, raw.l, mu, sd);
}

__device__ __forceinline__ float standardise(uint8_t code, float raw, float mu, float sd) {
    return standardise(code, ff{raw, 0.f}, mu, sd);
}

// a count as its two parts
__device__ __forceinline__ ff ff_count(int32_t i) {
    const float h = (float)i;
    return ff{h, i <= (1 << 24) && i >= -(1 << 24) ? 0.f : (float)((long long)i - (long long)h)};
}

// max(z, 0) + log1p(exp(-|z|))
__device__ __forceinline__ float softplus_c(float z) {
    const float a = fabsf(z);
    const ff e = ff_exp_neg(fminf(a, 60.f));
    // log(1 + e) = [ln 2] + 2 atanh((e - 1) / (e + 3)) above sqrt(2), else
    // 2 atanh(e / (e + 2))
    const bool big = e.h > 0x1.a8279ap-2f;
    const float one = big ? 1.f : 0.f;
    ff n = fast_two_sum(-one, e.h);
    n.l += e.l;
    ff d = fast_two_sum(2.f + one, e.h);
    d.l += e.l;
    const ff l2 = ff_atanh2(n, d);
    ff s = fast_two_sum(big ? 0x1.62e43p-1f : 0.f, l2.h);
    s.l += l2.l + (big ? -0x1.05c61p-29f : 0.f);
    ff r = two_sum(fmaxf(z, 0.f), s.h);
    r.l += s.l;
    float out;
    if (a <= 60.f && ff_round(r, FF_ERR * r.h, &out)) return out;
    return softplus_dp(z);
}

// 1 / (1 + exp(-s))
__device__ __forceinline__ float sigmoid_c(float s) {
    const float a = fabsf(s);
    const ff e = ff_exp_neg(fminf(a, 60.f));
    ff d = fast_two_sum(1.f, e.h);
    d.l += e.l;
    const ff r = ff_div(s >= 0.f ? ff{1.f, 0.f} : e, d);
    float out;
    if (a <= 60.f && ff_round(r, FF_ERR * r.h, &out)) return out;
    return sigmoid_dp(s);
}

}  // namespace hwr
