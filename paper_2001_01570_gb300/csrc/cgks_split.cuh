// cgks_split.cuh -- unevaluated sums of two FP32 numbers (x = h + l, about 47
// bits) for the parts of the reconstruction that are small corrections of FP64
// values, and the nonlinear part of the normal reconstruction written in them.
//
// Why: on GB300 a warp's FP64 instruction holds its sub-core's FP64 unit for 68
// cycles whatever the number of active lanes or independent chains (measured, 1
// to 8 chains, 8 to 32 lanes), while an FP32 instruction takes 1.1 to 1.5; the
// record kernel had the FP64 unit 99.6 % busy with about 320 instructions per
// (face row, variable), 240 of them in the WENO-Z pair.  A pair product takes 4
// FP32 instructions and a pair sum 8 to 11.
//
// Why no precision is lost: the values themselves stay FP64.  What is carried in
// pairs is a correction made of third differences (and the weights), and
// split_ok lets a face row take this path only where the third differences are
// below 2^-7 of the variable's scale, so the pairs' rounding (about 2^-48 of the
// correction) stays at or below the last bit of the FP64 value the correction is
// added to (tests/test_split_host.py: against 113-bit arithmetic the values' largest
// and rms errors are those of the FP64 formulas or smaller).  Everywhere else -- at shocks and on under-resolved data -- the FP64
// formulas of cgks_device.cuh run.  The choice depends on the row's own data
// alone, so every arrangement of the work gives the same bits.
//
// The operations are explicitly rounded (no contraction); the header compiles
// for the host too.
#pragma once
#include <stdint.h>
#ifndef __CUDACC__
#include <math.h>
#include <string.h>
#endif

namespace cgks {

#ifdef __CUDACC__
#define CGKS_SPLIT_FN __device__ __forceinline__
CGKS_SPLIT_FN float f_add(float a, float b) { return __fadd_rn(a, b); }
CGKS_SPLIT_FN float f_sub(float a, float b) { return __fsub_rn(a, b); }
CGKS_SPLIT_FN float f_mul(float a, float b) { return __fmul_rn(a, b); }
CGKS_SPLIT_FN float f_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
CGKS_SPLIT_FN float f_rcp(float a) { float y; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a)); return y; }
CGKS_SPLIT_FN float f_rsqrt(float a) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a)); return y; }
CGKS_SPLIT_FN float f_bits(uint32_t b) { return __uint_as_float(b); }
CGKS_SPLIT_FN uint32_t f_word(float a) { return __float_as_uint(a); }
CGKS_SPLIT_FN float f_int(int i) { return __int2float_rn(i); }
CGKS_SPLIT_FN int d_hi(double x) { return __double2hiint(x); }
CGKS_SPLIT_FN int d_lo(double x) { return __double2loint(x); }
CGKS_SPLIT_FN double d_make(int hi, int lo) { return __hiloint2double(hi, lo); }
CGKS_SPLIT_FN int i_max(int a, int b) { return max(a, b); }
CGKS_SPLIT_FN int i_min(int a, int b) { return min(a, b); }
#else
#define CGKS_SPLIT_FN inline
inline float f_add(float a, float b) { return a + b; }
inline float f_sub(float a, float b) { return a - b; }
inline float f_mul(float a, float b) { return a * b; }
inline float f_fma(float a, float b, float c) { return ::fmaf(a, b, c); }
inline float f_rcp(float a) { return 1.0f / a; }
inline float f_rsqrt(float a) { return 1.0f / ::sqrtf(a); }
inline float f_bits(uint32_t b) { float a; memcpy(&a, &b, 4); return a; }
inline uint32_t f_word(float a) { uint32_t b; memcpy(&b, &a, 4); return b; }
inline float f_int(int i) { return (float)i; }
#define CGKS_HOST_DOUBLE decltype(0.0)
inline int64_t d_word(CGKS_HOST_DOUBLE x) { int64_t b; memcpy(&b, &x, 8); return b; }
inline int d_hi(CGKS_HOST_DOUBLE x) { return (int)(d_word(x) >> 32); }
inline int d_lo(CGKS_HOST_DOUBLE x) { return (int)(uint32_t)d_word(x); }
inline CGKS_HOST_DOUBLE d_make(int hi, int lo)
{
    const int64_t b = ((int64_t)hi << 32) | (uint32_t)lo;
    CGKS_HOST_DOUBLE x;
    memcpy(&x, &b, 8);
    return x;
}
inline int i_max(int a, int b) { return a > b ? a : b; }
inline int i_min(int a, int b) { return a < b ? a : b; }
#endif

struct ff { float h, l; };

// The exponent field and the leading mantissa bits of |x|, from its high word, as a float's:
// the float's bits shifted right by 3.  A float below 2^-126 for |x| below that; infinity's bits from
// 2^128 on (NaN included).
CGKS_SPLIT_FN uint32_t f_upper(uint32_t hi)
{
#ifdef __CUDACC__
    return (uint32_t)__viaddmin_s32_relu((int)(hi & 0x7fffffffu), -(896 << 20), 0x0ff00000);
#else
    return (uint32_t)i_max(i_min((int)(hi & 0x7fffffffu) - (896 << 20), 0x0ff00000), 0);
#endif
}

// the pair nearest below |x| in its leading 24 bits, the remaining 29 bits rounded
// to 24; integer operations, since a conversion instruction occupies the FP64
// unit like an addition.  For |x| in [2^-74, 2^128) the pair has 47 bits; below 2^-74 it
// has the leading 24 alone (error below 2^-97) and below 2^-126 next to nothing.  ff_from is for
// numbers that a bound on the FP64 values keeps below 2^128 (from there on its exponent wraps
// around); with ff_from_any, h is infinite or NaN from 2^128 on and for infinity and NaN.  (One
// instruction more at every conversion of the flux kernel: 512^2, stage 1 907 us, so 902.)
CGKS_SPLIT_FN ff ff_of(uint32_t hi, uint32_t lo, uint32_t t)
{
    const uint32_t sgn = hi & 0x80000000u;
#ifdef __CUDACC__
    const uint32_t hb = __funnelshift_l(lo, t, 3);
#else
    const uint32_t hb = (t << 3) | (lo >> 29);
#endif
    const uint32_t sc = (uint32_t)i_max((int)(hb & 0x7f800000u) - (52 << 23), 0);
    ff r;
    r.h = f_bits(hb | sgn);
    r.l = f_mul(f_int((int)(lo & 0x1fffffffu)), f_bits(sc | sgn));
    return r;
}
CGKS_SPLIT_FN ff ff_from(double x)
{
    const uint32_t hi = (uint32_t)d_hi(x);
    return ff_of(hi, (uint32_t)d_lo(x), (uint32_t)i_max((int)(hi & 0x7fffffffu) - (896 << 20), 0));
}
CGKS_SPLIT_FN ff ff_from_any(double x)
{
    const uint32_t hi = (uint32_t)d_hi(x);
    return ff_of(hi, (uint32_t)d_lo(x), f_upper(hi));
}

// the leading 21 bits of x as a float (truncated; something below 2^-126 for |x| below that, infinite from
// 2^128 on and for NaN)
CGKS_SPLIT_FN float f_lead(double x)
{
    const uint32_t hi = (uint32_t)d_hi(x);
    return f_bits((hi & 0x80000000u) | (f_upper(hi) << 3));
}

// a finite float as a double (zero and denormals give zero; infinity and NaN give 2^128 and more,
// which no bound on a correction admits), integer operations
CGKS_SPLIT_FN double d_from(float a)
{
    const uint32_t b = f_word(a), m = b & 0x7fffffffu;
    const uint32_t hi = m < 0x00800000u ? 0u : (b & 0x80000000u) | ((m >> 3) + (896u << 20));
    return d_make((int)hi, m < 0x00800000u ? 0 : (int)(b << 29));
}

// a pair in the 64 bits of a double
CGKS_SPLIT_FN double ff_pack(ff a) { return d_make((int)f_word(a.h), (int)f_word(a.l)); }
CGKS_SPLIT_FN ff ff_unpack(double x) { return ff{f_bits((uint32_t)d_hi(x)), f_bits((uint32_t)d_lo(x))}; }

CGKS_SPLIT_FN ff ff_neg(ff a) { return ff{-a.h, -a.l}; }
// renormalise (|h| >= |l|)
CGKS_SPLIT_FN ff ff_norm(float h, float l)
{
    const float s = f_add(h, l);
    return ff{s, f_sub(l, f_sub(s, h))};
}
// a + b without renormalisation: for addends of one sign, and where a result's rounding need
// only be small beside its addends (after a cancellation l may be as large as h, and the
// products below leave out l times l)
CGKS_SPLIT_FN ff ff_addp(ff a, ff b)
{
    const float s = f_add(a.h, b.h), t = f_sub(s, a.h);
    const float e = f_add(f_sub(a.h, f_sub(s, t)), f_sub(b.h, t));
    return ff{s, f_add(e, f_add(a.l, b.l))};
}
CGKS_SPLIT_FN ff ff_add(ff a, ff b)
{
    const ff s = ff_addp(a, b);
    return ff_norm(s.h, s.l);
}
CGKS_SPLIT_FN ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }
CGKS_SPLIT_FN ff ff_mul(ff a, ff b)
{
    const float p = f_mul(a.h, b.h);
    return ff{p, f_fma(a.l, b.h, f_fma(a.h, b.l, f_fma(a.h, b.h, -p)))};
}
CGKS_SPLIT_FN ff ff_sqr(ff a)
{
    const float p = f_mul(a.h, a.h);
    return ff{p, f_fma(f_add(a.h, a.h), a.l, f_fma(a.h, a.h, -p))};
}
// times a float constant; times a power of two (exact)
CGKS_SPLIT_FN ff ff_mulf(float c, ff a)
{
    const float p = f_mul(c, a.h);
    return ff{p, f_fma(c, a.l, f_fma(c, a.h, -p))};
}
CGKS_SPLIT_FN ff ff_scale(float c, ff a) { return ff{f_mul(c, a.h), f_mul(c, a.l)}; }
// 1 / a (a.h normal, |a.l| a few last places of a.h): the hardware approximation and one correction
CGKS_SPLIT_FN ff ff_rcp(ff a)
{
    const float y = f_rcp(a.h);
    const float t = f_fma(-a.l, y, f_fma(-a.h, y, 1.0f));
    return ff{y, f_mul(y, f_fma(t, t, t))};
}
// a pair constant from its FP64 value
#define CGKS_FF(c) (ff{(float)(c), (float)((c) - (decltype(0.0))(float)(c))})

// ------------------------------------------------------------------------
// The nonlinear normal reconstruction of Sec. 3.3 in differences of the stencil
// data.  With d1 = b-a, d2 = c-b, d3 = d-c (values) and A..D the h * slopes:
//   s3 = d2-d1, s4 = d3-d2                                  second differences
//   t = s3 - 2(d1-A), u = s4 - 2(D-d3), w = s4-s3,
//   p = B - (d1+d2)/2, q = C - (d2+d3)/2                    third differences
// each sub-stencil polynomial q_k of the paper has at x_{i+1/2}
//   value - (b+c)/2 + s3/6:  k=0: -t/3;  1, 3: 0;  2: -w/6 - u/8;  4: -w/6;
//                            5: t/20 + 7p/10;  6: -w/6 + u/20 - 7q/10
//   h slope - d2:            k=0: -t;  1, 3, 4: 0;  2: u/8;  5: t/4 + 3p/2;  6: 3q/2 - u/4
// and its smoothness indicator is a sum of squares (Legendre form of the
// derivatives over the cell: mean slope L, second derivative M, c3, c4)
//   beta = L^2 + 13/12 M^2 + 781/20 c3^2 + (1421461/2275) c4^2
//   k=0: L = G - t/2,       M = s3 - t
//   k=1 (cubic of Sec. 3.3): L = G - t/4,  M = s3,  c3 = t/4
//   k=2: L = H - u/2,       M = s4 + 3u/2,  c3 = -u/4
//   k=3: L = G, M = s3;     k=4: L = H, M = s4       (G = d2 - s3/2, H = d2 - s4/2)
//   k=5: L = G + p,         c3 = -p, c4 = -(t/4 + p),    M = s3 + 3t/4 + 3p + (63/65) c4
//   k=6: L = H + u/2 - 4q,  c3 = u - 5q, c4 = q - u/4,   M = s4 - 9u/4 + 15q + (63/65) c4
// The squares have no cancellation, which the expanded quadratic forms in the
// products of first differences do (coefficients up to 1.6e3 times a beta).
// The right-biased side is the same with the mirrored data: s3 <-> s4, t <-> u,
// w -> -w, p -> -q, q -> -p, d2 -> -d2.
struct DiffData { ff d2, s3, s4, w, t, u, p, q; };

// (value - ((b+c)/2 - s3/6), h slope - d2) of the left-biased side.  ORDER selects
// the linear weights (times 98 or 70: integers).
template <int ORDER>
CGKS_SPLIT_FN void weno_side_split(const DiffData& x, ff eps, ff& dval, ff& dslope)
{
    const ff G = ff_sub(x.d2, ff_scale(0.5f, x.s3)), H = ff_sub(x.d2, ff_scale(0.5f, x.s4));
    const ff c1312 = CGKS_FF(13.0 / 12.0), c3k = CGKS_FF(781.0 / 320.0);
    // eps + 13/12 M^2 of the quadratics, shared
    const ff k3 = ff_addp(ff_mul(c1312, ff_sqr(x.s3)), eps), k4 = ff_addp(ff_mul(c1312, ff_sqr(x.s4)), eps);
    const ff e3 = ff_addp(ff_sqr(G), k3), e4 = ff_addp(ff_sqr(H), k4);
    const ff t4 = ff_scale(0.25f, x.t), u4 = ff_scale(0.25f, x.u);
    const ff e1 = ff_addp(ff_addp(ff_sqr(ff_sub(G, t4)), k3), ff_mul(c3k, ff_sqr(x.t)));
    const ff e0 = ff_addp(ff_addp(ff_sqr(ff_sub(G, ff_scale(0.5f, x.t))), ff_mul(c1312, ff_sqr(ff_sub(x.s3, x.t)))), eps);
    const ff e2 = ff_addp(ff_addp(ff_sqr(ff_sub(H, ff_scale(0.5f, x.u))),
                                  ff_mul(c1312, ff_sqr(ff_add(x.s4, ff_mulf(1.5f, x.u))))),
                          ff_addp(ff_mul(c3k, ff_sqr(x.u)), eps));
    const ff c4c = CGKS_FF(1421461.0 / 2275.0), c3c = CGKS_FF(781.0 / 20.0), kap = CGKS_FF(63.0 / 65.0);
    ff e5, e6;
    {
        const ff c4 = ff_add(t4, x.p);      // -c4
        const ff M = ff_add(x.s3, ff_sub(ff_mulf(3.0f, c4), ff_mul(kap, c4)));   // 3t/4 + 3p = 3 (t/4 + p)
        e5 = ff_addp(ff_addp(ff_sqr(ff_add(G, x.p)), ff_mul(c1312, ff_sqr(M))),
                     ff_addp(ff_addp(ff_mul(c3c, ff_sqr(x.p)), ff_mul(c4c, ff_sqr(c4))), eps));
    }
    {
        const ff c4 = ff_sub(x.q, u4), c3 = ff_sub(x.u, ff_mulf(5.0f, x.q));
        // 15 q - 9u/4 = 15 c4 + 3u/2
        const ff M = ff_add(ff_add(x.s4, ff_mulf(1.5f, x.u)), ff_add(ff_mulf(15.0f, c4), ff_mul(kap, c4)));
        const ff L = ff_add(ff_sub(H, ff_scale(0.5f, x.u)), ff_scale(-4.0f, c4));   // H + u/2 - 4q = H - u/2 - 4 c4
        e6 = ff_addp(ff_addp(ff_sqr(L), ff_mul(c1312, ff_sqr(M))),
                     ff_addp(ff_addp(ff_mul(c3c, ff_sqr(c3)), ff_mul(c4c, ff_sqr(c4))), eps));
    }
    // Z_ref = |3 (e0 - e4) + (e4 - e3)| (the epsilons cancel)
    ff Z = ff_add(ff_mulf(3.0f, ff_sub(e0, e4)), ff_sub(e4, e3));
    if (Z.h < 0.0f) Z = ff_neg(Z);
    // alpha_k = d_k (1 + Z / e_k)
    auto alpha = [&](float d, ff e) {
        const ff z = ff_mul(Z, ff_rcp(e));
        return ff_mulf(d, ff_addp(ff{1.0f, 0.0f}, z));
    };
    const ff a0 = alpha(3.0f, e0), a2 = alpha(8.0f, e2), a4 = alpha(7.0f, e4);
    const ff a13 = ff_addp(alpha(5.0f, e1), alpha(7.0f, e3));
    const ff a5 = alpha(ORDER == 6 ? 20.0f : 34.0f, e5), a6 = alpha(ORDER == 6 ? 20.0f : 34.0f, e6);
    const ff right = ff_addp(ff_addp(a2, a4), a6);
    const ff sum = ff_addp(ff_addp(ff_addp(a0, a13), a5), right);
    const ff inv = ff_rcp(sum);
    const ff c13 = CGKS_FF(1.0 / 3.0), c16 = CGKS_FF(1.0 / 6.0), c07 = CGKS_FF(0.7), c05 = CGKS_FF(0.05);
    const ff y5 = ff_add(ff_mul(c05, x.t), ff_mul(c07, x.p)), y6 = ff_sub(ff_mul(c05, x.u), ff_mul(c07, x.q));
    ff nv = ff_add(ff_mul(a5, y5), ff_mul(a6, y6));
    nv = ff_sub(nv, ff_mul(a0, ff_mul(c13, x.t)));
    nv = ff_sub(nv, ff_mul(a2, ff_scale(0.125f, x.u)));
    nv = ff_sub(nv, ff_mul(right, ff_mul(c16, x.w)));
    const ff g5 = ff_add(t4, ff_mulf(1.5f, x.p)), g6 = ff_sub(ff_mulf(1.5f, x.q), u4);
    ff ns = ff_add(ff_mul(a5, g5), ff_mul(a6, g6));
    ns = ff_sub(ns, ff_mul(a0, x.t));
    ns = ff_add(ns, ff_mul(a2, ff_scale(0.125f, x.u)));
    dval = ff_mul(nv, inv);
    dslope = ff_mul(ns, inv);
}

// Whether the pair arithmetic carries a row's nonlinear part: the third
// differences' magnitudes (and s3's) against the variable's scale, compared as
// the high words of FP64 numbers (for finite non-negative values their order is
// the values'; NaN and infinity compare above everything).  scale_hi: high word
// of the variable's scale; the ranges 2^-30..2^25 of the scale and of eps keep every
// FP32 intermediate normal where it counts.
constexpr int kHiOne = 1023 << 20;   // high word of 1.0; one binary order is 1 << 20
CGKS_SPLIT_FN int hi_abs(double x) { return d_hi(x) & 0x7fffffff; }
CGKS_SPLIT_FN bool split_scale_ok(int scale_hi, double eps)
{
    return scale_hi >= kHiOne - (30 << 20) && scale_hi < kHiOne + (25 << 20) && d_hi(eps) >= kHiOne - (30 << 20) &&
           d_hi(eps) < kHiOne + (25 << 20);
}
CGKS_SPLIT_FN bool split_ok(int scale_hi, double eps, double w, double t, double u, double p, double q, double s3)
{
    const int m3 = i_max(i_max(i_max(hi_abs(w), hi_abs(t)), hi_abs(u)), i_max(hi_abs(p), hi_abs(q)));
    return split_scale_ok(scale_hi, eps) && m3 < scale_hi - (7 << 20) && hi_abs(s3) < scale_hi;
}

// ------------------------------------------------------------------------
// The values and derivatives along a face (cgks_segment.cuh) as corrections; taken where the
// first and third differences (the slope's correction) are below these powers of two of
// the scale.
constexpr int kTangFirst = -3, kTangThird = -6, kTangSlope = -11;

// The quartic through five means from the four differences a..d of neighbours: the
// centre's difference A = b + c, second difference s, the third differences t0, t1, their
// sum ts and difference td.
struct QuarticParts { ff A, s, t0, t1, ts, td; };
CGKS_SPLIT_FN QuarticParts quartic_split(ff a, ff b, ff c, ff d)
{
    QuarticParts q;
    q.A = ff_add(b, c);
    q.s = ff_sub(c, b);
    q.t0 = ff_sub(q.s, ff_sub(b, a));
    q.t1 = ff_sub(ff_sub(d, c), q.s);
    q.ts = ff_add(q.t0, q.t1);
    q.td = ff_sub(q.t1, q.t0);
    return q;
}
// a float's bits for a scale's high word (within split_scale_ok's range)
CGKS_SPLIT_FN int f_scale_word(int scale_hi) { return (scale_hi - (896 << 20)) << 3; }
CGKS_SPLIT_FN int f_abs_word(float x) { return (int)(f_word(x) & 0x7fffffffu); }

// Five means: D1 - sum_k w_k D_k = w_0 t0 + w_2 t1 at both Gauss points, from D1, the
// centre's second difference s1, the third differences t0, t1 and 4 x epsilon; dlo,
// dhi: the linear weights over the centre's.
CGKS_SPLIT_FN void tang_weno5_split(ff D1, ff s1, ff t0, ff t1, ff eps4, ff dlo, ff dhi, ff& minus, ff& plus)
{
    const ff c133 = CGKS_FF(13.0 / 3.0);
    auto e = [&](ff D, ff s) { return ff_addp(ff_addp(ff_sqr(D), ff_mul(c133, ff_sqr(s))), eps4); };
    const ff e0 = e(ff_sub(D1, t0), ff_sub(s1, t0)), e1 = e(D1, s1), e2 = e(ff_sub(D1, t1), ff_add(s1, t1));
    ff Z = ff_sub(e0, e2);
    if (Z.h < 0.0f) Z = ff_neg(Z);
    const ff one = ff{1.0f, 0.0f};
    const ff a0 = ff_addp(one, ff_mul(Z, ff_rcp(e0))), a1 = ff_addp(one, ff_mul(Z, ff_rcp(e1))),
             a2 = ff_addp(one, ff_mul(Z, ff_rcp(e2)));
    const ff l0 = ff_mul(dlo, a0), h0 = ff_mul(dhi, a0), l2 = ff_mul(dlo, a2), h2 = ff_mul(dhi, a2);
    const ff dp = ff_addp(ff_addp(l0, h2), a1), dm = ff_addp(ff_addp(h0, l2), a1);
    plus = ff_mul(ff_add(ff_mul(l0, t0), ff_mul(h2, t1)), ff_rcp(dp));
    minus = ff_mul(ff_add(ff_mul(h0, t0), ff_mul(l2, t1)), ff_rcp(dm));
}

// Three means, slopes dm, dp to the neighbours, A = dp + dm, s = dp - dm: the nonlinear
// slope is (A - c) / 2 with c = Z sA s / (2 e0 e1 + Z (e0 + e1)), Z = |sA|: all of one
// sign below, so c keeps the pairs' relative accuracy.
CGKS_SPLIT_FN ff tang_weno3_split(ff A, ff s, ff eps)
{
    const ff dm = ff_scale(0.5f, ff_sub(A, s)), dp = ff_scale(0.5f, ff_add(A, s));
    const ff e0 = ff_addp(ff_sqr(dm), eps), e1 = ff_addp(ff_sqr(dp), eps);
    const ff sA = ff_mul(s, A);
    const ff Z = sA.h < 0.0f ? ff_neg(sA) : sA;
    const ff den = ff_addp(ff_scale(2.0f, ff_mul(e0, e1)), ff_mul(Z, ff_addp(e0, e1)));
    return ff_mul(ff_mul(ff_mul(Z, sA), s), ff_rcp(den));
}

// ------------------------------------------------------------------------
// Ranges.  The pairs' floats hold a number's 47 bits from 2^-74 to 2^128, and its leading 24 with an
// error below 2^-97 beneath that; the quantities of a face's time derivatives and slope moments carry
// units (density rho, a speed a, a rate or length), so their pairs are used only where the units keep
// the operands that matter and all results inside.  Logarithms here are base 2, in units of 2^-20, read
// off the high words (exact at powers of two, up to 0.09 too small between them); zero gives -1023,
// infinity and NaN 1024.
constexpr int kOct = 1 << 20;
CGKS_SPLIT_FN int hi_log(double x) { return hi_abs(x) - kHiOne; }
CGKS_SPLIT_FN int clamp_log(int x) { return i_max(i_min(x, 60 * kOct), -60 * kOct); }

// W_tt.  Density rho, energy E (so a = sqrt(E / rho)) and the time step: with the rate k = 1/(a dt) and
// derivatives up to k and k^2 times their variables (the caller's bound), the operands are of size rho^i
// a^j k^m with |i| <= 1, j <= 3, m <= 2 and no result exceeds rho^i a^j k^m with i <= 2, j <= 4, m <= 2.  Operands
// of 2^-50 and more lose at most 2^-47 of themselves, results stay below 2^110 (16 orders left for the
// sums).
CGKS_SPLIT_FN bool wtt_range_ok(int lrho, int lE, int ldt)
{
    const int r = clamp_log(lrho), a = clamp_log((lE - lrho) >> 1), k = clamp_log(-ldt - a);
    return (i_max(2 * r, -r) + i_max(4 * a, 0) + i_max(2 * k, 0) <= 110 * kOct) &
           (-i_max(r, -r) + i_min(3 * a, 0) + i_min(2 * k, 0) >= -50 * kOct);
}

// Slope moments of both sides.  Their densities and thetas lie between rlo, rhi and tlo, thi, |U| and |V|
// below speed; inv is the inverse spacing along the face, weight the larger weight's word (a float >= 0).
// Moments to the third power of the speeds a (2^-16 to 2^16) are operands, and a slope's absolute error
// of 2^-97 (times the inverse spacing where that is above 1) reaches the fluxes of size rho a, rho a^2,
// rho a^3 as weight a, weight and weight / a times itself over rho, which has to stay below 2^-56.  Slopes too
// large for a float give results that no bound admits.
CGKS_SPLIT_FN int f_log(float w) { return (int)(f_word(w) >> 3) - (127 << 20); }
CGKS_SPLIT_FN bool slopes_range_ok(int rlo, int rhi, int tlo, int thi, int speed, int inv, int weight)
{
    const int lc = tlo >> 1, la = i_max(thi >> 1, speed);
    return (i_max(rhi, -rlo) <= 40 * kOct) & (lc >= -16 * kOct) & (la <= 16 * kOct) & (inv <= 60 * kOct) &
           (weight - rlo + i_max(la, -lc) + i_max(inv, 0) <= 40 * kOct);
}

// The rows of normal derivatives along a face, of size scale x inverse spacing: operands of 2^-45 and more
// keep the absolute error of 2^-97 below 2^-52 of the row.
CGKS_SPLIT_FN bool deriv_rows_range_ok(int lscale, int linv) { return i_min(linv, 60 * kOct) + lscale >= -45 * kOct; }

}  // namespace cgks
