// cgks_segment.cuh -- the per-face-segment arithmetic of the flux kernel
// (cgks_stage.cuh): the layout of a tile's face-row records in shared memory,
// the reconstruction along a face at a Gauss point (SegmentPoint) and one
// segment's two Gauss points with their Gauss average (segment_results).
#pragma once
#include "cgks_device.cuh"
#include "cgks_flux.cuh"
#include "cgks_internal.h"

namespace cgks {

constexpr int kThreads = 128, kPairs = kThreads / 2;

template <int STAGE> struct FaceQ { static constexpr int n = (STAGE == 1) ? 16 : 8; };

// Face-row records of one orientation in shared memory: T own rows of F faces.
// Group A (RV, RN: 8 planes) on rows -2..T+1, group B (RL, RR, RLN, RRN: 16
// planes) on rows -1..T, group C (RNN: 4 planes) on rows 0..T-1 -- the rows each
// field is read on.
template <int T, int F>
struct RecGroups {
    static constexpr int pa = (T + 4) * F, pb = (T + 2) * F, pc = T * F;
    static constexpr int n = 8 * pa + 16 * pb + 4 * pc;
};

// field f, variable k, row `off` relative to the row of r0 = row * F + face
__device__ __forceinline__ double rec_at(const double* rec, int pa, int pb, int pc, int r0, int F, int f, int k,
                                         int off)
{
    if (f == RV || f == RN) return rec[(f * 4 + k) * pa + r0 + (off + 2) * F];
    if (f == RNN) return rec[8 * pa + 16 * pb + k * pc + r0 + off * F];
    return rec[8 * pa + ((f - RL) * 4 + k) * pb + r0 + (off + 1) * F];
}

// Parts of a variable: W0, twice its tangential slope per unit eta and its normal derivative
// at eta = -g and +g; twice the slopes of W_l and W_r; what the second derivatives need (d2/deta2 =
// PTT0 + eta PTT1, d2/dn deta = PNT0 + eta PNT1), as pairs of FP32, or in FP64 where the other
// parts are (and in the host operation count).  kRough: the slot of a bit per variable with FP64 parts.
enum { PV = 0, PT = 2, PN = 4, PS = 6, PTT0 = 8, PTT1, PNT0, PNT1, kPartsVar, kRough = 4 * kPartsVar, kParts };

template <int TX, int TY, int STAGE>
struct StageLayout {
    static constexpr int n_rx = RecGroups<TY, TX + 1>::n;
    static constexpr int n_ry = RecGroups<TX, TY + 1>::n;
    static constexpr int n_rec = n_rx + n_ry;
    // a slice per pair of threads: what the two Gauss points of its segment share
    static constexpr int n_parts = kParts * kPairs;
    // record buffers: two where the shape's CTAs still fit an SM (static shared memory and
    // the 1 KB the system takes per CTA included)
    static constexpr int buffers =
        stage_ctas(TX, TY) * (sizeof(double) * (size_t)(2 * n_rec + n_parts) + 2560) <= 228 * 1024 ? 2 : 1;
    static constexpr size_t bytes = sizeof(double) * (size_t)(buffers * n_rec + n_parts);
};

// The quartic through the segment means m_{j-2..j+2} (m0 the centre row): with A1 = m_1 -
// m_-1, the second difference s1, the sum ts and the difference td of the two third
// differences,
//   p(eta)   = m0 - td/4320 + eta (A1/2 - 7 ts/72) + O(eta^2 - 1/12)
//   p'(eta)  = A1/2 - ts/12 + eta (s1 - td/9) + O(eta^2 - 1/12)
//   p''(eta) = s1 - td/12 + eta ts/2 + O(eta^2 - 1/12)
// (exact at the Gauss points eta = +-1/(2 sqrt 3), where eta^2 = 1/12)
__device__ __forceinline__ double quartic_v0(const RegK& r, double m0, const TangDiffs& x) { return r.kfma(FK_M4320TH, r.sub(x.t1, x.t0), m0); }
__device__ __forceinline__ double quartic_v1(const RegK& r, const TangDiffs& x) { return r.kfma(FK_M7_72, r.add(x.t0, x.t1), r.kmul(FK_HALF, x.A1)); }
__device__ __forceinline__ double quartic_t0(const RegK& r, const TangDiffs& x) { return r.kfma(FK_M12TH, r.add(x.t0, x.t1), r.kmul(FK_HALF, x.A1)); }
__device__ __forceinline__ double quartic_t1(const RegK& r, const TangDiffs& x) { return r.kfma(FK_M9TH, r.sub(x.t1, x.t0), x.s1); }
__device__ __forceinline__ double quartic_tt0(const RegK& r, const TangDiffs& x) { return r.kfma(FK_M12TH, r.sub(x.t1, x.t0), x.s1); }
__device__ __forceinline__ double quartic_tt1(const RegK& r, const TangDiffs& x) { return r.kmul(FK_HALF, r.add(x.t0, x.t1)); }

// One Gauss point of a face segment: the face rows around it (records of rows
// j-2..j+2 of one face) and the reconstruction along the face there.  The
// segment's slice (segment_parts; part j of variable k at part[(kPartsVar k + j)
// * stride]) holds what its two Gauss points share.
constexpr double kGauss = 0.28867513459481287;   // 1/(2 sqrt 3): Gauss points at +-kGauss

struct SegmentPoint {
    RegK r;
    const double* rec;
    int pa, pb, pc, r0, rstride;
    double eta, iht, hiht;        // inverse spacing along the face and its half
    int gp;                       // 0: eta = -g, 1: +g
    const double* part;
    int stride;
    int ihp;                      // table index of iht as a pair

    __device__ __forceinline__ double at(int f, int k, int off) const
    {
        return rec_at(rec, pa, pb, pc, r0, rstride, f, k, off);
    }
    __device__ __forceinline__ double P(int k, int j) const { return part[(kPartsVar * k + j) * stride]; }
#ifdef CGKS_PAIRS
    // the same where a slot may hold a pair instead: read again where it is used (a value kept from the
    // pair's read to there costs two registers for each of 16 slots, 100 B of spills in all)
    __device__ __forceinline__ double P64(int k, int j) const { return ((volatile const double*)part)[(kPartsVar * k + j) * stride]; }
    // the variables with FP64 parts (segment_parts), a bit each
    __device__ __forceinline__ int rough() const
    {
        const volatile int* m = (const volatile int*)(part + kRough * stride);
        return m[0] | m[1];
    }
#endif

    __device__ __forceinline__ void eq_value(double W[4]) const
    {
#pragma unroll
        for (int k = 0; k < 4; ++k) W[k] = P(k, PV + gp);
    }

    __device__ __forceinline__ void eq_first(double W0n[4], double W0t[4]) const
    {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            W0n[k] = P(k, PN + gp);
            W0t[k] = r.mul(P(k, PT + gp), hiht);
        }
    }

    // the second derivatives in FP64: from the slice where it holds their parts so, else from the rows (always
    // from the rows took 124 of a rough point's FP64 instructions)
    __device__ __forceinline__ void eq_second(double W0nn[4], double W0nt[4], double W0tt[4]) const
    {
        const double iht2 = r.mul(iht, iht);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            W0nn[k] = at(RNN, k, 0);
#ifndef CGKS_PAIRS
            W0tt[k] = r.mul(fma(eta, P(k, PTT1), P(k, PTT0)), iht2);
            W0nt[k] = r.mul(fma(eta, P(k, PNT1), P(k, PNT0)), iht);
#else
            if (rough() >> k & 1) {
                W0tt[k] = r.mul(fma(eta, P64(k, PTT1), P64(k, PTT0)), iht2);
                W0nt[k] = r.mul(fma(eta, P64(k, PNT1), P64(k, PNT0)), iht);
                continue;
            }
            TangDiffs x;
            tang_diffs(r, at(RV, k, -2), at(RV, k, -1), at(RV, k, 0), at(RV, k, 1), at(RV, k, 2), x);
            W0tt[k] = r.mul(fma(eta, quartic_tt1(r, x), quartic_tt0(r, x)), iht2);
            tang_diffs(r, at(RN, k, -2), at(RN, k, -1), at(RN, k, 0), at(RN, k, 1), at(RN, k, 2), x);
            W0nt[k] = r.mul(fma(eta, quartic_t1(r, x), quartic_t0(r, x)), iht);
#endif
        }
    }

#ifdef CGKS_PAIRS
    __device__ __forceinline__ void eq_second_split(ff W0nn[4], ff W0nt[4], ff W0tt[4]) const
    {
        const ff ih = ff_unpack(r.k(ihp)), ih2 = ff_mul(ih, ih), et = gp ? CGKS_FF(kGauss) : CGKS_FF(-kGauss);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            W0tt[k] = ff_mul(ff_addp(ff_unpack(P(k, PTT0)), ff_mul(et, ff_unpack(P(k, PTT1)))), ih2);
            W0nt[k] = ff_mul(ff_addp(ff_unpack(P(k, PNT0)), ff_mul(et, ff_unpack(P(k, PNT1)))), ih);
            W0nn[k] = ff_from_any(at(RNN, k, 0));
        }
    }
#endif

    __device__ __forceinline__ void ne_value(int side, double W[4]) const
    {
        const int f = side ? RR : RL;
        const double heta = r.k(gp ? FK_HG : FK_MHG);   // eta / 2
#pragma unroll
        for (int k = 0; k < 4; ++k) W[k] = fma(heta, P(k, PS + side), at(f, k, 0));
    }

    __device__ __forceinline__ void ne_slopes(int side, double Wn[4], double Wt[4]) const
    {
        const int f = side ? RRN : RLN;
        const double he = r.kmul(FK_HALF, eta);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Wn[k] = fma(he, r.sub(at(f, k, 1), at(f, k, -1)), at(f, k, 0));
            Wt[k] = r.mul(P(k, PS + side), hiht);
        }
    }

#ifdef CGKS_PAIRS
    __device__ __forceinline__ void ne_slopes_split(int side, ff Wn[4], ff Wt[4]) const
    {
        const int f = side ? RRN : RLN;
        const ff he = gp ? CGKS_FF(0.5 * kGauss) : CGKS_FF(-0.5 * kGauss), ih = ff_scale(0.5f, ff_unpack(r.k(ihp)));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Wn[k] = ff_addp(ff_mul(he, ff_addp(ff_from_any(at(f, k, 1)), ff_neg(ff_from_any(at(f, k, -1))))), ff_from_any(at(f, k, 0)));
            Wt[k] = ff_mul(ff_from_any(P(k, PS + side)), ih);
        }
    }
#endif
};

// What the Gauss points of a segment share, for variables k0..k1-1.  Corrections in
// pairs of FP32 where the rows' differences are small beside the variable's scale (ihn:
// inverse spacing along the normal, for the derivative rows' differences), else in FP64.
// A variable whose rows are too rough for that has its second derivatives' parts in FP64 and its bit in the
// kRough slot set.  On rough data everywhere (512^2, stage 1 / 2) an all-FP64 kernel took 2170 /
// 1805 us, this one 2411 / 2050 with pairs tried first for every part of every point, and 2137 / 1800 where a rough
// variable is left out of what hardly ever qualifies then.
// A rolled loop: unrolled, its instructions alone outgrow the instruction cache.
__device__ __forceinline__ void segment_parts(const RegK& r, const double* rec, int pa, int pb, int pc, int r0,
                                              int rstride, double ihn, int k0, int k1, double* part, int stride)
{
    const double weps = r.k(FK_WEPS), weps4 = r.k(FK_WEPS4);
    int rough = 0;
    auto R = [&](int f, int k, int off) { return rec_at(rec, pa, pb, pc, r0, rstride, f, k, off); };
#ifdef CGKS_PAIRS
    // scales (high words): the smallest of the three states' densities and energies; a
    // momentum also against sqrt(rho E)
    const int sc0 = i_min(i_min(hi_abs(R(RV, 0, 0)), hi_abs(R(RL, 0, 0))), hi_abs(R(RR, 0, 0)));
    const int sc3 = i_min(i_min(hi_abs(R(RV, 3, 0)), hi_abs(R(RL, 3, 0))), hi_abs(R(RR, 3, 0)));
#endif
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
        double* p = part + kPartsVar * k * stride;
        int sc = 0;
        bool split = false;
        const double m0 = R(RV, k, 0), n0 = R(RN, k, 0);
#ifdef CGKS_PAIRS
        sc = k == 0 ? sc0 : k == 3 ? sc3 : i_max(hi_abs(m0), (sc0 >> 1) + (sc3 >> 1));
        {
            const double vm = R(RV, k, -1), vp = R(RV, k, 1), nm = R(RN, k, -1), np = R(RN, k, 1);
            const double va = r.sub(vm, R(RV, k, -2)), vb = r.sub(m0, vm), vc = r.sub(vp, m0), vd = r.sub(R(RV, k, 2), vp);
            const double na = r.sub(nm, R(RN, k, -2)), nb = r.sub(n0, nm), nc = r.sub(np, n0), nd = r.sub(R(RN, k, 2), np);
            const QuarticParts v = quartic_split(ff_from(va), ff_from(vb), ff_from(vc), ff_from(vd));
            const int m1 = i_max(i_max(hi_abs(va), hi_abs(vb)), i_max(hi_abs(vc), hi_abs(vd)));
            const int mn = i_max(i_max(hi_abs(na), hi_abs(nb)), i_max(hi_abs(nc), hi_abs(nd)));
            const int lim = sc + kTangFirst * (1 << 20);
            split = split_scale_ok(sc, weps4) && deriv_rows_range_ok(sc - kHiOne, hi_log(ihn)) && m1 < lim && mn < lim + i_min(hi_abs(ihn), kHiOne + (60 << 20)) - kHiOne &&
                    i_max(f_abs_word(v.t0.h), f_abs_word(v.t1.h)) < f_scale_word(sc) + kTangThird * (1 << 23);
            if (split) {
                const ff g = CGKS_FF(kGauss), m12 = CGKS_FF(-1.0 / 12.0), c9 = CGKS_FF(1.0 / 9.0);
                auto sum = [&](double base, ff c) { return r.add(base, r.add(d_from(c.h), d_from(c.l))); };
                const double A1 = r.sub(vp, vm);
                ff lo, hi;
                tang_weno5_split(v.A, v.s, v.t0, v.t1, ff_unpack(r.k(FK_PWEPS4)), CGKS_FF(kTangLo), CGKS_FF(kTangHi), lo, hi);
                p[(PV + 0) * stride] = r.kfma(FK_MHG, sum(A1, ff_neg(lo)), m0);
                p[(PV + 1) * stride] = r.kfma(FK_HG, sum(A1, ff_neg(hi)), m0);
                // the quartic of SegmentPoint: slope A1/2 - ts/12 + eta (s - td/9), second derivative
                // s - td/12 + eta ts/2, value + eta (A1/2 - 7 ts/72) - td/4320
                const ff x = ff_mul(CGKS_FF(-1.0 / 6.0), v.ts), y = ff_mul(CGKS_FF(2.0 * kGauss), ff_sub(v.s, ff_mul(c9, v.td)));
                p[(PT + 0) * stride] = sum(A1, ff_sub(x, y));
                p[(PT + 1) * stride] = sum(A1, ff_add(x, y));
                p[PTT0 * stride] = ff_pack(ff_add(v.s, ff_mul(m12, v.td)));
                p[PTT1 * stride] = ff_pack(ff_scale(0.5f, v.ts));
                const QuarticParts n = quartic_split(ff_from(na), ff_from(nb), ff_from(nc), ff_from(nd));
                const ff hB = ff_scale(0.5f, n.A), u = ff_mul(CGKS_FF(-1.0 / 4320.0), n.td),
                         w = ff_mul(g, ff_add(hB, ff_mul(CGKS_FF(-7.0 / 72.0), n.ts)));
                p[(PN + 0) * stride] = sum(n0, ff_sub(u, w));
                p[(PN + 1) * stride] = sum(n0, ff_add(u, w));
                p[PNT0 * stride] = ff_pack(ff_add(hB, ff_mul(m12, n.ts)));
                p[PNT1 * stride] = ff_pack(ff_sub(n.s, ff_mul(c9, n.td)));
            }
        }
#endif
        if (!split) {
            rough |= 1 << k;
            TangDiffs x;
            tang_diffs(r, R(RV, k, -2), R(RV, k, -1), m0, R(RV, k, 1), R(RV, k, 2), x);
            tang_weno5_pair(r, m0, x, weps4, p[(PV + 0) * stride], p[(PV + 1) * stride]);
            const double t0 = quartic_t0(r, x), t2 = r.add(t0, t0), gt = r.mul(2.0 * kGauss, quartic_t1(r, x));
            p[(PT + 0) * stride] = r.sub(t2, gt);
            p[(PT + 1) * stride] = r.add(t2, gt);
            p[PTT0 * stride] = quartic_tt0(r, x);
            p[PTT1 * stride] = quartic_tt1(r, x);
            tang_diffs(r, R(RN, k, -2), R(RN, k, -1), n0, R(RN, k, 1), R(RN, k, 2), x);
            const double v0 = quartic_v0(r, n0, x), gv = r.mul(kGauss, quartic_v1(r, x));
            p[(PN + 0) * stride] = r.sub(v0, gv);
            p[(PN + 1) * stride] = r.add(v0, gv);
            p[PNT0 * stride] = quartic_t0(r, x);
            p[PNT1 * stride] = quartic_t1(r, x);
        }
        // (a scale of 0 admits no pairs)
        tang_weno3_slopes(r, R(RL, k, -1), R(RL, k, 0), R(RL, k, 1), R(RR, k, -1), R(RR, k, 0), R(RR, k, 1), weps,
                          split ? sc : 0, p[(PS + 0) * stride], p[(PS + 1) * stride]);
    }
#ifdef CGKS_PAIRS
    // each of a pair's lanes has a half of the slot (one thread with all variables has both)
    int* m = (int*)(part + kRough * stride);
    m[k0 >> 1] = rough;
    if (k1 - k0 == 4) m[1] = rough;
#endif
}

// The results of one Gauss point (stage 1: Fb, Ft, Wm, Wb; stage 2: Ft, Wtt in a, b).
template <int STAGE> struct PointResult { double a[4], b[4], c[4], d[4]; };

template <int STAGE>
__device__ __forceinline__ bool segment_point(const SegmentPoint& src, PointResult<STAGE>& o)
{
    if constexpr (STAGE == 1) return gks_point<1>(src.r, src, o.a, o.b, o.c, o.d, o.d);
    else return gks_point<2>(src.r, src, o.c, o.a, o.c, o.d, o.b);
}

// Variable k of a segment's results (face frame) from the sums of its two points' results:
// the Gauss weight 1/2 times the stage's time factors; stage 1: the W* and R flux
// combinations and the interface states W(dt/2), W(dt); stage 2: dt^2/3 F_t, dt^2/3 W_tt.
// put(q, value): result group q.
template <int STAGE, class Put>
__device__ __forceinline__ void gauss_average(const RegK& r, double a, double b, double c, double d, Put put)
{
    if constexpr (STAGE == 1) {
        put(0, r.kfma(FK_W1B, b, r.kmul(FK_W1A, a)));
        put(1, r.kfma(FK_W2B, b, r.kmul(FK_W2A, a)));
        put(2, r.kmul(FK_HALF, c));
        put(3, r.kmul(FK_HALF, d));
    } else {
        put(0, r.kmul(FK_W3, a));
        put(1, r.kmul(FK_W3, b));
    }
}

// One face segment by one thread (the flux kernel gives each Gauss point a thread of its
// own, the same operations): parts, both points, the average into acc (face frame).
// Returns false if a state was non-physical.
template <int STAGE>
__device__ __forceinline__ bool segment_results(const RegK& r, const double* rec, int pa, int pb, int pc, int r0,
                                                int rstride, bool xo, double* part, int stride,
                                                double acc[FaceQ<STAGE>::n])
{
    const double iht = r.k(xo ? FK_IDY : FK_IDX);
    const int ihp = xo ? FK_PIDY : FK_PIDX;
    segment_parts(r, rec, pa, pb, pc, r0, rstride, r.k(xo ? FK_IDX : FK_IDY), 0, 4, part, stride);
    PointResult<STAGE> s;
    bool ok = true;
#pragma unroll 1
    for (int gp = 0; gp < 2; ++gp) {
        const SegmentPoint src{r, rec, pa, pb, pc, r0, rstride, gp ? kGauss : -kGauss, iht, r.k(xo ? FK_HIDY : FK_HIDX), gp, part,
                               stride, ihp};
        PointResult<STAGE> o;
        ok &= segment_point<STAGE>(src, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            s.a[k] = gp ? r.add(s.a[k], o.a[k]) : o.a[k];
            s.b[k] = gp ? r.add(s.b[k], o.b[k]) : o.b[k];
            if (STAGE == 1) {
                s.c[k] = gp ? r.add(s.c[k], o.c[k]) : o.c[k];
                s.d[k] = gp ? r.add(s.d[k], o.d[k]) : o.d[k];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        gauss_average<STAGE>(r, s.a[k], s.b[k], s.c[k], s.d[k], [&](int q, double v) { acc[4 * q + k] = v; });
    return ok;
}

}  // namespace cgks
