// cgks_segment.cuh -- the per-face-segment arithmetic of the flux kernel
// (cgks_stage.cuh): the layout of a tile's face-row records in shared memory,
// the reconstruction along a face at a Gauss point (SegmentRows) and one
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

template <int TX, int TY, int STAGE>
struct StageLayout {
    static constexpr int NF = FaceQ<STAGE>::n;
    static constexpr int n_rx = RecGroups<TY, TX + 1>::n;
    static constexpr int n_ry = RecGroups<TX, TY + 1>::n;
    // a slice per pair of threads: what the two Gauss points of its segment share
    static constexpr int n_parts = 48 * kPairs;
    static constexpr size_t bytes = sizeof(double) * (size_t)(n_rx + n_ry + n_parts);
};

// One Gauss point of a face segment: the face rows around it (records of rows
// j-2..j+2 of one face) and the reconstruction along the face there.  The
// segment's slice (segment_parts; part j of variable k at part[(kPartsVar k + j)
// * stride]) holds what its two Gauss points share.
enum { kPartsVar = 12, kParts = 4 * kPartsVar };   // 0..7: deriv_parts, 8, 9: W0 at eta = -g, +g, 10, 11: slopes of W_l, W_r

struct SegmentPoint {
    RegK r;
    const double* rec;
    int pa, pb, pc, r0, rstride;
    double eta, iht;
    int gp;                       // 0: eta = -g, 1: +g
    const double* part;
    int stride;

    __device__ __forceinline__ double at(int f, int k, int off) const
    {
        return rec_at(rec, pa, pb, pc, r0, rstride, f, k, off);
    }
    __device__ __forceinline__ double P(int k, int j) const { return part[(kPartsVar * k + j) * stride]; }

    __device__ __forceinline__ void eq_value(double W[4]) const
    {
#pragma unroll
        for (int k = 0; k < 4; ++k) W[k] = P(k, 8 + gp);
    }

    // The quartic through the segment means m_{j-2..j+2} (m0 the centre row): with A1 =
    // m_1 - m_-1, the second difference s1, the sum ts and the difference td of the two
    // third differences,
    //   p(eta)   = m0 - td/4320 + eta (A1/2 - 7 ts/72) + O(eta^2 - 1/12)
    //   p'(eta)  = A1/2 - ts/12 + eta (s1 - td/9) + O(eta^2 - 1/12)
    //   p''(eta) = s1 - td/12 + eta ts/2 + O(eta^2 - 1/12)
    // (exact at the Gauss points eta = +-1/(2 sqrt 3), where eta^2 = 1/12)
    __device__ __forceinline__ void eq_derivs(double W0n[4], double W0t[4], double W0nn[4], double W0nt[4],
                                              double W0tt[4]) const
    {
        const double iht2 = r.mul(iht, iht);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            W0t[k] = r.mul(fma(eta, P(k, 1), P(k, 0)), iht);
            W0tt[k] = r.mul(fma(eta, P(k, 3), P(k, 2)), iht2);
            W0n[k] = fma(eta, P(k, 5), P(k, 4));
            W0nt[k] = r.mul(fma(eta, P(k, 7), P(k, 6)), iht);
            W0nn[k] = at(RNN, k, 0);
        }
    }

    __device__ __forceinline__ void ne_value(int side, double W[4]) const
    {
        const int f = side ? RR : RL;
#pragma unroll
        for (int k = 0; k < 4; ++k) W[k] = fma(eta, P(k, 10 + side), at(f, k, 0));
    }

    __device__ __forceinline__ void ne_slopes(int side, double Wn[4], double Wt[4]) const
    {
        const int f = side ? RRN : RLN;
        const double he = r.kmul(FK_HALF, eta);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Wn[k] = fma(he, r.sub(at(f, k, 1), at(f, k, -1)), at(f, k, 0));
            Wt[k] = r.mul(P(k, 10 + side), iht);
        }
    }

#ifndef CGKS_OPCOUNT_HOST
    __device__ __forceinline__ void ne_slopes_split(int side, ff Wn[4], ff Wt[4]) const
    {
        const int f = side ? RRN : RLN;
        const ff he = ff_from(r.kmul(FK_HALF, eta)), ih = ff_from(iht);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Wn[k] = ff_add(ff_mul(he, ff_sub(ff_from(at(f, k, 1)), ff_from(at(f, k, -1)))), ff_from(at(f, k, 0)));
            Wt[k] = ff_mul(ff_from(P(k, 10 + side)), ih);
        }
    }
#endif
};

// the eta-independent parts of the quartic's derivatives for one variable (differences x
// of the values, rows n_{-2..2} of the normal derivatives), part j at p[j * stride]
__device__ __forceinline__ void deriv_parts(const RegK& r, double* p, int stride, const TangDiffs& x, double n2m,
                                            double nm, double n0, double np, double n2p)
{
    {
        const double ts = r.add(x.t0, x.t1), td = r.sub(x.t1, x.t0);
        p[0 * stride] = r.kfma(FK_M12TH, ts, r.kmul(FK_HALF, x.A1));
        p[1 * stride] = r.kfma(FK_M9TH, td, x.s1);
        p[2 * stride] = r.kfma(FK_M12TH, td, x.s1);
        p[3 * stride] = r.kmul(FK_HALF, ts);
    }
    const double B1 = r.sub(np, nm), hB = r.kmul(FK_HALF, B1), s1 = r.kfma(FK_M2, n0, r.add(np, nm));
    const double ts = r.kfma(FK_M2, B1, r.sub(n2p, n2m));
    const double td = r.kfma(FK_M4, s1, r.kfma(FK_M2, n0, r.add(n2p, n2m)));
    p[4 * stride] = r.kfma(FK_M4320TH, td, n0);
    p[5 * stride] = r.kfma(FK_M7_72, ts, hB);
    p[6 * stride] = r.kfma(FK_M12TH, ts, hB);
    p[7 * stride] = r.kfma(FK_M9TH, td, s1);
}

// What the Gauss points of a segment share, for variables k0..k1-1: the nonlinear values
// along the face at both points, the non-equilibrium slopes, the derivatives' parts.  A
// rolled loop: unrolled, its instructions alone outgrow the instruction cache.
__device__ __forceinline__ void segment_parts(const RegK& r, const double* rec, int pa, int pb, int pc, int r0,
                                              int rstride, int k0, int k1, double* part, int stride)
{
    const double weps = r.k(FK_WEPS), weps4 = r.k(FK_WEPS4);
    auto R = [&](int f, int k, int off) { return rec_at(rec, pa, pb, pc, r0, rstride, f, k, off); };
#ifndef CGKS_OPCOUNT_HOST
    // scales (high words): the smallest of the three states' densities and energies; a
    // momentum also against sqrt(rho E)
    const int sc0 = i_min(i_min(hi_abs(R(RV, 0, 0)), hi_abs(R(RL, 0, 0))), hi_abs(R(RR, 0, 0)));
    const int sc3 = i_min(i_min(hi_abs(R(RV, 3, 0)), hi_abs(R(RL, 3, 0))), hi_abs(R(RR, 3, 0)));
#endif
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
        double* p = part + kPartsVar * k * stride;
        const double m0 = R(RV, k, 0);
        TangDiffs x;
        tang_diffs(r, R(RV, k, -2), R(RV, k, -1), m0, R(RV, k, 1), R(RV, k, 2), x);
#ifdef CGKS_OPCOUNT_HOST
        const int sc = 0;
#else
        const int sc = k == 0 ? sc0 : k == 3 ? sc3 : i_max(hi_abs(m0), (sc0 >> 1) + (sc3 >> 1));
#endif
        tang_weno5_pair(r, m0, x, weps4, sc, p[8 * stride], p[9 * stride]);
        deriv_parts(r, p, stride, x, R(RN, k, -2), R(RN, k, -1), R(RN, k, 0), R(RN, k, 1), R(RN, k, 2));
        tang_weno3_slopes(r, R(RL, k, -1), R(RL, k, 0), R(RL, k, 1), R(RR, k, -1), R(RR, k, 0), R(RR, k, 1), weps, sc,
                          p[10 * stride], p[11 * stride]);
    }
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
                                                int rstride, double iht, double* part, int stride,
                                                double acc[FaceQ<STAGE>::n])
{
    constexpr double gq = 0.28867513459481287;   // 1/(2 sqrt 3): Gauss points at +-gq
    segment_parts(r, rec, pa, pb, pc, r0, rstride, 0, 4, part, stride);
    PointResult<STAGE> s;
    bool ok = true;
#pragma unroll 1
    for (int gp = 0; gp < 2; ++gp) {
        const SegmentPoint src{r, rec, pa, pb, pc, r0, rstride, gp ? gq : -gq, iht, gp, part, stride};
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
