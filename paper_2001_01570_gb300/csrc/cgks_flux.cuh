// cgks_flux.cuh -- device arithmetic of the flux kernel: the reconstruction
// along a face (Gauss-point values and derivatives), the Maxwellian moments,
// the micro-slopes, the Euler time derivatives and the gas-kinetic evaluation
// at one interface quadrature point (Sec. 2.1-2.2, Sec. 4).
//
// All of it is written in the register-only DFMA forms of RegK (see
// cgks_device.cuh): x + y = fma(x, 1, y), x * y = fma(x, y, -0), and every
// coefficient -- the fixed ones and the per-grid / per-tile ones (gamma, K,
// dt and their combinations) -- is read from the shared-memory table FluxK at
// its point of use.
#pragma once
#include "cgks_device.cuh"
#include "cgks_internal.h"

namespace cgks {

// A branch that the compiler may not turn into predicated instructions: those occupy the
// FP64 unit whether their predicate holds or not (the interface state's non-equilibrium
// terms, skipped by almost every warp, cost stage 1 a ninth of its FP64 instructions so).
#define CGKS_BRANCH(cond) _Pragma("unroll 1") for (bool go_ = (cond); go_; go_ = false)

// Layout of the flux kernel's shared-memory table.  Fixed constants first
// (copied from global memory), then the values of the tile's grid and time step
// (written by the CTA's four warps when a tile's grid is not the tile's before).
enum FluxK {
    FK_ONE = 0, FK_NZERO, FK_HALF, FK_MHALF, FK_2, FK_3,
    FK_T13_3, FK_DLO, FK_DHI,              // tangential WENO-Z: 4 x beta weight, linear weights at the Gauss points
    FK_HG, FK_MHG,                         // +-eta/2 at the Gauss point eta = 1/(2 sqrt 3)
    FK_M12TH, FK_M9TH, FK_M4320TH, FK_M7_72,         // quartic through the five means: coefficients
    FK_C1P, FK_C1M,                                  // +-1/sqrt(pi)
    FK_X32LN2, FK_SHIFT, FK_LN2HI, FK_LN2LO,         // exponential: argument reduction
    FK_P2, FK_P3, FK_P4, FK_P5, FK_P6,               // exponential: 1/k! of the Taylor polynomial
    FK_NFIX,
    FK_EXP2 = FK_NFIX,                               // 2^(j/32), j = 0..31
    FK_NFIX2 = FK_EXP2 + 32,
    // per grid and tile
    FK_DT = FK_NFIX2, FK_IDT, FK_4IDT2, FK_HDT, FK_MHDT, FK_EPSDT, FK_CTAUDT, FK_C8, FK_C6,
    FK_W1A, FK_W1B, FK_W2A, FK_W2B, FK_W3,          // Gauss-average weights of the face results
    FK_GAMMA, FK_GM1, FK_K1, FK_K3, FK_K2INV2, FK_KHEAT, FK_MU,
    FK_IDX, FK_IDY, FK_HIDX, FK_HIDY, FK_WEPS, FK_WEPS4,
    // the same as pairs of FP32 (ff_pack): gamma, gamma - 1, K + 1, K + 3, inverse spacings, epsilons
    FK_PGAMMA, FK_PGM1, FK_PK1, FK_PK3, FK_PIDX, FK_PIDY, FK_PWEPS, FK_PWEPS4,
    FK_DT80,                                        // dt / 80 (its high word is compared)
    FK_N
};

// the linear weights of the outer candidates along a face over the centre one's, 11/18
constexpr double kTangLo = (7.0 / 36.0 - 1.7320508075688772 / 1080.0) * (18.0 / 11.0);
constexpr double kTangHi = (7.0 / 36.0 + 1.7320508075688772 / 1080.0) * (18.0 / 11.0);

struct FluxFixed { double v[FK_NFIX2]; };

constexpr FluxFixed make_flux_fixed()
{
    FluxFixed t{};
    double* k = t.v;
    k[FK_ONE] = 1.0; k[FK_NZERO] = -0.0; k[FK_HALF] = 0.5; k[FK_MHALF] = -0.5; k[FK_2] = 2.0;
    k[FK_3] = 3.0;
    const double gq = 0.28867513459481287;               // 1/(2 sqrt 3)
    k[FK_T13_3] = 13.0 / 3.0;
    k[FK_DLO] = kTangLo;
    k[FK_DHI] = kTangHi;
    k[FK_HG] = 0.5 * gq; k[FK_MHG] = -0.5 * gq;
    // the quartic p(eta) through the five segment means (quartic_v0 and the functions after it, cgks_segment.cuh)
    k[FK_M12TH] = -1.0 / 12.0; k[FK_M9TH] = -1.0 / 9.0; k[FK_M4320TH] = -1.0 / 4320.0; k[FK_M7_72] = -7.0 / 72.0;
    k[FK_C1P] = 0.56418958354775628; k[FK_C1M] = -0.56418958354775628;
    k[FK_X32LN2] = 32.0 / 0.6931471805599453;             // 32 / ln 2
    k[FK_SHIFT] = 6755399441055744.0;                      // 1.5 * 2^52: rounds to an integer in the low bits
    k[FK_LN2HI] = 0.6931471805599453 / 32.0;               // ln 2 / 32 and the remainder of its rounding
    k[FK_LN2LO] = 2.3190468138462996e-17 / 32.0;
    k[FK_P2] = 1.0 / 2.0; k[FK_P3] = 1.0 / 6.0; k[FK_P4] = 1.0 / 24.0; k[FK_P5] = 1.0 / 120.0;
    k[FK_P6] = 1.0 / 720.0;
    const double e2[32] = {                                // 2^(j/32)
        1.0, 1.0218971486541166, 1.0442737824274138, 1.0671404006768237,
        1.0905077326652577, 1.1143867425958924, 1.1387886347566916, 1.1637248587775775,
        1.189207115002721, 1.215247359980469, 1.241857812073484, 1.2690509571917332,
        1.2968395546510096, 1.3252366431597413, 1.3542555469368927, 1.383909881963832,
        1.4142135623730951, 1.4451808069770467, 1.4768261459394993, 1.5091644275934228,
        1.5422108254079407, 1.5759808451078865, 1.6104903319492543, 1.6457554781539649,
        1.681792830507429, 1.7186192981224779, 1.7562521603732995, 1.7947090750031072,
        1.8340080864093424, 1.8741676341103, 1.9152065613971474, 1.9571441241754002};
    for (int j = 0; j < 32; ++j) k[FK_EXP2 + j] = e2[j];
    return t;
}

// the table's entries for a grid and its time step, in four parts of about equal length
// for a warp each (one thread's chain took 4,300 cycles, the longest part's takes a third)
__device__ __forceinline__ void flux_table_part(double* t, const GridDev& G, double dt, int part)
{
    if (part == 0) {
        t[FK_DT] = dt;
        t[FK_HDT] = 0.5 * dt;
        t[FK_MHDT] = -0.5 * dt;
        t[FK_EPSDT] = G.eps_tau * dt;
        t[FK_CTAUDT] = G.c_tau * dt;
        t[FK_C8] = 0.125 * dt * dt;
        // stage 1: half of (dt/2, dt^2/8) and of (dt, dt^2/6) per Gauss point; stage 2: half of dt^2/3
        t[FK_W1A] = 0.25 * dt;
        t[FK_W1B] = dt * dt * (1.0 / 16.0);
        t[FK_W2A] = 0.5 * dt;
        t[FK_W2B] = dt * dt * (1.0 / 12.0);
        t[FK_W3] = dt * dt * (1.0 / 6.0);
    } else if (part == 1) {
        t[FK_IDT] = __drcp_rn(dt);
        t[FK_4IDT2] = 4.0 * __drcp_rn(dt * dt);
        t[FK_GAMMA] = G.gamma;
        t[FK_MU] = G.mu;
        t[FK_IDX] = G.inv_dx;
        t[FK_IDY] = G.inv_dy;
        t[FK_HIDX] = 0.5 * G.inv_dx;
        t[FK_HIDY] = 0.5 * G.inv_dy;
    } else if (part == 2) {
        t[FK_C6] = dt * dt / 6.0;
        t[FK_GM1] = G.gamma - 1.0;
        t[FK_K1] = G.K + 1.0;
        t[FK_K3] = G.K + 3.0;
        t[FK_K2INV2] = 2.0 * __drcp_rn(G.K + 2.0);
        t[FK_KHEAT] = 0.5 * (G.K + 4.0);
        t[FK_WEPS] = G.weno_eps;
        t[FK_WEPS4] = 4.0 * G.weno_eps;
    } else {
#ifdef CGKS_PAIRS
        t[FK_PGAMMA] = ff_pack(ff_from_any(G.gamma));
        t[FK_PGM1] = ff_pack(ff_from_any(G.gamma - 1.0));
        t[FK_PK1] = ff_pack(ff_from_any(G.K + 1.0));
        t[FK_PK3] = ff_pack(ff_from_any(G.K + 3.0));
        t[FK_PIDX] = ff_pack(ff_from_any(G.inv_dx));
        t[FK_PIDY] = ff_pack(ff_from_any(G.inv_dy));
        t[FK_PWEPS] = ff_pack(ff_from_any(G.weno_eps));
        t[FK_PWEPS4] = ff_pack(ff_from_any(4.0 * G.weno_eps));
        t[FK_DT80] = dt * (1.0 / 80.0);
#endif
    }
}

__device__ __forceinline__ void flux_table_tile(double* t, const GridDev& G, double dt)
{
    for (int part = 0; part < 4; ++part) flux_table_part(t, G, dt, part);
}

#ifndef CGKS_OPCOUNT_HOST
// The table for the grid of a CTA's next tile (four warps, between two barriers): `held` is
// the grid that it holds.  dt and `done` are fixed for the launch, so consecutive tiles of one
// grid share it; made anew for each tile it took the first warp, and with it one of the SM's four
// FP64 units, 75 instructions beside the some 800 of a tile's fluxes.
__device__ __forceinline__ void flux_table_grid(double* t, const GridDev& G, int grid, int& held, int& skip)
{
    if (grid == held) return;
    held = grid;
    if (threadIdx.x & 31) return;
    const Ctrl* C = G.ctrl;
    const int done = C->done;
    if (threadIdx.x == 0) skip = done;
    if (!done) flux_table_part(t, G, C->dt, (int)(threadIdx.x >> 5));
}
#endif

// ------------------------------------------------------------------------
// Nonlinear point values along a face (2D): WENO-Z over the line averages of
// neighbouring face rows at the Gauss points eta = +-1/(2 sqrt 3) of the face
// segment (the linear tangential fits turn negative across a discontinuity
// that runs through the faces).
//
// Five means v_{-2..2}: three quadratic candidates on consecutive segments.  At
// a Gauss point each one is v_0 + (eta/2) D_k with
//   D_0 = 3 v_0 - 4 v_-1 + v_-2,  D_1 = v_1 - v_-1,  D_2 = 4 v_1 - v_2 - 3 v_0;
// linear weights (d_lo, 11/18, d_hi) at eta > 0 and (d_hi, 11/18, d_lo) at
// eta < 0, d_lo,hi = 7/36 -+ sqrt(3)/1080, make the combination the quartic
// through the five means; beta_k = 13/12 (second difference)^2 + D_k^2 / 4 is
// the indicator of candidate k over the central segment; Z = |beta_0 - beta_2|;
// alpha_k = d_k (e_k + Z) / e_k with e_k = beta_k + eps, normalised with one
// reciprocal through the common denominator e_0 e_1 e_2.
// Both Gauss points are evaluated at once (eta = -g and +g): the indicators
// and the unnormalised weights are shared, only the linear weights and the
// final normalisation differ.  The weights are homogeneous in (e_k, Z) and in
// (d_k), so the code carries 4 e_k = D_k^2 + 13/3 (second difference)^2 + 4 eps
// (eps4 = 4 eps) and the linear weights divided by 11/18.
// With the differences of the means, D_1 = A1 = v_1 - v_-1, D_0 = A1 - t0, D_2 = A1 - t1
// (t0, t1 the third differences), so a point value is v_0 + (eta/2) (A1 - w_0 t0 - w_2 t1):
// the weights enter through third differences alone, which is what the split form
// (cgks_split.cuh) carries in pairs of FP32 where they are small beside the scale.
struct TangDiffs { double A1, s1, t0, t1; };

__device__ __forceinline__ void tang_diffs(const RegK& r, double vmm, double vm, double v0, double vp, double vpp,
                                           TangDiffs& x)
{
    const double dA = r.sub(vm, vmm), dB = r.sub(v0, vm), dC = r.sub(vp, v0), dD = r.sub(vpp, vp);
    x.s1 = r.sub(dC, dB);
    x.t0 = r.sub(x.s1, r.sub(dB, dA));
    x.t1 = r.sub(r.sub(dD, dC), x.s1);
    x.A1 = r.add(dB, dC);
}

__device__ __forceinline__ void tang_weno5_pair(const RegK& r, double v0, const TangDiffs& x, double eps4,
                                                double& at_minus, double& at_plus)
{
    const double D0 = r.sub(x.A1, x.t0), D2 = r.sub(x.A1, x.t1), s0 = r.sub(x.s1, x.t0), s2 = r.add(x.s1, x.t1);
    const double e0 = fma(D0, D0, fma(r.kmul(FK_T13_3, s0), s0, eps4));
    const double e1 = fma(x.A1, x.A1, fma(r.kmul(FK_T13_3, x.s1), x.s1, eps4));
    const double e2 = fma(D2, D2, fma(r.kmul(FK_T13_3, s2), s2, eps4));
    const double Z = fabs(r.sub(e0, e2));
    // (e_k + Z) times the other two = E + Z times the other two, E = e0 e1 e2
    const double e12 = r.mul(e1, e2), E = r.mul(e0, e12);
    const double P0 = fma(Z, e12, E);
    const double P1 = fma(Z, r.mul(e0, e2), E);
    const double P2 = fma(Z, r.mul(e0, e1), E);
    const double Q0 = r.mul(P0, x.t0), Q2 = r.mul(P2, x.t1);
    const double np = r.kfma(FK_DHI, Q2, r.kmul(FK_DLO, Q0)), dp = r.kfma(FK_DHI, P2, r.kfma(FK_DLO, P0, P1));
    const double nm = r.kfma(FK_DLO, Q2, r.kmul(FK_DHI, Q0)), dm = r.kfma(FK_DLO, P2, r.kfma(FK_DHI, P0, P1));
    const double inv = r.rcp(r.mul(dp, dm));             // one reciprocal for both points
    at_plus = r.kfma(FK_HG, fma(-np, r.mul(dm, inv), x.A1), v0);
    at_minus = r.kfma(FK_MHG, fma(-nm, r.mul(dp, inv), x.A1), v0);
}

// Three means v_{-1..1}: two linear candidates with slopes v_0 - v_-1 and
// v_1 - v_0, linear weights 1/2 at both Gauss points (the quadratic through the
// three means has no eta^2 - 1/12 term there), beta_k = slope_k^2, Z = |beta_0 -
// beta_1|.  The weights do not depend on eta: the nonlinear slope per unit eta
// is num / den; the point value is v_0 + eta * slope.
__device__ __forceinline__ void tang_weno3_parts(const RegK& r, double vm, double v0, double vp, double eps,
                                                 double& num, double& den)
{
    const double dm = r.sub(v0, vm), dp = r.sub(vp, v0);
    const double e0 = fma(dm, dm, eps), e1 = fma(dp, dp, eps);
    const double Z = fabs(r.sub(e0, e1));
    const double e01 = r.mul(e0, e1);
    const double n0 = fma(Z, e1, e01), n1 = fma(Z, e0, e01);          // (e0 + Z) e1, (e1 + Z) e0
    num = fma(n1, dp, r.mul(n0, dm));
    den = r.add(n0, n1);
}

// Twice one row's slope in the split form: false where the correction it carries is not
// below 2^-11 of the scale (its relative error is about 2^-44).
#ifdef CGKS_PAIRS
__device__ __forceinline__ bool tang_weno3_small(const RegK& r, double vm, double v0, double vp, double eps,
                                                 int scale_hi, double& slope2)
{
    const double dm = r.sub(v0, vm), dp = r.sub(vp, v0), A = r.add(dp, dm), s = r.sub(dp, dm);
    if (!(split_scale_ok(scale_hi, eps) && i_max(hi_abs(A), hi_abs(s)) < scale_hi + (1 << 20))) return false;
    const ff c = tang_weno3_split(ff_from(A), ff_from(s), ff_unpack(r.k(FK_PWEPS)));
    const double ch = d_from(c.h);
    slope2 = r.sub(A, r.add(ch, d_from(c.l)));
    return hi_abs(ch) < scale_hi + kTangSlope * (1 << 20);
}
#endif

// twice the slopes of the left and right states' rows, with one reciprocal for both
__device__ __forceinline__ void tang_weno3_slopes(const RegK& r, double lm, double l0, double lp, double rm,
                                                  double r0, double rp, double eps, int scale_hi, double& sl,
                                                  double& sr)
{
#ifdef CGKS_PAIRS
    if (tang_weno3_small(r, lm, l0, lp, eps, scale_hi, sl) && tang_weno3_small(r, rm, r0, rp, eps, scale_hi, sr)) return;
#endif
    double nl, dl, nr, dr;
    tang_weno3_parts(r, lm, l0, lp, eps, nl, dl);
    tang_weno3_parts(r, rm, r0, rp, eps, nr, dr);
    const double inv = r.rcp(r.mul(dl, dr));
    sl = r.mul(r.add(nl, nl), r.mul(dr, inv));
    sr = r.mul(r.add(nr, nr), r.mul(dl, inv));
}

// ------------------------------------------------------------------------
// e^x for x <= 0 by Tang's table-driven method (ACM TOMS 15, 1989): x = (32 m +
// j) ln2/32 + r with |r| <= ln2/64, e^x = 2^m 2^(j/32) e^r, e^r from its Taylor
// polynomial of degree 6 (truncation below 4e-18 relative), 2^(j/32) from the
// table, 2^m added to the exponent field.  Below -700 (e^x < 1e-304) it returns 0.
__device__ __forceinline__ double exp_neg(const RegK& r, double x)
{
#ifdef CGKS_OPCOUNT_HOST
    return cgks_opcount_exp(x);   // one exponential in the host operation count
#endif
#ifndef CGKS_OPCOUNT_HOST
    if ((unsigned)d_hi(x) > 0xc085e000u) return 0.0;      // high word of -700
#endif
    const double t = r.kfma(FK_X32LN2, x, r.k(FK_SHIFT));
    const double n = r.sub(t, r.k(FK_SHIFT));             // round(32 x / ln 2), exactly
    const int ni = (int)(unsigned)__double_as_longlong(t);
    const double q = r.kfma(FK_LN2LO, -n, r.kfma(FK_LN2HI, -n, x));
    double p = fma(r.k(FK_P6), q, r.k(FK_P5));
    p = fma(p, q, r.k(FK_P4));
    p = fma(p, q, r.k(FK_P3));
    p = fma(p, q, r.k(FK_P2));
    p = fma(p, q, r.one);
    p = fma(p, q, r.one);
    const double y = r.mul(r.k(FK_EXP2 + (ni & 31)), p);
    return __longlong_as_double(__double_as_longlong(y) + ((long long)(ni >> 5) << 52));
}

// ------------------------------------------------------------------------
// erfc(t) for t >= 0 from e = exp(-t^2): e * erfcx(t), erfcx from the piecewise
// polynomials of cgks_erfcx_table.h (relative error ~2e-16) instead of a full erfc
// evaluation, since the half-line moments need e anyway.  Past t = 27.3 e underflows to 0;
// a NaN t selects the last piece and stays NaN.  With |z| <= 1/8 the terms from z^3 on are
// below 2^-10 of the value, so Horner's steps down to the z^3 coefficient run in pairs of
// FP32 (their 2^-46 is 2^-56 of the value) and only the last three in FP64.
#ifndef CGKS_OPCOUNT_HOST
constexpr int kErfcxPairs = CGKS_ERFCX_DEG - 2;      // coefficients of z^11 .. z^3
struct ErfcxPairs { float2 c[CGKS_ERFCX_PIECES][kErfcxPairs]; };
constexpr ErfcxPairs make_erfcx_pairs()
{
    ErfcxPairs t{};
    for (int k = 0; k < CGKS_ERFCX_PIECES; ++k)
        for (int m = 0; m < kErfcxPairs; ++m) {
            const double x = cgks_erfcx_coef[k][m];
            t.c[k][m].x = (float)x;
            t.c[k][m].y = (float)(x - (double)(float)x);
        }
    return t;
}
static __device__ const ErfcxPairs kErfcxTab = make_erfcx_pairs();
#endif
__device__ __forceinline__ double erfc_scaled(const RegK& r, double t, double e)
{
#ifdef CGKS_OPCOUNT_HOST
    return cgks_opcount_erfc(t);   // one erfc in the host operation count
#endif
#ifndef CGKS_OPCOUNT_HOST
    // the piece and its centre in FP32 (a t on the border may take either piece)
    const int k = (int)f_mul(4.0f, fminf(f_lead(t), 27.9f));
    const double* c = cgks_erfcx_coef[k];
    const double z = r.sub(t, d_from(f_fma(0.25f, f_int(k), 0.125f)));
    const float2* cp = kErfcxTab.c[k];
    const ff zf = ff_from(z);
    ff w{cp[0].x, cp[0].y};
#pragma unroll
    for (int m = 1; m < kErfcxPairs; ++m) {
        // c + w z, the coefficient the larger addend
        const ff p = ff_mul(w, zf);
        const float2 a = cp[m];
        const float s = f_add(a.x, p.h);
        w = ff{s, f_add(f_sub(p.h, f_sub(s, a.x)), f_add(a.y, p.l))};
    }
    double v = r.add(d_from(w.h), d_from(w.l));
#pragma unroll
    for (int m = kErfcxPairs; m <= CGKS_ERFCX_DEG; ++m) v = fma(v, z, c[m]);
    return r.mul(e, v);
#endif
}

// ------------------------------------------------------------------------
// Sec. 2.1: half-line velocity moments of a Maxwellian per unit density, mean
// (U, V), theta = p/rho = 1/(2 lambda), sqrt(lambda) = sq: m_n = <u^n> over u > 0
// (side 0) or u < 0 (side 1), n = 0..3, and the signed density at u = 0,
//   g = +-e^{-s^2} / sqrt(2 pi theta), s = U sqrt(lambda):
//   m_0 = erfc(-+ s)/2,  m_1 = U m_0 + theta g,  m_{n+1} = U m_n + n theta m_{n-1}.
struct HalfMoments { double m[4], g; };

__device__ __forceinline__ void half_moments(const RegK& r, int side, double U, double theta, double th2, double sq,
                                             HalfMoments& h)
{
    const double s = r.mul(U, sq);
    const double e = exp_neg(r, -r.mul(s, s));
    const double hE = r.kmul(FK_HALF, erfc_scaled(r, fabs(s), e));    // erfc(|s|)/2
    // u > 0: erfc(-s)/2 = 1 - erfc(s)/2 for s >= 0, erfc(|s|)/2 for s < 0; u < 0 mirrored
#ifdef CGKS_OPCOUNT_HOST
    const bool neg = s < 0.0;
#else
    const bool neg = d_hi(s) < 0;
#endif
    h.m[0] = (neg == (side != 0)) ? r.sub(r.one, hE) : hE;
    h.g = r.kmul(side ? FK_C1M : FK_C1P, r.mul(e, sq));
    h.m[1] = fma(U, h.m[0], r.mul(theta, h.g));
    h.m[2] = fma(U, h.m[1], r.mul(theta, h.m[0]));
    h.m[3] = fma(U, h.m[2], r.mul(th2, h.m[1]));
}

// The slope terms of the half-line moments: <psi u (u a_n + v a_t)> (the flux part,
// Th) and <psi (u a_n + v a_t)> (the interface-state part, Wsl), rho a_n and rho a_t
// being the Maxwellian's relative slopes along the normal and the tangent (Sec. 2.1).
// Since rho <phi a_n> is the normal derivative of rho <phi>, they are the
// derivatives of the half-line moments rho <u^2 psi>, rho <u v psi> (and rho <u psi>,
// rho <v psi>) along the conservative slopes, taken through the primitive variables:
//   dm_n = n m_{n-1} dU + n(n-1)/2 m_{n-2} dtheta   (n >= 2),
//   dm_1 = m_0 dU + g/2 dtheta,   dm_0 = g (dU - U/(2 theta) dtheta).
// No micro-slope system is solved and moments to order 4 suffice (the form with
// the micro-slope coefficients needs order 6 and half again the operations).  (R, A, B, C) = (rho', rho U', rho V',
// rho theta').  Ar supplies the arithmetic (FP64 or split).
template <class T> struct PrimSlope { T R, A, B, C; };

template <class Ar, class T = typename Ar::T>
__device__ __forceinline__ PrimSlope<T> prim_slope(const Ar& q, T U, T V, T hq2, T theta, const T b[4])
{
    PrimSlope<T> s;
    s.R = b[0];
    s.A = q.nmad(U, b[0], b[1]);
    s.B = q.nmad(V, b[0], b[2]);
    // e' = E' - (rho q^2/2)', e = rho theta / (gamma - 1)
    const T de = q.nmad(hq2, b[0], q.nmad(V, s.B, q.nmad(U, s.A, b[3])));
    s.C = q.nmad(theta, b[0], q.mul(q.gm1(), de));
    return s;
}

template <class Ar, class T = typename Ar::T>
__device__ __forceinline__ void slope_moments(const Ar& q, bool ne, T U, T V, T theta, T itheta, const T m[4], T g,
                                              const T bn[4], const T bt[4], T Th[4], T Wsl[4])
{
    const T VV = q.mul(V, V), hq2 = q.half(q.mad(U, U, VV));
    const PrimSlope<T> X = prim_slope(q, U, V, hq2, theta, bn), Y = prim_slope(q, U, V, hq2, theta, bt);
    const T V2 = q.dbl(V), qt = q.mad(q.K1(), theta, VV), w = q.mad(q.K3(), theta, VV), v2 = q.add(VV, theta);
    const T m4 = q.mad(U, m[3], q.mul(q.tri(theta), m[2]));
    // y_n = (rho m_n)' along the normal (x) and the tangent (y)
    auto y1 = [&](const PrimSlope<T>& s) { return q.mad(s.R, m[1], q.mad(s.A, m[0], q.mul(q.half(s.C), g))); };
    auto y2 = [&](const PrimSlope<T>& s) { return q.mad(s.R, m[2], q.mad(q.dbl(s.A), m[1], q.mul(s.C, m[0]))); };
    auto y3 = [&](const PrimSlope<T>& s) { return q.mad(s.R, m[3], q.tri(q.mad(s.A, m[2], q.mul(s.C, m[1])))); };
    const T x2 = y2(X), x3 = y3(X), a1 = y1(Y), a2 = y2(Y), a3 = y3(Y);
    const T x4 = q.mad(X.R, m4, q.dbl(q.mad(q.dbl(X.A), m[3], q.mul(q.tri(X.C), m[2]))));
    const T xv = q.mad(V2, X.B, q.mul(q.K1(), X.C));                            // (V^2 + (K+1) theta)' rho
    const T yv = q.mad(V, q.mad(V2, Y.B, q.mul(q.K3(), Y.C)), q.mul(Y.B, w));   // (V w)' rho
    const T yt = q.mad(V2, Y.B, Y.C);                                           // (V^2 + theta)' rho
    Th[0] = q.add(x2, q.mad(V, a1, q.mul(Y.B, m[1])));
    Th[1] = q.add(x3, q.mad(V, a2, q.mul(Y.B, m[2])));
    Th[2] = q.mad(V, x2, q.mad(X.B, m[2], q.mad(v2, a1, q.mul(m[1], yt))));
    Th[3] = q.half(q.add(q.mad(m[2], xv, q.mad(qt, x2, x4)),
                         q.mad(m[1], yv, q.mad(Y.B, m[3], q.mul(V, q.mad(w, a1, a3))))));
    CGKS_BRANCH(ne)
    {
        const T x1 = y1(X);
        const T a0 = q.mad(Y.R, m[0], q.mul(g, q.nmad(q.half(q.mul(U, itheta)), Y.C, Y.A)));
        Wsl[0] = q.add(x1, q.mad(V, a0, q.mul(Y.B, m[0])));
        Wsl[1] = q.add(x2, q.mad(V, a1, q.mul(Y.B, m[1])));
        Wsl[2] = q.mad(V, x1, q.mad(X.B, m[1], q.mad(v2, a0, q.mul(m[0], yt))));
        Wsl[3] = q.half(q.add(q.mad(m[1], xv, q.mad(qt, x1, x3)),
                              q.mad(m[0], yv, q.mad(Y.B, m[2], q.mul(V, q.mad(w, a0, a2))))));
    }
}

// FP64 arithmetic of slope_moments in the register forms
struct Ar64 {
    using T = double;
    const RegK& r;
    __device__ __forceinline__ double add(double a, double b) const { return r.add(a, b); }
    __device__ __forceinline__ double sub(double a, double b) const { return r.sub(a, b); }
    __device__ __forceinline__ double mul(double a, double b) const { return r.mul(a, b); }
    __device__ __forceinline__ double mad(double a, double b, double c) const { return fma(a, b, c); }
    __device__ __forceinline__ double nmad(double a, double b, double c) const { return fma(-a, b, c); }
    __device__ __forceinline__ double half(double a) const { return r.kmul(FK_HALF, a); }
    __device__ __forceinline__ double dbl(double a) const { return r.add(a, a); }
    __device__ __forceinline__ double tri(double a) const { return r.kmul(FK_3, a); }
    __device__ __forceinline__ double gm1() const { return r.k(FK_GM1); }
    __device__ __forceinline__ double K1() const { return r.k(FK_K1); }
    __device__ __forceinline__ double K3() const { return r.k(FK_K3); }
};

#ifdef CGKS_PAIRS
// the same in pairs of FP32 (cgks_split.cuh), not renormalised: the results' weights leave room
struct ArSplit {
    using T = ff;
    ff g1, k1, k3;
    __device__ __forceinline__ ff add(ff a, ff b) const { return ff_addp(a, b); }
    __device__ __forceinline__ ff sub(ff a, ff b) const { return ff_addp(a, ff_neg(b)); }
    __device__ __forceinline__ ff mul(ff a, ff b) const { return ff_mul(a, b); }
    __device__ __forceinline__ ff mad(ff a, ff b, ff c) const { return ff_addp(ff_mul(a, b), c); }
    __device__ __forceinline__ ff nmad(ff a, ff b, ff c) const { return ff_addp(c, ff_neg(ff_mul(a, b))); }
    __device__ __forceinline__ ff half(ff a) const { return ff_scale(0.5f, a); }
    __device__ __forceinline__ ff dbl(ff a) const { return ff_scale(2.0f, a); }
    __device__ __forceinline__ ff tri(ff a) const { return ff_mulf(3.0f, a); }
    __device__ __forceinline__ ff gm1() const { return g1; }
    __device__ __forceinline__ ff K1() const { return k1; }
    __device__ __forceinline__ ff K3() const { return k3; }
};
#endif

// ------------------------------------------------------------------------
// Euler time derivatives by Cauchy-Kowalevski in primitive variables.
// Inputs: conservative W and its x (normal), y (tangential) derivatives up to
// second order, 1/rho, the velocity, the pressure p and the internal energy per
// volume e = p / (gamma - 1).  The pressure's derivatives are carried as those
// of e (p_x = (gamma - 1) e_x, ...), which are differences of the energy's and
// the kinetic energy's.  Outputs conservative W_t, W_tt and the flux time
// derivative F_t of the normal Euler flux.
// TNS is rho <(a_n u + a_t v + A) u psi> of the equilibrium state, i.e. the
// Chapman-Enskog Navier-Stokes flux of the BGK model per unit collision time
// (mu = tau p, bulk part 2/(K+2), heat conduction (K+4)/2 tau p grad(p/rho)).
struct EulerTD { double Wt[4], Wtt[4], Ft[4], F[4], TNS[4]; };

// the state, its primitive first derivatives and first time derivatives
template <class T> struct EulerFirst {
    T rho, U, V, ir, gir, hq2, e;               // gir = (gamma - 1) / rho, hq2 = (U^2 + V^2)/2
    T rx, ry, Ux, Uy, Vx, Vy, ex, ey, Dv;       // Dv = U_x + V_y
    T rt, Ut, Vt, et, uut;                      // uut = U U_t + V V_t
};

// W_tt from the first-order quantities and the conservative second derivatives
template <class Ar, class T = typename Ar::T>
__device__ __forceinline__ void euler_second(const Ar& q, const EulerFirst<T>& f, T gamma, const T Wxx[4],
                                             const T Wxy[4], const T Wyy[4], T Wtt[4])
{
    const T rxx = Wxx[0], rxy = Wxy[0], ryy = Wyy[0], rx2 = q.dbl(f.rx), ry2 = q.dbl(f.ry);
    // primitive second derivatives; KE = rho q^2 / 2: KE_xx = rho |u_x|^2 + u . m_xx - rho_xx q^2/2,
    // KE_xy = rho u_x . u_y + u . m_xy - rho_xy q^2/2
    const T Uxx = q.mul(q.nmad(f.U, rxx, q.nmad(f.Ux, rx2, Wxx[1])), f.ir);
    const T Uxy = q.mul(q.nmad(f.U, rxy, q.nmad(f.Uy, f.rx, q.nmad(f.Ux, f.ry, Wxy[1]))), f.ir);
    const T Uyy = q.mul(q.nmad(f.U, ryy, q.nmad(f.Uy, ry2, Wyy[1])), f.ir);
    const T Vxx = q.mul(q.nmad(f.V, rxx, q.nmad(f.Vx, rx2, Wxx[2])), f.ir);
    const T Vxy = q.mul(q.nmad(f.V, rxy, q.nmad(f.Vy, f.rx, q.nmad(f.Vx, f.ry, Wxy[2]))), f.ir);
    const T Vyy = q.mul(q.nmad(f.V, ryy, q.nmad(f.Vy, ry2, Wyy[2])), f.ir);
    auto ke = [&](const T W2[4], T a, T b, T c, T d) {   // rho (a b + c d) + u . m'' - rho'' q^2/2
        return q.nmad(f.hq2, W2[0], q.mad(f.V, W2[2], q.mad(f.U, W2[1], q.mul(f.rho, q.mad(a, b, q.mul(c, d))))));
    };
    const T exx = q.sub(Wxx[3], ke(Wxx, f.Ux, f.Ux, f.Vx, f.Vx)), exy = q.sub(Wxy[3], ke(Wxy, f.Ux, f.Uy, f.Vx, f.Vy)),
            eyy = q.sub(Wyy[3], ke(Wyy, f.Uy, f.Uy, f.Vy, f.Vy));
    // mixed derivatives d/dx, d/dy of the (negated) first time derivatives
    const T Dx = q.add(Uxx, Vxy), Dy = q.add(Uxy, Vyy);
    const T nrxt = q.mad(f.rho, Dx, q.mad(f.rx, f.Dv, q.mad(f.V, rxy, q.mad(f.Vx, f.ry, q.mad(f.U, rxx, q.mul(f.Ux, f.rx))))));
    const T nryt = q.mad(f.rho, Dy, q.mad(f.ry, f.Dv, q.mad(f.V, ryy, q.mad(f.Vy, f.ry, q.mad(f.U, rxy, q.mul(f.Uy, f.rx))))));
    const T nUxt = q.mad(q.nmad(q.mul(f.ex, f.rx), f.ir, exx), f.gir, q.mad(f.V, Uxy, q.mad(f.Vx, f.Uy, q.mad(f.U, Uxx, q.mul(f.Ux, f.Ux)))));
    const T nVyt = q.mad(q.nmad(q.mul(f.ey, f.ry), f.ir, eyy), f.gir, q.mad(f.V, Vyy, q.mad(f.Vy, f.Vy, q.mad(f.U, Vxy, q.mul(f.Uy, f.Vx)))));
    const T nUyt = q.mad(q.nmad(q.mul(f.ex, f.ry), f.ir, exy), f.gir, q.mad(f.V, Uyy, q.mad(f.Vy, f.Uy, q.mad(f.U, Uxy, q.mul(f.Uy, f.Ux)))));
    const T nVxt = q.mad(q.nmad(q.mul(f.ey, f.rx), f.ir, exy), f.gir, q.mad(f.V, Vxy, q.mad(f.Vx, f.Vy, q.mad(f.U, Vxx, q.mul(f.Ux, f.Vx)))));
    const T next = q.mad(gamma, q.mad(f.e, Dx, q.mul(f.ex, f.Dv)), q.mad(f.V, exy, q.mad(f.Vx, f.ey, q.mad(f.U, exx, q.mul(f.Ux, f.ex)))));
    const T neyt = q.mad(gamma, q.mad(f.e, Dy, q.mul(f.ey, f.Dv)), q.mad(f.V, eyy, q.mad(f.Vy, f.ey, q.mad(f.U, exy, q.mul(f.Uy, f.ex)))));
    // second time derivatives (the mixed ones enter negated)
    const T nDt = q.add(nUxt, nVyt);
    const T rtt = q.mad(f.rho, nDt, q.nmad(f.rt, f.Dv, q.mad(f.V, nryt, q.nmad(f.Vt, f.ry, q.nmad(f.Ut, f.rx, q.mul(f.U, nrxt))))));
    const T Utt = q.mad(q.mad(q.mul(f.ex, f.rt), f.ir, next), f.gir, q.mad(f.V, nUyt, q.nmad(f.Vt, f.Uy, q.nmad(f.Ut, f.Ux, q.mul(f.U, nUxt)))));
    const T Vtt = q.mad(q.mad(q.mul(f.ey, f.rt), f.ir, neyt), f.gir, q.mad(f.V, nVyt, q.nmad(f.Vt, f.Vy, q.nmad(f.Ut, f.Vx, q.mul(f.U, nVxt)))));
    const T ett = q.mad(gamma, q.nmad(f.et, f.Dv, q.mul(f.e, nDt)), q.mad(f.V, neyt, q.nmad(f.Vt, f.ey, q.nmad(f.Ut, f.ex, q.mul(f.U, next)))));
    // back to conservative variables (E = e + KE)
    const T rt2 = q.dbl(f.rt);
    Wtt[0] = rtt;
    Wtt[1] = q.mad(f.rho, Utt, q.mad(rt2, f.Ut, q.mul(rtt, f.U)));
    Wtt[2] = q.mad(f.rho, Vtt, q.mad(rt2, f.Vt, q.mul(rtt, f.V)));
    Wtt[3] = q.mad(f.rho, q.mad(f.V, Vtt, q.mad(f.Vt, f.Vt, q.mad(f.U, Utt, q.mul(f.Ut, f.Ut)))),
                   q.mad(rt2, f.uut, q.mad(rtt, f.hq2, ett)));
}

#ifdef CGKS_PAIRS
// W_tt in pairs of FP32: it enters the interface state as dt^2/8 W_tt and dt^2/6 W_tt,
// second order in the changes over a time step.  False (nothing written) unless
//   (a dt)^2 (sum of second derivatives + squared sum of first ones) < 2^-6
// of the variables' scales rho, rho a, rho a^2 (a = |U| + |V| + 2 sqrt(theta)), so that
// the pairs' rounding of W_tt (about 2^-45 of its largest term) stays below the last bit
// of the state, and unless the units let the pairs hold all terms (wtt_range_ok).  A derivative
// that is out of a float's range itself, infinite or NaN is so in the sum, which then is not
// below the bound.  Nor on a rough segment (its bound hardly ever holds, and its slice holds the
// second derivatives' parts in FP64).
template <class Src>
__device__ __forceinline__ bool euler_second_split(const RegK& r, const Src& src, const EulerFirst<double>& f,
                                                   double E, double Wtt[4])
{
    // (with the size below, not as a branch of its own: the conversions wait for no FP64 result so)
    const bool in = wtt_range_ok(hi_log(f.rho), hi_log(E), hi_log(r.k(FK_DT))) & (src.rough() == 0);
    EulerFirst<ff> g;
    g.rho = ff_from(f.rho); g.U = ff_from(f.U); g.V = ff_from(f.V); g.ir = ff_from(f.ir); g.gir = ff_from(f.gir);
    g.hq2 = ff_from(f.hq2); g.e = ff_from(f.e);
    g.rx = ff_from_any(f.rx); g.ry = ff_from_any(f.ry); g.Ux = ff_from_any(f.Ux); g.Uy = ff_from_any(f.Uy);
    g.Vx = ff_from_any(f.Vx); g.Vy = ff_from_any(f.Vy); g.ex = ff_from_any(f.ex); g.ey = ff_from_any(f.ey); g.Dv = ff_from(f.Dv);
    g.rt = ff_from(f.rt); g.Ut = ff_from(f.Ut); g.Vt = ff_from(f.Vt); g.et = ff_from(f.et); g.uut = ff_from(f.uut);
    ff xx[4], xy[4], yy[4], o[4];
    src.eq_second_split(xx, xy, yy);
    {
        // theta = (gamma - 1) e / rho; e * gir
        const float th = f_mul(g.e.h, g.gir.h), a = f_add(f_add(fabsf(g.U.h), fabsf(g.V.h)), f_mul(2.0f, f_mul(th, f_rsqrt(th))));
        const float ia = f_rcp(a), ad = f_mul(a, f_lead(r.k(FK_DT))), ir = g.ir.h, ir1 = f_mul(ir, ia), ir2 = f_mul(ir1, ia);
        // sums, not maxima: a NaN has to fail the comparison (a maximum drops it)
        auto m3 = [](ff a, ff b, ff c) { return f_add(f_add(fabsf(a.h), fabsf(b.h)), fabsf(c.h)); };
        const float s2 = f_fma(m3(xx[3], xy[3], yy[3]), ir2,
                               f_fma(f_add(m3(xx[1], xy[1], yy[1]), m3(xx[2], xy[2], yy[2])), ir1, f_mul(m3(xx[0], xy[0], yy[0]), ir)));
        const float s1 = f_fma(f_add(fabsf(g.ex.h), fabsf(g.ey.h)), ir2,
                               f_fma(f_add(m3(g.Ux, g.Uy, g.Vx), fabsf(g.Vy.h)), ia, f_mul(f_add(fabsf(g.rx.h), fabsf(g.ry.h)), ir)));
        if (!(in & (f_mul(f_mul(ad, ad), f_fma(s1, s1, s2)) < 1.0f / 64.0f))) return false;
    }
    euler_second(ArSplit{}, g, ff_unpack(r.k(FK_PGAMMA)), xx, xy, yy, o);
#pragma unroll
    for (int k = 0; k < 4; ++k) Wtt[k] = r.add(d_from(o[k].h), d_from(o[k].l));
    return true;
}
#endif

template <class Src>
__device__ __forceinline__ void euler_time_derivs(const RegK& r, const Src& src, const double W[4], double ir, double U,
                                                  double V, double p, double e, EulerTD& o)
{
    double Wx[4], Wy[4];
    src.eq_first(Wx, Wy);
    EulerFirst<double> f;
    f.rho = W[0]; f.U = U; f.V = V; f.ir = ir; f.e = e;
    const double rho = W[0], m = W[1], E = W[3];
    // primitive first derivatives
    f.rx = Wx[0]; f.ry = Wy[0];
    f.Ux = r.mul(fma(-U, f.rx, Wx[1]), ir); f.Uy = r.mul(fma(-U, f.ry, Wy[1]), ir);
    f.Vx = r.mul(fma(-V, f.rx, Wx[2]), ir); f.Vy = r.mul(fma(-V, f.ry, Wy[2]), ir);
    // kinetic energy KE = rho q^2 / 2: KE_x = u . m_x - rho_x q^2/2
    f.hq2 = r.kmul(FK_HALF, fma(U, U, r.mul(V, V)));
    const double KEx = fma(-f.hq2, f.rx, fma(V, Wx[2], r.mul(U, Wx[1])));
    const double KEy = fma(-f.hq2, f.ry, fma(V, Wy[2], r.mul(U, Wy[1])));
    f.ex = r.sub(Wx[3], KEx); f.ey = r.sub(Wy[3], KEy);
    // first time derivatives (p_x / rho = e_x gir)
    const double gamma = r.k(FK_GAMMA);
    f.gir = r.mul(r.k(FK_GM1), ir);
    f.Dv = r.add(f.Ux, f.Vy);
    f.rt = -fma(rho, f.Dv, fma(V, f.ry, r.mul(U, f.rx)));
    f.Ut = -fma(f.ex, f.gir, fma(V, f.Uy, r.mul(U, f.Ux)));
    f.Vt = -fma(f.ey, f.gir, fma(V, f.Vy, r.mul(U, f.Vx)));
    f.et = -fma(r.mul(gamma, e), f.Dv, fma(V, f.ey, r.mul(U, f.ex)));
    f.uut = fma(V, f.Vt, r.mul(U, f.Ut));
    o.Wt[0] = f.rt;
    o.Wt[1] = fma(rho, f.Ut, r.mul(f.rt, U));
    o.Wt[2] = fma(rho, f.Vt, r.mul(f.rt, V));
    o.Wt[3] = fma(rho, f.uut, fma(f.rt, f.hq2, f.et));
    // normal Euler flux and its time derivative
    const double Ep = r.add(E, p);
    const double pt = r.mul(r.k(FK_GM1), f.et);
    o.F[0] = m;
    o.F[1] = fma(m, U, p);
    o.F[2] = r.mul(m, V);
    o.F[3] = r.mul(U, Ep);
    const double mt = o.Wt[1];
    o.Ft[0] = mt;
    o.Ft[1] = fma(m, f.Ut, fma(mt, U, pt));
    o.Ft[2] = fma(m, f.Vt, r.mul(mt, V));
    o.Ft[3] = fma(U, r.add(o.Wt[3], pt), r.mul(f.Ut, Ep));
    // BGK Navier-Stokes flux per unit tau in the face-normal direction
    const double sxx = r.mul(p, fma(-r.k(FK_K2INV2), f.Dv, r.add(f.Ux, f.Ux)));
    const double sxy = r.mul(p, r.add(f.Uy, f.Vx));
    const double thx = r.mul(fma(-r.mul(e, ir), f.rx, f.ex), f.gir);      // d/dx (p / rho)
    o.TNS[0] = 0.0;
    o.TNS[1] = sxx;
    o.TNS[2] = sxy;
    o.TNS[3] = fma(r.mul(r.k(FK_KHEAT), p), thx, fma(V, sxy, r.mul(U, sxx)));
#ifdef CGKS_PAIRS
    if (euler_second_split(r, src, f, E, o.Wtt)) return;
#endif
    double Wxx[4], Wxy[4], Wyy[4];
    src.eq_second(Wxx, Wxy, Wyy);
    euler_second(Ar64{r}, f, gamma, Wxx, Wxy, Wyy, o.Wtt);
}

#ifdef CGKS_PAIRS
// The slope moments in pairs of FP32.  They enter a face's flux through the weights
// of order tau^2/dt and its state through h dt, a small correction where the
// collision time is: false (nothing to be used) unless every weighted term is below
// 2^-7 of the side's half-line flux of the same kind (a momentum's scale is the
// normal momentum flux), so that the pairs' rounding stays below that flux's last
// bit.  Only where the units let the pairs hold the terms (slopes_range_ok).  wth, wsl:
// the weights' magnitudes.
template <class Src>
__device__ __forceinline__ bool slope_moments_split(const RegK& r, const Src& src, int side, bool ne, double rho,
                                                    double U, double V, double th, double sq, const HalfMoments& h,
                                                    float wth, float wsl, ff Th[4], ff Wsl[4])
{
    const ff K1 = ff_unpack(r.k(FK_PK1));
    const ArSplit q{ff_unpack(r.k(FK_PGM1)), K1, ff_unpack(r.k(FK_PK3))};
    ff m[4], n[4], s[4], T[4], S[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = ff_from(h.m[k]);
    src.ne_slopes_split(side, n, s);
    const ff fV = ff_from(V), fth = ff_from(th);
    const ff isq = ff_from(sq);
    slope_moments(q, ne, ff_from(U), fV, fth, ff_scale(2.0f, ff_mul(isq, isq)), m, ff_from(h.g), n, s, T, S);
    const float fr = f_lead(rho), qt = f_fma(fV.h, fV.h, f_mul(K1.h, fth.h)), f0 = f_mul(fr, fabsf(m[1].h)),
                f1 = f_mul(fr, m[2].h), f3 = f_mul(f_mul(0.5f, fr), f_fma(fabsf(m[1].h), qt, fabsf(m[3].h)));
    const float w = f_mul(128.0f, wth), v = f_mul(128.0f, wsl);
    // sums, not maxima: a NaN has to fail the comparisons (a maximum drops it)
    bool ok = f0 > 1e-15f && f1 > 1e-15f && f3 > 1e-15f && f_mul(w, fabsf(T[0].h)) < f0 &&
              f_mul(w, f_add(fabsf(T[1].h), fabsf(T[2].h))) < f1 && f_mul(w, fabsf(T[3].h)) < f3;
    if (ne)
        ok = ok && f_mul(v, fabsf(S[0].h)) < fr && f_mul(v, f_add(fabsf(S[1].h), fabsf(S[2].h))) < f0 &&
             f_mul(v, fabsf(S[3].h)) < f_mul(f_mul(0.5f, fr), f_fma(m[0].h, qt, m[2].h));
#pragma unroll
    for (int k = 0; k < 4; ++k) Th[k] = ff_add(Th[k], T[k]);
    if (ne)
#pragma unroll
        for (int k = 0; k < 4; ++k) Wsl[k] = ff_add(Wsl[k], S[k]);
    return ok;
}
#endif

// the sums of both sides' half-line terms: fluxes Fh = <u psi>, states Wh = <psi> (where
// the interface state needs them) and their slope terms Th, Wsl
struct HalfSums { double Fh[4], Th[4], Wh[4], Wsl[4]; };

// Side by side in a rolled loop: one copy of its instructions for both.  The slope terms
// in pairs of FP32 first; where a side's do not qualify, the loop runs again with them in
// FP64.
template <class Src>
__device__ __forceinline__ void half_sums(const RegK& r, const Src& src, const double Wl[4], const double Wr[4],
                                          double Ul, double Vl, double thl, double Ur, double Vr, double thr,
                                          bool need_ne, float wth, float wsl, HalfSums& o)
{
#ifndef CGKS_PAIRS
    bool split = false;
#else
    const int rl = hi_log(Wl[0]), rr = hi_log(Wr[0]), tl = hi_log(thl), tr = hi_log(thr);
    const int speed = i_max(i_max(hi_log(Ul), hi_log(Vl)), i_max(hi_log(Ur), hi_log(Vr)));
    bool split = slopes_range_ok(i_min(rl, rr), i_max(rl, rr), i_min(tl, tr), i_max(tl, tr), speed, hi_log(src.iht),
                                 f_log(wth > wsl ? wth : wsl));
    ff Ts[4], Ss[4];
#endif
    for (;;) {
        bool ok = true;
#pragma unroll
        for (int k = 0; k < 4; ++k) { o.Fh[k] = 0.0; o.Th[k] = 0.0; o.Wh[k] = 0.0; o.Wsl[k] = 0.0; }
#ifdef CGKS_PAIRS
#pragma unroll
        for (int k = 0; k < 4; ++k) { Ts[k] = ff{0.0f, 0.0f}; Ss[k] = ff{0.0f, 0.0f}; }
#endif
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            const double rho = side ? Wr[0] : Wl[0], U = side ? Ur : Ul, V = side ? Vr : Vl, th = side ? thr : thl;
            HalfMoments h;
            const double th2 = r.add(th, th);
            const double sq = r.rsq(th2);                     // sqrt(lambda) = 1/sqrt(2 theta)
            half_moments(r, side, U, th, th2, sq, h);
            const double qt = fma(V, V, r.mul(r.k(FK_K1), th));       // <v^2 + xi^2>
            o.Fh[0] = fma(rho, h.m[1], o.Fh[0]);
            o.Fh[1] = fma(rho, h.m[2], o.Fh[1]);
            o.Fh[2] = fma(rho, r.mul(V, h.m[1]), o.Fh[2]);
            o.Fh[3] = fma(rho, r.kmul(FK_HALF, fma(h.m[1], qt, h.m[3])), o.Fh[3]);
            CGKS_BRANCH(need_ne)
            {
                o.Wh[0] = fma(rho, h.m[0], o.Wh[0]);
                o.Wh[1] = fma(rho, h.m[1], o.Wh[1]);
                o.Wh[2] = fma(rho, r.mul(V, h.m[0]), o.Wh[2]);
                o.Wh[3] = fma(rho, r.kmul(FK_HALF, fma(h.m[0], qt, h.m[2])), o.Wh[3]);
            }
#ifdef CGKS_PAIRS
            if (split) {
                ok &= slope_moments_split(r, src, side, need_ne, rho, U, V, th, sq, h, wth, wsl, Ts, Ss);
                continue;
            }
#endif
            double bn[4], bt[4], t[4], ws[4];
            src.ne_slopes(side, bn, bt);
            const double ith = r.mul(r.add(sq, sq), sq);     // 1/theta = 2 lambda
            slope_moments(Ar64{r}, need_ne, U, V, th, ith, h.m, h.g, bn, bt, t, ws);
#pragma unroll
            for (int k = 0; k < 4; ++k) o.Th[k] = r.add(o.Th[k], t[k]);
            CGKS_BRANCH(need_ne)
#pragma unroll
            for (int k = 0; k < 4; ++k) o.Wsl[k] = r.add(o.Wsl[k], ws[k]);
        }
        if (!split) return;
#ifdef CGKS_PAIRS
        if (ok) {
#pragma unroll
            for (int k = 0; k < 4; ++k) o.Th[k] = r.add(d_from(Ts[k].h), d_from(Ts[k].l));
            CGKS_BRANCH(need_ne)
#pragma unroll
            for (int k = 0; k < 4; ++k) o.Wsl[k] = r.add(d_from(Ss[k].h), d_from(Ss[k].l));
            return;
        }
#endif
        split = false;
    }
}

#ifndef CGKS_OPCOUNT_HOST
// dt < 80 tau, from the high words (in any unit of time, off the FP64 unit); true for a NaN
__device__ __forceinline__ bool nonequilibrium(const RegK& r, double tau) { return d_hi(r.k(FK_DT80)) < d_hi(tau); }
#endif

// ------------------------------------------------------------------------
// One interface quadrature point in the face frame (Sec. 2.1-2.2).
// Inputs of one Gauss point are pulled from the caller's loader when they are
// consumed, so that the 48 reconstructed quantities are never live at once:
//   src.eq_value(W0)                          equilibrium state
//   src.eq_first(W0n, W0t)                    its derivatives (face frame) ...
//   src.eq_second(W0nn, W0nt, W0tt)           ... and second derivatives
//   src.ne_value(side, W)                     left (0) / right (1) state
//   src.ne_slopes(side, Wn, Wt)               its normal and tangential derivatives
// The caller's table holds the grid's gamma, K and the time step.
template <int STAGE, class Src>
__device__ __forceinline__ bool gks_point(const RegK& r, const Src& src, double Fb[4], double Ft[4], double Wm[4],
                                          double Wb[4], double Wtt[4])
{
    // equilibrium state g0
    double W0[4];
    src.eq_value(W0);
    const double ir0 = r.rcp3(W0[0]);
    const double U0 = r.mul(W0[1], ir0), V0 = r.mul(W0[2], ir0);
    const double e0 = r.kfma(FK_MHALF, fma(W0[2], V0, r.mul(W0[1], U0)), W0[3]);   // p0 / (gamma - 1)
    const double p0 = r.mul(r.k(FK_GM1), e0);
    // non-equilibrium states
    double Wl[4], Wr[4];
    src.ne_value(0, Wl);
    src.ne_value(1, Wr);
    const double irl = r.rcp3(Wl[0]);
    const double Ul = r.mul(Wl[1], irl), Vl = r.mul(Wl[2], irl);
    const double pl = r.mul(r.k(FK_GM1), r.kfma(FK_MHALF, fma(Wl[2], Vl, r.mul(Wl[1], Ul)), Wl[3]));
    const double irr = r.rcp3(Wr[0]);
    const double Ur = r.mul(Wr[1], irr), Vr = r.mul(Wr[2], irr);
    const double pr = r.mul(r.k(FK_GM1), r.kfma(FK_MHALF, fma(Wr[2], Vr, r.mul(Wr[1], Ur)), Wr[3]));
    const bool ok = positive(W0[0]) && positive(p0) && positive(Wl[0]) && positive(pl) && positive(Wr[0]) && positive(pr);
    const double thl = r.mul(pl, irl), thr = r.mul(pr, irr);

    // Sec. 4: collision time with pressure-jump enhancement; viscous flow: mu/p
    // with p the equilibrium pressure at the point
    const double mu = r.k(FK_MU), dt = r.k(FK_DT);
    double tau0 = r.k(FK_EPSDT);
    CGKS_BRANCH(positive(mu)) tau0 = r.mul(mu, r.rcp3(p0));
    const double tau = fma(r.k(FK_CTAUDT), fabs(r.mul(r.sub(pl, pr), r.rcp3(r.add(pl, pr)))), tau0);
    // h = exp(-dt / (2 tau)) weights the non-equilibrium part of the interface state.
    // For dt > 80 tau, h < 4e-18: then 1 - h and 3 - h round to 1 and 3, and the
    // remaining h-terms change the window coefficients by under 2e-14 of a term
    // that is itself O(tau^2), so h is taken as 0 without evaluating the exponential.
    // Below h = 1e-20 that part is under 1e-20 of the state it is added to: far below one
    // ulp, so its velocity moments are not evaluated (the flux terms, weighted by O(tau),
    // are).
    double h = 0.0;
#ifdef CGKS_OPCOUNT_HOST
    if (tau > 0.0 && dt < 80.0 * tau) h = exp_neg(r, r.mul(r.k(FK_MHDT), r.rcp3(tau)));
    const bool need_ne = (STAGE == 1) && (h >= 1e-20);
#else
    CGKS_BRANCH(nonequilibrium(r, tau)) h = exp_neg(r, r.mul(r.k(FK_MHDT), r.rcp3(tau)));
    const bool need_ne = (STAGE == 1) && d_hi(h) >= 0x3bc79ca1;       // high word of 1e-20
#endif
#ifdef CGKS_PAIRS
    // bounds of the slope terms' weights (FP32, for the choice of their arithmetic): beside F
    // |b4| and |f4| dt/4 below are at most 4 tau (tau + h dt) / dt, beside W it is h dt
    const float ft = f_lead(tau), wsl = f_mul(f_lead(dt), f_lead(h));
    const float wth = f_mul(f_mul(4.0f, ft), f_mul(f_add(ft, wsl), f_lead(r.k(FK_IDT))));
#else
    const float wth = 0.0f, wsl = 0.0f;
#endif

    HalfSums o;
    half_sums(r, src, Wl, Wr, Ul, Vl, thl, Ur, Vr, thr, need_ne, wth, wsl, o);

    // Euler derivatives of the equilibrium state (W_t, W_tt, F, F_t), evaluated after the
    // half-line moments so that the two sets of intermediates are never live together
    EulerTD e;
    euler_time_derivs(r, src, W0, ir0, U0, V0, p0, e0, e);

    // tau-terms of g0: rho <(a_n u + a_t v) u psi> = TNS - F_t (the time part is the Euler F_t)
    // window coefficients over [0, dt]
    const double idt = r.k(FK_IDT);
    const double omh = r.sub(r.one, h);
    const double ta = r.mul(tau, omh);                       // tau (1 - h)
    const double q4 = r.mul(ta, r.k(FK_4IDT2));              // 4 tau (1 - h) / dt^2
    const double g = r.mul(q4, omh);
    const double dh = r.mul(dt, h);
    const double f4 = r.mul(q4, r.sub(dh, ta));
    const double tat = r.mul(ta, r.sub(r.k(FK_3), h));       // tau (1 - h) (3 - h)
    const double a = r.mul(tat, idt);
    const double b4 = r.mul(r.mul(tau, fma(-dh, r.sub(r.k(FK_2), h), tat)), idt);
    for (int k = 0; k < 4; ++k) {
        const double dTh = (k == 0) ? -r.add(e.Ft[0], o.Th[0]) : r.sub(r.sub(e.TNS[k], e.Ft[k]), o.Th[k]);
        const double dFh = r.sub(o.Fh[k], e.F[k]);
        Ft[k] = fma(f4, dTh, fma(-g, dFh, e.Ft[k]));
        if (STAGE == 1) Fb[k] = fma(b4, dTh, (k == 0) ? fma(a, dFh, e.F[0]) : fma(-tau, e.TNS[k], fma(a, dFh, e.F[k])));
    }
    if (STAGE == 1) {
        // interface state W(t) = W0 + t W_t + t^2/2 W_tt + e^{-t/tau} [W_ne(t) - W0 - t W_t]
        const double hdt = r.k(FK_HDT);
        for (int k = 0; k < 4; ++k) {
            Wm[k] = fma(r.k(FK_C8), e.Wtt[k], fma(hdt, e.Wt[k], W0[k]));
            Wb[k] = fma(r.k(FK_C6), e.Wtt[k], fma(dt, e.Wt[k], W0[k]));
        }
        CGKS_BRANCH(need_ne)
        {
            const double h2 = r.mul(h, h);
            for (int k = 0; k < 4; ++k) {
                Wm[k] = fma(h, fma(-hdt, e.Wt[k], r.sub(fma(-hdt, o.Wsl[k], o.Wh[k]), W0[k])), Wm[k]);
                Wb[k] = fma(h2, fma(-dt, e.Wt[k], r.sub(fma(-dt, o.Wsl[k], o.Wh[k]), W0[k])), Wb[k]);
            }
        }
    } else {
        for (int k = 0; k < 4; ++k) Wtt[k] = e.Wtt[k];
    }
    return ok;
}

}  // namespace cgks
