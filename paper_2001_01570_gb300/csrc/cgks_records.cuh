// cgks_records.cuh -- the arithmetic of one face-row record (the record
// kernel of cgks_records.cu runs it once per face row of a grid): the stencil
// cells with the boundary conditions applied on the fly (x-boundaries first,
// then y, so the corners match the oracle's ghost layers), the linear compact
// reconstruction (Sec. 3.2, Eq. recons-8th-val) and the nonlinear WENO-Z left
// and right states with their slopes (Sec. 3.3), in conservative or
// characteristic variables.
#pragma once
#include "cgks_device.cuh"
#include "cgks_internal.h"

namespace cgks {

// plane p of ghost cell (i, j) from the value v of its source cell: kx, ky are
// map_axis's transform kinds along x and y (x first, then y)
__device__ __forceinline__ double bc_value(const GridDev& G, double v, int i, int j, int kx, int ky, int p)
{
    if (kx == 1) { if (p == 1 || p == 4 || p == 6 || p == 7 || p == 9) v = -v; }
    else if (kx == 2) v = p < 4 ? G.inflow[i < 0 ? 0 : 1][p] : 0.0;
    else if (kx == 3) { if (p >= 4 && p < 8) v = 0.0; }
    if (ky == 1) { if (p == 2 || p == 6 || p == 8 || p == 9 || p == 11) v = -v; }
    else if (ky == 2) v = p < 4 ? G.inflow[j < 0 ? 2 : 3][p] : 0.0;
    else if (ky == 3) { if (p >= 8) v = 0.0; }
    return v;
}

// plane p of cell (i, j) with the boundary conditions applied outside the grid
__device__ __forceinline__ double cell_value(const GridDev& G, const double* src, size_t PL, int i, int j,
                                             int p)
{
    int kx, ky;
    const int si = map_axis(i, G.nx, G.bc[0], G.bc[1], kx);
    const int sj = map_axis(j, G.ny, G.bc[2], G.bc[3], ky);
    if (!CGKS_IN_BOUNDS(si >= 0 && si < G.nx && sj >= 0 && sj < G.ny && p >= 0 && p < 12, G.ctrl)) return 0.0;
    return bc_value(G, src[(size_t)p * PL + (size_t)sj * G.nx + si], i, j, kx, ky, p);
}

// geometry of record r of a grid: orientation, stencil start cell and step,
// frame of the variables, global record index
struct RowRef {
    bool xo, inner;
    int i0, j0, di, dj;     // stencil cell c is (i0 + c di, j0 + c dj)
    int gn;                 // first plane of the normal gradient
    double h, ih;
    double* base;           // record array of this orientation
    size_t stride;          // distance between (field, variable) slices
    size_t idx;             // index of this record inside a slice
};

__device__ __forceinline__ RowRef row_ref(const GridDev& G, int r)
{
    RowRef q;
    const int nx = G.nx, ny = G.ny;
    if (G.dim == 1) r += 2 * (nx + 1);      // the grid's only row: no neighbours along the faces are read
    const int nrx = (nx + 1) * (ny + 4);
    q.xo = r < nrx;
    if (q.xo) {
        const int f = r % (nx + 1), j = r / (nx + 1) - 2;
        q.inner = (j >= -1) && (j <= ny);
        q.i0 = f - 2; q.j0 = j; q.di = 1; q.dj = 0;
        q.gn = 4; q.h = G.dx; q.ih = G.inv_dx;
        q.base = G.recx; q.stride = (size_t)(ny + 4) * (nx + 1); q.idx = (size_t)r;
    } else {
        const int rr = r - nrx;
        const int g = rr % (ny + 1), i = rr / (ny + 1) - 2;
        q.inner = (i >= -1) && (i <= nx);
        q.i0 = i; q.j0 = g - 2; q.di = 0; q.dj = 1;
        q.gn = 8; q.h = G.dy; q.ih = G.inv_dy;
        q.base = G.recy; q.stride = (size_t)(nx + 4) * (ny + 1); q.idx = (size_t)rr;
    }
    return q;
}

// The four stencil cells of a row: where each one's values are read (its source cell inside
// the grid) and the boundary transforms along x and y.  The index across the row is the same
// for the four, so it is mapped once, and all of a row's values are read before the first is
// transformed: mapping and reading value by value (ten, in characteristic mode 32 copies of
// the mapping, one memory latency each) took 12,000 of a boundary row's 19,000 cycles, and
// the copies outgrew the instruction cache.
struct Stencil {
    size_t at[4];
    int kn[4], kt;          // transform kinds along and across the row
    bool ghost;             // some cell lies outside the grid
    __device__ __forceinline__ int kind(int c) const { return kn[c] | kt; }
    // plane p of cell c from the value v of its source cell
    __device__ __forceinline__ double value(const GridDev& G, const RowRef& q, int c, double v, int p) const
    {
        return bc_value(G, v, q.i0 + c * q.di, q.j0 + c * q.dj, q.xo ? kn[c] : kt, q.xo ? kt : kn[c], p);
    }
};

__device__ __forceinline__ void map_stencil(const GridDev& G, const RowRef& q, Stencil& s)
{
    const int i3 = q.i0 + 3 * q.di, j3 = q.j0 + 3 * q.dj;
    s.ghost = !(q.i0 >= 0 && q.j0 >= 0 && i3 < G.nx && j3 < G.ny);
    s.kt = 0;
    const size_t step = q.di ? 1 : (size_t)G.nx, base = (size_t)q.j0 * G.nx + q.i0;
#pragma unroll
    for (int c = 0; c < 4; ++c) { s.at[c] = base + c * step; s.kn[c] = 0; }
    if (!s.ghost) return;
    const int bn = q.xo ? 0 : 2, bt = 2 - bn;           // the axes' boundary conditions
    const int nn = q.xo ? G.nx : G.ny, nt = q.xo ? G.ny : G.nx;
    int st = map_axis(q.xo ? q.j0 : q.i0, nt, G.bc[bt], G.bc[bt + 1], s.kt);
    if (!CGKS_IN_BOUNDS(st >= 0 && st < nt, G.ctrl)) st = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        int sn = map_axis((q.xo ? q.i0 : q.j0) + c, nn, G.bc[bn], G.bc[bn + 1], s.kn[c]);
        if (!CGKS_IN_BOUNDS(sn >= 0 && sn < nn, G.ctrl)) sn = 0;
        s.at[c] = q.xo ? (size_t)st * G.nx + sn : (size_t)sn * G.nx + st;
    }
}

// one cell of the stencil, for the lane that reads it alone
struct StencilCell {
    size_t at;
    int kn, kt;
    __device__ __forceinline__ double value(const GridDev& G, const RowRef& q, int c, double v, int p) const
    {
        return bc_value(G, v, q.i0 + c * q.di, q.j0 + c * q.dj, q.xo ? kn : kt, q.xo ? kt : kn, p);
    }
};

__device__ __forceinline__ void map_cell(const GridDev& G, const RowRef& q, int c, StencilCell& s)
{
    const int i = q.i0 + c * q.di, j = q.j0 + c * q.dj;
    int kx, ky, si = map_axis(i, G.nx, G.bc[0], G.bc[1], kx), sj = map_axis(j, G.ny, G.bc[2], G.bc[3], ky);
    if (!CGKS_IN_BOUNDS(si >= 0 && si < G.nx && sj >= 0 && sj < G.ny, G.ctrl)) si = sj = 0;
    s.at = (size_t)sj * G.nx + si;
    s.kn = q.xo ? kx : ky;
    s.kt = q.xo ? ky : kx;
}

// Coefficient table of the register-form reconstruction, one block per order
// (index 0: the 8th-order scheme, 1: the 6th-order variant); copied to shared
// memory by each CTA.
struct ReconTab { double v[2][RK_N]; };

constexpr ReconTab make_recon_tab()
{
    ReconTab t{};
    for (int o = 0; o < 2; ++o) {
        double* k = t.v[o];
        const bool six = (o == 1);
        k[RK_ONE] = 1.0; k[RK_NZERO] = -0.0;
        k[RK_HALF] = 0.5; k[RK_MHALF] = -0.5; k[RK_M2] = -2.0; k[RK_M6TH] = -1.0 / 6.0;
        k[RK_DV + 0] = -1.0 / 12.0; k[RK_DV + 1] = six ? 0.2 : 17.0 / 70.0; k[RK_DV + 2] = six ? 0.0 : 1.0 / 140.0;
        k[RK_DS + 0] = six ? -11.0 / 36.0 : -10.0 / 27.0; k[RK_DS + 1] = six ? -2.0 / 3.0 : -11.0 / 12.0;
        k[RK_DS + 2] = six ? 0.0 : -1.0 / 72.0;
        k[RK_DC + 0] = six ? -1.5 : -2.25; k[RK_DC + 1] = six ? 0.0 : -0.125;
        const double e0[3] = {16.0 / 3.0, -38.0 / 3.0, 25.0 / 3.0};
        const double e1[6] = {801.0 / 80.0, -2443.0 / 80.0, 761.0 / 80.0, 23627.0 / 960.0, -7769.0 / 480.0,
                              3443.0 / 960.0};
        const double e2[6] = {1641.0 / 80.0, 2401.0 / 80.0, -5523.0 / 80.0, 12683.0 / 960.0, -25169.0 / 480.0,
                              56387.0 / 960.0};
        const double e3[3] = {4.0 / 3.0, -5.0 / 3.0, 4.0 / 3.0};
        const double e4[3] = {10.0 / 3.0, -11.0 / 3.0, 4.0 / 3.0};
        const double e5[10] = {4405.0 / 28.0, 4405.0 / 7.0, -110433.0 / 140.0, -21717.0 / 140.0, 93707.0 / 140.0,
                               -226333.0 / 140.0, -48901.0 / 140.0, 209917.0 / 210.0, 17063.0 / 42.0, 5153.0 / 105.0};
        const double e6[10] = {265067.0 / 140.0, 11104.0 / 7.0, -160551.0 / 140.0, -592783.0 / 140.0, 9529.0 / 28.0,
                               -65327.0 / 140.0, -252323.0 / 140.0, 38131.0 / 210.0, 52763.0 / 42.0, 251276.0 / 105.0};
        for (int i = 0; i < 3; ++i) { k[RK_E0 + i] = e0[i]; k[RK_E3 + i] = e3[i]; k[RK_E4 + i] = e4[i]; }
        for (int i = 0; i < 6; ++i) { k[RK_E1 + i] = e1[i]; k[RK_E2 + i] = e2[i]; }
        for (int i = 0; i < 10; ++i) { k[RK_E5 + i] = e5[i]; k[RK_E6 + i] = e6[i]; }
        k[RK_Z + 0] = 3.0; k[RK_Z + 1] = -2.0;
        // Sec. 3.3 linear weights d^8 (the 6th-order variant: d^6)
        const double w8[7] = {3.0 / 98.0, 5.0 / 98.0, 4.0 / 49.0, 7.0 / 98.0, 7.0 / 98.0, 17.0 / 49.0, 17.0 / 49.0};
        const double w6[7] = {3.0 / 70.0, 5.0 / 70.0, 8.0 / 70.0, 7.0 / 70.0, 7.0 / 70.0, 20.0 / 70.0, 20.0 / 70.0};
        const double* w = six ? w6 : w8;
        for (int i = 0; i < 7; ++i) k[RK_W + i] = w[i];
        const double d0 = w[0], d2w = w[2], d5 = w[5], d6 = w[6];
        k[RK_Q0 + 0] = d0 * 7.0 / 6.0; k[RK_Q0 + 1] = -(d0 * 2.0 / 3.0);
        k[RK_Q13 + 0] = 1.0 / 6.0; k[RK_Q13 + 1] = 1.0 / 3.0;
        k[RK_Q2 + 0] = d2w * 0.25; k[RK_Q2 + 1] = d2w * 19.0 / 24.0; k[RK_Q2 + 2] = -(d2w * 13.0 / 24.0);
        k[RK_Q4 + 0] = 2.0 / 3.0; k[RK_Q4 + 1] = -1.0 / 6.0;
        k[RK_Q5 + 0] = d5 * 0.1; k[RK_Q5 + 1] = d5 * 0.7; k[RK_Q5 + 2] = -(d5 / 3.0); k[RK_Q5 + 3] = d5 / 30.0;
        k[RK_Q6 + 0] = d6 * 29.0 / 30.0; k[RK_Q6 + 1] = d6 / 3.0; k[RK_Q6 + 2] = -(d6 * 0.7);
        k[RK_Q6 + 3] = -(d6 * 0.1);
        k[RK_S0 + 0] = d0 * 3.0; k[RK_S0 + 1] = -(d0 * 2.0);
        k[RK_S2 + 0] = d2w * 0.875; k[RK_S2 + 1] = d2w * 0.375; k[RK_S2 + 2] = -(d2w * 0.25);
        k[RK_S5 + 0] = d5 * 0.5; k[RK_S5 + 1] = d5 * 1.5; k[RK_S5 + 2] = -(d5 * 1.5); k[RK_S5 + 3] = d5 * 0.5;
        k[RK_S6 + 0] = d6 * 1.5; k[RK_S6 + 1] = d6 * 0.5; k[RK_S6 + 2] = d6 * 0.5; k[RK_S6 + 3] = -(d6 * 1.5);
    }
    return t;
}


// The arithmetic of one record in conservative variables: variable k from its
// four stencil cells (values Q, h times the normal gradients S), written through
// out(field, k, value); the WENO-Z fields only where `inner` (the rows the
// non-equilibrium states are needed on).  scale_hi: see scale_of.
template <int ORDER, class Out>
__device__ __forceinline__ void cons_record(const RegK& r, const double Q[4], const double S[4], double ih,
                                            double weno_eps, bool inner, int k, int scale_hi, Out out)
{
    double v, hvx, h2vxx;
    RowDiffs x;
    row_diffs_rk(r, Q, S, x);
    const double hd2 = r.kmul(RK_HALF, x.d2);
    linear_diff_rk<ORDER>(r, Q[1], hd2, x, v, hvx, h2vxx);
    out(RV, k, v);
    out(RN, k, r.mul(hvx, ih));
    out(RNN, k, r.mul(r.mul(h2vxx, ih), ih));
    if (inner) {
        double vl, sl, vr, sr;
#ifndef CGKS_PAIRS
        weno_pair_rk(r, Q[0], Q[1], Q[2], Q[3], S[0], S[1], S[2], S[3], weno_eps, vl, sl, vr, sr);
#else
        weno_pair_row<ORDER>(r, Q, S, x, hd2, weno_eps, scale_hi, vl, sl, vr, sr);
#endif
        out(RL, k, vl);
        out(RR, k, vr);
        out(RLN, k, r.mul(sl, ih));
        out(RRN, k, r.mul(sr, ih));
    }
}

#ifndef CGKS_PAIRS
inline int scale_of(int, double, double, double, double) { return 0; }
inline int char_scale(int, double, double) { return 0; }
#else
// High word of the scale a variable's rounding is measured against: density and
// energy against the values on the face's two sides (b, c); a momentum also
// against sqrt(rho E) (its high word: the mean of the two), the momentum whose
// changes the pressure fluxes' last bits amount to -- a gas at rest has no
// momentum of its own to measure against.
__device__ __forceinline__ int scale_of(int k, double b, double c, double rho, double E)
{
    int s = i_max(hi_abs(b), hi_abs(c));
    if (k == 1 || k == 2) s = i_max(s, (int)(((unsigned)hi_abs(rho) + (unsigned)hi_abs(E)) >> 1));
    return s;
}

// The same for characteristic field m: the density, whose dimension the acoustic and the entropy fields
// have; the shear field (2) has a momentum's, so sqrt(rho E).
__device__ __forceinline__ int char_scale(int m, double rho, double E)
{
    const int s = hi_abs(rho);
    return m == 2 ? (int)(((unsigned)s + (unsigned)hi_abs(E)) >> 1) : s;
}
#endif

// The linear part of one variable's record (values Q, normal gradients N), through
// out(field, k, value).
template <int ORDER, class Out>
__device__ __forceinline__ void linear_fields(const RegK& r, const double Q[4], const double N[4], double h, double ih,
                                              int k, Out out)
{
    double v, hvx, h2vxx, S[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) S[c] = r.mul(h, N[c]);
    RowDiffs x;
    row_diffs_rk(r, Q, S, x);
    linear_diff_rk<ORDER>(r, Q[1], r.kmul(RK_HALF, x.d2), x, v, hvx, h2vxx);
    out(RV, k, v);
    out(RN, k, r.mul(hvx, ih));
    out(RNN, k, r.mul(r.mul(h2vxx, ih), ih));
}

// Characteristic variables: the basis is taken at the mean of the two cells sharing the face (b, c) ...
__device__ __forceinline__ double char_mean(const RegK& r, double b, double c) { return r.mul(0.5, r.add(b, c)); }

// ... and a field's WENO-Z step, from its projections Q and h times its projected gradients S (scale_hi:
// char_scale); w[0..3]: left and right value, left and right slope per unit length.
template <int ORDER>
__device__ __forceinline__ void char_weno(const RegK& r, int scale_hi, const double Q[4], const double S[4], double ih,
                                          double weno_eps, double w[4])
{
#ifndef CGKS_PAIRS
    weno_pair_rk(r, Q[0], Q[1], Q[2], Q[3], S[0], S[1], S[2], S[3], weno_eps, w[0], w[2], w[1], w[3]);
#else
    RowDiffs x;
    row_diffs_rk(r, Q, S, x);
    weno_pair_row<ORDER>(r, Q, S, x, r.kmul(RK_HALF, x.d2), weno_eps, scale_hi, w[0], w[2], w[1], w[3]);
#endif
    w[2] = r.mul(w[2], ih);
    w[3] = r.mul(w[3], ih);
}

// The arithmetic of one record in characteristic variables by one thread: all four
// variables from the stencil cells' values Qa[var][cell] and normal gradients
// Na[var][cell] (face frame), written through out(field, k, value).  (The record kernel
// gives each field a lane of its own, the same operations.)
template <int ORDER, class Out>
__device__ __forceinline__ void char_record(const RegK& r, double gamma, const double Qa[4][4], const double Na[4][4],
                                            double h, double ih, double weno_eps, bool inner, Out out)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) linear_fields<ORDER>(r, Qa[k], Na[k], h, ih, k, out);
    if (!inner) return;
    CharState cs;
    double Wref[4], w[4][4], o4[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) Wref[k] = char_mean(r, Qa[k][1], Qa[k][2]);
    char_state(r, Wref, gamma, cs);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        double l[4], Q[4], S[4], v[4];
        char_left_row(r, cs, m, l);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            Q[c] = char_project(r, m, l, Qa[0][c], Qa[1][c], Qa[2][c], Qa[3][c]);
            S[c] = r.mul(h, char_project(r, m, l, Na[0][c], Na[1][c], Na[2][c], Na[3][c]));
        }
        char_weno<ORDER>(r, char_scale(m, Wref[0], Wref[3]), Q, S, ih, weno_eps, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q][m] = v[q];
    }
    const int fields[4] = {RL, RR, RLN, RRN};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        char_to_cons(r, cs, w[q], o4);
#pragma unroll
        for (int k = 0; k < 4; ++k) out(fields[q], k, o4[k]);
    }
}

// Conservative variables: variable k of face row `row`.
template <int ORDER>
__device__ __forceinline__ void cons_row(const RegK& r, const GridDev& G, const double* src, size_t PL,
                                         int row, int k)
{
    const RowRef q = row_ref(G, row);
    if (!CGKS_IN_BOUNDS(q.idx < q.stride, G.ctrl)) return;
    const int pv = q.xo ? k : ((k == 1) ? 2 : (k == 2) ? 1 : k);   // face frame: normal momentum first
    double Q[4], S[4], rho = 0.0, E = 0.0;   // rho, E: cell b's, where a momentum's scale needs them
    Stencil c4;
    map_stencil(G, q, c4);
    const double *v = src + (size_t)pv * PL, *d = src + (size_t)(q.gn + pv) * PL;
#pragma unroll
    for (int c = 0; c < 4; ++c) { Q[c] = v[c4.at[c]]; S[c] = d[c4.at[c]]; }
    const bool mom = (k == 1 || k == 2) && q.inner;
    if (mom) { rho = src[c4.at[1]]; E = src[3 * PL + c4.at[1]]; }
    if (c4.ghost) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (!c4.kind(c)) continue;
            Q[c] = c4.value(G, q, c, Q[c], pv);
            S[c] = c4.value(G, q, c, S[c], q.gn + pv);
        }
        if (mom && c4.kind(1)) { rho = c4.value(G, q, 1, rho, 0); E = c4.value(G, q, 1, E, 3); }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) S[c] = r.mul(q.h, S[c]);
    double* o = q.base + q.idx;
    const size_t st = q.stride;
    cons_record<ORDER>(r, Q, S, q.ih, G.weno_eps, q.inner, k, scale_of(k, Q[1], Q[2], rho, E),
                       [&](int f, int kk, double x) { o[(f * 4 + kk) * st] = x; });
}

#ifdef CGKS_OPCOUNT_HOST
// the stencil cells of a row, all four variables in the face frame
__device__ __forceinline__ void char_stencil(const GridDev& G, const double* src, size_t PL, const RowRef& q,
                                             double Qa[4][4], double Na[4][4])
{
    const int p1 = q.xo ? 1 : 2, p2 = q.xo ? 2 : 1;         // planes of the normal and tangential momentum
    Stencil c4;
    map_stencil(G, q, c4);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const double* v = src + c4.at[c];
        const double* n = v + (size_t)q.gn * PL;
        Qa[0][c] = v[0]; Qa[1][c] = v[p1 * PL]; Qa[2][c] = v[p2 * PL]; Qa[3][c] = v[3 * PL];
        Na[0][c] = n[0]; Na[1][c] = n[p1 * PL]; Na[2][c] = n[p2 * PL]; Na[3][c] = n[3 * PL];
    }
    if (!c4.ghost) return;
    const int pk[4] = {0, p1, p2, 3};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (!c4.kind(c)) continue;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Qa[k][c] = c4.value(G, q, c, Qa[k][c], pk[k]);
            Na[k][c] = c4.value(G, q, c, Na[k][c], q.gn + pk[k]);
        }
    }
}

// Characteristic variables: all four variables of face row `row` by one thread (the host count)
template <int ORDER>
__device__ __forceinline__ void char_row(const RegK& r, const GridDev& G, const double* src, size_t PL,
                                         int row)
{
    const RowRef q = row_ref(G, row);
    if (!CGKS_IN_BOUNDS(q.idx < q.stride, G.ctrl)) return;
    double Qa[4][4], Na[4][4];
    char_stencil(G, src, PL, q, Qa, Na);
    double* o = q.base + q.idx;
    const size_t st = q.stride;
    char_record<ORDER>(r, G.gamma, Qa, Na, q.h, q.ih, G.weno_eps, q.inner,
                       [&](int f, int kk, double x) { o[(f * 4 + kk) * st] = x; });
}
#else
// a 4x4 matrix over a quad of lanes, lane m holding row m, becomes its transpose
__device__ __forceinline__ void quad_transpose(unsigned quad, int m, double a[4])
{
#pragma unroll
    for (int s = 1; s < 4; s <<= 1) {
        const bool up = m & s;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i & s) continue;                // the pair of columns i, i + s
            const double got = __shfl_xor_sync(quad, up ? a[i] : a[i | s], s);
            if (up) a[i] = got;
            else a[i | s] = got;
        }
    }
}

// Characteristic variables: face row `row` by four lanes (a quad of a warp).  Lane m reads cell m of the stencil and projects it on
// the four left eigenvectors; transposed, it has variable m of the four cells for the linear
// fields and field m for the WENO-Z step, and, transposed again, quantity m (left, right value, left,
// right slope) of the four fields, which it brings back to conservative variables.  One thread per row
// ran the four fields in turn: 600 FP64 instructions in one chain and 254 registers; with every lane
// of the quad reading the whole stencil the kernel waited for its instructions (200x50: 65 us, 58 here).
template <int ORDER>
__device__ __forceinline__ void char_row_quad(const RegK& r, const GridDev& G, const double* src, size_t PL,
                                              int row, int m, unsigned quad)
{
    const RowRef q = row_ref(G, row);
    if (!CGKS_IN_BOUNDS(q.idx < q.stride, G.ctrl)) return;
    const int p1 = q.xo ? 1 : 2, p2 = q.xo ? 2 : 1;         // planes of the normal and tangential momentum
    StencilCell c;
    map_cell(G, q, m, c);
    const double *v = src + c.at, *n = v + (size_t)q.gn * PL;
    double Q[4] = {v[0], v[p1 * PL], v[p2 * PL], v[3 * PL]}, N[4] = {n[0], n[p1 * PL], n[p2 * PL], n[3 * PL]};
    if (c.kn | c.kt) {
        const int pk[4] = {0, p1, p2, 3};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Q[k] = c.value(G, q, m, Q[k], pk[k]);
            N[k] = c.value(G, q, m, N[k], q.gn + pk[k]);
        }
    }
    double Qm[4] = {Q[0], Q[1], Q[2], Q[3]}, Nm[4] = {N[0], N[1], N[2], N[3]};
    quad_transpose(quad, m, Qm);
    quad_transpose(quad, m, Nm);
    double* o = q.base + q.idx;
    const size_t st = q.stride;
    linear_fields<ORDER>(r, Qm, Nm, q.h, q.ih, m, [&](int f, int kk, double x) { o[(f * 4 + kk) * st] = x; });
    if (!q.inner) return;                     // the same for the quad's lanes (one row)
    CharState cs;
    const double mean = char_mean(r, Qm[1], Qm[2]);
    double Wref[4], P[4], S[4], w[4], o4[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) Wref[k] = __shfl_sync(quad, mean, k, 4);
    char_state(r, Wref, G.gamma, cs);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        double l[4];
        char_left_row(r, cs, f, l);
        P[f] = char_project(r, f, l, Q[0], Q[1], Q[2], Q[3]);
        S[f] = r.mul(q.h, char_project(r, f, l, N[0], N[1], N[2], N[3]));
    }
    quad_transpose(quad, m, P);
    quad_transpose(quad, m, S);
    char_weno<ORDER>(r, char_scale(m, Wref[0], Wref[3]), P, S, q.ih, G.weno_eps, w);
    quad_transpose(quad, m, w);
    char_to_cons(r, cs, w, o4);
    const int f = m == 0 ? RL : m == 1 ? RR : m == 2 ? RLN : RRN;
#pragma unroll
    for (int k = 0; k < 4; ++k) o[(f * 4 + k) * st] = o4[k];
}
#endif

}  // namespace cgks
