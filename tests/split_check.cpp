// Host check of the split (pairs of FP32) arithmetic of the kernels against the FP64 formulas it
// stands in for: both are compared with long double evaluations of the same rows.  Prints one line
// per check: name, amplitude exponent, rows taken, rows, then max and rms errors (split, FP64).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#define CGKS_OPCOUNT_HOST 1   // the plain FP64 forms of the device headers
#define CGKS_SPLIT_CHECK 1    // and the pairs' arithmetic beside them
inline double cgks_opcount_rcp(double x) { return 1.0 / x; }
inline double cgks_opcount_exp(double x) { return std::exp(x); }
inline double cgks_opcount_erfc(double x) { return std::erfc(x); }
inline double __drcp_rn(double x) { return 1.0 / x; }
inline double __ddiv_rn(double a, double b) { return a / b; }
inline double __dmul_rn(double a, double b) { return a * b; }
inline double __dadd_rn(double a, double b) { return a + b; }
inline double __dsub_rn(double a, double b) { return a - b; }
inline double __dsqrt_rn(double a) { return std::sqrt(a); }
inline double rsqrt(double a) { return 1.0 / std::sqrt(a); }
inline long long __double_as_longlong(double x) { long long b; memcpy(&b, &x, 8); return b; }
inline double __longlong_as_double(long long b) { double x; memcpy(&x, &b, 8); return x; }
template <class T> inline T __ldg(const T* p) { return *p; }
inline int min(int a, int b) { return a < b ? a : b; }
inline int max(int a, int b) { return a > b ? a : b; }
#include "cgks_split.cuh"
#include "cgks_device.cuh"
#include "cgks_internal.h"
#include "cgks_records.cuh"
#include "cgks_flux.cuh"

using namespace cgks;
typedef long double Q;

static double err(Q x, Q y) { return (double)std::fabs(x - y); }
static double val(ff a) { return (double)a.h + (double)a.l; }

struct Stat {
    double mx[2] = {0, 0}, sq[2] = {0, 0};
    long n = 0;
    void add(double a, double b)
    {
        mx[0] = std::max(mx[0], a); mx[1] = std::max(mx[1], b);
        sq[0] += a * a; sq[1] += b * b; ++n;
    }
    void print(const char* name, int lev, long rows) const
    {
        printf("%s %d %ld %ld %.4e %.4e %.4e %.4e\n", name, lev, n, rows, mx[0], mx[1], std::sqrt(sq[0] / std::max(1l, n)),
               std::sqrt(sq[1] / std::max(1l, n)));
    }
};

// a random smooth row of four cells: base + amp * (two sines), averages and h * slopes
struct Row {
    double Q4[4], S[4];
    template <class G, class U> Row(G& g, U& u, double base, double amp)
    {
        const double k1 = 0.3 + 1.5 * u(g), k2 = 0.3 + 2.5 * u(g), p1 = 6.28 * u(g), p2 = 6.28 * u(g), a1 = u(g), a2 = 0.5 * u(g);
        auto F = [&](double x) { return base * x - amp * (a1 * std::cos(k1 * x + p1) / k1 + a2 * std::cos(k2 * x + p2) / k2); };
        auto f = [&](double x) { return base + amp * (a1 * std::sin(k1 * x + p1) + a2 * std::sin(k2 * x + p2)); };
        for (int c = 0; c < 4; ++c) { Q4[c] = F(c - 0.5) - F(c - 1.5); S[c] = f(c - 0.5) - f(c - 1.5); }
    }
};

// the left-biased value and h * slope of Sec. 3.3 by its definition, on (1, i-1..i+2) data relative to cell i
static void left_side(int order, const Q d[3], const Q S[4], Q eps, Q& v, Q& sl)
{
    const Q d1 = d[0], d2 = d[1], d3 = d[2], s3 = d2 - d1, s4 = d3 - d2, a = d1 - S[0], dd = S[3] - d3;
    const Q t = s3 - 2 * a, u = s4 - 2 * dd, w = s4 - s3, p = S[1] - (d1 + d2) / 2, q = S[2] - (d2 + d3) / 2;
    const Q G = d2 - s3 / 2, H = d2 - s4 / 2;
    const Q c45 = -(t / 4 + p), c46 = q - u / 4;
    // sum over r of the integrals of the squared r-th derivatives, c2 half the second derivative at the centre
    auto beta = [](Q L, Q c2, Q c3, Q c4) {
        return L * L + 13 * c2 * c2 / 3 + 21 * c2 * c4 / 5 + 781 * c3 * c3 / 20 +
               c4 * c4 * (Q(103) / 100 + Q(16) / 2800 + Q(4) / 5 + 48 + 576);
    };
    const Q e[7] = {beta(G - t / 2, (s3 - t) / 2, 0, 0) + eps, beta(G - t / 4, s3 / 2, t / 4, 0) + eps,
                    beta(H - u / 2, s4 / 2 + 3 * u / 4, -u / 4, 0) + eps, beta(G, s3 / 2, 0, 0) + eps,
                    beta(H, s4 / 2, 0, 0) + eps, beta(G + p, s3 / 2 + 3 * t / 8 + 3 * p / 2, -p, c45) + eps,
                    beta(H + u / 2 - 4 * q, s4 / 2 - 9 * u / 8 + 15 * q / 2, u - 5 * q, c46) + eps};
    const Q Z = std::fabs(3 * (e[0] - e[4]) + (e[4] - e[3]));
    const int w8[7] = {3, 5, 8, 7, 7, 34, 34}, w6[7] = {3, 5, 8, 7, 7, 20, 20};
    const Q y[7] = {-t / 3, 0, -w / 6 - u / 8, 0, -w / 6, t / 20 + 7 * p / 10, -w / 6 + u / 20 - 7 * q / 10};
    const Q z[7] = {-t, 0, u / 8, 0, 0, t / 4 + 3 * p / 2, 3 * q / 2 - u / 4};
    Q s = 0, nv = 0, ns = 0;
    for (int k = 0; k < 7; ++k) {
        const Q al = (order == 6 ? w6 : w8)[k] * (1 + Z / e[k]);
        s += al; nv += al * y[k]; ns += al * z[k];
    }
    v = d2 / 2 - s3 / 6 + nv / s;
    sl = d2 + ns / s;
}

template <int ORDER> static void check_rows(int lev, double base, double unit)
{
    static double tab[2 * RK_N];
    const ReconTab T = make_recon_tab();
    for (int o = 0; o < 2; ++o) for (int i = 0; i < RK_N; ++i) tab[o * RK_N + i] = T.v[o][i];
    const RegK r{tab + (ORDER == 6 ? RK_N : 0), 1.0, -0.0};
    std::mt19937_64 g(11 + lev);
    std::uniform_real_distribution<double> u01(0.0, 1.0);
    auto u = [&](std::mt19937_64& x) { return u01(x); };
    const double eps = 1e-6;
    Stat sv, ss;
    const long rows = 20000;
    for (long it = 0; it < rows; ++it) {
        const Row row(g, u, base * (0.5 + u(g)), std::ldexp(unit, -lev));
        const double *q = row.Q4, *S = row.S;
        const double d1 = q[1] - q[0], d2 = q[2] - q[1], d3 = q[3] - q[2], s3 = d2 - d1, s4 = d3 - d2, w = s4 - s3;
        const double t = fma(-2.0, d1 - S[0], s3), ut = fma(-2.0, S[3] - d3, s4), p = fma(-0.5, d1 + d2, S[1]), pq = fma(-0.5, d2 + d3, S[2]);
        const int scale = std::max(hi_abs(q[1]), std::max(hi_abs(q[2]), hi_abs(unit)));
        if (!split_ok(scale, eps, w, t, ut, p, pq, s3)) continue;
        double vl, sl, vr, sr;
        weno_pair_rk(r, q[0], q[1], q[2], q[3], S[0], S[1], S[2], S[3], eps, vl, sl, vr, sr);
        DiffData m{ff_from(d2), ff_from(s3), ff_from(s4), ff_from(w), ff_from(t), ff_from(ut), ff_from(p), ff_from(pq)};
        ff dv, ds, rv, rs;
        weno_side_split<ORDER>(m, ff_from(eps), dv, ds);
        weno_side_split<ORDER>(DiffData{ff_neg(m.d2), m.s4, m.s3, ff_neg(m.w), m.u, m.t, ff_neg(m.q), ff_neg(m.p)}, ff_from(eps), rv, rs);
        const double hd = 0.5 * d2;
        const double nvl = q[1] + (fma(-1.0 / 6.0, s3, hd) + val(dv)), nvr = q[2] + (fma(-1.0 / 6.0, s4, -hd) + val(rv));
        const Q D[3] = {(Q)q[1] - q[0], (Q)q[2] - q[1], (Q)q[3] - q[2]}, E[3] = {-D[2], -D[1], -D[0]};
        const Q A[4] = {S[0], S[1], S[2], S[3]}, B[4] = {-A[3], -A[2], -A[1], -A[0]};
        Q xl, yl, xr, yr;
        left_side(ORDER, D, A, eps, xl, yl);
        left_side(ORDER, E, B, eps, xr, yr);
        xl += q[1]; xr += q[2];
        sv.add(std::max(err(nvl, xl), err(nvr, xr)), std::max(err(vl, xl), err(vr, xr)));
        ss.add(std::max(err(d2 + val(ds), yl), err(d2 - val(rs), -yr)), std::max(err(sl, yl), err(sr, -yr)));
    }
    char name[64];
    snprintf(name, sizeof name, "weno%d_value_base%g", ORDER, base);
    sv.print(name, lev, rows);
    snprintf(name, sizeof name, "weno%d_slope_base%g", ORDER, base);
    ss.print(name, lev, rows);
}

// double -> pair -> double keeps 47 bits, exactly representable values keep all
static void check_pairs()
{
    std::mt19937_64 g(3);
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    double worst = 0.0, exact = 0.0, back = 0.0;
    for (int it = 0; it < 200000; ++it) {
        const double x = std::ldexp(u(g), (int)(60 * u(g)));
        worst = std::max(worst, std::fabs(val(ff_from(x)) - x) / std::fabs(x));
        const float f = (float)x;
        exact = std::max(exact, std::fabs(val(ff_from((double)f)) - (double)f));
        back = std::max(back, std::fabs(d_from(f) - (double)f));
    }
    printf("pairs 0 0 0 %.4e %.4e %.4e %.4e\n", worst, exact, back, std::fabs(val(ff_from(0.0))) + std::fabs(d_from(0.0f)));
}

// arithmetic of slope_moments and euler_second in long double
struct ArLD {
    using T = Q;
    Q g1, k1, k3;
    Q add(Q a, Q b) const { return a + b; }
    Q sub(Q a, Q b) const { return a - b; }
    Q mul(Q a, Q b) const { return a * b; }
    Q mad(Q a, Q b, Q c) const { return a * b + c; }
    Q nmad(Q a, Q b, Q c) const { return c - a * b; }
    Q half(Q a) const { return a / 2; }
    Q dbl(Q a) const { return a + a; }
    Q tri(Q a) const { return 3 * a; }
    Q gm1() const { return g1; }
    Q K1() const { return k1; }
    Q K3() const { return k3; }
};

struct FluxTable {
    double t[FK_N];
    RegK r;
    FluxTable()
    {
        const FluxFixed f = make_flux_fixed();
        for (int i = 0; i < FK_N; ++i) t[i] = 0.0;
        for (int i = 0; i < FK_NFIX; ++i) t[i] = f.v[i];
        t[FK_GM1] = 0.4; t[FK_GAMMA] = 1.4; t[FK_K1] = 4.0; t[FK_K3] = 6.0;
        r = RegK{t, 1.0, -0.0};
    }
};

// the two point values and the slope along a face, from five (three) means of a smooth function
static void check_tangential(int lev)
{
    const FluxTable F;
    const RegK& r = F.r;
    std::mt19937_64 g(5 + lev);
    std::uniform_real_distribution<double> u(0.0, 1.0);
    const double eps = 1e-6, hg = 0.5 * 0.28867513459481287;
    Stat s5, s3;
    const long rows = 20000;
    for (long it = 0; it < rows; ++it) {
        const double base = 0.5 + u(g), amp = std::ldexp(1.0, -lev), k1 = 0.2 + u(g), k2 = 0.2 + 2.0 * u(g), p1 = 6.28 * u(g), p2 = 6.28 * u(g);
        double v[5];
        for (int c = 0; c < 5; ++c) v[c] = base + amp * (std::sin(k1 * c + p1) + 0.5 * std::sin(k2 * c + p2));
        TangDiffs x;
        tang_diffs(r, v[0], v[1], v[2], v[3], v[4], x);
        const int sc = hi_abs(v[2]);
        const ff da = ff_from(v[1] - v[0]), db = ff_from(v[2] - v[1]), dc = ff_from(v[3] - v[2]), dd = ff_from(v[4] - v[3]);
        const QuarticParts q = quartic_split(da, db, dc, dd);
        if (std::max(std::max(hi_abs(v[1] - v[0]), hi_abs(v[2] - v[1])), std::max(hi_abs(v[3] - v[2]), hi_abs(v[4] - v[3]))) < sc + kTangFirst * (1 << 20) &&
            i_max(hi_abs(x.t0), hi_abs(x.t1)) < sc + kTangThird * (1 << 20)) {
            double om, op;
            tang_weno5_pair(r, v[2], x, 4.0 * eps, om, op);
            ff m, p;
            tang_weno5_split(q.A, q.s, q.t0, q.t1, ff_from(4.0 * eps), CGKS_FF(kTangLo), CGKS_FF(kTangHi), m, p);
            const double A1 = v[3] - v[1], nm = fma(-hg, A1 - val(m), v[2]), np = fma(hg, A1 - val(p), v[2]);
            const Q V[5] = {v[0], v[1], v[2], v[3], v[4]}, D[3] = {3 * V[2] - 4 * V[1] + V[0], V[3] - V[1], 4 * V[3] - V[4] - 3 * V[2]};
            Q e[3];
            for (int k = 0; k < 3; ++k) { const Q s2 = V[k] - 2 * V[k + 1] + V[k + 2]; e[k] = D[k] * D[k] + 13 * s2 * s2 / 3 + 4 * (Q)eps; }
            const Q Z = std::fabs(e[0] - e[2]);
            Q ref[2];
            for (int side = 0; side < 2; ++side) {
                const Q w[3] = {side ? (Q)kTangLo : (Q)kTangHi, 1, side ? (Q)kTangHi : (Q)kTangLo};
                Q n = 0, d = 0;
                for (int k = 0; k < 3; ++k) { const Q a = w[k] * (1 + Z / e[k]); n += a * D[k]; d += a; }
                ref[side] = V[2] + (side ? (Q)hg : -(Q)hg) * n / d;
            }
            s5.add(std::max(err(nm, ref[0]), err(np, ref[1])), std::max(err(om, ref[0]), err(op, ref[1])));
        }
        {
            const double dm = v[2] - v[1], dp = v[3] - v[2], A = dp + dm, s = dp - dm;
            const ff c = tang_weno3_split(ff_from(A), ff_from(s), ff_from(eps));
            if (hi_abs(d_from(c.h)) < sc + kTangSlope * (1 << 20)) {
                double n, d;
                tang_weno3_parts(r, v[1], v[2], v[3], eps, n, d);
                const Q a = (Q)v[2] - v[1], b = (Q)v[3] - v[2], e0 = a * a + (Q)eps, e1 = b * b + (Q)eps, z = std::fabs(e0 - e1);
                const Q w0 = 1 + z / e0, w1 = 1 + z / e1, ref = (w0 * a + w1 * b) / (w0 + w1);
                s3.add(err(0.5 * (A - val(c)), ref), err(n / d, ref));
            }
        }
    }
    s5.print("tang_value", lev, rows);
    s3.print("tang_slope", lev, rows);
}

// slope moments and W_tt against long double, relative to the size of their terms
static void check_moments()
{
    const FluxTable F;
    std::mt19937_64 g(17);
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    const ArLD ql{(Q)0.4, 4, 6};
    const ArSplit qs{ff_from(0.4), ff_from(4.0), ff_from(6.0)};
    const Ar64 q64{F.r};
    Stat st, se;
    const long rows = 20000;
    for (long it = 0; it < rows; ++it) {
        const double U = 1.5 * u(g), V = 1.5 * u(g), th = 0.3 + std::fabs(u(g)), sq = std::sqrt(0.5 / th);
        const int side = it & 1;
        double m[4], bn[4], bt[4];
        m[0] = 0.5 * std::erfc((side ? 1 : -1) * U * sq);
        const double gd = (side ? -1 : 1) * std::exp(-U * U * sq * sq) * sq / std::sqrt(M_PI);
        m[1] = U * m[0] + th * gd; m[2] = U * m[1] + th * m[0]; m[3] = U * m[2] + 2 * th * m[1];
        for (int k = 0; k < 4; ++k) { bn[k] = u(g); bt[k] = u(g); }
        Q Lm[4], Ln[4], Lt[4], T[4], W[4];
        double T64[4], W64[4];
        ff Sm[4], Sn[4], St[4], Ts[4], Ws[4];
        for (int k = 0; k < 4; ++k) {
            Lm[k] = m[k]; Ln[k] = bn[k]; Lt[k] = bt[k];
            Sm[k] = ff_from(m[k]); Sn[k] = ff_from(bn[k]); St[k] = ff_from(bt[k]);
        }
        const double ith = 1.0 / th;
        slope_moments(ql, true, (Q)U, (Q)V, (Q)th, (Q)ith, Lm, (Q)gd, Ln, Lt, T, W);
        slope_moments(q64, true, U, V, th, ith, m, gd, bn, bt, T64, W64);
        slope_moments(qs, true, ff_from(U), ff_from(V), ff_from(th), ff_from(ith), Sm, ff_from(gd), Sn, St, Ts, Ws);
        double size = 0.0, a = 0.0, b = 0.0;
        for (int k = 0; k < 4; ++k) size += std::fabs(bn[k]) + std::fabs(bt[k]);
        size *= std::pow(1.0 + U * U + V * V + th, 2);
        for (int k = 0; k < 4; ++k) {
            a = std::max(a, std::max(err(val(Ts[k]), T[k]), err(val(Ws[k]), W[k])));
            b = std::max(b, std::max(err(T64[k], T[k]), err(W64[k], W[k])));
        }
        st.add(a / size, b / size);

        EulerFirst<double> f;
        double* fd = (double*)&f;
        for (size_t i = 0; i < sizeof f / sizeof(double); ++i) fd[i] = u(g);
        f.rho = 0.5 + std::fabs(u(g)); f.U = U; f.V = V; f.ir = 1.0 / f.rho; f.gir = 0.4 * f.ir; f.hq2 = 0.5 * (U * U + V * V); f.e = f.rho * th / 0.4;
        EulerFirst<Q> fl;
        EulerFirst<ff> fs;
        for (size_t i = 0; i < sizeof f / sizeof(double); ++i) { ((Q*)&fl)[i] = fd[i]; ((ff*)&fs)[i] = ff_from(fd[i]); }
        double w2[3][4], o64[4], sec = 0.0;
        Q l2[3][4], ol[4];
        ff s2[3][4], os[4];
        for (int d = 0; d < 3; ++d)
            for (int k = 0; k < 4; ++k) { w2[d][k] = u(g); l2[d][k] = w2[d][k]; s2[d][k] = ff_from(w2[d][k]); sec += std::fabs(w2[d][k]); }
        euler_second(ql, fl, (Q)1.4, l2[0], l2[1], l2[2], ol);
        euler_second(q64, f, 1.4, w2[0], w2[1], w2[2], o64);
        euler_second(qs, fs, ff_from(1.4), s2[0], s2[1], s2[2], os);
        const double sp = 1.0 + std::fabs(U) + std::fabs(V) + 2.0 * std::sqrt(th);
        double first = 0.0;
        for (size_t i = 0; i < sizeof f / sizeof(double); ++i) first += std::fabs(fd[i]);
        const double sz = sp * sp * sp * sp * (sec + first * first) * (1.0 + f.rho) * (1.0 + f.ir);
        a = b = 0.0;
        for (int k = 0; k < 4; ++k) { a = std::max(a, err(val(os[k]), ol[k])); b = std::max(b, err(o64[k], ol[k])); }
        se.add(a / sz, b / sz);
    }
    st.print("slope_moments", 0, rows);
    se.print("euler_second", 0, rows);
}

int main()
{
    check_pairs();
    for (int lev : {2, 4, 6, 9, 14}) check_tangential(lev);
    check_moments();
    for (double base : {1.0, 0.0})
        for (int lev : {1, 3, 5, 8, 12, 20}) { check_rows<8>(lev, base, 1.0); check_rows<6>(lev, base, 1.0); }
    return 0;
}
