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
#include "cgks_device.cuh"
#include "cgks_internal.h"
#include "cgks_records.cuh"
#include "cgks_split.cuh"

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

int main()
{
    check_pairs();
    for (double base : {1.0, 0.0})
        for (int lev : {1, 3, 5, 8, 12, 20}) { check_rows<8>(lev, base, 1.0); check_rows<6>(lev, base, 1.0); }
    return 0;
}
