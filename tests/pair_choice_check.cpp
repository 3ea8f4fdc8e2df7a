// The choices between pairs of FP32 and FP64 themselves, on the host: each of the kernels' functions that
// makes one is driven with random data from well inside to well outside its bound and compared with the
// bound worked out in FP64.  Prints per choice: name, how often the pairs were allowed, how often not, how
// often the function and the bound disagreed (points within 1 % of the bound are left out).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#define CGKS_OPCOUNT_HOST 1
#define CGKS_SPLIT_CHECK 1
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
#include "cgks_internal.h"
#include "cgks_records.cuh"
#include "cgks_segment.cuh"

using namespace cgks;
using RG = RecGroups<1, 1>;

static std::mt19937_64 g(99);
static double u(double lo = -1.0, double hi = 1.0) { return std::uniform_real_distribution<double>(lo, hi)(g); }

struct Tally {
    long yes = 0, no = 0, bad = 0;
    // got: the pairs were allowed; x: the largest of the bounded quantities over their bounds
    void add(bool got, double x, double margin = 0.01)
    {
        if (std::fabs(x - 1.0) < margin) return;
        (got ? yes : no)++;
        bad += got != (x < 1.0);
    }
    void print(const char* n) const { printf("%s %ld %ld %ld\n", n, yes, no, bad); }
};

// what the slope moments and W_tt pull from a segment
struct Source {
    double n[2][4], t[2][4], xx[4], xy[4], yy[4], iht = 1.0;
    int bits = 0;
    int rough() const { return bits; }
    void ne_slopes_split(int side, ff a[4], ff b[4]) const { for (int k = 0; k < 4; ++k) { a[k] = ff_from_any(n[side][k]); b[k] = ff_from_any(t[side][k]); } }
    void eq_second_split(ff a[4], ff b[4], ff c[4]) const
    {
        for (int k = 0; k < 4; ++k) { a[k] = ff_from_any(xx[k]); b[k] = ff_from_any(xy[k]); c[k] = ff_from_any(yy[k]); }
    }
};

struct Table {
    double t[FK_N];
    RegK r;
    Table(double dt, double eps = 1e-6)
    {
        const FluxFixed f = make_flux_fixed();
        for (int i = 0; i < FK_NFIX2; ++i) t[i] = f.v[i];
        GridDev G;
        memset(&G, 0, sizeof G);
        G.dx = G.dy = G.inv_dx = G.inv_dy = 1.0; G.gamma = 1.4; G.K = 3.0; G.eps_tau = 0.01; G.c_tau = 1.0; G.weno_eps = eps;
        flux_table_tile(t, G, dt);
        r = RegK{t, 1.0, -0.0};
    }
};

static void slope_choice()
{
    const Table T(0.25);
    Tally flux, state;
    for (int it = 0; it < 40000; ++it) {
        const bool ne = it & 1;
        const int side = (it >> 1) & 1;
        const double rho = u(0.5, 1.5), U = u(), V = u(), th = u(0.5, 1.5), th2 = th + th, sq = 1.0 / std::sqrt(th2);
        HalfMoments h;
        half_moments(T.r, side, U, th, th2, sq, h);
        Source s;
        for (int k = 0; k < 4; ++k) { s.n[side][k] = u(); s.t[side][k] = u(); }
        double t[4], w[4];
        slope_moments(Ar64{T.r}, true, U, V, th, 1.0 / th, h.m, h.g, s.n[side], s.t[side], t, w);
        const double f0 = rho * std::fabs(h.m[1]), f1 = rho * h.m[2], q = V * V + 4.0 * th;
        const double f3 = 0.5 * rho * (std::fabs(h.m[1]) * q + std::fabs(h.m[3])), w3 = 0.5 * rho * (h.m[0] * q + h.m[2]);
        const double wth = std::exp(u(-12.0, 0.0)), wsl = ne ? std::exp(u(-12.0, 0.0)) : 0.0;
        const double x = 128.0 * wth * std::max(std::fabs(t[0]) / f0, std::max((std::fabs(t[1]) + std::fabs(t[2])) / f1, std::fabs(t[3]) / f3));
        const double y = 128.0 * wsl * std::max(std::fabs(w[0]) / rho, std::max((std::fabs(w[1]) + std::fabs(w[2])) / f0, std::fabs(w[3]) / w3));
        ff a[4] = {}, b[4] = {};
        const bool ok = slope_moments_split(T.r, s, side, ne, rho, U, V, th, sq, h, (float)wth, (float)wsl, a, b);
        if (!ne) flux.add(ok, x);
        else if (y > x) state.add(ok, y);
        else flux.add(ok, x);
        s.n[side][it & 3] = it & 4 ? 1e39 : INFINITY;           // out of a float's range: refused however small the weight
        ff c[4] = {}, d[4] = {};
        if (slope_moments_split(T.r, s, side, ne, rho, U, V, th, sq, h, 1e-30f, 1e-30f, c, d)) flux.bad++;
    }
    flux.print("slope_moments_flux");
    state.print("slope_moments_state");
}

static void wtt_choice()
{
    const Table T(0.25);
    Tally n;
    for (int it = 0; it < 40000; ++it) {
        const double amp = std::exp(u(-7.0, 0.0)), rho = u(0.5, 1.5), th = u(0.5, 1.5);
        EulerFirst<double> f;
        double* fd = (double*)&f;
        for (size_t i = 0; i < sizeof f / sizeof(double); ++i) fd[i] = amp * u();
        f.rho = rho; f.U = u(); f.V = u(); f.ir = 1.0 / rho; f.gir = 0.4 / rho; f.hq2 = 0.5 * (f.U * f.U + f.V * f.V); f.e = rho * th / 0.4;
        Source s;
        for (int k = 0; k < 4; ++k) { s.xx[k] = amp * amp * u(); s.xy[k] = amp * amp * u(); s.yy[k] = amp * amp * u(); }
        const double a = std::fabs(f.U) + std::fabs(f.V) + 2.0 * std::sqrt(th);
        double s1 = (std::fabs(f.rx) + std::fabs(f.ry)) / rho + (std::fabs(f.Ux) + std::fabs(f.Uy) + std::fabs(f.Vx) + std::fabs(f.Vy)) / a +
                    (std::fabs(f.ex) + std::fabs(f.ey)) / (rho * a * a), s2 = 0.0;
        for (int k = 0; k < 4; ++k)
            s2 += (std::fabs(s.xx[k]) + std::fabs(s.xy[k]) + std::fabs(s.yy[k])) / (rho * (k == 0 ? 1.0 : k == 3 ? a * a : a));
        double o[4];
        const double E = f.e + rho * f.hq2;
        n.add(euler_second_split(T.r, s, f, E, o), 64.0 * (a * 0.25) * (a * 0.25) * (s1 * s1 + s2));
        Source z;
        memset(&z, 0, sizeof z);
        EulerFirst<double> e = f;
        e.rx = e.ry = e.Ux = e.Uy = e.Vx = e.Vy = e.ex = e.ey = 0.0;
        if (!euler_second_split(T.r, z, e, E, o)) n.bad++;
        z.bits = 1 << (it & 3);
        if (euler_second_split(T.r, z, e, E, o)) n.bad++;       // a rough variable
        z.bits = 0;
        (it & 4 ? z.xx : it & 8 ? z.xy : z.yy)[it & 3] = it & 16 ? 1e39 : NAN;
        if (euler_second_split(T.r, z, e, E, o)) n.bad++;       // out of range
    }
    n.print("wtt");
}

// the bits of segment_parts: first differences, third differences and the derivative rows' first
// differences, one of them scaled over its bound and the others far below theirs
static void segment_choice()
{
    const Table T(0.25);
    const char* names[3] = {"first_differences", "third_differences", "derivative_rows"};
    for (int what = 0; what < 3; ++what) {
        Tally n;
        for (int it = 0; it < 20000; ++it) {
            const int k = it & 1 ? 3 : 0;                       // density or energy
            double rec[RG::n];
            for (double& x : rec) x = 0.0;
            for (int y = 0; y < 5; ++y) { rec[(RV * 4 + 0) * RG::pa + y] = 1.0; rec[(RV * 4 + 3) * RG::pa + y] = 2.5; }
            for (int f = 0; f < 2; ++f)
                for (int y = 0; y < 3; ++y) { rec[8 * RG::pa + (f * 4 + 0) * RG::pb + y] = 2.0; rec[8 * RG::pa + (f * 4 + 3) * RG::pb + y] = 4.0; }
            const double scale = k ? 2.5 : 1.0, amp = scale * std::exp(u(-6.0, 0.0));
            double* v = rec + (RV * 4 + k) * RG::pa;
            double* d = rec + (RN * 4 + k) * RG::pa;
            double x = 0.0;
            if (what == 0) {                                    // a ramp: no third differences
                for (int y = 0; y < 5; ++y) v[y] += amp * (y - 2);
                x = amp / (0.125 * scale);
            } else if (what == 1) {                             // third differences alternate: v = c (-1)^y, t = 4 c
                for (int y = 0; y < 5; ++y) v[y] += (y & 1 ? -1.0 : 1.0) * amp / 32.0;
                const double t = amp / 4.0, first = amp / 16.0, s = std::fabs(v[2]);
                x = std::max(t / (s / 64.0), first / (0.125 * s));
            } else {
                for (int y = 0; y < 5; ++y) d[y] = amp * (y - 2);
                x = amp / (0.125 * scale);
            }
            double part[kParts];
            segment_parts(T.r, rec, RG::pa, RG::pb, RG::pc, 0, 1, 1.0, 0, 4, part, 1);
            const SegmentPoint src{T.r, rec, RG::pa, RG::pb, RG::pc, 0, 1, kGauss, 1.0, 0.5, 1, part, 1, FK_PIDY};
            const int rough = src.rough();
            n.add(!(rough >> k & 1), x);
            if (rough & ~(1 << k)) n.bad++;
        }
        n.print(names[what]);
    }
}

static void tangential_slope_choice()
{
    const Table T(0.25, 1e-3);
    Tally n;
    for (int it = 0; it < 40000; ++it) {
        const double amp = std::exp(u(-6.0, 0.0)), v0 = u(0.5, 1.5), vm = v0 + amp * u(), vp = v0 + amp * u();
        const double a = v0 - vm, b = vp - v0, e0 = a * a + 1e-3, e1 = b * b + 1e-3, z = std::fabs(e0 - e1);
        const double w0 = 1.0 + z / e0, w1 = 1.0 + z / e1, c = (a + b) - 2.0 * (w0 * a + w1 * b) / (w0 + w1);
        double s2;
        // (the scale's word stands for its power of two and leading bits; the correction's word is compared with it)
        const bool got = tang_weno3_small(T.r, vm, v0, vp, 1e-3, hi_abs(v0), s2);
        n.add(got, std::max(std::fabs(c) / (v0 / 2048.0), std::max(std::fabs(a + b), std::fabs(b - a)) / (2.0 * v0)), 0.1);
    }
    n.print("tangential_slope");
}

static void row_choice()
{
    Tally n, s;
    for (int it = 0; it < 40000; ++it) {
        const double scale = std::ldexp(u(1.0, 2.0), (int)u(-34.0, 30.0)), eps = std::ldexp(u(1.0, 2.0), (int)u(-34.0, 30.0));
        double x[5];
        const double amp = scale * std::exp(u(-9.0, 0.0));
        double m = 0.0;
        for (double& y : x) { y = amp * u(); m = std::max(m, std::fabs(y)); }
        const double s3 = scale * u(-1.5, 1.5);
        const bool in = scale >= 0x1p-30 && scale < 0x1p25 && eps >= 0x1p-30 && eps < 0x1p25;
        const bool got = split_ok(hi_abs(scale), eps, x[0], x[1], x[2], x[3], x[4], s3);
        n.add(got, in ? std::max(128.0 * m / scale, std::fabs(s3) / scale) : 2.0);
        s.add(split_scale_ok(hi_abs(scale), eps), in ? 0.5 : 2.0);
        if (split_ok(hi_abs(scale), eps, x[0], NAN, x[2], x[3], x[4], s3)) n.bad++;
    }
    n.print("row");
    s.print("scale");
}

int main()
{
    slope_choice();
    wtt_choice();
    segment_choice();
    tangential_slope_choice();
    row_choice();
    return 0;
}
