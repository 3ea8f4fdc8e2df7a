// The flux kernel's Gauss-point evaluation on the host over units of density, velocity and length:
// the records of random smooth face segments in, the point's results out, in binary on stdout.  Built
// twice, with the forms in pairs of FP32 and the choices that guard them (CGKS_SPLIT_CHECK) and in FP64
// alone; the test compares the two outputs.
//
// Per point: kN results (stage 1: Fb, Ft, Wm, Wb; stage 2: Wtt), then the kN scales they are measured
// against (rho a^k fluxes, over dt for F_t; the state; the state over dt^2).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#define CGKS_OPCOUNT_HOST 1
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

constexpr int kN = 20;
using RG = RecGroups<1, 1>;

struct Case { int er, ea, el; double amp; bool viscous; };

static void segment(std::mt19937_64& g, const Case& c)
{
    std::uniform_real_distribution<double> u01(0.0, 1.0);
    auto u = [&] { return u01(g); };
    const double rho = std::ldexp(0.7 + 0.6 * u(), c.er), a = std::ldexp(0.7 + 0.6 * u(), c.ea), dx = std::ldexp(0.7 + 0.6 * u(), c.el);
    const double dy = dx * (0.7 + 0.6 * u()), U = 1.6 * u() - 0.8, V = 1.6 * u() - 0.8;
    const double s[4] = {rho, rho * a, rho * a, rho * a * a}, b[4] = {1.0, U, V, 2.5 + 0.5 * (U * U + V * V)};
    double k1[4], k2[4], ph[4], jump[4];
    for (int k = 0; k < 4; ++k) { k1[k] = 0.2 + 0.5 * u(); k2[k] = 0.2 + 0.5 * u(); ph[k] = 6.28 * u(); jump[k] = c.amp * 1e-3 * (u() - 0.5); }
    double rec[RG::n];
    // d-th derivative along the normal (per cell) of variable k on row y
    auto f = [&](int k, int d, double y) {
        const double x = ph[k] + k2[k] * y;
        return s[k] * (d == 0 ? b[k] + c.amp * std::sin(x) : d == 1 ? c.amp * k1[k] * std::cos(x) : -c.amp * k1[k] * k1[k] * std::sin(x));
    };
    for (int k = 0; k < 4; ++k) {
        for (int y = -2; y <= 2; ++y) {
            rec[(RV * 4 + k) * RG::pa + y + 2] = f(k, 0, y);
            rec[(RN * 4 + k) * RG::pa + y + 2] = f(k, 1, y) / dx;
        }
        for (int y = -1; y <= 1; ++y)
            for (int side = 0; side < 2; ++side) {
                const double j = (side ? 0.5 : -0.5) * jump[k];
                rec[8 * RG::pa + ((side ? 4 : 0) + k) * RG::pb + y + 1] = f(k, 0, y) + s[k] * j;          // RL, RR
                rec[8 * RG::pa + ((side ? 12 : 8) + k) * RG::pb + y + 1] = (f(k, 1, y) + s[k] * j) / dx;  // RLN, RRN
            }
        rec[8 * RG::pa + 16 * RG::pb + k] = f(k, 2, 0.0) / dx / dx;
    }
    static_assert(RL == 3 && RR == 4 && RLN == 5 && RRN == 6);
    GridDev G;
    memset(&G, 0, sizeof G);
    G.dx = dx; G.dy = dy; G.inv_dx = 1.0 / dx; G.inv_dy = 1.0 / dy;
    G.gamma = 1.4; G.K = 3.0; G.eps_tau = 0.01; G.c_tau = 1.0; G.weno_eps = 1e-6;
    const double dt = 0.4 * std::min(dx, dy) / (a * (1.2 + std::fabs(U) + std::fabs(V)));
    G.mu = c.viscous ? 0.05 * rho * a * a * dt : 0.0;
    double t[FK_N];
    const FluxFixed fix = make_flux_fixed();
    for (int i = 0; i < FK_NFIX2; ++i) t[i] = fix.v[i];
    flux_table_tile(t, G, dt);
    const RegK r{t, 1.0, -0.0};
    double part[kParts];
    segment_parts(r, rec, RG::pa, RG::pb, RG::pc, 0, 1, G.inv_dx, 0, 4, part, 1);
    for (int gp = 0; gp < 2; ++gp) {
        const SegmentPoint src{r, rec, RG::pa, RG::pb, RG::pc, 0, 1, gp ? kGauss : -kGauss, r.k(FK_IDY), r.k(FK_HIDY), gp, part, 1, FK_PIDY};
        PointResult<1> o;
        PointResult<2> q;
        double out[2 * kN];
        if (!segment_point<1>(src, o) || !segment_point<2>(src, q)) { fprintf(stderr, "non-physical\n"); exit(1); }
        for (int k = 0; k < 4; ++k) {
            const double v[5] = {o.a[k], o.b[k], o.c[k], o.d[k], q.b[k]};
            const double z[5] = {s[k] * a, s[k] * a / dt, s[k], s[k], s[k] / dt / dt};
            for (int j = 0; j < 5; ++j) { out[4 * j + k] = v[j]; out[kN + 4 * j + k] = z[j]; }
        }
        fwrite(out, sizeof(double), 2 * kN, stdout);
    }
}

int main()
{
    std::mt19937_64 g(2024);
    for (int er : {-60, -50, -38, -30, -20, 0, 10, 13, 20})
        for (int ea : {-24, -12, 0, 10, 15, 20, 26, 30})
            for (int el : {-120, -60, -30, -23, -13, -7, 0, 10, 13, 17, 30, 33, 60, 120})
                for (int lev : {2, 3, 6, 10})
                    for (int n = 0; n < 6; ++n) segment(g, Case{er, ea, el, std::ldexp(1.0, -lev), n % 2 == 1});
    return 0;
}
