// Records in characteristic variables on the host, for gases whose speed of sound is 2^-j of the unit of
// velocity: random rows of four cells in, the record's fields out, in binary on stdout.  Built twice, with
// the pairs of FP32 (CGKS_SPLIT_CHECK) and in FP64 alone; the test compares the two outputs.
//
// Per row: the WENO-Z values of both sides (8), then the scales they are measured against (rho, and
// rho c for the momenta, rho c^2).
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

using namespace cgks;

int main()
{
    const ReconTab T = make_recon_tab();
    const RegK r{T.v[0], 1.0, -0.0};
    std::mt19937_64 g(7);
    std::uniform_real_distribution<double> u(-1.0, 1.0);
    for (int j = 0; j <= 12; ++j)
        for (int lev = 0; lev < 4; ++lev)
            for (int n = 0; n < 500; ++n) {
                // a shear layer that the grid does not resolve, in a gas at rest otherwise
                const double c = std::ldexp(1.0, -j), amp = std::ldexp(c, -2 * lev), h = 0.01;
                double Q[4][4], N[4][4];
                for (int i = 0; i < 4; ++i) {
                    const double m = amp * u(g);
                    Q[0][i] = 1.0; Q[1][i] = 0.0; Q[2][i] = m; Q[3][i] = c * c / (1.4 * 0.4) + 0.5 * m * m;
                    const double dm = amp * u(g) / h;
                    N[0][i] = 0.0; N[1][i] = 0.0; N[2][i] = dm; N[3][i] = m * dm;
                }
                double out[16] = {1, c, c, c * c, 1, c, c, c * c, 1, c, c, c * c, 1, c, c, c * c};
                char_record<8>(r, 1.4, Q, N, h, 1.0 / h, 0x1p-29, true, [&](int f, int k, double v) {
                    if (f == RL) out[k] = v;
                    if (f == RR) out[4 + k] = v;
                });
                fwrite(out, sizeof(double), 16, stdout);
            }
    return 0;
}
