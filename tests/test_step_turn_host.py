"""The end of a step and the start of the next as one thread runs them (csrc/cgks_control.cuh), on the host: a
state without a usable time step is an error of the step that is asked of it, not of the step that led to it."""
import os
import subprocess

from conftest import ROOT

SRC = r'''
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#define CGKS_OPCOUNT_HOST 1
using std::isinf;
inline double __drcp_rn(double x) { return 1.0 / x; }
inline double __ddiv_rn(double a, double b) { return a / b; }
inline double __dmul_rn(double a, double b) { return a * b; }
inline double __dadd_rn(double a, double b) { return a + b; }
inline double __dsub_rn(double a, double b) { return a - b; }
inline double __dsqrt_rn(double a) { return std::sqrt(a); }
inline long long __double_as_longlong(double x) { long long b; memcpy(&b, &x, 8); return b; }
inline double __longlong_as_double(long long b) { double x; memcpy(&x, &b, 8); return x; }
template <class T> T __shfl_xor_sync(unsigned, T v, int) { return v; }
template <class T> void atomicMax(T*, T) {}
inline void atomicOr(int*, int) {}
inline long long max(long long a, long long b) { return a > b ? a : b; }
struct { int x = 0; } threadIdx;
#include "cgks_control.cuh"
using namespace cgks;
static void speeds(Ctrl& c, double x, double y) { c.amax_bits[0] = __double_as_longlong(x); c.amax_bits[1] = __double_as_longlong(y); }
static void show(const Ctrl& c) { printf("%d %d %d %lld %.17g %.17g\n", c.status, c.done, c.par, (long long)c.steps, c.t, c.dt); }
int main()
{
    for (double bad : {(double)INFINITY, 0.0})
        for (double t_end : {0.0, 0.25}) {
            GridDev G;
            memset(&G, 0, sizeof G);
            G.dim = 2; G.dx = G.dy = 1.0; G.cfl = 0.5;
            Ctrl c;
            memset(&c, 0, sizeof c);
            c.steps_target = -1; c.t_end = t_end;
            speeds(c, 2.0, 1.0);
            begin_step(G, &c);                  // dt = 0.25
            show(c);
            speeds(c, bad, bad);
            turn_step(G, &c);                   // the step is taken; the state it leads to has no dt
            show(c);
            turn_step(G, &c);                   // a step asked of that state
            show(c);
            Ctrl d = c;
            d.status = d.done = 0;
            speeds(d, bad, bad);
            begin_step(G, &d);                  // or asked by the next call
            show(d);
        }
    return 0;
}
'''


def test_a_state_without_a_time_step_is_the_next_steps_error(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    exe = str(tmp_path / "t")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-std=c++17", "-w", "-I", cuda, "-I", os.path.join(ROOT, "paper_2001_01570_gb300", "csrc"), "-o", exe,
                    str(src)], check=True)
    out = [ln.split() for ln in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]
    err = "5"                                                # CGKS_E_NONPHYSICAL
    for k, t_end in enumerate((0.0, 0.25, 0.0, 0.25)):
        first, taken, asked, call = out[4 * k:4 * k + 4]
        assert first == ["0", "0", "0", "0", "0", "0.25"]
        assert taken[:5] == ["0", str(int(t_end > 0)), "1", "1", "0.25"]     # done where t_end is reached
        if t_end > 0:
            assert asked == taken and call[0] == "0" and call[1] == "1"
        else:
            assert asked[:5] == [err, "1", "1", "1", "0.25"] and call[:2] == [err, "1"]
