// cgks_control.cuh -- the end and the start of a grid's time step, run by one thread:
// the last chunk of the stage-2 update (cgks_update.cu) and the control kernels
// (cgks_control.cu).
#pragma once
#include "cgks_internal.h"
#include "../../include/cgks.h"

namespace cgks {

// whether a step can be taken with dt
__device__ __forceinline__ bool usable_dt(double dt) { return dt > 0.0 && !isinf(dt); }

// Start of a step: dt = CFL * (min over cells of dx/(|U|+c+2 nu/dx), dy/(|V|+c+2 nu/dy)) of the
// current state, clipped so that t does not pass t_end; marks a grid that is finished.  A
// function of the control block alone that it leaves valid: running it again before the
// step gives the same dt.  A state without a usable dt is an error if a step is asked of it: right away
// (raise), or at the end of the step that was begun with it (turn_step, which cannot know whether
// another step follows).
template <class C_>
__device__ __forceinline__ void begin_step(const GridDev& G, C_* C, bool raise = true)
{
    if (C->done) return;
    if (C->status) { C->done = 1; return; }
    if (C->steps_target >= 0 && C->steps >= C->steps_target) { C->done = 1; return; }
    if (C->t_end > 0.0 && C->t >= C->t_end) { C->done = 1; return; }
    double d = G.dx / __longlong_as_double((long long)C->amax_bits[0]);
    if (G.dim != 1) d = fmin(d, G.dy / __longlong_as_double((long long)C->amax_bits[1]));
    double dt = G.cfl * d;
    if (!usable_dt(dt)) {
        if (raise) { C->status |= CGKS_E_NONPHYSICAL; C->done = 1; }
        else C->dt = dt;
        return;
    }
    if (C->t_end > 0.0 && C->t + dt > C->t_end) dt = C->t_end - C->t;
    C->dt = dt;
}

// End of a step: the new state becomes current unless a kernel raised an error.
template <class C_>
__device__ __forceinline__ void end_step(C_* C)
{
    if (C->done) return;
    if (C->status) { C->done = 1; return; }
    C->par ^= 1;
    C->t += C->dt;
    C->steps += 1;
}

// The end of a step and the start of the next, the control block read once: as field after
// field between their branches the reads took a memory latency each (with the rest of the last
// chunk's end 9,400 cycles).
__device__ __forceinline__ void turn_step(const GridDev& G, volatile Ctrl* C)
{
    Ctrl c;
    c.dt = C->dt; c.t = C->t; c.t_end = C->t_end; c.amax_bits[0] = C->amax_bits[0]; c.amax_bits[1] = C->amax_bits[1];
    c.status = C->status; c.done = C->done; c.par = C->par; c.steps = C->steps; c.steps_target = C->steps_target;
    if (!usable_dt(c.dt)) c.status |= CGKS_E_NONPHYSICAL;   // the step just run had none: the state before it stays
    end_step(&c);
    begin_step(G, &c, false);
    C->dt = c.dt; C->t = c.t; C->status = c.status; C->done = c.done; C->par = c.par; C->steps = c.steps;
}

// A warp's speed maxima into the grid's control block (positive doubles compare as their
// bits); the maximum is read first, since few warps raise it.
__device__ __forceinline__ void speed_max_warp(Ctrl* C, SpeedMax& s)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int d = 0; d < 2; ++d) {   // as integers, off the FP64 unit
            const long long v = __double_as_longlong(s.a[d]);
            s.a[d] = __longlong_as_double(max(v, __shfl_xor_sync(0xffffffffu, v, o)));
        }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const unsigned long long v = (unsigned long long)__double_as_longlong(s.a[d]);
            if (v > ((volatile Ctrl*)C)->amax_bits[d]) atomicMax(&C->amax_bits[d], v);
        }
    if (s.bad) atomicOr(&C->status, (int)CGKS_E_NONPHYSICAL);
}

}  // namespace cgks
