// cgks_control.cu -- step-control kernels (CFL time step, step begin/end),
// state layout conversions and the stage-kernel dispatcher.
#include "cgks_control.cuh"
#include "cgks_internal.h"
#include "../../include/cgks.h"
#include <math.h>

namespace cgks {

#define CGKS_DECLARE_TILE(w, h)                                                                          \
    cudaError_t launch_stage_##w##x##h(int, const GridDev*, const TileRef*, int, int, cudaStream_t, const int*); \
    size_t smem_##w##x##h(int);
CGKS_FOR_EACH_TILE(CGKS_DECLARE_TILE)
#undef CGKS_DECLARE_TILE

cudaError_t launch_stage(int shape, int stage, const GridDev* grids, const TileRef* tiles, int ntiles, int nblocks,
                         cudaStream_t st, const int* dcount)
{
    switch (shape) {
#define CGKS_LAUNCH_CASE(w, h) \
    case TILE_##w##x##h: return launch_stage_##w##x##h(stage, grids, tiles, ntiles, nblocks, st, dcount);
    CGKS_FOR_EACH_TILE(CGKS_LAUNCH_CASE)
#undef CGKS_LAUNCH_CASE
    default: return cudaErrorInvalidValue;
    }
}

size_t stage_smem_bytes(int shape, int stage)
{
    switch (shape) {
#define CGKS_SMEM_CASE(w, h) \
    case TILE_##w##x##h: return smem_##w##x##h(stage);
    CGKS_FOR_EACH_TILE(CGKS_SMEM_CASE)
#undef CGKS_SMEM_CASE
    default: return 0;
    }
}

__global__ void begin_step_kernel(const GridDev* grids, int n, int reset)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    Ctrl* C = grids[g].ctrl;
    begin_step(grids[g], C);
    if (reset && !C->done) C->amax_bits[0] = C->amax_bits[1] = 0;
}

__global__ void end_step_kernel(const GridDev* grids, int n)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n) end_step(grids[g].ctrl);
}

// speed maxima of the current state (after a state is set)
__global__ void cfl_kernel(const GridDev* grids, int gidx)
{
    const GridDev& G = grids[gidx];
    const size_t PL = (size_t)G.nx * G.ny;
    const double* W = G.buf[G.ctrl->par];
    SpeedMax s;
    for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < PL; c += (size_t)gridDim.x * blockDim.x)
        s.cell(G, W[c], W[PL + c], W[2 * PL + c], W[3 * PL + c]);
    speed_max_warp(G.ctrl, s);
}

__device__ __forceinline__ void set_ctrl(Ctrl* c, double t, double t_end, long long steps_target, int reset,
                                         long long steps0)
{
    if (reset) {
        c->t = t;
        c->steps = steps0;
        c->status = 0;
        c->done = 0;
        c->par = 0;
        c->dt = 0.0;
        c->amax_bits[0] = c->amax_bits[1] = 0;
        c->arrived = 0;
    } else if (!c->status) {
        // a new request may continue a solve that was stopped by its step target or t_end
        c->done = 0;
    }
    c->t_end = t_end;
    c->steps_target = steps_target;
}

__global__ void set_ctrl_kernel(Ctrl* c, double t, double t_end, long long steps_target, int reset, long long steps0)
{
    set_ctrl(c, t, t_end, steps_target, reset, steps0);
}

// a batch call continues every grid of the batch that has no error: no step
// target, no end time
__global__ void batch_resume_kernel(const GridDev* grids, int n)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    Ctrl* c = grids[g].ctrl;
    if (!c->status) c->done = 0;
    c->t_end = 0.0;
    c->steps_target = -1;
}

// The state of a 1D grid (6 planes: rho, rhoU, rhoE, their x-gradients) into the internal
// 2D layout, with the state's speed maxima and, run by one CTA (one_cta), the control block of a solve
// that starts there; before several CTAs a launch of its own has reset the block.
__global__ void __launch_bounds__(256) set_state_1d_kernel(const GridDev* grids, const double* src, double t,
                                                           long long steps0, int one_cta)
{
    const GridDev& G = grids[0];
    Ctrl* C = G.ctrl;
    if (one_cta) {
        if (threadIdx.x == 0) {
            set_ctrl(C, t, 0.0, -1, 1, steps0);
            __threadfence_block();
        }
        __syncthreads();
    }
    const int nx = G.nx;
    double* dst = G.buf[0];
    SpeedMax s;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nx; i += gridDim.x * blockDim.x) {
        double v[6];
#pragma unroll
        for (int p = 0; p < 6; ++p) v[p] = src[(size_t)p * nx + i];
        const int map[12] = {0, 1, -1, 2, 3, 4, -1, 5, -1, -1, -1, -1};
#pragma unroll
        for (int p = 0; p < 12; ++p) dst[(size_t)p * nx + i] = map[p] < 0 ? 0.0 : v[map[p]];
        s.cell(G, v[0], v[1], 0.0, v[2]);
    }
    speed_max_warp(C, s);
}

// The current state, whichever buffer holds it, as the caller's planes.
__global__ void get_state_kernel(const GridDev* grids, double* dst)
{
    const GridDev& G = grids[0];
    const double* src = G.buf[G.ctrl->par & 1];
    const size_t PL = (size_t)G.nx * G.ny, n = (G.dim == 1 ? 6 : 12) * PL;
    const int map[6] = {0, 1, 3, 4, 5, 7};
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t p = i / PL;
        dst[i] = src[G.dim == 1 ? (size_t)map[p] * PL + (i - p * PL) : i];
    }
}

cudaError_t launch_begin_step(const GridDev* grids, int n, cudaStream_t st, int reset)
{
    begin_step_kernel<<<(n + 127) / 128, 128, 0, st>>>(grids, n, reset);
    return cudaGetLastError();
}

cudaError_t launch_end_step(const GridDev* grids, int n, cudaStream_t st)
{
    end_step_kernel<<<(n + 127) / 128, 128, 0, st>>>(grids, n);
    return cudaGetLastError();
}

cudaError_t launch_cfl(const GridDev* grids, int gidx, const GridDev& host, cudaStream_t st)
{
    const size_t cells = (size_t)host.nx * host.ny;
    int blocks = (int)((cells + 255) / 256);
    if (blocks > 1024) blocks = 1024;
    cfl_kernel<<<blocks, 256, 0, st>>>(grids, gidx);
    return cudaGetLastError();
}

cudaError_t launch_set_ctrl(Ctrl* c, double t, double t_end, long long steps_target, int reset, cudaStream_t st,
                            long long steps0)
{
    set_ctrl_kernel<<<1, 1, 0, st>>>(c, t, t_end, steps_target, reset, steps0);
    return cudaGetLastError();
}

cudaError_t launch_batch_resume(const GridDev* grids, int n, cudaStream_t st)
{
    batch_resume_kernel<<<(n + 127) / 128, 128, 0, st>>>(grids, n);
    return cudaGetLastError();
}

// A thread per cell; one CTA's worth in one launch (a batch of small grids is set one by one), more after
// a launch for the control block.  A whole call with one CTA at any size / so: 256 cells 14.7 / 14.9 us,
// 512 17.9 / 16.5, 2048 33 / 16, 2^20 10766 / 89 (four launches of a kind each: 24, 23, 23, 136).
cudaError_t launch_set_state_1d(const GridDev* grids, const GridDev& host, const double* src, double t, long long steps0,
                                cudaStream_t st)
{
    const int blocks = host.nx < 1024 * 256 ? (host.nx + 255) / 256 : 1024;
    if (blocks > 1) {
        const cudaError_t e = launch_set_ctrl(host.ctrl, t, 0.0, -1, 1, st, steps0);
        if (e != cudaSuccess) return e;
    }
    set_state_1d_kernel<<<blocks, 256, 0, st>>>(grids, src, t, steps0, blocks == 1);
    return cudaGetLastError();
}

cudaError_t launch_get_state(const GridDev* grids, const GridDev& host, double* dst, cudaStream_t st)
{
    const size_t n = (size_t)(host.dim == 1 ? 6 : 12) * host.nx * host.ny;
    const size_t blocks = (n + 255) / 256;
    get_state_kernel<<<(int)(blocks < 1216 ? blocks : 1216), 256, 0, st>>>(grids, dst);
    return cudaGetLastError();
}

}  // namespace cgks
