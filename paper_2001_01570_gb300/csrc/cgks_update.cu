// cgks_update.cu -- the cell update of one stage of the two-stage fourth-order
// step (Sec. 2.2, Eq. step-hyper-1) from the face results the flux kernel wrote
// (each face evaluated once): cell averages by the Gauss-averaged fluxes, cell-
// averaged gradients by the Gauss theorem on the interface states (Sec. 3.1,
// Eq. compact-deriv-1).
//   stage 1: W* = W - (dt/2 F + dt^2/8 F_t) differences,  grad* from W(dt/2);
//            R  = W - (dt F + dt^2/6 F_t) differences,    R_grad from W(dt)
//            (the face results already carry the dt factors and the Gauss weights)
//   stage 2: W^{n+1} = R - dt^2/3 F_t* differences, grad^{n+1} = R_grad + dt^2/3
//            differences of W_tt*; the signal speeds of W^{n+1}; the grid's last chunk
//            to finish ends the step and starts the next one (its dt)
#include "cgks_control.cuh"
#include "cgks_update.cuh"

namespace cgks {

// One CTA per chunk of kCellChunk cells of one grid; CPT cells per thread, the cells of a
// thread kCellChunk / CPT apart so that every pass of the CTA reads and writes contiguous
// cells.
// What bounds it: HBM on large grids; on small ones the chain of one thread's 80 (stage 1)
// to 150 FP64 instructions per cell, so those run one cell per thread.  Measured, stage 1 / 2,
// before (four cells per thread, chunks of 256, two quotients per cell, the step's end and
// start in launches of their own) and now: 64^2 27 / 29 -> 10.3 / 14.5 us (5 of them the event
// pair's), 2048^2 537 / 693 -> 543 / 561 us.
template <int STAGE, int CPT>
__global__ void __launch_bounds__(kCellChunk / CPT) update_kernel(const GridDev* __restrict__ grids,
                                                                  const TileRef* __restrict__ chunks, int nchunks,
                                                                  const int* __restrict__ dcount)
{
    constexpr int NT = kCellChunk / CPT;
    wait_previous();
    if (dcount) nchunks = *dcount;   // queue length in device memory (a server's patched queue)
    for (int ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const TileRef tr = chunks[ch];
        const GridDev& G = grids[tr.grid];
        Ctrl* C = G.ctrl;
        if (C->done) continue;                      // uniform over the block (one grid per chunk)
        const int par = C->par;
        const long long PL = (long long)G.nx * G.ny;
        // dt has been taken from the maxima of the state the step started from
        if (STAGE == 1 && tr.x0 == 0 && threadIdx.x == 0) C->amax_bits[0] = C->amax_bits[1] = 0;
        SpeedMax smax;
#pragma unroll
        for (int m = 0; m < CPT; ++m) {
            const long long cell = (long long)tr.x0 + threadIdx.x + m * NT;
            if (cell < PL) update_cell<STAGE>(G, par, cell, smax);
        }
        if (STAGE == 2) {
            speed_max_warp(C, smax);
            __syncthreads();
            if (threadIdx.x == 0) {
                // every chunk's maxima and status are in the control block before its arrival is
                __threadfence();
                const int last = (int)((PL + kCellChunk - 1) / kCellChunk) - 1;
                if (atomicAdd(&C->arrived, 1) == last) {
                    __threadfence();
                    C->arrived = 0;
                    turn_step(G, C);
                }
            }
        }
    }
    release_next();
}

std::vector<TileRef> cell_chunks(int nx, int ny, int grid)
{
    const long long cells = (long long)nx * ny;
    std::vector<TileRef> c;
    for (long long s = 0; s < cells; s += kCellChunk) c.push_back(TileRef{grid, (int)s, 0, 0});
    return c;
}

cudaError_t launch_update(int stage, const GridDev* grids, const TileRef* chunks, int nchunks, int nblocks,
                          cudaStream_t st, const int* dcount, int cpt)
{
    if (nchunks <= 0 || nblocks <= 0) return cudaSuccess;
    auto* kernel = stage == 1 ? (cpt == 4 ? update_kernel<1, 4> : cpt == 2 ? update_kernel<1, 2> : update_kernel<1, 1>)
                              : (cpt == 4 ? update_kernel<2, 4> : cpt == 2 ? update_kernel<2, 2> : update_kernel<2, 1>);
    const int threads = kCellChunk / (cpt == 4 ? 4 : cpt == 2 ? 2 : 1);
    return launch_chained(kernel, nblocks, threads, 0, st, grids, chunks, nchunks, dcount);
}

}  // namespace cgks
