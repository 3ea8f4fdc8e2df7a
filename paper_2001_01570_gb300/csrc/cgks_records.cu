// cgks_records.cu -- the face-row records of one stage: the normal
// reconstruction of every face row of a grid (linear compact reconstruction,
// Sec. 3.2, Eq. recons-8th-val; nonlinear WENO-Z left and right states with
// their slopes, Sec. 3.3), computed once per row and written to global memory,
// where the flux kernels of all tiles that share the row read it.
//
// A record holds 7 fields x 4 variables (face frame: density, normal momentum,
// tangential momentum, energy): RV, RN, RNN (P7, P7_n, P7_nn) and, for the rows
// the non-equilibrium states are needed on, RL, RR (WENO-Z values) and RLN, RRN
// (their normal slopes).  x-face rows: faces 0..nx, rows -2..ny+1; y-face rows
// (2D): faces 0..ny, columns -2..nx+1.  Ghost cells of the stencils are the
// boundary conditions applied on the fly: x-boundaries first, then y, so the
// corners match the oracle's ghost layers.
#include "cgks_records.cuh"

namespace cgks {

// in global memory: lanes that read different words of constant memory are served one by one
static __device__ const ReconTab kReconTab = make_recon_tab();

// CHAR = 0: conservative variables, one (record, variable) per thread;
// CHAR = 1: characteristic variables, one (record, field) per lane of a quad.
// The reconstruction order is per grid (a uniform branch per chunk).
// Bound by the FP64 unit and FP32 issue together: about 55 FP64 instructions of 68
// cycles per warp (differences, linear reconstruction, the sums that bring the
// corrections back) beside some 1,900 FP32 and integer ones of the split WENO-Z
// pair (cgks_split.cuh); rows that fail split_ok take 240 more FP64 instructions.
// Measured per stage on the 2048^2 vortex: 15.73 ms with the pair in FP64, 3.74 ms now;
// 512^2: 1.010 -> 0.257 ms; 64^2 (two warps per FP64 unit): 24 -> 14.3 us.
// Characteristic mode with a thread per row ran 600 FP64 instructions and four WENO-Z pairs
// in one chain (401 cells in 1D: 78 us; a lane per field, and only the grid's own row of the
// five a 1D stencil would take: 41 us; the stencil mapped once: 26; a cell per lane: 24.7;
// 200x50: 99 -> 58 us).  Two lanes per row, one for each side of the face, changed nothing
// on small grids (100 cells in 1D: 69.1 and 69.4 us per step).
// CTAs of 128 threads, four per SM: one of 256 left a small grid's items on half
// of the SMs (100 cells in 1D: 24.7 us; spread over twice the CTAs: 20.9, 12.6 now).
// Three, four, five per SM: 2048^2 3.98, 3.73, 3.78 ms; 512^2 272, 258, 256 us.
template <int STAGE, int CHAR>
__global__ void __launch_bounds__(kRecordChunk, 4) records_kernel(const GridDev* __restrict__ grids,
                                                                    const TileRef* __restrict__ chunks, int nchunks,
                                                                    const int* __restrict__ dcount)
{
    __shared__ double s_tab[2 * RK_N];
    for (int i = threadIdx.x; i < 2 * RK_N; i += blockDim.x) s_tab[i] = kReconTab.v[i / RK_N][i % RK_N];
    __syncthreads();
    const double one = ((volatile const double*)s_tab)[RK_ONE];
    const double nzero = ((volatile const double*)s_tab)[RK_NZERO];
    wait_previous();
    if (dcount) nchunks = *dcount;   // queue length in device memory (a server's patched queue)
    for (int ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const TileRef tr = chunks[ch];
        const GridDev& G = grids[tr.grid];
        if (G.ctrl->done) continue;
        const double* src = (STAGE == 1) ? G.buf[G.ctrl->par] : G.ws;
        const size_t PL = (size_t)G.nx * G.ny;
        const int nrec = record_work_rows(G.nx, G.ny, G.dim);
        const int item = tr.x0 + (int)threadIdx.x;
        if (item >= 4 * nrec) continue;
        if (!CHAR) {
            const int k = item / nrec;
            if (G.order == 6) cons_row<6>(RegK{s_tab + RK_N, one, nzero}, G, src, PL, item - k * nrec, k);
            else cons_row<8>(RegK{s_tab, one, nzero}, G, src, PL, item - k * nrec, k);
        } else {
            const unsigned quad = 0xfu << (threadIdx.x & 28);
            if (G.order == 6) char_row_quad<6>(RegK{s_tab + RK_N, one, nzero}, G, src, PL, item >> 2, item & 3, quad);
            else char_row_quad<8>(RegK{s_tab, one, nzero}, G, src, PL, item >> 2, item & 3, quad);
        }
    }
    release_next();
}

std::vector<TileRef> record_chunks(int nx, int ny, int dim, int grid)
{
    const long long items = 4LL * record_work_rows(nx, ny, dim);
    std::vector<TileRef> c;
    for (long long s = 0; s < items; s += kRecordChunk) c.push_back(TileRef{grid, (int)s, 0, 0});
    return c;
}

cudaError_t launch_records(int stage, int char_vars, const GridDev* grids, const TileRef* chunks, int nchunks,
                           int nblocks, cudaStream_t st, const int* dcount)
{
    if (nchunks <= 0 || nblocks <= 0) return cudaSuccess;
    auto* kernel = char_vars ? (stage == 1 ? records_kernel<1, 1> : records_kernel<2, 1>)
                             : (stage == 1 ? records_kernel<1, 0> : records_kernel<2, 0>);
    return launch_chained(kernel, nblocks, kRecordChunk, 0, st, grids, chunks, nchunks, dcount);
}

}  // namespace cgks
