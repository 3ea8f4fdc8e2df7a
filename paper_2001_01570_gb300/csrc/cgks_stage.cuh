// cgks_stage.cuh -- the per-stage flux kernel of the two-stage fourth-order
// compact GKS (Sec. 2.2, Eq. step-hyper-1).  It runs after the record kernel
// (cgks_records.cu), which did the normal reconstruction of every face row of
// the grid once, and before the update kernel (cgks_update.cu), which applies
// the face results to the cells.
//
// One CTA owns a TX x TY tile of cells of one grid and runs, in shared memory:
//   phase 1  stage the face-row records the tile needs (its faces on its rows
//            and two rows either side) with asynchronous copies, for the CTA's
//            next tile while it works on this one where two buffers fit
//   phase 2  per face segment the tile owns (the x- and y-faces on the low side
//            of its cells; the grid's last faces have tiles of their own, so every
//            face is evaluated once) a pair of lanes.  Together they compute what
//            its two Gauss points share, two variables each, into the pair's slice
//            of shared memory: WENO-Z point values along the face over rows
//            j-2..j+2 (equilibrium) and j-1..j+1 (non-equilibrium states, with
//            their tangential slopes) and the parts of the quartic through the same
//            line averages.  Then each lane evaluates one point; their results are
//            exchanged by shuffles, averaged, weighted by the stage's time factors
//            and written to the face results, two variables per lane (stage 1: the
//            W* and R flux combinations and the interface states W(dt/2), W(dt);
//            stage 2: dt^2/3 F_t and dt^2/3 W_tt)
// What bounds it: the FP64 unit (68 cycles per warp instruction) with FP32 issue beside
// it: 792 (stage 1) and 690 FP64 instructions and some 20,000 others per 32 segments.  One
// thread per segment ran both points in turn with the first one's sums and the shared
// parts in registers (255 of them, 1.8 KB of spills once the FP32 pairs came in); one
// thread per point needs 168 and halves the chain of dependent instructions that a small
// grid waits for.  Measured per launch, stage 1 / 2: 2048^2 27.66 / 25.41 -> 17.8 / 14.4
// ms with this split, 14.0 / 12.2 now; 512^2 1.93 / 1.77 -> 1.14 / 0.94, 0.90 / 0.79 ms now;
// 64^2 155 / 138 -> 43 / 38, 37 / 34 us now.
// Coefficients (fixed, and the tile's grid and dt) come from the shared-memory
// table of cgks_flux.cuh; all arithmetic is in the register-only DFMA forms.
// The kernel is persistent: CTAs stride over a flattened tile queue that may
// span many grids of different sizes (each with its own dt in its Ctrl).
#pragma once
#include "cgks_segment.cuh"
#include "../../include/cgks.h"

#include <mutex>

namespace cgks {

// (in global memory: lanes that read different words of constant memory are served one by one, which
// with 2^(j/32) computed per CTA took 2,300 cycles at the start of every launch)
static __device__ const FluxFixed kFluxFixed = make_flux_fixed();

template <int TX, int TY, int STAGE>
__global__ void __launch_bounds__(kThreads, stage_ctas(TX, TY))
stage_kernel(const GridDev* __restrict__ grids, const TileRef* __restrict__ tiles, int ntiles,
             const int* __restrict__ dcount)
{
    using L = StageLayout<TX, TY, STAGE>;
    extern __shared__ double smem[];
    double* part = smem + L::buffers * L::n_rec + (threadIdx.x >> 1);   // [kParts][kPairs]: this pair's slice
    __shared__ double s_fk[FK_N];       // coefficient table (fixed part, then the tile's grid and dt)
    __shared__ int s_skip;
    const int tid = threadIdx.x;

    for (int i = tid; i < FK_NFIX2; i += kThreads) s_fk[i] = kFluxFixed.v[i];
    __syncthreads();
    const RegK r{s_fk, ((volatile const double*)s_fk)[FK_ONE], ((volatile const double*)s_fk)[FK_NZERO]};

    wait_previous();

    // ---------------- phase 1: a tile's face-row records (the record kernel wrote them for
    // every face row of the grid) into buffer `buf`: x-faces x0..x0+TX on rows y0-2..y0+TY+1,
    // y-faces y0..y0+TY on columns x0-2..x0+TX+1, each field on the rows it is read on; rows
    // beyond the grid's last ghost row are zero and unused.  Asynchronous 8-byte copies,
    // zero-filled where invalid.
    auto issue = [&](int tile, int buf) {
        const TileRef tr = tiles[tile];
        const GridDev& G = grids[tr.grid];
        const int nx = G.nx, ny = G.ny, x0 = tr.x0, y0 = tr.y0;
        const size_t sx = (size_t)(ny + 4) * (nx + 1), sy = (size_t)(nx + 4) * (ny + 1);
        const unsigned sbx = (unsigned)__cvta_generic_to_shared(smem + buf * L::n_rec), sby = sbx + 8u * L::n_rx;
        // group g of one orientation: plane p of the group is global plane p0 + p, its
        // local row q is record row base + q (records carry two ghost rows first)
        auto stage = [&](unsigned sbase, int sofs, int np, int plane, int F, int p0, const double* g, size_t gs,
                         int gfaces, int row0, int face0, int nface_max, int row_max, int nsmem) {
            const int n = np * plane;
            for (int idx = tid; idx < n; idx += kThreads) {
                const int p = idx / plane, rem = idx - p * plane;
                const int q = rem / F, fc = rem - q * F;
                bool valid = (face0 + fc <= nface_max) && (row0 + q <= row_max);
                if (!CGKS_IN_BOUNDS(sofs + idx < nsmem, G.ctrl)) continue;
                if (valid)
                    valid = CGKS_IN_BOUNDS(row0 + q >= 0 && face0 + fc >= 0 &&
                                               (size_t)(p0 + p) * gs + (size_t)(row0 + q) * gfaces + face0 + fc <
                                                   28 * gs,
                                           G.ctrl);
                const double* src = valid ? g + (size_t)(p0 + p) * gs + (size_t)(row0 + q) * gfaces + face0 + fc
                                          : G.recx;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(sbase + 8u * (unsigned)(sofs + idx)),
                             "l"(src), "r"(valid ? 8 : 0) : "memory");
            }
        };
        using RX = RecGroups<TY, TX + 1>;
        using RY = RecGroups<TX, TY + 1>;
        // x-faces: record rows y0 + 2 + (own row); group A starts two rows earlier, B one
        stage(sbx, 0, 8, RX::pa, TX + 1, 0, G.recx, sx, nx + 1, y0, x0, nx, ny + 3, RX::n);
        stage(sbx, 8 * RX::pa, 16, RX::pb, TX + 1, 4 * RL, G.recx, sx, nx + 1, y0 + 1, x0, nx, ny + 3, RX::n);
        stage(sbx, 8 * RX::pa + 16 * RX::pb, 4, RX::pc, TX + 1, 4 * RNN, G.recx, sx, nx + 1, y0 + 2, x0, nx, ny + 3,
              RX::n);
        stage(sby, 0, 8, RY::pa, TY + 1, 0, G.recy, sy, ny + 1, x0, y0, ny, nx + 3, RY::n);
        stage(sby, 8 * RY::pa, 16, RY::pb, TY + 1, 4 * RL, G.recy, sy, ny + 1, x0 + 1, y0, ny, nx + 3, RY::n);
        stage(sby, 8 * RY::pa + 16 * RY::pb, 4, RY::pc, TY + 1, 4 * RNN, G.recy, sy, ny + 1, x0 + 2, y0, ny, nx + 3,
              RY::n);
    };
    // the queue length: the kernel argument, or the int in device memory behind dcount (a server's
    // queue, patched between replays), read at each tile
    auto length = [&] { return dcount ? *(volatile const int*)dcount : ntiles; };

    // with two buffers the next tile's records are copied while this one's are used
    if (L::buffers == 2 && (int)blockIdx.x < length()) issue(blockIdx.x, 0);
    int buf = 0, held = -1;
    for (int tile = blockIdx.x; tile < length(); tile += gridDim.x) {
        __syncthreads();                              // the tile before is finished: table and buffer are free
        const TileRef tr = tiles[tile];
        const GridDev& G = grids[tr.grid];
        if (L::buffers == 1) issue(tile, 0);
        flux_table_grid(s_fk, G, tr.grid, held, s_skip);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        const double* rx = smem + buf * L::n_rec;     // x-face records, RecGroups<TY, TX+1>
        const double* ry = rx + L::n_rx;              // y-face records, RecGroups<TX, TY+1>
        if (L::buffers == 2) {
            if (tile + (int)gridDim.x < length()) issue(tile + gridDim.x, buf ^ 1);
            buf ^= 1;
        }
        if (s_skip) continue;
        const int nx = G.nx, ny = G.ny, x0 = tr.x0, y0 = tr.y0;

        // ---------------- phase 2: face segments, two Gauss points each
        bool bad = false;
        // the tile's own faces: x-faces x0..x0+TX-1 and y-faces y0..y0+TY-1 (a tile with
        // x0 = nx or y0 = ny has the grid's last faces alone); every face is evaluated by
        // exactly one tile
        constexpr int nseg = 2 * TX * TY;
        const size_t nfx = (size_t)ny * (nx + 1), nfy = (size_t)(ny + 1) * nx;
        const int gp = tid & 1;
        const unsigned pair = 3u << (tid & 30);         // the two lanes of this pair
        for (int item = tid >> 1; item < nseg; item += kPairs) {
            const bool xo = item < TX * TY;
            const int it = xo ? item : item - TX * TY, fl = it % TX, jl = it / TX;   // cell of the tile
            const double* rec;
            int pa, pb, pc, r0, rstride;
            double* out;
            size_t ostride, oidx;
            if (xo) {
                if (!((x0 + fl <= nx) && (y0 + jl < ny))) continue;
                rec = rx; pa = RecGroups<TY, TX + 1>::pa; pb = RecGroups<TY, TX + 1>::pb; pc = RecGroups<TY, TX + 1>::pc;
                r0 = jl * (TX + 1) + fl; rstride = TX + 1;
                out = G.facex; ostride = nfx; oidx = (size_t)(y0 + jl) * (nx + 1) + x0 + fl;
            } else {
                if (!((y0 + jl <= ny) && (x0 + fl < nx))) continue;
                rec = ry; pa = RecGroups<TX, TY + 1>::pa; pb = RecGroups<TX, TY + 1>::pb; pc = RecGroups<TX, TY + 1>::pc;
                r0 = fl * (TY + 1) + jl; rstride = TY + 1;
                out = G.facey; ostride = nfy; oidx = (size_t)(y0 + jl) * nx + x0 + fl;
            }
            // the segment's record window (rows -2..2 of group A, -1..1 of group B, 0 of group C)
            // and its output index
            if (!CGKS_IN_BOUNDS(r0 >= 0 && r0 + 4 * rstride < pa && r0 + 2 * rstride < pb && r0 < pc &&
                                    oidx < ostride,
                                G.ctrl))
                continue;
            __syncwarp(pair);   // the slice's reads of the segment before
            // the pair's lanes compute two variables' parts each, then a Gauss point each
            segment_parts(r, rec, pa, pb, pc, r0, rstride, r.k(xo ? FK_IDX : FK_IDY), 2 * gp, 2 * gp + 2, part, kPairs);
            __syncwarp(pair);
            const SegmentPoint src{r, rec, pa, pb, pc, r0, rstride, gp ? kGauss : -kGauss, r.k(xo ? FK_IDY : FK_IDX),
                                   r.k(xo ? FK_HIDY : FK_HIDX), gp, part, kPairs, xo ? FK_PIDY : FK_PIDX};
            PointResult<STAGE> o;
            bad |= !segment_point<STAGE>(src, o);
            // each lane averages and writes two variables: the other lane's sums for them come by
            // shuffle
            auto sum = [&](const double v[4], int m) {
                const double mine = gp ? v[2 + m] : v[m], theirs = gp ? v[m] : v[2 + m];
                return r.add(mine, __shfl_xor_sync(pair, theirs, 1));
            };
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const double a = sum(o.a, m), b = sum(o.b, m);
                double c = 0.0, d = 0.0;
                if (STAGE == 1) { c = sum(o.c, m); d = sum(o.d, m); }
                // back to the physical frame (y-faces: swap momentum components)
                const int k = 2 * gp + m, kp = (k == 1 || k == 2) && !xo ? 3 - k : k;
                gauss_average<STAGE>(r, a, b, c, d, [&](int q, double v) { out[(4 * q + kp) * ostride + oidx] = v; });
            }
        }
        if (bad) atomicOr(&G.ctrl->status, (int)CGKS_E_NONPHYSICAL);
    }
    release_next();
}

// The kernel's attributes (more than 48 KB of dynamic shared memory, the
// largest carveout) belong to one device's context: they are set once per
// device, thread-safely, before the first launch on that device.
template <int TX, int TY, int STAGE>
cudaError_t configure_stage_t()
{
    using L = StageLayout<TX, TY, STAGE>;
    static std::once_flag once[kMaxDevices];
    static cudaError_t status[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::call_once(once[dev], [dev] {
        cudaError_t r = cudaFuncSetAttribute(stage_kernel<TX, TY, STAGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)L::bytes);
        // the largest shared-memory carveout, so that two CTAs fit where the shape allows
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(stage_kernel<TX, TY, STAGE>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared);
        status[dev] = r;
    });
    return status[dev];
}

template <int TX, int TY, int STAGE>
cudaError_t launch_stage_t(const GridDev* grids, const TileRef* tiles, int ntiles, int nblocks, cudaStream_t st,
                           const int* dcount)
{
    using L = StageLayout<TX, TY, STAGE>;
    cudaError_t e = configure_stage_t<TX, TY, STAGE>();
    if (e != cudaSuccess) return e;
    if (ntiles <= 0 || nblocks <= 0) return cudaSuccess;
    return launch_chained(stage_kernel<TX, TY, STAGE>, nblocks, kThreads, L::bytes, st, grids, tiles, ntiles, dcount);
}

// The launcher and shared-memory size of one tile shape (one translation unit
// per shape, so the shapes compile in parallel).
#define CGKS_STAGE_INSTANCE(W, H) CGKS_STAGE_INSTANCE_(W, H, work_w(W, H), work_h(W, H))
#define CGKS_STAGE_INSTANCE_(W, H, TX, TY)                                                                  \
    static_assert(StageLayout<TX, TY, 1>::bytes + sizeof(double) * FK_N + 16 <= 227 * 1024,                 \
                  "stage-1 tile exceeds shared memory");                                                    \
    cudaError_t launch_stage_##W##x##H(int stage, const GridDev* grids, const TileRef* tiles, int ntiles,  \
                                         int nblocks, cudaStream_t st, const int* dcount)                   \
    {                                                                                                       \
        return stage == 1 ? launch_stage_t<TX, TY, 1>(grids, tiles, ntiles, nblocks, st, dcount)            \
                          : launch_stage_t<TX, TY, 2>(grids, tiles, ntiles, nblocks, st, dcount);           \
    }                                                                                                       \
    size_t smem_##W##x##H(int stage)                                                                      \
    {                                                                                                       \
        return stage == 1 ? StageLayout<TX, TY, 1>::bytes : StageLayout<TX, TY, 2>::bytes;                  \
    }

}  // namespace cgks
