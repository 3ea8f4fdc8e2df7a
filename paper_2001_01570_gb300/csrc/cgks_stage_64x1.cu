// cgks_stage_64x1.cu -- the flux kernel of a 1D grid (tile shape 64x1): the
// gas-kinetic evaluation of cgks_flux.cuh with nothing varying along the face and no
// tangential velocity (Sec. 2.1-2.2 in one dimension; the kinetic model keeps the 2D
// one's internal degrees of freedom, whose tangential velocity plays the additional
// one of the 1D model).
//
// The two Gauss points of a face coincide, so one evaluation serves both; the state
// and its slopes are read straight from the grid's one row of records; a pair of lanes
// shares a face, each with one of the two half-line sides, whose sums they exchange by
// shuffles.  What bounds it on the grids 1D is used for (12 to a few hundred cells) is the
// chain of dependent FP64 instructions of one warp, 68 cycles each: about 220 here
// against some 550 per lane of the 2D kernel (100 cells, stage 1: 81.9 us with one thread
// per face, 43.7 with one per Gauss point, 18.3 here).
#include "cgks_flux.cuh"
#include "cgks_segment.cuh"

namespace cgks {

static __device__ const FluxFixed kFluxFixed1d = make_flux_fixed();

namespace {

// variables of a 1D state: density, momentum, energy (indices 0, 1, 3 of the records)
struct State1 { double r, m, e; };

// one side's half-line sums (fluxes, slope terms of the fluxes, states, slope terms of the states)
struct Half1 { State1 F, T, W, S; };

__device__ __forceinline__ void half_1d(const RegK& r, int side, const State1& W, const State1& Wn, double U, double th,
                                        bool ne, Half1& o)
{
    HalfMoments h;
    const double th2 = r.add(th, th), sq = r.rsq(th2);
    half_moments(r, side, U, th, th2, sq, h);
    const double m0 = h.m[0], m1 = h.m[1], m2 = h.m[2], m3 = h.m[3], K1 = r.k(FK_K1), qt = r.mul(K1, th);
    o.F.r = r.mul(W.r, m1);
    o.F.m = r.mul(W.r, m2);
    o.F.e = r.mul(W.r, r.kmul(FK_HALF, fma(m1, qt, m3)));
    // slope_moments without tangential slopes: (rho', rho U', rho theta') and y_n = (rho m_n)'
    const double R = Wn.r, A = fma(-U, R, Wn.m), hq2 = r.kmul(FK_HALF, r.mul(U, U));
    const double de = fma(-hq2, R, fma(-U, A, Wn.e)), C = fma(-th, R, r.mul(r.k(FK_GM1), de));
    const double A2 = r.add(A, A), C3 = r.kmul(FK_3, C), m4 = fma(U, m3, r.mul(r.kmul(FK_3, th), m2));
    const double y2 = fma(R, m2, fma(A2, m1, r.mul(C, m0)));
    const double y3 = fma(R, m3, r.kmul(FK_3, fma(A, m2, r.mul(C, m1))));
    const double z4 = fma(A2, m3, r.mul(C3, m2)), y4 = fma(R, m4, r.add(z4, z4)), xv = r.mul(K1, C);
    o.T.r = y2;
    o.T.m = y3;
    o.T.e = r.kmul(FK_HALF, fma(m2, xv, fma(qt, y2, y4)));
    CGKS_BRANCH(ne)
    {
        const double y1 = fma(R, m1, fma(A, m0, r.mul(r.kmul(FK_HALF, C), h.g)));
        o.W.r = r.mul(W.r, m0);
        o.W.m = o.F.r;
        o.W.e = r.mul(W.r, r.kmul(FK_HALF, fma(m0, qt, m2)));
        o.S.r = y1;
        o.S.m = y2;
        o.S.e = r.kmul(FK_HALF, fma(m1, xv, fma(qt, y1, y3)));
    }
}

// Euler time derivatives (cgks_flux.cuh: euler_time_derivs) without tangential terms
struct Euler1 { State1 Wt, Wtt, F, Ft, T; };

__device__ __forceinline__ void euler_1d(const RegK& r, const State1& W, const State1& Wx, const State1& Wxx, double ir,
                                         double U, double p, double e, Euler1& o)
{
    const double gamma = r.k(FK_GAMMA), gir = r.mul(r.k(FK_GM1), ir), hq2 = r.kmul(FK_HALF, r.mul(U, U));
    const double Ux = r.mul(fma(-U, Wx.r, Wx.m), ir);
    const double ex = r.sub(Wx.e, fma(-hq2, Wx.r, r.mul(U, Wx.m)));
    const double rt = -fma(W.r, Ux, r.mul(U, Wx.r)), Ut = -fma(ex, gir, r.mul(U, Ux));
    const double et = -fma(r.mul(gamma, e), Ux, r.mul(U, ex)), uut = r.mul(U, Ut);
    o.Wt = State1{rt, fma(W.r, Ut, r.mul(rt, U)), fma(W.r, uut, fma(rt, hq2, et))};
    const double Ep = r.add(W.e, p), pt = r.mul(r.k(FK_GM1), et);
    o.F = State1{W.m, fma(W.m, U, p), r.mul(U, Ep)};
    o.Ft = State1{o.Wt.m, fma(W.m, Ut, fma(o.Wt.m, U, pt)), fma(U, r.add(o.Wt.e, pt), r.mul(Ut, Ep))};
    const double sxx = r.mul(p, fma(-r.k(FK_K2INV2), Ux, r.add(Ux, Ux)));
    const double thx = r.mul(fma(-r.mul(e, ir), Wx.r, ex), gir);
    o.T = State1{0.0, sxx, fma(r.mul(r.k(FK_KHEAT), p), thx, r.mul(U, sxx))};
    // second order (the mixed derivatives enter negated)
    const double rx2 = r.add(Wx.r, Wx.r), Uxx = r.mul(fma(-U, Wxx.r, fma(-Ux, rx2, Wxx.m)), ir);
    const double exx = r.sub(Wxx.e, fma(-hq2, Wxx.r, fma(U, Wxx.m, r.mul(W.r, r.mul(Ux, Ux)))));
    const double nrxt = fma(W.r, Uxx, fma(rx2, Ux, r.mul(U, Wxx.r)));
    const double nUxt = fma(fma(-r.mul(ex, Wx.r), ir, exx), gir, fma(U, Uxx, r.mul(Ux, Ux)));
    const double next = fma(gamma, fma(e, Uxx, r.mul(ex, Ux)), fma(U, exx, r.mul(Ux, ex)));
    const double rtt = fma(W.r, nUxt, fma(-rt, Ux, fma(-Ut, Wx.r, r.mul(U, nrxt))));
    const double Utt = fma(fma(r.mul(ex, rt), ir, next), gir, fma(-Ut, Ux, r.mul(U, nUxt)));
    const double ett = fma(gamma, fma(-et, Ux, r.mul(e, nUxt)), fma(-Ut, ex, r.mul(U, next)));
    const double rt2 = r.add(rt, rt);
    o.Wtt = State1{rtt, fma(W.r, Utt, fma(rt2, Ut, r.mul(rtt, U))),
                   fma(W.r, fma(U, Utt, r.mul(Ut, Ut)), fma(rt2, uut, fma(rtt, hq2, ett)))};
}

template <int STAGE>
__global__ void __launch_bounds__(kThreads, 2)
flux1d_kernel(const GridDev* __restrict__ grids, const TileRef* __restrict__ tiles, int ntiles,
              const int* __restrict__ dcount)
{
    __shared__ double s_fk[FK_N];
    __shared__ int s_skip;
    const int tid = threadIdx.x, side = tid & 1;
    const unsigned pair = 3u << (tid & 30);
    for (int i = tid; i < FK_NFIX2; i += kThreads) s_fk[i] = kFluxFixed1d.v[i];
    __syncthreads();
    const RegK r{s_fk, ((volatile const double*)s_fk)[FK_ONE], ((volatile const double*)s_fk)[FK_NZERO]};
    wait_previous();
    int held = -1;
    for (int tile = blockIdx.x; tile < (dcount ? *(volatile const int*)dcount : ntiles); tile += gridDim.x) {
        __syncthreads();
        const TileRef tr = tiles[tile];
        const GridDev& G = grids[tr.grid];
        flux_table_grid(s_fk, G, tr.grid, held, s_skip);
        __syncthreads();
        if (s_skip) continue;
        const int face = tr.x0 + (tid >> 1), nx = G.nx;
        if (face > nx) continue;                      // both lanes of the pair
        // the grid's row (j = 0) of the records [7][4][5][nx+1]
        const size_t sx = (size_t)5 * (nx + 1), at0 = (size_t)2 * (nx + 1) + face;
        if (!CGKS_IN_BOUNDS(27 * sx + at0 < 28 * sx && face >= 0, G.ctrl)) continue;
        auto rec = [&](int f, int k) { return G.recx[(size_t)(f * 4 + k) * sx + at0]; };
        auto state = [&](int f) { return State1{rec(f, 0), rec(f, 1), rec(f, 3)}; };
        const State1 W = state(RV), Wx = state(RN), Wxx = state(RNN), H = state(RL + side), Hn = state(RLN + side);
        const double ir = r.rcp3(W.r), U = r.mul(W.m, ir), e = r.kfma(FK_MHALF, r.mul(W.m, U), W.e);
        const double p = r.mul(r.k(FK_GM1), e);
        const double irh = r.rcp3(H.r), Uh = r.mul(H.m, irh);
        const double ph = r.mul(r.k(FK_GM1), r.kfma(FK_MHALF, r.mul(H.m, Uh), H.e)), thh = r.mul(ph, irh);
        const bool ok = positive(W.r) && positive(p) && positive(H.r) && positive(ph);
        // collision time and its weight, as gks_point (the other side's pressure by shuffle)
        const double po = __shfl_xor_sync(pair, ph, 1);
        const double mu = r.k(FK_MU), dt = r.k(FK_DT);
        double tau0 = r.k(FK_EPSDT);
        CGKS_BRANCH(positive(mu)) tau0 = r.mul(mu, r.rcp3(p));
        const double tau = fma(r.k(FK_CTAUDT), fabs(r.mul(r.sub(ph, po), r.rcp3(r.add(ph, po)))), tau0);
        double h = 0.0;
        CGKS_BRANCH(nonequilibrium(r, tau)) h = exp_neg(r, r.mul(r.k(FK_MHDT), r.rcp3(tau)));
        const bool need_ne = (STAGE == 1) && d_hi(h) >= 0x3bc79ca1;       // h >= 1e-20
        Half1 o;
        half_1d(r, side, H, Hn, Uh, thh, need_ne, o);
        auto both = [&](State1& s) {
            s.r = r.add(s.r, __shfl_xor_sync(pair, s.r, 1));
            s.m = r.add(s.m, __shfl_xor_sync(pair, s.m, 1));
            s.e = r.add(s.e, __shfl_xor_sync(pair, s.e, 1));
        };
        both(o.F);
        both(o.T);
        CGKS_BRANCH(need_ne) { both(o.W); both(o.S); }        // tau is the pair's, so need_ne is too
        Euler1 E;
        euler_1d(r, W, Wx, Wxx, ir, U, p, e, E);
        // window coefficients over [0, dt] (gks_point)
        const double idt = r.k(FK_IDT), omh = r.sub(r.one, h), ta = r.mul(tau, omh), q4 = r.mul(ta, r.k(FK_4IDT2));
        const double g = r.mul(q4, omh), dh = r.mul(dt, h), f4 = r.mul(q4, r.sub(dh, ta)), tat = r.mul(ta, r.sub(r.k(FK_3), h));
        const double a = r.mul(tat, idt), b4 = r.mul(r.mul(tau, fma(-dh, r.sub(r.k(FK_2), h), tat)), idt);
        const double hdt = r.k(FK_HDT), h2 = r.mul(h, h);
        double* out = G.facex + face;
        const size_t os = (size_t)nx + 1;
        // one variable's results: lane 0 writes the flux combinations, lane 1 the states; both
        // Gauss points are this one, so the sums gauss_average takes are twice the point's
        auto finish = [&](int k, double W0, double Fh, double Th, double Wh, double Ws, double F, double Ft, double TNS,
                          double Wt, double Wtt) {
            const double dTh = r.sub(r.sub(TNS, Ft), Th), dFh = r.sub(Fh, F);
            const double ft_ = fma(f4, dTh, fma(-g, dFh, Ft)), ft2 = r.add(ft_, ft_);
            if (STAGE == 1) {
                const double fb = fma(b4, dTh, fma(-tau, TNS, fma(a, dFh, F))), fb2 = r.add(fb, fb);
                double wm = fma(r.k(FK_C8), Wtt, fma(hdt, Wt, W0)), wb = fma(r.k(FK_C6), Wtt, fma(dt, Wt, W0));
                CGKS_BRANCH(need_ne)
                {
                    wm = fma(h, fma(-hdt, Wt, r.sub(fma(-hdt, Ws, Wh), W0)), wm);
                    wb = fma(h2, fma(-dt, Wt, r.sub(fma(-dt, Ws, Wh), W0)), wb);
                }
                gauss_average<1>(r, fb2, ft2, r.add(wm, wm), r.add(wb, wb), [&](int q, double v) {
                    if ((q >> 1) == side) out[(4 * q + k) * os] = v;
                });
            } else {
                gauss_average<2>(r, ft2, r.add(Wtt, Wtt), 0.0, 0.0, [&](int q, double v) {
                    if (q == side) out[(4 * q + k) * os] = v;
                });
            }
        };
        finish(0, W.r, o.F.r, o.T.r, o.W.r, o.S.r, E.F.r, E.Ft.r, E.T.r, E.Wt.r, E.Wtt.r);
        finish(1, W.m, o.F.m, o.T.m, o.W.m, o.S.m, E.F.m, E.Ft.m, E.T.m, E.Wt.m, E.Wtt.m);
        finish(3, W.e, o.F.e, o.T.e, o.W.e, o.S.e, E.F.e, E.Ft.e, E.T.e, E.Wt.e, E.Wtt.e);
        // no tangential momentum
        out[(STAGE == 1 ? 8 * side + 2 : 4 * side + 2) * os] = 0.0;
        if (STAGE == 1) out[(8 * side + 6) * os] = 0.0;
        if (!ok) atomicOr(&G.ctrl->status, (int)CGKS_E_NONPHYSICAL);
    }
    release_next();
}

}  // namespace

cudaError_t launch_stage_64x1(int stage, const GridDev* grids, const TileRef* tiles, int ntiles, int nblocks,
                              cudaStream_t st, const int* dcount)
{
    if (ntiles <= 0 || nblocks <= 0) return cudaSuccess;
    return launch_chained(stage == 1 ? flux1d_kernel<1> : flux1d_kernel<2>, nblocks, kThreads, 0, st, grids, tiles, ntiles,
                          dcount);
}

size_t smem_64x1(int) { return 0; }

}  // namespace cgks
