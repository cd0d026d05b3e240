// update.cu -- the cell update of a stage (Liska et al. 2019, Sec. 2.5-2.7):
// U = U(P^n) + dt (Q - div F), the inversion, the floors and, in the
// corrector of a single block, the CFL rate of the new state.
//
// Two forms: FP64 (b_update64), and the mixed forms with FP64 under the learned
// guess (b_update). Around the mixed form's FP32 parts its FP64 arithmetic keeps its
// operations and their order: the state is rounded to FP32 for the next stage, and
// where a value sits at a rounding boundary a change of its last bit moves that stage
// by an FP32 unit, which limiters and the inversion of magnetised cells then amplify
// (measured with the same arithmetic in double-float, 2^-46: one cell in 3000 off by
// more than 1e-8 after four steps). FP64 cells under the network keep Newton in FP64:
// with newton_wv_ff a test of tree periods gave other outcomes from run to run (cells
// whose rescue by the network sits on a knife edge: a change of the last bit of rho and
// u moves a tilted disk's step by 1e-2 in either form). They keep the rest of b_update
// with it only because no FP64 form with the network has been made from b_update64: a
// step of the 256x128x64 torus takes 13.1 / 12.3 ms with the network first / as rescue,
// 10.0 without. Inversions in which the network has no part (internal-SMR groups,
// refluxed cells, drift-frame floors) take the same form on every FP64 grid.
#include "mlp.cuh"
#include "stage.cuh"

namespace hamr {
namespace {

// the learned guess of a CTA's 128 cells (mlp.cuh): Newton starts from it with the start from the previous
// primitives as fallback, or (rescue) from those primitives first and from the network where that fails;
// the CTA runs the network only if one of its cells needs it. The weight image has been asked for
// (mlp_begin) unless rescue.
__device__ __forceinline__ void mlp_attempts(MlpCta& C, uint8_t* smem, const PhysArgs& ph, bool rescue, bool active,
                                             C2PWork& w, const double U[NCONS], const Metric<double>& m, double x1) {
    if (rescue && active) c2p_attempt_plain(w, ph.gam);
    if (__syncthreads_or(active && !w.ok)) {
        if (rescue) mlp_begin(C, smem, ph.mlp_img);
        float f[MLP_NIN], y[MLP_NOUT];
        if (active) mlp_features(w.S, U[C_RHO], U[C_ENT], m, x1, ph.gam, f);
        const bool ran = mlp_infer(C, f, active, y);
        mlp_end(C);
        if (!C.ok && threadIdx.x == 0 && ph.mlp_err) atomicExch(ph.mlp_err, 1);
        if (active && ran && !w.ok) {
            double g2[2];
            mlp_guess(w.S.D, y, g2);
            c2p_attempt(w, ph.gam, g2[0], g2[1]);
        }
    } else if (!rescue) {
        mlp_end(C);
    }
}

// ---------------------------------------------------------------- FP64
// Bound by the FP64 pipe: what counts is FP64 instructions per cell. COR: the corrector (U^n from the
// cache); rate: with the CFL rate of the new state, which is formed only where its FP32 estimate is not
// certainly below the largest rate found so far. 256x128x64 torus, predictor and corrector together: 3.00 ms
// with b^mu, b_mu and the rate of every cell, 2.52 ms now.
template <bool COR>
__device__ __forceinline__ void b_update64(const BlockView& v, const PhysArgs& ph, bool rate,
                                           const double* __restrict__ Pf, const double* __restrict__ F1,
                                           const double* __restrict__ F2, const double* __restrict__ F3,
                                           const double* __restrict__ Bn, double* Un, double* Po,
                                           uint8_t* __restrict__ status, const double* __restrict__ dscal, double fac,
                                           unsigned long long* dmax, unsigned long long* dcnt, long t) {
    bool active = t < (long)v.n1 * v.n2 * v.n3;  // false again for a cell whose inversion its internal-SMR group does
    double inv = 0.0;
    int st = -1, fl = 0, its = 0;
    const double gam = ph.gam;
    Metric<double> m;
    double U[NCONS], Bc[3], pr[NPRIM], start[2];
    long c = 0, g = 0;
    if (active) {
        const int i = (int)(t % v.n1);
        const int j = (int)((t / v.n1) % v.n2), k = (int)(t / ((long)v.n1 * v.n2));
        c = cidx(v, i, j, k);
        g = gidx(v, i, j);
        const long nc = v.nc;
        load_metric(v.gc, v.n2d, g, m);
#pragma unroll
        for (int q = 0; q < NPRIM; q++) pr[q] = Pf[q * nc + c];
        // the stage state: the source, the inversion's start and, in the predictor, U^n
        Side64 s;
        side64(pr, m, m.alpha * m.c01, s);
        if (!COR) {
            // U^n (the rows of hll_side64 with cF = 0, cU = 1); kappa from the entropy-tracer pass
            const double w = fma(gam, pr[UU], pr[RHO]) + s.s2;
            const double a = w * s.ut, Z = s.Y * s.ut, mass = pr[RHO] * s.ut;
            const double ptot = (gam - 1.0) * pr[UU] + 0.5 * s.bsq;
            U[C_RHO] = mass * m.gdet;
            U[C_EN] = (a * s.c0 + (-Z * s.k0 + (ptot + mass))) * m.gdet;
            U[C_S1] = (a * s.c1 - Z * s.k1) * m.gdet;
            U[C_S2] = (a * s.c2 - Z * s.k2) * m.gdet;
            U[C_S3] = (a * s.c3 - Z * s.k3) * m.gdet;
            U[C_ENT] = Un[C_ENT * nc + c] * U[C_RHO];
#pragma unroll
            for (int q = 0; q < NCONS; q++) Un[q * nc + c] = U[q];
        } else {
#pragma unroll
            for (int q = 0; q < NCONS; q++) U[q] = Un[q * nc + c];
        }
        const double dts = dscal[0] * fac;
        double Q1, Q2;
        source64(v.gc, v.n2d, g, m, pr, s, gam, Q1, Q2);
        const double dg = dts * m.gdet;
        U[C_S1] = fma(dg, Q1, U[C_S1]);
        U[C_S2] = fma(dg, Q2, U[C_S2]);
        const double a1 = dts * v.idx1, a2 = dts * v.idx2, a3 = dts * v.idx3;  // dt / dx^i
        const long sj = v.n1p, sk = (long)v.n1p * v.n2p;
#pragma unroll
        for (int q = 0; q < NCONS; q++) {
            // U + dt (Q - div F): the flux differences times dt/dx^i taken off one by one
            double u = fma(-a1, F1[q * nc + c + 1] - F1[q * nc + c], U[q]);
            u = fma(-a2, F2[q * nc + c + sj] - F2[q * nc + c], u);
            U[q] = fma(-a3, F3[q * nc + c + sk] - F3[q * nc + c], u);
        }
        centre_field(v, Bn, i, j, k, m.igdet, Bc);
        start[0] = s.g2;
        start[1] = s.g2 - 1.0;
        pr[B1] = Bc[0];
        pr[B2] = Bc[1];
        pr[B3] = Bc[2];
        if (ph.smr > 0 && smr_width(v, ph, j) > 1) {  // inverted with its group (k_smr_cells)
#pragma unroll
            for (int q = 0; q < NCONS; q++) ph.smr_u[q * nc + c] = U[q];
            active = false;
        }
    }
    // inversion: the energy equation, then the entropy backup
    C2PWork w;
    if (active) {
        c2p_prepare(U, Bc, m, gam, pr, w, ph.inversion, C2P_NEWTON_FF, nullptr, ph.igam, ph.gfac, start);
        c2p_attempt_plain(w, gam);
    }
    // the lanes come out of the attempt by several ways: together again, or the entropy backup runs once for
    // each (pair of launches on a 24x12x8 block 207 -> 120 us, 96x64x48 disk with MINMOD 1180 -> 720 us)
    __syncwarp();
    if (active) {
        its = w.its;
        st = c2p_finish(w, U, m, gam, pr);
        uint8_t sb = (st == INV_ENTROPY) ? ST_ENTROPY : ((st == INV_FAIL) ? ST_FAIL : 0);
        // the floors take b^2 of the returned primitives, not of the inversion's own (W, v^2), which differ
        // from them by the Newton tolerance (more where v^2 was clamped): the floor rho = b^2/50 would
        // carry that
        if (ph.floors || (COR && rate)) {
            Side64 s;
            side64(pr, m, m.alpha * m.c01, s);
            if (ph.floors) {
                fl = cell_floors_b2(v, g, m, ph, pr, s.bsq);
                if (fl) sb |= ST_FLOOR;
            }
            if (COR && rate) {
                if (ph.floor_frame == HAMR_FLOOR_DRIFT) {  // the floors may have moved the velocity
                    inv = inv_dt_cell(v, pr, m, gam);
                } else {
                    const int sh = scale_of(pr[RHO], pr[UU], s.bsq);
                    const float ud[3] = {ff_of(s.u1).h, ff_of(s.u2).h, ff_of(s.u3).h};
                    const float est = rate_estimate(v, ph, ff_of(pr[RHO], sh).h, ff_of(pr[UU], sh).h, ff_of(s.bsq, sh).h,
                                                    ff_of(s.ut).h, ud, ff_of(m.c00).h, ff_of(m.c01).h, ff_of(m.c11).h,
                                                    ff_of(m.c22).h, ff_of(m.c33).h);
                    if (!rate_below(est, dmax)) inv = inv_dt_cell(v, pr, m, gam);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NPRIM; q++) Po[q * v.nc + c] = pr[q];
        status[c] |= sb;
    }
    count_cells(st, fl, active ? its : 0, dcnt);
    if (COR && rate) reduce_rate(inv, dmax);
}

// ---------------------------------------------------------------- mixed, and FP64 with the network
// U = U(P^n) + dts (Q(Pf) - div F); inversion with guess Pf; floors; the corrector (1) also reduces the CFL
// rate of the new state (2: the batched corrector, without it). TS: precision of the floors' b^2 and of the
// CFL rate (float in the mixed forms; the conserved accumulation and the inversion are FP64 always). INV64:
// the FP64 source and Newton in FP64 only (HAMR_PREC_MIXED_FP64INV, and FP64 with the network); else the
// FP32 source and Newton starting in FP32 (c2p.cuh).
template <bool MLP, typename TS, bool INV64>
__device__ __forceinline__ void b_update(const BlockView& v, const PhysArgs& ph, int corrector,
                                               const double* __restrict__ Pf, const double* __restrict__ F1,
                                               const double* __restrict__ F2, const double* __restrict__ F3,
                                               const double* __restrict__ Bn, double* Un, double* Po,
                                               uint8_t* __restrict__ status, const double* __restrict__ dscal,
                                               double fac, unsigned long long* dmax, unsigned long long* dcnt, long t) {
    const long n = (long)v.n1 * v.n2 * v.n3;
    bool active = t < n;  // false again for a cell whose inversion its internal-SMR group does
    double inv = 0.0;
    int st = -1, fl = 0, its = 0;
    const double gam = ph.gam;
    Metric<double> m;
    double U[NCONS], Bc[3], pr[NPRIM];
    long c = 0, g = 0;
    int i = 0, j = 0;
    MlpCta C;
    float start32[2] = {0.0f, 0.0f};  // mixed form: the inversion's start in FP32 (see the source)
    bool have32 = false;
    const bool rescue = MLP && ph.mlp_mode == HAMR_MLP_RESCUE;
    extern __shared__ __align__(16) uint8_t mlp_smem[];
    if (MLP && !rescue) mlp_begin(C, mlp_smem, ph.mlp_img);  // the weight image streams in while U is formed
    if (active) {
        i = (int)(t % v.n1);
        j = (int)((t / v.n1) % v.n2);
        const int k = (int)(t / ((long)v.n1 * v.n2));
        c = cidx(v, i, j, k);
        g = gidx(v, i, j);
        const long nc = v.nc;
        load_metric(v.gc, v.n2d, g, m);
        double pf[NPRIM];
#pragma unroll
        for (int q = 0; q < NPRIM; q++) pf[q] = Pf[q * nc + c];
        Fluid<double> sf;  // FP64 source: one fluid state serves U^n and the source
        if (INV64) fluid_state(pf, m, sf);
        // U^n, with kappa from the entropy-tracer pass
        if (!corrector) {
            double row[NFLUX];
            if (!INV64) fluid_state(pf, m, sf);
            flux_row(pf, sf, 0, 1, gam, Un[C_ENT * nc + c], row);
#pragma unroll
            for (int q = 0; q < NCONS; q++) {
                U[q] = row[q] * m.gdet;
                Un[q * nc + c] = U[q];
            }
        } else {
#pragma unroll
            for (int q = 0; q < NCONS; q++) U[q] = Un[q * nc + c];
        }
        // source sqrt(-g) T^k_l Gamma^l_{nu k} at the centre, from Pf
        double Q[4];
        if constexpr (INV64) {
            source_q_dg(v.gc, v.n2d, g, m, pf, sf, gam, Q);
        } else {
            // the FP32 source of the stage state: its FP32 copy, the values (float)pf exactly
            Metric<float> mf;
            load_metric(v.gc32, v.n2d, g, mf);
            float p32[NPRIM];
#pragma unroll
            for (int q = 0; q < NPRIM; q++) p32[q] = v.P32[q * nc + c];
            Fluid<float> s32;
            fluid_state(p32, mf, s32);
            float Qf[4];
            source_q_state(v.gc32, v.n2d, g, mf, p32, s32, narrow(gam), Qf);
#pragma unroll
            for (int q = 0; q < 4; q++) Q[q] = widen(Qf[q]);
            // the inversion's start from the same state (it only seeds the FP32 iterations)
            const float qsq = p32[U1] * s32.ucov[1] + p32[U2] * s32.ucov[2] + p32[U3] * s32.ucov[3];
            const float gsq = 1.0f + qsq;
            start32[0] = (p32[RHO] + narrow(gam) * p32[UU]) * gsq;
            start32[1] = qsq / gsq;
            have32 = true;
        }
        const double dts = dscal[0] * fac;
        const double a1 = dts * v.idx1, a2 = dts * v.idx2, a3 = dts * v.idx3;  // dt / dx^i
        const long sj = v.n1p, sk = (long)v.n1p * v.n2p;
#pragma unroll
        for (int q = 0; q < NCONS; q++) {
            // U + dt (Q - div F): the flux differences times dt/dx^i taken off one by one
            double u = (q >= C_EN && q <= C_S3) ? fma(dts, Q[q - C_EN], U[q]) : U[q];
            u = fma(-a1, F1[q * nc + c + 1] - F1[q * nc + c], u);
            u = fma(-a2, F2[q * nc + c + sj] - F2[q * nc + c], u);
            U[q] = fma(-a3, F3[q * nc + c + sk] - F3[q * nc + c], u);
        }
        centre_field(v, Bn, i, j, k, m.igdet, Bc);
#pragma unroll
        for (int q = 0; q < NPRIM; q++) pr[q] = pf[q];
        pr[B1] = Bc[0];
        pr[B2] = Bc[1];
        pr[B3] = Bc[2];
        if (ph.smr > 0 && smr_width(v, ph, j) > 1) {  // inverted with its group (k_smr_cells)
#pragma unroll
            for (int q = 0; q < NCONS; q++) ph.smr_u[q * nc + c] = U[q];
            active = false;
        }
    }
    // inversion: energy attempts from the start(s), then the entropy backup
    C2PWork w;
    if (active)
        c2p_prepare(U, Bc, m, gam, pr, w, ph.inversion, INV64 ? C2P_NEWTON64 : C2P_NEWTON32,
                    have32 ? start32 : nullptr, ph.igam, ph.gfac);
    if (MLP) mlp_attempts(C, mlp_smem, ph, rescue, active, w, U, m, v.x1min + (i + 0.5) * v.dx1);
    if (active && !rescue) c2p_attempt_plain(w, gam);
    __syncwarp();  // as in b_update64 (24x12x8 pair, mixed: 225 -> 185 us)
    if (active) {
        its = w.its;
        st = c2p_finish(w, U, m, gam, pr);
        uint8_t sb = (st == INV_ENTROPY) ? ST_ENTROPY : ((st == INV_FAIL) ? ST_FAIL : 0);
        // the fluid state of the returned primitives serves the floors (b^2) and the CFL rate (u^mu,
        // b^mu and b^2 do not depend on rho and u_g, which are all the floors change). The floors take
        // b^2 of these primitives, not of the inversion's own (W, v^2), which differ from them by the
        // Newton tolerance (more where v^2 was clamped), and the floor rho = b^2/50 would carry that.
        if constexpr (std::is_same<TS, double>::value) {
            Fluid<double> s;
            const bool need_fluid = ph.floors || corrector == 1;
            if (need_fluid) fluid_state(pr, m, s);
            if (ph.floors) {
                fl = cell_floors(v, g, m, ph, pr, s);
                if (fl) sb |= ST_FLOOR;
            }
#pragma unroll
            for (int q = 0; q < NPRIM; q++) Po[q * v.nc + c] = pr[q];
            if (corrector == 1) inv = inv_dt_fluid(v, pr, s, m, gam);
        } else {
            // mixed precision: one FP32 fluid state of the returned primitives gives the floors'
            // b^2 (the thresholds b^2/50 and b^2/750 to FP32 accuracy, like the fluxes) and the
            // FP32 CFL rate; drift-frame floors form the FP64 state they need themselves
            Metric<TS> mf;
            load_metric(v.gc32, v.n2d, g, mf);
            TS pf32[NPRIM];
#pragma unroll
            for (int q = 0; q < NPRIM; q++) pf32[q] = to_t<TS>(pr[q]);
            Fluid<TS> s32;
            fluid_state(pf32, mf, s32);
            if (ph.floors) {
                fl = cell_floors_f32(v, g, m, ph, pr, pf32, s32.bsq);
                if (fl) {
                    sb |= ST_FLOOR;
                    if (ph.floor_frame == HAMR_FLOOR_DRIFT && corrector == 1) fluid_state(pf32, mf, s32);
                }
            }
#pragma unroll
            for (int q = 0; q < NPRIM; q++) Po[q * v.nc + c] = pr[q];
            if (corrector == 1) inv = inv_dt_fluid(v, pf32, s32, mf, to_t<TS>(gam));
            if (ph.stage32) store_stage32(v, ph, corrector, c, pf32);
        }
        status[c] |= sb;
    }
    count_cells(st, fl, active ? its : 0, dcnt);
    if (corrector == 1) reduce_rate(inv, dmax);
}

#define HAMR_UPD_PARAMS                                                                                              \
    const double *__restrict__ Pf, const double *__restrict__ F1, const double *__restrict__ F2,                     \
        const double *__restrict__ F3, const double *__restrict__ Bn, double *Un, double *Po,                        \
        uint8_t *__restrict__ status, const double *__restrict__ dscal, double fac, unsigned long long *dmax,        \
        unsigned long long *dcnt

template <bool COR>
__global__ void __launch_bounds__(BS) k_update64(BlockView v, PhysArgs ph, HAMR_UPD_PARAMS) {
    b_update64<COR>(v, ph, true, Pf, F1, F2, F3, Bn, Un, Po, status, dscal, fac, dmax, dcnt, tidx());
}
// four CTAs per SM (128 registers, a few spilled) without the network: the FP64 pipe waits less between the
// FP32 stretches (256x128x64 torus, mixed predictor: 1.03 -> 0.94 ms; 384 threads per CTA: 1.09 ms)
template <bool MLP, typename TS, bool INV64>
__global__ void __launch_bounds__(BS, MLP ? 3 : 4) k_update(BlockView v, PhysArgs ph, int corrector, HAMR_UPD_PARAMS) {
    b_update<MLP, TS, INV64>(v, ph, corrector, Pf, F1, F2, F3, Bn, Un, Po, status, dscal, fac, dmax, dcnt, tidx());
}

// batched: block list[blockIdx.y]; predictor or corrector of the block's step (no CFL rate here). Under
// internal SMR the grouped cells' conserved states go to the right edge values (free once the fluxes exist).
#define HAMR_UPD_BLOCK(D, COR)                                                                                \
    (COR) ? D.Ph : D.P, D.F1, D.F2, D.F3, (COR) ? D.B : D.Bh, D.Un, (COR) ? D.P : D.Ph, D.status, D.dscal,    \
        (COR) ? 1.0 : 0.5, D.dmax, D.dcnt, tidx()

template <bool COR>
__global__ void __launch_bounds__(BS, 3) kb_update64(const DevBlock* tab, const int* list, PhysArgs ph) {
    const DevBlock& D = tab[list[blockIdx.y]];
    ph.smr_u = D.QR;
    b_update64<COR>(D.v, ph, false, HAMR_UPD_BLOCK(D, COR));
}
template <bool MLP, typename TS, bool INV64>
__global__ void __launch_bounds__(BS, MLP ? 3 : 4) kb_update(const DevBlock* tab, const int* list, PhysArgs ph, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    ph.smr_u = D.QR;
    b_update<MLP, TS, INV64>(D.v, ph, sigma ? 2 : 0, HAMR_UPD_BLOCK(D, sigma));
}

}  // namespace

cudaError_t launch_update(const BlockView& v, const PhysArgs& ph, int corrector, const double* Pflux,
                          double* const F[3], const double* Bnew, double* Un, double* Pout, uint8_t* status,
                          const double* dscal, double dt_factor, unsigned long long* dmax, unsigned long long* dcnt,
                          cudaStream_t s) {
    const long n = (long)v.n1 * v.n2 * v.n3;
    const int bs = ph.mlp_img ? MLP_ROWS : ph.bs_update;  // the network needs one row per thread of 128
    const unsigned nb = nblk(n, bs);
    const int sm = ph.mlp_img ? MLP_SMEM_BYTES : 0;
#define HAMR_UPD_ARGS Pflux, F[0], F[1], F[2], Bnew, Un, Pout, status, dscal, dt_factor, dmax, dcnt
    if (!ph.mixed && !ph.mlp_img) {
        corrector ? k_update64<true><<<nb, bs, 0, s>>>(v, ph, HAMR_UPD_ARGS)
                  : k_update64<false><<<nb, bs, 0, s>>>(v, ph, HAMR_UPD_ARGS);
    } else {
        auto k = !ph.mixed    ? k_update<true, double, true>
                 : ph.mlp_img ? (ph.fp64_inv ? k_update<true, float, true> : k_update<true, float, false>)
                              : (ph.fp64_inv ? k_update<false, float, true> : k_update<false, float, false>);
        k<<<nb, bs, sm, s>>>(v, ph, corrector, HAMR_UPD_ARGS);
    }
#undef HAMR_UPD_ARGS
    return cudaGetLastError();
}

cudaError_t launch_update_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, const PhysArgs& ph,
                                int sigma, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    const int bs = ph.mlp_img ? MLP_ROWS : ph.bs_update;
    const dim3 gr = bgrid(maxwork, nlist, bs);
    const int sm = ph.mlp_img ? MLP_SMEM_BYTES : 0;
    if (!ph.mixed && !ph.mlp_img) {
        sigma ? kb_update64<true><<<gr, bs, 0, s>>>(tab, list, ph) : kb_update64<false><<<gr, bs, 0, s>>>(tab, list, ph);
    } else {
        auto k = !ph.mixed    ? kb_update<true, double, true>
                 : ph.mlp_img ? (ph.fp64_inv ? kb_update<true, float, true> : kb_update<true, float, false>)
                              : (ph.fp64_inv ? kb_update<false, float, true> : kb_update<false, float, false>);
        k<<<gr, bs, sm, s>>>(tab, list, ph, sigma);
    }
    return cudaGetLastError();
}

}  // namespace hamr
