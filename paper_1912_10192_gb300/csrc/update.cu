// update.cu -- the cell update of a stage (Liska et al. 2019, Sec. 2.5-2.7):
// U = U(P^n) + dt (Q - div F), the inversion, the floors and, in the
// corrector of a single block, the CFL rate of the new state.
#include "mlp.cuh"
#include "stage.cuh"

namespace hamr {
namespace {

// ---------------------------------------------------------------- cell update
// U = U(P^n) + dts (Q(Pf) - div F); inversion with guess Pf; floors;
// the corrector also reduces the CFL rate of the new state.
// MLP: the CTA's 128 cells first run the learned guess (mlp.cuh) on the
// tensor cores; Newton starts from it, with the start from Pf as fallback.
// TS: precision of the connection source and of the CFL rate (float in mixed
// precision; the conserved accumulation and the inversion are FP64 always). With
// ph.fp64_inv the mixed form takes the FP64 source and iterates Newton in FP64
// only (without it, its Newton iteration starts in FP32, c2p.cuh).
template <bool MLP, typename TS>
__device__ __forceinline__ void b_update(const BlockView& v, PhysArgs ph, int corrector, const double* Pb,
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
        // in the predictor the base state is the stage state (Pb == Pf): with an FP64
        // source one fluid state serves U^n and the source
        const bool share = std::is_same<TS, double>::value && !corrector && Pb == Pf;
        Fluid<double> sf;
        if (share) fluid_state(pf, m, sf);
        // U^n
        if (!corrector) {
            double row[NFLUX];
            if (share) {  // kappa of P^n from the predictor's entropy-tracer pass
                flux_row(pf, sf, 0, 1, gam, Un[C_ENT * nc + c], row);
            } else {
                double pb[NPRIM];
#pragma unroll
                for (int q = 0; q < NPRIM; q++) pb[q] = Pb[q * nc + c];
                Fluid<double> s;
                fluid_state(pb, m, s);
                flux_row(pb, s, 0, 1, gam, Un[C_ENT * nc + c], row);  // kappa from the tracer pass
            }
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
        if constexpr (std::is_same<TS, double>::value) {
            if (share) {
                source_q_dg(v.gc, v.n2d, g, m, pf, sf, gam, Q);
            } else {
                Fluid<double> s;
                fluid_state(pf, m, s);
                source_q_dg(v.gc, v.n2d, g, m, pf, s, gam, Q);
            }
        } else if (ph.fp64_inv) {  // mixed form with the FP64 source of the FP64 path
            Fluid<double> s;
            fluid_state(pf, m, s);
            source_q_dg(v.gc, v.n2d, g, m, pf, s, gam, Q);
        } else {
            // the FP32 source of the stage state: its FP32 copy, the values (float)pf exactly
            Metric<float> mf;
            load_metric(v.gc32, v.n2d, g, mf);
            float p32[NPRIM];
#pragma unroll
            for (int q = 0; q < NPRIM; q++) p32[q] = v.P32[q * nc + c];
            Fluid<float> s32;
            fluid_state(p32, mf, s32);
            source_q_state(v.gc32, v.n2d, g, mf, p32, s32, narrow(gam), Q);
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
        c2p_prepare(U, Bc, m, gam, pr, w, ph.inversion, (std::is_same<TS, float>::value && !ph.fp64_inv) ? 1 : 0,
                    have32 ? start32 : nullptr, ph.igam, ph.gfac);
    if (MLP) {
        // first: the network's start, then the plain one; rescue: the plain start, then the
        // network's where it failed (the CTA runs the network only if one of its cells failed)
        if (rescue && active) c2p_attempt_plain(w, gam);
        if (__syncthreads_or(active && !w.ok)) {
            if (rescue) mlp_begin(C, mlp_smem, ph.mlp_img);
            float f[MLP_NIN], y[MLP_NOUT];
            if (active) mlp_features(w.S, U[C_RHO], U[C_ENT], m, v.x1min + (i + 0.5) * v.dx1, gam, f);
            const bool ran = mlp_infer(C, f, active, y);
            mlp_end(C);
            if (!C.ok && threadIdx.x == 0 && ph.mlp_err) atomicExch(ph.mlp_err, 1);
            if (active && ran && !w.ok) {
                double g2[2];
                mlp_guess(w.S.D, y, g2);
                c2p_attempt(w, gam, g2[0], g2[1]);
            }
        } else if (!rescue) {
            mlp_end(C);
        }
    }
    if (active) {
        if (!rescue) c2p_attempt_plain(w, gam);
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
    // warp-aggregated counters and CFL max
    const unsigned lane = threadIdx.x & 31u;
    const unsigned long long c_ok = warp_sum((unsigned long long)(st == INV_OK));
    const unsigned long long c_en = warp_sum((unsigned long long)(st == INV_ENTROPY));
    const unsigned long long c_fa = warp_sum((unsigned long long)(st == INV_FAIL));
    const unsigned long long c_fl = warp_sum((unsigned long long)fl);
    const unsigned long long c_it = warp_sum((unsigned long long)(active ? its : 0));
    const double wmax = warp_max(inv);
    if (lane == 0) {
        if (c_ok) atomicAdd(&dcnt[0], c_ok);
        if (c_en) atomicAdd(&dcnt[1], c_en);
        if (c_fa) atomicAdd(&dcnt[2], c_fa);
        if (c_fl) atomicAdd(&dcnt[3], c_fl);
        if (c_it) atomicAdd(&dcnt[4], c_it);
        if (corrector == 1 && wmax > 0.0) atomicMax(dmax, (unsigned long long)__double_as_longlong(wmax));
    }
}

template <bool MLP, typename TS>
__global__ void __launch_bounds__(BS) k_update(BlockView v, PhysArgs ph, int corrector, const double* Pb,
                                               const double* __restrict__ Pf, const double* __restrict__ F1,
                                               const double* __restrict__ F2, const double* __restrict__ F3,
                                               const double* __restrict__ Bn, double* Un, double* Po,
                                               uint8_t* __restrict__ status, const double* __restrict__ dscal,
                                               double fac, unsigned long long* dmax, unsigned long long* dcnt) {
    b_update<MLP, TS>(v, ph, corrector, Pb, Pf, F1, F2, F3, Bn, Un, Po, status, dscal, fac, dmax, dcnt,
                      (long)blockIdx.x * blockDim.x + threadIdx.x);
}

template <bool MLP, typename TS>
__global__ void __launch_bounds__(BS, 3) kb_update(const DevBlock* tab, const int* list, PhysArgs ph, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    const bool c = sigma != 0;  // predictor (0) or corrector (2, no CFL rate here) of the block's step
    PhysArgs pb = ph;
    pb.smr_u = D.QR;  // internal SMR: the grouped cells' conserved states (free once the fluxes exist)
    b_update<MLP, TS>(D.v, pb, c ? 2 : 0, D.P, c ? D.Ph : D.P, D.F1, D.F2, D.F3, c ? D.B : D.Bh, D.Un, c ? D.P : D.Ph,
                      D.status, D.dscal, c ? 1.0 : 0.5, D.dmax, D.dcnt, tidx());
}

}  // namespace

cudaError_t launch_update(const BlockView& v, const PhysArgs& ph, int corrector, const double* Pbase,
                          const double* Pflux, double* const F[3], const double* Bnew, double* Un, double* Pout,
                          uint8_t* status, const double* dscal, double dt_factor, unsigned long long* dmax,
                          unsigned long long* dcnt, cudaStream_t s) {
    const long n = (long)v.n1 * v.n2 * v.n3;
    const int bs = ph.mlp_img ? MLP_ROWS : ph.bs_update;  // the network needs one row per thread of 128
    const unsigned nb = nblk(n, bs);
    const int sm = ph.mlp_img ? MLP_SMEM_BYTES : 0;
#define HAMR_UPD_ARGS v, ph, corrector, Pbase, Pflux, F[0], F[1], F[2], Bnew, Un, Pout, status, dscal, dt_factor, dmax, dcnt
    if (ph.mlp_img && ph.mixed)
        k_update<true, float><<<nb, bs, sm, s>>>(HAMR_UPD_ARGS);
    else if (ph.mlp_img)
        k_update<true, double><<<nb, bs, sm, s>>>(HAMR_UPD_ARGS);
    else if (ph.mixed)
        k_update<false, float><<<nb, bs, 0, s>>>(HAMR_UPD_ARGS);
    else
        k_update<false, double><<<nb, bs, 0, s>>>(HAMR_UPD_ARGS);
#undef HAMR_UPD_ARGS
    return cudaGetLastError();
}

cudaError_t launch_update_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, const PhysArgs& ph,
                                int sigma, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    const int bs = ph.mlp_img ? MLP_ROWS : ph.bs_update;
    const dim3 gr = bgrid(maxwork, nlist, bs);
    const int sm = ph.mlp_img ? MLP_SMEM_BYTES : 0;
    if (ph.mlp_img && ph.mixed)
        kb_update<true, float><<<gr, bs, sm, s>>>(tab, list, ph, sigma);
    else if (ph.mlp_img)
        kb_update<true, double><<<gr, bs, sm, s>>>(tab, list, ph, sigma);
    else if (ph.mixed)
        kb_update<false, float><<<gr, bs, 0, s>>>(tab, list, ph, sigma);
    else
        kb_update<false, double><<<gr, bs, 0, s>>>(tab, list, ph, sigma);
    return cudaGetLastError();
}

}  // namespace hamr
