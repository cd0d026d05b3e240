// stage.cuh -- what the stage kernels (step.cu, update.cu) share: indices, the
// centre field, fluid states, sources, floors, the CFL rate, reductions.
#pragma once
#include <type_traits>

#include "c2p.cuh"
#include "ff.cuh"
#include "grmhd.cuh"
#include "hamr_internal.h"

namespace hamr {
namespace {

constexpr int BS = 128;

__device__ __forceinline__ long cidx(const BlockView& v, int i, int j, int k) {
    return ((long)(k + NG) * v.n2p + (j + NG)) * v.n1p + (i + NG);
}
__device__ __forceinline__ long gidx(const BlockView& v, int i, int j) { return (long)(j + NG) * v.n1p + (i + NG); }

inline unsigned nblk(long n, int bs = BS) { return (unsigned)((n + bs - 1) / bs); }

// ---------------------------------------------------------------- centre B
// B^i = (Bbar^i_lo + Bbar^i_hi) / 2 / sqrt(-g)_centre (Sec. 2.5)
__device__ __forceinline__ void centre_field_at(const BlockView& v, const double* __restrict__ B, long stride, long c,
                                                double ig, double Bc[3]) {  // ig = 1 / sqrt(-g)
    const double hig = 0.5 * ig;
    Bc[0] = (B[c] + B[c + 1]) * hig;
    Bc[1] = (B[stride + c] + B[stride + c + v.n1p]) * hig;
    Bc[2] = (B[2 * stride + c] + B[2 * stride + c + (long)v.n1p * v.n2p]) * hig;
}
__device__ __forceinline__ void centre_field(const BlockView& v, const double* __restrict__ B, int i, int j, int k,
                                             double ig, double Bc[3]) {
    centre_field_at(v, B, v.nc, cidx(v, i, j, k), ig, Bc);
}

__device__ __forceinline__ long tidx() { return (long)blockIdx.x * blockDim.x + threadIdx.x; }
inline dim3 bgrid(long maxwork, int nlist, int bs = BS) { return dim3(nblk(maxwork, bs), (unsigned)nlist); }

// What an FP64 face flux keeps of one side. No b^mu or b_mu is formed: with B_nu = g_{nu i} B^i,
// b^t = B^i u_i and i2 = 1/(u^t)^2, b^mu = (B^mu + b^t u^mu)/u^t (B^t = 0), so
//   b^2 = i2 B^2 + Y b^t with B^2 = B^i B_i, Y = i2 b^t,
// and the rows are combinations of u_nu and B_nu (hll_side64).
struct Side64 {
    double ut, u1, u2, u3;   // u^mu
    double c0, c1, c2, c3;   // u_mu
    double k0, k1, k2, k3;   // B_mu
    double iut, s2, Y, bsq;  // 1/u^t, i2 B^2, i2 b^t, b^2
    double g2, i2;           // Gamma^2, 1/(u^t)^2
};

__device__ __forceinline__ void side64(const double pr[NPRIM], const Metric<double>& m, double ac01, Side64& s) {
    const double q1 = pr[U1], q2 = pr[U2], q3 = pr[U3];
    s.c1 = m.g11 * q1 + m.g13 * q3;
    s.c2 = m.g22 * q2;
    s.c3 = m.g13 * q1 + m.g33 * q3;
    s.g2 = fma(q1, s.c1, fma(q2, s.c2, fma(q3, s.c3, 1.0)));
    const double ig = rsqrt(s.g2);
    const double gamma = s.g2 * ig;
    s.ut = gamma * m.ialpha;
    s.u1 = q1 - gamma * ac01;
    s.u2 = q2;
    s.u3 = q3;
    s.c0 = m.g01 * q1 + m.g03 * q3 - m.alpha * gamma;
    const double b1 = pr[B1], b2 = pr[B2], b3 = pr[B3];
    s.k0 = m.g01 * b1 + m.g03 * b3;
    s.k1 = m.g11 * b1 + m.g13 * b3;
    s.k2 = m.g22 * b2;
    s.k3 = m.g13 * b1 + m.g33 * b3;
    const double bt = b1 * s.c1 + b2 * s.c2 + b3 * s.c3;
    s.iut = m.alpha * ig;
    s.i2 = s.iut * s.iut;
    s.s2 = s.i2 * (b1 * s.k1 + b2 * s.k2 + b3 * s.k3);
    s.Y = s.i2 * bt;
    s.bsq = s.s2 + s.Y * bt;
}

// ---------------------------------------------------------------- reductions
// sum_i v_f^i / dx^i at a cell centre (Sec. 2.1 CFL condition), given the fluid state
// (max(|v+|, |v-|) = (|B| + sd)/|A| per direction; the three terms over one denominator)
template <typename T>
__device__ __forceinline__ double inv_dt_fluid(const BlockView& v, const T pr[NPRIM], const Fluid<T>& s,
                                               const Metric<T>& m, T gam) {
    // the quadratic's leading coefficient A = (u^t)^2 (w - gam p) - (b^2 + gam p) g^{tt} is the same
    // in every direction: max(|v+|, |v-|) = (|B_d| + sqrt(B_d^2 - A C_d)) / |A| and one division
    const T p = (gam - T(1)) * pr[UU];
    const T gp = gam * p;
    const T num = s.bsq + gp;
    const T dn = pr[RHO] + pr[UU] + p - gp;
    const T ut = s.ucon[0];
    const T A = ut * ut * dn - num * m.c00;
    const T idx[3] = {to_t<T>(v.idx1), to_t<T>(v.idx2), to_t<T>(v.idx3)};
    T nsum = T(0);
#pragma unroll
    for (int d = 1; d <= 3; d++) {
        const T ud = s.ucon[d];
        const T B = ut * ud * dn - num * gcon0(m, d);
        const T C = ud * ud * dn - num * gcondd(m, d);
        nsum += (fabs(B) + root_pos(B * B - A * C)) * idx[d - 1];
    }
    return to_d(nsum / fabs(A));
}

template <typename T>
__device__ __forceinline__ double inv_dt_cell(const BlockView& v, const T pr[NPRIM], const Metric<T>& m, T gam) {
    Fluid<T> s;
    fluid_state(pr, m, s);
    return inv_dt_fluid(v, pr, s, m, gam);
}

// source sqrt(-g) T^k_l Gamma^l_{nu k} at a cell centre in precision T
// (tables gc: metric and connection planes of that precision)
template <typename T, typename TT>
__device__ __forceinline__ void source_q_state(const TT* __restrict__ gc, long n2d, long g, const Metric<T>& m,
                                              const T pf[NPRIM], const Fluid<T>& s, T gam, T Q[4]) {
    const T p = (gam - T(1)) * pf[UU];
    const T eta = pf[RHO] + pf[UU] + p + s.bsq;
    const T ptot = p + T(0.5) * s.bsq;
    T Tm[4][4];
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++)
            Tm[a][b] = eta * s.ucon[a] * s.ucov[b] - s.bcon[a] * s.bcov[b] + ((a == b) ? ptot : T(0));
    const TT* cn = gc + (long)C_CONN * n2d + g;
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
        T acc = T(0);
#pragma unroll
        for (int l = 0; l < 4; l++)
#pragma unroll
            for (int kk = 0; kk < 4; kk++) acc += Tm[kk][l] * (T)cn[(l * 10 + sym(nu, kk)) * n2d];
        Q[nu] = acc * m.gdet;
    }
}

// The same source in FP64 from the stored metric derivatives: with the Christoffel
// symbols formed from the derivatives d_s g of the metric whose inverse raises T,
// T^k_l Gamma^l_{nu k} = (1/2) T^{kl} d_nu g_{kl} (the terms with d_k g_{l nu} - d_l g_{nu k}
// cancel against the symmetric T^{kl}), so Q_t = Q_phi = 0 (stationary, axisymmetric
// metric) and Q_1, Q_2 contract the 7 non-zero d_s g_{mn}; the same number up to
// rounding order, with a third of the operations. With b^mu = (B^mu + b^t u^mu)/u^t
//   T^{mn} = (rho h + i2 B^2) u^m u^n - Y (B^m u^n + u^m B^n) - i2 B^m B^n + ptot g^{mn}
//          = h^m u^n - B^n g^m + ptot g^{mn}, h = (rho h + i2 B^2) u - Y B, g = Y u + i2 B.
// Q: Q_1 and Q_2 without sqrt(-g).
__device__ __forceinline__ void source64(const double* __restrict__ gc, long n2d, long g, const Metric<double>& m,
                                         const double pf[NPRIM], const Side64& s, double gam, double& Q1, double& Q2) {
    const double w = fma(gam, pf[UU], pf[RHO]) + s.s2;
    const double ptot = (gam - 1.0) * pf[UU] + 0.5 * s.bsq;
    const double b1 = pf[B1], b2 = pf[B2], b3 = pf[B3];
    const double h1 = w * s.u1 - s.Y * b1, h2 = w * s.u2 - s.Y * b2, h3 = w * s.u3 - s.Y * b3;
    const double g1 = s.Y * s.u1 + s.i2 * b1, g2 = s.Y * s.u2 + s.i2 * b2, g3 = s.Y * s.u3 + s.i2 * b3;
    const double T[7] = {w * s.ut * s.ut + ptot * m.c00,           h1 * s.ut + ptot * m.c01,
                         h3 * s.ut,                                h1 * s.u1 + (-b1 * g1 + ptot * m.c11),
                         h1 * s.u3 + (-b3 * g1 + ptot * m.c13),    h2 * s.u2 + (-b2 * g2 + ptot * m.c22),
                         h3 * s.u3 + (-b3 * g3 + ptot * m.c33)};
    const double* d = gc + (long)C_DG * n2d + g;
    Q1 = Q2 = 0.0;
#pragma unroll
    for (int k = 0; k < 7; k++) {
        Q1 += T[k] * d[k * n2d];
        Q2 += T[k] * d[(7 + k) * n2d];
    }
}

// The same from b^mu, as the mixed form with the FP64 source takes it (Q: all four, times sqrt(-g)).
__device__ __forceinline__ void source_q_dg(const double* __restrict__ gc, long n2d, long g, const Metric<double>& m,
                                            const double pf[NPRIM], const Fluid<double>& s, double gam, double Q[4]) {
    const double p = (gam - 1.0) * pf[UU];
    const double eta = pf[RHO] + pf[UU] + p + s.bsq;
    const double ptot = p + 0.5 * s.bsq;
    const double* u = s.ucon;
    const double* b = s.bcon;
    const double e0 = eta * u[0], e1 = eta * u[1], e3 = eta * u[3];
    const double T[7] = {e0 * u[0] - b[0] * b[0] + ptot * m.c00, e0 * u[1] - b[0] * b[1] + ptot * m.c01,
                         e0 * u[3] - b[0] * b[3],                e1 * u[1] - b[1] * b[1] + ptot * m.c11,
                         e1 * u[3] - b[1] * b[3] + ptot * m.c13, eta * u[2] * u[2] - b[2] * b[2] + ptot * m.c22,
                         e3 * u[3] - b[3] * b[3] + ptot * m.c33};
    const double* d = gc + (long)C_DG * n2d + g;
    double q1 = 0.0, q2 = 0.0;
#pragma unroll
    for (int k = 0; k < 7; k++) {
        q1 += T[k] * d[k * n2d];
        q2 += T[k] * d[(7 + k) * n2d];
    }
    Q[0] = 0.0;
    Q[1] = q1 * m.gdet;
    Q[2] = q2 * m.gdet;
    Q[3] = 0.0;
}

// adds the warp's cells to the counters of a step: inversions by outcome st (-1: none), floors, iterations
__device__ __forceinline__ void count_cells(int st, int fl, int its, unsigned long long* dcnt) {
    const unsigned all = 0xffffffffu;
    const int c[5] = {__popc(__ballot_sync(all, st == INV_OK)), __popc(__ballot_sync(all, st == INV_ENTROPY)),
                      __popc(__ballot_sync(all, st == INV_FAIL)), __popc(__ballot_sync(all, fl != 0)),
                      __reduce_add_sync(all, its)};
    if ((threadIdx.x & 31u) == 0) {
#pragma unroll
        for (int q = 0; q < 5; q++)
            if (c[q]) atomicAdd(&dcnt[q], (unsigned long long)c[q]);
    }
}

// ---- the CFL rate in FP32, to leave out the FP64 one where it cannot be the largest
// Estimate of inv_dt_fluid from (rho, u, b^2), all scaled by one factor, and u^mu; negative where it says
// nothing. Its discriminant may lose all digits to cancellation: the root's error is then below
// sqrt(2^-22) = 5e-4 of |B|, so the estimate is within 1e-3 of the rate wherever num g^{dd} stays in range.
__device__ __forceinline__ float rate_estimate(const BlockView& v, const PhysArgs& ph, float rho, float u, float bsq,
                                               float ut, const float ud[3], float c00, float c01, float c11, float c22,
                                               float c33) {
    const float num = bsq + ph.cs2h * u, dn = rho + ph.wmph * u;
    const float A = ut * ut * dn - num * c00;
    const float c0[3] = {c01, 0.0f, 0.0f}, cd[3] = {c11, c22, c33};
    const float idx[3] = {narrow(v.idx1), narrow(v.idx2), narrow(v.idx3)};
    float sum = 0.0f;
    bool ok = A > 1e-15f;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const float B = ut * ud[d] * dn - num * c0[d];
        const float C = ud[d] * ud[d] * dn - num * cd[d];
        const float s = B * B - A * C;
        sum += (fabsf(B) + (s > 0.0f ? sqrtf(s) : 0.0f)) * idx[d];
        ok = ok && num * cd[d] > 1e-20f;
    }
    return ok ? sum / A : -1.0f;
}
// true where a rate of this estimate is certainly below the largest found so far (margin 1%)
__device__ __forceinline__ bool rate_below(float est, const unsigned long long* dmax) {
    const float cur = narrow(__longlong_as_double((long long)*(const volatile unsigned long long*)dmax));
    return est >= 0.0f && est * 1.01f < cur;
}
// 2^(sh >> 20) brings the largest of three values to [1, 2) (0 where that is not above 2^-767)
__device__ __forceinline__ int scale_of(double a, double b, double c) {
    const int e = max(max(__double2hiint(a), __double2hiint(b)), __double2hiint(c)) & 0x7ff00000;
    return e > 0x10000000 ? 0x3ff00000 - e : 0;
}

// largest of the warp's (non-negative) rates into *dmax
__device__ __forceinline__ void reduce_rate(double inv, unsigned long long* dmax) {
    const bool some = inv > 0.0;  // NaNs count as nothing
    if (!__any_sync(0xffffffffu, some)) return;
    unsigned long long b = some ? (unsigned long long)__double_as_longlong(inv) : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, b, o);
        b = x > b ? x : b;
    }
    if ((threadIdx.x & 31u) == 0) atomicMax(dmax, b);
}

// Floors in the drift frame (Sec. 2.7, after Ressler et al. 2017): the floor
// material, drho = rho_f - rho and du = u_f - u (each >= 0), moves with the
// drift velocity of the field lines, the part of the normal-frame velocity
// across B, v_d = v - (v.Bn / Bn^2) Bn (v_d = v where B = 0). Its stress-energy
// (no field) is added to the cell's in conserved form, the entropy slot keeps
// the cell's kappa, and the sum is inverted with the same B from rho_f, u_f at
// the drift velocity. The material brings no momentum along B, so a flow along
// the field slows as mass is added; the fluid-frame floor is applied to the
// result. false when the inversion fails (the caller then takes the fluid-frame
// floor).
__device__ __forceinline__ bool drift_floor(const Metric<double>& m, const PhysArgs& ph, double pr[NPRIM],
                                            const Fluid<double>& s, double rf, double uf) {
    const double gam = ph.gam;
    const double q1 = pr[U1], q2 = pr[U2], q3 = pr[U3];
    const double qsq = m.g11 * q1 * q1 + m.g22 * q2 * q2 + m.g33 * q3 * q3 + 2.0 * m.g13 * q1 * q3;
    const double ig = 1.0 / sqrt(1.0 + qsq);
    const double v1 = q1 * ig, v2 = q2 * ig, v3 = q3 * ig;
    const double b1 = m.alpha * pr[B1], b2 = m.alpha * pr[B2], b3 = m.alpha * pr[B3];
    const double bn2 = m.g11 * b1 * b1 + m.g22 * b2 * b2 + m.g33 * b3 * b3 + 2.0 * m.g13 * b1 * b3;
    const double vb = m.g11 * v1 * b1 + m.g22 * v2 * b2 + m.g33 * v3 * b3 + m.g13 * (v1 * b3 + v3 * b1);
    const double f = (bn2 > 0.0) ? vb / bn2 : 0.0;
    const double d1 = v1 - f * b1, d2 = v2 - f * b2, d3 = v3 - f * b3;
    const double vd2 = m.g11 * d1 * d1 + m.g22 * d2 * d2 + m.g33 * d3 * d3 + 2.0 * m.g13 * d1 * d3;
    const double gd = 1.0 / sqrt(1.0 - vd2);
    double pa[NPRIM] = {fmax(rf - pr[RHO], 0.0), fmax(uf - pr[UU], 0.0), gd * d1, gd * d2, gd * d3, 0.0, 0.0, 0.0};
    Fluid<double> sa;
    fluid_state(pa, m, sa);
    double uo[NFLUX], ua[NFLUX];
    flux_row(pr, s, 0, 1, gam, entropy_kappa(pr, gam), uo);
    flux_row(pa, sa, 0, 1, gam, 0.0, ua);
    double U[NCONS];
#pragma unroll
    for (int q = 0; q < 5; q++) U[q] = m.gdet * (uo[q] + ua[q]);
    U[C_ENT] = m.gdet * uo[5] / uo[0] * (uo[0] + ua[0]);
    double x[NPRIM];
#pragma unroll
    for (int q = 0; q < NPRIM; q++) x[q] = pr[q];
    x[RHO] = fmax(pr[RHO], rf);
    x[UU] = fmax(pr[UU], uf);
    x[U1] = pa[U1];
    x[U2] = pa[U2];
    x[U3] = pa[U3];
    const double Bc[3] = {pr[B1], pr[B2], pr[B3]};
    int its = 0;
    if (invert(U, Bc, m, gam, x, &its, false, nullptr, ph.inversion, ph.mixed ? C2P_NEWTON64 : C2P_NEWTON_FF) ==
        INV_FAIL)
        return false;
    pr[RHO] = fmax(x[RHO], rf);
    pr[UU] = fmax(x[UU], uf);
    pr[U1] = x[U1];
    pr[U2] = x[U2];
    pr[U3] = x[U3];
    return true;
}

// Floors (Sec. 2.7): rho >= max(1e-7/r^2, b^2/50), u >= max(1e-9/r^(10/3),
// b^2/750) with b^2 of pr; HAMR_FLOOR_FLUID raises rho and u (utilde kept),
// HAMR_FLOOR_DRIFT adds the material in the drift frame. s: the fluid state
// of pr on entry, and again on return (recomputed where the velocity moved).
// Returns 1 where a floor applied.
__device__ __forceinline__ int cell_floors(const BlockView& v, long g, const Metric<double>& m, const PhysArgs& ph,
                                           double pr[NPRIM], Fluid<double>& s) {
    const double rf = fmax(v.gc[C_RHOFLR * v.n2d + g], s.bsq * (1.0 / 50.0));
    const double uf = fmax(v.gc[C_UFLR * v.n2d + g], s.bsq * (1.0 / 750.0));
    if (!(pr[RHO] < rf) && !(pr[UU] < uf)) return 0;
    if (ph.floor_frame == HAMR_FLOOR_DRIFT && drift_floor(m, ph, pr, s, rf, uf)) {
        fluid_state(pr, m, s);
        return 1;
    }
    if (pr[RHO] < rf) pr[RHO] = rf;
    if (pr[UU] < uf) pr[UU] = uf;
    return 1;
}

// The same floors with b^2 given (the cell updates; the mixed-precision one takes it from its FP32 fluid
// state); the drift frame forms the FP64 fluid state of pr where a floor applies.
__device__ __forceinline__ int cell_floors_b2(const BlockView& v, long g, const Metric<double>& m, const PhysArgs& ph,
                                              double pr[NPRIM], double bsq) {
    const double rf = fmax(v.gc[C_RHOFLR * v.n2d + g], bsq * (1.0 / 50.0));
    const double uf = fmax(v.gc[C_UFLR * v.n2d + g], bsq * (1.0 / 750.0));
    if (!(pr[RHO] < rf) && !(pr[UU] < uf)) return 0;
    if (ph.floor_frame == HAMR_FLOOR_DRIFT) {
        Fluid<double> s;
        fluid_state(pr, m, s);
        if (drift_floor(m, ph, pr, s, rf, uf)) return 1;
    }
    if (pr[RHO] < rf) pr[RHO] = rf;
    if (pr[UU] < uf) pr[UU] = uf;
    return 1;
}

// the next stage's FP32 copy of cell c (p: the returned primitives rounded to FP32) and its entropy
// tracer kappa = (gam - 1) u / rho^gam formed as the kappa pass forms it; in the corrector also the
// next step's U^n kappa (the entropy slot of the U^n cache, which the predictor reads)
__device__ __forceinline__ void store_stage32(const BlockView& v, const PhysArgs& ph, int corrector, long c,
                                              const float p[NPRIM]) {
#pragma unroll
    for (int q = 0; q < NPRIM; q++) ph.p32w[q * v.nc + c] = p[q];
    const float g32 = narrow(ph.gam);
    const float kap = (g32 - 1.0f) * p[UU] * pow_pos(p[RHO], -g32);
    ph.k32[c] = kap;
    if (corrector == 1) ph.un[(long)C_ENT * v.nc + c] = widen(kap);
}

// The fluid-frame floors of the mixed form in FP32: b^2 of the FP32 fluid state (like the fluxes),
// thresholds, comparisons and floor values in FP32 (pf: the returned primitives rounded to FP32, updated
// with pr)
__device__ __forceinline__ int cell_floors_fluid32(const BlockView& v, long g, double pr[NPRIM], float pf[NPRIM],
                                                   float bsq) {
    const float rf = fmaxf(narrow(v.gc[C_RHOFLR * v.n2d + g]), bsq * (1.0f / 50.0f));
    const float uf = fmaxf(narrow(v.gc[C_UFLR * v.n2d + g]), bsq * (1.0f / 750.0f));
    const bool lr = pf[RHO] < rf, lu = pf[UU] < uf;
    if (!lr && !lu) return 0;
    if (lr) {
        pf[RHO] = rf;
        pr[RHO] = widen(rf);
    }
    if (lu) {
        pf[UU] = uf;
        pr[UU] = widen(uf);
    }
    return 1;
}

// The same, or the drift frame's by the FP64 path of cell_floors_b2
__device__ __forceinline__ int cell_floors_f32(const BlockView& v, long g, const Metric<double>& m, const PhysArgs& ph,
                                               double pr[NPRIM], float pf[NPRIM], float bsq) {
    if (ph.floor_frame == HAMR_FLOOR_DRIFT) {
        const int fl = cell_floors_b2(v, g, m, ph, pr, widen(bsq));
        if (fl)
#pragma unroll
            for (int q = 0; q < NPRIM; q++) pf[q] = narrow(pr[q]);
        return fl;
    }
    return cell_floors_fluid32(v, g, pr, pf, bsq);
}

}  // namespace
}  // namespace hamr
