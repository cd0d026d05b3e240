// c2p.cuh -- conserved-to-primitive inversion (Liska et al. 2019, Sec. 2.6).
//
// Primary: 2-D Newton-Raphson on W = w Gamma^2 and v^2 = 1 - 1/Gamma^2 for
// the two scalar equations of the energy and the projected momentum in the
// normal-observer frame (the formulation of Noble et al. 2006). Backup when
// it fails: the entropy equation replaces the energy one, p = kappa rho^gam
// with kappa = U_kappa / U_rho, and a 1-D Newton in W solves the projected
// momentum equation (Noble et al. 2009). A state where both fail keeps its
// guess.
//
// Stopping rule: |dW|/W + |dv^2| < 1e-10 (quadratic convergence leaves the
// accepted iterate at round-off), at most 30 iterations; v^2 is kept
// in [0, 1 - 1/50^2].
#pragma once
#include "../../include/hamr.h"
#include "ff.cuh"
#include "grmhd.cuh"

namespace hamr {

constexpr double C2P_TOL = 1.0e-10;
constexpr int C2P_NMAX = 30;
constexpr double C2P_VSQMAX = 1.0 - 1.0 / (50.0 * 50.0);

enum { INV_OK = 0, INV_ENTROPY = 1, INV_FAIL = 2 };

// how Newton iterates: in double-float with an FP64 last solve (newton_wv_ff), in FP32 with one FP64
// refinement step (newton_wv_mixed), or in FP64 (newton_wv: grids of the mixed forms, update.cu).
// C2P_NEWTON_ANY: newton_wv_ff from a start that may be anywhere (the standalone inversion), which gives up
// its double-float iterations early, and the FP64 entropy backup alone
enum { C2P_NEWTON_FF = 0, C2P_NEWTON32 = 1, C2P_NEWTON64 = 2, C2P_NEWTON_ANY = 3 };

// The normal-frame scalars of a conserved state (Sec. 2.6, Noble et al. 2006).
struct C2PScalars {
    double D, Qdotn, Qtsq, Bsq, QdotB, QB2;
    double Qc1, Qc2, Qc3, Bn1, Bn2, Bn3;
};

// U: sqrt(-g) (rho u^t, T^t_t + rho u^t, T^t_i, kappa rho u^t); Bc: centre B^i.
__device__ __forceinline__ void c2p_scalars(const double U[NCONS], const double Bc[3], const Metric<double>& m,
                                            C2PScalars& S) {
    const double al = m.alpha;
    const double aig = al * m.igdet;  // alpha / sqrt(-g), formed once
    S.D = U[C_RHO] * aig;
    // Q_mu = alpha T^t_mu, raised with the sparse inverse metric
    const double Q0 = (U[C_EN] - U[C_RHO]) * aig;
    const double Q1 = U[C_S1] * aig;
    const double Q2 = U[C_S2] * aig;
    const double Q3 = U[C_S3] * aig;
    const double Qc0 = m.c00 * Q0 + m.c01 * Q1;
    S.Qc1 = m.c01 * Q0 + m.c11 * Q1 + m.c13 * Q3;
    S.Qc2 = m.c22 * Q2;
    S.Qc3 = m.c13 * Q1 + m.c33 * Q3;
    S.Bn1 = al * Bc[0];
    S.Bn2 = al * Bc[1];
    S.Bn3 = al * Bc[2];
    S.Qdotn = -al * Qc0;
    S.Qtsq = Q0 * Qc0 + Q1 * S.Qc1 + Q2 * S.Qc2 + Q3 * S.Qc3 + S.Qdotn * S.Qdotn;
    S.Bsq = m.g11 * S.Bn1 * S.Bn1 + m.g22 * S.Bn2 * S.Bn2 + m.g33 * S.Bn3 * S.Bn3 + 2.0 * m.g13 * S.Bn1 * S.Bn3;
    S.QdotB = Q1 * S.Bn1 + Q2 * S.Bn2 + Q3 * S.Bn3;
    S.QB2 = S.QdotB * S.QdotB;
}

// 2-D Newton on (W, v^2) from the given start; true when it met the
// stopping rule. `it` returns the iterations taken.
__device__ __forceinline__ bool newton_wv(const C2PScalars& S, double gfac, double& W, double& vsq, int& it) {
    const double D = S.D, Bsq = S.Bsq, QB2 = S.QB2, Qdotn = S.Qdotn, Qtsq = S.Qtsq;
    bool ok = false;
    for (it = 1; it <= C2P_NMAX; it++) {
        const double omv = 1.0 - vsq;
        const double rs = rsqrt(omv);
        const double sq = omv * rs;
        const double W2 = W * W, W3 = W2 * W;
        const double BW = Bsq + W;
        const double p = gfac * (W * omv - D * sq);
        // the residuals f1, f2 times W^2 and the Jacobian's first column (d/dW) times W^3, so that no
        // 1/W is formed: with det' = det W^3 the Newton step is dW = W (j12 f2' - j22 f1') / det',
        // dv = (j21' f1' - j11' f2') / (W^2 det'), both from the one reciprocal of W^2 det'
        const double f1 = (-0.5 * Bsq * (1.0 + vsq) - W + p - Qdotn) * W2 + 0.5 * QB2;
        const double f2 = (vsq * BW * BW - Qtsq) * W2 - QB2 * (Bsq + 2.0 * W);
        const double j11 = (gfac * omv - 1.0) * W3 - QB2;
        const double j12 = -0.5 * Bsq + gfac * (0.5 * D * rs - W);
        const double j21 = 2.0 * BW * (vsq * W3 + QB2);
        const double j22 = BW * BW;
        const double r = 1.0 / ((j11 * j22 - j12 * j21) * W2);
        const double dW = (j12 * f2 - j22 * f1) * W3 * r;
        const double dv = (j21 * f1 - j11 * f2) * r;
        const double Wn = W + dW;
        const double vn = fmin(fmax(vsq + dv, 0.0), C2P_VSQMAX);
        if (!(Wn > 0.0)) break;
        const double err = fabs(Wn - W) + fabs(vn - vsq) * Wn;
        W = Wn;
        vsq = vn;
        if (err < C2P_TOL * Wn) {
            ok = true;
            break;
        }
    }
    if (it > C2P_NMAX) it = C2P_NMAX;
    return ok;
}

// newton_wv out of line, for the callers below whose common path it is not (its registers and code
// stay out of theirs)
struct NewtonOut {
    double W, vsq;
    int it;
    bool ok;
};
static __device__ __noinline__ NewtonOut newton_wv_call(const C2PScalars* S, double gfac, double W, double vsq) {
    NewtonOut o;
    o.ok = newton_wv(*S, gfac, W, vsq, o.it);
    o.W = W;
    o.vsq = vsq;
    return o;
}

// newton_wv with its iterations in double-float (ff.cuh) and the last word from FP64: the same
// iterations, from the same start to the same stopping rule, on the equations scaled by the power of two
// that brings the start's W to [1, 2) (f1 ~ W, f2 ~ W^2), on the FP32 pipe; then the FP64 residuals at
// that root, solved with the Jacobian of the last iteration. The double-float root is 1e-13 or better, so
// that solve (relative error of the Jacobian 1e-7 times its cancellation) leaves what FP64 residuals
// resolve, like newton_wv's own last iterate. Where the steps still shrink slowly at the end (not by 1e-3;
// v^2 near its limit), newton_wv stops short of the root by up to its tolerance, and where a step is within
// the double-float steps' noise (1e-13 times the cancellation) of the tolerance, rounding decides whether it
// stops: both are left to it. Taken when the step and the step times the cancellation
// (|j11 j22| + |j12 j21|) / |det| are as small as that argument needs; otherwise, and wherever the
// double-float iteration meets no root or leaves its range, newton_wv decides. `it` counts the iterations,
// not the solve. rs: 1/sqrt(1 - v^2) at the root where it comes for free, else 0.
// An FP64 iteration is ~52 FP64 instructions (64 cycles each per scheduler), here ~340 FP32 ones, plus
// ~28 FP64 for the solve: 1M states from a 5% start (4.7 iterations) 1035 -> 626 us, the FP64
// cell update of the 256x128x64 torus 2.00 -> 1.50 ms with the entropy backup below.
// any: the start may be far off (no previous state). From such starts many states meet no root, and a warp
// with one of them waits for 30 iterations in double-float and then for 30 in FP64: a fourth step that still
// moves the root by a quarter of W ends the first. 1M states at rest (14% without an energy root) take
// 12.7 ms, 16.8 without the rule, 12.0 with FP64 alone; 30 to 50% off 8.1, 6.9 and 7.9 ms. The cell updates do
// without it: their failing cells are few, and cells that get there in more steps would go to FP64.
// Lanes leave by several ways (root taken, FP64 after each of the breaks, early break there), and the compiler
// brings them together as late as it may: callers put a __syncwarp() behind the attempt, without which the
// entropy backup ran once for each way (1M states at rest 17.5 ms).
__device__ __forceinline__ bool newton_wv_ff(const C2PScalars& S, double gfac, double& W, double& vsq, int& it,
                                             double& rs64, bool any) {
    rs64 = 0.0;
    const unsigned eW = (unsigned)__double2hiint(W) & 0xfff00000u;  // sign and exponent of the start
    bool ok = false;
    if (eW - 0x2b000000u < 0x2a000000u) {  // W positive, 2^-334 .. 2^337
        const unsigned sh = 0x3ff00000u - eW;
        const ff D = ff_of(S.D, (int)sh), B2 = ff_of(S.Bsq, (int)sh), Qn = ff_of(S.Qdotn, (int)sh);
        const ff Qt = ff_of(S.Qtsq, (int)(2u * sh)), QB = ff_of(S.QB2, (int)(3u * sh));
        const ff gf = ff_of(gfac), one{1.0f, 0.0f};
        const ff vmax{(float)C2P_VSQMAX, (float)(C2P_VSQMAX - (double)(float)C2P_VSQMAX)};
        const ff hB = ff_scale(B2, 0.5f), c1 = ff_neg(ff_add(hB, Qn));
        ff w = ff_of(W, (int)sh), v = ff_of(vsq);
        float j11h = 0.0f, j12h = 0.0f, j21h = 0.0f, j22h = 0.0f, idh = 0.0f, iwh = 0.0f, rsh = 0.0f;
        float before = 1e30f, cancel = 0.0f;  // the step before; the Jacobian's cancellation
        for (it = 1; it <= C2P_NMAX; it++) {
            const ff omv = ff_sub(one, v);
            const ff rs = ff_rsqrt(omv);
            const ff bw = ff_add(B2, w);
            const ff p = ff_mul(gf, ff_sub(ff_mul(w, omv), ff_mul(D, ff_mul(omv, rs))));
            const ff iw = ff_rcp(w);
            const ff q2 = ff_mul(QB, ff_mul(iw, iw)), q3 = ff_mul(q2, iw);
            const ff j22 = ff_mul(bw, bw);
            // f1 = -B^2 (1 + v)/2 + QB2/(2 W^2) - W + p - Q.n, f2 = v (B^2 + W)^2 - QB2 (B^2 + 2 W)/W^2 - Qt^2
            const ff f1 = ff_add(ff_sub(ff_sub(ff_scale(q2, 0.5f), w), ff_mul(hB, v)), ff_add(p, c1));
            const ff f2 = ff_sub(ff_sub(ff_mul(v, j22), Qt), ff_mul(q2, ff_add(bw, w)));
            const ff j11 = ff_sub(ff_sub(ff_mul(gf, omv), one), q3);
            const ff j12 = ff_sub(ff_mul(gf, ff_sub(ff_scale(ff_mul(D, rs), 0.5f), w)), hB);
            const ff j21 = ff_scale(ff_mul(bw, ff_add(v, q3)), 2.0f);
            const ff id = ff_rcp(ff_sub(ff_mul(j11, j22), ff_mul(j12, j21)));
            const ff dw = ff_mul(ff_sub(ff_mul(j12, f2), ff_mul(j22, f1)), id);
            const ff dv = ff_mul(ff_sub(ff_mul(j21, f1), ff_mul(j11, f2)), id);
            const ff wn = ff_add(w, dw);
            ff vn = ff_add(v, dv);
            if (vn.h < 0.0f) vn = ff{0.0f, 0.0f};
            if (!ff_less(vn, vmax)) vn = vmax;
            if (!(wn.h > 0.0f && wn.h < 1e9f)) break;  // NaNs too
            const float err = fabsf(dw.h) + fabsf((vn.h - v.h) + (vn.l - v.l)) * wn.h;
            w = wn;
            v = vn;
            // the steps' noise: 2^-46 or so times the Jacobian's cancellation. Where that comes near the
            // tolerance, or the steps have stopped shrinking, FP64 decides
            cancel = (fabsf(j11.h * j22.h) + fabsf(j12.h * j21.h)) * fabsf(id.h);
            const float tol = (float)C2P_TOL * wn.h, noise = 1e-13f * cancel * wn.h;
            if (noise > 0.5f * tol || (err > 0.25f * before && before < 1e-6f * wn.h)) break;
            if (any && it >= 4 && err > 0.25f * wn.h) break;
            if (err < tol) {
                ok = err + noise < tol && before > tol + noise && (err < 1e-3f * before || err < 0.1f * tol);
                j11h = j11.h;
                j12h = j12.h;
                j21h = j21.h;
                j22h = j22.h;
                idh = id.h;
                iwh = iw.h;
                rsh = rs.h;
                break;
            }
            before = err;
        }
        if (ok) {
            double Wd = ff_d(w);  // in [2^-40, 2^30]: the exponent added back as an integer
            Wd = __hiloint2double((int)((unsigned)__double2hiint(Wd) - sh), __double2loint(Wd));
            const double vd = ff_d(v);
            const double omv = 1.0 - vd;
            const double r = rsqrt(omv);
            const double W2 = Wd * Wd, BW = S.Bsq + Wd;
            const double p = gfac * (Wd * omv - S.D * (omv * r));
            const double f1 = (-0.5 * S.Bsq * (1.0 + vd) - Wd + p - S.Qdotn) * W2 + 0.5 * S.QB2;
            const double f2 = (vd * BW * BW - S.Qtsq) * W2 - S.QB2 * (BW + Wd);
            const float iw2 = iwh * iwh;
            const float r1 = ff_of(f1, (int)(3u * sh)).h * iw2, r2 = ff_of(f2, (int)(4u * sh)).h * iw2;
            const float dw = (j12h * r2 - j22h * r1) * idh, dv = (j21h * r1 - j11h * r2) * idh;
            const float step = fabsf(dw) + fabsf(dv) * w.h;
            const double vn = vd + widen(dv);
            const long long vb = __double_as_longlong(vn);
            if (step < 1e-9f * w.h && step * cancel < 1e-8f * w.h && vb >= 0 &&
                vb <= __double_as_longlong(C2P_VSQMAX)) {
                W = fma(widen(dw), __hiloint2double((int)eW, 0), Wd);  // 2^e dw
                vsq = vn;
                // the root moved by dv: 1/sqrt(1 - v^2) moves by half of y = dv / (1 - v^2), to second order
                const float y = dv * rsh * rsh;
                if (fabsf(y) < 1e-8f) rs64 = fma(r, widen(0.5f * y), r);
                return true;
            }
        }
    }
    const C2PScalars T = S;
    const NewtonOut o = newton_wv_call(&T, gfac, W, vsq);
    W = o.W;
    vsq = o.vsq;
    it = o.it;
    return o.ok;
}

// Mixed precision (the FP32-flux form only): FP32 Newton iterations first, on
// the two equations scaled by k = 2^-e, e the binary exponent of the start's W
// (an exact scaling; every term then O(1): f1 ~ W, f2 ~ W^2, so D, B^2, Q.n
// scale by k, Qt^2 by k^2, (Q.B)^2 by k^3), until a step is below 1e-5 W (at
// most 8). Then one refinement step in the manner of mixed-precision iterative
// refinement: the FP64 residuals at the FP32 root, solved with the FP32
// Jacobian there; it shrinks the root's error (~1e-7 W) by the Jacobian's
// relative error times its condition, to the FP64 level. It is accepted when
// the step is below 1e-5 W and that bound times the Jacobian's cancellation
// (|j11 j22| + |j12 j21|) / |det| stays below 1e-3 W (the remaining error of
// order 1e-10 W, the FP64 rule's); otherwise FP64 Newton iterations run from
// the refined point, stopping at the usual rule. When the FP32 stage does not
// converge the FP64 iteration runs from the original start alone. `it` counts
// the iterations of both precisions (the refinement as one).
__device__ __forceinline__ bool newton_wv_mixed(const C2PScalars& S, double gfac, double& W, double& vsq, int& it) {
    // the scalars rounded to FP32 first and scaled there (their magnitudes stay far inside FP32's
    // range for admissible states; a start outside the normal FP32 range takes the FP64 iteration)
    const float Wf = narrow(W);
    const unsigned eb = (__float_as_uint(Wf) >> 23) & 0xffu;  // biased exponent of the start
    if (!(Wf > 0.0f) || eb == 0u || eb >= 254u) {
        const C2PScalars T = S;
        const NewtonOut o = newton_wv_call(&T, gfac, W, vsq);
        W = o.W;
        vsq = o.vsq;
        it = o.it;
        return o.ok;
    }
    const float k = __uint_as_float((254u - eb) << 23);  // 2^(127 - eb): w = W k in [1, 2)
    const float k2 = k * k;
    const float D = narrow(S.D) * k, Bsq = narrow(S.Bsq) * k, Qdotn = narrow(S.Qdotn) * k;
    const float Qtsq = narrow(S.Qtsq) * k2, QB2 = narrow(S.QB2) * (k2 * k);
    const float gf = narrow(gfac), vmax = (float)C2P_VSQMAX;
    float w = Wf * k, v = narrow(vsq);
    bool ok32 = false;
    int it32 = 0;
    for (it32 = 1; it32 <= 8; it32++) {
        const float omv = 1.0f - v;
        const float rs = rsqrtf(omv);
        const float sq = omv * rs;
        const float iw = 1.0f / w;
        const float iw2 = iw * iw;
        const float bw = Bsq + w;
        const float p = gf * (w * omv - D * sq);
        const float f1 = -0.5f * Bsq * (1.0f + v) + 0.5f * QB2 * iw2 - w + p - Qdotn;
        const float f2 = v * bw * bw - QB2 * (Bsq + 2.0f * w) * iw2 - Qtsq;
        const float j11 = -QB2 * iw2 * iw - 1.0f + gf * omv;
        const float j12 = -0.5f * Bsq + gf * (0.5f * D * rs - w);
        const float j21 = 2.0f * bw * (v + QB2 * iw2 * iw);
        const float j22 = bw * bw;
        const float idet = 1.0f / (j11 * j22 - j12 * j21);
        const float wn = w + (j12 * f2 - j22 * f1) * idet;
        const float vn = fminf(fmaxf(v + (j21 * f1 - j11 * f2) * idet, 0.0f), vmax);
        if (!(wn > 0.0f) || !(wn < 1e30f)) break;
        const float err = fabsf(wn - w) + fabsf(vn - v) * wn;
        w = wn;
        v = vn;
        if (err < 1e-5f * wn) {
            ok32 = true;
            break;
        }
    }
    if (it32 > 8) it32 = 8;
    if (!ok32) {  // the FP64 iteration from the original start
        const C2PScalars T = S;
        const NewtonOut o = newton_wv_call(&T, gfac, W, vsq);
        W = o.W;
        vsq = o.vsq;
        it = o.it + it32;
        return o.ok;
    }
    const double D64 = S.D, Bsq64 = S.Bsq, QB264 = S.QB2, Qdotn64 = S.Qdotn, Qtsq64 = S.Qtsq;
    // the FP32 root in FP64 (W = w / k exactly) and the exact powers 1/k, k^3, k^4 in FP64
    const int ed = (int)eb - 127;  // 1/k = 2^ed
    const double ik = __hiloint2double((1023 + ed) << 20, 0);
    const double k3 = __hiloint2double((1023 - 3 * ed) << 20, 0), k4 = __hiloint2double((1023 - 4 * ed) << 20, 0);
    double Wd = widen(w) * ik, vd = widen(v);
    {
        // FP64 residuals of newton_wv's form (times W^2) at the root
        const double omv = 1.0 - vd;
        const double sq = omv * rsqrt(omv);
        const double W2 = Wd * Wd;
        const double BW = Bsq64 + Wd;
        const double p = gfac * (Wd * omv - D64 * sq);
        const double f1 = (-0.5 * Bsq64 * (1.0 + vd) - Wd + p - Qdotn64) * W2 + 0.5 * QB264;
        const double f2 = (vd * BW * BW - Qtsq64) * W2 - QB264 * (Bsq64 + 2.0 * Wd);
        // in the FP32 stage's scaled form: k f1 / W^2 = k^3 f1 / w^2, k^2 f2 / W^2 = k^4 f2 / w^2
        const float iw = 1.0f / w, iw2 = iw * iw;
        const float r1 = narrow(f1 * k3) * iw2, r2 = narrow(f2 * k4) * iw2;
        // the FP32 Jacobian at the root
        const float om = 1.0f - v;
        const float rs = rsqrtf(om);
        const float bw = Bsq + w;
        const float j11 = -QB2 * iw2 * iw - 1.0f + gf * om;
        const float j12 = -0.5f * Bsq + gf * (0.5f * D * rs - w);
        const float j21 = 2.0f * bw * (v + QB2 * iw2 * iw);
        const float j22 = bw * bw;
        const float det = j11 * j22 - j12 * j21;
        const float idet = 1.0f / det;
        const float dw = (j12 * r2 - j22 * r1) * idet, dv = (j21 * r1 - j11 * r2) * idet;
        const float step = fabsf(dw) + fabsf(dv) * w;
        const float cancel = (fabsf(j11 * j22) + fabsf(j12 * j21)) * fabsf(idet);
        const double Wn = Wd + widen(dw) * ik;
        const double vn = clamp_pos(vd + widen(dv), C2P_VSQMAX);
        const bool in = is_pos(Wn);
        if (in && step < 1e-5f * w && step * cancel < 1e-3f * w) {
            it = it32 + 1;
            W = Wn;
            vsq = vn;
            return true;
        }
        if (in) {
            Wd = Wn;
            vd = vn;
        }
    }
    const C2PScalars T = S;
    const NewtonOut o = newton_wv_call(&T, gfac, Wd, vd);
    it = it32 + 1 + o.it;
    W = o.W;
    vsq = o.vsq;
    return o.ok;
}

// Aitken-accelerated inversion (Sec. 2.6 names it beside Newton; Newman &
// Hamlin 2014). With E = -Q.n, S^2 = Qt^2, T = Q.B the two equations give, for
// a trial pressure p, a cubic in phi = W + B^2: phi^3 - a phi^2 + d = 0,
// a = E + p + B^2/2, d = (S^2 B^2 - T^2)/2. Its largest root (closed form
// (a/3)(1 + 2 cos(acos(1 - 27 d / (2 a^3)) / 3))), v^2 from the momentum
// equation and the ideal-gas pressure of (W, v^2) map p to the next p.
// Returns false when W <= 0 or the pressure is not finite.
__device__ __forceinline__ bool nh_map(const C2PScalars& S, double gfac, double p, double& W, double& vsq,
                                       double& pn) {
    const double B2 = S.Bsq;
    const double a = -S.Qdotn + p + 0.5 * B2;
    const double d = fmax(0.5 * (S.Qtsq * B2 - S.QB2), 0.0);
    if (!(a > 0.0)) return false;
    const double x = fmin(fmax(1.0 - 27.0 * d / (2.0 * a * a * a), -1.0), 1.0);
    const double phi = a / 3.0 * (1.0 + 2.0 * cos(acos(x) / 3.0));
    const double w = phi - B2;
    if (!(w > 0.0)) return false;
    const double v = fmin(fmax((S.Qtsq * w * w + S.QB2 * (2.0 * w + B2)) / (w * w * phi * phi), 0.0), C2P_VSQMAX);
    W = w;
    vsq = v;
    pn = gfac * (w * (1.0 - v) - S.D * sqrt(1.0 - v));
    return isfinite(pn);
}

// Steffensen's form of the Aitken delta-squared acceleration of p -> map(p):
// two evaluations from p0 give p1, p2, and the next cycle starts from
// p0 - (p1 - p0)^2 / (p2 - 2 p1 + p0) (from p2 when that is not a valid
// pressure). Pressures stay >= max(0, (27 d / 4)^(1/3) - E - B^2/2), where
// the cubic has its root. An extrapolation step below C2P_TOL W ends the
// iteration, and one more evaluation gives (W, v^2). `it` counts evaluations.
__device__ __forceinline__ bool aitken_wv(const C2PScalars& S, double gfac, double p, double& W, double& vsq,
                                          int& it) {
    const double d = fmax(0.5 * (S.Qtsq * S.Bsq - S.QB2), 0.0);
    const double pmin = fmax(cbrt(6.75 * d) + S.Qdotn - 0.5 * S.Bsq, 0.0);
    if (!(p >= pmin)) p = pmin;
    it = 0;
    for (int cycle = 1; cycle <= C2P_NMAX; cycle++) {
        double W1, v1, p1, W2, v2, p2;
        it++;
        if (!nh_map(S, gfac, p, W1, v1, p1)) return false;
        p1 = fmax(p1, pmin);
        it++;
        if (!nh_map(S, gfac, p1, W2, v2, p2)) return false;
        p2 = fmax(p2, pmin);
        const double den = p2 - 2.0 * p1 + p;
        double pa = p2;
        if (den != 0.0) {
            const double e = p - (p1 - p) * (p1 - p) / den;
            if (e >= pmin && isfinite(e)) pa = e;
        }
        const double step = fabs(pa - p);
        p = pa;
        if (step < C2P_TOL * W2) {
            it++;
            double pn;
            return nh_map(S, gfac, p, W, vsq, pn);
        }
    }
    return false;
}

// rho and u_g of a converged (W, v^2) (u_g = p / (gam - 1) = (W (1 - v^2) - D sqrt(1 - v^2)) / gam);
// false unless both are positive. rs: 1/sqrt(1 - v^2), the Lorentz factor, for the velocity (in: the
// same where the caller has it, else 0).
__device__ __forceinline__ bool energy_result(const C2PScalars& S, double igam, double W, double vsq, double& rho,
                                              double& u, double& rs) {
    const double omv = 1.0 - vsq;
    if (__double2hiint(rs) == 0) rs = rsqrt(omv);
    const double sq = omv * rs;
    rho = S.D * sq;
    u = (W * omv - S.D * sq) * igam;
    return is_pos(rho) && is_pos(u);
}

// The inversion in three pieces (invert() below composes them):
// c2p_prepare (scalars and the start from the guess primitives), any number of
// energy-equation attempts from given starts, c2p_finish (entropy backup when
// no attempt succeeded, then the primitives).
struct C2PWork {
    C2PScalars S;
    double W0, vsq0;  // the start from the guess primitives
    double p0;        // ... and its pressure (the Aitken inversion's start)
    int method;       // HAMR_INV_NEWTON or HAMR_INV_AITKEN
    int form;         // Newton: C2P_NEWTON_FF, _32, _64 or _ANY
    double igam, gfac;  // 1/gam and (gam - 1)/gam, from one division per inversion
    double W, vsq, rho, u;
    double rs;        // 1/sqrt(1 - v^2) of an energy result
    bool ok;
    int its;          // Newton iterations of every energy attempt
};

// start32 (mixed form, optional): the start (W, v^2) already formed in FP32 from the guess primitives;
// igam, gfac (optional, > 0): 1/gam and (gam - 1)/gam formed once by the caller (else here, per state);
// start64 (optional): Gamma^2 and Gamma^2 v^2 of the guess primitives where the caller has them
__device__ __forceinline__ void c2p_prepare(const double U[NCONS], const double Bc[3], const Metric<double>& m,
                                            double gam, const double pr[NPRIM], C2PWork& w,
                                            int method = HAMR_INV_NEWTON, int form = C2P_NEWTON_FF,
                                            const float* start32 = nullptr, double igam = 0.0, double gfac = 0.0,
                                            const double* start64 = nullptr) {
    c2p_scalars(U, Bc, m, w.S);
    if (igam > 0.0) {
        w.igam = igam;
        w.gfac = gfac;
    } else {
        w.igam = 1.0 / gam;
        w.gfac = (gam - 1.0) * w.igam;
    }
    w.method = method;
    w.form = form;
    w.p0 = (method == HAMR_INV_AITKEN) ? (gam - 1.0) * pr[UU] : 0.0;
    if (form == C2P_NEWTON32 && start32) {
        w.W0 = widen(start32[0]);
        w.vsq0 = widen(fminf(start32[1], (float)C2P_VSQMAX));
    } else if (form == C2P_NEWTON32) {
        // the start only seeds the FP32 iterations (and, where they fail, the FP64 ones): in FP32
        const float q1 = narrow(pr[U1]), q2 = narrow(pr[U2]), q3 = narrow(pr[U3]);
        const float qsq = narrow(m.g11) * q1 * q1 + narrow(m.g22) * q2 * q2 + narrow(m.g33) * q3 * q3 +
                          2.0f * narrow(m.g13) * q1 * q3;
        const float gsq = 1.0f + qsq;
        w.W0 = widen((narrow(pr[RHO]) + narrow(gam) * narrow(pr[UU])) * gsq);
        w.vsq0 = widen(fminf(qsq / gsq, (float)C2P_VSQMAX));
    } else if (start64) {
        w.W0 = (pr[RHO] + gam * pr[UU]) * start64[0];
        w.vsq0 = fmin(start64[1] * (1.0 / start64[0]), C2P_VSQMAX);
    } else {
        const double q1 = pr[U1], q2 = pr[U2], q3 = pr[U3];
        const double qsq = m.g11 * q1 * q1 + m.g22 * q2 * q2 + m.g33 * q3 * q3 + 2.0 * m.g13 * q1 * q3;
        const double gsq = 1.0 + qsq;
        w.W0 = (pr[RHO] + gam * pr[UU]) * gsq;
        w.vsq0 = fmin(qsq * (1.0 / gsq), C2P_VSQMAX);
    }
    w.W = w.W0;
    w.vsq = 0.0;
    w.rho = w.u = w.rs = 0.0;
    w.ok = false;
    w.its = 0;
}

// one energy-equation attempt from the pressure p (Aitken inversion)
__device__ __forceinline__ void c2p_attempt_p(C2PWork& w, double gam, double p) {
    if (w.ok) return;
    (void)gam;
    int it = 0;
    double W = 0.0, vsq = 0.0;
    bool ok = aitken_wv(w.S, w.gfac, p, W, vsq, it);
    w.its += it;
    if (ok) {
        w.W = W;
        w.vsq = vsq;
        w.rs = 0.0;
        ok = energy_result(w.S, w.igam, W, vsq, w.rho, w.u, w.rs);
    }
    w.ok = ok;
}

// one energy-equation attempt from (W, v^2); no-op once an attempt succeeded.
// The Aitken inversion starts from the pressure of (W, v^2).
__device__ __forceinline__ void c2p_attempt(C2PWork& w, double gam, double W, double vsq) {
    if (w.ok || !is_pos(W)) return;
    const double gfac = w.gfac;
    vsq = clamp_pos(vsq, C2P_VSQMAX);
    if (w.method == HAMR_INV_AITKEN) {
        c2p_attempt_p(w, gam, gfac * (W * (1.0 - vsq) - w.S.D * sqrt(1.0 - vsq)));
        return;
    }
    int it = 0;
    w.rs = 0.0;
    bool ok = (w.form == C2P_NEWTON32)   ? newton_wv_mixed(w.S, gfac, W, vsq, it)
              : (w.form == C2P_NEWTON64) ? newton_wv(w.S, gfac, W, vsq, it)
                                         : newton_wv_ff(w.S, gfac, W, vsq, it, w.rs, w.form == C2P_NEWTON_ANY);
    w.its += it;
    w.W = W;
    w.vsq = vsq;
    if (ok) ok = energy_result(w.S, w.igam, W, vsq, w.rho, w.u, w.rs);
    w.ok = ok;
}

// the attempt from the guess primitives: (W, v^2) for Newton, their pressure for Aitken
__device__ __forceinline__ void c2p_attempt_plain(C2PWork& w, double gam) {
    if (w.method == HAMR_INV_AITKEN)
        c2p_attempt_p(w, gam, w.p0);
    else
        c2p_attempt(w, gam, w.W0, w.vsq0);
}

// The entropy backup: Newton in W on f = W (1 - v^2) - rho - gam p / (gam - 1), p = kappa rho^gam,
// v^2(W) from the momentum equation, rho = D sqrt(1 - v^2).
struct EntropyOut {
    double W, vsq, rho, u;
    bool ok;
};

__device__ __forceinline__ bool entropy_newton(const C2PScalars& S, double kappa, double gam, double& W) {
    const double gr = gam / (gam - 1.0);
    for (int k = 1; k <= C2P_NMAX; k++) {
        const double W2 = W * W;
        const double BW = S.Bsq + W;
        const double num = S.Qtsq * W2 + S.QB2 * (S.Bsq + 2.0 * W);
        const double den = W2 * BW * BW;
        const double iden = 1.0 / den;
        double vs = num * iden;
        double dvs = (2.0 * (S.Qtsq * W + S.QB2) - num * 2.0 * W * BW * (S.Bsq + 2.0 * W) * iden) * iden;
        if (vs > C2P_VSQMAX) {
            vs = C2P_VSQMAX;
            dvs = 0.0;
        }
        const double s1 = 1.0 - vs;
        const double sq = sqrt(s1);
        const double rh = S.D * sq;
        const double p = kappa * pow(rh, gam);
        const double f = W * s1 - rh - gr * p;
        const double drh = -0.5 * S.D / sq * dvs;
        const double df = s1 - W * dvs - drh * (1.0 + gr * gam * p / rh);
        const double Wn = W - f / df;
        if (!(Wn > 0.0)) return false;
        const double err = fabs(Wn - W);
        W = Wn;
        if (err < C2P_TOL * Wn) return true;
    }
    return false;
}

// v^2 and rho at W; with the base point's rho and rho^gam (r0, pw0) also rho^gam, by the binomial series
// in x = rho / r0 - 1 (|x| < 1e-3: the terms to x^4 leave 1e-15 x^... < 1e-16), which a pow would cost
// five times
__device__ __forceinline__ void entropy_point(const C2PScalars& S, double gam, double W, double r0, double pw0,
                                              double& vsq, double& rh, double& pw, double& x) {
    const double W2 = W * W, BW = S.Bsq + W;
    vsq = fmin((S.Qtsq * W2 + S.QB2 * (BW + W)) / (W2 * BW * BW), C2P_VSQMAX);
    rh = S.D * sqrt(1.0 - vsq);
    x = 0.0;
    if (r0 > 0.0) {
        x = (rh - r0) / r0;
        const double g1 = gam - 1.0, g2 = gam - 2.0, g3 = gam - 3.0;
        pw = pw0 * fma(gam * x, fma(0.5 * g1 * x, fma(g2 * x * (1.0 / 3.0), fma(0.25 * g3, x, 1.0), 1.0), 1.0), 1.0);
    } else {
        pw = pow(rh, gam);
    }
}

// The iterations run in FP32 first (scaled by the power of two of the start's W; p through base-2
// logarithms), until a step is below 1e-5 W; two FP64 residuals with the FP32 slope then take the root from
// there to the stopping rule, one power and its series for both and the result. Where the FP32 iteration
// meets no root, or the second FP64 step is not below the rule, the FP64 iteration runs from the start.
// Few cells come here (0.2% of a large torus, 4% of a small one), but their warps wait for this chain:
// five or six FP64 iterations of ~145 FP64 instructions each before. On a 64x32x16 block the cell update,
// which such warps end, takes 49 us a launch, 98 with FP64 iterations alone (newton_wv's too). fast = false:
// the FP64 iteration alone, in the mixed forms, whose results stay bit for bit (update.cu), and in the
// standalone inversion, where many states of a warp may have no entropy root either (1M inversions by
// entropy alone, 10% of them failing: 9.41 ms, 9.96 with the FP32 start).
static __device__ __noinline__ EntropyOut entropy_backup(const C2PScalars* Sp, double kappa, double gam, double W0,
                                                         bool fast) {
    const C2PScalars& S = *Sp;
    EntropyOut o;
    o.ok = false;
    const unsigned eW = (unsigned)__double2hiint(W0) & 0xfff00000u;
    if (fast && eW - 0x2b000000u < 0x2a000000u && kappa > 0.0) {
        const unsigned sh = 0x3ff00000u - eW;
        const float D = ff_of(S.D, (int)sh).h, B2 = ff_of(S.Bsq, (int)sh).h;
        const float Qt = ff_of(S.Qtsq, (int)(2u * sh)).h, QB = ff_of(S.QB2, (int)(3u * sh)).h;
        const float gf = (float)gam, gr = gf / (gf - 1.0f);
        const float e = (float)((int)(eW >> 20) - 1023);
        // log2 p = log2 kappa + gam (log2 rho_scaled + e) - e
        const int ke = (__double2hiint(kappa) >> 20) - 1023;
        const float km = __uint_as_float(0x3f800000u | (((unsigned)__double2hiint(kappa) & 0xfffffu) << 3));
        const float lk = (float)ke + log2f(km) + (gf - 1.0f) * e;
        float w = ff_of(W0, (int)sh).h, df = 0.0f;
        bool ok32 = false;
        for (int k = 0; k < C2P_NMAX && !ok32; k++) {
            const float bw = B2 + w, den = w * w * bw * bw, iden = 1.0f / den;
            const float num = Qt * w * w + QB * (B2 + 2.0f * w);
            float vs = num * iden;
            float dvs = (2.0f * (Qt * w + QB) - num * 2.0f * w * bw * (B2 + 2.0f * w) * iden) * iden;
            if (vs > (float)C2P_VSQMAX) {
                vs = (float)C2P_VSQMAX;
                dvs = 0.0f;
            }
            const float s1 = 1.0f - vs, sq = sqrtf(s1), rh = D * sq;
            const float p = exp2f(lk + gf * log2f(rh));
            const float f = w * s1 - rh - gr * p;
            df = s1 - w * dvs + 0.5f * D / sq * dvs * (1.0f + gr * gf * p / rh);
            const float wn = w - f / df;
            if (!(wn > 0.02f * w && wn < 1e9f)) break;  // near wn = 0 rounding decides whether FP64 fails
            ok32 = k < 12 && fabsf(wn - w) < 1e-5f * wn;
            w = wn;
        }
        if (ok32 && fabsf(df) > 1e-6f) {
            const double gr64 = gam / (gam - 1.0);
            double W = widen(w);
            W = __hiloint2double((int)((unsigned)__double2hiint(W) - sh), __double2loint(W));
            const double idf = 1.0 / widen(df);
            double vs, rh, pw, x, r0, pw0;
            entropy_point(S, gam, W, 0.0, 0.0, vs, r0, pw0, x);
            const double d1 = (W * (1.0 - vs) - r0 - gr64 * kappa * pw0) * idf;
            W -= d1;
            entropy_point(S, gam, W, r0, pw0, vs, rh, pw, x);
            const double d2 = (W * (1.0 - vs) - rh - gr64 * kappa * pw) * idf;
            W -= d2;
            // the rule on the second step, and both small enough for the slope's error (the contraction
            // d2 / d1) to leave the third below round-off
            if (W > 0.0 && fabs(d1) < 1e-4 * W && fabs(d2) < C2P_TOL * W && d2 * d2 <= 1e-16 * fabs(d1) * W) {
                entropy_point(S, gam, W, r0, pw0, o.vsq, o.rho, pw, x);
                if (fabs(x) < 1e-3) {
                    o.W = W;
                    o.u = kappa * pw / (gam - 1.0);
                    o.ok = (o.rho > 0.0) && (o.u > 0.0) && (o.vsq >= 0.0);
                    return o;
                }
            }
        }
    }
    double W = W0;
    if (entropy_newton(S, kappa, gam, W)) {
        const double W2 = W * W;
        const double BW = S.Bsq + W;
        o.W = W;
        o.vsq = fmin((S.Qtsq * W2 + S.QB2 * (S.Bsq + 2.0 * W)) / (W2 * BW * BW), C2P_VSQMAX);
        o.rho = S.D * sqrt(1.0 - o.vsq);
        o.u = kappa * pow(o.rho, gam) / (gam - 1.0);
        o.ok = (o.rho > 0.0) && (o.u > 0.0) && (o.vsq >= 0.0);
    }
    return o;
}

// pr: out the result (slots 0..4) unless INV_FAIL (then untouched)
__device__ __forceinline__ int c2p_finish(C2PWork& w, const double U[NCONS], const Metric<double>& m, double gam,
                                          double pr[NPRIM]) {
    const C2PScalars& S = w.S;
    const double Bsq = S.Bsq;
    double W = w.W, vsq = w.vsq, rho = w.rho, u = w.u;
    int status = INV_OK;
    if (!w.ok) {
        const C2PScalars T = S;
        const EntropyOut o = entropy_backup(&T, U[C_ENT] / U[C_RHO], gam, w.W0, w.form == C2P_NEWTON_FF);
        if (!o.ok) return INV_FAIL;
        W = o.W;
        vsq = o.vsq;
        rho = o.rho;
        u = o.u;
        status = INV_ENTROPY;
    }
    // utilde^i = Gamma/(W + B^2) (Qt^i + (Q.B) Bn^i / W), Qt^i = Q^i - alpha g^{ti} (Q.n);
    // 1/(W + B^2) and 1/W from one reciprocal of W (W + B^2)
    const double gamma = (status == INV_OK) ? w.rs : rsqrt(1.0 - vsq);
    const double WB = W + Bsq;
    const double r = 1.0 / (W * WB);
    const double pre = gamma * W * r;
    const double qbw = S.QdotB * WB * r;
    pr[U1] = pre * (S.Qc1 - m.alpha * m.c01 * S.Qdotn + qbw * S.Bn1);
    pr[U2] = pre * (S.Qc2 + qbw * S.Bn2);
    pr[U3] = pre * (S.Qc3 + qbw * S.Bn3);
    pr[RHO] = rho;
    pr[UU] = u;
    w.W = W;
    w.vsq = vsq;
    return status;
}

// pr: in the guess (slots 0..4), out the result (slots 0..4) unless INV_FAIL.
// guess2 (optional): a first start (W, v^2) tried before the one of pr; the
// start from pr is then the fallback. `iters` counts the energy-inversion
// Newton iterations of every start tried.
__device__ __forceinline__ int invert(const double U[NCONS], const double Bc[3], const Metric<double>& m, double gam,
                                      double pr[NPRIM], int* iters, bool entropy_only,
                                      const double* guess2 = nullptr, int method = HAMR_INV_NEWTON,
                                      int form = C2P_NEWTON_FF) {
    C2PWork w;
    c2p_prepare(U, Bc, m, gam, pr, w, method, form);
    if (!entropy_only) {
        if (guess2) c2p_attempt(w, gam, guess2[0], guess2[1]);
        c2p_attempt_plain(w, gam);
    }
    if (iters) *iters = w.its;
    return c2p_finish(w, U, m, gam, pr);
}

}  // namespace hamr
