// c2p.cu -- the standalone inversion entry point (Sec. 2.6): one thread per
// state, the metric evaluated analytically at each state's position.
#include "c2p.cuh"
#include "hamr_internal.h"
#include "metric.cuh"
#include "mlp.cuh"

namespace hamr {
namespace {

// FORM: how Newton iterates without HAMR_C2P_MIXED (C2P_NEWTON_ANY or C2P_NEWTON64, launch_con2prim)
template <bool MLP, int FORM>
__global__ void __launch_bounds__(128) k_con2prim(hamr_c2p_desc d, const uint8_t* __restrict__ img, int* err,
                                                  int64_t n, const double* __restrict__ U,
                                                  const double* __restrict__ B, const double* __restrict__ x1,
                                                  const double* __restrict__ x2, double* __restrict__ prim,
                                                  int32_t* __restrict__ status, int32_t* __restrict__ iters) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = s < n;
    if (!MLP && !active) return;
    Metric<double> m;
    double u[NCONS], bc[3], pr[NPRIM];
    if (active) {
        FullMetric M;
        metric_at(d.metric, d.a, x1[s], x2[s], M);
        to_sparse(M, m);
#pragma unroll
        for (int q = 0; q < NCONS; q++) u[q] = U[q * n + s];
#pragma unroll
        for (int q = 0; q < 3; q++) bc[q] = B[q * n + s];
#pragma unroll
        for (int q = 0; q < NPRIM; q++) pr[q] = prim[q * n + s];
        pr[B1] = bc[0];
        pr[B2] = bc[1];
        pr[B3] = bc[2];
    }
    const bool entropy_only = (d.flags & HAMR_C2P_ENTROPY_ONLY) != 0;
    const bool rescue = (d.flags & HAMR_C2P_MLP_RESCUE) != 0;
    C2PWork w;
    if (active)
        c2p_prepare(u, bc, m, d.gam, pr, w, (d.flags & HAMR_C2P_AITKEN) ? HAMR_INV_AITKEN : HAMR_INV_NEWTON,
                    (d.flags & HAMR_C2P_MIXED) ? C2P_NEWTON32 : FORM);
    if (MLP && !entropy_only) {  // the 128 states of the CTA through the network (mlp.cuh)
        if (rescue && active) c2p_attempt_plain(w, d.gam);
        if (__syncthreads_or(active && !w.ok)) {
            extern __shared__ __align__(16) uint8_t mlp_smem[];
            MlpCta C;
            mlp_begin(C, mlp_smem, img);
            float f[MLP_NIN], y[MLP_NOUT];
            if (active) mlp_features(w.S, u[C_RHO], u[C_ENT], m, x1[s], d.gam, f);
            const bool ran = mlp_infer(C, f, active, y);
            mlp_end(C);
            if (!C.ok && threadIdx.x == 0 && err) atomicExch(err, 1);
            if (active && ran && !w.ok) {
                double g2[2];
                mlp_guess(w.S.D, y, g2);
                c2p_attempt(w, d.gam, g2[0], g2[1]);
            }
        }
    }
    if (active && !entropy_only && !(MLP && rescue)) c2p_attempt_plain(w, d.gam);
    __syncwarp();  // the lanes come out of the attempt by several ways: together again for the backup
    if (!active) return;
    const int st = c2p_finish(w, u, m, d.gam, pr);
    const int it = w.its;
#pragma unroll
    for (int q = 0; q < NPRIM; q++) prim[q * n + s] = pr[q];
    status[s] = st;
    if (iters) iters[s] = it;
}

}  // namespace

cudaError_t launch_con2prim(const hamr_c2p_desc& d, int64_t n, const double* U, const double* B, const double* x1,
                            const double* x2, double* prim, int32_t* status, int32_t* iters, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int bs = 128;
    const unsigned nb = (unsigned)((n + bs - 1) / bs);
    // Up to one warp per scheduler (a CTA per SM) the call waits for one warp's chain of dependent instructions,
    // which is shorter in FP64: 24.3 us for 1024 to 16384 states 5% off, 26.5 to 27 in double-float. Beyond, the
    // FP64 pipe is shared: 42.5 against 37.5 us at 32768 states, 81 against 63 at 65536.
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const bool chain = (int64_t)nb <= sms;
    if ((d.flags & (HAMR_C2P_MLP | HAMR_C2P_MLP_RESCUE)) && d.mlp)
        (chain ? k_con2prim<true, C2P_NEWTON64> : k_con2prim<true, C2P_NEWTON_ANY>)<<<nb, bs, MLP_SMEM_BYTES, s>>>(
            d, mlp_image(d.mlp), mlp_error_ptr(d.mlp), n, U, B, x1, x2, prim, status, iters);
    else
        (chain ? k_con2prim<false, C2P_NEWTON64> : k_con2prim<false, C2P_NEWTON_ANY>)<<<nb, bs, 0, s>>>(
            d, nullptr, nullptr, n, U, B, x1, x2, prim, status, iters);
    return cudaGetLastError();
}

}  // namespace hamr
