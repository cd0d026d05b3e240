// mlp.cu -- the learned starting point of the inversion: model state,
// primitive -> conserved for training pairs, the ten inputs and two
// targets, standardisation, training (forward and backward on the CUDA cores
// in FP32, Adam), the bf16 inference image and the standalone inference.
// The paper has no counterpart (its Newton starts from the previous
// primitives, Sec. 2.6); the network only moves Newton's starting point.
#include <cmath>
#include <cstring>
#include <vector>

#include "hamr_internal.h"
#include "metric.cuh"
#include "mlp.cuh"

namespace hamr {
namespace {

constexpr int TB = 128;   // batches are multiples of this
constexpr int TSMP = 64;  // samples per CTA of the training kernel
constexpr int TTHR = 256; // its threads
constexpr int HS = 68;    // row stride of its 64-wide arrays: 16-byte aligned rows, 16 bytes apart modulo the banks
constexpr int XS = 12;    // row stride of its 10-wide arrays (two zeros)
// shared memory of k_mlp_fb (floats): W2, W3, three hidden layers, W1, inputs, biases and W4, output errors,
// four warps' sums of squares
constexpr int FB_W2 = 0, FB_W3 = 64 * HS, FB_H1 = 2 * 64 * HS, FB_H2 = FB_H1 + TSMP * HS, FB_H3 = FB_H2 + TSMP * HS,
              FB_W1 = FB_H3 + TSMP * HS, FB_X = FB_W1 + 64 * XS, FB_B = FB_X + TSMP * XS, FB_W4 = FB_B + 192,
              FB_B4 = FB_W4 + 128, FB_DY = FB_B4 + 4, FB_R2 = FB_DY + TSMP * 2, FB_N = FB_R2 + 4;
constexpr int FB_SMEM = FB_N * 4;

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {  // Steele, Lea & Flood (2014)
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

__device__ __forceinline__ void metric_sparse(const hamr_c2p_desc& d, double x1, double x2, Metric<double>& m) {
    FullMetric M;
    metric_at(d.metric, d.a, x1, x2, M);
    to_sparse(M, m);
}

// ---------------------------------------------------------------- data
__global__ void k_prim2cons(hamr_c2p_desc d, int64_t n, const double* __restrict__ prim,
                            const double* __restrict__ x1, const double* __restrict__ x2, double* __restrict__ U) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    Metric<double> m;
    metric_sparse(d, x1[s], x2[s], m);
    double pr[NPRIM];
#pragma unroll
    for (int q = 0; q < NPRIM; q++) pr[q] = prim[q * n + s];
    Fluid<double> st;
    fluid_state(pr, m, st);
    double row[NFLUX];
    flux_row(pr, st, 0, 1, d.gam, entropy_kappa(pr, d.gam), row);
#pragma unroll
    for (int q = 0; q < NCONS; q++) U[q * n + s] = row[q] * m.gdet;
}

__global__ void k_features(hamr_c2p_desc d, int64_t n, const double* __restrict__ U, const double* __restrict__ B,
                           const double* __restrict__ x1, const double* __restrict__ x2,
                           const double* __restrict__ prim, float* __restrict__ feat, float* __restrict__ targ) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    Metric<double> m;
    metric_sparse(d, x1[s], x2[s], m);
    double u[NCONS], bc[3];
#pragma unroll
    for (int q = 0; q < NCONS; q++) u[q] = U[q * n + s];
#pragma unroll
    for (int q = 0; q < 3; q++) bc[q] = B[q * n + s];
    C2PScalars S;
    c2p_scalars(u, bc, m, S);
    float f[MLP_NIN];
    mlp_features(S, u[C_RHO], u[C_ENT], m, x1[s], d.gam, f);
#pragma unroll
    for (int q = 0; q < MLP_NIN; q++) feat[q * n + s] = f[q];
    if (prim && targ) {
        const double q1 = prim[U1 * n + s], q2 = prim[U2 * n + s], q3 = prim[U3 * n + s];
        const double qsq = m.g11 * q1 * q1 + m.g22 * q2 * q2 + m.g33 * q3 * q3 + 2.0 * m.g13 * q1 * q3;
        const double h = 1.0 + d.gam * prim[UU * n + s] / prim[RHO * n + s];
        targ[s] = (float)log(h * sqrt(1.0 + qsq));
        targ[n + s] = (float)log1p(qsq);
    }
}

// sums and sums of squares of the 12 columns (inputs, targets), FP64
__global__ void k_norm_sums(int64_t n, const float* __restrict__ feat, const float* __restrict__ targ,
                            double* __restrict__ sums) {
    __shared__ double red[24][4];
    double acc[24];
#pragma unroll
    for (int q = 0; q < 24; q++) acc[q] = 0.0;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int q = 0; q < 12; q++) {
            const double v = (q < MLP_NIN) ? feat[q * n + s] : targ[(q - MLP_NIN) * n + s];
            acc[q] += v;
            acc[12 + q] += v * v;
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 24; q++) {
        double v = acc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[q][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < 24) {
        double v = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); k++) v += red[threadIdx.x][k];
        atomicAdd(&sums[threadIdx.x], v);
    }
}

// ---------------------------------------------------------------- inference image
__global__ void k_pack(const float* __restrict__ P, const float* __restrict__ norm, uint8_t* __restrict__ img) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    // bf16 operands: W1 padded to 64 x 16, W2 and W3 64 x 64 (row = output unit n, column = input k)
    if (t < 64 * 16) {
        const int r = t / 16, k = t % 16;
        const float w = (k < MLP_NIN) ? P[P_W1 + r * MLP_NIN + k] : 0.0f;
        *reinterpret_cast<__nv_bfloat16*>(img + IMG_W1 + core_off(r, k, 16)) = __float2bfloat16_rn(w);
    } else if (t < 64 * 16 + 2 * 4096) {
        const int u = t - 64 * 16;
        const int which = u / 4096, e = u % 4096, r = e / 64, k = e % 64;
        const float w = P[(which ? P_W3 : P_W2) + r * 64 + k];
        *reinterpret_cast<__nv_bfloat16*>(img + (which ? IMG_W3 : IMG_W2) + core_off(r, k, 64)) =
            __float2bfloat16_rn(w);
    } else if (t < 64 * 16 + 2 * 4096 + IMGF_N) {
        const int q = t - 64 * 16 - 2 * 4096;
        float v = 0.0f;
        if (q < IMGF_W4) v = P[(q < 64 ? P_B1 : (q < 128 ? P_B2 : P_B3)) + (q & 63)];
        else if (q < IMGF_B4) v = __bfloat162float(__float2bfloat16_rn(P[P_W4 + q - IMGF_W4]));
        else if (q < IMGF_B4 + 2) v = P[P_B4 + q - IMGF_B4];
        else if (q < IMGF_FM) v = 0.0f;
        else if (q < IMGF_FI) v = norm[q - IMGF_FM];
        else if (q < IMGF_YM) v = 1.0f / norm[10 + q - IMGF_FI];
        else if (q < IMGF_YS) v = norm[20 + q - IMGF_YM];
        else v = norm[22 + q - IMGF_YS];
        reinterpret_cast<float*>(img + IMG_F)[q] = v;
    }
}
constexpr int PACK_THREADS = 64 * 16 + 2 * 4096 + IMGF_N;

// ---------------------------------------------------------------- training (FP32)
// 64 x 64 products of a CTA's 64 samples, 256 threads with 4 x 4 results each in registers (tx = t & 15,
// ty = t >> 4); operands in shared memory, read 16 bytes at a time without bank conflicts.

// acc[r][q] += sum_i A[(ty + 16 r)][i] W[(tx + 16 q)][i], i < K (a multiple of 4)
template <int K, int LD>
__device__ __forceinline__ void mm_nt(const float* A, const float* W, int tx, int ty, float acc[4][4]) {
#pragma unroll 4
    for (int i = 0; i < K; i += 4) {
        float4 a[4], w[4];
#pragma unroll
        for (int r = 0; r < 4; r++) a[r] = *reinterpret_cast<const float4*>(A + (ty + 16 * r) * LD + i);
#pragma unroll
        for (int q = 0; q < 4; q++) w[q] = *reinterpret_cast<const float4*>(W + (tx + 16 * q) * LD + i);
#pragma unroll
        for (int r = 0; r < 4; r++)
#pragma unroll
            for (int q = 0; q < 4; q++) {
                acc[r][q] = fmaf(a[r].x, w[q].x, acc[r][q]);
                acc[r][q] = fmaf(a[r].y, w[q].y, acc[r][q]);
                acc[r][q] = fmaf(a[r].z, w[q].z, acc[r][q]);
                acc[r][q] = fmaf(a[r].w, w[q].w, acc[r][q]);
            }
    }
}

// one hidden layer: out[s][o] = tanh(b[o] + sum_i in[s][i] W[o][i])
template <int K, int LD>
__device__ __forceinline__ void mlp_layer(const float* in, const float* W, const float* b, float* out, int tx, int ty) {
    float acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[r][q] = b[tx + 16 * q];
    mm_nt<K, LD>(in, W, tx, ty, acc);
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
        for (int q = 0; q < 4; q++) out[(ty + 16 * r) * HS + tx + 16 * q] = tanhf(acc[r][q]);
}

// One CTA: TSMP samples, forward and backward; the parameter gradient of
// loss = sum over samples and outputs of r^2 / (2 count), r = yn - tn, is
// accumulated into grad; sum r^2 into loss[0].
// mode 0: samples off + 0.., mode 1: sample ids splitmix64(seed ^ (step * batch + b)) mod n.
// ~26000 FMAs per sample, latency-bound: a batch of 8192 took 104 us with one thread per sample (two shared
// loads per FMA, 64 CTAs of 4 warps), 24 us with register tiles (128 CTAs of 8 warps).
__global__ void __launch_bounds__(TTHR) k_mlp_fb(const float* __restrict__ Pg, const float* __restrict__ norm,
                                                 const float* __restrict__ feat, const float* __restrict__ targ,
                                                 int64_t n, int mode, int64_t off, int64_t count, uint64_t seed,
                                                 int64_t step, float* __restrict__ grad, float* __restrict__ loss) {
    extern __shared__ __align__(16) float fsm[];
    float *W2 = fsm + FB_W2, *W3 = fsm + FB_W3, *H1 = fsm + FB_H1, *H2 = fsm + FB_H2, *H3 = fsm + FB_H3;
    float *W1 = fsm + FB_W1, *X = fsm + FB_X, *Bs = fsm + FB_B, *W4 = fsm + FB_W4, *B4 = fsm + FB_B4, *DY = fsm + FB_DY, *R2 = fsm + FB_R2;
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    auto sample = [&](int s, int64_t& g) {  // whether sample s of the CTA counts, and its row
        const int64_t b = (int64_t)blockIdx.x * TSMP + s;
        if (mode == 0) {
            g = off + b;
            return (b < count) && (g < n);
        }
        g = (int64_t)(splitmix64(seed ^ (uint64_t)(step * count + b)) % (uint64_t)n);
        return b < count;
    };
#pragma unroll
    for (int q = 0; q < 4; q++) {  // 1024 float4 of W2 and of W3
        const int e = t + TTHR * q, o = e >> 4, i = (e & 15) * 4;
        *reinterpret_cast<float4*>(W2 + o * HS + i) = *reinterpret_cast<const float4*>(Pg + P_W2 + o * 64 + i);
        *reinterpret_cast<float4*>(W3 + o * HS + i) = *reinterpret_cast<const float4*>(Pg + P_W3 + o * 64 + i);
    }
    for (int e = t; e < 64 * XS; e += TTHR) {
        const int o = e / XS, i = e % XS;
        W1[e] = i < MLP_NIN ? Pg[P_W1 + o * MLP_NIN + i] : 0.0f;
    }
    if (t < 64) {
        Bs[t] = Pg[P_B1 + t];
        Bs[64 + t] = Pg[P_B2 + t];
        Bs[128 + t] = Pg[P_B3 + t];
    } else if (t < 192) {
        W4[t - 64] = Pg[P_W4 + t - 64];
    } else if (t < 194) {
        B4[t - 192] = Pg[P_B4 + t - 192];
    }
    {
        const int s = t & 63;
        int64_t g;
        const bool on = sample(s, g);
        for (int i = t >> 6; i < XS; i += 4)
            X[s * XS + i] = (on && i < MLP_NIN) ? (feat[i * n + g] - norm[i]) / norm[10 + i] : 0.0f;
    }
    __syncthreads();
    // forward
    mlp_layer<XS, XS>(X, W1, Bs, H1, tx, ty);
    __syncthreads();
    mlp_layer<64, HS>(H1, W2, Bs + 64, H2, tx, ty);
    __syncthreads();
    mlp_layer<64, HS>(H2, W3, Bs + 128, H3, tx, ty);
    __syncthreads();
    if (t < 2 * TSMP) {
        const int s = t >> 1, j = t & 1;
        int64_t g;
        const bool on = sample(s, g);
        float y = B4[j];
        for (int o = 0; o < 64; o += 4) {
            const float4 h = *reinterpret_cast<const float4*>(H3 + s * HS + o);
            const float4 w = *reinterpret_cast<const float4*>(W4 + j * 64 + o);
            y = fmaf(w.x, h.x, y);
            y = fmaf(w.y, h.y, y);
            y = fmaf(w.z, h.z, y);
            y = fmaf(w.w, h.w, y);
        }
        const float r = on ? y - (targ[j * n + g] - norm[20 + j]) / norm[22 + j] : 0.0f;
        DY[s * 2 + j] = r * (1.0f / (float)count);
        float v = r * r;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((t & 31) == 0) R2[t >> 5] = v;
    }
    __syncthreads();
    // output layer gradients: (j, o) over half the samples each
    {
        const int o = t & 63, j = (t >> 6) & 1, s0 = (t >> 7) * (TSMP / 2);
        float a = 0.0f;
        for (int s = s0; s < s0 + TSMP / 2; s++) a = fmaf(DY[s * 2 + j], H3[s * HS + o], a);
        atomicAdd(&grad[P_W4 + j * 64 + o], a);
        if (t < 2) {
            float bsum = 0.0f;
            for (int s = 0; s < TSMP; s++) bsum += DY[s * 2 + t];
            atomicAdd(&grad[P_B4 + t], bsum);
        }
    }
    __syncthreads();
    // dz3 = (W4^T dy) (1 - h3^2)
    {
        const int o = t & 63;
        for (int s = t >> 6; s < TSMP; s += 4) {
            const float h = H3[s * HS + o];
            H3[s * HS + o] = (W4[o] * DY[s * 2] + W4[64 + o] * DY[s * 2 + 1]) * (1.0f - h * h);
        }
    }
    __syncthreads();
    // hidden layers 3 and 2: dW = dz^T h_prev, db = sum dz; then dz_prev = (W^T dz) (1 - h_prev^2)
#pragma unroll 1
    for (int layer = 3; layer >= 2; layer--) {
        const float* Z = (layer == 3) ? H3 : H2;
        float* Hp = (layer == 3) ? H2 : H1;
        const float* Wl = (layer == 3) ? W3 : W2;
        const int pw = (layer == 3) ? P_W3 : P_W2, pb = (layer == 3) ? P_B3 : P_B2;
        float acc[4][4];
#pragma unroll
        for (int r = 0; r < 4; r++)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[r][q] = 0.0f;
#pragma unroll 4
        for (int s = 0; s < TSMP; s++) {  // outputs 4 ty + r, inputs 4 tx + q
            const float4 z = *reinterpret_cast<const float4*>(Z + s * HS + 4 * ty);
            const float4 h = *reinterpret_cast<const float4*>(Hp + s * HS + 4 * tx);
            const float zr[4] = {z.x, z.y, z.z, z.w}, hq[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int r = 0; r < 4; r++)
#pragma unroll
                for (int q = 0; q < 4; q++) acc[r][q] = fmaf(zr[r], hq[q], acc[r][q]);
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {  // pairs: the gradient's base is 8-byte aligned
            float2* g = reinterpret_cast<float2*>(grad + pw + (4 * ty + r) * 64 + 4 * tx);
            atomicAdd(g, make_float2(acc[r][0], acc[r][1]));
            atomicAdd(g + 1, make_float2(acc[r][2], acc[r][3]));
        }
        if (t < 64) {
            float bs = 0.0f;
            for (int s = 0; s < TSMP; s++) bs += Z[s * HS + t];
            atomicAdd(&grad[pb + t], bs);
        }
#pragma unroll
        for (int r = 0; r < 4; r++)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[r][q] = 0.0f;
#pragma unroll 4
        for (int o = 0; o < 64; o += 4) {  // samples ty + 16 r, inputs 4 tx + q
            float4 z[4], w[4];
#pragma unroll
            for (int r = 0; r < 4; r++) z[r] = *reinterpret_cast<const float4*>(Z + (ty + 16 * r) * HS + o);
#pragma unroll
            for (int u = 0; u < 4; u++) w[u] = *reinterpret_cast<const float4*>(Wl + (o + u) * HS + 4 * tx);
#pragma unroll
            for (int r = 0; r < 4; r++) {
                const float zu[4] = {z[r].x, z[r].y, z[r].z, z[r].w};
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    acc[r][0] = fmaf(zu[u], w[u].x, acc[r][0]);
                    acc[r][1] = fmaf(zu[u], w[u].y, acc[r][1]);
                    acc[r][2] = fmaf(zu[u], w[u].z, acc[r][2]);
                    acc[r][3] = fmaf(zu[u], w[u].w, acc[r][3]);
                }
            }
        }
        __syncthreads();  // every thread has read h_prev
#pragma unroll
        for (int r = 0; r < 4; r++) {
            float4* d = reinterpret_cast<float4*>(Hp + (ty + 16 * r) * HS + 4 * tx);
            const float4 h = *d;
            *d = make_float4(acc[r][0] * (1.0f - h.x * h.x), acc[r][1] * (1.0f - h.y * h.y),
                             acc[r][2] * (1.0f - h.z * h.z), acc[r][3] * (1.0f - h.w * h.w));
        }
        __syncthreads();
    }
    // first layer: dW1 = dz1^T x (three of the twelve columns per thread), db1
    {
        const int o = t >> 2, i0 = (t & 3) * 3;
        float acc[3] = {0.0f, 0.0f, 0.0f};
        float bs = 0.0f;
        for (int s = 0; s < TSMP; s++) {
            const float z = H1[s * HS + o];
            bs += z;
#pragma unroll
            for (int q = 0; q < 3; q++) acc[q] = fmaf(z, X[s * XS + i0 + q], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < 3; q++)
            if (i0 + q < MLP_NIN) atomicAdd(&grad[P_W1 + o * MLP_NIN + i0 + q], acc[q]);
        if ((t & 3) == 0) atomicAdd(&grad[P_B1 + o], bs);
    }
    // loss: one sum per CTA, as the running sum's rounding grows with the number of its terms
    if (t == 0) atomicAdd(loss, (R2[0] + R2[1]) + (R2[2] + R2[3]));
}

__global__ void k_adam(float* __restrict__ P, float* __restrict__ grad, float* __restrict__ m1,
                       float* __restrict__ m2, float lr, float c1, float c2) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= MLP_NPARAM) return;
    const float g = grad[q];
    const float a = 0.9f * m1[q] + 0.1f * g;
    const float b = 0.999f * m2[q] + 0.001f * g * g;
    m1[q] = a;
    m2[q] = b;
    P[q] -= lr * (a * c1) / (sqrtf(b * c2) + 1e-8f);
    grad[q] = 0.0f;
}

// FP32 forward of the training path, one thread per sample
__global__ void k_fwd32(const float* __restrict__ Pg, const float* __restrict__ norm, const float* __restrict__ feat,
                        int64_t n, float* __restrict__ out) {
    extern __shared__ __align__(16) float P[];
    for (int q = threadIdx.x; q < MLP_NPARAM; q += blockDim.x) P[q] = Pg[q];
    __syncthreads();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float x[MLP_NIN], h[64], h2[64];
#pragma unroll
    for (int i = 0; i < MLP_NIN; i++) x[i] = (feat[i * n + s] - norm[i]) / norm[10 + i];
    for (int o = 0; o < 64; o++) {
        float z = P[P_B1 + o];
#pragma unroll
        for (int i = 0; i < MLP_NIN; i++) z = fmaf(P[P_W1 + o * MLP_NIN + i], x[i], z);
        h[o] = tanhf(z);
    }
    for (int o = 0; o < 64; o++) {
        float z = P[P_B2 + o];
        for (int i = 0; i < 64; i++) z = fmaf(P[P_W2 + o * 64 + i], h[i], z);
        h2[o] = tanhf(z);
    }
    for (int o = 0; o < 64; o++) {
        float z = P[P_B3 + o];
        for (int i = 0; i < 64; i++) z = fmaf(P[P_W3 + o * 64 + i], h2[i], z);
        h[o] = tanhf(z);
    }
    for (int j = 0; j < 2; j++) {
        float y = P[P_B4 + j];
        for (int o = 0; o < 64; o++) y = fmaf(P[P_W4 + j * 64 + o], h[o], y);
        out[j * n + s] = y * norm[22 + j] + norm[20 + j];
    }
}

// bf16 tensor-core inference of given inputs, 128 samples per CTA
__global__ void __launch_bounds__(MLP_ROWS) k_fwd16(const uint8_t* __restrict__ img, const float* __restrict__ feat,
                                                   int64_t n, float* __restrict__ out, int* err) {
    extern __shared__ __align__(16) uint8_t sm[];
    const int64_t s = (int64_t)blockIdx.x * MLP_ROWS + threadIdx.x;
    const bool active = s < n;
    MlpCta C;
    mlp_begin(C, sm, img);
    float f[MLP_NIN], y[MLP_NOUT];
#pragma unroll
    for (int q = 0; q < MLP_NIN; q++) f[q] = active ? feat[q * n + s] : 0.0f;
    const bool ran = mlp_infer(C, f, active, y);
    mlp_end(C);
    if (!C.ok && threadIdx.x == 0) atomicExch(err, 1);
    if (active) {
        out[s] = ran ? y[0] : __int_as_float(0x7fc00000);
        out[n + s] = ran ? y[1] : __int_as_float(0x7fc00000);
    }
}

int check_model(const hamr_mlp* m) {
    if (!m) return set_error(HAMR_EINVAL, "model is NULL");
    int dev = -1;
    cudaGetDevice(&dev);
    if (dev != m->device) return set_error(HAMR_EINVAL, "the model lives on device %d, device %d is current", m->device,
                                           dev);
    return HAMR_OK;
}

#define MLP_CUDA(x)                                                                       \
    do {                                                                                  \
        cudaError_t e_ = (x);                                                             \
        if (e_ != cudaSuccess) return set_error(HAMR_ECUDA, "%s: %s", #x, cudaGetErrorString(e_)); \
    } while (0)

int repack(hamr_mlp* m, cudaStream_t s) {
    k_pack<<<(PACK_THREADS + 255) / 256, 256, 0, s>>>(m->params, m->norm, m->img);
    MLP_CUDA(cudaGetLastError());
    return HAMR_OK;
}

}  // namespace

// inference launch of the standalone inversion (c2p.cu) and the grid
const uint8_t* mlp_image(const hamr_mlp* m) { return m ? m->img : nullptr; }
int* mlp_error_ptr(const hamr_mlp* m) { return m ? m->err : nullptr; }

}  // namespace hamr

using namespace hamr;

extern "C" {

int hamr_prim2cons(const hamr_c2p_desc* d, int64_t n, const double* prim, const double* x1, const double* x2,
                   double* U, void* stream) {
    if (!d || n < 0) return set_error(HAMR_EINVAL, "descriptor NULL or n < 0");
    if (n == 0) return HAMR_OK;
    if (!prim || !x1 || !x2 || !U) return set_error(HAMR_EINVAL, "NULL array");
    k_prim2cons<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(*d, n, prim, x1, x2, U);
    MLP_CUDA(cudaGetLastError());
    return HAMR_OK;
}

int hamr_mlp_create(hamr_mlp** out, uint64_t seed) {
    if (!out) return set_error(HAMR_EINVAL, "out is NULL");
    *out = nullptr;
    hamr_mlp* m = new hamr_mlp;
    cudaGetDevice(&m->device);
    auto fail_free = [&](cudaError_t e) {
        hamr_mlp_destroy(m);
        return set_error(HAMR_ECUDA, "model allocation failed: %s", cudaGetErrorString(e));
    };
    cudaError_t e;
    if ((e = cudaMalloc(&m->params, 4 * MLP_NPARAM * sizeof(float))) != cudaSuccess) return fail_free(e);
    m->grad = m->params + MLP_NPARAM;
    m->m1 = m->grad + MLP_NPARAM;
    m->m2 = m->m1 + MLP_NPARAM;
    if ((e = cudaMalloc(&m->norm, MLP_NNORM * sizeof(float))) != cudaSuccess) return fail_free(e);
    if ((e = cudaMalloc(&m->img, MLP_IMG_BYTES)) != cudaSuccess) return fail_free(e);
    if ((e = cudaMalloc(&m->sums, 24 * sizeof(double))) != cudaSuccess) return fail_free(e);
    if ((e = cudaMalloc(&m->err, sizeof(int))) != cudaSuccess) return fail_free(e);
    // Glorot-uniform weights (bound sqrt(6 / (fan_in + fan_out))), zero biases; uniform
    // numbers from SplitMix64 of seed ^ parameter index
    std::vector<float> P(MLP_NPARAM, 0.0f);
    auto sm64 = [](uint64_t x) {
        x += 0x9E3779B97F4A7C15ull;
        x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
        x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
        return x ^ (x >> 31);
    };
    const int offs[4] = {P_W1, P_W2, P_W3, P_W4}, fin[4] = {MLP_NIN, 64, 64, 64}, fout[4] = {64, 64, 64, 2};
    for (int l = 0; l < 4; l++) {
        const double bound = std::sqrt(6.0 / (fin[l] + fout[l]));
        for (int q = 0; q < fin[l] * fout[l]; q++) {
            const uint64_t z = sm64(seed ^ (uint64_t)(offs[l] + q));
            const double u = (double)(z >> 11) * (1.0 / 9007199254740992.0);
            P[offs[l] + q] = (float)((2.0 * u - 1.0) * bound);
        }
    }
    std::vector<float> norm(MLP_NNORM, 0.0f);
    for (int q = 0; q < 10; q++) norm[10 + q] = 1.0f;
    norm[22] = norm[23] = 1.0f;
    if ((e = cudaMemcpy(m->params, P.data(), MLP_NPARAM * sizeof(float), cudaMemcpyHostToDevice)) != cudaSuccess)
        return fail_free(e);
    if ((e = cudaMemset(m->grad, 0, 3 * MLP_NPARAM * sizeof(float))) != cudaSuccess) return fail_free(e);
    if ((e = cudaMemcpy(m->norm, norm.data(), MLP_NNORM * sizeof(float), cudaMemcpyHostToDevice)) != cudaSuccess)
        return fail_free(e);
    if ((e = cudaMemset(m->err, 0, sizeof(int))) != cudaSuccess) return fail_free(e);
    int rc = repack(m, 0);
    if (rc) {
        hamr_mlp_destroy(m);
        return rc;
    }
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) return fail_free(e);
    *out = m;
    return HAMR_OK;
}

int hamr_mlp_destroy(hamr_mlp* m) {
    if (!m) return HAMR_OK;
    cudaFree(m->params);
    cudaFree(m->norm);
    cudaFree(m->img);
    cudaFree(m->sums);
    cudaFree(m->loss);
    cudaFree(m->err);
    delete m;
    return HAMR_OK;
}

int hamr_mlp_get_params(const hamr_mlp* m, float* params, float* norm) {
    if (int rc = check_model(m)) return rc;
    MLP_CUDA(cudaDeviceSynchronize());
    if (params) MLP_CUDA(cudaMemcpy(params, m->params, MLP_NPARAM * sizeof(float), cudaMemcpyDeviceToHost));
    if (norm) MLP_CUDA(cudaMemcpy(norm, m->norm, MLP_NNORM * sizeof(float), cudaMemcpyDeviceToHost));
    return HAMR_OK;
}

int hamr_mlp_set_params(hamr_mlp* m, const float* params, const float* norm) {
    if (int rc = check_model(m)) return rc;
    if (norm)
        for (int q = 0; q < MLP_NNORM; q++)
            if (!std::isfinite(norm[q]) || (((q >= 10 && q < 20) || q >= 22) && !(norm[q] > 0.0f)))
                return set_error(HAMR_EINVAL, "norm[%d] must be finite (standard deviations > 0)", q);
    MLP_CUDA(cudaDeviceSynchronize());
    if (params) MLP_CUDA(cudaMemcpy(m->params, params, MLP_NPARAM * sizeof(float), cudaMemcpyHostToDevice));
    if (norm) MLP_CUDA(cudaMemcpy(m->norm, norm, MLP_NNORM * sizeof(float), cudaMemcpyHostToDevice));
    if (int rc = repack(m, 0)) return rc;
    MLP_CUDA(cudaDeviceSynchronize());
    return HAMR_OK;
}

int hamr_mlp_features(const hamr_c2p_desc* d, int64_t n, const double* U, const double* B, const double* x1,
                      const double* x2, const double* prim, float* feat, float* targ, void* stream) {
    if (!d || n < 0) return set_error(HAMR_EINVAL, "descriptor NULL or n < 0");
    if (n == 0) return HAMR_OK;
    if (!U || !B || !x1 || !x2 || !feat) return set_error(HAMR_EINVAL, "NULL array");
    if ((prim == nullptr) != (targ == nullptr)) return set_error(HAMR_EINVAL, "prim and targ go together");
    k_features<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(*d, n, U, B, x1, x2, prim, feat, targ);
    MLP_CUDA(cudaGetLastError());
    return HAMR_OK;
}

int hamr_mlp_fit_norm(hamr_mlp* m, int64_t n, const float* feat, const float* targ, void* stream) {
    if (int rc = check_model(m)) return rc;
    if (n < 2 || !feat || !targ) return set_error(HAMR_EINVAL, "need n >= 2 samples with targets");
    cudaStream_t s = (cudaStream_t)stream;
    MLP_CUDA(cudaMemsetAsync(m->sums, 0, 24 * sizeof(double), s));
    k_norm_sums<<<1216, 128, 0, s>>>(n, feat, targ, m->sums);
    MLP_CUDA(cudaGetLastError());
    double h[24];
    MLP_CUDA(cudaMemcpyAsync(h, m->sums, sizeof(h), cudaMemcpyDeviceToHost, s));
    MLP_CUDA(cudaStreamSynchronize(s));
    float norm[MLP_NNORM];
    for (int q = 0; q < 12; q++) {
        const double mean = h[q] / (double)n;
        const double var = std::max(h[12 + q] / (double)n - mean * mean, 0.0);
        const double sd = std::max(std::sqrt(var), 1e-6 * std::max(1.0, std::fabs(mean)));
        if (q < MLP_NIN) {
            norm[q] = (float)mean;
            norm[10 + q] = (float)sd;
        } else {
            norm[20 + q - MLP_NIN] = (float)mean;
            norm[22 + q - MLP_NIN] = (float)sd;
        }
    }
    return hamr_mlp_set_params(m, nullptr, norm);
}

int hamr_mlp_train(hamr_mlp* m, int64_t n, const float* feat, const float* targ, const hamr_mlp_train_args* a,
                   float* loss, void* stream) {
    if (int rc = check_model(m)) return rc;
    if (!a || n < 1 || !feat || !targ) return set_error(HAMR_EINVAL, "need arguments, n >= 1 and data");
    if (a->steps < 1 || a->batch < TB || a->batch % TB) return set_error(HAMR_EINVAL, "steps >= 1, batch a multiple of 128");
    if (!(a->lr > 0.0f) || !(a->lr_final >= 0.0f)) return set_error(HAMR_EINVAL, "lr > 0, lr_final >= 0");
    cudaStream_t s = (cudaStream_t)stream;
    if (m->loss_cap < a->steps) {
        cudaFree(m->loss);
        m->loss = nullptr;
        MLP_CUDA(cudaMalloc(&m->loss, (size_t)a->steps * sizeof(float)));
        m->loss_cap = a->steps;
    }
    MLP_CUDA(cudaFuncSetAttribute(k_mlp_fb, cudaFuncAttributeMaxDynamicSharedMemorySize, FB_SMEM));
    MLP_CUDA(cudaMemsetAsync(m->loss, 0, (size_t)a->steps * sizeof(float), s));
    MLP_CUDA(cudaMemsetAsync(m->grad, 0, MLP_NPARAM * sizeof(float), s));
    const unsigned nb = (unsigned)(a->batch / TSMP);
    for (int64_t k = 0; k < a->steps; k++) {
        k_mlp_fb<<<nb, TTHR, FB_SMEM, s>>>(m->params, m->norm, feat, targ, n, 1, 0, a->batch, a->seed, k, m->grad,
                                         m->loss + k);
        m->adam_t++;
        const double tt = (double)m->adam_t;
        const double frac = (a->steps > 1) ? (double)k / (double)(a->steps - 1) : 1.0;
        const double lr = a->lr_final + 0.5 * (a->lr - a->lr_final) * (1.0 + std::cos(3.14159265358979323846 * frac));
        const float c1 = (float)(1.0 / (1.0 - std::pow(0.9, tt)));
        const float c2 = (float)(1.0 / (1.0 - std::pow(0.999, tt)));
        k_adam<<<(MLP_NPARAM + 255) / 256, 256, 0, s>>>(m->params, m->grad, m->m1, m->m2, (float)lr, c1, c2);
    }
    MLP_CUDA(cudaGetLastError());
    if (int rc = repack(m, s)) return rc;
    if (loss) {
        MLP_CUDA(cudaMemcpyAsync(loss, m->loss, (size_t)a->steps * sizeof(float), cudaMemcpyDeviceToHost, s));
        MLP_CUDA(cudaStreamSynchronize(s));
        for (int64_t k = 0; k < a->steps; k++) loss[k] /= (float)(2 * a->batch);
    }
    MLP_CUDA(cudaStreamSynchronize(s));
    return HAMR_OK;
}

int hamr_mlp_loss_grad(hamr_mlp* m, int64_t n, const float* feat, const float* targ, float* grad, float* loss,
                       void* stream) {
    if (int rc = check_model(m)) return rc;
    if (n < 1 || !feat || !targ || !grad || !loss) return set_error(HAMR_EINVAL, "need n >= 1, data and outputs");
    cudaStream_t s = (cudaStream_t)stream;
    if (m->loss_cap < 1) {
        MLP_CUDA(cudaMalloc(&m->loss, sizeof(float)));
        m->loss_cap = 1;
    }
    MLP_CUDA(cudaFuncSetAttribute(k_mlp_fb, cudaFuncAttributeMaxDynamicSharedMemorySize, FB_SMEM));
    MLP_CUDA(cudaMemsetAsync(m->loss, 0, sizeof(float), s));
    MLP_CUDA(cudaMemsetAsync(m->grad, 0, MLP_NPARAM * sizeof(float), s));
    const unsigned nb = (unsigned)((n + TSMP - 1) / TSMP);
    k_mlp_fb<<<nb, TTHR, FB_SMEM, s>>>(m->params, m->norm, feat, targ, n, 0, 0, n, 0, 0, m->grad, m->loss);
    MLP_CUDA(cudaGetLastError());
    MLP_CUDA(cudaMemcpyAsync(grad, m->grad, MLP_NPARAM * sizeof(float), cudaMemcpyDeviceToHost, s));
    MLP_CUDA(cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
    MLP_CUDA(cudaMemsetAsync(m->grad, 0, MLP_NPARAM * sizeof(float), s));
    MLP_CUDA(cudaStreamSynchronize(s));
    loss[0] /= (float)(2 * n);
    return HAMR_OK;
}

int hamr_mlp_forward(const hamr_mlp* m, int64_t n, const float* feat, float* out, int tensor_cores, void* stream) {
    if (int rc = check_model(m)) return rc;
    if (n < 0 || (n > 0 && (!feat || !out))) return set_error(HAMR_EINVAL, "n >= 0 with arrays");
    if (n == 0) return HAMR_OK;
    cudaStream_t s = (cudaStream_t)stream;
    if (tensor_cores) {
        MLP_CUDA(cudaFuncSetAttribute(k_fwd16, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_SMEM_BYTES));
        k_fwd16<<<(unsigned)((n + MLP_ROWS - 1) / MLP_ROWS), MLP_ROWS, MLP_SMEM_BYTES, s>>>(m->img, feat, n, out,
                                                                                         m->err);
    } else {
        MLP_CUDA(cudaFuncSetAttribute(k_fwd32, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_NPARAM * 4));
        k_fwd32<<<(unsigned)((n + 127) / 128), 128, MLP_NPARAM * 4, s>>>(m->params, m->norm, feat, n, out);
    }
    MLP_CUDA(cudaGetLastError());
    return HAMR_OK;
}

int hamr_mlp_error_flag(hamr_mlp* m, int* flag) {
    if (int rc = check_model(m)) return rc;
    if (!flag) return set_error(HAMR_EINVAL, "flag is NULL");
    MLP_CUDA(cudaDeviceSynchronize());
    MLP_CUDA(cudaMemcpy(flag, m->err, sizeof(int), cudaMemcpyDeviceToHost));
    MLP_CUDA(cudaMemset(m->err, 0, sizeof(int)));
    return HAMR_OK;
}

}  // extern "C"
