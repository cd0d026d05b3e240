// step.cu -- the per-block stage kernels of the midpoint step
// (Liska et al. 2019, Sec. 2.1 and 2.5-2.7).
//
// One stage = boundary conditions (one launch) -> per direction: edge values
// (reconstruction) and face fluxes -> edge EMFs -> CT face update ->
// cell update + inversion + floors (+ CFL reduction in the corrector), the
// last in update.cu.
// Fluxes, EMFs and edge values go through HBM: the FP64 path is bound by the
// FP64 pipe, so every face flux and every parabola is computed exactly once
// and re-read from memory instead of recomputed in a halo.
#include "stage.cuh"

namespace hamr {
namespace {

__device__ __forceinline__ void b_centre_b(const BlockView& v, double* __restrict__ P, const double* __restrict__ B, long t) {
    const long n = (long)v.n1 * v.n2 * v.n3;
    if (t >= n) return;
    const int i = (int)(t % v.n1), j = (int)((t / v.n1) % v.n2), k = (int)(t / ((long)v.n1 * v.n2));
    double Bc[3];
    centre_field(v, B, i, j, k, v.gc[G_IGDET * v.n2d + gidx(v, i, j)], Bc);
    const long c = cidx(v, i, j, k);
    P[B1 * v.nc + c] = Bc[0];
    P[B2 * v.nc + c] = Bc[1];
    P[B3 * v.nc + c] = Bc[2];
}

__global__ void k_centre_b(BlockView v, double* __restrict__ P, const double* __restrict__ B) {
    b_centre_b(v, P, B, (long)blockIdx.x * blockDim.x + threadIdx.x);
}


// ---------------------------------------------------------------- boundaries
// The conditions of x3, x2, x1 in this order, each over the full padded extent of the other two
// directions, composed: a ghost cell takes the interior cell that its x1, then x2, then x3 map lead to.
// Polar (x2): ghost (j = -1-m, k) takes (j = m, k + n3/2) with utilde^2, B^2 and Bbar^2 negated; axis
// faces 0. Outflow: copy of the last interior cell/face; NOINFLOW clamps utilde^1. Periodic: wrap; face n
// takes face 0.
__device__ __forceinline__ int cell_src(int bc, int n, int g) {
    if (bc == HAMR_BC_PERIODIC) return g < 0 ? g + n : g - n;
    if (bc == HAMR_BC_POLAR) return g < 0 ? -1 - g : 2 * n - 1 - g;
    return g < 0 ? 0 : n - 1;
}
__device__ __forceinline__ int face_src(int bc, int n, int g) {
    if (bc == HAMR_BC_PERIODIC) return g < 0 ? g + n : g - n;
    if (bc == HAMR_BC_POLAR) return g < 0 ? -g : 2 * n - g;
    return g < 0 ? 0 : n;
}

// the interior location that (x[1], x[2], x[3]) takes its value from, in place; f: the direction of a face
// field's component (0: a cell field). Returns whether a polar map was passed.
__device__ __forceinline__ bool bc_source(const BlockView& v, int f, int x[4]) {
    const int n[4] = {0, v.n1, v.n2, v.n3};
    bool polar = false;
#pragma unroll
    for (int e = 1; e <= 3; e++) {
        const int hi = n[e] + ((f == e && v.bc[2 * e - 1] != HAMR_BC_PERIODIC) ? 1 : 0);  // first ghost above
        if (x[e] >= 0 && x[e] < hi) continue;
        const int bc = v.bc[2 * (e - 1) + (x[e] < 0 ? 0 : 1)];
        x[e] = (f == e) ? face_src(bc, n[e], x[e]) : cell_src(bc, n[e], x[e]);
        if (bc == HAMR_BC_POLAR) {
            polar = true;
            x[3] = ((x[3] + v.n3 / 2) % v.n3 + v.n3) % v.n3;
        }
    }
    return polar;
}

// Every ghost cell and face in one launch (threads over the x3 slabs, then the x2 and x1 ones without
// them, then the axis faces of the lower pole): sources are interior, so no pass waits for another. Four
// dependent launches before: a 256x128x64 block 38 -> 20 us, a 64x32x16 block 21 -> 7 us.
// P32, K32 (mixed precision on a single block, else null): the ghost cells of the FP32 copy of the
// primitives and of its entropy tracer kappa, from the same sources
__global__ void k_bc(BlockView v, double* __restrict__ P, double* __restrict__ B, float* __restrict__ P32,
                     float* __restrict__ K32) {
    long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long s3 = 2L * NG * v.n1p * v.n2p, s2 = 2L * NG * v.n1p * v.n3, s1 = 2L * NG * v.n2 * v.n3;
    int i, j, k;
    if (t < s3) {
        const int m = (int)(t / ((long)v.n1p * v.n2p));
        i = (int)(t % v.n1p) - NG;
        j = (int)((t / v.n1p) % v.n2p) - NG;
        k = m < NG ? m - NG : v.n3 + m - NG;
    } else if ((t -= s3) < s2) {
        const int m = (int)((t / v.n1p) % (2 * NG));
        i = (int)(t % v.n1p) - NG;
        j = m < NG ? m - NG : v.n2 + m - NG;
        k = (int)(t / (2L * NG * v.n1p));
    } else if ((t -= s2) < s1) {
        const int m = (int)(t % (2 * NG));
        i = m < NG ? m - NG : v.n1 + m - NG;
        j = (int)((t / (2 * NG)) % v.n2);
        k = (int)(t / (2L * NG * v.n2));
    } else if ((t -= s1) < (long)v.n1 * v.n3) {
        if (v.bc[2] == HAMR_BC_POLAR) B[v.nc + cidx(v, (int)(t % v.n1), 0, (int)(t / v.n1))] = 0.0;
        return;
    } else {
        return;
    }
    const long dst = cidx(v, i, j, k);
    {
        int x[4] = {0, i, j, k};
        const bool polar = bc_source(v, 0, x);
        const long src = cidx(v, x[1], x[2], x[3]);
        const bool nolo = i < 0 && v.bc[0] == HAMR_BC_OUTFLOW_NOINFLOW;
        const bool nohi = i >= v.n1 && v.bc[1] == HAMR_BC_OUTFLOW_NOINFLOW;
#pragma unroll
        for (int q = 0; q < NPRIM; q++) {
            double p = P[q * v.nc + src];
            if (polar && (q == U2 || q == B2)) p = -p;
            if (q == U1) {
                if (nohi && p < 0.0) p = 0.0;
                if (nolo && p > 0.0) p = 0.0;
            }
            P[q * v.nc + dst] = p;
            if (P32) P32[q * v.nc + dst] = (float)p;
        }
        if (K32) K32[dst] = K32[src];  // kappa depends on rho and u only, which the map keeps
    }
#pragma unroll
    for (int f = 1; f <= 3; f++) {
        int x[4] = {0, i, j, k};
        const bool polar = bc_source(v, f, x);
        double* b = B + (f - 1) * v.nc;
        const bool axis = f == 2 && ((j == 0 && v.bc[2] == HAMR_BC_POLAR) || (j == v.n2 && v.bc[3] == HAMR_BC_POLAR));
        const long src = cidx(v, x[1], x[2], x[3]);
        if (axis)
            b[dst] = 0.0;
        else if (src != dst)
            b[dst] = (polar && f == 2) ? -b[src] : b[src];
    }
}

// ---------------------------------------------------------------- reconstruction
// Edge values of every cell that borders a flux face of direction dir: cells
// -1..n_dir along dir, -1..n_e across, for the 7 primitives other than B^dir
// and the entropy tracer kappa of the cells (an eighth variable, read from K,
// whose edge values go to the B^dir fields of QL and QR).
// Every slope and every PPM interface value is formed once and shared by the
// two cells that use it: along x1 a warp holds 32 consecutive cells (28 of
// them produced) and passes values between lanes by shuffles; along x2 and
// x3 a thread sweeps recon_seg cells of one pencil (consecutive threads on
// consecutive i, so loads and stores coalesce). T = float (mixed precision)
// reads the FP32 copy of the primitives and writes FP32 edge values.
// Shock flattening (Colella & Woodward 1984), optional with PPM: a coefficient
// f in [0, 1] per cell of the reconstruction range, from p = (gam - 1) u and
// the velocity primitive w along dir. A relative pressure jump across the
// cell above 0.33 of the smaller neighbour with converging flow (w(c-1) >
// w(c+1)) marks a shock; f = 10 (|dp1| / |dp2| - 3/4) clamped to [0, 1], dp1 =
// p(c+1) - p(c-1), dp2 = p(c+2) - p(c-2), and f = 1 for dp2 = 0 (the ratio in
// magnitude: at a narrow pressure peak dp2 is zero up to rounding, and a
// signed ratio would follow the rounding noise). The coefficient stays with its cell
// (no max with the upwind neighbour: its stencil would pass three ghost
// layers). It is written to field 0 of the dir-flux array, which the flux
// kernel of dir fills only afterwards; the reconstruction blends both
// interface values of the cell toward its value, f q + (1 - f) a, before the
// parabola constraints.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

template <int DIR, typename T>
__device__ __forceinline__ void b_flatten(const BlockView& v, PhysArgs ph, const T* __restrict__ P,
                                          T* __restrict__ Fl, long t) {
    const int e1 = v.n1 + 2, e2 = v.n2 + 2, e3 = v.n3 + 2;
    if (t >= (long)e1 * e2 * e3) return;
    const int i = (int)(t % e1) - 1, j = (int)((t / e1) % e2) - 1, k = (int)(t / ((long)e1 * e2)) - 1;
    const long c = cidx(v, i, j, k);
    const long st = (DIR == 1) ? 1 : ((DIR == 2) ? (long)v.n1p : (long)v.n1p * v.n2p);
    const T* u = P + UU * v.nc + c;
    const T* w = P + (U1 + DIR - 1) * v.nc + c;
    const T gm1 = (T)(ph.gam - 1.0);
    // products rounded on their own (no contraction into the differences)
    const T pm = mul_rn(gm1, u[-st]), pp = mul_rn(gm1, u[st]);
    const T dp1 = pp - pm;
    const T dp2 = mul_rn(gm1, u[2 * st] - u[-2 * st]);
    const T pmin = pm < pp ? pm : pp;
    const T a1 = fabs(dp1), a2 = fabs(dp2);
    T f = T(0);
    if (a1 > mul_rn(T(0.33), pmin) && w[-st] > w[st]) {
        if (a2 == T(0)) {
            f = T(1);
        } else {
            const T x = mul_rn(T(10), a1 / a2 - T(0.75));
            f = x < T(0) ? T(0) : (x > T(1) ? T(1) : x);
        }
    }
    Fl[c] = f;
}

template <int DIR, typename T>
__global__ void k_flatten(BlockView v, PhysArgs ph, const T* __restrict__ P, T* __restrict__ Fl) {
    b_flatten<DIR, T>(v, ph, P, Fl, (long)blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename T>
__device__ __forceinline__ void flatten_edges(T f, T qc, T& l, T& r) {
    l = f * qc + (T(1) - f) * l;
    r = f * qc + (T(1) - f) * r;
}

// entropy tracer kappa = p / rho^gam of every padded cell into K: one power per
// cell; the reconstruction carries kappa to the faces like a primitive
// (predictor: also into Kn, the entropy slot of the U^n cache, where the cell
// update takes it for U^n instead of forming the power again; in mixed
// precision this kappa is the FP32 one, like the entropy fluxes)
template <typename T>
__device__ __forceinline__ void b_kappa(const BlockView& v, T gam, const T* __restrict__ P, T* __restrict__ K,
                                        long t, double* __restrict__ Kn = nullptr) {
    const long n = (long)v.n1p * v.n2p * v.n3p;
    if (t >= n) return;
    const T kap = (gam - T(1)) * P[UU * v.nc + t] * pow_pos(P[RHO * v.nc + t], -gam);
    K[t] = kap;
    if (Kn) Kn[t] = (double)kap;
}

template <typename T>
__global__ void k_kappa(BlockView v, T gam, const T* __restrict__ P, T* __restrict__ K, double* __restrict__ Kn) {
    b_kappa<T>(v, gam, P, K, (long)blockIdx.x * blockDim.x + threadIdx.x, Kn);
}

template <int DIR>
__device__ __forceinline__ int recon_var(int n) {  // the n-th of the 7 reconstructed primitives
    return n + (n >= B1 + DIR - 1 ? 1 : 0);
}

template <typename T>
__device__ __forceinline__ T limited_slope(int recon, T qm, T q0, T qp) {
    return (recon == HAMR_RECON_MC) ? mc_slope_i(qm, q0, qp) : minmod_slope_i(qm, q0, qp);
}

// the n-th reconstructed variable's source field and its edge-value field
template <int DIR, typename T>
__device__ __forceinline__ const T* recon_src(const BlockView& v, int n, const T* P, const T* K) {
    return (n < 7) ? P + (long)recon_var<DIR>(n) * v.nc : K;
}
template <int DIR>
__device__ __forceinline__ int recon_dst(int n) {
    return (n < 7) ? recon_var<DIR>(n) : B1 + DIR - 1;
}

template <typename T>
__device__ __forceinline__ void b_recon_row(const BlockView& v, PhysArgs ph, const T* __restrict__ P,
                                            const T* __restrict__ K, const T* __restrict__ Fl,
                                            T* __restrict__ QL, T* __restrict__ QR, long t) {
    const int n2 = v.n2 + 2, n3 = v.n3 + 2;
    const int ntile = (v.n1 + 2 + RECON_TILE - 1) / RECON_TILE;
    const long w = t >> 5;  // whole warps leave or stay together
    if (w >= (long)ntile * n2 * n3 * 8) return;
    const int lane = (int)(t & 31);
    const int tile = (int)(w % ntile);
    long rest = w / ntile;
    const int j = (int)(rest % n2) - 1;
    rest /= n2;
    const int k = (int)(rest % n3) - 1;
    const int nv = (int)(rest / n3);
    const int q = recon_dst<1>(nv);
    const int i = RECON_TILE * tile - 3 + lane;               // lanes 2..29 produce cells tile*28-1 .. +27
    const int ic = min(max(i, -NG), v.n1 + NG - 1);           // loads stay inside the padded row
    const long c = cidx(v, 0, j, k);
    const T qc = recon_src<1>(v, nv, P, K)[c + ic];
    const T qm = __shfl_up_sync(0xffffffffu, qc, 1);
    const T qp = __shfl_down_sync(0xffffffffu, qc, 1);
    T l, r;
    if (ph.recon == HAMR_RECON_PPM) {
        // the same differences and formulas as the pencil sweep (identical edge values)
        const T dr = qp - qc;
        const T dl = __shfl_up_sync(0xffffffffu, dr, 1);
        const T sc = mc_slope_d(dl, dr, qp - qm);             // valid on lanes 1..30
        const T sp = __shfl_down_sync(0xffffffffu, sc, 1);
        r = ppm_face_d(qc, dr, sc, sp);                       // interface i+1/2, valid on lanes 1..29
        l = __shfl_up_sync(0xffffffffu, r, 1);                // interface i-1/2, valid on lanes 2..30
        if (ph.flatten) flatten_edges(Fl[c + ic], qc, l, r);
        ppm_limit(qc, l, r);
    } else {
        const T dq = limited_slope(ph.recon, qm, qc, qp);
        l = qc - T(0.5) * dq;
        r = qc + T(0.5) * dq;
    }
    if (lane >= 2 && lane <= 29 && i <= v.n1) {
        QL[q * v.nc + c + i] = l;
        QR[q * v.nc + c + i] = r;
    }
}

template <int DIR, typename T>
__device__ __forceinline__ void b_recon_sweep(const BlockView& v, PhysArgs ph, const T* __restrict__ P,
                                              const T* __restrict__ K, const T* __restrict__ Fl,
                                              T* __restrict__ QL, T* __restrict__ QR, long t) {
    // cells along the sweep: -1..n_dir; across: the two other directions, the faster one first
    // (x1 for the x2 and x3 sweeps, so that loads and stores coalesce; x2 for the x1 sweep)
    const int na = (DIR == 1 ? v.n1 : (DIR == 2 ? v.n2 : v.n3)) + 2;
    const int seglen = ph.recon_seg;
    const int nseg = (na + seglen - 1) / seglen;
    const int n1 = (DIR == 1 ? v.n2 : v.n1) + 2, no = (DIR == 3 ? v.n2 : v.n3) + 2;
    if (t >= (long)n1 * no * nseg * 8) return;
    const int i = (int)(t % n1) - 1;
    long rest = t / n1;
    const int o = (int)(rest % no) - 1;
    rest /= no;
    const int seg = (int)(rest % nseg);
    const int nv = (int)(rest / nseg);
    const long st = (DIR == 1) ? 1L : ((DIR == 2) ? (long)v.n1p : (long)v.n1p * v.n2p);
    const int a0 = seg * seglen - 1;
    const int ncell = min(seglen, na - 1 - a0);           // cells a0 .. a0 + ncell - 1 (<= n_dir)
    const long co = (DIR == 1) ? cidx(v, a0, i, o) : ((DIR == 2) ? cidx(v, i, a0, o) : cidx(v, i, o, a0));
    const long c0 = (long)recon_dst<DIR>(nv) * v.nc + co;
    const T* p = recon_src<DIR>(v, nv, P, K) + co;
    if (ph.recon == HAMR_RECON_PPM) {
        // each difference of neighbours is formed once and serves two slopes and a face
        const T qmm = p[-2 * st], qm = p[-st];
        T qc = p[0], qp = p[st];
        const T dmm = qm - qmm, dm = qc - qm;
        T dc = qp - qc;
        const T sm = mc_slope_d(dmm, dm, qc - qmm);
        T sc = mc_slope_d(dm, dc, qp - qm);
        T fl = ppm_face_d(qm, dm, sm, sc);  // interface a0 - 1/2
        for (int m = 0; m < ncell; m++) {
            const T qpp = p[(m + 2) * st];
            const T dp = qpp - qp;
            const T sp = mc_slope_d(dc, dp, qpp - qc);
            const T fr = ppm_face_d(qc, dc, sc, sp);  // interface a + 1/2
            T l = fl, r = fr;
            if (ph.flatten) flatten_edges(Fl[co + m * st], qc, l, r);
            ppm_limit(qc, l, r);
            QL[c0 + m * st] = l;
            QR[c0 + m * st] = r;
            qc = qp;
            qp = qpp;
            dc = dp;
            sc = sp;
            fl = fr;
        }
    } else {
        T qm = p[-st], qc = p[0];
        for (int m = 0; m < ncell; m++) {
            const T qp = p[(m + 1) * st];
            const T dq = limited_slope(ph.recon, qm, qc, qp);
            QL[c0 + m * st] = qc - T(0.5) * dq;
            QR[c0 + m * st] = qc + T(0.5) * dq;
            qm = qc;
            qc = qp;
        }
    }
}

// FP32: M cells per thread along dir, their M + 4 values of a variable loaded together (a sweep that loads
// cell by cell is latency-bound), every slope and interface value formed once for them. Bound by
// instruction issue (comparisons and selects run at half rate) on large launches: with M = 4 a cell takes
// 1.5 slopes and 1.25 interface values instead of 3 and 2 (256x128x64 torus, x2 / x3: 91 / 83 -> 58 / 73 us;
// x1 with M = 2: 61 -> 60). On small launches the threads are what is missing: M = 1 (53x37x22:
// 5.8 us per direction, 9 with M = 4).
template <int DIR, int M, typename T>
__device__ __forceinline__ void b_recon_cells(const BlockView& v, PhysArgs ph, const T* __restrict__ P,
                                              const T* __restrict__ K, const T* __restrict__ Fl,
                                              T* __restrict__ QL, T* __restrict__ QR, long t) {
    const int nd = (DIR == 1) ? v.n1 : ((DIR == 2) ? v.n2 : v.n3);
    const int ng = (nd + 2 + M - 1) / M;  // groups of cells -1 .. nd
    const int e1 = (DIR == 1) ? ng : v.n1 + 2, e2 = (DIR == 2) ? ng : v.n2 + 2, e3 = (DIR == 3) ? ng : v.n3 + 2;
    if (t >= (long)e1 * e2 * e3) return;
    const int x1 = (int)(t % e1), x2 = (int)((t / e1) % e2), x3 = (int)(t / ((long)e1 * e2));
    const int a0 = M * ((DIR == 1) ? x1 : ((DIR == 2) ? x2 : x3)) - 1;  // the first cell along dir
    const long c = cidx(v, (DIR == 1) ? a0 : x1 - 1, (DIR == 2) ? a0 : x2 - 1, (DIR == 3) ? a0 : x3 - 1);
    const long st = (DIR == 1) ? 1 : ((DIR == 2) ? (long)v.n1p : (long)v.n1p * v.n2p);
#pragma unroll (M == 1 ? 8 : 2)
    for (int n = 0; n < 8; n++) {
        const long q = (long)recon_dst<DIR>(n) * v.nc + c;
        const T* p = recon_src<DIR>(v, n, P, K) + c;
        T x[M + 4];
#pragma unroll
        for (int m = 0; m < M + 4; m++)  // the last group stays in the block
            x[m] = p[(M == 1 ? m - 2 : min(m - 2, nd + 2 - a0)) * st];
        if (ph.recon == HAMR_RECON_PPM) {
            T d[M + 3], sl[M + 2], f[M + 1];
#pragma unroll
            for (int m = 0; m < M + 3; m++) d[m] = x[m + 1] - x[m];
#pragma unroll
            for (int m = 0; m < M + 2; m++) sl[m] = mc_slope_d(d[m], d[m + 1], x[m + 2] - x[m]);
#pragma unroll
            for (int m = 0; m < M + 1; m++) f[m] = ppm_face_d(x[m + 1], d[m + 1], sl[m], sl[m + 1]);
#pragma unroll
            for (int m = 0; m < M; m++) {
                if (a0 + m > nd) break;
                T l = f[m], r = f[m + 1];
                if (ph.flatten) flatten_edges(Fl[c + m * st], x[m + 2], l, r);
                ppm_limit(x[m + 2], l, r);
                QL[q + m * st] = l;
                QR[q + m * st] = r;
            }
        } else {
#pragma unroll
            for (int m = 0; m < M; m++) {
                if (a0 + m > nd) break;
                const T dq = limited_slope(ph.recon, x[m + 1], x[m + 2], x[m + 3]);
                QL[q + m * st] = x[m + 2] - T(0.5) * dq;
                QR[q + m * st] = x[m + 2] + T(0.5) * dq;
            }
        }
    }
}

// FP64: the non-redundant row and pencil forms; FP32: a few cells per thread
// M: cells per thread in FP32 (0: FP64)
template <int DIR, typename T, int M>
__device__ __forceinline__ void b_recon(const BlockView& v, PhysArgs ph, const T* __restrict__ P,
                                        const T* __restrict__ K, const T* __restrict__ Fl, T* __restrict__ QL,
                                        T* __restrict__ QR, long t) {
    if constexpr (M > 0)
        b_recon_cells<DIR, M>(v, ph, P, K, Fl, QL, QR, t);
    else if constexpr (DIR == 1) {
        if (ph.recon_x1_sweep)
            b_recon_sweep<1>(v, ph, P, K, Fl, QL, QR, t);
        else
            b_recon_row(v, ph, P, K, Fl, QL, QR, t);
    } else {
        b_recon_sweep<DIR>(v, ph, P, K, Fl, QL, QR, t);
    }
}

template <int DIR, typename T, int M>
__global__ void k_recon(BlockView v, PhysArgs ph, const T* __restrict__ P, const T* __restrict__ K,
                        const T* __restrict__ Fl, T* __restrict__ QL, T* __restrict__ QR) {
    b_recon<DIR, T, M>(v, ph, P, K, Fl, QL, QR, (long)blockIdx.x * blockDim.x + threadIdx.x);
}

// FP32 copy of the 8 primitive fields over the whole padded block (mixed precision)
__device__ __forceinline__ void b_to_f32(const BlockView& v, const double* __restrict__ P, float* __restrict__ P32,
                                         long t) {
    const long n = (long)v.n1p * v.n2p * v.n3p;
    if (t >= n) return;
#pragma unroll
    for (int q = 0; q < NPRIM; q++) P32[q * v.nc + t] = (float)P[q * v.nc + t];
}

__global__ void k_to_f32(BlockView v, const double* __restrict__ P, float* __restrict__ P32) {
    b_to_f32(v, P, P32, (long)blockIdx.x * blockDim.x + threadIdx.x);
}

// the tables a face flux of direction DIR reads, in the flux precision
template <int DIR, typename T>
__device__ __forceinline__ const T* face_table(const BlockView& v) {
    if constexpr (std::is_same<T, double>::value)
        return (DIR == 1) ? v.gf1 : ((DIR == 2) ? v.gf2 : v.gc);
    else
        return (DIR == 1) ? v.gf1_32 : ((DIR == 2) ? v.gf2_32 : v.gc32);
}


// ---------------------------------------------------------------- fluxes
// One side's share of an HLL face flux: cF F + cU U of that side's state, where F is its flux row
// along DIR and U its conserved row (both without sqrt(-g), which the weights carry), accumulated
// into acc (FIRST: acc is set). Uses that the two rows differ only in the contravariant index:
//   cF F_q + cU U_q = eta (cF u^D + cU u^t) u_q - (cF b^D + cU b^t) b_q + (cF delta^D_q + cU delta^t_q) ptot,
// the mass row rho (cF u^D + cU u^t), the energy row adding it, the entropy row kappa times it, and
// the transverse B slots cF (b^i u^D - b^D u^i) + cU B^i (U's B^i slot is the edge value itself).
template <int DIR, bool FIRST, typename T>
__device__ __forceinline__ void hll_side(const T pr[NPRIM], const Fluid<T>& s, T gam, T kappa, T cF, T cU,
                                         T acc[NFLUX]) {
    const T p = (gam - T(1)) * pr[UU];
    const T eta = pr[RHO] + pr[UU] + p + s.bsq;
    const T ptot = p + T(0.5) * s.bsq;
    const T tu = cF * s.ucon[DIR] + cU * s.ucon[0];
    const T tb = cF * s.bcon[DIR] + cU * s.bcon[0];
    const T a = eta * tu;
    const T mass = pr[RHO] * tu;
    const T cfp = cF * ptot;
    constexpr int i1 = (DIR == 1) ? 2 : 1, i2 = (DIR == 3) ? 2 : 3;
    const T fu = cF * s.ucon[DIR], fb = cF * s.bcon[DIR];
    // the second side's terms are summed into the running total innermost, so its products fuse
    // with the accumulation (no separate addition per component)
    T r[NFLUX];
#pragma unroll
    for (int q = 0; q < NFLUX; q++) r[q] = acc[q];
    if constexpr (FIRST) {
        acc[0] = mass;
        acc[1] = a * s.ucov[0] + (-tb * s.bcov[0] + (cU * ptot + mass));
        acc[2] = (DIR == 1) ? a * s.ucov[1] + (-tb * s.bcov[1] + cfp) : a * s.ucov[1] - tb * s.bcov[1];
        acc[3] = (DIR == 2) ? a * s.ucov[2] + (-tb * s.bcov[2] + cfp) : a * s.ucov[2] - tb * s.bcov[2];
        acc[4] = (DIR == 3) ? a * s.ucov[3] + (-tb * s.bcov[3] + cfp) : a * s.ucov[3] - tb * s.bcov[3];
        acc[5] = kappa * mass;
        acc[6] = s.bcon[i1] * fu + (-fb * s.ucon[i1] + cU * pr[B1 + i1 - 1]);
        acc[7] = s.bcon[i2] * fu + (-fb * s.ucon[i2] + cU * pr[B1 + i2 - 1]);
    } else {
        acc[0] = r[0] + mass;
        acc[1] = a * s.ucov[0] + (-tb * s.bcov[0] + (cU * ptot + (mass + r[1])));
        acc[2] = a * s.ucov[1] + (-tb * s.bcov[1] + ((DIR == 1) ? cfp + r[2] : r[2]));
        acc[3] = a * s.ucov[2] + (-tb * s.bcov[2] + ((DIR == 2) ? cfp + r[3] : r[3]));
        acc[4] = a * s.ucov[3] + (-tb * s.bcov[3] + ((DIR == 3) ? cfp + r[4] : r[4]));
        acc[5] = kappa * mass + r[5];
        acc[6] = s.bcon[i1] * fu + (-fb * s.ucon[i1] + (cU * pr[B1 + i1 - 1] + r[6]));
        acc[7] = s.bcon[i2] * fu + (-fb * s.ucon[i2] + (cU * pr[B1 + i2 - 1] + r[7]));
    }
}

// ---- FP64 face fluxes
// One side's cF F + cU U (without sqrt(-g)) onto acc (FIRST: acc is set). With X = cF B^D,
// tu = cF u^D + cU u^t and Z = i2 X + Y tu,
//   cF T^D_nu + cU T^t_nu = ((rho h + i2 B^2) tu - Y X) u_nu - Z B_nu + (cF delta^D_nu + cU delta^t_nu) ptot
// (the b^t u_nu parts of the field's two terms cancel against those of b^2), and the field slots
//   cF (b^i u^D - b^D u^i) + cU B^i = B^i (cF u^D / u^t + cU) - (X / u^t) u^i.
template <int DIR, bool FIRST>
__device__ __forceinline__ void hll_side64(const double pr[NPRIM], const Side64& s, double gam, double kappa,
                                           double cF, double cU, double acc[NFLUX]) {
    const double ud = (DIR == 1) ? s.u1 : ((DIR == 2) ? s.u2 : s.u3);
    const double ptot = (gam - 1.0) * pr[UU] + 0.5 * s.bsq;
    const double w = fma(gam, pr[UU], pr[RHO]) + s.s2;
    const double tu = cF * ud + cU * s.ut;
    const double X = cF * pr[B1 + DIR - 1];
    const double a = w * tu - s.Y * X;
    const double Xi = X * s.iut;
    const double Z = Xi * s.iut + s.Y * tu;
    const double mass = pr[RHO] * tu;
    const double cfp = cF * ptot;
    const double fu = cF * s.iut * ud + cU;
    constexpr int i1 = (DIR == 1) ? 2 : 1, i2 = (DIR == 3) ? 2 : 3;
    const double v1 = (i1 == 1) ? s.u1 : s.u2, v2 = (i2 == 2) ? s.u2 : s.u3;
    double r[NFLUX];
#pragma unroll
    for (int q = 0; q < NFLUX; q++) r[q] = FIRST ? 0.0 : acc[q];
    const double e0 = FIRST ? mass : mass + r[1];
    acc[0] = FIRST ? mass : r[0] + mass;
    acc[1] = a * s.c0 + (-Z * s.k0 + (cU * ptot + e0));
    const double f1 = (DIR == 1) ? (FIRST ? cfp : cfp + r[2]) : r[2];
    const double f2 = (DIR == 2) ? (FIRST ? cfp : cfp + r[3]) : r[3];
    const double f3 = (DIR == 3) ? (FIRST ? cfp : cfp + r[4]) : r[4];
    acc[2] = (FIRST && DIR != 1) ? a * s.c1 - Z * s.k1 : a * s.c1 + (-Z * s.k1 + f1);
    acc[3] = (FIRST && DIR != 2) ? a * s.c2 - Z * s.k2 : a * s.c2 + (-Z * s.k2 + f2);
    acc[4] = (FIRST && DIR != 3) ? a * s.c3 - Z * s.k3 : a * s.c3 + (-Z * s.k3 + f3);
    acc[5] = FIRST ? kappa * mass : kappa * mass + r[5];
    acc[6] = FIRST ? pr[B1 + i1 - 1] * fu - Xi * v1 : pr[B1 + i1 - 1] * fu + (-Xi * v1 + r[6]);
    acc[7] = FIRST ? pr[B1 + i2 - 1] * fu - Xi * v2 : pr[B1 + i2 - 1] * fu + (-Xi * v2 + r[7]);
}

// HLL weights of a face: F = wl F_L + wr F_R - wc (U_R - U_L) with wl + wr = sqrt(-g).
struct Weights64 {
    double wl, wr, wc;
};

// in FP64: the LLF option, and faces whose numbers leave the range of hll_weights_ff. Out of line: rare
// faces (and LLF), whose registers the common path does not carry.
__device__ __noinline__ Weights64 hll_weights_fp64(int riemann, double gam, double gdet, double c00, double c0d,
                                                   double cdd, double rl, double ul, double bl, double utl, double udl,
                                                   double rr, double ur, double br, double utr, double udr) {
    const double gm = gam - 1.0;
    double v[4];
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const double rho = e ? rr : rl, u = e ? ur : ul, bsq = e ? br : bl, ut = e ? utr : utl, ud = e ? udr : udl;
        const double p = gm * u, gp = gam * p, num = bsq + gp, dn = rho + u + p - gp;
        const double A = ut * ut * dn - num * c00, B = ut * ud * dn - num * c0d, C = ud * ud * dn - num * cdd;
        const double sd = root_pos(B * B - A * C), iA = 1.0 / A;
        v[2 * e] = (B + sd) * iA;
        v[2 * e + 1] = (B - sd) * iA;
    }
    const double cmax = max_i(0.0, max_i(v[0], v[2])), cmin = max_i(0.0, max_i(-v[1], -v[3]));
    const double half = 0.5 * gdet;
    Weights64 w;
    if (riemann == HAMR_FLUX_LLF) {
        w.wl = w.wr = half;
        w.wc = half * max_i(cmax, cmin);
    } else if (cmax + cmin > 0.0) {
        const double r = gdet / (cmax + cmin);
        w.wl = cmax * r;
        w.wr = cmin * r;
        w.wc = cmax * w.wr;
    } else {
        w.wl = w.wr = half;
        w.wc = 0.0;
    }
    return w;
}

// The signal speeds of one side in double-float, from the fast-speed quadratic (wave_quadratic); its
// coefficients scale with (rho, u, b^2), so these enter times a power of two, 2^(sh >> 20), that brings the
// largest to [1, 2): the speeds (B +- sd)/A do not change. ok: every factor in binary32's normal range with room
// for the low words of the squares under the root (NaNs fail too), and the root not lost to cancellation.
struct WaveFF {
    ff vp, vm;  // (B +- sd)/A
    float isd;  // 1/(2 sd), sd = sqrt(B^2 - A C)
    int sh;
    bool ok;
};
template <int DIR>
__device__ __forceinline__ WaveFF wave_ff(const PhysArgs& ph, double rho, double u, double bsq, double ut, double ud,
                                          ff c00, ff c0d, ff cdd) {
    WaveFF w;
    w.sh = scale_of(rho, u, bsq);
    const ff R = ff_of(rho, w.sh), U = ff_of(u, w.sh), b = ff_of(bsq, w.sh), t = ff_of(ut), d = ff_of(ud);
    const ff num = ff_add(b, ff_mul(ff{ph.cs2h, ph.cs2l}, U));
    const ff dn = ff_add(R, ff_mul(ff{ph.wmph, ph.wmpl}, U));
    const ff td = ff_mul(t, dn);
    const ff A = ff_sub(ff_mul(td, t), ff_mul(num, c00));
    ff B = ff_mul(td, d);
    if (DIR == 1) B = ff_sub(B, ff_mul(num, c0d));
    const ff C = ff_sub(ff_mul(ff_mul(d, dn), d), ff_mul(num, cdd));
    const ff sd = ff_sqrt_pos(ff_sub(ff_mul(B, B), ff_mul(A, C)));
    const ff iA = ff_rcp(A);
    w.vp = ff_norm(ff_mul(ff_add(B, sd), iA));
    w.vm = ff_norm(ff_mul(ff_sub(B, sd), iA));
    w.isd = 0.5f * rcp_approx(sd.h);
    w.ok = A.h > 1e-12f && A.h < 1e18f && sd.h > 1e-13f && sd.h < 1e18f && sd.h > 4e-6f * fabsf(B.h);
    return w;
}

// One Newton step in FP64 on a double-float root x of the fast-speed quadratic A x^2 - 2 B x + C, written as
// dn (u^t x - u^d)^2 - num (g^tt x^2 - 2 g^td x + g^dd), whose two parts meet at the root without the cancellation
// of B^2 - A C. hi: 1/(the quadratic's slope) up to its sign, +-1/(2 sd).
template <int DIR>
__device__ __forceinline__ double wave_root64(const PhysArgs& ph, double rho, double u, double bsq, double ut,
                                              double ud, double c00, double c0d, double cdd, ff v, float hi, int sh) {
    const double x = ff_d(v);
    const double num = fma(ph.cs2, u, bsq), dn = fma(ph.wmp, u, rho);
    const double w = fma(ut, x, -ud);
    const double g = fma((DIR == 1) ? fma(c00, x, -2.0 * c0d) : c00 * x, x, cdd);
    const double res = fma(dn * w, w, -(num * g));
    return x + widen(ff_of(res, sh).h * hi);
}

// HLL weights: the speeds in double-float on the FP32 pipe, the largest and the smallest then taken to FP64 by a
// Newton step each, the weights in FP64. The double-float speeds alone (2^-46, times the cancellation in
// B^2 - A C) are not enough: a face between dense and thin gas carries their error into the thin cell as many
// times larger as the gas is thinner (17x9x16 torus, one step: utilde^2 8e-13 off, 5e-14 with FP64 weights, 6e-14 here).
// The step leaves what FP64 residuals resolve, no more than the FP64 form's own error, in cold flow less. Which
// side has the larger speed is decided in double-float, which can err only where the two speeds differ by less
// than its error. About 30 FP64 instructions of the 170 a face takes, the FP64 form about 65: a direction of the
// 256x128x64 torus takes 0.66 ms, 0.55 with the weights left in double-float, a pass of two steps 20.4 ms against
// 23.0 with the FP64 form. false where a number leaves the range or the root is lost to cancellation:
// hll_weights_fp64 then.
template <int DIR>
__device__ __forceinline__ bool hll_weights_ff(const PhysArgs& ph, const Metric<double>& m, const double pl[NPRIM],
                                               const Side64& sl, const double pr[NPRIM], const Side64& sr,
                                               Weights64& w) {
    const double cdd = gcondd(m, DIR);
    const ff c00 = ff_of(m.c00), c0d = (DIR == 1) ? ff_of(m.c01) : ff{0.0f, 0.0f}, cddf = ff_of(cdd);
    const double udl = (DIR == 1) ? sl.u1 : ((DIR == 2) ? sl.u2 : sl.u3);
    const double udr = (DIR == 1) ? sr.u1 : ((DIR == 2) ? sr.u2 : sr.u3);
    const WaveFF L = wave_ff<DIR>(ph, pl[RHO], pl[UU], sl.bsq, sl.ut, udl, c00, c0d, cddf);
    const WaveFF R = wave_ff<DIR>(ph, pr[RHO], pr[UU], sr.bsq, sr.ut, udr, c00, c0d, cddf);
    if (!(L.ok && R.ok)) return false;
    auto root = [&](bool right, ff v, float hi, int sh) {
        return wave_root64<DIR>(ph, right ? pr[RHO] : pl[RHO], right ? pr[UU] : pl[UU], right ? sr.bsq : sl.bsq,
                                right ? sr.ut : sl.ut, right ? udr : udl, m.c00, m.c01, cdd, v, hi, sh);
    };
    const bool rp = ff_less(L.vp, R.vp), rm = ff_less(R.vm, L.vm);
    const double vp = root(rp, rp ? R.vp : L.vp, rp ? -R.isd : -L.isd, rp ? R.sh : L.sh);
    const double vm = root(rm, rm ? R.vm : L.vm, rm ? R.isd : L.isd, rm ? R.sh : L.sh);
    const double cmax = max_i(0.0, vp), cmin = max_i(0.0, -vm), sum = cmax + cmin;
    const float s32 = ff_of(sum).h;
    if (!(s32 > 1e-18f && s32 < 1e18f)) return false;
    const double y = widen(rcp_approx(s32)), e = fma(-sum, y, 1.0);  // 1/sum = y (1 + e + e^2 + ...), |e| < 2^-21
    const double r = m.gdet * fma(y, fma(e, e, e), y);
    w.wl = cmax * r;
    w.wr = cmin * r;
    w.wc = cmax * w.wr;
    return true;
}

// HLLE (or LLF) flux in FP64 through every dir-face: faces 0..n_dir, -1..n_e across. Bound by the FP64
// pipe (2 lanes per SM and cycle), so what counts is FP64 instructions per face: the side states
// without b^mu and b_mu, and the weights (30 of the former 65 or so) started on the idle FP32 pipe.
// 256x128x64 torus, one direction: 0.857 ms with the FP64 weights and lowered b^mu, 0.66 ms now; the
// error of a step against 80-bit arithmetic is that of FP64 throughout.
template <int DIR>
__device__ __forceinline__ void b_flux64(const BlockView& v, const PhysArgs& ph, const double* __restrict__ QL,
                                         const double* __restrict__ QR, const double* __restrict__ Bf,
                                         double* __restrict__ F, long t) {
    const int e1 = (DIR == 1) ? v.n1 + 1 : v.n1 + 2;
    const int e2 = (DIR == 2) ? v.n2 + 1 : v.n2 + 2;
    const int e3 = (DIR == 3) ? v.n3 + 1 : v.n3 + 2;
    if (t >= (long)e1 * e2 * e3) return;
    const int i = (int)(t % e1) - (DIR == 1 ? 0 : 1);
    const int j = (int)((t / e1) % e2) - (DIR == 2 ? 0 : 1);
    const int k = (int)(t / ((long)e1 * e2)) - (DIR == 3 ? 0 : 1);
    const long c = cidx(v, i, j, k);
    const long st = (DIR == 1) ? 1 : ((DIR == 2) ? (long)v.n1p : (long)v.n1p * v.n2p);
    Metric<double> m;
    load_metric(face_table<DIR, double>(v), v.n2d, gidx(v, i, j), m);
    if (m.gdet == 0.0) {  // face on the polar axis: no area
#pragma unroll
        for (int q = 0; q < NFLUX; q++) F[q * v.nc + c] = 0.0;
        return;
    }
    double pl[NPRIM], pr[NPRIM];
#pragma unroll
    for (int q = 0; q < NPRIM; q++) {
        if (q == B1 + DIR - 1) continue;
        pl[q] = QR[q * v.nc + c - st];
        pr[q] = QL[q * v.nc + c];
    }
    const double bn = Bf[(DIR - 1) * v.nc + c] * m.igdet;
    pl[B1 + DIR - 1] = bn;
    pr[B1 + DIR - 1] = bn;
    // the entropy tracer's edge values sit in the B^dir fields
    const double kapl = QR[(B1 + DIR - 1) * v.nc + c - st], kapr = QL[(B1 + DIR - 1) * v.nc + c];
    const double ac01 = m.alpha * m.c01;
    Side64 sl, sr;
    side64(pl, m, ac01, sl);
    side64(pr, m, ac01, sr);
    Weights64 w;
    if (ph.riemann == HAMR_FLUX_LLF || !hll_weights_ff<DIR>(ph, m, pl, sl, pr, sr, w))
        w = hll_weights_fp64(ph.riemann, ph.gam, m.gdet, m.c00, gcon0(m, DIR), gcondd(m, DIR), pl[RHO], pl[UU], sl.bsq,
                             sl.ut, (DIR == 1) ? sl.u1 : ((DIR == 2) ? sl.u2 : sl.u3), pr[RHO], pr[UU], sr.bsq, sr.ut,
                             (DIR == 1) ? sr.u1 : ((DIR == 2) ? sr.u2 : sr.u3));
    double acc[NFLUX];
    hll_side64<DIR, true>(pl, sl, ph.gam, kapl, w.wl, w.wc, acc);
    hll_side64<DIR, false>(pr, sr, ph.gam, kapr, w.wr, -w.wc, acc);
#pragma unroll
    for (int q = 0; q < NFLUX; q++) F[q * v.nc + c] = acc[q];
}

// HLLE (or LLF) flux in FP32 (mixed precision).
template <int DIR>
__device__ __forceinline__ void b_flux32(const BlockView& v, const PhysArgs& ph, const float* __restrict__ QL,
                                         const float* __restrict__ QR, const double* __restrict__ Bf,
                                         double* __restrict__ F, long t) {
    using T = float;
    const int nn[4] = {0, v.n1, v.n2, v.n3};
    const int e1 = (DIR == 1) ? nn[1] + 1 : nn[1] + 2;
    const int e2 = (DIR == 2) ? nn[2] + 1 : nn[2] + 2;
    const int e3 = (DIR == 3) ? nn[3] + 1 : nn[3] + 2;
    if (t >= (long)e1 * e2 * e3) return;
    const int i = (int)(t % e1) - (DIR == 1 ? 0 : 1);
    const int j = (int)((t / e1) % e2) - (DIR == 2 ? 0 : 1);
    const int k = (int)(t / ((long)e1 * e2)) - (DIR == 3 ? 0 : 1);
    const long c = cidx(v, i, j, k);
    const long st = (DIR == 1) ? 1 : ((DIR == 2) ? (long)v.n1p : (long)v.n1p * v.n2p);
    Metric<T> m;
    load_metric(face_table<DIR, T>(v), v.n2d, gidx(v, i, j), m);
    // single-block mixed precision: the two field slots (6, 7) also in FP32, after the FP64 fields
    float* F32 = ph.flux32 ? reinterpret_cast<float*>(F + NFLUX * v.nc) : nullptr;
    if (m.gdet == T(0)) {  // face on the polar axis: no area
#pragma unroll
        for (int q = 0; q < NFLUX; q++) F[q * v.nc + c] = 0.0;
        if (F32) F32[c] = F32[v.nc + c] = 0.0f;
        return;
    }
    T pl[NPRIM], pr[NPRIM];
#pragma unroll
    for (int q = 0; q < NPRIM; q++) {
        if (q == B1 + DIR - 1) continue;
        pl[q] = QR[q * v.nc + c - st];
        pr[q] = QL[q * v.nc + c];
    }
    const T bn = (T)Bf[(DIR - 1) * v.nc + c] * m.igdet;
    pl[B1 + DIR - 1] = bn;
    pr[B1 + DIR - 1] = bn;
    // the entropy tracer's edge values sit in the B^dir fields
    const T kapl = QR[(B1 + DIR - 1) * v.nc + c - st], kapr = QL[(B1 + DIR - 1) * v.nc + c];
    const T gam = (T)ph.gam;
    Fluid<T> sl, sr;
    T Al, Bl, sdl, Ar, Br, sdr;
    fluid_state(pl, m, sl);
    wave_quadratic(pl, sl, m, DIR, gam, Al, Bl, sdl);
    fluid_state(pr, m, sr);
    wave_quadratic(pr, sr, m, DIR, gam, Ar, Br, sdr);
    // F sqrt(-g) = wl F_L + wr F_R - wc (U_R - U_L): the weights first, then each side's
    // wl F_L + wc U_L (wr F_R - wc U_R) from its fluid state in one pass (hll_side), which forms no
    // U or F row on its own
    T wl, wr, wc;
    const T half = T(0.5) * m.gdet;
    // the two sides' 1/A from one division
    const T iAA = T(1) / (Al * Ar);
    const T iAl = Ar * iAA, iAr = Al * iAA;
    const T vpl = (Bl + sdl) * iAl, vml = (Bl - sdl) * iAl;
    const T vpr = (Br + sdr) * iAr, vmr = (Br - sdr) * iAr;
    const T cmax = max_i(T(0), max_i(vpl, vpr));
    const T cmin = max_i(T(0), max_i(-vml, -vmr));
    if (ph.riemann == HAMR_FLUX_LLF) {
        wl = wr = half;
        wc = half * max_i(cmax, cmin);
    } else if (cmax + cmin > T(0)) {
        // (cmin F_R + cmax F_L - cmax cmin (U_R - U_L)) sqrt(-g) / (cmax + cmin)
        const T w = m.gdet / (cmax + cmin);
        wl = cmax * w;
        wr = cmin * w;
        wc = cmax * wr;
    } else {
        wl = wr = half;
        wc = T(0);
    }
    T acc[NFLUX];
    hll_side<DIR, true>(pl, sl, gam, kapl, wl, wc, acc);
    hll_side<DIR, false>(pr, sr, gam, kapr, wr, -wc, acc);
#pragma unroll
    for (int q = 0; q < NFLUX; q++) F[q * v.nc + c] = (double)acc[q];
    if (F32) {
        F32[c] = acc[6];
        F32[v.nc + c] = acc[7];
    }
}

template <int DIR, typename T>
__device__ __forceinline__ void b_flux(const BlockView& v, const PhysArgs& ph, const T* __restrict__ QL,
                                       const T* __restrict__ QR, const double* __restrict__ Bf, double* __restrict__ F,
                                       long t) {
    if constexpr (std::is_same<T, double>::value)
        b_flux64<DIR>(v, ph, QL, QR, Bf, F, t);
    else
        b_flux32<DIR>(v, ph, QL, QR, Bf, F, t);
}

template <int DIR, typename T>
__global__ void __launch_bounds__(256, 2) k_flux(BlockView v, PhysArgs ph, const T* __restrict__ QL,
                                             const T* __restrict__ QR, const double* __restrict__ Bf,
                                             double* __restrict__ F) {
    b_flux<DIR, T>(v, ph, QL, QR, Bf, F, (long)blockIdx.x * blockDim.x + threadIdx.x);
}


// ---------------------------------------------------------------- EMFs
// edge EMFs as the average of the 4 neighbouring face fluxes of B (Sec. 2.5).
// E1 and E3 on the polar axis are 0. With T = float (mixed precision) the
// average is formed in FP32; every face shares the one stored edge value, so
// the FP64 curl in the CT update still keeps div B at FP64 roundoff.
//
// Upwinded EMFs (Ec != nullptr; Gardiner & Stone 2005, the paper's usual
// setting): for an edge between face directions p and q, with e_p / e_q the
// EMF values the p- / q-faces carry and Ec the EMF of the cell-centred state,
//   E = average + 1/4 [D_q(q-3/4) - D_q(q-1/4)] + 1/4 [D_p(p-3/4) - D_p(p-1/4)],
//   D_q(q-1/4) = Ec(c, q) - e_q(c, q-1/2), D_q(q-3/4) = e_q(c, q-1/2) - Ec(c, q-1),
// in the cell column c (p-1 or p) upwind of the mass flux through the p-face
// beside the edge (both averaged when it is zero); D_p likewise.

// the cell-centred EMFs sqrt(-g)(b^2 u^3 - b^3 u^2, b^3 u^1 - b^1 u^3, b^1 u^2 - b^2 u^1)
// of every cell -1..n of the block, from the stage state (centre B in slots 5..7)
__device__ __forceinline__ void b_cell_emf(const BlockView& v, const double* __restrict__ P, double* __restrict__ Ec,
                                           long t) {
    const int e1 = v.n1 + 2, e2 = v.n2 + 2, e3 = v.n3 + 2;
    if (t >= (long)e1 * e2 * e3) return;
    const int i = (int)(t % e1) - 1, j = (int)((t / e1) % e2) - 1, k = (int)(t / ((long)e1 * e2)) - 1;
    const long c = cidx(v, i, j, k);
    Metric<double> m;
    load_metric(v.gc, v.n2d, gidx(v, i, j), m);
    double pr[NPRIM];
#pragma unroll
    for (int q = 0; q < NPRIM; q++) pr[q] = P[q * v.nc + c];
    Fluid<double> s;
    fluid_state(pr, m, s);
    Ec[c] = (s.bcon[2] * s.ucon[3] - s.bcon[3] * s.ucon[2]) * m.gdet;
    Ec[v.nc + c] = (s.bcon[3] * s.ucon[1] - s.bcon[1] * s.ucon[3]) * m.gdet;
    Ec[2 * v.nc + c] = (s.bcon[1] * s.ucon[2] - s.bcon[2] * s.ucon[1]) * m.gdet;
}

__global__ void k_cell_emf(BlockView v, const double* __restrict__ P, double* __restrict__ Ec) {
    b_cell_emf(v, P, Ec, (long)blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename T>
__device__ __forceinline__ T upwind_pick(T mass_flux, T lower, T upper) {
    return mass_flux > T(0) ? lower : (mass_flux < T(0) ? upper : T(0.5) * (lower + upper));
}

// the Gardiner-Stone corrections of one edge. Offsets are cells along p and q from the
// edge's cell c: sp, sq the index strides of p and q; Fp / Fq the flux arrays of the p / q
// faces, slp / slq their B-flux slots with signs gp / gq (the EMF a face carries is g F[sl]);
// ec the cell-EMF field of the component
// field slot `slot` (6 or 7) of a face flux at cell offset i as T: the FP64 field converted, or (F32)
// the FP32 copy of slots 6 and 7 kept after the FP64 fields
template <typename T, bool F32>
__device__ __forceinline__ T ld_bflux(const double* __restrict__ F, int slot, long nc, long i) {
    if constexpr (F32) {
        static_assert(std::is_same<T, float>::value, "the FP32 slot copy serves the FP32 EMFs");
        return reinterpret_cast<const float*>(F + NFLUX * nc)[(slot - 6) * nc + i];
    } else {
        return (T)F[slot * nc + i];
    }
}

template <typename T>
__device__ __forceinline__ T gs_correction(long c, long sp, long sq, long nc, const double* __restrict__ Fp,
                                           const double* __restrict__ Fq, int slp, int slq, T gp, T gq,
                                           const double* __restrict__ ec) {
    auto ep = [&](long o) { return gp * (T)Fp[slp * nc + c + o]; };  // p-face value at cell offset o
    auto eq = [&](long o) { return gq * (T)Fq[slq * nc + c + o]; };
    auto E = [&](long o) { return (T)ec[c + o]; };
    auto mp = [&](long o) { return (T)Fp[c + o]; };  // mass flux (slot 0) through a p-face
    auto mq = [&](long o) { return (T)Fq[c + o]; };
    const T dq_lo = upwind_pick(mp(-sq), eq(-sp) - E(-sp - sq), eq(0) - E(-sq));  // D_q(q-3/4)
    const T dq_hi = upwind_pick(mp(0), E(-sp) - eq(-sp), E(0) - eq(0));           // D_q(q-1/4)
    const T dp_lo = upwind_pick(mq(-sp), ep(-sq) - E(-sp - sq), ep(0) - E(-sp));  // D_p(p-3/4)
    const T dp_hi = upwind_pick(mq(0), E(-sq) - ep(-sq), E(0) - ep(0));           // D_p(p-1/4)
    return T(0.25) * (dq_lo - dq_hi) + T(0.25) * (dp_lo - dp_hi);
}

template <typename T, bool F32 = false>
__device__ __forceinline__ void b_emf(const BlockView& v, const double* __restrict__ F1, const double* __restrict__ F2,
                      const double* __restrict__ F3, double* __restrict__ E, const double* __restrict__ Ec, long t) {
    const int e1 = v.n1 + 1, e2 = v.n2 + 1, e3 = v.n3 + 1;
    if (t >= (long)e1 * e2 * e3) return;
    const int i = (int)(t % e1), j = (int)((t / e1) % e2), k = (int)(t / ((long)e1 * e2));
    const long c = cidx(v, i, j, k);
    const long si = 1, sj = v.n1p, sk = (long)v.n1p * v.n2p, nc = v.nc;
    const bool axis = (v.bc[2] == HAMR_BC_POLAR && j == 0) || (v.bc[3] == HAMR_BC_POLAR && j == v.n2);
    const T q = T(0.25);
    // flux slots: F1 -> (B2: 6, B3: 7), F2 -> (B1: 6, B3: 7), F3 -> (B1: 6, B2: 7)
    if (i < v.n1) {
        T x = q * (ld_bflux<T, F32>(F3, 7, nc, c) + ld_bflux<T, F32>(F3, 7, nc, c - sj) -
                   ld_bflux<T, F32>(F2, 7, nc, c - sk) - ld_bflux<T, F32>(F2, 7, nc, c));
        // p = x2 faces (value -F2(B3)), q = x3 faces (value F3(B2))
        if (Ec) x += gs_correction<T>(c, sj, sk, nc, F2, F3, 7, 7, T(-1), T(1), Ec);
        E[c] = axis ? 0.0 : (double)x;
    }
    if (j < v.n2) {
        T x = q * (ld_bflux<T, F32>(F1, 7, nc, c - sk) + ld_bflux<T, F32>(F1, 7, nc, c) -
                   ld_bflux<T, F32>(F3, 6, nc, c) - ld_bflux<T, F32>(F3, 6, nc, c - si));
        // p = x1 faces (value F1(B3)), q = x3 faces (value -F3(B1))
        if (Ec) x += gs_correction<T>(c, si, sk, nc, F1, F3, 7, 6, T(1), T(-1), Ec + nc);
        E[nc + c] = (double)x;
    }
    if (k < v.n3) {
        T x = q * (ld_bflux<T, F32>(F2, 6, nc, c - si) + ld_bflux<T, F32>(F2, 6, nc, c) -
                   ld_bflux<T, F32>(F1, 6, nc, c) - ld_bflux<T, F32>(F1, 6, nc, c - sj));
        // p = x1 faces (value -F1(B2)), q = x2 faces (value F2(B1))
        if (Ec) x += gs_correction<T>(c, si, sj, nc, F1, F2, 6, 6, T(-1), T(1), Ec + 2 * nc);
        E[2 * nc + c] = axis ? 0.0 : (double)x;
    }
}

template <typename T, bool F32 = false>
__global__ void k_emf(BlockView v, const double* __restrict__ F1, const double* __restrict__ F2,
                      const double* __restrict__ F3, double* __restrict__ E, const double* __restrict__ Ec) {
    b_emf<T, F32>(v, F1, F2, F3, E, Ec, (long)blockIdx.x * blockDim.x + threadIdx.x);
}


// ---------------------------------------------------------------- CT
// staggered face update Bbar += dt curl E (Sec. 2.5, the three CT equations)
__device__ __forceinline__ void b_ct(const BlockView& v, const double* __restrict__ E, const double* Bb, double* Bo,
                     const double* __restrict__ dscal, double fac, long t) {
    const int e1 = v.n1 + 1, e2 = v.n2 + 1, e3 = v.n3 + 1;
    if (t >= (long)e1 * e2 * e3) return;
    const int i = (int)(t % e1), j = (int)((t / e1) % e2), k = (int)(t / ((long)e1 * e2));
    const long c = cidx(v, i, j, k);
    const long sj = v.n1p, sk = (long)v.n1p * v.n2p, nc = v.nc;
    const double dt = dscal[0] * fac;
    const double* E1 = E;
    const double* E2 = E + nc;
    const double* E3 = E + 2 * nc;
    if (j < v.n2 && k < v.n3) {
        const double r = (E2[c + sk] - E2[c]) * v.idx3 - (E3[c + sj] - E3[c]) * v.idx2;
        Bo[c] = Bb[c] + dt * r;
    }
    if (i < v.n1 && k < v.n3) {
        const bool axis = (v.bc[2] == HAMR_BC_POLAR && j == 0) || (v.bc[3] == HAMR_BC_POLAR && j == v.n2);
        const double r = (E3[c + 1] - E3[c]) * v.idx1 - (E1[c + sk] - E1[c]) * v.idx3;
        Bo[nc + c] = axis ? 0.0 : Bb[nc + c] + dt * r;
    }
    if (i < v.n1 && j < v.n2) {
        const double r = (E1[c + sj] - E1[c]) * v.idx2 - (E2[c + 1] - E2[c]) * v.idx1;
        Bo[2 * nc + c] = Bb[2 * nc + c] + dt * r;
    }
}

__global__ void k_ct(BlockView v, const double* __restrict__ E, const double* Bb, double* Bo,
                     const double* __restrict__ dscal, double fac) {
    b_ct(v, E, Bb, Bo, dscal, fac, (long)blockIdx.x * blockDim.x + threadIdx.x);
}


// largest CFL rate of the block's cells. The FP64 rate of a cell is formed only where its FP32 estimate is
// not certainly below the largest rate found so far (rate_below): in a spherical block nearly every cell is
// (the largest rates sit next to the axis at the inner edge), and the result is the same bits.
__device__ __forceinline__ double cell_rate(const BlockView& v, const PhysArgs& ph, int i, int j, const double pr[NPRIM],
                                            const unsigned long long* dmax) {
    Metric<double> m;
    load_metric(v.gc, v.n2d, gidx(v, i, j), m);
    const int w = smr_width(v, ph, j);
    BlockView vw = v;
    if (w > 1) vw.idx3 = v.idx3 / w;  // an internal-SMR group: its width in x3
    // the estimate's fluid state in FP32, (rho, u, B^2) scaled to O(1) by 2^sh, sh even
    const int sh = scale_of(pr[RHO], pr[UU], 0.0) & ~0x100000;
    Metric<float> mf;
    mf.g01 = narrow(m.g01), mf.g03 = narrow(m.g03), mf.g11 = narrow(m.g11), mf.g13 = narrow(m.g13);
    mf.g22 = narrow(m.g22), mf.g33 = narrow(m.g33);
    const float q1 = narrow(pr[U1]), q2 = narrow(pr[U2]), q3 = narrow(pr[U3]);
    const float u1 = mf.g11 * q1 + mf.g13 * q3, u2 = mf.g22 * q2, u3 = mf.g13 * q1 + mf.g33 * q3;
    const float g2 = 1.0f + q1 * u1 + q2 * u2 + q3 * u3, gamma = sqrtf(g2);
    const float al = narrow(m.alpha), c01 = narrow(m.c01);
    const float b1 = ff_of(pr[B1], sh / 2).h, b2 = ff_of(pr[B2], sh / 2).h, b3 = ff_of(pr[B3], sh / 2).h;
    const float bt = b1 * u1 + b2 * u2 + b3 * u3;
    const float bb = mf.g11 * b1 * b1 + mf.g22 * b2 * b2 + mf.g33 * b3 * b3 + 2.0f * mf.g13 * b1 * b3;
    const float bsq = al * al * (bb + bt * bt) / g2;
    const float ud[3] = {q1 - gamma * al * c01, q2, q3};
    const float est = rate_estimate(vw, ph, ff_of(pr[RHO], sh).h, ff_of(pr[UU], sh).h, bsq, gamma / al, ud,
                                    narrow(m.c00), c01, narrow(m.c11), narrow(m.c22), narrow(m.c33));
    return rate_below(est, dmax) ? 0.0 : inv_dt_cell(vw, pr, m, ph.gam);
}

__device__ __forceinline__ void b_dt_reduce(const BlockView& v, const PhysArgs& ph, const double* __restrict__ P,
                                            unsigned long long* dmax, long t) {
    double inv = 0.0;
    if (t < (long)v.n1 * v.n2 * v.n3) {
        const int i = (int)(t % v.n1), j = (int)((t / v.n1) % v.n2), k = (int)(t / ((long)v.n1 * v.n2));
        const long c = cidx(v, i, j, k);
        double pr[NPRIM];
#pragma unroll
        for (int q = 0; q < NPRIM; q++) pr[q] = P[q * v.nc + c];
        inv = cell_rate(v, ph, i, j, pr, dmax);
    }
    reduce_rate(inv, dmax);
}

__global__ void k_dt_reduce(BlockView v, PhysArgs ph, const double* __restrict__ P, unsigned long long* dmax) {
    b_dt_reduce(v, ph, P, dmax, (long)blockIdx.x * blockDim.x + threadIdx.x);
}

// A state load from device memory in one pass over the padded block: prim and bface (field stride n) into
// P and B (and, in a block tree, into the old state Po and Bo), the centre field of interior cells from the
// faces, the CFL rate. It replaces 11 copies (13 in a tree), the centre-field pass and the rate's pass over
// memory: per block of the 512-block tree 15 operations became 2, the tree's load and read-out 61 -> 10 ms.
__global__ void k_load(BlockView v, PhysArgs ph, const double* __restrict__ prim, const double* __restrict__ bface,
                       double* __restrict__ P, double* __restrict__ B, double* __restrict__ Po, double* __restrict__ Bo,
                       unsigned long long* dmax) {
    const long n = (long)v.n1p * v.n2p * v.n3p;
    const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
    double inv = 0.0;
    if (c < n) {
        const int i = (int)(c % v.n1p) - NG, j = (int)((c / v.n1p) % v.n2p) - NG;
        const int k = (int)(c / ((long)v.n1p * v.n2p)) - NG;
        const bool in = i >= 0 && i < v.n1 && j >= 0 && j < v.n2 && k >= 0 && k < v.n3;
        double pr[NPRIM];
#pragma unroll
        for (int q = 0; q < NPRIM; q++) pr[q] = (in && q >= B1) ? 0.0 : prim[q * n + c];
        if (in) {
            centre_field_at(v, bface, n, c, v.gc[G_IGDET * v.n2d + gidx(v, i, j)], pr + B1);
            inv = cell_rate(v, ph, i, j, pr, dmax);
        }
#pragma unroll
        for (int q = 0; q < NPRIM; q++) {
            P[q * v.nc + c] = pr[q];
            if (Po) Po[q * v.nc + c] = pr[q];
        }
#pragma unroll
        for (int q = 0; q < 3; q++) {
            const double b = bface[q * n + c];
            B[q * v.nc + c] = b;
            if (Bo) Bo[q * v.nc + c] = b;
        }
    }
    reduce_rate(inv, dmax);
}

// the state out, in the caller's field stride n; prim or bface may be null
__global__ void k_store(BlockView v, const double* __restrict__ P, const double* __restrict__ B,
                        double* __restrict__ prim, double* __restrict__ bface) {
    const long n = (long)v.n1p * v.n2p * v.n3p;
    const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    double x[NPRIM + 3];
    if (prim)
#pragma unroll
        for (int q = 0; q < NPRIM; q++) x[q] = P[q * v.nc + c];
    if (bface)
#pragma unroll
        for (int q = 0; q < 3; q++) x[NPRIM + q] = B[q * v.nc + c];
    if (prim)
#pragma unroll
        for (int q = 0; q < NPRIM; q++) prim[q * n + c] = x[q];
    if (bface)
#pragma unroll
        for (int q = 0; q < 3; q++) bface[q * n + c] = x[NPRIM + q];
}


// dt of this step: the caller's, or C0 / max rate of the current state;
// resets the accumulators of the new step.
__global__ void k_dt_select(double cour, double user_dt, double* dscal, unsigned long long* dmax,
                            unsigned long long* dcnt) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const double mx = __longlong_as_double((long long)dmax[0]);
    dscal[0] = (user_dt > 0.0) ? user_dt : cour / mx;
    dmax[0] = 0ull;
    dcnt[0] = dcnt[1] = dcnt[2] = dcnt[3] = dcnt[4] = 0ull;
}

// ---------------------------------------------------------------- batched (multi-block) wrappers
// blockIdx.y selects the block list[blockIdx.y] of the table; blockIdx.x and
// threadIdx.x index the work inside it exactly as in the single-block kernels.

// kappa goes to field 0 of the EMF array (free until the EMFs), the flattening
// coefficients of dir to field 0 of the dir-flux array
template <int DIR, typename T, int M>
__global__ void kb_recon(const DevBlock* tab, const int* list, PhysArgs ph, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    const double* Fl = (DIR == 1) ? D.F1 : ((DIR == 2) ? D.F2 : D.F3);
    if constexpr (std::is_same<T, double>::value)
        b_recon<DIR, T, M>(D.v, ph, sigma ? D.Ph : D.P, D.E, Fl, D.QL, D.QR, tidx());
    else  // the FP32 copy holds the stage's state
        b_recon<DIR, T, M>(D.v, ph, D.P32, reinterpret_cast<const float*>(D.E), reinterpret_cast<const float*>(Fl),
                        reinterpret_cast<float*>(D.QL), reinterpret_cast<float*>(D.QR), tidx());
}

template <int DIR, typename T>
__global__ void kb_flatten(const DevBlock* tab, const int* list, PhysArgs ph, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    double* Fl = (DIR == 1) ? D.F1 : ((DIR == 2) ? D.F2 : D.F3);
    if constexpr (std::is_same<T, double>::value)
        b_flatten<DIR, T>(D.v, ph, sigma ? D.Ph : D.P, Fl, tidx());
    else
        b_flatten<DIR, T>(D.v, ph, D.P32, reinterpret_cast<float*>(Fl), tidx());
}

template <typename T>
__global__ void kb_kappa(const DevBlock* tab, const int* list, PhysArgs ph, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    if constexpr (std::is_same<T, double>::value)
        b_kappa<T>(D.v, ph.gam, sigma ? D.Ph : D.P, D.E, tidx(), sigma ? nullptr : D.Un + (long)C_ENT * D.v.nc);
    else
        b_kappa<T>(D.v, (float)ph.gam, D.P32, reinterpret_cast<float*>(D.E), tidx(),
                   sigma ? nullptr : D.Un + (long)C_ENT * D.v.nc);
}

__global__ void kb_to_f32(const DevBlock* tab, const int* list, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    b_to_f32(D.v, sigma ? D.Ph : D.P, D.P32, tidx());
}

template <int DIR, typename T>
__global__ void __launch_bounds__(256, 2) kb_flux(const DevBlock* tab, const int* list, PhysArgs ph, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    double* F = (DIR == 1) ? D.F1 : ((DIR == 2) ? D.F2 : D.F3);
    b_flux<DIR, T>(D.v, ph, reinterpret_cast<const T*>(D.QL), reinterpret_cast<const T*>(D.QR), sigma ? D.Bh : D.B, F,
                   tidx());
}

template <typename T, bool F32 = false>
__global__ void kb_emf(const DevBlock* tab, const int* list, int upwind) {
    const DevBlock& D = tab[list[blockIdx.y]];
    b_emf<T, F32>(D.v, D.F1, D.F2, D.F3, D.E, upwind ? D.QL : nullptr, tidx());
}

// cell EMFs of the stage state into the edge-value scratch (free once the fluxes exist)
__global__ void kb_cell_emf(const DevBlock* tab, const int* list, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    b_cell_emf(D.v, sigma ? D.Ph : D.P, D.QL, tidx());
}

__global__ void kb_ct(const DevBlock* tab, const int* list, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    if (sigma == 0)
        b_ct(D.v, D.E, D.B, D.Bh, D.dscal, 0.5, tidx());
    else if (sigma == 1)
        b_ct(D.v, D.E, D.B, D.B, D.dscal, 1.0, tidx());
    else
        b_ct(D.v, D.E, D.B, D.B, D.dscal + 1, 1.0, tidx());
}

__global__ void kb_dt_reduce(const DevBlock* tab, const int* list, PhysArgs ph) {
    const DevBlock& D = tab[list[blockIdx.y]];
    b_dt_reduce(D.v, ph, D.P, D.dmax, tidx());
}

// state at the start of a step (the source of finer neighbours' time interpolation), status reset
__global__ void kb_save_old(const DevBlock* tab, const int* list) {
    const DevBlock& D = tab[list[blockIdx.y]];
    const long t = tidx();
    const long n = (long)D.v.n1p * D.v.n2p * D.v.n3p;
    if (t >= n) return;
#pragma unroll
    for (int q = 0; q < NPRIM; q++) D.Pold[q * D.v.nc + t] = D.P[q * D.v.nc + t];
#pragma unroll
    for (int q = 0; q < 3; q++) D.Bold[q * D.v.nc + t] = D.B[q * D.v.nc + t];
    D.status[t] = 0;
}

// refluxed cells: U(P) with the field before the correction, plus the flux corrections
__global__ void k_reflux_u0(const DevBlock* tab, int n, const int* cblk, const long* cix, const int* nrec,
                            const int* recs, const double* rec_dU, int nrec_tot, double* Ucorr, PhysArgs ph) {
    const long i = tidx();
    if (i >= n) return;
    const DevBlock& D = tab[cblk[i]];
    const BlockView& v = D.v;
    const long c = cix[i];
    const long ip = c % v.n1p, jp = (c / v.n1p) % v.n2p;
    Metric<double> m;
    load_metric(v.gc, v.n2d, jp * v.n1p + ip, m);
    double pr[NPRIM];
#pragma unroll
    for (int q = 0; q < NPRIM; q++) pr[q] = D.P[q * v.nc + c];
    Fluid<double> s;
    fluid_state(pr, m, s);
    double row[NFLUX];
    flux_row(pr, s, 0, 1, ph.gam, entropy_kappa(pr, ph.gam), row);
    for (int q = 0; q < NCONS; q++) {
        double du = 0.0;
        for (int r = 0; r < nrec[i]; r++) du += rec_dU[(long)q * nrec_tot + recs[3 * i + r]];
        Ucorr[(long)q * n + i] = row[q] * m.gdet + du;
    }
}

// inversion of the refluxed cells with the corrected field; floors. Ucorr: stride `stride` per field
__global__ void k_reflux_cells(const DevBlock* tab, int n, const int* cblk, const long* cix, const double* Ucorr,
                               long stride, PhysArgs ph) {
    const long i = tidx();
    if (i >= n) return;
    const DevBlock& D = tab[cblk[i]];
    const BlockView& v = D.v;
    const long c = cix[i];
    const int ii = (int)(c % v.n1p) - NG, jj = (int)((c / v.n1p) % v.n2p) - NG, kk = (int)(c / ((long)v.n1p * v.n2p)) - NG;
    const long g = gidx(v, ii, jj);
    Metric<double> m;
    load_metric(v.gc, v.n2d, g, m);
    double U[NCONS];
    for (int q = 0; q < NCONS; q++) U[q] = Ucorr[(long)q * stride + i];
    double Bc[3];
    centre_field(v, D.B, ii, jj, kk, m.igdet, Bc);
    double pr[NPRIM];
#pragma unroll
    for (int q = 0; q < NPRIM; q++) pr[q] = D.P[q * v.nc + c];
    pr[B1] = Bc[0];
    pr[B2] = Bc[1];
    pr[B3] = Bc[2];
    int its;
    const int st = invert(U, Bc, m, ph.gam, pr, &its, false, nullptr, ph.inversion,
                          ph.mixed ? C2P_NEWTON64 : C2P_NEWTON_FF);
    if (st == INV_FAIL)
#pragma unroll
        for (int q = 0; q < 5; q++) pr[q] = D.P[q * v.nc + c];
    int fl = 0;
    if (ph.floors) {
        Fluid<double> s;
        fluid_state(pr, m, s);
        fl = cell_floors(v, g, m, ph, pr, s);
    }
#pragma unroll
    for (int q = 0; q < NPRIM; q++) D.P[q * v.nc + c] = pr[q];
    atomicAdd(&D.dcnt[st == INV_OK ? 0 : (st == INV_ENTROPY ? 1 : 2)], 1ull);
    if (fl) atomicAdd(&D.dcnt[3], 1ull);
}

// refluxed internal-SMR groups (its w cells consecutive in the list from position first[g]): the mean
// of the cells' corrected states inverted once with the mean corrected centre field, from the mean
// primitives; every cell takes the result and keeps its own centre field; floors
__global__ void k_reflux_groups(const DevBlock* tab, int ngrp, const int* first, const int* gw, const int* cblk,
                                const long* cix, const double* Ucorr, long stride, PhysArgs ph) {
    const long t = tidx();
    if (t >= ngrp) return;
    const int f = first[t], w = gw[t];
    const DevBlock& D = tab[cblk[f]];
    const BlockView& v = D.v;
    const long c0 = cix[f];
    const int ii = (int)(c0 % v.n1p) - NG, jj = (int)((c0 / v.n1p) % v.n2p) - NG;
    const int k0 = (int)(c0 / ((long)v.n1p * v.n2p)) - NG;
    const long g = gidx(v, ii, jj);
    Metric<double> m;
    load_metric(v.gc, v.n2d, g, m);
    double U[NCONS], Bc[3] = {0.0, 0.0, 0.0}, pr[NPRIM];
#pragma unroll
    for (int q = 0; q < NCONS; q++) U[q] = 0.0;
#pragma unroll
    for (int q = 0; q < NPRIM; q++) pr[q] = 0.0;
    for (int a = 0; a < w; a++) {
        const long c = cix[f + a];
#pragma unroll
        for (int q = 0; q < NCONS; q++) U[q] += Ucorr[(long)q * stride + f + a];
        double b[3];
        centre_field(v, D.B, ii, jj, k0 + a, m.igdet, b);
        for (int e = 0; e < 3; e++) Bc[e] += b[e];
#pragma unroll
        for (int q = 0; q < 5; q++) pr[q] += D.P[q * v.nc + c];
    }
#pragma unroll
    for (int q = 0; q < NCONS; q++) U[q] /= w;
    for (int e = 0; e < 3; e++) Bc[e] /= w;
#pragma unroll
    for (int q = 0; q < 5; q++) pr[q] /= w;
    double p0[5];
#pragma unroll
    for (int q = 0; q < 5; q++) p0[q] = pr[q];
    pr[B1] = Bc[0];
    pr[B2] = Bc[1];
    pr[B3] = Bc[2];
    int its;
    const int st = invert(U, Bc, m, ph.gam, pr, &its, false, nullptr, ph.inversion,
                          ph.mixed ? C2P_NEWTON64 : C2P_NEWTON_FF);
    if (st == INV_FAIL)
#pragma unroll
        for (int q = 0; q < 5; q++) pr[q] = p0[q];
    int fl = 0;
    if (ph.floors) {
        Fluid<double> s;
        fluid_state(pr, m, s);
        fl = cell_floors(v, g, m, ph, pr, s);
    }
    for (int a = 0; a < w; a++) {
        const long c = cix[f + a];
        double b[3];
        centre_field(v, D.B, ii, jj, k0 + a, m.igdet, b);
#pragma unroll
        for (int q = 0; q < 5; q++) D.P[q * v.nc + c] = pr[q];
        for (int e = 0; e < 3; e++) D.P[(B1 + e) * v.nc + c] = b[e];
    }
    atomicAdd(&D.dcnt[st == INV_OK ? 0 : (st == INV_ENTROPY ? 1 : 2)], (unsigned long long)w);
    if (fl) atomicAdd(&D.dcnt[3], (unsigned long long)w);
}

// ---------------------------------------------------------------- internal SMR
// Rows next to a polar face grouped into cells smr_width wide in x3 (Sec. 3.3.2:
// a group's fluxes and conserved state are averaged). The field: before CT, along
// each x2-line of edges with group width W (that of the adjacent row closer to the
// pole) the E3 of a group take their mean and the inner E1 are linear between the
// group's outer ones; inside each grouped row the inner E2 are linear between the
// group's outer ones. The changes of a group's x1- and x2-faces are then uniform
// and those of its inner x3-faces linear (a wide cell's), and CT keeps div B. The
// cells: after the cell update (which leaves the group's conserved states in the
// scratch U) the group's mean state is inverted once with the mean centre field,
// from the mean primitives, and every cell takes the result (its own centre field
// kept); the CFL rate uses the group's width.
__device__ __forceinline__ int smr_line_width(const BlockView& v, const PhysArgs& ph, int je) {
    int w = 1;
    if (je >= 1) w = max(w, smr_width(v, ph, je - 1));
    if (je < v.n2) w = max(w, smr_width(v, ph, je));
    return w;
}

// sum of w = 2^n values as a balanced binary tree (w equal values sum to exactly w times the
// value): element m closes the subtrees its trailing one bits end
__device__ __forceinline__ double pair_sum_strided(const double* __restrict__ a, long stride, int w) {
    double st[12];
    for (int m = 0; m < w; m++) {
        double t = a[m * stride];
        int l = 0;
        while ((m >> l) & 1) {
            t = st[l] + t;
            l++;
        }
        st[l] = t;
    }
    return st[__ffs(w) - 1];
}

// Threads: i in [0, n1], q over the nr + 1 edge lines and nr rows next to each polar face
// (lines je = 0..nr and n2 - nr..n2, a line counted once when n2 = 2 nr), gi over the groups.
__device__ __forceinline__ void b_smr_emf(const BlockView& v, const PhysArgs& ph, double* __restrict__ E, long t) {
    const int nr = smr_rows(v, ph);
    const int ng = v.n3 / 2;
    const int nq = 2 * (nr + 1);
    if (nr == 0 || t >= (long)(v.n1 + 1) * nq * ng) return;
    const int i = (int)(t % (v.n1 + 1));
    const int q = (int)((t / (v.n1 + 1)) % nq);
    const int gi = (int)(t / ((long)(v.n1 + 1) * nq));
    const long sk = (long)v.n1p * v.n2p;
    double* E1 = E;
    double* E2 = E + v.nc;
    double* E3 = E + 2 * v.nc;
    // the edge line: lower side je = q, upper side je = n2 - 2 nr - 1 + q
    const bool upper = q > nr;
    const int je = upper ? v.n2 - 2 * nr - 1 + q : q;
    const int W = (upper && je <= nr) ? 1 : smr_line_width(v, ph, je);
    if (W > 1 && gi < v.n3 / W) {
        const int k0 = gi * W;
        const long c0 = cidx(v, i, je, k0);
        const double s3 = pair_sum_strided(E3 + c0, sk, W);
        for (int m = 0; m < W; m++) E3[c0 + m * sk] = s3 / W;
        if (i < v.n1) {
            const double e0 = E1[c0], ew = E1[c0 + W * sk];
            for (int m = 1; m < W; m++) E1[c0 + m * sk] = e0 + (ew - e0) * m / W;
        }
    }
    // the row: lower side j = q (q < nr), upper side j = n2 - 2 nr - 1 + q (nr < q <= 2 nr)
    const int j = (q < nr) ? q : ((q > nr && q <= 2 * nr) ? v.n2 - 2 * nr - 1 + q : -1);
    if (j < 0) return;
    const int w = smr_width(v, ph, j);
    if (w > 1 && gi < v.n3 / w) {
        const int k0 = gi * w;
        const long c0 = cidx(v, i, j, k0);
        const double e0 = E2[c0], ew = E2[c0 + w * sk];
        for (int m = 1; m < w; m++) E2[c0 + m * sk] = e0 + (ew - e0) * m / w;
    }
}

// the grouped row of cell-thread row r: rows [0, nr) and [n2 - nr, n2), nr = smr_rows
__device__ __forceinline__ int smr_row(const BlockView& v, const PhysArgs& ph, int r) {
    const int nr = smr_rows(v, ph);
    return (r < nr) ? r : v.n2 - 2 * nr + r;
}

__device__ __forceinline__ void b_smr_cells(const BlockView& v, const PhysArgs& ph, int corrector,
                                            const double* __restrict__ Pf, const double* __restrict__ Bn,
                                            const double* __restrict__ Us, double* Po, uint8_t* __restrict__ status,
                                            unsigned long long* dmax, unsigned long long* dcnt, long t) {
    const int nr = smr_rows(v, ph);
    const int ng = v.n3 / 2;
    if (nr == 0 || t >= (long)v.n1 * 2 * nr * ng) return;
    const int i = (int)(t % v.n1);
    const int r = (int)((t / v.n1) % (2 * nr));
    const int gi = (int)(t / ((long)v.n1 * 2 * nr));
    const int j = smr_row(v, ph, r);
    const int w = smr_width(v, ph, j);
    if (w == 1 || gi >= v.n3 / w) return;
    const int k0 = gi * w;
    const long g = gidx(v, i, j);
    Metric<double> m;
    load_metric(v.gc, v.n2d, g, m);
    double U[NCONS], Bc[3] = {0.0, 0.0, 0.0}, pr[NPRIM];
#pragma unroll
    for (int q = 0; q < NCONS; q++) U[q] = 0.0;
#pragma unroll
    for (int q = 0; q < NPRIM; q++) pr[q] = 0.0;
    for (int a = 0; a < w; a++) {
        const long c = cidx(v, i, j, k0 + a);
#pragma unroll
        for (int q = 0; q < NCONS; q++) U[q] += Us[q * v.nc + c];
        double b[3];
        centre_field(v, Bn, i, j, k0 + a, m.igdet, b);
        for (int e = 0; e < 3; e++) Bc[e] += b[e];
#pragma unroll
        for (int q = 0; q < 5; q++) pr[q] += Pf[q * v.nc + c];
    }
#pragma unroll
    for (int q = 0; q < NCONS; q++) U[q] /= w;
    for (int e = 0; e < 3; e++) Bc[e] /= w;
#pragma unroll
    for (int q = 0; q < 5; q++) pr[q] /= w;
    double pf[5];
#pragma unroll
    for (int q = 0; q < 5; q++) pf[q] = pr[q];
    pr[B1] = Bc[0];
    pr[B2] = Bc[1];
    pr[B3] = Bc[2];
    int its = 0;
    const int st = invert(U, Bc, m, ph.gam, pr, &its, false, nullptr, ph.inversion,
                          ph.mixed ? C2P_NEWTON64 : C2P_NEWTON_FF);
    if (st == INV_FAIL)
#pragma unroll
        for (int q = 0; q < 5; q++) pr[q] = pf[q];
    Fluid<double> s;
    fluid_state(pr, m, s);
    const int fl = ph.floors ? cell_floors(v, g, m, ph, pr, s) : 0;
    const uint8_t sb = ((st == INV_ENTROPY) ? ST_ENTROPY : ((st == INV_FAIL) ? ST_FAIL : 0)) | (fl ? ST_FLOOR : 0);
    for (int a = 0; a < w; a++) {
        const long c = cidx(v, i, j, k0 + a);
        double b[3];
        centre_field(v, Bn, i, j, k0 + a, m.igdet, b);
#pragma unroll
        for (int q = 0; q < 5; q++) Po[q * v.nc + c] = pr[q];
        for (int e = 0; e < 3; e++) Po[(B1 + e) * v.nc + c] = b[e];
        status[c] |= sb;
        if (ph.stage32) {
            float p8[NPRIM];
#pragma unroll
            for (int q = 0; q < 5; q++) p8[q] = narrow(pr[q]);
            for (int e = 0; e < 3; e++) p8[B1 + e] = narrow(b[e]);
            store_stage32(v, ph, corrector, c, p8);
        }
    }
    atomicAdd(&dcnt[st == INV_OK ? 0 : (st == INV_ENTROPY ? 1 : 2)], (unsigned long long)w);
    if (fl) atomicAdd(&dcnt[3], (unsigned long long)w);
    atomicAdd(&dcnt[4], (unsigned long long)(w * its));
    if (corrector == 1) {  // the CFL rate over the group's width, of each cell with its own centre field
        BlockView vw = v;
        vw.idx3 = v.idx3 / w;
        double inv = 0.0;
        for (int a = 0; a < w; a++) {
            double pa[NPRIM];
#pragma unroll
            for (int q = 0; q < NPRIM; q++) pa[q] = Po[q * v.nc + cidx(v, i, j, k0 + a)];
            Fluid<double> sa;
            fluid_state(pa, m, sa);
            inv = fmax(inv, inv_dt_fluid(vw, pa, sa, m, ph.gam));
        }
        if (inv > 0.0) atomicMax(dmax, (unsigned long long)__double_as_longlong(inv));
    }
}

__global__ void k_smr_emf(BlockView v, PhysArgs ph, double* __restrict__ E) {
    b_smr_emf(v, ph, E, (long)blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void k_smr_cells(BlockView v, PhysArgs ph, int corrector, const double* __restrict__ Pf,
                            const double* __restrict__ Bn, double* Po, uint8_t* __restrict__ status,
                            unsigned long long* dmax, unsigned long long* dcnt) {
    b_smr_cells(v, ph, corrector, Pf, Bn, ph.smr_u, Po, status, dmax, dcnt, (long)blockIdx.x * blockDim.x + threadIdx.x);
}

// batched: the EMFs of the stage (after the edge synchronisation) and the cells of the block's
// predictor (sigma 0) or corrector (1, no CFL rate: the period sets dt); scratch: the block's right
// edge values, free once the fluxes are formed
__global__ void kb_smr_emf(const DevBlock* tab, const int* list, PhysArgs ph) {
    const DevBlock& D = tab[list[blockIdx.y]];
    b_smr_emf(D.v, ph, D.E, tidx());
}

__global__ void kb_smr_cells(const DevBlock* tab, const int* list, PhysArgs ph, int sigma) {
    const DevBlock& D = tab[list[blockIdx.y]];
    const bool c = sigma != 0;
    b_smr_cells(D.v, ph, c ? 2 : 0, c ? D.Ph : D.P, c ? D.B : D.Bh, D.QR, c ? D.P : D.Ph, D.status, D.dmax, D.dcnt,
                tidx());
}

// maximum of field q over the interior cells, as ordered bits (ordered_bits)
__global__ void k_block_max(BlockView v, const double* __restrict__ P, int q, unsigned long long* out) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long n = (long)v.n1 * v.n2 * v.n3;
    unsigned long long m = 0ull;
    if (t < n) {
        const int i = (int)(t % v.n1), j = (int)((t / v.n1) % v.n2), k = (int)(t / ((long)v.n1 * v.n2));
        m = ordered_bits(P[q * v.nc + cidx(v, i, j, k)]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_down_sync(0xffffffffu, m, o);
        m = x > m ? x : m;
    }
    if ((threadIdx.x & 31u) == 0 && m) atomicMax(out, m);
}

}  // namespace

cudaError_t launch_smr_emf(const BlockView& v, const PhysArgs& ph, double* E, cudaStream_t s) {
    const long n = smr_emf_threads(v, ph);
    if (n > 0) k_smr_emf<<<nblk(n), BS, 0, s>>>(v, ph, E);
    return cudaGetLastError();
}

cudaError_t launch_smr_cells(const BlockView& v, const PhysArgs& ph, int corrector, const double* Pf, const double* Bn,
                             double* Po, uint8_t* status, unsigned long long* dmax, unsigned long long* dcnt,
                             cudaStream_t s) {
    const long n = smr_cell_threads(v, ph);
    if (n > 0) k_smr_cells<<<nblk(n), BS, 0, s>>>(v, ph, corrector, Pf, Bn, Po, status, dmax, dcnt);
    return cudaGetLastError();
}

long smr_emf_threads(const BlockView& v, const PhysArgs& ph) {
    const int nr = smr_rows(v, ph);
    return nr ? (long)(v.n1 + 1) * 2 * (nr + 1) * (v.n3 / 2) : 0;
}

long smr_cell_threads(const BlockView& v, const PhysArgs& ph) { return (long)v.n1 * 2 * smr_rows(v, ph) * (v.n3 / 2); }

cudaError_t launch_smr_emf_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, const PhysArgs& ph,
                                 cudaStream_t s) {
    if (nlist == 0 || maxwork == 0) return cudaSuccess;
    kb_smr_emf<<<dim3(nblk(maxwork), nlist), BS, 0, s>>>(tab, list, ph);
    return cudaGetLastError();
}

cudaError_t launch_smr_cells_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, const PhysArgs& ph,
                                   int sigma, cudaStream_t s) {
    if (nlist == 0 || maxwork == 0) return cudaSuccess;
    kb_smr_cells<<<dim3(nblk(maxwork), nlist), BS, 0, s>>>(tab, list, ph, sigma);
    return cudaGetLastError();
}

cudaError_t launch_block_max(const BlockView& v, const double* P, int q, unsigned long long* out, cudaStream_t s) {
    k_block_max<<<nblk((long)v.n1 * v.n2 * v.n3), BS, 0, s>>>(v, P, q, out);
    return cudaGetLastError();
}

cudaError_t launch_centre_b(const BlockView& v, double* P, const double* B, cudaStream_t s) {
    k_centre_b<<<nblk((long)v.n1 * v.n2 * v.n3), BS, 0, s>>>(v, P, B);
    return cudaGetLastError();
}

cudaError_t launch_bc(const BlockView& v, double* P, double* B, cudaStream_t s, float* P32, float* K32) {
    const long n = 2L * NG * ((long)v.n1p * v.n2p + (long)v.n1p * v.n3 + (long)v.n2 * v.n3) + (long)v.n1 * v.n3;
    k_bc<<<nblk(n), BS, 0, s>>>(v, P, B, P32, K32);
    return cudaGetLastError();
}

cudaError_t launch_load(const BlockView& v, const PhysArgs& ph, const double* prim, const double* bface, double* P,
                        double* B, double* Po, double* Bo, unsigned long long* dmax, cudaStream_t s) {
    k_load<<<nblk((long)v.n1p * v.n2p * v.n3p), BS, 0, s>>>(v, ph, prim, bface, P, B, Po, Bo, dmax);
    return cudaGetLastError();
}

cudaError_t launch_store(const BlockView& v, const double* P, const double* B, double* prim, double* bface,
                         cudaStream_t s) {
    k_store<<<nblk((long)v.n1p * v.n2p * v.n3p), BS, 0, s>>>(v, P, B, prim, bface);
    return cudaGetLastError();
}

cudaError_t launch_flatten(const BlockView& v, const PhysArgs& ph, int dir, const double* P, const float* P32,
                           double* Fl, cudaStream_t s) {
    const long n = (long)(v.n1 + 2) * (v.n2 + 2) * (v.n3 + 2);
    if (ph.mixed) {
        float* F = reinterpret_cast<float*>(Fl);
        if (dir == 1) k_flatten<1, float><<<nblk(n), BS, 0, s>>>(v, ph, P32, F);
        if (dir == 2) k_flatten<2, float><<<nblk(n), BS, 0, s>>>(v, ph, P32, F);
        if (dir == 3) k_flatten<3, float><<<nblk(n), BS, 0, s>>>(v, ph, P32, F);
    } else {
        if (dir == 1) k_flatten<1, double><<<nblk(n), BS, 0, s>>>(v, ph, P, Fl);
        if (dir == 2) k_flatten<2, double><<<nblk(n), BS, 0, s>>>(v, ph, P, Fl);
        if (dir == 3) k_flatten<3, double><<<nblk(n), BS, 0, s>>>(v, ph, P, Fl);
    }
    return cudaGetLastError();
}

cudaError_t launch_kappa(const BlockView& v, const PhysArgs& ph, const double* P, const float* P32, double* K,
                         double* Un, cudaStream_t s) {
    const long n = (long)v.n1p * v.n2p * v.n3p;
    if (ph.mixed)
        k_kappa<float><<<nblk(n), BS, 0, s>>>(v, (float)ph.gam, P32, reinterpret_cast<float*>(K),
                                              Un ? Un + (long)C_ENT * v.nc : nullptr);
    else
        k_kappa<double><<<nblk(n), BS, 0, s>>>(v, ph.gam, P, K, Un ? Un + (long)C_ENT * v.nc : nullptr);
    return cudaGetLastError();
}

cudaError_t launch_recon(const BlockView& v, const PhysArgs& ph, int dir, const double* P, const float* P32,
                         const double* K, const double* Fl, double* QL, double* QR, cudaStream_t s) {
    const int m = recon_cells((long)v.n1 * v.n2 * v.n3, dir);
    const long n = recon_threads(v, dir, ph.mixed ? m : 0, ph.recon_seg, ph.recon_x1_sweep);
    const unsigned nb = nblk(n, ph.bs_recon);
    const int bs = ph.bs_recon;
    if (ph.mixed) {
        const float* K32 = reinterpret_cast<const float*>(K);
        const float* F32 = reinterpret_cast<const float*>(Fl);
        float* L = reinterpret_cast<float*>(QL);
        float* R = reinterpret_cast<float*>(QR);
        if (dir == 1) (m == 1 ? k_recon<1, float, 1> : k_recon<1, float, 2>)<<<nb, bs, 0, s>>>(v, ph, P32, K32, F32, L, R);
        if (dir == 2) (m == 1 ? k_recon<2, float, 1> : k_recon<2, float, 4>)<<<nb, bs, 0, s>>>(v, ph, P32, K32, F32, L, R);
        if (dir == 3) (m == 1 ? k_recon<3, float, 1> : k_recon<3, float, 4>)<<<nb, bs, 0, s>>>(v, ph, P32, K32, F32, L, R);
    } else {
        if (dir == 1) k_recon<1, double, 0><<<nb, bs, 0, s>>>(v, ph, P, K, Fl, QL, QR);
        if (dir == 2) k_recon<2, double, 0><<<nb, bs, 0, s>>>(v, ph, P, K, Fl, QL, QR);
        if (dir == 3) k_recon<3, double, 0><<<nb, bs, 0, s>>>(v, ph, P, K, Fl, QL, QR);
    }
    return cudaGetLastError();
}

cudaError_t launch_to_f32(const BlockView& v, const double* P, float* P32, cudaStream_t s) {
    k_to_f32<<<nblk((long)v.n1p * v.n2p * v.n3p), BS, 0, s>>>(v, P, P32);
    return cudaGetLastError();
}

cudaError_t launch_flux(const BlockView& v, const PhysArgs& ph, int dir, const double* QL, const double* QR,
                        const double* Bf, double* F, cudaStream_t s) {
    const long n1 = v.n1 + (dir == 1 ? 1 : 2), n2 = v.n2 + (dir == 2 ? 1 : 2), n3 = v.n3 + (dir == 3 ? 1 : 2);
    const long n = n1 * n2 * n3;
    const unsigned nb = nblk(n, ph.bs_flux);
    const int bs = ph.bs_flux;
    if (ph.mixed) {
        const float* L = reinterpret_cast<const float*>(QL);
        const float* R = reinterpret_cast<const float*>(QR);
        if (dir == 1) k_flux<1, float><<<nb, bs, 0, s>>>(v, ph, L, R, Bf, F);
        if (dir == 2) k_flux<2, float><<<nb, bs, 0, s>>>(v, ph, L, R, Bf, F);
        if (dir == 3) k_flux<3, float><<<nb, bs, 0, s>>>(v, ph, L, R, Bf, F);
    } else {
        if (dir == 1) k_flux<1, double><<<nb, bs, 0, s>>>(v, ph, QL, QR, Bf, F);
        if (dir == 2) k_flux<2, double><<<nb, bs, 0, s>>>(v, ph, QL, QR, Bf, F);
        if (dir == 3) k_flux<3, double><<<nb, bs, 0, s>>>(v, ph, QL, QR, Bf, F);
    }
    return cudaGetLastError();
}

cudaError_t launch_emf(const BlockView& v, double* const F[3], double* E, int mixed, const double* P, double* Ec,
                       cudaStream_t s) {
    const long n = (long)(v.n1 + 1) * (v.n2 + 1) * (v.n3 + 1);
    if (Ec) {  // upwinded EMFs: the cell EMFs of the stage state P first
        k_cell_emf<<<nblk((long)(v.n1 + 2) * (v.n2 + 2) * (v.n3 + 2)), BS, 0, s>>>(v, P, Ec);
    }
    if (mixed == 2)  // FP32 EMFs of fluxes stored in FP32
        k_emf<float, true><<<nblk(n), BS, 0, s>>>(v, F[0], F[1], F[2], E, Ec);
    else if (mixed)
        k_emf<float><<<nblk(n), BS, 0, s>>>(v, F[0], F[1], F[2], E, Ec);
    else
        k_emf<double><<<nblk(n), BS, 0, s>>>(v, F[0], F[1], F[2], E, Ec);
    return cudaGetLastError();
}

cudaError_t launch_ct(const BlockView& v, const double* E, const double* Bbase, double* Bout, const double* dscal,
                      double dt_factor, cudaStream_t s) {
    const long n = (long)(v.n1 + 1) * (v.n2 + 1) * (v.n3 + 1);
    k_ct<<<nblk(n), BS, 0, s>>>(v, E, Bbase, Bout, dscal, dt_factor);
    return cudaGetLastError();
}

cudaError_t launch_dt_reduce(const BlockView& v, const PhysArgs& ph, const double* P, unsigned long long* dmax,
                             cudaStream_t s) {
    k_dt_reduce<<<nblk((long)v.n1 * v.n2 * v.n3), BS, 0, s>>>(v, ph, P, dmax);
    return cudaGetLastError();
}

cudaError_t launch_dt_select(const PhysArgs& ph, double user_dt, double* dscal, unsigned long long* dmax,
                             unsigned long long* dcnt, uint8_t* status, long nc, cudaStream_t s) {
    k_dt_select<<<1, 32, 0, s>>>(ph.cour, user_dt, dscal, dmax, dcnt);
    cudaMemsetAsync(status, 0, (size_t)nc, s);
    return cudaGetLastError();
}

cudaError_t launch_recon_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, int m,
                               const PhysArgs& ph, int dir, int sigma, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    const int bs = ph.bs_recon;
    const dim3 g = bgrid(maxwork, nlist, bs);
    if (ph.mixed) {
        if (dir == 1) (m == 1 ? kb_recon<1, float, 1> : kb_recon<1, float, 2>)<<<g, bs, 0, s>>>(tab, list, ph, sigma);
        if (dir == 2) (m == 1 ? kb_recon<2, float, 1> : kb_recon<2, float, 4>)<<<g, bs, 0, s>>>(tab, list, ph, sigma);
        if (dir == 3) (m == 1 ? kb_recon<3, float, 1> : kb_recon<3, float, 4>)<<<g, bs, 0, s>>>(tab, list, ph, sigma);
    } else {
        if (dir == 1) kb_recon<1, double, 0><<<g, bs, 0, s>>>(tab, list, ph, sigma);
        if (dir == 2) kb_recon<2, double, 0><<<g, bs, 0, s>>>(tab, list, ph, sigma);
        if (dir == 3) kb_recon<3, double, 0><<<g, bs, 0, s>>>(tab, list, ph, sigma);
    }
    return cudaGetLastError();
}

cudaError_t launch_flatten_batch(const DevBlock* tab, const int* list, int nlist, long maxcells, const PhysArgs& ph,
                                 int dir, int sigma, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    const dim3 g = bgrid(maxcells, nlist);
    if (ph.mixed) {
        if (dir == 1) kb_flatten<1, float><<<g, BS, 0, s>>>(tab, list, ph, sigma);
        if (dir == 2) kb_flatten<2, float><<<g, BS, 0, s>>>(tab, list, ph, sigma);
        if (dir == 3) kb_flatten<3, float><<<g, BS, 0, s>>>(tab, list, ph, sigma);
    } else {
        if (dir == 1) kb_flatten<1, double><<<g, BS, 0, s>>>(tab, list, ph, sigma);
        if (dir == 2) kb_flatten<2, double><<<g, BS, 0, s>>>(tab, list, ph, sigma);
        if (dir == 3) kb_flatten<3, double><<<g, BS, 0, s>>>(tab, list, ph, sigma);
    }
    return cudaGetLastError();
}

cudaError_t launch_kappa_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, const PhysArgs& ph,
                               int sigma, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    if (ph.mixed)
        kb_kappa<float><<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list, ph, sigma);
    else
        kb_kappa<double><<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list, ph, sigma);
    return cudaGetLastError();
}

cudaError_t launch_to_f32_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, int sigma,
                                cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    kb_to_f32<<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list, sigma);
    return cudaGetLastError();
}

cudaError_t launch_flux_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, const PhysArgs& ph,
                              int dir, int sigma, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    const int bs = ph.bs_flux;
    const dim3 g = bgrid(maxwork, nlist, bs);
    if (ph.mixed) {
        if (dir == 1) kb_flux<1, float><<<g, bs, 0, s>>>(tab, list, ph, sigma);
        if (dir == 2) kb_flux<2, float><<<g, bs, 0, s>>>(tab, list, ph, sigma);
        if (dir == 3) kb_flux<3, float><<<g, bs, 0, s>>>(tab, list, ph, sigma);
    } else {
        if (dir == 1) kb_flux<1, double><<<g, bs, 0, s>>>(tab, list, ph, sigma);
        if (dir == 2) kb_flux<2, double><<<g, bs, 0, s>>>(tab, list, ph, sigma);
        if (dir == 3) kb_flux<3, double><<<g, bs, 0, s>>>(tab, list, ph, sigma);
    }
    return cudaGetLastError();
}

cudaError_t launch_emf_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, int mixed, int upwind,
                             long maxcells, int sigma, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    if (upwind) kb_cell_emf<<<bgrid(maxcells, nlist), BS, 0, s>>>(tab, list, sigma);
    if (mixed == 2 && !upwind)  // FP32 EMFs of the FP32 copies of the flux field slots
        kb_emf<float, true><<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list, upwind);
    else if (mixed)
        kb_emf<float><<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list, upwind);
    else
        kb_emf<double><<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list, upwind);
    return cudaGetLastError();
}

cudaError_t launch_ct_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, int sigma, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    kb_ct<<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list, sigma);
    return cudaGetLastError();
}

cudaError_t launch_dt_reduce_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, const PhysArgs& ph,
                                   cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    kb_dt_reduce<<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list, ph);
    return cudaGetLastError();
}

cudaError_t launch_save_old_batch(const DevBlock* tab, const int* list, int nlist, long maxwork, cudaStream_t s) {
    if (nlist <= 0) return cudaSuccess;
    kb_save_old<<<bgrid(maxwork, nlist), BS, 0, s>>>(tab, list);
    return cudaGetLastError();
}

cudaError_t launch_reflux_u0(const DevBlock* tab, int n, const int* cblk, const long* cidx_, const int* nrec,
                             const int* recs, const double* rec_dU, int nrec_tot, double* Ucorr, const PhysArgs& ph,
                             cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_reflux_u0<<<nblk(n), BS, 0, s>>>(tab, n, cblk, cidx_, nrec, recs, rec_dU, nrec_tot, Ucorr, ph);
    return cudaGetLastError();
}

cudaError_t launch_reflux_cells(const DevBlock* tab, int n, const int* cblk, const long* cidx_, const double* Ucorr,
                                long stride, const PhysArgs& ph, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_reflux_cells<<<nblk(n), BS, 0, s>>>(tab, n, cblk, cidx_, Ucorr, stride, ph);
    return cudaGetLastError();
}

cudaError_t launch_reflux_groups(const DevBlock* tab, int ngrp, const int* first, const int* w, const int* cblk,
                                 const long* cidx_, const double* Ucorr, long stride, const PhysArgs& ph,
                                 cudaStream_t s) {
    if (ngrp <= 0) return cudaSuccess;
    k_reflux_groups<<<nblk(ngrp), BS, 0, s>>>(tab, ngrp, first, w, cblk, cidx_, Ucorr, stride, ph);
    return cudaGetLastError();
}

}  // namespace hamr
