// geom.cu -- geometry tables of a block (Liska et al. 2019, Sec. 2.2).
//
// The Kerr metric is evaluated analytically in Kerr-Schild coordinates and
// carried to the internal coordinates x1 = log r, x2 = theta, x3 = phi with
// the exact Jacobian dr/dx1 = r. Christoffel symbols are finite differences
// of the internal-coordinate metric: 4th-order central differences with
// step h = 1e-3 in x1 and x2 (the metric does not depend on t or phi); the
// same derivatives are also stored themselves for the FP64 source term.
// Tables are 2-D over the padded (i, j) plane because the metric is
// stationary and axisymmetric; each component is one contiguous plane.
#include "grmhd.cuh"
#include "hamr_internal.h"
#include "metric.cuh"

namespace hamr {

namespace {

constexpr double CONN_H = 1.0e-3;

__device__ void store_metric(double* __restrict__ tab, long stride, long q, const FullMetric& M, bool pole) {
    tab[G_00 * stride + q] = M.g[0][0];
    tab[G_01 * stride + q] = M.g[0][1];
    tab[G_03 * stride + q] = M.g[0][3];
    tab[G_11 * stride + q] = M.g[1][1];
    tab[G_13 * stride + q] = M.g[1][3];
    tab[G_22 * stride + q] = M.g[2][2];
    tab[G_33 * stride + q] = M.g[3][3];
    tab[GI_00 * stride + q] = M.gi[0][0];
    tab[GI_01 * stride + q] = M.gi[0][1];
    tab[GI_11 * stride + q] = M.gi[1][1];
    tab[GI_13 * stride + q] = M.gi[1][3];
    tab[GI_22 * stride + q] = M.gi[2][2];
    tab[GI_33 * stride + q] = pole ? 0.0 : M.gi[3][3];
    tab[G_DET * stride + q] = pole ? 0.0 : M.gdet;
    tab[G_ALPHA * stride + q] = 1.0 / sqrt(-M.gi[0][0]);
    tab[G_IALPHA * stride + q] = sqrt(-M.gi[0][0]);
    tab[G_IGDET * stride + q] = pole ? 0.0 : 1.0 / M.gdet;
}

// One thread per (i, j) point: the least work, for planes that fill the chip with it.
__global__ void k_geometry_points(GeomArgs A) {
    const long n2d = A.table_stride;
    const long q = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (long)A.n1p * A.n2p) return;
    const int i = (int)(q % A.n1p) - NG;
    const int j = (int)(q / A.n1p) - NG;
    const double x1c = A.x1min + (i + 0.5) * A.dx1, x2c = A.x2min + (j + 0.5) * A.dx2;
    const double x1f = A.x1min + i * A.dx1, x2f = A.x2min + j * A.dx2;
    FullMetric M;
    metric_at(A.metric, A.a, x1c, x2c, M);
    store_metric(A.centre, n2d, q, M, false);
    // Christoffel symbols at the centre
    double dg[3][4][4];  // d/dx1, d/dx2 (index 1, 2); index 0 unused
    for (int m = 0; m < 4; m++)
        for (int n = 0; n < 4; n++) dg[0][m][n] = dg[1][m][n] = dg[2][m][n] = 0.0;
    if (A.metric != HAMR_METRIC_MINKOWSKI) {
        for (int s = 1; s <= 2; s++) {
            const double e1 = (s == 1) ? CONN_H : 0.0, e2 = (s == 2) ? CONN_H : 0.0;
            FullMetric p2, p1, m1, m2;
            metric_at(A.metric, A.a, x1c + 2.0 * e1, x2c + 2.0 * e2, p2);
            metric_at(A.metric, A.a, x1c + e1, x2c + e2, p1);
            metric_at(A.metric, A.a, x1c - e1, x2c - e2, m1);
            metric_at(A.metric, A.a, x1c - 2.0 * e1, x2c - 2.0 * e2, m2);
            for (int m = 0; m < 4; m++)
                for (int n = 0; n < 4; n++)
                    dg[s][m][n] = (8.0 * (p1.g[m][n] - m1.g[m][n]) - (p2.g[m][n] - m2.g[m][n])) / (12.0 * CONN_H);
        }
    }
    // Gamma^l_{mn} = 1/2 g^{lk} (d_m g_{kn} + d_n g_{km} - d_k g_{mn})
    for (int l = 0; l < 4; l++)
        for (int m = 0; m < 4; m++)
            for (int n = m; n < 4; n++) {
                double s = 0.0;
                for (int k = 0; k < 4; k++) {
                    const double dm = (m == 1 || m == 2) ? dg[m][k][n] : 0.0;
                    const double dn = (n == 1 || n == 2) ? dg[n][k][m] : 0.0;
                    const double dk = (k == 1 || k == 2) ? dg[k][m][n] : 0.0;
                    s += M.gi[l][k] * (dm + dn - dk);
                }
                A.centre[(C_CONN + l * 10 + sym(m, n)) * n2d + q] = 0.5 * s;
            }
    {
        const int pm[7] = {0, 0, 0, 1, 1, 2, 3}, pn[7] = {0, 1, 3, 1, 3, 2, 3};
        for (int s = 1; s <= 2; s++)
            for (int p = 0; p < 7; p++)
                A.centre[(C_DG + (s - 1) * 7 + p) * n2d + q] = (pm[p] == pn[p] ? 0.5 : 1.0) * dg[s][pm[p]][pn[p]];
    }
    const double r = (A.metric != HAMR_METRIC_MINKOWSKI) ? exp(x1c) : 1.0;
    A.centre[C_RHOFLR * n2d + q] = 1.0e-7 / (r * r);
    A.centre[C_UFLR * n2d + q] = 1.0e-9 * pow(r, -10.0 / 3.0);

    metric_at(A.metric, A.a, x1f, x2c, M);
    store_metric(A.face1, n2d, q, M, false);
    metric_at(A.metric, A.a, x1c, x2f, M);
    const bool pole = (A.pole_lo && j == 0) || (A.pole_hi && j == A.n2);
    store_metric(A.face2, n2d, q, M, pole);
}

// Twelve threads per (i, j) point, for smaller planes. The point's metric is wanted at eleven places (the
// centre, four around it in x1 and four in x2 for the derivatives, the two faces), each a chain of FP64
// transcendental functions: one place per thread, the covariant entries shared through shared memory, then
// the Christoffel symbols spread over the threads. Bound by that chain's latency: the tables of a 24x12x8
// block, which the no-allocation step forms on every call, take 20 us, 57 with a thread per point, which takes
// that long up to 15000 points. Every warp also runs the floors' power for a few of its lanes, so the time
// here grows with the points: 43 us at 4000, 62 at 6144, 295 at 35108 (256x128; 108 with a thread per point).
// The two meet between: from 6144 points on k_geometry_points.
constexpr int GEO_T = 12, GEO_P = 8;  // threads per point (eleven places and the floors), points per CTA

__global__ void __launch_bounds__(GEO_T* GEO_P) k_geometry(GeomArgs A) {
    __shared__ double sg[GEO_P][9][7];   // covariant entries: centre, x1 + 2h, + h, - h, - 2h, the same in x2
    __shared__ double sdg[GEO_P][2][7];  // derivatives
    __shared__ double sgi[GEO_P][6];     // contravariant entries at the centre
    const long n2d = A.table_stride;
    const int pt = threadIdx.x / GEO_T, r = threadIdx.x % GEO_T;
    const long q = (long)blockIdx.x * GEO_P + pt;
    const bool on = q < (long)A.n1p * A.n2p;
    const int i = (int)(q % A.n1p) - NG;
    const int j = (int)(q / A.n1p) - NG;
    const double x1c = A.x1min + (i + 0.5) * A.dx1, x2c = A.x2min + (j + 0.5) * A.dx2;
    const double x1f = A.x1min + i * A.dx1, x2f = A.x2min + j * A.dx2;
    if (on && r < 11) {
        const double st[4] = {2.0 * CONN_H, CONN_H, -CONN_H, -2.0 * CONN_H};
        const double x1 = (r == 9) ? x1f : ((r >= 1 && r <= 4) ? x1c + st[(r - 1) & 3] : x1c);
        const double x2 = (r == 10) ? x2f : ((r >= 5 && r <= 8) ? x2c + st[(r - 5) & 3] : x2c);
        FullMetric M;
        metric_at(A.metric, A.a, x1, x2, M);
        if (r < 9) {
            double* o = sg[pt][r];
            o[0] = M.g[0][0], o[1] = M.g[0][1], o[2] = M.g[0][3], o[3] = M.g[1][1], o[4] = M.g[1][3];
            o[5] = M.g[2][2], o[6] = M.g[3][3];
        }
        if (r == 0) {
            double* o = sgi[pt];
            o[0] = M.gi[0][0], o[1] = M.gi[0][1], o[2] = M.gi[1][1], o[3] = M.gi[1][3], o[4] = M.gi[2][2];
            o[5] = M.gi[3][3];
            store_metric(A.centre, n2d, q, M, false);
        }
        if (r == 9) store_metric(A.face1, n2d, q, M, false);
        if (r == 10) store_metric(A.face2, n2d, q, M, (A.pole_lo && j == 0) || (A.pole_hi && j == A.n2));
    } else if (on && r == 11) {
        const double rr = (A.metric != HAMR_METRIC_MINKOWSKI) ? exp(x1c) : 1.0;
        A.centre[C_RHOFLR * n2d + q] = 1.0e-7 / (rr * rr);
        A.centre[C_UFLR * n2d + q] = 1.0e-9 * pow(rr, -10.0 / 3.0);
    }
    __syncthreads();
    // 4th-order differences of the 7 non-zero entries
    const int pm[7] = {0, 0, 0, 1, 1, 2, 3}, pn[7] = {0, 1, 3, 1, 3, 2, 3};
    for (int c = r; on && c < 14; c += GEO_T) {
        const int s = c / 7, e = c % 7;
        const double(*g)[7] = &sg[pt][1 + 4 * s];
        const double d = (A.metric != HAMR_METRIC_MINKOWSKI)
                             ? (8.0 * (g[1][e] - g[2][e]) - (g[0][e] - g[3][e])) / (12.0 * CONN_H)
                             : 0.0;
        sdg[pt][s][e] = d;
        A.centre[(C_DG + s * 7 + e) * n2d + q] = (pm[e] == pn[e] ? 0.5 : 1.0) * d;
    }
    __syncthreads();
    // Gamma^l_{mn} = 1/2 g^{lk} (d_m g_{kn} + d_n g_{km} - d_k g_{mn}), d_t = d_phi = 0
    if (!on) return;
    auto dg = [&](int s, int m, int n) {  // d_s g_{mn}, zero where structurally so
        if (s != 1 && s != 2) return 0.0;
        const int lo = m < n ? m : n, hi = m < n ? n : m;
        const int e = (lo == 0) ? (hi == 0 ? 0 : (hi == 1 ? 1 : (hi == 3 ? 2 : -1)))
                                : (lo == 1 ? (hi == 1 ? 3 : (hi == 3 ? 4 : -1)) : (lo == hi ? lo + 3 : -1));
        return e < 0 ? 0.0 : sdg[pt][s - 1][e];
    };
    auto gi = [&](int l, int k) {
        const int lo = l < k ? l : k, hi = l < k ? k : l;
        const int e = (lo == 0) ? (hi <= 1 ? hi : -1) : (lo == 1 ? (hi == 1 ? 2 : (hi == 3 ? 3 : -1)) : (lo == hi ? lo + 2 : -1));
        return e < 0 ? 0.0 : sgi[pt][e];
    };
    for (int c = r; c < 40; c += GEO_T) {
        const int l = c / 10;
        int m = 0, n = c % 10;  // the pair (m <= n) of sym()'s order
        while (n >= 4 - m) {
            n -= 4 - m;
            m++;
        }
        n += m;
        double s = 0.0;
        for (int k = 0; k < 4; k++) {
            const double c_lk = gi(l, k);
            if (c_lk != 0.0) s += c_lk * (dg(m, k, n) + dg(n, k, m) - dg(k, m, n));
        }
        A.centre[(C_CONN + c) * n2d + q] = 0.5 * s;
    }
}

}  // namespace

__global__ void k_table_f32(const double* __restrict__ src, float* __restrict__ dst, long n) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) dst[t] = (float)src[t];
}

cudaError_t launch_table_f32(const double* src, float* dst, int nplanes, long stride, cudaStream_t s) {
    const long n = (long)nplanes * stride;
    k_table_f32<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_geometry(const GeomArgs& A, cudaStream_t s) {
    const long n2d = (long)A.n1p * A.n2p;
    if (n2d >= 6144)
        k_geometry_points<<<(unsigned)((n2d + 127) / 128), 128, 0, s>>>(A);
    else
        k_geometry<<<(unsigned)((n2d + GEO_P - 1) / GEO_P), GEO_T * GEO_P, 0, s>>>(A);
    return cudaGetLastError();
}

}  // namespace hamr
