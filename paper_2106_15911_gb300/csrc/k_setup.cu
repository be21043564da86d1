// k_setup.cu -- one-time device work of pfmm_build_trees: expansion tables and the nearfield
// quadrature of V_h and K_h.
//
// Tables (Section 3.1, 3.4):
//   Sx[x][kappa]    = int_{gamma_x} T_{Y,kappa}(y) ds_y           (S2M / L2T space part, Eq. s2m, l2t)
//   SK[x][v][kappa] = int_{gamma_x} alpha n_x . grad T_{Y,kappa}(y) phi_v(y) ds_y
//                     (double-layer moments: the normal derivative falls on the expansion of
//                      the source variable, Section 3 "slight modifications")
//   E1[D][a][b][o][k][l] = E_{k,l}(r_o, d_ab) of Eq. exp_coeffs_1d for the interval gap D in {2,3}
//                          and grid offset o of one level; pref[D][a][b] = (4 pi alpha dt_ab)^{-3/2}
// Nearfield (Eq. eval_sl_nf_block with the entries of Section 2): collapsed Gauss-Legendre
// n_r x n_r per triangle for regular pairs; Sauter-Schwab (Sauter & Schwab, Boundary Element
// Methods, Sec. 5.2) with n_s points per direction for triangles sharing a vertex at d = 0, 1.
#include <algorithm>
#include <cstdio>

#include "device_math.cuh"
#include "kernels.h"
#include "nf_geom.cuh"

namespace pfmm {

using namespace dev;

// ------------------------------------------------------------------------------------------
// Sx, SK: thread per (triangle, kappa)
__global__ void k_space_tables(const double *__restrict__ verts, const int *__restrict__ tri, const int *__restrict__ tri_leaf,
                               const int *__restrict__ leaf_grid, double c0, double c1, double c2, double hx, double hxp,
                               int nt, int mx, int nk, const int *__restrict__ kidx, const double *__restrict__ rule,
                               int nq, double alpha, double *__restrict__ Sx, double *__restrict__ SK)
{
    int gid = blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= nt * nk) return;
    int x = gid / nk, ik = gid % nk;
    int k0 = kidx[3 * ik], k1 = kidx[3 * ik + 1], k2 = kidx[3 * ik + 2];
    const int *t = tri + 3 * x;
    double P[3][3];
    for (int v = 0; v < 3; ++v)
        for (int c = 0; c < 3; ++c) P[v][c] = verts[3 * t[v] + c];
    double e1[3], e2[3], cr[3];
    for (int c = 0; c < 3; ++c) { e1[c] = P[1][c] - P[0][c]; e2[c] = P[2][c] - P[1][c]; }
    cr[0] = e1[1] * e2[2] - e1[2] * e2[1];
    cr[1] = e1[2] * e2[0] - e1[0] * e2[2];
    cr[2] = e1[0] * e2[1] - e1[1] * e2[0];
    double J = sqrt(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]);
    double n[3] = {cr[0] / J, cr[1] / J, cr[2] / J};
    const int *g = leaf_grid + 3 * tri_leaf[x];
    double cen[3] = {c0 + (2.0 * g[0] + 1.0) * hx, c1 + (2.0 * g[1] + 1.0) * hx, c2 + (2.0 * g[2] + 1.0) * hx};
    double s = 0.0, sk[3] = {0.0, 0.0, 0.0};
    double T[3][kMaxMx + 1], dT[3][kMaxMx + 1];
    for (int q = 0; q < nq; ++q) {
        double s1 = rule[q], s2 = rule[nq + q], w = rule[2 * nq + q] * J;
        double yh[3];
        for (int c = 0; c < 3; ++c) yh[c] = (P[0][c] + s1 * e1[c] + s2 * e2[c] - cen[c]) / hxp;
        for (int c = 0; c < 3; ++c) {
            cheb_all(yh[c], mx, T[c]);
            cheb_deriv_all(yh[c], mx, dT[c]);
        }
        double tv = T[0][k0] * T[1][k1] * T[2][k2];
        s += w * tv;
        double gr[3] = {dT[0][k0] * T[1][k1] * T[2][k2] / hxp, T[0][k0] * dT[1][k1] * T[2][k2] / hxp,
                        T[0][k0] * T[1][k1] * dT[2][k2] / hxp};
        double dn = alpha * (n[0] * gr[0] + n[1] * gr[1] + n[2] * gr[2]);
        double by[3] = {1.0 - s1, s1 - s2, s2};
        for (int v = 0; v < 3; ++v) sk[v] += w * dn * by[v];
    }
    Sx[(size_t)x * nk + ik] = s;
    for (int v = 0; v < 3; ++v) SK[((size_t)x * 3 + v) * nk + ik] = sk[v];
}

void launch_space_tables(const SetupArgs &a, cudaStream_t st)
{
    int n = a.nt * a.nk;
    k_space_tables<<<(n + 127) / 128, 128, 0, st>>>(a.verts, a.tri, a.tri_leaf, a.leaf_grid, a.corner[0], a.corner[1],
                                                    a.corner[2], a.hx_leaf, a.hxp_leaf, a.nt, a.mx, a.nk, a.kidx,
                                                    a.rule_tab, a.nq_tab, a.alpha, a.Sx, a.SK);
}

// ------------------------------------------------------------------------------------------
// E1 tables of one level: thread per (D, a, b, o, k, l).  E_{k,l}(-r) = (-1)^{k+l} E_{k,l}(r) holds
// exactly in the table (the value of the offset's mirror image with its sign, 0 for o = 0 and odd
// k + l): the folded M2L relies on it, and the double layer's far field amplifies the asymmetry that
// rounding leaves otherwise about a hundredfold (1.3e-13; either table leaves it 3.5e-13 from exact ones)
__global__ void k_e1_table(int na, int mt, int mx, int G, double hx, double hxp, double ht, double alpha,
                           double *__restrict__ E1, double *__restrict__ pref)
{
    const int m1 = mx + 1, no = 2 * G - 1;
    int gid = blockIdx.x * blockDim.x + threadIdx.x;
    int total = 2 * na * na * no * m1 * m1;
    if (gid >= total) return;
    int l = gid % m1, r_ = gid / m1;
    int k = r_ % m1;
    r_ /= m1;
    int o = r_ % no;
    r_ /= no;
    int b = r_ % na;
    r_ /= na;
    int a = r_ % na;
    int D = r_ / na + 2;
    double L = 2.0 * ht;
    double xb = cos((2.0 * b + 1.0) * kPi / (2.0 * mt + 2.0)), xa = cos((2.0 * a + 1.0) * kPi / (2.0 * mt + 2.0));
    double dt = D * L + ht * (xb - xa);  // xi_{I,b} - xi_{J,a}, J = I - D intervals
    double dab = 4.0 * alpha * dt / (hxp * hxp);
    if (o == 0 && k == 0 && l == 0) pref[((D - 2) * na + a) * na + b] = pow(4.0 * kPi * alpha * dt, -1.5);
    double val = 0.0;
    if (k + l <= mx) {
        const int off = o - (G - 1);
        double r = 2.0 * hx * (off < 0 ? -off : off) / hxp;
        double s = 0.0;
        for (int n = 0; n <= mx; ++n) {
            double xn = cos((2.0 * n + 1.0) * kPi / (2.0 * mx + 2.0));
            double Tl = cos(l * acos(xn));
            for (int mm = 0; mm <= mx; ++mm) {
                double xm = cos((2.0 * mm + 1.0) * kPi / (2.0 * mx + 2.0));
                double z = r + xn - xm;
                s += exp(-z * z / dab) * Tl * cos(k * acos(xm));
            }
        }
        double lam = (k == 0 ? 1.0 : 2.0) * (l == 0 ? 1.0 : 2.0);
        val = lam / ((mx + 1.0) * (mx + 1.0)) * s;
        if ((k + l) & 1) val = off < 0 ? -val : (off == 0 ? 0.0 : val);
    }
    E1[gid] = val;
}

void launch_e1_table(int na, int mt, int mx, int G, double hx, double hxp, double ht, double alpha, double *E1,
                     double *pref, cudaStream_t st)
{
    int m1 = mx + 1, no = 2 * G - 1;
    int total = 2 * na * na * no * m1 * m1;
    k_e1_table<<<(total + 127) / 128, 128, 0, st>>>(na, mt, mx, G, hx, hxp, ht, alpha, E1, pref);
}

// ------------------------------------------------------------------------------------------
// Regular nearfield quadrature of both layers.  Thread per (row, column) of one panel; bound by the
// FP64 (FP32) pipe and the special functions, which the two layers share (see time_integrals).
// One launch for all panels (grid z): a small mesh's panels have too few rows to fill the GPU alone.
template <typename R, int ND>
__global__ void __launch_bounds__(256) k_nf_regular(NfQuadArgs a, const PanelGPU *__restrict__ panels,
                                                      R *__restrict__ AVs, R *__restrict__ AKs)
{
    const PanelGPU &P = panels[blockIdx.z];
    int col = blockIdx.x * blockDim.x + threadIdx.x;
    int row = blockIdx.y * blockDim.y + threadIdx.y;
    if (row >= P.nrows || col >= P.ncolV) return;
    int y = a.colV[P.colV_at + col];
    if (y < 0) return;
    int x = P.row0 + row;
    R accV[ND], accK[3 * ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) accV[i] = R(0);
#pragma unroll
    for (int i = 0; i < 3 * ND; ++i) accK[i] = R(0);
    const int d0 = nf_regular_pair<R, true, true, ND>(a, x, y, accV, accK);
    R *AV = AVs + P.offV, *AK = AKs + P.offK;
#pragma unroll
    for (int d = 0; d < ND; ++d)
        if (d >= d0) AV[((size_t)d * P.rows_pad + row) * P.colsV_pad + col] = accV[d];
    for (int v = 0; v < 3; ++v) {
        const int kc = a.kmap[(size_t)P.index * a.nv + a.tri[3 * y + v]];
#pragma unroll
        for (int d = 0; d < ND; ++d)
            if (d >= d0) atomicAdd(&AK[((size_t)d * P.rows_pad + row) * P.colsK_pad + kc], accK[3 * d + v]);
    }
}

template <typename R>
void launch_nf_regular_T(const NfQuadArgs &a, const PanelGPU *panels, dim3 grd, R *AV, R *AK, cudaStream_t st)
{
    auto kf = a.nd == 2 ? k_nf_regular<R, 2> : a.nd == 4 ? k_nf_regular<R, 4> : a.nd == 6 ? k_nf_regular<R, 6> : k_nf_regular<R, 8>;
    kf<<<grd, dim3(32, 8), 0, st>>>(a, panels, AV, AK);
}

void launch_nf_regular(const NfQuadArgs &a, const PanelGPU *panels, int npanel, int max_rows, int max_cols, void *AV,
                       void *AK, bool mixed, cudaStream_t st)
{
    for (int p0 = 0; p0 < npanel; p0 += 65535) {  // grid z limit
        const dim3 grd((max_cols + 31) / 32, (max_rows + 7) / 8, std::min(npanel - p0, 65535));
        if (mixed)
            launch_nf_regular_T<float>(a, panels + p0, grd, (float *)AV, (float *)AK, st);
        else
            launch_nf_regular_T<double>(a, panels + p0, grd, (double *)AV, (double *)AK, st);
    }
}

// ------------------------------------------------------------------------------------------
// Sauter-Schwab quadrature of touching pairs at d = 0, 1: one warp per pair, FP64.
// Output: into the stored panels (AV, AK), or, when cV is given (on-the-fly nearfield), compactly
// per pair: cV[pair][d], cK[pair][d][v] (v: the source triangle's vertices in mesh order).
template <typename S>
__global__ void __launch_bounds__(128) k_nf_singular(NfQuadArgs a, const int *__restrict__ sing /*[n][12]*/, int nsing,
                                                       const PanelGPU *__restrict__ panels, S *__restrict__ AV,
                                                       S *__restrict__ AK, double *__restrict__ cV,
                                                       double *__restrict__ cK)
{
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= nsing) return;
    const int *sp = sing + 12 * warp;
    int x = sp[0], y = sp[1], panel = sp[2], row = sp[3], colV = sp[4], code = sp[5];
    int cls = code & 3;
    int ox[3] = {(code >> 2) & 3, (code >> 4) & 3, (code >> 6) & 3};
    int oy[3] = {(code >> 8) & 3, (code >> 10) & 3, (code >> 12) & 3};
    double PXo[3][3], PYo[3][3], PX[3][3], PY[3][3], ny[3], nx[3];
    load_tri(a.verts, a.tri, x, PXo);
    load_tri(a.verts, a.tri, y, PYo);
    tri_normal_orig(PYo, ny);
    for (int v = 0; v < 3; ++v)
        for (int c = 0; c < 3; ++c) {
            PX[v][c] = PXo[ox[v]][c];
            PY[v][c] = PYo[oy[v]][c];
        }
    double Jx = tri_jac(PX, nx), Jy = tri_jac(PY, nx);
    const int n = a.nq_sing;
    const double *gx = a.gl_sing, *gw = a.gl_sing + n;
    double accV[2] = {0, 0}, accK[2][3] = {{0, 0, 0}, {0, 0, 0}};
    const int n4 = n * n * n * n;
    for (int q = lane; q < n4; q += 32) {
        int i0 = q / (n * n * n), i1 = (q / (n * n)) % n, i2 = (q / n) % n, i3 = q % n;
        double xi = gx[i0], e1 = gx[i1], e2 = gx[i2], e3 = gx[i3];
        double w4 = gw[i0] * gw[i1] * gw[i2] * gw[i3];
        double pts[6][4], jac[6];
        const int np = ss_points(cls, xi, e1, e2, e3, pts, jac);
        for (int u = 0; u < np; ++u) {
            double xp[3], yp[3], dx[3];
            for (int c = 0; c < 3; ++c) {
                xp[c] = PX[0][c] + pts[u][0] * (PX[1][c] - PX[0][c]) + pts[u][1] * (PX[2][c] - PX[1][c]);
                yp[c] = PY[0][c] + pts[u][2] * (PY[1][c] - PY[0][c]) + pts[u][3] * (PY[2][c] - PY[1][c]);
                dx[c] = xp[c] - yp[c];
            }
            double r = sqrt(dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2]);
            double wt = w4 * jac[u] * Jx * Jy;
            double vv[2], kk[2];
            time_integrals<double, true, true, 2>(r, a.tc, vv, kk);
            accV[0] += wt * vv[0];
            accV[1] += wt * vv[1];
            double dn = dx[0] * ny[0] + dx[1] * ny[1] + dx[2] * ny[2];
            double byl[3] = {1.0 - pts[u][2], pts[u][2] - pts[u][3], pts[u][3]}, by[3];
            for (int v = 0; v < 3; ++v) by[oy[v]] = byl[v];
            for (int d = 0; d < 2; ++d)
                for (int v = 0; v < 3; ++v) accK[d][v] += wt * dn * kk[d] * by[v];
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        for (int d = 0; d < 2; ++d) {
            accV[d] += __shfl_xor_sync(0xffffffffu, accV[d], off);
            for (int v = 0; v < 3; ++v) accK[d][v] += __shfl_xor_sync(0xffffffffu, accK[d][v], off);
        }
    }
    if (lane == 0 && cV) {
        for (int d = 0; d < 2; ++d) {
            cV[2 * (size_t)warp + d] = d < a.nd ? accV[d] : 0.0;
            for (int v = 0; v < 3; ++v) cK[6 * (size_t)warp + 3 * d + v] = d < a.nd ? accK[d][v] : 0.0;
        }
    } else if (lane == 0) {
        const PanelGPU &P = panels[panel];
        for (int d = 0; d < 2 && d < a.nd; ++d) {
            AV[P.offV + ((size_t)d * P.rows_pad + row) * P.colsV_pad + colV] = S(accV[d]);
            for (int v = 0; v < 3; ++v)
                atomicAdd(&AK[P.offK + ((size_t)d * P.rows_pad + row) * P.colsK_pad + sp[6 + v]], S(accK[d][v]));
        }
    }
}

void launch_nf_singular(const NfQuadArgs &a, const int *sing, int nsing, const PanelGPU *panels, void *AV, void *AK,
                        bool mixed, cudaStream_t st, double *cV, double *cK)
{
    if (nsing == 0) return;
    int blocks = (nsing * 32 + 127) / 128;
    if (mixed)
        k_nf_singular<float><<<blocks, 128, 0, st>>>(a, sing, nsing, panels, (float *)AV, (float *)AK, cV, cK);
    else
        k_nf_singular<double><<<blocks, 128, 0, st>>>(a, sing, nsing, panels, (double *)AV, (double *)AK, cV, cK);
}

}  // namespace pfmm
