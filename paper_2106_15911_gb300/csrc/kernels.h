// kernels.h -- launch interfaces between the host orchestration (capi.cpp) and the CUDA files.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "device_math.cuh"
#include "pfmm_internal.h"

namespace pfmm {

struct PanelGPU {  // device copy of Panel
    int index, row0, nrows, rows_pad;
    int ncolV, colsV_pad, ncolK, colsK_pad;
    long long offV, offK;
    int colV_at, colK_at;
};

struct SetupArgs {
    const double *verts;   // [nv][3]
    const int *tri;        // [nt][3] internal order
    const int *tri_leaf;   // [nt]
    const int *leaf_grid;  // [nbox_p][3]
    double corner[3], hx_leaf, hxp_leaf, alpha;
    int nt, mx, nk;
    const int *kidx;       // [nk][3] graded multi-indices
    const double *rule_tab;// collapsed rule s1[nq], s2[nq], w[nq] (exact for degree m_x)
    int nq_tab;
    double *Sx, *SK;       // [nt][nk], [nt][3][nk]
};

struct NfQuadArgs {
    const double *verts;
    const int *tri;        // internal order
    int nv, nd;            // nd = 2 leaf_steps step offsets
    double h, alpha;
    const double *rule_reg;// collapsed rule s1, s2, w (n_r^2 points)
    int nq_reg;
    const double *gl_sing; // Gauss-Legendre on [0,1]: x[n], w[n]
    int nq_sing;
    const int *colV;       // all panels' V columns
    const int *kmap;       // [npanel][nv]
    dev::TimeConst<double> tc;  // constants of the nd step ends
    dev::TimeConst<float> tcf;
};

void launch_space_tables(const SetupArgs &a, cudaStream_t st);
void launch_e1_table(int na, int mt, int mx, int G, double hx, double hxp, double ht, double alpha, double *E1,
                     double *pref, cudaStream_t st);
// panels: device array; max_rows, max_cols: largest nrows and ncolV of the panels
void launch_nf_regular(const NfQuadArgs &a, const PanelGPU *panels, int npanel, int max_rows, int max_cols, void *AV,
                       void *AK, bool mixed, cudaStream_t st);
void launch_nf_singular(const NfQuadArgs &a, const int *sing, int nsing, const PanelGPU *panels, void *AV, void *AK,
                        bool mixed, cudaStream_t st, double *cV = nullptr, double *cK = nullptr);

// on-the-fly nearfield (quadrature fused into the apply, no stored panels)
struct OtfArgs {
    NfQuadArgs q;              // geometry, time step, regular rule
    const PanelGPU *panels;
    const int *tiles;          // [ntiles][2] (panel, first row) of 64-row tiles
    int ntiles;
    const int *tile_sing;      // [ntiles + 1] ranges of the singular list per tile
    const int *sing;           // [n][12] singular pairs (x, y, panel, row, colV, code, ...)
    const double *singV;       // [n][2] Sauter-Schwab values, d = 0, 1
    const double *singK;       // [n][2][3]
    const void *x;             // V: permuted input [rhs][Et][nt]; K: nodal input [rhs][Et][nv] (arithmetic type)
    int ncolg, Et, ls, nrhs, ndmax;
    double *f;                 // [rhs][Et][nt] internal rows, accumulated (+=)
    int nt;
};
// f += nearfield(x) with the panels recomputed tile by tile; kop: double layer (node columns)
void launch_nf_otf(bool mixed, bool kop, const OtfArgs &a, int nsm, cudaStream_t st);

// ---- apply ------------------------------------------------------------------------------
// unit tables of the folded M2L (k_m2l.cu) on the device; units null: not built
constexpr int kM2LMaxSlices = 8;
struct M2LFoldDev {
    int urows, nslice, nunits, first3, ntask3, q3;  // rows of U, units, pass 3: first unit, tasks (in all, per warp)
    int first1[kM2LMaxSlices], ntask1[kM2LMaxSlices], first2[kM2LMaxSlices], ntask2[kM2LMaxSlices];
    const int *units, *urow;
    size_t smem;
};

struct ApplyGeo {
    int nt, nv, Et, ls, nd, na, nk, mx, p;
    const int *perm;       // [nt] internal -> caller triangle
    const int *tri;        // [nt][3] internal order
    const int *leaf_start; // [nbox_p + 1]
    int nbox_leaf;
    const int *kidx;       // [nk][3] graded
    const int *kinv;       // [(m+1)^3] -> graded index
    int ne;                // C(m_x+4, 4): budget-indexed entries of the separable M2L intermediates
    const int *eoff;       // [nk] offset of the budget range of each triple
    const int *tiles;      // [ntiles][2] (leaf box, first row) of the 64-row tiles of every leaf box
    int ntiles;
    const int *box_tiles;  // [nbox_p + 1] first tile of each leaf box (tiles are box-major)
    int nsm;               // streaming multiprocessors of the device (grid sizing)
    int m2l_force;         // M2L engine asked for by the batch autotuner (PFMM_M2L_* code, 0: none)
    const M2LFoldDev *fold;// [3] unit tables of the folded M2L: 4^3 with T2 whole, sliced; 8^3
};

// prec of the FMM launchers: 0 FP64, 1 FP32 (mixed mode), 2 double-FP32 (FP64 mode); every
// moment, local and table buffer holds 8-byte elements in modes 0 and 2, 4-byte ones in mode 1
void launch_permute_in(const double *w, void *w_int, bool to_float, int nrhs, const ApplyGeo &g, cudaStream_t st);
void launch_permute_out(const double *f_int, double *f, int nrhs, const ApplyGeo &g, cudaStream_t st);
void launch_cast_to_float(const double *x, float *y, size_t n, cudaStream_t st);
// rewrite n FP64 values in place as double-FP32 pairs (hi, lo) of the same 8 bytes
void launch_to_df64(double *x, size_t n, cudaStream_t st);
// FP32 panels held only as the tensor-core engine's FP16 parts: A = (hi + lo) * inv_scale
struct NfHalfSplit {
    const uint16_t *parts = nullptr;  // FP16 bit patterns (nf_split_index)
    float inv_scale = 1.f;            // 2^-E of the split's scale (exact)
};
// Position of the high part of entry (target triangle x in internal order, step offset d < 4, column c)
// of a layout with 32 * nkb columns; the low part is kSplitPart further.  Both parts of 128 rows x 32
// columns at one offset are 16 KB in one piece, [tile][column block][d][part][row][32], with the
// 16-byte chunks of row r at chunk ^ ((r / 2) mod 4) (the 64-byte swizzle of the MMA's operands).
constexpr size_t kSplitPart = 4096;
__host__ __device__ inline size_t nf_split_index(int x, int d, int c, int nkb)
{
    const int r = x & 127;
    return (((size_t)(x >> 7) * nkb + (c >> 5)) * 4 + d) * (2 * kSplitPart) + r * 32 +
           ((((c >> 3) & 3) ^ ((r >> 1) & 3)) << 3) + (c & 7);
}
void launch_nf_apply(bool mixed, bool kop, const void *A, const int *colidx, const int *tiles, int ntiles,
                     const PanelGPU *panels, const void *x, int ncolg, int nrhs, const ApplyGeo &g, double *f_int,
                     cudaStream_t st,
                     bool same_step = false,            // offset 0 only, each of the g.Et steps a slice of its own
                     const NfHalfSplit *hs = nullptr);  // FP32 only: blocks from the FP16 parts, A unused
// ws: scratch of ws_elems elements of the arithmetic type for the per-tile partial moments (the
// M2L workspace, idle at this point); too small: one CTA per whole leaf box instead
void launch_s2m(int prec, bool kop, const void *x, int ncolg, const void *Stab /*Sx or SK*/, const void *St,
                void *mu_leaf, int nrhs, const ApplyGeo &g, cudaStream_t st, void *ws = nullptr, size_t ws_elems = 0);
void launch_m2m(int prec, const DevLevel &par, const DevLevel &ch, int l, const void *qt, void *mu, int nrhs,
                const ApplyGeo &g, int64_t mu_stride, cudaStream_t st);
// M2L of the levels 2 .. p (dl[l]); T1, T2: scratch of ws_elems elements each; -1: one interval of a
// three-pass level does not fit it
int launch_m2l_levels(int prec, const DevLevel *dl, int p, const void *mu, void *lam, int nrhs, const ApplyGeo &g, void *T1,
                      void *T2, size_t ws_elems, cudaStream_t st);
// M2L kernel of a level with a G^3 grid (launch_m2l_levels' choice).  kM2LThreePass needs T1 and T2; the others
// take T1 where it is large enough: the fused kernels for a launch by source terms, the slab kernel for its
// folded moments (else it runs unfolded)
enum { kM2LThreePass = 0, kM2LFused = 1, kM2LSlab = 2, kM2LFusedSliced = 3 };
int m2l_engine(int prec, int G, int nk, int ne, int mx);
// the engine of a level when an autotuner asks for `force` (a PFMM_M2L_* code; 0: none): the forced
// engine where it can run that level, else m2l_engine's choice
int m2l_engine_for(int prec, int G, int nk, int ne, int mx, int force);
void launch_l2l(int prec, const DevLevel &par, const DevLevel &ch, int l, const void *qt, void *lam, int nrhs,
                const ApplyGeo &g, int64_t mu_stride, cudaStream_t st);
// ws: scratch (ws_elems elements of the arithmetic type) for the temporal factor of every (step,
// leaf box), the M2L workspace idle at this point; too small: computed per CTA
void launch_l2t(int prec, const void *lam_leaf, const void *Sx, const void *St, double *f_int, int nrhs,
                const ApplyGeo &g, int64_t mu_stride, cudaStream_t st, void *ws = nullptr, size_t ws_elems = 0);
void launch_apply_M(const double *g_in, double *f, const int *tri_user, const double *area, int nrhs, int nt, int nv,
                    int Et, double h, cudaStream_t st);
// representation formula u[rhs][p] = V~ w - W g at the points pts [np][4] = (x, y, z, t)
// (caller's triangle and node order; g may be null: single-layer potential only)
void launch_repr(const double *verts, const int *tri, int nt, int nv, const double *rule, int nq, const double *w,
                 const double *g, const double *pts, int np, int nrhs, int Et, double h, double alpha, double *u,
                 cudaStream_t st);

}  // namespace pfmm
