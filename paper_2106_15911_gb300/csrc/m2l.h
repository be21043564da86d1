// m2l.h -- the folded M2L of the 4^3 levels (k_m2l.cu): its unit tables and launch interface.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <vector>

#include "kernels.h"

namespace pfmm {

// largest shared memory of a CTA
constexpr size_t kM2LFoldSmemMax = 227 * 1024;

// Unit tables of the three passes (see k_m2l.cu): pass 1, pass 2 per slice, pass 3; two words a unit
struct M2LFoldPlan {
    int nk = 0, ne = 0, urows = 0, nslice = 1, first3 = 0, q3 = 0;
    int ntask[2] = {0, 0};  // passes 1 and 3
    int first2[kM2LMaxSlices] = {0}, ntask2[kM2LMaxSlices] = {0};
    std::vector<int> units, urow;
    size_t smem = 0;
};

// sliced: T2 is formed a few values of nu1 at a time, so that it needs no more rows than the moments
M2LFoldPlan m2l_fold_plan(int prec, int mx, const std::vector<int> &kinv, bool sliced);

struct M2LFoldArgs {
    int na, nk, mx, ne, nint, nbox, urows, nslice, nunits, first3, tpc, nchunk, k_lo;
    int ntask[2], first2[kM2LMaxSlices], ntask2[kM2LMaxSlices];
    const int2 *units;
    const int *urow, *cellbox;  // [nk], [64]
    const float *EF;
    const void *pref;           // (R)
    void *part;                 // chunk slices of the locals (R), or null: write the locals
    size_t nlev;                // elements of a slice
};

size_t m2l_fold_table_floats(int na, int mx, int prec);
void launch_m2l_fold_table(const double *E1, int na, int mx, int ntr, int prec, float *EF, cudaStream_t st);
int launch_m2l_folded(int prec, const DevLevel &L, const M2LFoldDev &P, const void *mu, void *lam, int nrhs,
                      const ApplyGeo &g, void *ws, size_t ws_elems, cudaStream_t st);

}  // namespace pfmm
