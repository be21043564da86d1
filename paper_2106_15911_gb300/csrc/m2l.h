// m2l.h -- the folded M2L of the 4^3 and 8^3 levels (k_m2l.cu): unit tables and launch interfaces.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <vector>

#include "kernels.h"

namespace pfmm {

// largest shared memory of a CTA
constexpr size_t kM2LFoldSmemMax = 227 * 1024;

// Unit tables of the three passes (see k_m2l.cu): pass 1 (per slice in the 8^3 kernel), pass 2 per
// slice, pass 3; two words a unit
struct M2LFoldPlan {
    M2LFoldDev d{};  // counts, without the device arrays
    std::vector<int> units, urow;
};

// 4^3 levels.  sliced: T2 is formed a few values of nu1 at a time, so that it needs no more rows than
// the moments
M2LFoldPlan m2l_fold_plan(int prec, int mx, const std::vector<int> &kinv, bool sliced);
// 8^3 levels (FP32): T1 and T2 both by slices of nu1
M2LFoldPlan m2l_slab_plan(int mx, const std::vector<int> &kinv);

struct M2LFoldArgs {
    int na, nk, mx, ne, nint, nbox, tpc, nchunk, k_lo;
    int truncated;              // the interaction radius leaves cells out: moments that are not finite count as zeros
    M2LFoldDev p;
    const int *cellbox;         // [G^3]
    const float *EF;
    const void *pref;           // (R)
    void *part;                 // chunk slices of the locals (R), or null: write the locals
    size_t nlev;                // elements of a slice
};

// folded coefficients of a level with G = 4 or 8 cells per direction
size_t m2l_fold_table_floats(int na, int mx, int G, int prec);
void launch_m2l_fold_table(const double *E1, int na, int mx, int G, int ntr, int prec, float *EF, cudaStream_t st);
int launch_m2l_folded(int prec, bool sliced, const DevLevel &L, const M2LFoldDev &P, const void *mu, void *lam, int nrhs,
                      const ApplyGeo &g, void *ws, size_t ws_elems, cudaStream_t st);
// 8^3 level, FP32; ws: scratch of ws_elems floats for the folded moments of some source intervals.
// Returns 1 (nothing launched) when ws does not hold those of one target interval
int launch_m2l_slab_folded(const DevLevel &L, const M2LFoldDev &P, const float *mu, float *lam, int nrhs,
                           const ApplyGeo &g, float *ws, size_t ws_elems, cudaStream_t st);

}  // namespace pfmm
