// nf_crt.h -- launch interface of the FP64-accurate tensor-core nearfield (k_nf_crt.cu): the
// block-Toeplitz product computed exactly modulo 16 primes on tcgen05 and combined by the Chinese
// remainder theorem.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"

namespace pfmm {

constexpr int kCrtModuli = 16;

struct NfCrtParams {
    const unsigned char *A;  // residue bytes of the blocks [modulus][tile][column block][d][128][64]
    int ntiles, nkb, nitems; // 128-row tiles, 64-column blocks; nitems is set by the launch
    int nint, Et, nt, nrhs;
    const int *shared;       // CrtInput.shared
    unsigned char *res;      // out: residues [modulus][rhs][Et][nt] in [0, p)
    int *err;                // set non-zero when a bounded wait gave up
};

// moduli tables into constant memory of the current device (once per device); 0 or -1
int crt_upload_constants(cudaStream_t st);
// fixed-point bits b of both operands for a reduction over k_total terms: 2 k_total 2^(2b) < M
int crt_bits(long long k_total);
// per-row exponents of the stored FP64 panels by triangle (largest |A| of the row over d and columns
// in [2^(b-1), 2^b) after scaling)
void launch_crt_row_exps(const double *A, const PanelGPU *panels, int npanel, int kop, int nd, int b,
                         unsigned long long *rowmax, int nt, int *rowexp, cudaStream_t st);
// residues of the scaled, rounded panels of nd step offsets (all of ncp columns) for NfCrtParams.A
size_t crt_panel_bytes(int nt, int ncp, int nd);
void launch_crt_split_panel(const double *A, const PanelGPU *panels, const int *tri_leaf, const int *rowexp, int kop,
                            int nt, int ncp, int nd, unsigned char *res, cudaStream_t st);
// one product's input, and the stored blocks for the entries that are not finite
struct CrtInput {
    const double *x;          // [rhs][Et][ncol]
    const int *perm;          // internal -> caller column (V), or null
    int ncol, ncol_pad, nrhs, Et, ls, nt, b, kop;
    // scratch (k_crt_scales): CTAs done (0 between launches); largest finite |x| as FP64 bits of each rhs, of the
    // (rhs, leaf interval)s and of their parts; scale exponents of the outputs (x 2, + 1 where values that are not
    // finite reach them); 1 where all intervals of a tile [rhs][tile] have the scale of the one before
    unsigned *ticket;
    unsigned long long *all, *wmax, *part;
    int *win, *shared;
    const double *A;          // FP64 panels
    const PanelGPU *panels;
    const int *tri_leaf;
};
// scratch of a product: its words (the first zero before the first launch), and the pointers into it
size_t crt_scratch_words(int nrhs, int Et, int ls);
void crt_scratch(CrtInput &in, unsigned long long *p);
// scales and residues [kCrtModuli][nrhs][leaf intervals][2 ls][ncol_pad] of the scaled, rounded,
// permuted (V) or padded (K) input: every interval's own steps after those of the one before (these only in
// tiles of ni intervals that are not shared)
void launch_crt_split_input(const CrtInput &in, int ni, void *res, cudaStream_t st);
// f[rhs][t][row] (overwritten) from the residues of the exact products
void launch_crt_combine(const unsigned char *res, const CrtInput &in, const int *rowexp, double *f, cudaStream_t st);
// leaf intervals per work item: rows of the W tensor map's box
int nf_crt_intervals(int nint, int ls, int form);
// form 1: work items of up to 128 leaf intervals; form 2: of up to 64 (twice the items, each of half
// the MMAs on the same blocks)
int launch_nf_apply_crt(const CUtensorMap &W, const NfCrtParams &P, int ls, int nsm, cudaStream_t st, int form);

}  // namespace pfmm
