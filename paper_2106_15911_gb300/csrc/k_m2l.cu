// k_m2l.cu -- M2L of the levels with 4^3 cells (Eq. m2l with Eq. exp_coeffs_3d, one direction at a
// time; the passes and their budget rows are described at M2LArgs in k_apply.cu), with every direction folded
// into its even and odd part.
//
// The one-directional coefficients satisfy E_{k,nu}(-o) = (-1)^{k+nu} E_{k,nu}(o), so on the four
// cells of a direction they are a 4 x 4 Toeplitz matrix that the reflection of the cells maps to
// itself (k + nu even) or to its negative (odd).  In the folded coordinates
//   (y0 + y3, y1 + y2 | y0 - y3, y1 - y2)   (index = 2 sector + j, sector 0: even, 1: odd)
// it is two 2 x 2 blocks, input sector s to output sector s ^ ((k + nu) & 1), with
//   M^s_ij = (t_{i-j} + (-1)^s t_{i-(3-j)}) / 2,  t_o = E_{k,nu}(o),
// so a step costs 8 multiply-adds per fibre of four cells instead of 16, and 8 coefficients
// instead of 7.  The moments are folded once when a CTA loads them, the locals unfolded once when
// it writes them; the factor 1/2 of the inverse sits in M.
//
// One CTA per (target interval k, time node b, chunk of source terms (J, a), rhs).  T1 and T2 live
// in shared memory, one row of 64 cells per (triple, budget) entry; a row is 16 chunks of four
// consecutive values, and the four values of a chunk are a fibre of the direction that the next
// pass sums over, so a fibre is one vector load:
//   U  row (k2, k3; k1):        [Y3][Y2][Y1]       pass 1 sums over k1, Y1
//   T1 row (nu1, k3; k2, C):    [X1][Y3][Y2]       pass 2 sums over k2, Y2   (C: budget of T1)
//   T2 row (nu1, nu2, B'; k3):  [X2][X1][Y3]       pass 3 sums over k3, Y3
// The rows of one sum are consecutive (passes 1 and 3) or at steps that shrink by one row (pass 2),
// so all passes are the same short chain: a unit (its rows and its nu) is given to 16 / NF lanes,
// each with NF fibres in registers, and a warp takes a task of 2 NF units of one length.  Where the lengths allow it the units of a task share nu
// (their coefficient loads are one broadcast) and differ in the row key (k3 of T1, nu1 of T2, modulo
// 4): the chunks of a row are stored at chunk ^ 2 key, so the units' stores go to different banks.
// Tasks are dealt to the warps longest first, back and forth.  The parity of k + nu alternates with
// k, so the accumulators are kept relative to the parity of nu and swapped by addressing when they
// are written.  Double-FP32 rows hold 64 high then 64 low parts.
//
// Folding mixes all cells of a fibre, so where the interaction radius leaves some out, what is not finite would
// reach them and their zeros would come out as rounding noise: there such moments are folded as zeros and
// k_m2l_outside settles the cells afterwards.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include "df64.cuh"
#include "kernels.h"
#include "m2l.h"

namespace pfmm {

namespace {

constexpr int kSlabThreads = 512;  // 8^3 kernel

template <typename R>
// planes: FP32 words per value; NF: fibres per lane; threads and CTAs per SM (sliced: threads of the
// sliced form, whose shared memory leaves room for one CTA per SM)
struct Form;
template <>
struct Form<float> {
    static constexpr int planes = 1, NF = 2, threads = 256, ctas = 2, sliced = 512;
};
template <>
struct Form<df64> {
    static constexpr int planes = 2, NF = 1, threads = 384, ctas = 1, sliced = 384;
};

__device__ __forceinline__ void load4(const float *p, float (&v)[4])
{
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void load4(const float *p, df64 (&v)[4])
{
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 64);
    v[0] = df_make(a.x, b.x); v[1] = df_make(a.y, b.y); v[2] = df_make(a.z, b.z); v[3] = df_make(a.w, b.w);
}
__device__ __forceinline__ void store1(float *p, float v) { *p = v; }
__device__ __forceinline__ void store1(float *p, df64 v)
{
    v = df_fast_two_sum(v.hi, v.lo);
    p[0] = v.hi;
    p[64] = v.lo;
}
__device__ __forceinline__ void store4(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(float *p, const df64 (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0].hi, v[1].hi, v[2].hi, v[3].hi);
    *reinterpret_cast<float4 *>(p + 64) = make_float4(v[0].lo, v[1].lo, v[2].lo, v[3].lo);
}
// the eight coefficients of (nu, k)
__device__ __forceinline__ void load8(const float *p, float (&e)[8])
{
    const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
    e[0] = a.x; e[1] = a.y; e[2] = a.z; e[3] = a.w;
    e[4] = b.x; e[5] = b.y; e[6] = b.z; e[7] = b.w;
}
__device__ __forceinline__ void load8(const float *p, df64 (&e)[8])
{
    float h[8], l[8];
    load8(p, h);
    load8(p + 8, l);
#pragma unroll
    for (int i = 0; i < 8; ++i) e[i] = df_make(h[i], l[i]);
}
// acc += a b.  Double-FP32: the high parts by an error-free sum, everything else into the low part,
// which is normalised only when the sum is stored (12 operations instead of 15)
__device__ __forceinline__ void step(float &acc, float a, float b) { acc = fmaf(a, b, acc); }
__device__ __forceinline__ void step(df64 &acc, df64 a, df64 b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    float s, t;
    df_two_sum(acc.hi, p, s, t);
    acc.hi = s;
    acc.lo = __fadd_rn(acc.lo, __fadd_rn(t, e));
}
__device__ __forceinline__ float norm(float v) { return v; }
__device__ __forceinline__ df64 norm(df64 v) { return df_fast_two_sum(v.hi, v.lo); }
__device__ __forceinline__ float head(float v) { return v; }
__device__ __forceinline__ float head(df64 v) { return v.hi; }
__device__ __forceinline__ float diff(float a, float b) { return a - b; }
__device__ __forceinline__ df64 diff(df64 a, df64 b) { return a + (-b); }
__device__ __forceinline__ float shfl_x(float v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ df64 shfl_x(df64 v, int m)
{
    return df_make(__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m));
}

// one (k, nu) step of a fibre; `odd`: k is odd, the input sectors feed the other accumulators
template <typename R>
__device__ __forceinline__ void fibre_step(R (&acc)[4], const R (&in)[4], const R (&e)[8], bool odd)
{
    const int o = odd ? 2 : 0;
    step(acc[o], e[0], in[0]);
    step(acc[o + 1], e[2], in[0]);
    step(acc[2 - o], e[4], in[2]);
    step(acc[3 - o], e[6], in[2]);
    step(acc[o], e[1], in[1]);
    step(acc[o + 1], e[3], in[1]);
    step(acc[2 - o], e[5], in[3]);
    step(acc[3 - o], e[7], in[3]);
}

// the chain of a unit: len steps from row address p (rows `stride` words apart, then `stride - dec` and
// so on; the second fibre fstep words further on) with the coefficients at e; after(j) sees the partial
// sums of every step.  Two steps at a time: unrolled for every length the passes outgrow the
// instruction cache (M2L of 12288 x 256: double-FP32 1.79 instead of 0.93 ms, FP32 with 4 rhs 1.11
// instead of 1.07 ms)
template <typename R, typename After>
__device__ __forceinline__ void chain_of(int len, R (&acc)[Form<R>::NF][4], const float *p, int stride, int dec, int fstep,
                                         const float *e, After after)
{
    constexpr int PL = Form<R>::planes, NF = Form<R>::NF;
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[f][r] = R(0);
#pragma unroll 1
    for (int j = 0; j < len; j += 2) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && j + 1 >= len) break;
            R ev[8], in[NF][4];
            load8(e, ev);
            load4(p, in[0]);
            if (NF == 2) load4(p + fstep, in[NF - 1]);
#pragma unroll
            for (int f = 0; f < NF; ++f) fibre_step(acc[f], in[f], ev, h == 1);
            after(j + h);
            e += 8 * PL;
            p += stride;
            stride -= dec;
        }
    }
}

// offsets within a row of the four values of chunk c's output fibre: position pos of the chunk goes
// to chunk (4 pos + c / 4) ^ 2 key, word c % 4; the relative position r is pos ^ 2 (nu mod 2)
__device__ __forceinline__ void out_offsets(int (&q)[4], int c, int nu, int key)
{
    const int base = ((((c >> 2) ^ ((key & 1) << 1)) << 2) | (c & 3)), x = (((nu & 1) << 1) ^ (key >> 1)) << 4;
#pragma unroll
    for (int r = 0; r < 4; ++r) q[r] = base + ((r << 4) ^ x);
}

// a unit's words
struct UnitBits {
    int row, nu, key, okey, step, slice, len, out;
    bool valid;
    __device__ __forceinline__ explicit UnitBits(int2 d)
    {
        row = d.x & 1023;
        nu = (d.x >> 10) & 15;
        key = (d.x >> 14) & 3;
        okey = (d.x >> 16) & 3;
        step = (d.x >> 18) & 15;
        len = (d.x >> 22) & 15;
        slice = (d.x >> 26) & 7;
        valid = d.x < 0;
        out = d.y;
    }
};

}  // namespace

template <typename R, int Q3, int NT>
__global__ void __launch_bounds__(NT, NT == Form<R>::threads ? Form<R>::ctas : 1)
k_m2l_folded(M2LFoldArgs A, const R *__restrict__ mu, R *__restrict__ lam)
{
    using F = Form<R>;
    constexpr int PL = F::planes, NF = F::NF, LPU = 16 / NF, UPW = 32 / LPU, W = NT / 32, RW = 64 * PL;
    extern __shared__ __align__(16) float sm[];
    const int nk = A.nk, na = A.na, m1 = A.mx + 1;
    float *T1 = sm, *U = T1 + A.ne * RW, *Es = U + A.p.urows * RW;
    int2 *un = reinterpret_cast<int2 *>(Es + m1 * m1 * 8 * PL);
    int *cbo = reinterpret_cast<int *>(un + A.p.nunits);  // [z][x][y] element offset of the cell's box, -1: empty
    int *urow = cbo + 64;                               // [nk] row of U of a moment
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane / LPU, cl = lane % LPU;
    // grid x: (interval, node, chunk); even intervals have half the terms of odd ones
    const int chunk = blockIdx.x % A.nchunk, kb = blockIdx.x / A.nchunk;
    const int b = kb % na, k = A.k_lo + kb / na, rhs = blockIdx.y;
    const int nterm = k < 2 ? 0 : (k & 1 ? 2 * na : na);
    const int t_lo = chunk * A.tpc, t_hi = min(nterm, t_lo + A.tpc);
    if (A.part && t_lo >= t_hi) return;
    for (int i = threadIdx.x; i < A.p.nunits; i += NT) un[i] = reinterpret_cast<const int2 *>(A.p.units)[i];
    for (int i = threadIdx.x; i < nk; i += NT) urow[i] = A.p.urow[i];
    for (int i = threadIdx.x; i < 64; i += NT) {
        const int box = A.cellbox[i];
        cbo[(i & 3) * 16 + (i >> 2)] = box < 0 ? -1 : box * na * nk;
    }

    R lamr[Q3][NF][4];
#pragma unroll
    for (int q = 0; q < Q3; ++q)
#pragma unroll
        for (int f = 0; f < NF; ++f)
#pragma unroll
            for (int r = 0; r < 4; ++r) lamr[q][f][r] = R(0);

    for (int t = t_lo; t < t_hi; ++t) {
        // terms (J, a): odd intervals J = k - 3 then k - 2, even ones k - 2
        const int a = t % na, D = (k & 1) ? 3 - t / na : 2, J = k - D;
        __syncthreads();  // tables in place; the previous term's pass 3 is done with U and Es
        const float4 *Eg = reinterpret_cast<const float4 *>(A.EF) + (size_t)(((D - 2) * na + a) * na + b) * m1 * m1 * 2 * PL;
        for (int i = threadIdx.x; i < m1 * m1 * 2 * PL; i += NT) reinterpret_cast<float4 *>(Es)[i] = Eg[i];
        const R coef = reinterpret_cast<const R *>(A.pref)[((D - 2) * na + a) * na + b];
        // moments of (J, a): lane = (multi-index, Y3) takes the 16 cells (Y1, Y2), folds them in x and
        // y and, with the lane of the mirrored Y3, in z
        const R *mJ = mu + (((size_t)rhs * A.nint + J) * A.nbox * na + a) * nk;
        for (int i = threadIdx.x; i < ((nk + 7) & ~7) * 4; i += NT) {
            const int z = i & 3, ik = i >> 2;
            const bool ok = ik < nk;
            const R *mi = mJ + (ok ? ik : 0);
            R v[4][4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const int4 o = *reinterpret_cast<const int4 *>(cbo + z * 16 + x * 4);
                v[x][0] = o.x >= 0 ? mi[o.x] : R(0);
                v[x][1] = o.y >= 0 ? mi[o.y] : R(0);
                v[x][2] = o.z >= 0 ? mi[o.z] : R(0);
                v[x][3] = o.w >= 0 ? mi[o.w] : R(0);
            }
            if (A.truncated) {
#pragma unroll
                for (int x = 0; x < 4; ++x)
#pragma unroll
                    for (int y = 0; y < 4; ++y)
                        if (!isfinite(head(v[x][y]))) v[x][y] = R(0);
            }
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const R a0 = v[0][y], a1 = v[1][y], a2 = v[2][y], a3 = v[3][y];
                v[0][y] = a0 + a3; v[1][y] = a1 + a2; v[2][y] = diff(a0, a3); v[3][y] = diff(a1, a2);
            }
            float *p = U + (ok ? urow[ik] : 0) * RW + (z < 2 ? z : 5 - z) * 16;
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const R a0 = v[x][0], a1 = v[x][1], a2 = v[x][2], a3 = v[x][3];
                v[x][0] = a0 + a3; v[x][1] = a1 + a2; v[x][2] = diff(a0, a3); v[x][3] = diff(a1, a2);
            }
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                R s[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const R o = shfl_x(v[x][y], 3);
                    s[x] = z < 2 ? v[x][y] + o : diff(o, v[x][y]);
                }
                if (ok) store4(p + y * 4, s);
            }
        }
        __syncthreads();
        // pass 1: unit (k2, k3, nu1); the sum over k1 is cumulative, every partial sum is a row of T1
        for (int ts = warp; ts < A.p.ntask1[0]; ts += W) {
            const UnitBits u(un[ts * UPW + sub]);
            int q[NF][4];
#pragma unroll
            for (int f = 0; f < NF; ++f) out_offsets(q[f], cl + f * LPU, u.nu, u.okey);
            float *o = T1 + u.out * RW;
            R acc[NF][4];
            chain_of(u.len, acc, U + u.row * RW + cl * 4, RW, 0, LPU * 4, Es + u.nu * m1 * 8 * PL, [&](int j) {
                if (u.valid) {
#pragma unroll
                    for (int f = 0; f < NF; ++f)
#pragma unroll
                        for (int r = 0; r < 4; ++r) store1(o + q[f][r] + j * RW, acc[f][r]);
                }
            });
        }
        __syncthreads();
        for (int sl = 0; sl < A.p.nslice; ++sl) {
            if (sl > 0) __syncthreads();  // pass 3 of the previous slice is done with U
            // pass 2: unit = row of T2
            for (int ts = warp; ts < A.p.ntask2[sl]; ts += W) {
                const UnitBits u(un[A.p.first2[sl] + ts * UPW + sub]);
                R acc[NF][4];
                chain_of(u.len, acc, T1 + u.row * RW + ((cl ^ (u.key << 1)) << 2), u.step * RW, RW, LPU * 4,
                            Es + u.nu * m1 * 8 * PL, [](int) {});
                if (u.valid) {
                    float *o = U + u.out * RW;
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        int q[4];
                        out_offsets(q, cl + f * LPU, u.nu, u.okey);
#pragma unroll
                        for (int r = 0; r < 4; ++r) store1(o + q[r], acc[f][r]);
                    }
                }
            }
            __syncthreads();
            // pass 3: unit = multi-index of the locals, fixed per lane over all terms
#pragma unroll
            for (int q = 0; q < Q3; ++q) {
                const int ts = warp + q * W;
                if (ts >= A.p.ntask3) break;
                const UnitBits u(un[A.p.first3 + ts * UPW + sub]);
                if (u.slice != sl) continue;
                R acc[NF][4];
                chain_of(u.len, acc, U + u.row * RW + ((cl ^ (u.key << 1)) << 2), RW, 0, LPU * 4,
                            Es + u.nu * m1 * 8 * PL, [](int) {});
#pragma unroll
                for (int f = 0; f < NF; ++f)
#pragma unroll
                    for (int r = 0; r < 4; ++r) step(lamr[q][f][r], coef, norm(acc[f][r]));
            }
        }
    }
    // unfold: in z per lane (row = multi-index: [X3][X2][X1]), then in y and x per (multi-index, X3)
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q3; ++q) {
        const int ts = warp + q * W;
        if (ts >= A.p.ntask3) break;
        const UnitBits u(un[A.p.first3 + ts * UPW + sub]);
        if (!u.valid) continue;
        const bool odd = u.nu & 1;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const R(&l)[4] = lamr[q][f];
            const R p0 = norm(odd ? l[2] : l[0]), p1 = norm(odd ? l[3] : l[1]), n0 = norm(odd ? l[0] : l[2]),
                    n1 = norm(odd ? l[1] : l[3]);
            float *p = U + u.out * RW + cl + f * LPU;
            store1(p, p0 + n0);
            store1(p + 16, p1 + n1);
            store1(p + 32, diff(p1, n1));
            store1(p + 48, diff(p0, n0));
        }
    }
    __syncthreads();
    R *out = (A.part ? reinterpret_cast<R *>(A.part) + (size_t)chunk * A.nlev : lam) +
             (((size_t)rhs * A.nint + k) * A.nbox * na + b) * nk;
    for (int i = threadIdx.x; i < nk * 4; i += NT) {
        const int z = i & 3, iv = i >> 2;
        const float *p = U + iv * RW + z * 16;
        R v[4][4];  // [y][x]
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            R q[4];
            load4(p + y * 4, q);
            v[y][0] = q[0] + q[2]; v[y][1] = q[1] + q[3]; v[y][2] = diff(q[1], q[3]); v[y][3] = diff(q[0], q[2]);
        }
        const int4 *co = reinterpret_cast<const int4 *>(cbo + z * 16);
        R *ov = out + iv;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const R q0 = v[0][x], q1 = v[1][x], q2 = v[2][x], q3 = v[3][x];
            const int4 o = co[x];
            if (o.x >= 0) ov[o.x] = q0 + q2;
            if (o.y >= 0) ov[o.y] = q1 + q3;
            if (o.z >= 0) ov[o.z] = diff(q1, q3);
            if (o.w >= 0) ov[o.w] = diff(q0, q2);
        }
    }
}

// lam = sum of the chunk slices in order; interval k has ceil(terms / tpc) slices (none for k < 2)
template <typename R>
__global__ void k_m2l_sum_chunks(const R *__restrict__ part, int na, int tpc, size_t n, size_t per_k, int nint,
                                 R *__restrict__ lam)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int k = (int)((i / per_k) % nint);
    const int nterm = k < 2 ? 0 : (k & 1 ? 2 * na : na), nc = (nterm + tpc - 1) / tpc;
    R s = R(0);
    for (int t = 0; t < nc; ++t) s += part[(size_t)t * n + i];
    lam[i] = s;
}

// Locals of a level whose interaction radius leaves cells out: zero where no moment within the radius is other
// than zero, NaN where one is not finite.  CTA: (target interval, rhs); reads the moments of its one or two source
// intervals once.  Bound by the latency of these reads: many warps, eight loads each in flight
constexpr int kOutsideThreads = 1024;
template <typename R>
__global__ void __launch_bounds__(kOutsideThreads) k_m2l_outside(const R *__restrict__ mu, R *__restrict__ lam,
                                                     const int *__restrict__ boxcell, int G, int ntr, int na, int nk, int nint,
                                                     int nbox)
{
    __shared__ int flag[2][512];  // bit 0: a moment that is not zero, bit 1: one that is not finite
    const int k = blockIdx.x + 2, rhs = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = na * nk, G3 = G * G * G;
    for (int i = threadIdx.x; i < G3; i += kOutsideThreads) flag[0][i] = 0;
    __syncthreads();
    for (int w = warp; w < nbox * (1 + (k & 1)); w += kOutsideThreads / 32) {
        const int b = w % nbox;
        const R *m = mu + (((size_t)rhs * nint + k - 2 - w / nbox) * nbox + b) * n;
        int f = 0;
#pragma unroll 8
        for (int i = lane; i < n; i += 32) {
            const float v = head(m[i]);
            f |= isfinite(v) ? (v != 0.f ? 1 : 0) : 3;
        }
        f = __reduce_or_sync(0xffffffffu, f);
        if (lane == 0 && f) atomicOr(&flag[0][boxcell[b]], f);
    }
    __syncthreads();
    for (int dir = 0, st = 1; dir < 3; ++dir, st *= G) {  // the cells within the radius, one direction at a time
        for (int i = threadIdx.x; i < G3; i += kOutsideThreads) {
            const int c = i / st % G;
            int f = 0;
            for (int o = max(-ntr, -c); o <= min(ntr, G - 1 - c); ++o) f |= flag[dir & 1][i + o * st];
            flag[~dir & 1][i] = f;
        }
        __syncthreads();
    }
    for (int b = warp; b < nbox; b += kOutsideThreads / 32) {
        const int f = flag[1][boxcell[b]];
        if (f == 1) continue;
        R *o = lam + (((size_t)rhs * nint + k) * nbox + b) * n;
        for (int i = lane; i < n; i += 32) o[i] = f ? R(__int_as_float(0x7fffffff)) : R(0);
    }
}

template <typename R>
static void settle_outside(const DevLevel &L, const R *mu, R *lam, int nrhs, const ApplyGeo &g, cudaStream_t st)
{
    if (L.ntr < L.G - 1 && L.nint > 2)
        k_m2l_outside<R><<<dim3(L.nint - 2, nrhs), kOutsideThreads, 0, st>>>(mu, lam, L.boxcell, L.G, L.ntr, g.na, g.nk, L.nint, L.nbox);
}

// folded coefficients of a level from its FP64 table E1 [D][a][b][o][k][nu] (offsets beyond the
// interaction radius are zero): EF [D][a][b][nu][k][2 (G/2)^2] (sector, i, j), in FP32 or as high and low
// parts
__global__ void k_m2l_fold_table(const double *__restrict__ E1, int na, int m1, int G, int ntr, int planes,
                                 float *__restrict__ EF)
{
    const int gid = blockIdx.x * blockDim.x + threadIdx.x, esz = m1 * m1, H = G / 2, n = 2 * H * H;
    if (gid >= 2 * na * na * esz) return;
    const int k = gid % m1, nu = (gid / m1) % m1;
    const double *E = E1 + ((size_t)(gid / esz) * (2 * G - 1) + G - 1) * esz + k * m1 + nu;
    float *o = EF + (size_t)gid * n * planes;
    for (int s = 0; s < 2; ++s)
        for (int i = 0; i < H; ++i)
            for (int j = 0; j < H; ++j) {
                const int o1 = i - j, o2 = i - (G - 1 - j);
                const double t1 = (o1 < 0 ? -o1 : o1) <= ntr ? E[o1 * esz] : 0.0;
                const double t2 = (o2 < 0 ? -o2 : o2) <= ntr ? E[o2 * esz] : 0.0;
                const double m = 0.5 * (s == 0 ? t1 + t2 : t1 - t2);
                const int at = (s * H + i) * H + j;
                o[at] = (float)m;
                if (planes == 2) o[at + n] = (float)(m - (double)(float)m);
            }
}

void launch_m2l_fold_table(const double *E1, int na, int mx, int G, int ntr, int prec, float *EF, cudaStream_t st)
{
    const int n = 2 * na * na * (mx + 1) * (mx + 1);
    k_m2l_fold_table<<<(n + 127) / 128, 128, 0, st>>>(E1, na, mx + 1, G, ntr, prec == 1 ? 1 : 2, EF);
}

size_t m2l_fold_table_floats(int na, int mx, int G, int prec)
{
    return (size_t)na * na * (mx + 1) * (mx + 1) * G * G * (prec == 1 ? 1 : 2);
}

namespace {

struct Unit {
    int row, nu, key, okey, step, slice, len, out;
    bool valid;
    int word() const
    {
        return row | nu << 10 | key << 14 | okey << 16 | step << 18 | len << 22 | slice << 26 | (valid ? INT32_MIN : 0);
    }
};

// units into tasks of `upw` of one length and slice, of one nu and different okey where that can be
// had; incomplete tasks are filled with units that store nothing.  Longest tasks first, dealt to
// `warps` warps back and forth.  Appends the units' words, returns the number of tasks
int deal(const std::vector<Unit> &u, int upw, int warps, std::vector<int> &out)
{
    std::vector<std::vector<Unit>> tasks;
    int maxlen = 0, maxslice = 0;
    for (const Unit &q : u) {
        maxlen = std::max(maxlen, q.len);
        maxslice = std::max(maxslice, q.slice);
    }
    for (int sl = 0; sl <= maxslice; ++sl)
        for (int len = maxlen; len >= 1; --len) {
            std::vector<Unit> g;
            for (const Unit &q : u)
                if (q.slice == sl && q.len == len) g.push_back(q);
            while (!g.empty()) {
                std::vector<Unit> t;
                while ((int)t.size() < upw && !g.empty()) {
                    size_t best = 0;
                    int score = -1;
                    for (size_t i = 0; i < g.size(); ++i) {
                        bool fresh = true;
                        for (const Unit &q : t) fresh = fresh && q.okey != g[i].okey;
                        const int sc = (fresh ? 2 : 0) + (t.empty() || t[0].nu == g[i].nu ? 1 : 0);
                        if (sc > score) {
                            score = sc;
                            best = i;
                        }
                    }
                    t.push_back(g[best]);
                    g.erase(g.begin() + best);
                }
                while ((int)t.size() < upw) {
                    Unit d = t[0];
                    d.valid = false;
                    t.push_back(d);
                }
                tasks.push_back(t);
            }
        }
    std::stable_sort(tasks.begin(), tasks.end(), [](const std::vector<Unit> &a, const std::vector<Unit> &b) { return a[0].len > b[0].len; });
    const int n = (int)tasks.size();
    const size_t at = out.size();
    out.resize(at + 2 * (size_t)n * upw);
    for (int t = 0; t < n; ++t) {
        const int r = t / warps, w = t % warps, last = std::min(warps, n - r * warps);
        const int pos = r * warps + (r & 1 ? last - 1 - w : w);
        for (int i = 0; i < upw; ++i) {
            out[at + 2 * ((size_t)pos * upw + i)] = tasks[t][i].word();
            out[at + 2 * ((size_t)pos * upw + i) + 1] = tasks[t][i].out;
        }
    }
    return n;
}

}  // namespace

// slab: 8^3 levels (T1 by slices as well, keys of one bit that alternate with the budget)
static M2LFoldPlan make_plan(int upw, int warps, int mx, const std::vector<int> &kinv, bool sliced, bool slab)
{
    const int m1 = mx + 1, nk = (mx + 1) * (mx + 2) * (mx + 3) / 6;
    auto iv = [&](int a, int b, int c) { return kinv[((size_t)a * m1 + b) * m1 + c]; };
    auto tri = [](int n) { return n * (n + 1) / 2; };
    M2LFoldPlan P;
    M2LFoldDev &D = P.d;
    // slices of nu1: consecutive values whose rows of T2 (as many as of T1) fit the rows of the moments
    std::vector<int> slice(m1, 0);
    auto rows2 = [&](int nu1) {
        int n = 0;
        for (int nu2 = 0; nu1 + nu2 <= mx; ++nu2) n += tri(mx - nu1 - nu2 + 1);
        return n;
    };
    D.nslice = 1;
    D.urows = nk;
    for (int v = 0, fill = 0; v <= mx; ++v) {
        if (sliced && fill && fill + rows2(v) > nk) {
            D.nslice++;
            fill = 0;
        }
        fill += rows2(v);
        slice[v] = D.nslice - 1;
        D.urows = std::max(D.urows, fill);
    }
    // rows of U: (k2, k3), then k1; of T1: (nu1, k3), then k2, then C = nu1 + k3 + k2 .. m_x
    P.urow.assign(nk, 0);
    std::vector<int> ub((size_t)m1 * m1, 0), tb((size_t)m1 * m1, 0), f1(D.nslice, 0);
    int r = 0;
    for (int i = 0; i <= mx; ++i)
        for (int j = 0; i + j <= mx; ++j) {
            ub[i * m1 + j] = r;
            for (int k1 = 0; k1 + i + j <= mx; ++k1) P.urow[iv(k1, i, j)] = r++;
            int &rt = f1[slab ? slice[i] : 0];
            tb[i * m1 + j] = rt;
            rt += tri(mx - i - j + 1);
        }
    std::vector<Unit> u3;
    std::vector<std::vector<Unit>> u1(slab ? D.nslice : 1), u2(D.nslice);
    for (int k2 = 0; k2 <= mx; ++k2)
        for (int k3 = 0; k2 + k3 <= mx; ++k3)
            for (int nu1 = 0; nu1 + k2 + k3 <= mx; ++nu1) {
                const int n = mx - nu1 - k3;  // T1 rows of k2 start after n + 1, n, ... rows of smaller k2
                u1[slab ? slice[nu1] : 0].push_back({ub[k2 * m1 + k3], nu1, 0, k3 & 3, 0, 0, n - k2 + 1,
                                                     tb[nu1 * m1 + k3] + k2 * (n + 1) - tri(k2 - 1), true});
            }
    std::vector<int> t2b((size_t)m1 * m1, 0), fill(D.nslice, 0);
    for (int nu1 = 0; nu1 <= mx; ++nu1)
        for (int nu2 = 0; nu1 + nu2 <= mx; ++nu2) {
            t2b[nu1 * m1 + nu2] = fill[slice[nu1]];
            fill[slice[nu1]] += tri(mx - nu1 - nu2 + 1);
        }
    for (int nu1 = 0; nu1 <= mx; ++nu1)
        for (int nu2 = 0; nu1 + nu2 <= mx; ++nu2) {
            for (int k3 = 0; nu1 + nu2 + k3 <= mx; ++k3)
                for (int B = nu1 + nu2 + k3; B <= mx; ++B) {
                    const int C = B - nu2, s = nu1 + k3;  // k2 = 0 .. C - s; from k2 to k2 + 1: n - k2 rows
                    u2[slice[nu1]].push_back({tb[nu1 * m1 + k3] + C - s, nu2, k3 & 3, slab ? B & 1 : nu1 & 3, mx - s, 0,
                                              C - s + 1, t2b[nu1 * m1 + nu2] + tri(B - nu1 - nu2) + k3, true});
                }
            for (int nu3 = 0; nu1 + nu2 + nu3 <= mx; ++nu3)
                u3.push_back({t2b[nu1 * m1 + nu2] + tri(mx - nu3 - nu1 - nu2), nu3, slab ? (mx - nu3) & 1 : nu1 & 3, 0, 0,
                              slice[nu1], mx - nu1 - nu2 - nu3 + 1, iv(nu1, nu2, nu3), true});
        }
    for (int s = 0; s < (slab ? D.nslice : 1); ++s) {
        D.first1[s] = (int)P.units.size() / 2;
        D.ntask1[s] = deal(u1[s], upw, warps, P.units);
    }
    for (int s = 0; s < D.nslice; ++s) {
        D.first2[s] = (int)P.units.size() / 2;
        D.ntask2[s] = deal(u2[s], upw, warps, P.units);
    }
    D.first3 = (int)P.units.size() / 2;
    D.ntask3 = deal(u3, upw, warps, P.units);
    D.q3 = (D.ntask3 + warps - 1) / warps;
    D.nunits = (int)P.units.size() / 2;
    return P;
}

M2LFoldPlan m2l_fold_plan(int prec, int mx, const std::vector<int> &kinv, bool sliced)
{
    const int m1 = mx + 1, nf = prec == 1 ? Form<float>::NF : Form<df64>::NF, planes = prec == 1 ? 1 : 2;
    const int warps = (prec == 1 ? (sliced ? Form<float>::sliced : Form<float>::threads)
                                 : (sliced ? Form<df64>::sliced : Form<df64>::threads)) / 32;
    M2LFoldPlan P = make_plan(2 * nf, warps, mx, kinv, sliced, false);
    const size_t nk = P.urow.size(), ne = nk * (mx + 4) / 4;
    P.d.smem = sizeof(float) * planes * ((ne + P.d.urows) * 64 + (size_t)m1 * m1 * 8) + sizeof(int) * P.units.size() +
               sizeof(int) * (64 + nk);
    return P;
}

M2LFoldPlan m2l_slab_plan(int mx, const std::vector<int> &kinv)
{
    M2LFoldPlan P = make_plan(2, kSlabThreads / 32, mx, kinv, true, true);
    P.d.smem = sizeof(float) * ((size_t)2 * P.d.urows * 256 + (size_t)(mx + 1) * (mx + 1) * 32) + sizeof(int) * P.units.size();
    return P;
}

template <typename R>
static int launch_T(const M2LFoldArgs &A, bool sliced, dim3 grd, const void *mu, void *lam, cudaStream_t st)
{
    constexpr int NT = Form<R>::threads, NS = Form<R>::sliced;
    auto kf = sliced && NS != NT ? (A.p.q3 <= 4 ? k_m2l_folded<R, 4, NS> : nullptr)
              : A.p.q3 <= 4     ? k_m2l_folded<R, 4, NT>
              : A.p.q3 <= 6     ? k_m2l_folded<R, 6, NT>
                                : nullptr;
    if (!kf || cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)A.p.smem) != cudaSuccess) return -1;
    kf<<<grd, sliced ? NS : NT, A.p.smem, st>>>(A, (const R *)mu, (R *)lam);
    return 0;
}

int launch_m2l_folded(int prec, bool sliced, const DevLevel &L, const M2LFoldDev &P, const void *mu, void *lam, int nrhs,
                      const ApplyGeo &g, void *ws, size_t ws_elems, cudaStream_t st)
{
    M2LFoldArgs A{};
    A.na = g.na;
    A.nk = g.nk;
    A.mx = g.mx;
    A.ne = g.ne;
    A.nint = L.nint;
    A.nbox = L.nbox;
    A.truncated = L.ntr < L.G - 1;
    A.p = P;
    A.cellbox = L.cellbox;
    A.EF = L.EF;
    A.pref = L.pref;
    const size_t per_k = (size_t)L.nbox * g.na * g.nk, nlev = (size_t)nrhs * L.nint * per_k;
    // terms per CTA: all 2 m_t + 2 of an interval, or, while that leaves fewer than eight CTAs per SM,
    // three, with the chunks' locals added afterwards
    const int all = 2 * g.na, tpc = 3, nchunk = (all + tpc - 1) / tpc;
    const int64_t few = (int64_t)8 * (g.nsm > 0 ? g.nsm : 152);
    const bool split = (int64_t)L.nint * g.na * nrhs < few && (size_t)nchunk * nlev <= ws_elems;
    A.tpc = split ? tpc : all;
    A.nchunk = split ? nchunk : 1;
    A.k_lo = split ? 2 : 0;
    A.part = split ? ws : nullptr;
    A.nlev = nlev;
    const dim3 grd((unsigned)((L.nint - A.k_lo) * g.na * A.nchunk), nrhs);
    const int rc = prec == 1 ? launch_T<float>(A, sliced, grd, mu, lam, st) : launch_T<df64>(A, sliced, grd, mu, lam, st);
    if (rc) return rc;
    if (split) {
        const unsigned blocks = (unsigned)((nlev + 255) / 256);
        if (prec == 1)
            k_m2l_sum_chunks<float><<<blocks, 256, 0, st>>>((const float *)ws, g.na, A.tpc, nlev, per_k, L.nint, (float *)lam);
        else
            k_m2l_sum_chunks<df64><<<blocks, 256, 0, st>>>((const df64 *)ws, g.na, A.tpc, nlev, per_k, L.nint, (df64 *)lam);
    }
    if (prec == 1)
        settle_outside(L, (const float *)mu, (float *)lam, nrhs, g, st);
    else
        settle_outside(L, (const df64 *)mu, (df64 *)lam, nrhs, g, st);
    return 0;
}

// ------------------------------------------------------------------------------------------
// 8^3 levels (FP32).  A direction folds into two sectors of four; the coefficients of (k, nu) are two
// 4 x 4 blocks.  T1 and T2 of a whole level's cells do not fit shared memory, so a CTA takes the target
// x-sector s1 (four X1 of a folded direction) and forms T1 and T2 a slice of nu1 at a time; rows have
// 256 cells (4 X1 x 64).  The folded moments of the source intervals are laid out once in global memory
// (every term is read by 5 b x 2 s1 CTAs of up to two intervals) and pass 1 reads them from L2.  The
// two CTAs of (k, b) are a cluster: at the end they exchange their sector's locals through
// distributed shared memory and each writes one half of the x range.  FP32 FMA and issue bound: a step
// of a lane is 64 FMAs on 8 or 12 vector loads (the unfolded kernel had one FMA per load).

// moments of (rhs, J, a) folded in x, y, z: F[((rhs, J, a)][row of U][X1][y >> 2][z][y & 3], positions of
// the folded directions; 12 multi-indices per CTA
constexpr int kFoldK = 12;
__global__ void __launch_bounds__(256) k_m2l_fold_moments(const float *__restrict__ mu, const int *__restrict__ cellbox,
                                                          const int *__restrict__ urow, int na, int nk, int nint, int nbox,
                                                          int J0, int nJ, int r0, int truncated, float *__restrict__ F)
{
    __shared__ float S[kFoldK][8][8][9];  // [k][x][y][z]
    const int J = J0 + blockIdx.x / na, a = blockIdx.x % na, k0 = blockIdx.y * kFoldK, kn = min(kFoldK, nk - k0);
    const float *mJ = mu + (((size_t)(r0 + blockIdx.z) * nint + J) * nbox * na + a) * nk + k0;
    for (int i = threadIdx.x; i < 512 * kFoldK; i += 256) {
        const int c = i / kFoldK, k = i % kFoldK, box = cellbox[c];
        const float v = box >= 0 && k < kn ? mJ[(size_t)box * na * nk + k] : 0.f;
        S[k][c >> 6][(c >> 3) & 7][c & 7] = truncated && !isfinite(v) ? 0.f : v;
    }
    __syncthreads();
#pragma unroll
    for (int dir = 0; dir < 3; ++dir) {
        for (int i = threadIdx.x; i < 64 * kFoldK; i += 256) {
            const int k = i >> 6, u = (i >> 3) & 7, w = i & 7;
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = dir == 0 ? S[k][j][u][w] : dir == 1 ? S[k][u][j][w] : S[k][u][w][j];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float p = v[j] + v[7 - j], m = v[j] - v[7 - j];
                if (dir == 0) {
                    S[k][j][u][w] = p;
                    S[k][4 + j][u][w] = m;
                } else if (dir == 1) {
                    S[k][u][j][w] = p;
                    S[k][u][4 + j][w] = m;
                } else {
                    S[k][u][w][j] = p;
                    S[k][u][w][4 + j] = m;
                }
            }
        }
        __syncthreads();
    }
    float *o = F + (((size_t)blockIdx.z * nJ + (J - J0)) * na + a) * nk * 512;
    for (int i = threadIdx.x; i < 512 * kn; i += 256) {
        const int k = i >> 9, c = i & 511, x = c >> 6, y = ((c >> 5) & 1) * 4 + (c & 3), z = (c >> 2) & 7;
        o[(size_t)urow[k0 + k] * 512 + c] = S[k][x][y][z];
    }
}

// one (k, nu) step of a fibre of eight: both sectors, 4 x 4 each
__device__ __forceinline__ void fibre8(float (&acc)[8], const float (&in)[8], const float (&e)[4], int s, int i, int o)
{
    float &a = acc[((s ^ o) << 2) + i];
#pragma unroll
    for (int j = 0; j < 4; ++j) a = fmaf(e[j], in[s * 4 + j], a);
}

// chain of passes 2 and 3: two fibres per lane (fstep words apart), the halves of a fibre at p + c0 and
// p + c1
__device__ __forceinline__ void chain8(int len, float (&acc)[2][8], const float *p, int c0, int c1, int stride, int dec,
                                       int fstep, const float *e)
{
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[f][r] = 0.f;
#pragma unroll 1
    for (int j = 0; j < len; j += 2) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && j + 1 >= len) break;
            float in[2][8];
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                float h0[4], h1[4];
                load4(p + f * fstep + c0, h0);
                load4(p + f * fstep + c1, h1);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    in[f][q] = h0[q];
                    in[f][4 + q] = h1[q];
                }
            }
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float ev[4];
                    load4(e + s * 16 + i * 4, ev);
                    fibre8(acc[0], in[0], ev, s, i, h);
                    fibre8(acc[1], in[1], ev, s, i, h);
                }
            p += stride;
            stride -= dec;
            e += 32;
        }
    }
}

template <int Q3>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSlabThreads, 1)
k_m2l_slab_folded(M2LFoldArgs A, const float *__restrict__ F, float *__restrict__ lam, int J0, int nJ, int r0)
{
    constexpr int W = kSlabThreads / 32, RW = 256;
    extern __shared__ __align__(16) float sm[];
    const int nk = A.nk, na = A.na, m1 = A.mx + 1;
    float *T1 = sm, *T2 = T1 + A.p.urows * RW, *Es = T2 + A.p.urows * RW;
    int2 *un = reinterpret_cast<int2 *>(Es + m1 * m1 * 32);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane >> 4, cl = lane & 15;
    const int s1 = blockIdx.x & 1, kb = blockIdx.x >> 1, b = kb % na, k = A.k_lo + kb / na, rhs = r0 + blockIdx.y;
    const int nterm = k < 2 ? 0 : (k & 1 ? 2 * na : na);
    for (int i = threadIdx.x; i < A.p.nunits; i += kSlabThreads) un[i] = reinterpret_cast<const int2 *>(A.p.units)[i];

    float lamr[Q3][2][8];
#pragma unroll
    for (int q = 0; q < Q3; ++q)
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int r = 0; r < 8; ++r) lamr[q][f][r] = 0.f;

    for (int t = 0; t < nterm; ++t) {
        const int a = t % na, D = (k & 1) ? 3 - t / na : 2, J = k - D;
        __syncthreads();  // units in place; the previous term's passes are done with Es
        const float4 *Eg = reinterpret_cast<const float4 *>(A.EF) + (size_t)(((D - 2) * na + a) * na + b) * m1 * m1 * 8;
        for (int i = threadIdx.x; i < m1 * m1 * 8; i += kSlabThreads) reinterpret_cast<float4 *>(Es)[i] = Eg[i];
        const float coef = reinterpret_cast<const float *>(A.pref)[((D - 2) * na + a) * na + b];
        const float *Fj = F + (((size_t)blockIdx.y * nJ + (J - J0)) * na + a) * nk * 512 + cl * 4;
        for (int sl = 0; sl < A.p.nslice; ++sl) {
            __syncthreads();  // Es in place; pass 2 of the previous slice is done with T1
            // pass 1: unit (k2, k3, nu1); lane = four cells (y of one half, z); inputs of the sector that
            // feeds s1, outputs the four X1 of s1
            for (int ts = warp; ts < A.p.ntask1[sl]; ts += W) {
                const UnitBits u(un[A.p.first1[sl] + ts * 2 + sub]);
                float acc[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
                const int s0 = s1 ^ (u.nu & 1);
                const float *src = Fj + (size_t)u.row * 512;
                const float *e = Es + u.nu * m1 * 32;
                float *o = T1 + u.out * RW + cl * 4;
                float4 nx[4];  // the next step's inputs, one L2 latency ahead
#pragma unroll
                for (int q = 0; q < 4; ++q) nx[q] = __ldg(reinterpret_cast<const float4 *>(src + s0 * 256 + q * 64));
#pragma unroll 1
                for (int j = 0; j < u.len; ++j) {
                    const int s = s0 ^ (j & 1);
                    float4 in[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) in[q] = nx[q];
                    if (j + 1 < u.len)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            nx[q] = __ldg(reinterpret_cast<const float4 *>(src + (j + 1) * 512 + (s ^ 1) * 256 + q * 64));
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float ev[4];
                        load4(e + j * 32 + s * 16 + i * 4, ev);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            acc[i][0] = fmaf(ev[q], in[q].x, acc[i][0]);
                            acc[i][1] = fmaf(ev[q], in[q].y, acc[i][1]);
                            acc[i][2] = fmaf(ev[q], in[q].z, acc[i][2]);
                            acc[i][3] = fmaf(ev[q], in[q].w, acc[i][3]);
                        }
                        if (u.valid) store4(o + j * RW + i * 64, acc[i]);
                    }
                }
            }
            __syncthreads();
            // pass 2: unit = row of T2; lane: fibres (X1, z) with X1 = cl / 8 and cl / 8 + 2
            for (int ts = warp; ts < A.p.ntask2[sl]; ts += W) {
                const UnitBits u(un[A.p.first2[sl] + ts * 2 + sub]);
                const int z = cl & 7, i0 = cl >> 3;
                float acc[2][8];
                chain8(u.len, acc, T1 + u.row * RW + i0 * 64 + z * 4, 0, 32, u.step * RW, RW, 128, Es + u.nu * m1 * 32);
                if (u.valid) {
                    // to [X1][z / 4][X2 ^ swizzle][z % 4]: the lanes' eight groups of four words on all banks
                    float *o = T2 + u.out * RW + i0 * 64 + (z >> 2) * 32 + (z & 3);
                    const int sw = (z >> 2) | i0 << 1 | u.okey << 2, fl = (u.nu & 1) << 2;
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        const int x2 = ((r ^ fl) ^ sw) << 2;
                        o[x2] = acc[0][r];
                        o[x2 + 128] = acc[1][r];
                    }
                }
            }
            __syncthreads();
            // pass 3: unit = multi-index of the locals; lane: fibres (X1, X2)
#pragma unroll
            for (int q = 0; q < Q3; ++q) {
                const int ts = warp + q * W;
                if (ts >= A.p.ntask3) break;
                const UnitBits u(un[A.p.first3 + ts * 2 + sub]);
                if (u.slice != sl) continue;
                const int X2 = cl & 7, i0 = cl >> 3;
                float acc[2][8];
                // the halves of a fibre (z / 4) lie at different swizzles
                chain8(u.len, acc, T2 + u.row * RW + i0 * 64, (X2 ^ (i0 << 1 | u.key << 2)) << 2,
                       32 + ((X2 ^ (1 | i0 << 1 | u.key << 2)) << 2), RW, 0, 128, Es + u.nu * m1 * 32);
#pragma unroll
                for (int f = 0; f < 2; ++f)
#pragma unroll
                    for (int r = 0; r < 8; ++r) lamr[q][f][r] = fmaf(coef, acc[f][r], lamr[q][f][r]);
            }
        }
    }
    // unfold in z per lane into rows [multi-index][X1][X2][X3] over T1 and T2 (nk <= urows)
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q3; ++q) {
        const int ts = warp + q * W;
        if (ts >= A.p.ntask3) break;
        const UnitBits u(un[A.p.first3 + ts * 2 + sub]);
        if (!u.valid) continue;
        const int X2 = cl & 7, i0 = cl >> 3;
        const bool odd = u.nu & 1;
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            float *p = T1 + u.out * RW + (i0 + 2 * f) * 64 + X2 * 8;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float P = odd ? lamr[q][f][4 + i] : lamr[q][f][i], M = odd ? lamr[q][f][i] : lamr[q][f][4 + i];
                p[i] = P + M;
                p[7 - i] = P - M;
            }
        }
    }
    __syncthreads();
    // unfold in y
    for (int i = threadIdx.x; i < nk * 32; i += kSlabThreads) {
        float *p = T1 + (i >> 5) * RW + ((i >> 3) & 3) * 64 + (i & 7);
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = p[j * 8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            p[j * 8] = v[j] + v[4 + j];
            p[(7 - j) * 8] = v[j] - v[4 + j];
        }
    }
    // unfold in x with the other CTA's sector: sector 0 writes X1 = i (sum), sector 1 X1 = 7 - i (difference)
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    uint32_t mine = (uint32_t)__cvta_generic_to_shared(T1), other;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(other) : "r"(mine), "r"(s1 ^ 1));
    float *out = lam + (((size_t)rhs * A.nint + k) * A.nbox * na + b) * nk;
    for (int i = threadIdx.x; i < nk * 256; i += kSlabThreads) {
        const int iv = i % nk, c = i / nk, i1 = c >> 6;
        const int box = A.cellbox[(s1 ? 7 - i1 : i1) * 64 + (c & 63)];
        if (box < 0) continue;
        float o;
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(o) : "r"(other + 4u * (iv * RW + c)) : "memory");
        const float m = T1[iv * RW + c];
        out[(size_t)box * na * nk + iv] = s1 ? o - m : m + o;
    }
    // the other CTA has read this one's rows
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

int launch_m2l_slab_folded(const DevLevel &L, const M2LFoldDev &P, const float *mu, float *lam, int nrhs,
                           const ApplyGeo &g, float *ws, size_t ws_elems, cudaStream_t st)
{
    // folded moments: per_int floats an interval and right-hand side; a target interval needs two
    // intervals (k - 3, k - 2), n targets n + 1
    const size_t per_int = (size_t)512 * g.na * g.nk, cap = ws_elems / per_int;
    if (!P.units || cap < 2) return 1;
    M2LFoldArgs A{};
    A.na = g.na;
    A.nk = g.nk;
    A.mx = g.mx;
    A.nint = L.nint;
    A.nbox = L.nbox;
    A.truncated = L.ntr < L.G - 1;
    A.p = P;
    A.cellbox = L.cellbox;
    A.EF = L.EF;
    A.pref = L.pref;
    auto kf = P.q3 <= 2 ? k_m2l_slab_folded<2> : k_m2l_slab_folded<3>;
    if (P.q3 > 3 || cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P.smem) != cudaSuccess) return -1;
    const int rc = (int)std::min<size_t>(nrhs, std::max<size_t>(1, cap / std::min(L.nint, 16)));  // rhs at a time
    const int nt = (int)std::min<size_t>(cap / rc - 1, L.nint);                                    // targets at a time
    for (int r0 = 0; r0 < nrhs; r0 += rc)
        for (int k0 = 0; k0 < L.nint; k0 += nt) {
            const int nr = std::min(rc, nrhs - r0), k1 = std::min(L.nint, k0 + nt);
            const int J0 = std::max(0, k0 - 3), nJ = std::max(0, k1 - 2 - J0);
            if (nJ > 0)
                k_m2l_fold_moments<<<dim3(nJ * g.na, (g.nk + kFoldK - 1) / kFoldK, nr), 256, 0, st>>>(
                    mu, L.cellbox, P.urow, g.na, g.nk, L.nint, L.nbox, J0, nJ, r0, A.truncated, ws);
            A.k_lo = k0;
            kf<<<dim3((unsigned)((k1 - k0) * g.na * 2), nr), kSlabThreads, P.smem, st>>>(A, ws, lam, J0, nJ, r0);
        }
    settle_outside(L, mu, lam, nrhs, g, st);
    return 0;
}

}  // namespace pfmm
