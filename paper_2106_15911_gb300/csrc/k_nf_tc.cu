// k_nf_tc.cu -- nearfield apply (Alg. 2, last loop; Eq. eval_sl_nf_block) on the sm_103a
// tensor cores: tcgen05.mma (kind::f16, FP16 operands) with TMA-staged operands and TMEM
// accumulators.
//
// The block-Toeplitz nearfield product is a dense GEMM
//   F[rows][t] += sum_{d} A_d[rows][k] W[t - d][k]      (k: all triangles or nodes)
// with t = i*2 + s (leaf interval i, step s of the interval) and d = 0 .. 2 + s.  All panels index the
// same columns, so rows are tiled regardless of panels (leaf boxes of fewer than 128 rows leave no
// empty rows: 6 tiles instead of 56 on 768 triangles).  A CTA tile is 128 rows x (NI intervals x 2
// phases).  W is seen by TMA as a 4D tensor [rhs][interval][phase][col], so the time shift by d is a
// coordinate offset, and the causality mask (t - d < 0) is the out-of-bounds zero fill.  For one block
// of 32 columns the four offsets need four W tiles, (phase 0 or 1) x (interval shift 1 or 0); in the
// order (0, 1), (1, 1), (0, 0), (1, 0) phase ph of offset d is tile 2 + ph - d and both phases are one
// operand of 2 NI rows, so each tile is brought in once for its two uses.  FP32 accuracy comes from a
// two-part FP16 split with power-of-two
// scales (FP16 keeps 11 significant bits, as TF32 does, at twice the rate and half the bytes):
//   A W ~ (A_hi W_hi + A_hi W_lo + A_lo W_hi) / (s_A s_W),
//   A_hi = rn_f16(s_A A), A_lo = rn_f16(s_A A - A_hi)     (same for W with s_W per rhs),
// where s_A (per operator, at build) and s_W (per rhs and apply, from max |W|) bring the largest
// magnitude into [2^14, 2^15): the parts are normal FP16 down to 2^-29 of the maximum, and
// |A - (A_hi + A_lo) / s_A| <= 2^-22 |A| above that.  Both parts of a tile's 32 columns at offset d are
// one 16 KB piece of memory (nf_split_index), one bulk copy.  The products are accumulated in FP32 in
// TMEM over sub-chunks of 4 column blocks (512 products: the tensor cores truncate each sum to the
// accumulator's FP32 grid, so a long accumulation is biased: over 16 blocks 12288 triangles x 256 steps
// came out 5.3e-6 from 64-bit arithmetic, over 4 it is 1.8e-6), four sub-chunks are added in FP32 registers (rounded to
// nearest), unscaled exactly (powers of two) to FP64 and added, in order and by the one CTA that owns
// the work item, into the item's FP64 partial plane; the ksplit planes of a tile (split K, for SM
// balance) are then summed in plane order by k_nf_tc_reduce: bitwise reproducible.  The planes take their sums as
// reductions at the memory: reading, adding and writing them here kept the epilogue longer than the
// MMAs of a sum (2.44 instead of 1.89 ms below).
// Warp roles (384 threads): 0 TMA of W (two stages), 1 TMEM allocation and MMA issue, 2 bulk copies of A
// (one slot per offset), 4-11 drain TMEM (32-lane quadrant, one phase each).  Two TMEM accumulators,
// persistent CTAs over (tile, K chunk) work items.  Every mbarrier
// wait gives up after a deadline, sets an error word and lets the CTA finish cleanly.
// Bound: the MMAs (2688 cycles a column block against 128 KB of operands), for one right-hand side the
// FP16 parts of A from memory.  12288 triangles x 256 steps, kernel with 1 / 4 right-hand sides: 0.59 /
// 1.89 ms (0.59 = 4.9 TB/s, 1.89 = 1720 TFLOP/s of FP16 products); with one 96 KB stage per offset and
// 64 columns, W brought in once per offset, and an FP64 epilogue it was 3.1 ms for 4.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "kernels.h"
#include "nf_tc.h"
#include "tc_ptx.cuh"

namespace pfmm {

namespace {

using namespace tc;

constexpr int BM = 128, BK = 32;      // BK fp16 = 64 bytes = one row of the 64-byte swizzle
constexpr int A_PART = BM * BK * 2;    // 8 KB
constexpr int A_SLOT = 2 * A_PART;     // hi, lo of one offset
constexpr int NW = 2;                  // column blocks of W in flight
constexpr int kSub = 4;                // column blocks per accumulation in TMEM (512 products)
constexpr int kFlush = 4;              // accumulations per FP32 sum in registers (2048 products)
constexpr int kTcThreads = 384;

template <int NI>
struct TcShape {
    static constexpr int W_TILE = NI * BK * 2, W_PART = 4 * W_TILE, W_STAGE = 2 * W_PART;
    static constexpr int NA = NI == 128 ? 6 : 8;  // A slots
    static constexpr size_t bytes = (size_t)NW * W_STAGE + NA * A_SLOT + 1024 + 256;
};

__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(su32(dst)),
                 "l"(src), "r"(bytes), "r"(su32(bar))
                 : "memory");
}

__device__ __forceinline__ void tma_4d(void *dst, const CUtensorMap *map, int x, int y, int z, int w, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(su32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(su32(bar))
        : "memory");
}

// instruction descriptor: kind::f16 with FP16 A and B (format 0), FP32 accumulate, both
// K-major, M x N
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N)
{
    return (1u << 4)                      // D format F32
           | ((uint32_t)(N >> 3) << 17)   // N / 8
           | ((uint32_t)(M >> 4) << 24);  // M / 16
}

// operands at descriptor low words alo, blo (K-major, 64-byte swizzle)
__device__ __forceinline__ void mma_f16(uint32_t issue, uint32_t dt, uint32_t alo, uint32_t blo, uint32_t idesc,
                                        uint32_t acc)
{
    constexpr uint32_t hi = (512 >> 4) | 1u << 14 | 4u << 29;  // 8-row groups 512 bytes apart, version, swizzle
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %6};\n\tmov.b64 b, {%2, %6};\n\tsetp.ne.b32 p, %4, "
        "0;\n\tsetp.ne.b32 q, %5, 0;\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}\n" ::"r"(dt),
        "r"(alo), "r"(blo), "r"(idesc), "r"(acc), "r"(issue), "n"(hi)
        : "memory");
}

struct Item {
    int tile, ib, rhs, kc, kb0, kb1;  // row tile, interval block, rhs, K chunk (partial plane), its column blocks
    __device__ __forceinline__ Item(const NfTcParams &P, int nib, int it)
    {
        // right-hand sides and interval blocks inner: CTAs that run together read the same blocks of A,
        // which then come from memory once (12288 triangles x 256 steps, 4 right-hand sides: 2.11 -> 1.78 ms
        // against right-hand sides outermost)
        int t = it;
        rhs = t % P.nrhs;
        t /= P.nrhs;
        ib = t % nib;
        t /= nib;
        kc = t % P.ksplit;
        tile = t / P.ksplit;
        kb0 = (int)((long long)P.nkb * kc / P.ksplit);
        kb1 = (int)((long long)P.nkb * (kc + 1) / P.ksplit);
    }
};

// FP32 bits times 2^(shift - 896) as FP64, exactly, without the FP64 unit (a conversion and a product
// there would take longer than the tile's MMAs).  Sums of products of FP16 numbers are zero or at least
// 2^-48: no subnormals.  |shift - 896| <= 200
__device__ __forceinline__ double widen(uint32_t v, int shift)
{
    const uint32_t e = (v >> 23) & 255u, m = v & 0x7fffffu;
    const uint32_t E = e == 255u ? 2047u : e + shift;
    const uint32_t hi = (v & 0x80000000u) | (e ? (E << 20) | (m >> 3) : 0u);
    return __hiloint2double((int)hi, (int)(e ? m << 29 : 0u));
}

}  // namespace

template <int NI>
__global__ void __launch_bounds__(kTcThreads, 1) k_nf_apply_tc(const __grid_constant__ CUtensorMap mapWhi,
                                                                const __grid_constant__ CUtensorMap mapWlo, NfTcParams P)
{
    using S = TcShape<NI>;
    constexpr int NA = S::NA;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte alignment of the tiles (swizzle atoms)
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = smem + NW * S::W_STAGE;
    uint64_t *wfull = (uint64_t *)(sA + NA * A_SLOT), *wempty = wfull + NW, *afull = wempty + NW, *aempty = afull + NA;
    uint64_t *tfull = aempty + NA, *tempty = tfull + 2;
    uint32_t *tmem_slot = (uint32_t *)(tempty + 2);
    __shared__ volatile int s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NW; ++s) {
            mbar_init(&wfull[s], 1);
            mbar_init(&wempty[s], 1);
        }
        for (int s = 0; s < NA; ++s) {
            mbar_init(&afull[s], 1);
            mbar_init(&aempty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 8);  // one arrival per epilogue warp
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const int nib = (P.nint + NI - 1) / NI;
    auto wait = [&](uint64_t *bar, uint32_t parity, int code) {
        if (mbar_wait_bounded(bar, parity)) return true;
        atomicExch(P.err, code);
        s_abort = 1;
        return false;
    };

    if (warp == 0) {
        // ---------------- TMA of W: hi and lo of the four (phase, shift) tiles of a column block
        if (lane == 0) {
            int g = 0;
            for (int it = blockIdx.x; it < P.nitems && !s_abort; it += gridDim.x) {
                const Item I(P, nib, it);
                for (int kb = I.kb0; kb < I.kb1; ++kb, ++g) {
                    const int s = g % NW;
                    if (!wait(&wempty[s], ((g / NW) & 1) ^ 1, 1) || s_abort) break;
                    unsigned char *d = smem + s * S::W_STAGE;
                    mbar_expect_tx(&wfull[s], S::W_STAGE);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int i0 = I.ib * NI - (q < 2 ? 1 : 0);
                        tma_4d(d + q * S::W_TILE, &mapWhi, kb * BK, q & 1, i0, I.rhs, &wfull[s]);
                        tma_4d(d + S::W_PART + q * S::W_TILE, &mapWlo, kb * BK, q & 1, i0, I.rhs, &wfull[s]);
                    }
                }
            }
            // before the CTA exits, the copies it issued must have landed (bounded wait)
            for (int j = (g > NW ? g - NW : 0); j < g; ++j) mbar_wait_bounded(&wfull[j % NW], (j / NW) & 1);
        }
    } else if (warp == 2) {
        // ---------------- bulk copies of A: hi and lo of one offset per slot
        if (lane == 0) {
            int g = 0;
            for (int it = blockIdx.x; it < P.nitems && !s_abort; it += gridDim.x) {
                const Item I(P, nib, it);
                const unsigned char *src = P.A + ((size_t)I.tile * P.nkb + I.kb0) * 4 * A_SLOT;
                for (int j = 0; j < (I.kb1 - I.kb0) * 4; ++j, ++g, src += A_SLOT) {
                    const int s = g % NA;
                    if (!wait(&aempty[s], ((g / NA) & 1) ^ 1, 2) || s_abort) break;
                    mbar_expect_tx(&afull[s], A_SLOT);
                    bulk_copy(sA + s * A_SLOT, src, A_SLOT, &afull[s]);
                }
            }
            for (int j = (g > NA ? g - NA : 0); j < g; ++j) mbar_wait_bounded(&afull[j % NA], (j / NA) & 1);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        const uint32_t issue = elect_lane(), tm = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t wbase = __shfl_sync(0xffffffffu, (su32(smem) >> 4) & 0x3FFFu, 0) | 1u << 16;
        const uint32_t abase = __shfl_sync(0xffffffffu, (su32(sA) >> 4) & 0x3FFFu, 0) | 1u << 16;
        constexpr uint32_t id2 = idesc_f16(BM, 2 * NI), id1 = idesc_f16(BM, NI), WT = S::W_TILE >> 4, WP = S::W_PART >> 4;
        int ga = 0, gw = 0, n = 0;  // n: sub-chunks issued (the TMEM accumulators alternate per sub-chunk)
        for (int it = blockIdx.x; it < P.nitems && !s_abort; it += gridDim.x) {
            const Item I(P, nib, it);
            bool ok = true;
            for (int sc0 = I.kb0; sc0 < I.kb1 && ok; sc0 += kSub, ++n) {
                const int sc1 = min(I.kb1, sc0 + kSub), acc = n & 1;
                if (!(ok = wait(&tempty[acc], ((n >> 1) & 1) ^ 1, 3))) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t dcol = tm + acc * 256;
                for (int kb = sc0; kb < sc1 && ok; ++kb, ++gw) {
                    const int sw = gw % NW;
                    if (!(ok = wait(&wfull[sw], (gw / NW) & 1, 4))) break;
                    const uint32_t more = kb > sc0 ? 1u : 0u;  // a sub-chunk's first MMA starts both phases from zero
#pragma unroll
                    for (int d = 0; d < 4; ++d, ++ga) {
                        const int s = ga % NA;
                        if (!ok || !(ok = wait(&afull[s], (ga / NA) & 1, 5))) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t ah = abase + s * (A_SLOT >> 4), al = ah + (A_PART >> 4);
                        const uint32_t wh = wbase + sw * (S::W_STAGE >> 4) + (d < 3 ? 2 - d : 0) * WT, wl = wh + WP;
                        const uint32_t dc = d < 3 ? dcol : dcol + NI, id = d < 3 ? id2 : id1;
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {  // K = 16 fp16 (32 bytes) per MMA
                            mma_f16(issue, dc, ah + kk * 2, wh + kk * 2, id, d == 0 && kk == 0 ? more : 1u);
                            mma_f16(issue, dc, ah + kk * 2, wl + kk * 2, id, 1u);
                            mma_f16(issue, dc, al + kk * 2, wh + kk * 2, id, 1u);
                        }
                        mma_commit_if(issue, &aempty[s]);  // frees the slot once these MMAs have read it
                    }
                    mma_commit_if(issue, &wempty[sw]);
                }
                mma_commit_if(issue, &tfull[acc]);
            }
        }
    } else if (warp >= 4) {
        // ---------------- epilogue: warps 4..11, TMEM lane quadrant = warp % 4, one phase each
        const int quad = warp & 3, ph = warp >= 8 ? 1 : 0;
        int n = 0;
        bool ok = true;
        float sum[NI];
#pragma unroll
        for (int c = 0; c < NI; ++c) sum[c] = 0.f;
        for (int it = blockIdx.x; it < P.nitems && ok; it += gridDim.x) {
            const Item I(P, nib, it);
            const int row = I.tile * BM + quad * 32 + lane, nj = P.nint - I.ib * NI;
            double *fr = P.part + (((size_t)I.kc * P.nrhs + I.rhs) * P.Et + 2 * I.ib * NI + ph) * P.nt + row;
            const size_t step = 2 * (size_t)P.nt;
            const int shift = 896 - P.a_exp - f64_scale_exp(P.wmax[I.rhs]);  // FP64 exponent offset, unscaled
            bool first = true;
            for (int sc0 = I.kb0, j = 0; sc0 < I.kb1; sc0 += kSub, ++n) {
                const int acc = n & 1;
                bool go = true;
                if (lane == 0) go = wait(&tfull[acc], (n >> 1) & 1, 6) && !s_abort;
                if (!(ok = __all_sync(0xffffffffu, go) != 0)) break;  // the warp's TMEM loads are warp-wide
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int c0 = 0; c0 < NI; c0 += 16) {
                    uint32_t v[16];
                    tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + acc * 256 + ph * NI + c0, v);
#pragma unroll
                    for (int c = 0; c < 16; ++c) sum[c0 + c] += __uint_as_float(v[c]);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[acc]);
                if (++j < kFlush && sc0 + kSub < I.kb1) continue;
                j = 0;
                if (row < P.nt) {
                    // adds at the memory: nothing to wait for.  The plane is private to this work item and
                    // every element to one thread, whose operations on it keep their order
                    double *a0 = fr;
                    int left = nj;
#pragma unroll
                    for (int c = 0; c < NI; ++c, a0 += step, --left) {
                        if (c % 8 == 0) asm volatile("" : "+l"(a0), "+r"(left));  // addresses a few at a time
                        const double x = widen(__float_as_uint(sum[c]), shift);
                        if (left > 0) {
                            if (first)
                                *a0 = x;
                            else
                                atomicAdd(a0, x);
                        }
                    }
                }
#pragma unroll
                for (int c = 0; c < NI; ++c) sum[c] = 0.f;
                first = false;
                __syncwarp();
            }
        }
    }
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

// ------------------------------------------------------------------------------------------
// split kernels: with the scale s = 2^E, hi = rn_f16(s a) and lo = rn_f16(s a - hi).  s a - hi is
// exact in FP32 (and in FP64 for the input), so a - (hi + lo) / s is one FP16 rounding of the
// remainder: below 2^-22 |a| while lo is a normal FP16 number.

// largest |a| of n FP32 values into *out as ordered bits (non-negative floats order as integers)
__global__ void k_absmax_f32(const float *__restrict__ A, size_t n, unsigned *__restrict__ out)
{
    float m = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(A[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

// FP32 panels -> FP16 parts in the layout of nf_split_index (rows past the last triangle are zero).
// Thread per (row, d, eight columns: one 16-byte chunk of each part)
__global__ void k_split_panel(const float *__restrict__ A, const PanelGPU *__restrict__ panels,
                              const int *__restrict__ tri_leaf, int kop, int nt, int ntiles, int ncp, float scale,
                              __half *__restrict__ out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int nq = ncp / 8, c = (int)(i % nq) * 8;
    const size_t rd = i / nq;
    const int d = (int)(rd & 3), x = (int)(rd >> 2);
    if (x >= ntiles * BM) return;
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (x < nt) {
        const PanelGPU &Pn = panels[tri_leaf[x]];
        const float4 *a = reinterpret_cast<const float4 *>(
            A + (kop ? Pn.offK : Pn.offV) + ((size_t)d * Pn.rows_pad + (x - Pn.row0)) * ncp + c);
        const float4 p = a[0], q = a[1];
        v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
        v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
    }
    __half h[8], l[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float a = v[j] * scale;
        h[j] = __float2half_rn(a);
        l[j] = __float2half_rn(a - __half2float(h[j]));
    }
    const size_t o = nf_split_index(x, d, c, ncp / 32);
    *reinterpret_cast<uint4 *>(out + o) = *reinterpret_cast<const uint4 *>(h);
    *reinterpret_cast<uint4 *>(out + o + kSplitPart) = *reinterpret_cast<const uint4 *>(l);
}

// per-rhs max |x| of the FP64 input [rhs][Et][ncol], on the bits (non-negative doubles order as
// unsigned integers; no FP64 arithmetic)
__global__ void k_absmax_input(const double *__restrict__ x, size_t per_rhs, unsigned long long *__restrict__ wmax)
{
    const unsigned long long *xr = reinterpret_cast<const unsigned long long *>(x) + (size_t)blockIdx.y * per_rhs;
    unsigned long long m = 0ull;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < per_rhs; i += (size_t)gridDim.x * blockDim.x) {
        const unsigned long long v = xr[i] & 0x7fffffffffffffffull;
        m = v > m ? v : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
        m = v > m ? v : m;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(wmax + blockIdx.y, m);
}

// W split from FP64 input: permutes (V) or pads rows (K) into [rhs][t][ncol_pad].  x is rounded
// once to FP32 (2^-24 relative), scaled exactly by 2^E in FP32 and split there.
__global__ void k_split_input(const double *__restrict__ x, const int *__restrict__ perm, int ncol, int ncol_pad,
                              __half *__restrict__ hi, __half *__restrict__ lo, size_t per_rhs, size_t total,
                              const unsigned long long *__restrict__ wmax)
{
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    size_t rt = i / ncol_pad;
    int c = (int)(i - rt * ncol_pad);
    float v = 0.f;
    if (c < ncol) v = (float)x[rt * ncol + (perm ? perm[c] : c)];
    v *= __int_as_float((127 + f64_scale_exp(wmax[i / per_rhs])) << 23);  // 2^E, |E| <= 100
    const __half h = __float2half_rn(v);
    hi[i] = h;
    lo[i] = __float2half_rn(v - __half2float(h));
}

int panel_scale_exp(const float *A, size_t n, unsigned *scratch, cudaStream_t st)
{
    if (cudaMemsetAsync(scratch, 0, sizeof(unsigned), st) != cudaSuccess) return INT32_MIN;
    const unsigned grid = (unsigned)std::min<size_t>((n + 255) / 256, 4096);
    if (grid > 0) k_absmax_f32<<<grid, 256, 0, st>>>(A, n, scratch);
    unsigned bits = 0;
    if (cudaMemcpyAsync(&bits, scratch, sizeof(unsigned), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return INT32_MIN;
    return f32_scale_exp(bits);
}

size_t split_panel_halves(int nt, int ncp) { return (size_t)((nt + BM - 1) / BM) * BM * ncp * 8; }

void launch_split_panel(const float *A, const PanelGPU *panels, const int *tri_leaf, int kop, int nt, int ncp, int a_exp,
                        void *out, cudaStream_t st)
{
    const int ntiles = (nt + BM - 1) / BM;
    const size_t n = (size_t)ntiles * BM * 4 * (ncp / 8);
    k_split_panel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(A, panels, tri_leaf, kop, nt, ntiles, ncp,
                                                              std::ldexp(1.0f, a_exp), (__half *)out);
}

void launch_split_input(const double *x, const int *perm, int ncol, int ncol_pad, int nrhs, int Et, void *hi,
                        void *lo, unsigned long long *wmax, cudaStream_t st)
{
    cudaMemsetAsync(wmax, 0, sizeof(unsigned long long) * nrhs, st);
    const size_t per_in = (size_t)Et * ncol;
    const unsigned gx = (unsigned)std::max<size_t>(1, std::min<size_t>((per_in + 2047) / 2048, 1216));
    k_absmax_input<<<dim3(gx, nrhs), 256, 0, st>>>(x, per_in, wmax);
    const size_t per_rhs = (size_t)Et * ncol_pad, total = (size_t)nrhs * per_rhs;
    k_split_input<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(x, perm, ncol, ncol_pad, (__half *)hi,
                                                                   (__half *)lo, per_rhs, total, wmax);
}

void launch_absmax_input(const double *x, size_t per_rhs, int nrhs, unsigned grid_x, unsigned long long *wmax,
                         cudaStream_t st)
{
    k_absmax_input<<<dim3(grid_x, nrhs), 256, 0, st>>>(x, per_rhs, wmax);
}

// f[i] = sum over the K-chunk planes of part[kc][i], in plane order
__global__ void k_nf_tc_reduce(const double *__restrict__ part, int ks, size_t n, double *__restrict__ f)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = part[i];
    for (int kc = 1; kc < ks; ++kc) s += part[(size_t)kc * n + i];
    f[i] = s;
}

void launch_nf_tc_reduce(const double *part, int ks, size_t n, double *f, cudaStream_t st)
{
    if (n > 0) k_nf_tc_reduce<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(part, ks, n, f);
}

int nf_tc_intervals(int nint) { return nint <= 64 ? 64 : 128; }

int nf_tc_ksplit(int nt, int nint, int Et, int nrhs, int cols, int nsm)
{
    // K chunks (1 .. 16, of at least two column blocks) with the least estimated time: the rounds of the
    // persistent grid at 1.3 us a column block (2688 cycles of MMAs; half for 64 intervals) and a plane
    // written, read back and added at 6 TB/s
    const int ni = nf_tc_intervals(nint), nkb = cols / BK;
    const long long tiles = (long long)nrhs * ((nt + BM - 1) / BM) * ((nint + ni - 1) / ni);
    const double block = ni == 128 ? 1.3e-6 : 0.75e-6, plane = 16.0 * nt * Et * nrhs / 6e12;
    int best = 1;
    double best_t = 1e30;
    for (int ks = 1; ks <= std::min(16, std::max(1, nkb / 2)); ++ks) {
        const long long rounds = (tiles * ks + nsm - 1) / nsm;
        const double t = (double)rounds * ((nkb + ks - 1) / ks) * block + ks * plane;
        if (t < best_t * (1.0 - 1e-9)) {
            best_t = t;
            best = ks;
        }
    }
    return best;
}

template <int NI>
static int launch_tc_T(const CUtensorMap &Whi, const CUtensorMap &Wlo, NfTcParams P, int nsm, cudaStream_t st)
{
    P.nitems = P.nrhs * P.ntiles * ((P.nint + NI - 1) / NI) * P.ksplit;
    auto kf = k_nf_apply_tc<NI>;
    const size_t smem = TcShape<NI>::bytes;
    if (cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -1;
    kf<<<std::min(P.nitems, nsm), kTcThreads, smem, st>>>(Whi, Wlo, P);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_nf_apply_tc(const CUtensorMap &Whi, const CUtensorMap &Wlo, const NfTcParams &P, int nsm, cudaStream_t st)
{
    return nf_tc_intervals(P.nint) == 64 ? launch_tc_T<64>(Whi, Wlo, P, nsm, st) : launch_tc_T<128>(Whi, Wlo, P, nsm, st);
}

}  // namespace pfmm
