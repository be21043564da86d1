// k_nf_crt.cu -- FP64-accurate nearfield apply (Alg. 2, last loop; Eq. eval_sl_nf_block) on
// the sm_103a tensor cores, by exact integer arithmetic in residues (a multi-modular form of the
// Ozaki error-free splitting scheme for matrix products: Ozaki, Ogita, Oishi, Rump, Numerical
// Algorithms 59 (2012); here with the Chinese remainder theorem instead of digit slices, as in
// Ozaki, Uchino, Imamura, "Ozaki Scheme II", 2024).
//
// GB300 executes FP64 FMAs at about 1 TFLOP/s but FP16 tensor-core products at about 2 PFLOP/s.
// The block-Toeplitz nearfield product F[r][t] = sum_d sum_k A_d[r][k] W[t-d][k] is therefore
// computed exactly in integers and rounded to FP64 once:
//   * every row r of the stored FP64 blocks is scaled by 2^e_r (largest |A_d[r][k]| over d, k in
//     [2^(b-1), 2^b)) and rounded to the integer A'; the input by 2^s to W' (|W'| <= 2^b), with s
//     from the largest finite input of the two leaf intervals that an output's products read (or of
//     the whole right-hand side while that takes at most kCrtSlack bits from them),
//     b chosen so that the exact integer product X = sum A' W' satisfies 2 |X| < M;
//   * X is computed modulo 16 primes p_i < 256 (M = prod p_i ~ 2^123): the residues of A' and W'
//     in [-(p-1)/2, (p-1)/2] are exact FP16 numbers, their products are below 2^14, and a tcgen05
//     kind::f16 MMA chain accumulates them in FP32 exactly (integers below 2^24) over a chunk of
//     products; after each chunk the epilogue reduces the accumulator modulo p in place
//     (tcgen05.ld / .st), so the next chunk adds onto a small residue;
//   * the 16 residues of X are combined by Garner's mixed-radix algorithm (balanced digits, exact
//     FP32 arithmetic), X is assembled exactly in 128-bit integers and X 2^-(e_r + s) is rounded
//     to FP64 (relative error ~2^-52).
// The only rounding before the final FP64 result is that of A and W to b-bit fixed point per row /
// per output interval (b = 51..53): the error is that of an FP64 dot product whose terms are all of
// the size of the row's largest entry times the interval's largest input.  An input that is not
// finite has residues of zero, and its products are added in FP64 to the outputs that they reach.
//
// The residues of A' are stored as bytes (r + 128), half the bytes of FP16, because the stored
// blocks are the bulk of the traffic: 16 bytes per element.  All panels index the same columns, so
// the rows are tiled regardless of panels: tile t holds the target triangles 128 t .. 128 t + 127, and
// the 2 LS step offsets (LS steps per leaf) of one 64-column block of a tile are one piece, [modulus]
// [tile][column block][d][row][64], brought in by one bulk copy (32 KB at LS = 2).  Converter warps turn the bytes into FP16
// in registers (byte permute onto 1024 + u, one subtraction, exact) and write them to tensor memory,
// from where tcgen05.mma takes them as the A operand.
//
// Tiles: 128 rows x (NI leaf intervals x LS phases) columns; W is a TMA tensor [modulus][rhs]
// [interval][2 LS steps][column]: the steps of the interval before and then of the interval itself, both
// scaled for this interval's outputs.  Where all intervals of a tile have the scale of the one before
// (P.shared), the first LS steps are not stored but read as the interval before's own (a coordinate
// offset; the zero fill before the first): writing and reading both took 1.6 % of a product.
// For one column block the 2 LS step offsets need only these 2 LS W tiles; in this
// order phase ph of offset d is tile LS + ph - d, so all
// phases of an offset are one contiguous operand of up to LS NI rows, and each W tile is brought in
// once for its LS uses.  A work item is (modulus, row tile, interval block, rhs).  The accumulators
// are reduced modulo p every r column blocks (r by the modulus and LS: 128 LS r products of two
// residues stay below 2^24).  At LS = 2 the phases are reduced in turn, half a period apart, and the
// other phase's MMAs of that block are issued first and hide the reduction.
// The roles meet once per column block (16 MMAs): a wait, the issue and the commit of a step cost the
// issuing thread some 400 cycles, which one step per offset (448 cycles of MMAs) did not hide.
// Warps: 0 TMA of W, 1 TMEM allocation and MMA issue, 2-9 converters (two groups of four, two offsets
// each, one 32-lane TMEM quadrant per warp), 10-17 epilogue (two warps per quadrant, half the columns
// each), 18 bulk copies of A.  Every mbarrier wait is bounded (error word, clean exit).
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "kernels.h"
#include "nf_crt.h"
#include "nf_tc.h"
#include "tc_ptx.cuh"

namespace pfmm {

namespace {

using namespace tc;

__constant__ int c_p[kCrtModuli];              // the moduli
__constant__ float c_invp[kCrtModuli];         // 1 / p (FP32)
__constant__ float c_pf[kCrtModuli];           // the moduli (FP32)
__constant__ int c_red[5][kCrtModuli];         // [LS] column blocks between two reductions (LS = 2: even)
__constant__ float c_pow11[kCrtModuli][5];     // 2^(11 k) mod p_i (FP32), k = 0 .. 4
__constant__ float c_pjmodpif[kCrtModuli][kCrtModuli];  // (p_0 ... p_{j-1}) mod p_i, j < i (FP32)
__constant__ float c_invPif[kCrtModuli];       // (p_0 ... p_{i-1})^-1 mod p_i (FP32)

constexpr int BM = 128, BK = 64;
constexpr int A8_TILE = BM * BK;         // 8 KB of residue bytes
constexpr int NST = 2;                   // column blocks in flight (bytes, W)
constexpr int kCrtThreads = 608;
constexpr uint64_t kTimeoutNs = 2000000000ull;

__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(su32(dst)),
                 "l"(src), "r"(bytes), "r"(su32(bar))
                 : "memory");
}

__device__ __forceinline__ void tma_5d(void *dst, const CUtensorMap *map, int x, int y, int z, int w, int v,
                                       uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
        "[%7];" ::"r"(su32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(v), "r"(su32(bar))
        : "memory");
}

// kind::f16, FP16 A and B, FP32 accumulate, K-major, M x N
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N)
{
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// A from tensor memory, B from shared memory at descriptor low word blo (K-major, 128-byte swizzle)
__device__ __forceinline__ void mma_f16_ts(uint32_t issue, uint32_t dt, uint32_t a, uint32_t blo, uint32_t idesc,
                                           uint32_t acc)
{
    constexpr uint32_t hi = (1024 >> 4) | 1u << 14 | 2u << 29;  // 8-row groups 1024 bytes apart, version, swizzle
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 b;\n\tmov.b64 b, {%2, %6};\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, "
        "0;\n\t@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %3, p;\n\t}\n" ::"r"(dt),
        "r"(a), "r"(blo), "r"(idesc), "r"(acc), "r"(issue), "n"(hi)
        : "memory");
}
__device__ __forceinline__ void tmem_st32_async(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

struct CItem {
    int m, rhs, ib, tile;
    __device__ __forceinline__ CItem(const NfCrtParams &P, int nib, int it)
    {
        // modulus-major: consecutive CTAs share the modulus (its W residues stay in L2)
        const int per_m = P.ntiles * nib * P.nrhs;
        m = it / per_m;
        int r_ = it % per_m;
        rhs = r_ / (P.ntiles * nib);
        r_ %= P.ntiles * nib;
        ib = r_ % nib;
        tile = r_ / nib;
    }
};

// four residue bytes u = r + 128 to FP16: the bytes below 0x64 are 1024 + u, less 1152 is r (exact)
__device__ __forceinline__ void bytes_to_half(uint32_t w, uint32_t &lo, uint32_t &hi)
{
    const __half2 off = __half2half2(__ushort_as_half(0x6480));  // 1152
    const uint32_t a = __byte_perm(w, 0x64646464u, 0x4140), b = __byte_perm(w, 0x64646464u, 0x4342);
    const __half2 x = __hsub2(*reinterpret_cast<const __half2 *>(&a), off);
    const __half2 y = __hsub2(*reinterpret_cast<const __half2 *>(&b), off);
    lo = *reinterpret_cast<const uint32_t *>(&x);
    hi = *reinterpret_cast<const uint32_t *>(&y);
}

template <int NI, int LS>
struct CrtShape {
    static constexpr int ND = 2 * LS;  // step offsets
    static constexpr int W_TILE = NI * BK * 2, W_STAGE = ND * W_TILE, A8_STAGE = ND * A8_TILE;
    // tensor memory: LS NI accumulator columns, then TA stages of ND FP16 tiles of 32 columns
    static constexpr int TA = LS <= 3 ? 2 : 1, kTmemA = 512 - TA * ND * 32;
    static_assert(LS * NI <= kTmemA && LS * NI <= 256, "tensor memory");
    static constexpr int NG = LS == 2 ? 2 : 1, GC = LS * NI / NG;  // groups reduced together, their columns
    // one CTA per SM (it takes all of the tensor memory)
    static constexpr size_t used = (size_t)NST * (W_STAGE + A8_STAGE) + 1024 + 256, bytes = used > 118784 ? used : 118784;
};

// x mod p into [-(p-1)/2 - p, (p-1)/2 + p] for an integer-valued |x| < 2^24 (exact): the FP32
// quotient may be one off near a half-integer, which leaves a congruent value within 1.5 p.  The
// quotient (below 2^22) is rounded by adding and subtracting 1.5 2^23: rintf runs at an eighth of the
// FP32 rate, and 64 columns of an accumulator took 1650 cycles to reduce instead of 450
__device__ __forceinline__ float mod_small(float x, float p, float invp)
{
    const float q = __fsub_rn(__fmaf_rn(x, invp, 12582912.f), 12582912.f);
    return fmaf(-q, p, x);
}

}  // namespace

template <int NI, int LS>
__global__ void __launch_bounds__(kCrtThreads, 1) k_nf_apply_crt(const __grid_constant__ CUtensorMap mapW, NfCrtParams P)
{
    using S = CrtShape<NI, LS>;
    constexpr int ND = S::ND, A8_STAGE = S::A8_STAGE, TA = S::TA, kTmemA = S::kTmemA, NG = S::NG, GC = S::GC;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = smem + NST * S::W_STAGE;
    uint64_t *wfull = (uint64_t *)(sA + NST * A8_STAGE);  // W of a stage has arrived
    uint64_t *a8full = wfull + NST, *a8empty = a8full + NST;  // residue bytes arrived / read
    uint64_t *aready = a8empty + NST, *done = aready + NST;   // FP16 tiles in TMEM / the stage's MMAs have completed
    uint64_t *tfull = done + NST, *tempty = tfull + 2;
    uint32_t *tmem_slot = (uint32_t *)(tempty + 2);
    __shared__ volatile int s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&wfull[s], 1);
            mbar_init(&a8full[s], 1);
            mbar_init(&a8empty[s], 8);  // one arrival per converter warp
            mbar_init(&aready[s], 8);
            mbar_init(&done[s], 1);
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
    // each wait is bounded by about 2 s; the abort flag ends the other roles' loops
    auto wait = [&](uint64_t *bar, uint32_t parity, int code) {
        if (mbar_wait_bounded(bar, parity)) return true;
        atomicExch(P.err, code);
        s_abort = 1;
        return false;
    };
    // the same for a whole warp, which goes on or stops together (its TMEM accesses are warp-wide):
    // one lane polls
    auto warp_wait = [&](uint64_t *bar, uint32_t parity, int code) {
        bool go = true;
        if (lane == 0) go = wait(bar, parity, code) && !s_abort;
        return __all_sync(0xffffffffu, go) != 0;
    };

    if (warp == 0) {
        // ---------------- TMA of W: the tiles of a column block
        if (lane == 0) {
            int g = 0;
            for (int it = blockIdx.x; it < P.nitems && !s_abort; it += gridDim.x) {
                const CItem I(P, nib, it);
                const bool shared = P.shared[I.rhs * nib + I.ib] != 0;
                for (int kb = 0; kb < P.nkb; ++kb, ++g) {
                    const int s = g % NST;
                    if (!wait(&done[s], ((g / NST) & 1) ^ 1, 11) || s_abort) break;
                    unsigned char *d = smem + s * S::W_STAGE;
                    mbar_expect_tx(&wfull[s], S::W_STAGE);
#pragma unroll
                    for (int q = 0; q < ND; ++q)  // the steps of the interval before, then its own
                        tma_5d(d + q * S::W_TILE, &mapW, kb * BK, q < LS && shared ? LS + q : q,
                               I.ib * NI - (q < LS && shared ? 1 : 0), I.rhs, I.m, &wfull[s]);
                }
            }
            const uint64_t dl2 = gtimer() + kTimeoutNs / 20;
            for (int j = (g > NST ? g - NST : 0); j < g; ++j) mbar_wait(&wfull[j % NST], (j / NST) & 1, dl2);
        }
    } else if (warp == 18) {
        // ---------------- bulk copies of the A bytes
        if (lane == 0) {
            int g = 0;
            for (int it = blockIdx.x; it < P.nitems && !s_abort; it += gridDim.x) {
                const CItem I(P, nib, it);
                const unsigned char *src = P.A + ((size_t)I.m * P.ntiles + I.tile) * P.nkb * A8_STAGE;
                for (int kb = 0; kb < P.nkb; ++kb, ++g, src += A8_STAGE) {
                    const int s = g % NST;
                    if (!wait(&a8empty[s], ((g / NST) & 1) ^ 1, 12) || s_abort) break;
                    mbar_expect_tx(&a8full[s], A8_STAGE);
                    bulk_copy(sA + s * A8_STAGE, src, A8_STAGE, &a8full[s]);
                }
            }
            const uint64_t dl2 = gtimer() + kTimeoutNs / 20;
            for (int j = (g > NST ? g - NST : 0); j < g; ++j) mbar_wait(&a8full[j % NST], (j / NST) & 1, dl2);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        const uint32_t issue = elect_lane(), tm = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t wlo = __shfl_sync(0xffffffffu, (su32(smem) >> 4) & 0x3FFFu, 0) | 1u << 16;
        constexpr uint32_t WT = S::W_TILE >> 4;
        int g = 0;
        uint32_t ev0 = 0, ev1 = 0;  // accumulator hand-overs of the groups
        for (int it = blockIdx.x; it < P.nitems && !s_abort; it += gridDim.x) {
            const CItem I(P, nib, it);
            const int rp = c_red[LS][I.m];
            // the previous item's outputs have been read
            bool ok = (ev0 == 0 || wait(&tempty[0], (ev0 - 1) & 1, 13)) && (ev1 == 0 || wait(&tempty[1], (ev1 - 1) & 1, 13));
            int next0 = rp, next1 = rp / 2;  // column blocks before which a group is reduced
            for (int kb = 0; kb < P.nkb && ok; ++kb, ++g) {
                const int s = g % NST;
                const uint32_t w0 = wlo + s * (S::W_STAGE >> 4), at = tm + kTmemA + g % TA * (ND * 32);
                const bool r0 = kb == next0, r1 = NG == 2 && kb == next1;
                if (r0) {
                    mma_commit_if(issue, &tfull[0]);
                    ++ev0;
                    next0 += rp;
                }
                if (r1) {
                    mma_commit_if(issue, &tfull[1]);
                    ++ev1;
                    next1 += rp;
                }
                ok = wait(&wfull[s], (g / NST) & 1, 14) && wait(&aready[s], (g / NST) & 1, 15);
                if (ok && NG == 1 && r0) ok = wait(&tempty[0], (ev0 - 1) & 1, 16);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // offset d for the np phases from p0
                auto offset = [&](int d, int p0, int np, uint32_t first) {
                    const uint32_t id = idesc_f16(BM, np * NI);
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        mma_f16_ts(issue, tm + p0 * NI, at + d * 32 + kk * 8, w0 + (LS + p0 - d) * WT + kk * 2, id,
                                   kk == 0 ? first : 1u);
                };
                if (NG == 1 || (!r0 && !r1)) {
                    // the first MMA of an item, of offset 0, starts all phases from zero
#pragma unroll
                    for (int d = 0; d < ND; ++d) {
                        const int p0 = d > LS ? d - LS : 0;
                        offset(d, p0, LS - p0, d == 0 ? (kb > 0 ? 1u : 0u) : 1u);
                    }
                } else {
                    // the other phase first, while the epilogue reduces this one
                    auto phase = [&](int ph) {
#pragma unroll
                        for (int d = 0; d < ND; ++d)
                            if (d <= LS + ph) offset(d, ph, 1, 1u);
                    };
                    if (r0) {
                        phase(1);
                        if (!(ok = wait(&tempty[0], (ev0 - 1) & 1, 16))) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        phase(0);
                    } else {
                        phase(0);
                        if (!(ok = wait(&tempty[1], (ev1 - 1) & 1, 17))) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        phase(1);
                    }
                }
                mma_commit_if(issue, &done[s]);
            }
            mma_commit_if(issue, &tfull[0]);
            ++ev0;
            if (NG == 2) {
                mma_commit_if(issue, &tfull[1]);
                ++ev1;
            }
        }
    } else if (warp < 10) {
        // ---------------- converters: thread = row; the bytes of LS offsets to FP16 pairs in TMEM
        const int row = (warp & 3) * 32 + lane, d0 = ((warp - 2) >> 2) * LS;
        const uint32_t tq = tmem + ((uint32_t)((warp & 3) * 32) << 16) + kTmemA + d0 * 32;
        int g = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < P.nitems && ok; it += gridDim.x)
            for (int kb = 0; kb < P.nkb; ++kb, ++g) {
                const int s = g % NST;
                if (!(ok = warp_wait(&a8full[s], (g / NST) & 1, 18))) break;
                uint4 b[LS][4];
#pragma unroll
                for (int d = 0; d < LS; ++d) {
                    // 16-byte chunk c of row r is at c ^ ((r / 2) mod 4): a quarter warp reads all banks
                    const unsigned char *src = sA + s * A8_STAGE + (d0 + d) * A8_TILE + row * 64;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        b[d][c] = *reinterpret_cast<const uint4 *>(src + ((c ^ ((row >> 1) & 3)) << 4));
                }
                uint32_t v[32];
                auto convert = [&](const uint4(&q)[4]) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        bytes_to_half(q[c].x, v[8 * c], v[8 * c + 1]);
                        bytes_to_half(q[c].y, v[8 * c + 2], v[8 * c + 3]);
                        bytes_to_half(q[c].z, v[8 * c + 4], v[8 * c + 5]);
                        bytes_to_half(q[c].w, v[8 * c + 6], v[8 * c + 7]);
                    }
                };
                convert(b[0]);
                __syncwarp();
                if (lane == 0) mbar_arrive(&a8empty[s]);
                // the MMAs of column block g - TA, which read these tiles' place, have completed
                const int gd = g - TA;
                if (gd >= 0 && !(ok = warp_wait(&done[gd % NST], (gd / NST) & 1, 19))) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t ts = tq + g % TA * (ND * 32);
                tmem_st32_async(ts, v);
#pragma unroll
                for (int d = 1; d < LS; ++d) {
                    convert(b[d]);
                    tmem_st32_async(ts + d * 32, v);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&aready[s]);
            }
    } else {
        // ---------------- epilogue: warps 10..17, TMEM lane quadrant = warp % 4, every other 32 columns
        constexpr int NCH = GC / 32, NC = (NCH + 1) / 2;  // 32-column chunks of a group, of a warp
        const int quad = warp & 3, half = (warp - 10) >> 2;
        uint32_t ev[2] = {0, 0};
        bool ok = true;
        for (int it = blockIdx.x; it < P.nitems && ok; it += gridDim.x) {
            const CItem I(P, nib, it);
            const float p = c_pf[I.m], invp = c_invp[I.m];
            const int rp = c_red[LS][I.m] / NG;
            bool odd = NG == 2;  // of two groups the second is reduced first, then in turn
            for (int kb = rp; ok; kb += rp, odd = NG == 2 && !odd) {
                const bool last = kb >= P.nkb;
#pragma unroll
                for (int gr = 0; gr < NG; ++gr) {
                    if (!ok || (!last && (gr == 1) != odd)) continue;
                    if (!(ok = warp_wait(&tfull[gr], ev[gr]++ & 1, 20))) continue;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t tb = tmem + ((uint32_t)(quad * 32) << 16) + gr * GC;
                    if (!last) {
                        uint32_t v[NC][32];
#pragma unroll
                        for (int c = 0; c < NC; ++c)
                            if (2 * c + half < NCH) tmem_ld32_async(tb + (2 * c + half) * 32, v[c]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            if (2 * c + half >= NCH) continue;
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                v[c][j] = __float_as_uint(mod_small(__uint_as_float(v[c][j]), p, invp));
                            tmem_st32_async(tb + (2 * c + half) * 32, v[c]);
                        }
                        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    } else {
                        const int row = I.tile * BM + quad * 32 + lane;
                        unsigned char *out = P.res + ((size_t)I.m * P.nrhs + I.rhs) * P.Et * (size_t)P.nt + row;
#pragma unroll 1
                        for (int c = half; c < NCH; c += 2) {
                            uint32_t v[32];
                            tmem_ld32(tb + c * 32, v);
                            const int col = gr * GC + c * 32, ph = col / NI, iv0 = I.ib * NI + col % NI;
                            if (row < P.nt) {
#pragma unroll
                                for (int j = 0; j < 32; ++j) {
                                    float r = mod_small(__uint_as_float(v[j]), p, invp);
                                    r = r < 0.f ? r + p : r;
                                    r = r < 0.f ? r + p : r;
                                    r = r >= p ? r - p : r;
                                    if (iv0 + j < P.nint)
                                        out[(unsigned)(LS * (iv0 + j) + ph) * (unsigned)P.nt] = (unsigned char)(int)r;
                                }
                            }
                        }
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[gr]);
                }
                if (last) break;
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
// scaling and residues

// largest |A| of every target row over the step offsets and columns of its panel, as FP64 bits
// (non-negative doubles order as unsigned integers), into rowmax[row0 + r]
__global__ void k_row_absmax(const double *__restrict__ A, const PanelGPU *__restrict__ panels, int npanel, int kop,
                             int nd, unsigned long long *__restrict__ rowmax)
{
    const PanelGPU &Pn = panels[blockIdx.y];
    const int cols = kop ? Pn.colsK_pad : Pn.colsV_pad;
    const long long off = kop ? Pn.offK : Pn.offV;
    for (int r = blockIdx.x; r < Pn.nrows; r += gridDim.x) {
        unsigned long long m = 0ull;
        for (int d = 0; d < nd; ++d) {
            const unsigned long long *a =
                reinterpret_cast<const unsigned long long *>(A + off + ((size_t)d * Pn.rows_pad + r) * cols);
            for (int c = threadIdx.x; c < cols; c += blockDim.x) {
                const unsigned long long v = a[c] & 0x7fffffffffffffffull;
                m = v > m ? v : m;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
            m = v > m ? v : m;
        }
        if ((threadIdx.x & 31) == 0) atomicMax(rowmax + Pn.row0 + r, m);
    }
}

// exponent e with 2^e m in [2^(b-1), 2^b) for the FP64 bits of m (0 for m = 0 or non-finite)
__host__ __device__ inline int crt_scale_exp(unsigned long long bits, int b)
{
    bits &= 0x7fffffffffffffffull;
    const int be = (int)(bits >> 52);
    if (bits == 0ull || be == 2047) return 0;
    const int E = (be == 0) ? -1074 + 63 - __builtin_clzll(bits) : be - 1023;  // m in [2^E, 2^(E+1))
    return b - 1 - E;
}

// v 2^e, rounded once where the result is subnormal
__device__ __forceinline__ double scale2(double v, int e)
{
    if (e >= -1022 && e <= 1023) return v * __longlong_as_double((long long)(1023 + e) << 52);
    return ldexp(v, e);
}

// balanced residue of an integer-valued x (|x| < 2^22) modulo p, in [-(p-1)/2, (p-1)/2]: the
// FP32 quotient of mod_small is off by at most one, so one correction each way suffices
__device__ __forceinline__ float mod_balanced(float x, float p, float invp)
{
    float t = mod_small(x, p, invp);
    const float hp = 0.5f * (p - 1.f);
    t = t > hp ? t - p : t;
    return t < -hp ? t + p : t;
}

// balanced residues of the integer a (|a| < 2^55) modulo the 16 primes, exactly in FP32: |a| is
// cut into five 11-bit digits a_k and sum_k a_k (2^(11 k) mod p) < 5 * 2^11 * 2^8 < 2^22 is reduced
// once; the residue of -a is minus that of a
__device__ __forceinline__ void residues16(long long a, float (&r)[kCrtModuli])
{
    const bool neg = a < 0;
    const unsigned long long u = neg ? 0ull - (unsigned long long)a : (unsigned long long)a;
    float dg[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) dg[k] = (float)(unsigned)((u >> (11 * k)) & 0x7ffull);
#pragma unroll
    for (int m = 0; m < kCrtModuli; ++m) {
        float x = dg[0];
#pragma unroll
        for (int k = 1; k < 5; ++k) x = fmaf(dg[k], c_pow11[m][k], x);
        const float t = mod_balanced(x, c_pf[m], c_invp[m]);
        r[m] = neg ? -t : t;
    }
}

// FP64 panels -> residues of A' = rint(2^e_x A) for every modulus as bytes r + 128, [modulus][tile]
// [column block][d][128 rows][64 columns] with the 16-byte chunks of row r at c ^ ((r / 2) mod 4); rows
// past the last triangle are zero.  Thread per (row, d, four columns)
__global__ void k_crt_split_panel(const double *__restrict__ A, const PanelGPU *__restrict__ panels,
                                  const int *__restrict__ tri_leaf, const int *__restrict__ rowexp, int kop, int nt,
                                  int ntiles, int ncp, int nd, unsigned char *__restrict__ res)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int nq = ncp / 4, c = (int)(i % nq) * 4;
    const size_t rd = i / nq;
    const int x = (int)(rd / nd), d = (int)(rd - (size_t)x * nd);
    if (x >= ntiles * BM) return;
    const int nkb = ncp / BK, row = x & (BM - 1), ch = ((c & 63) >> 4) ^ ((row >> 1) & 3);
    double e[4] = {0.0, 0.0, 0.0, 0.0};
    if (x < nt) {
        const PanelGPU &Pn = panels[tri_leaf[x]];
        const double2 *a = reinterpret_cast<const double2 *>(
            A + (kop ? Pn.offK : Pn.offV) + ((size_t)d * Pn.rows_pad + (x - Pn.row0)) * ncp + c);
        const double2 p = a[0], q = a[1];
        const int sc = rowexp[x];
        e[0] = scale2(p.x, sc);
        e[1] = scale2(p.y, sc);
        e[2] = scale2(q.x, sc);
        e[3] = scale2(q.y, sc);
    }
    uint32_t w[kCrtModuli];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float r[kCrtModuli];
        residues16(__double2ll_rn(e[j]), r);
#pragma unroll
        for (int m = 0; m < kCrtModuli; ++m) w[m] = (j ? w[m] : 0u) | (uint32_t)((int)r[m] + 128) << (8 * j);
    }
    const size_t per_m = (size_t)ntiles * nkb * nd * A8_TILE;
    const size_t o = (((size_t)(x / BM) * nkb + c / BK) * nd + d) * A8_TILE + row * 64 + ch * 16 + (c & 15);
#pragma unroll
    for (int m = 0; m < kCrtModuli; ++m) *reinterpret_cast<uint32_t *>(res + m * per_m + o) = w[m];
}

// per-row exponents
__global__ void k_row_exps(const unsigned long long *__restrict__ rowmax, int nt, int b, int *__restrict__ rowexp)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < nt) rowexp[x] = crt_scale_exp(rowmax[x], b);
}

// scales of the input.  Every (rhs, leaf interval) goes to nsplit CTAs, each of which writes its largest finite |x|
// as FP64 bits (sign bit: there are other values) to part.  The last CTA to finish adds them up and sets, for the
// outputs of each interval (whose products read it and the one before), win = the scale exponent of the rhs's
// largest |x|, or of the two intervals' where that is more than kCrtSlack binary orders smaller; bit 0 of win
// tells of values that are not finite.  shared of a tile of ni intervals: the exponent never changes.
// ticket is zero between products.  With the split that follows 1 to 4 us more than one scale per rhs took
// (12288 triangles x 256 steps: product 4.43 -> 4.45 ms)
constexpr int kCrtSlack = 2;
__global__ void __launch_bounds__(256) k_crt_scales(CrtInput in, int nsplit, int ni)
{
    constexpr unsigned long long kNot = 1ull << 63;
    __shared__ unsigned long long red[8];
    __shared__ bool last;
    const int nint = in.Et / in.ls, nw = in.nrhs * nint, w = blockIdx.x / nsplit;
    const size_t per = (size_t)in.ls * in.ncol;
    const unsigned long long *xr = reinterpret_cast<const unsigned long long *>(in.x) + w * per;
    unsigned long long m = 0ull;
    bool nf = false;
    for (size_t i = (size_t)(blockIdx.x % nsplit) * blockDim.x + threadIdx.x; i < per; i += (size_t)nsplit * blockDim.x) {
        const unsigned long long v = xr[i] & ~kNot;
        const bool finite = v < 0x7ff0000000000000ull;
        nf |= !finite;
        m = finite && v > m ? v : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
        m = v > m ? v : m;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    nf = __syncthreads_or(nf) != 0;
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) m = red[q] > m ? red[q] : m;
        in.part[blockIdx.x] = nf ? m | kNot : m;
        __threadfence();
        last = atomicAdd(in.ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int nib = (nint + ni - 1) / ni;
    for (int i = threadIdx.x; i < in.nrhs * nib; i += blockDim.x) in.shared[i] = 1;
    for (int i = threadIdx.x; i < in.nrhs; i += blockDim.x) in.all[i] = 0ull;
    if (threadIdx.x == 0) *in.ticket = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < nw; i += blockDim.x) {
        unsigned long long v = 0ull, bad = 0ull;
        for (int q = 0; q < nsplit; ++q) {
            const unsigned long long u = __ldcg(in.part + (size_t)i * nsplit + q);
            v = (u & ~kNot) > v ? u & ~kNot : v;
            bad |= u & kNot;
        }
        in.wmax[i] = v | bad;
        atomicMax(in.all + i / nint, v);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nw; i += blockDim.x) {
        const int iv = i % nint;
        unsigned long long v[3], bad = 0ull;  // this interval's, the one's before and the one's before that
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            v[q] = iv >= q ? in.wmax[i - q] : 0ull;
            if (q < 2) bad |= v[q] & kNot;
            v[q] &= ~kNot;
        }
        const int ea = crt_scale_exp(__ldcg(in.all + i / nint), in.b);
        auto window = [&](unsigned long long x, unsigned long long y) {
            const unsigned long long m = x > y ? x : y;
            const int e = crt_scale_exp(m, in.b);
            return m == 0ull || e - ea <= kCrtSlack ? ea : e;
        };
        const int e = window(v[0], v[1]);
        in.win[i] = e * 2 + (bad ? 1 : 0);
        if (iv > 0 && e != window(v[1], v[2])) in.shared[i / nint * nib + iv / ni] = 0;
    }
}

// input: W' = rint(2^s x) permuted (V) or padded (K), 0 where x is not finite, with the scale of its own
// interval's outputs as steps ls .. 2 ls - 1 and, where a tile of ni intervals is not shared, with that of
// the next interval's as its steps 0 .. ls - 1; residues [modulus][rhs][interval][2 ls][ncol_pad]
__global__ void k_crt_split_input(CrtInput in, size_t total, int ni, __half *__restrict__ res)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int ls = in.ls, nint = in.Et / ls, nib = (nint + ni - 1) / ni;
    const unsigned rt = i >> 32 ? (unsigned)(i / in.ncol_pad) : (unsigned)i / (unsigned)in.ncol_pad, rhs = rt / (unsigned)in.Et;
    const int c = (int)(i - (size_t)rt * in.ncol_pad), t = (int)(rt - rhs * in.Et), iv = t / ls, s = t - iv * ls;
    const size_t w = (size_t)rhs * nint + iv;
    double v = c < in.ncol ? in.x[(size_t)rt * in.ncol + (in.perm ? in.perm[c] : c)] : 0.0;
    if (!isfinite(v)) v = 0.0;
    const bool more = iv + 1 < nint;  // the next interval's outputs read this step as well
    const int e0 = in.win[w] >> 1, e1 = more ? in.win[w + 1] >> 1 : e0;
    const bool next_shared = !more || in.shared[rhs * nib + (iv + 1) / ni], first_shared = iv > 0 || in.shared[rhs * nib];
    // element of (interval iv, step ls + s); the next interval's step s is ls steps on
    __half *o = res + (w * 2 * ls + ls + s) * in.ncol_pad + c;
    const size_t per_m = 2 * total, next = (size_t)ls * in.ncol_pad;
    if (!first_shared) {
#pragma unroll
        for (int m = 0; m < kCrtModuli; ++m) (o - next)[m * per_m] = __float2half_rn(0.f);
    }
#pragma unroll 1
    for (int q = 0; q < (next_shared ? 1 : 2); ++q, o += next) {
        float r[kCrtModuli];
        residues16(__double2ll_rn(scale2(v, q ? e1 : e0)), r);
#pragma unroll
        for (int m = 0; m < kCrtModuli; ++m) o[m * per_m] = __float2half_rn(r[m]);
    }
}

// f[rhs][t][row] = X 2^-(e_row + s), X from its residues by Garner's algorithm: the balanced
// mixed-radix digits v_j = (r_j - sum_{k<j} v_k P_k) P_j^-1 mod p_j (P_j = p_0 ... p_{j-1}) in exact
// FP32 arithmetic (every intermediate is an integer below 2^20), then X = sum_j v_j P_j by Horner's
// rule in 128-bit integers (|X| < M / 2 < 2^123, exact) and one conversion to FP64.  The products of inputs
// that are not finite follow in FP64 from the stored blocks
__global__ void k_crt_combine(const unsigned char *__restrict__ res, size_t per_mod, CrtInput in,
                              const int *__restrict__ rowexp, double *__restrict__ f)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= per_mod) return;
    if (i == 0) *in.ticket = 0u;  // whatever overlapped: the next product's scales count from zero
    float acc[kCrtModuli], v[kCrtModuli];
#pragma unroll
    for (int k = 0; k < kCrtModuli; ++k) acc[k] = 0.f;
#pragma unroll
    for (int j = 0; j < kCrtModuli; ++j) {
        const float p = c_pf[j], invp = c_invp[j];
        const float t = mod_small((float)res[(size_t)j * per_mod + i] - acc[j], p, invp);
        v[j] = mod_balanced(t * c_invPif[j], p, invp);
#pragma unroll
        for (int k = j + 1; k < kCrtModuli; ++k) acc[k] = fmaf(v[j], c_pjmodpif[j][k], acc[k]);
    }
    __int128 X = (__int128)(int)v[kCrtModuli - 1];
#pragma unroll
    for (int j = kCrtModuli - 2; j >= 0; --j) X = X * (__int128)c_p[j] + (__int128)(int)v[j];
    // |X| = hi 2^64 + lo: both parts non-negative, so the two roundings cannot cancel
    const bool neg = X < 0;
    const unsigned __int128 U = neg ? (unsigned __int128)0 - (unsigned __int128)X : (unsigned __int128)X;
    const unsigned long long hi = (unsigned long long)(U >> 64), lo = (unsigned long long)U;
    const double ax = hi ? fma((double)hi, 18446744073709551616.0, (double)lo) : (double)lo;
    const double x = neg ? -ax : ax;
    const unsigned rt = i >> 32 ? (unsigned)(i / in.nt) : (unsigned)i / (unsigned)in.nt, rhs = rt / (unsigned)in.Et;
    const int row = (int)(i - (size_t)rt * in.nt), t = (int)(rt - rhs * in.Et), nint = in.Et / in.ls, iv = t / in.ls;
    const int win = in.win[(size_t)rhs * nint + iv];
    double y = scale2(x, -(rowexp[row] + (win >> 1)));
    if (win & 1) {
        const PanelGPU &Pn = in.panels[in.tri_leaf[row]];
        const double *a = in.A + (in.kop ? Pn.offK : Pn.offV) + (size_t)(row - Pn.row0) * in.ncol_pad;
        for (int d = 0; d <= t - (iv - 1) * in.ls && d <= t; ++d, a += (size_t)Pn.rows_pad * in.ncol_pad)
            for (int c = 0; c < in.ncol && y == y; ++c) {  // NaN stays
                const double v = in.x[(size_t)(rt - d) * in.ncol + (in.perm ? in.perm[c] : c)];
                if (!isfinite(v)) y += a[c] * v;
            }
    }
    f[i] = y;
}

// ------------------------------------------------------------------------------------------
// host side

static int g_moduli[kCrtModuli] = {251, 241, 239, 233, 229, 227, 223, 211, 199, 197, 193, 191, 181, 179, 173, 167};

static long long modinv(long long a, long long p)
{
    long long t = 0, nt = 1, r = p, nr = ((a % p) + p) % p;
    while (nr) {
        long long q = r / nr, tmp = t - q * nt;
        t = nt;
        nt = tmp;
        tmp = r - q * nr;
        r = nr;
        nr = tmp;
    }
    return t < 0 ? t + p : t;
}

int crt_upload_constants(cudaStream_t st)
{
    static bool done[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
    if (done[dev]) return 0;
    float invp[kCrtModuli], pf[kCrtModuli], pow11[kCrtModuli][5];
    int red[5][kCrtModuli] = {{0}};
    float pj[kCrtModuli][kCrtModuli] = {{0.f}}, invPi[kCrtModuli];
    for (int i = 0; i < kCrtModuli; ++i) {
        pf[i] = (float)g_moduli[i];
        invp[i] = 1.0f / (float)g_moduli[i];
        // largest r (LS = 2: even) with 128 LS r ((p - 1) / 2)^2 + 1.5 p < 2^24
        const long long hp = (g_moduli[i] - 1) / 2;
        for (int ls = 1; ls <= 4; ++ls) red[ls][i] = (int)(((1ll << 24) - 2 * g_moduli[i]) / (128 * ls * hp * hp));
        red[2][i] &= ~1;
        long long q = 1;  // p_0 ... p_{j-1} mod p_i, for j = 0 .. i
        for (int j = 0; j < i; ++j) {
            pj[j][i] = (float)q;
            q = q * g_moduli[j] % g_moduli[i];
        }
        invPi[i] = (float)modinv(q, g_moduli[i]);
        long long w = 1;  // 2^(11 k) mod p_i
        for (int k = 0; k < 5; ++k) {
            pow11[i][k] = (float)w;
            w = (w << 11) % g_moduli[i];
        }
    }
    if (cudaMemcpyToSymbolAsync(c_p, g_moduli, sizeof(g_moduli), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_pf, pf, sizeof(pf), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_red, red, sizeof(red), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_invp, invp, sizeof(invp), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_pow11, pow11, sizeof(pow11), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_pjmodpif, pj, sizeof(pj), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_invPif, invPi, sizeof(invPi), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return -1;
    done[dev] = true;
    return 0;
}

int crt_bits(long long k_total)
{
    double l2m = 0.0;
    for (int i = 0; i < kCrtModuli; ++i) l2m += std::log2((double)g_moduli[i]);
    int lk = 0;
    while ((1ll << lk) < k_total) ++lk;
    const int b = (int)std::floor((l2m - 1.0 - lk) / 2.0);
    return std::min(b, 53);
}

void launch_crt_row_exps(const double *A, const PanelGPU *panels, int npanel, int kop, int nd, int b,
                         unsigned long long *rowmax, int nt, int *rowexp, cudaStream_t st)
{
    cudaMemsetAsync(rowmax, 0, sizeof(unsigned long long) * nt, st);
    k_row_absmax<<<dim3(64, npanel), 256, 0, st>>>(A, panels, npanel, kop, nd, rowmax);
    k_row_exps<<<(nt + 255) / 256, 256, 0, st>>>(rowmax, nt, b, rowexp);
}

size_t crt_panel_bytes(int nt, int ncp, int nd)
{
    return (size_t)kCrtModuli * ((nt + BM - 1) / BM) * (ncp / BK) * nd * A8_TILE;
}

void launch_crt_split_panel(const double *A, const PanelGPU *panels, const int *tri_leaf, const int *rowexp, int kop,
                            int nt, int ncp, int nd, unsigned char *res, cudaStream_t st)
{
    const int ntiles = (nt + BM - 1) / BM;
    const size_t n = (size_t)ntiles * BM * nd * (ncp / 4);
    k_crt_split_panel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(A, panels, tri_leaf, rowexp, kop, nt, ntiles, ncp, nd,
                                                                  res);
}

// CTAs of k_crt_scales per interval: about 2048 values each, or more where the intervals fill the GPU
static int crt_nsplit(size_t nw, size_t per)
{
    return (int)std::max<size_t>(1, std::min<size_t>((per + 2047) / 2048, (1216 + nw - 1) / nw));
}

// part: at most nw + 1216 CTAs
size_t crt_scratch_words(int nrhs, int Et, int ls) { return (size_t)nrhs * (Et / ls) * 3 + 1216 + nrhs + 1; }

void crt_scratch(CrtInput &in, unsigned long long *p)
{
    const size_t nw = (size_t)in.nrhs * (in.Et / in.ls);
    in.ticket = (unsigned *)p;
    in.all = p + 1;
    in.wmax = in.all + in.nrhs;
    in.part = in.wmax + nw;
    in.win = (int *)(in.part + nw + 1216);
    in.shared = in.win + nw;  // at most one a (rhs, interval)
}

void launch_crt_split_input(const CrtInput &in, int ni, void *res, cudaStream_t st)
{
    const size_t nw = (size_t)in.nrhs * (in.Et / in.ls), per = (size_t)in.ls * in.ncol;
    const int nsplit = crt_nsplit(nw, per);
    k_crt_scales<<<(unsigned)(nw * nsplit), 256, 0, st>>>(in, nsplit, ni);
    const size_t total = (size_t)in.nrhs * in.Et * in.ncol_pad;
    k_crt_split_input<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(in, total, ni, (__half *)res);
}

void launch_crt_combine(const unsigned char *res, const CrtInput &in, const int *rowexp, double *f, cudaStream_t st)
{
    const size_t per_mod = (size_t)in.nrhs * in.Et * in.nt;
    k_crt_combine<<<(unsigned)((per_mod + 255) / 256), 256, 0, st>>>(res, per_mod, in, rowexp, f);
}

int nf_crt_intervals(int nint, int ls, int form)
{
    // the MMA's columns are LS NI: few intervals take the narrowest block that holds them; three and
    // four steps per leaf leave room for 32 intervals beside the A tiles in tensor memory
    if (ls > 2) return 32;
    return nint <= 32 ? 32 : (nint <= 64 || form == 2 ? 64 : 128);
}

template <int NI, int LS>
static int launch_crt_T(const CUtensorMap &W, NfCrtParams P, int nsm, cudaStream_t st)
{
    P.nitems = kCrtModuli * P.ntiles * ((P.nint + NI - 1) / NI) * P.nrhs;
    auto kf = k_nf_apply_crt<NI, LS>;
    const size_t smem = CrtShape<NI, LS>::bytes;
    if (cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -1;
    kf<<<std::min(P.nitems, nsm), kCrtThreads, smem, st>>>(W, P);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_nf_apply_crt(const CUtensorMap &W, const NfCrtParams &P, int ls, int nsm, cudaStream_t st, int form)
{
    const int ni = nf_crt_intervals(P.nint, ls, form);
    switch (ls) {
    case 1:
        return ni == 32   ? launch_crt_T<32, 1>(W, P, nsm, st)
               : ni == 64 ? launch_crt_T<64, 1>(W, P, nsm, st)
                          : launch_crt_T<128, 1>(W, P, nsm, st);
    case 2:
        return ni == 32   ? launch_crt_T<32, 2>(W, P, nsm, st)
               : ni == 64 ? launch_crt_T<64, 2>(W, P, nsm, st)
                          : launch_crt_T<128, 2>(W, P, nsm, st);
    case 3: return launch_crt_T<32, 3>(W, P, nsm, st);
    case 4: return launch_crt_T<32, 4>(W, P, nsm, st);
    default: return -1;
    }
}

}  // namespace pfmm
