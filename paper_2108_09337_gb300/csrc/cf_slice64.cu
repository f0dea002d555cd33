// cf_slice64.cu -- CH-3 of the FP64 path on the tensor cores:
//     C -= L10 L10^T (lower), L10 m x w
//
// GB300 runs FP64 at ~2 fused multiply-adds per clock per SM (1.20 TFLOP/s
// measured), so the update as FP64 code is bound by that pipe; the BF16 tensor
// cores run 1500 times faster and form the same product exactly from small
// integers:
//   * per row of L10 the elements become integers of at most 62 bits relative
//     to the row's largest exponent and eight balanced base-256 digits (the top
//     one in [-64, 64], the others in [-128, 127]), exact in BF16;
//   * Q_d = sum_{s+t=d} sum_j d_s e_t, d = 0..7: for every row digit s one
//     chain of tcgen05 MMAs against the column digits t = 0..7-s, accumulating
//     into the TMEM columns of diagonal s + t.  A sum holds at most 128
//     products of each of at most 8 digit pairs, two of them with a top digit:
//     at most 7 x 2^21 < 2^24, so the FP32 accumulation is exact in any order;
//   * C -= 2^(E_i + E_k - 4158) sum_d Q_d 256^(7-d): the 76-bit integer sum is
//     rounded to FP64 once and subtracted with a second rounding.
// The error is a few 2^-62 of (max of row i) x (max of row k) per term and one
// rounding of the sum, where the FP64 loop rounds w partial sums.  A Cholesky
// factor's rows are bounded by the diagonal, |l_ij| <= sqrt(a_ii), so this is
// below the factorization's own error u sqrt(a_ii a_kk) whatever the rows'
// scales.  LU has no such bound (one large element of U in one column would take
// the bits of all others): its update is the FP64 loop.
// Every C element's value is a function of its row and its column alone, so it
// does not depend on how the update is cut into pieces.
//
// Rows with an infinity, a NaN or scales whose product could leave the normal
// range flag their tile, and flagged tiles are done by the FP64 loop
// (k_gemm_flagged), with that loop's results.
//
// Kernel layout: persistent CTAs over 128 x 64 tiles of C, column-tile major,
// so that a CTA's column digits (128 KB) stay in shared memory while the row
// digits (16 KB tiles, six in flight) stream through from L2; 8 diagonals x 64
// columns fill the 512 TMEM columns.  Per tile: 36 digit pairs = 9,200 tensor
// clocks; sixteen epilogue warps combine the diagonals in integers as they
// leave TMEM (the accumulators are free again after the read), then do the
// rounding and the one FP64 operation per element beside the next tile's MMAs.
#include <climits>

#include <cuda_bf16.h>

#include "cf_common.cuh"
#include "cf_kernels.cuh"
#include "cf_slice64.cuh"
#include "cf_tc.cuh"
#include "cf_umma.cuh"

namespace cf {

__device__ int g_slice64_status = 0;       // 0 or CF_ERR_TIMEOUT

namespace s64 {

using namespace umma;

constexpr int ND = 8;                  // digits per element
constexpr int BM = 128, BN = 64, BK = 64;
constexpr int UMMA_K = 16;
constexpr int AST = 6;                 // row digit tiles in flight
constexpr int EPI = 16;                // epilogue warps: 4 lane quarters x 4 groups of 16 columns
constexpr int kThreads = 64 + 32 * EPI;
constexpr uint32_t kABytes = BM * BK * 2;          // one digit of 128 rows x 64 k
constexpr uint32_t kBHalf = BN * BK * 2;           // one digit of 64 rows x 64 k
constexpr uint32_t kBBytes = 2 * ND * kBHalf;      // all digits of 64 columns x 128 k
constexpr uint32_t kTmemCols = 512;
constexpr int kCentre = 2046;          // E of a row whose largest scaled element is in [1, 2)
constexpr int kSpan = 450;             // E may be this far from it: E_i + E_k - kCentre - 994 - 95 >= 1, ... - 994 <= 2046

struct Smem {
    uint64_t afull[AST], aempty[AST];
    uint64_t bfull, bempty, acc_full, acc_empty, drain;
    uint32_t tmem_base;
    int abort_flag;
};

struct Problem {
    int m, c0, c1;                     // rows; columns [c0, c1), rows of the slices too; i >= j only
    int nkb;                           // K blocks of 64 (1 or 2)
    int ct0, ct1, nrt;                 // column tiles of 64, row tiles of 128
    long long units;
    const uint8_t *S;
    const int *E;
    const int *any, *flag;
    const int *skip;
    double *C;
    int ldc;
};

// Byte offset of the digit-d tile (128 rows x 64 k, 128-byte-swizzled image)
// of row tile rt and K block kb.
__host__ __device__ __forceinline__ size_t tile_offset(int rt, int kb, int d) {
    return (((size_t)rt * 2 + kb) * ND + d) * (size_t)kABytes;
}

// The units of a CTA: (column tile, row tile) pairs, row tiles fastest.
struct Walk {
    int ct, rt;
    __device__ void seek(const Problem &p, long long u) {
        ct = p.ct0;
        while (u >= p.nrt - ct / 2) { u -= p.nrt - ct / 2; ++ct; }
        rt = ct / 2 + (int)u;
    }
    __device__ void next(const Problem &p) {
        if (++rt >= p.nrt) { ++ct; rt = ct / 2; }
    }
};

#define TMEM_LD4(taddr, r, o)                                                                       \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"                       \
                 : "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3])                       \
                 : "r"(taddr))

// (hi 2^32 + lo) 2^(e - 2112), |hi| < 2^44, rounded to nearest (a
// tie between two doubles goes up in magnitude).  32-bit integer operations
// only (about 30): the FP64 pipe takes 64 clocks per instruction and quarter
// SM and is left to the subtraction.
__device__ __forceinline__ double scaled_double(long long hi, unsigned lo, int e) {
    const unsigned sign = (unsigned)(hi >> 63);               // all ones if negative
    unsigned long long low = ((unsigned long long)(unsigned)hi << 32) | lo;
    const unsigned long long mask = ((unsigned long long)sign << 32) | sign;
    low = (low ^ mask) - mask;
    unsigned w2 = ((unsigned)(hi >> 32) ^ sign) + ((sign != 0u && low == 0ull) ? 1u : 0u);
    unsigned w1 = (unsigned)(low >> 32), w0 = (unsigned)low;
    if (w2 == 0u) { w2 = w1; w1 = w0; w0 = 0u; e -= 32; }
    if (w2 == 0u) { w2 = w1; w1 = 0u; e -= 32; }
    const int lz = __clz((int)w2);
    const unsigned m1 = __funnelshift_lc(w1, w2, lz), m0 = __funnelshift_lc(w0, w1, lz);      // top bit of m1 set
    const unsigned field = (unsigned)(e - 2112 + 95 - lz + 1023);
    // 53 bits rounded; the leading bit adds the exponent's missing one, a carry one more
    unsigned long long b = ((unsigned long long)((m1 >> 11) + ((field - 1u) << 20)) << 32) | __funnelshift_r(m0, m1, 11);
    b += (m0 >> 10) & 1u;
    b |= (unsigned long long)(sign & 0x80000000u) << 32;
    return w2 == 0u ? 0.0 : __longlong_as_double((long long)b);
}

// An integer of magnitude at most 2^22 held in a float, without the conversion
// unit (16 lanes per clock).
__device__ __forceinline__ int small_int(float x) { return __float_as_int(x + 12582912.f) - 0x4B400000; }

__global__ void __launch_bounds__(kThreads, 1)
k_update_sliced(Problem p) {
    if (p.skip != nullptr && *p.skip != 0) return;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sB = base;
    uint8_t *sA = base + kBBytes;
    Smem &s = *reinterpret_cast<Smem *>(sA + AST * kABytes);
    volatile int *abort_flag = &s.abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long u0 = p.units * blockIdx.x / gridDim.x, u1 = p.units * (blockIdx.x + 1) / gridDim.x;

    if (threadIdx.x == 0) {
        for (int i = 0; i < AST; ++i) { mbar_init(&s.afull[i], 1); mbar_init(&s.aempty[i], 1); }
        mbar_init(&s.bfull, 1);
        mbar_init(&s.bempty, 1);
        mbar_init(&s.acc_full, 1);
        mbar_init(&s.acc_empty, EPI);
        mbar_init(&s.drain, 1);
        s.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s.tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s.tmem_base;

    if (warp == 0) {
        // ------------------------------------------------ copies
        if (lane == 0 && u0 < u1) {
            Walk wk;
            wk.seek(p, u0);
            int ia = 0, nb = 0, ct = -1;
            bool ok = true;
            for (long long u = u0; u < u1 && ok; ++u, wk.next(p)) {
                if (wk.ct != ct) {
                    ct = wk.ct;
                    if (!wait_bounded(&s.bempty, (uint32_t)(nb & 1) ^ 1u, abort_flag, &g_slice64_status)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&s.bfull, (uint32_t)p.nkb * ND * kBHalf);
                    for (int kb = 0; kb < p.nkb; ++kb)
                        for (int d = 0; d < ND; ++d)
                            asm volatile(
                                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
                                "[%3];" ::"r"(smem_u32(sB + (kb * ND + d) * kBHalf)),
                                "l"(p.S + tile_offset(ct / 2, kb, d) + (size_t)(ct & 1) * kBHalf), "r"(kBHalf),
                                "r"(smem_u32(&s.bfull))
                                : "memory");
                    ++nb;
                }
                for (int kb = 0; kb < p.nkb && ok; ++kb)
                    for (int d = 0; d < ND; ++d) {
                        const int st = ia % AST;
                        if (!wait_bounded(&s.aempty[st], ((uint32_t)(ia / AST) & 1u) ^ 1u, abort_flag,
                                          &g_slice64_status)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_expect_tx(&s.afull[st], kABytes);
                        asm volatile(
                            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                smem_u32(sA + st * kABytes)),
                            "l"(p.S + tile_offset(wk.rt, kb, d)), "r"(kABytes), "r"(smem_u32(&s.afull[st]))
                            : "memory");
                        ++ia;
                    }
            }
            if (!ok) {
                // every issued copy must land before the CTA exits
                for (long long i = 0; nb > 0 && i < kSpinLimit && !mbar_try_wait(&s.bfull, (uint32_t)(nb - 1) & 1u); ++i)
                    __nanosleep(64);
                for (int j = (ia > AST ? ia - AST : 0); j < ia; ++j) {
                    const uint32_t ph = (uint32_t)(j / AST) & 1u;
                    for (long long i = 0; i < kSpinLimit && !mbar_try_wait(&s.afull[j % AST], ph); ++i)
                        __nanosleep(64);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0 && u0 < u1) {
            Walk wk;
            wk.seek(p, u0);
            int ia = 0, nb = 0, ct = -1, n = 0;
            bool ok = true, issued = false;
            for (long long u = u0; u < u1 && ok; ++u, ++n) {
                if (wk.ct != ct) {
                    ct = wk.ct;
                    if (!wait_bounded(&s.bfull, (uint32_t)nb & 1u, abort_flag, &g_slice64_status)) { ok = false; break; }
                    ++nb;
                }
                if (!wait_bounded(&s.acc_empty, ((uint32_t)n & 1u) ^ 1u, abort_flag, &g_slice64_status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                for (int kb = 0; kb < p.nkb && ok; ++kb) {
                    const uint64_t bd = make_sw128_desc(smem_u32(sB + kb * ND * kBHalf));
                    for (int d = 0; d < ND; ++d) {
                        const int as = ia % AST;
                        if (!wait_bounded(&s.afull[as], (uint32_t)(ia / AST) & 1u, abort_flag, &g_slice64_status)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint64_t ad = make_sw128_desc(smem_u32(sA + as * kABytes));
                        // row digit d times column digits t = 0..7-d into the columns of diagonals d..7
                        const int ncol = BN * (ND - d);
                        const int n1 = ncol < 256 ? ncol : 256, n2 = ncol - n1;
                        const uint32_t id1 = make_idesc(true, BM, n1);
                        const uint32_t id2 = make_idesc(true, BM, n2 > 0 ? n2 : 16);
                        const uint32_t dst = tmem_base + (uint32_t)(BN * d);
#pragma unroll
                        for (int kk = 0; kk < BK / UMMA_K; ++kk) {
                            const uint32_t acc = (kb > 0 || d > 0 || kk > 0) ? 1u : 0u;
                            umma_f16(dst, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), id1, acc);
                            if (n2 > 0)      // 256 rows further: 32 KB
                                umma_f16(dst + 256, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2 + (256 * 128 >> 4)),
                                         id2, acc);
                        }
                        issued = true;
                        umma_commit(&s.aempty[as]);
                        ++ia;
                    }
                }
                if (!ok) break;
                umma_commit(&s.acc_full);
                wk.next(p);
                if (u + 1 < u1 && wk.ct != ct) umma_commit(&s.bempty);
            }
            if (issued) {
                umma_commit(&s.drain);
                for (long long i = 0; i < kSpinLimit && !mbar_try_wait(&s.drain, 0); ++i) __nanosleep(64);
            }
        }
    } else {
        // ------------------------------------------------ epilogue (warps 2..17)
        const int quarter = warp & 3;             // TMEM lanes 32 * quarter ..
        const int grp = (warp - 2) >> 2;          // columns 16 * grp ..
        const int any = *p.any;
        Walk wk;
        int n = 0;
        bool ok = true;
        if (u0 < u1) wk.seek(p, u0);
        for (long long u = u0; u < u1 && ok; ++u, ++n, wk.next(p)) {
            const int row = wk.rt * BM + quarter * 32 + lane;
            const int col0 = wk.ct * BN + grp * 16;
            const int Ei = row < p.m ? p.E[row] : kCentre;
            double *Cp = p.C + (size_t)row + (size_t)col0 * p.ldc;
            auto mine = [&](int c) { return row < p.m && col0 + c >= p.c0 && col0 + c < p.c1 && row >= col0 + c; };
            if (lane == 0) ok = wait_bounded(&s.acc_full, (uint32_t)n & 1u, abort_flag, &g_slice64_status);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(grp * 16);
            // the diagonals leave TMEM as one 96-bit integer per element, so that the
            // accumulators are free for the next tile before the rounding
            long long hi[16];
            unsigned lo[16];
#pragma unroll
            for (int c = 0; c < 16; c += 4) {
                uint32_t r[4 * ND];
#pragma unroll
                for (int d = 0; d < ND; ++d) TMEM_LD4(taddr + (uint32_t)(d * BN + c), r, 4 * d);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    // |S_0| <= 2^19, |S_d| <= d 2^21: S_0 .. S_2 by the FP32 pipe, and the sums
                    // formed in int32 fit it
                    const int S0 = small_int(__uint_as_float(r[q])), S1 = small_int(__uint_as_float(r[4 + q])),
                              S2 = small_int(__uint_as_float(r[8 + q]));
                    int S[ND];
#pragma unroll
                    for (int d = 3; d < ND; ++d) S[d] = __float2int_rn(__uint_as_float(r[4 * d + q]));
                    const long long low = (long long)S[4] * 16777216 + ((long long)S[5] * 65536 + ((long long)S[6] * 256 + S[7]));
                    hi[c + q] = (long long)(S0 * 256 + S1) * 65536 + (long long)(S2 * 256 + S[3]) + (low >> 32);
                    lo[c + q] = (unsigned)low;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&s.acc_empty);
            if (row >= p.m || (any && (p.flag[wk.rt] || p.flag[wk.ct / 2]))) continue;
            const int *Ek = p.E + col0;
            const int shift = Ei - kCentre;
#pragma unroll
            for (int c0 = 0; c0 < 16; c0 += 8) {
                double cv[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) cv[c] = mine(c0 + c) ? Cp[(size_t)(c0 + c) * p.ldc] : 0.0;
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (mine(c0 + c))
                        Cp[(size_t)(c0 + c) * p.ldc] = cv[c] - scaled_double(hi[c0 + c], lo[c0 + c], shift + Ek[c0 + c]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// Digit slices of the rows of L10 (A[i + j lda]).
// CTA: 32 rows x 128 j; the row's largest exponent, the digits, then
// each slice through shared memory as whole 128-byte tile rows.  Bound by the
// memory traffic of 24 bytes per element and ~40 integer operations.
// ---------------------------------------------------------------------------
constexpr int kRows = 32;
constexpr int kPitch = 2 * BK + 8;      // BF16 per staged row

__device__ __forceinline__ void digits8(double x, int sh, __nv_bfloat16 (&dg)[ND]) {
    const long long bits = __double_as_longlong(x);
    const int f = (int)((bits >> 52) & 0x7FF);
    const long long mant = bits & ((1ll << 52) - 1);
    const long long m53 = f == 0 ? mant : (mant | (1ll << 52));
    long long q;                                   // m53 2^sh, to nearest
    if (sh >= 0) q = m53 << (sh > 9 ? 9 : sh);
    else if (-sh >= 60) q = 0;
    else q = (m53 + (1ll << (-sh - 1))) >> (-sh);
    if (bits < 0) q = -q;
    // the seven low digits are the bytes of q + 128 (1 + 256 + ... + 256^6)
    // less 128 each, the top one what is left above them
    const long long t = q + 0x0080808080808080ll;
    const unsigned lo = (unsigned)t, hi = (unsigned)(t >> 32);
#pragma unroll
    for (int b = 0; b < 4; ++b) dg[ND - 1 - b] = __float2bfloat16_rn((float)((lo >> (8 * b)) & 255u) - 128.f);
#pragma unroll
    for (int b = 0; b < 3; ++b) dg[ND - 5 - b] = __float2bfloat16_rn((float)((hi >> (8 * b)) & 255u) - 128.f);
    dg[0] = __float2bfloat16_rn((float)(t >> 56));
}

struct SliceArgs {
    const double *A;
    int lda, rows, w, nkb;
    uint8_t *S;
    int *E;
    int *any, *flag;
    const int *skip;
};

__global__ void __launch_bounds__(256) k_slice_rows(SliceArgs a) {
    if (a.skip != nullptr && *a.skip != 0) return;
    __shared__ __align__(16) __nv_bfloat16 tile[kRows * kPitch];
    __shared__ int gmax[8][kRows];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = blockIdx.x * kRows;
    const int i = i0 + lane, j0 = warp * 16;
    double x[16];
#pragma unroll
    for (int c = 0; c < 16; ++c)
        x[c] = (i < a.rows && j0 + c < a.w) ? a.A[(size_t)i + (size_t)(j0 + c) * a.lda] : 0.0;
    int g[16];
    int top = INT_MIN;
    bool bad = false;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const int f = (int)((__double_as_longlong(x[c]) >> 52) & 0x7FF);
        g[c] = max(f, 1) + 1023;
        bad |= f == 0x7FF;
        if (x[c] != 0.0) top = max(top, g[c]);
    }
    gmax[warp][lane] = top;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) top = max(top, gmax[q][lane]);
    if (top == INT_MIN) top = kCentre;                  // a zero row: all digits zero
    bad |= top < kCentre - kSpan || top > kCentre + kSpan;
    if (i < a.rows) {
        if (warp == 0) a.E[i] = top;
        if (bad) {
            atomicOr(a.flag + i / BM, 1);
            atomicOr(a.any, 1);
        }
    }
    uint32_t pk[ND][8];
#pragma unroll
    for (int c = 0; c < 16; c += 2) {
        __nv_bfloat16 d0[ND], d1[ND];
        digits8(x[c], g[c] - top + 9, d0);
        digits8(x[c + 1], g[c + 1] - top + 9, d1);
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            __nv_bfloat162 h;
            h.x = d0[d];
            h.y = d1[d];
            pk[d][c / 2] = *reinterpret_cast<const uint32_t *>(&h);
        }
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        uint4 *sdst = reinterpret_cast<uint4 *>(tile + lane * kPitch + warp * 16);
        sdst[0] = make_uint4(pk[d][0], pk[d][1], pk[d][2], pk[d][3]);
        sdst[1] = make_uint4(pk[d][4], pk[d][5], pk[d][6], pk[d][7]);
        __syncthreads();
#pragma unroll
        for (int it = 0; it < 2; ++it) {
            const int c = tid + 256 * it;
            const int r = c >> 4, q = c & 15;
            const int kb = q >> 3, ch = q & 7;
            const int gi = i0 + r, rl = gi & (BM - 1);
            if (kb < a.nkb) {       // rows past m: zero digits, inside the padded tile
                const uint4 v = *reinterpret_cast<const uint4 *>(tile + r * kPitch + q * 8);
                *reinterpret_cast<uint4 *>(a.S + tile_offset(gi / BM, kb, d) + (size_t)rl * 128 +
                                           (size_t)((ch ^ (rl & 7)) * 16)) = v;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Flagged tiles in FP64: the 64 x 64 tiles of C that lie in a flagged row or
// column tile.  One element per thread at a time (the flag is rare); nothing
// flagged: one load per CTA.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_gemm_flagged(Problem p, int w, const double *__restrict__ A, int lda) {
    if (p.skip != nullptr && *p.skip != 0) return;
    if (*p.any == 0) return;
    const int nrt = (p.m + 63) / 64, ct0 = p.c0 / 64, ct1 = (p.c1 + 63) / 64;
    for (long long t = blockIdx.x; t < (long long)nrt * (ct1 - ct0); t += gridDim.x) {
        const int rt = (int)(t % nrt), ct = ct0 + (int)(t / nrt);
        if (!(p.flag[rt / 2] || p.flag[ct / 2])) continue;
        for (int e = threadIdx.x; e < 64 * 64; e += 256) {
            const int i = rt * 64 + (e & 63), j = ct * 64 + (e >> 6);
            if (i >= p.m || j < p.c0 || j >= p.c1 || i < j) continue;
            double acc = 0.0;
            for (int k = 0; k < w; ++k)
                acc = fma(A[(size_t)i + (size_t)k * lda], A[(size_t)j + (size_t)k * lda], acc);
            double *c = p.C + (size_t)i + (size_t)j * p.ldc;
            *c = *c - acc;
        }
    }
}

}  // namespace s64

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
static void carve(Carver &cv, int rows, Slice64 &s) {
    const size_t r = align_up((size_t)rows, s64::BM);
    s.rows = rows;
    s.S = cv.take<uint8_t>(r * 2 * s64::ND * 128, 1024);
    s.E = cv.take<int>(r);
    s.nflags = 4 + r / s64::BM;
    s.flags = cv.take<int>(s.nflags);
}

Slice64 slice64_carve(void *work, int rows) {
    Carver cv(work);
    Slice64 s;
    carve(cv, rows, s);
    return s;
}

size_t slice64_bytes(int rows) {
    Carver cv(nullptr);
    Slice64 s;
    carve(cv, rows, s);
    return cv.size();
}

int slice64_operand(const Slice64 &s, const double *L10, int lda, int rows, int w, const int *skip, cudaStream_t st) {
    CF_CUDA_TRY(cudaMemsetAsync(s.flags, 0, sizeof(int) * s.nflags, st));
    if (rows <= 0) return CF_OK;
    s64::SliceArgs a{};
    a.A = L10;
    a.lda = lda;
    a.rows = rows;
    a.w = w;
    a.nkb = ceil_div(w, s64::BK);
    a.S = s.S;
    a.E = s.E;
    a.any = s.any();
    a.flag = s.flag();
    a.skip = skip;
    s64::k_slice_rows<<<ceil_div(rows, s64::kRows), 256, 0, st>>>(a);
    CF_LAUNCH_CHECK();
    return CF_OK;
}

int slice64_update(const Slice64 &s, int rows, int c0, int c1, int w, const double *L10, int lda, double *C, int ldc,
                   const int *skip, cudaStream_t st) {
    using namespace s64;
    if (rows <= 0 || c1 <= c0 || w <= 0) return CF_OK;
    Problem p{};
    p.m = rows;
    p.c0 = c0;
    p.c1 = c1;
    p.nkb = ceil_div(w, BK);
    p.ct0 = c0 / BN;
    p.ct1 = ceil_div(c1, BN);
    p.nrt = ceil_div(rows, BM);
    p.units = 0;
    for (int ct = p.ct0; ct < p.ct1; ++ct) p.units += p.nrt - ct / 2;
    p.S = s.S;
    p.E = s.E;
    p.any = s.any();
    p.flag = s.flag();
    p.skip = skip;
    p.C = C;
    p.ldc = ldc;
    const int sms = device_sm_count();
    const size_t smem = 1024 + kBBytes + AST * kABytes + sizeof(Smem);
    CF_CUDA_TRY(cudaFuncSetAttribute(k_update_sliced, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_update_sliced<<<(int)(p.units < sms ? p.units : sms), kThreads, smem, st>>>(p);
    CF_LAUNCH_CHECK();
    k_gemm_flagged<<<sms, 256, 0, st>>>(p, w, L10, lda);
    CF_LAUNCH_CHECK();
    return CF_OK;
}

int slice64_take_status(cudaStream_t st, int *status) {
    int h = 0;
    CF_CUDA_TRY(cudaMemcpyFromSymbolAsync(&h, g_slice64_status, sizeof(int), 0, cudaMemcpyDeviceToHost, st));
    CF_CUDA_TRY(cudaStreamSynchronize(st));
    if (h != 0) {
        const int zero = 0;
        CF_CUDA_TRY(cudaMemcpyToSymbolAsync(g_slice64_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st));
        CF_CUDA_TRY(cudaStreamSynchronize(st));
    }
    *status = h;
    return CF_OK;
}

}  // namespace cf
