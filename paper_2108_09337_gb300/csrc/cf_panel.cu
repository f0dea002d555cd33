// cf_panel.cu -- the per-step block routines around the Schur update:
//   LU-3  A10 <- A10 U00^{-1}      (Alg. 1, "Factorize A10"; Table 2)
//   LU-4  A01 <- L00^{-1} A01      (Alg. 1, "Factorize A01")
//   A00   LU without pivoting of the selected rows (Fig. "prog_rep"): taken
//         over from the tournament's root (Sec. 7.2) where the driver has
//         room for it, which saves 0.59 ms of one SM per 128-column panel
//   CH-1  potrf of A00 (Listing "Cholesky Factorization"; Table 2, v^3/6)
//   CH-2  L10 <- A10 L00^{-T}      (Table 2: costed like the LU panel solve)
//
// The v x v triangle lives in shared memory.  LU's updates are a separately
// rounded multiply and subtract in the oracle's order, so step 0 of an LU
// reproduces the oracle's values bit for bit.
#include "cf_common.cuh"
#include "cf_kernels.cuh"

namespace cf {

constexpr int kPanelThreads = 256;
constexpr int kLdT = kMaxV;        // triangle tile leading dimension

// ---------------------------------------------------------------------------
// A00: LU without pivoting (w <= 128), one CTA.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kPanelThreads, 1)
k_getf2_nopiv(double *A, int lda, int w, int kglob, int *info, const double *lu, const int *lu_ok) {
    using T = double;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *t = reinterpret_cast<T *>(smem_raw);      // t[k*kLdT + r]
    const int tid = threadIdx.x;
    if (lu != nullptr && *lu_ok) {               // the tournament's root has done it: the same operations in the same order
        for (int idx = blockIdx.x * kPanelThreads + tid; idx < w * w; idx += gridDim.x * kPanelThreads) {
            const int k = idx / w, r = idx % w;
            A[r + (size_t)k * lda] = lu[r + (size_t)k * kMaxV];
        }
        return;
    }
    if (blockIdx.x != 0) return;
    for (int idx = tid; idx < w * w; idx += kPanelThreads) {
        const int k = idx / w, r = idx % w;
        t[k * kLdT + r] = A[r + (size_t)k * lda];
    }
    __syncthreads();
    const int r = tid & (kMaxV - 1), half = tid / kMaxV;
    for (int k = 0; k < w; ++k) {
        const T piv = t[k * kLdT + k];
        const bool act = (r > k && r < w);
        T l = T(0);
        if (act) l = (piv != T(0)) ? div_rn(t[k * kLdT + r], piv) : t[k * kLdT + r];
        if (piv == T(0) && tid == 0) atomicCAS(info, 0, kglob + k + 1);
        __syncthreads();
        if (act) {
            if (half == 0) t[k * kLdT + r] = l;
            for (int j = k + 1 + half; j < w; j += 2)
                t[j * kLdT + r] = sub_rn(t[j * kLdT + r], mul_rn(l, t[j * kLdT + k]));
        }
        __syncthreads();
    }
    for (int idx = tid; idx < w * w; idx += kPanelThreads) {
        const int k = idx / w, rr = idx % w;
        A[rr + (size_t)k * lda] = t[k * kLdT + rr];
    }
}

// ---------------------------------------------------------------------------
// A00: Cholesky (lower, w <= 128), one CTA.  Stops at the first pivot that is
// not positive (or NaN) and records info; later launches see info != 0.
//
// Bound by a chain of w pivots (square root, reciprocal, scaling, update of the
// next pivot: each FP64 operation 64 clocks) and by the FP64 pipe of one SM
// (w^3 / 6 multiply-adds, two lanes per clock).  Blocks of 16 columns, one row
// per lane: warp 0 (the block's first rows) runs the chain alone, with nothing
// else on its quarter of the SM; three helpers bring its later columns up to
// date and up to three warps follow with the rows below, from the columns, roots
// and reciprocals it leaves in shared memory; then all warps update the columns
// right of the block.  w = 128: 0.21 ms (0.56 with one barrier pair per column).
// ---------------------------------------------------------------------------
constexpr int kPB = 16;            // columns of a block
constexpr int kPotThreads = 512;
constexpr int kLdP = kMaxV + 1;

struct PotSmem {
    double t[kMaxV * kLdP];        // t[column * kLdP + row]
    double col[kPB][kPB];          // col[c][j]: finished column c at the block's row j
    double root[kPB], rinv[kPB];   // pivot and its reciprocal
    int dead[kPB];                 // 1 from the first failed pivot on
    int fail;                      // column of the failed pivot (-1: none)
};

// a / l from r ~ 1 / l (to a few ulp), corrected by the exact remainder; a zero
// is its own product, what else leaves the normal numbers is divided.
__device__ __forceinline__ double quot1(double a, double l, double r) {
    const double q0 = a * r;
    double q = fma(fma(-q0, l, a), r, q0);
    if (exp_bits(q0) - 100u >= 1900u) q = is_zero(a) && exp_bits(r) - 1u < 2046u ? q0 : div_call(a, l);
    return q;
}

// Square root of a pivot that is not a positive normal number, and its
// reciprocal; a root of -1: not positive.
static __device__ __noinline__ double2 odd_root(double d) {
    const double root = sqrt(d);
    return d > 0.0 ? make_double2(root, 1.0 / root) : make_double2(-1.0, -1.0);
}

__device__ __forceinline__ void named_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__global__ void __launch_bounds__(kPotThreads, 1)
k_potf2(double *A, int lda, int w, int kglob, int *info) {
    if (*info != 0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PotSmem &s = *reinterpret_cast<PotSmem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = warp; k < w; k += kPotThreads / 32)
        for (int r = lane; r < w; r += 32)
            if (r >= k) s.t[k * kLdP + r] = A[r + (size_t)k * lda];
    if (tid == 0) s.fail = -1;
    __syncthreads();
    for (int k0 = 0; k0 < w; k0 += kPB) {
        const int nb = min(kPB, w - k0);
        // ---- the block's columns, one row per lane.  (Loops, with the entries in
        // shared memory: unrolled with the entries in registers, the code outgrew
        // the instruction caches.)
        const int below = max(0, (w - k0 - 1) / 32);           // 32-row groups below the first
        if (warp == 0) {
            // the chain: pivot, column, the next column's own update
            const int row = k0 + lane;
            double *x = s.t + k0 * kLdP + min(row, w - 1);     // x[c * kLdP]: this row's entries
            bool dead = false;
            double a = x[0];
#pragma unroll 1
            for (int c = 0; c < nb; ++c) {
                const double d = __shfl_sync(0xffffffffu, a, c);
                double r = rsqrt(d);
                const double s0 = d * r;
                double root = fma(fma(-s0, s0, d), 0.5 * r, s0);
                if (!dead && (unsigned)__double2hiint(d) - 0x00100000u >= 0x7FE00000u) {
                    const double2 o = odd_root(d);
                    root = o.x;
                    r = o.y;
                    if (__double2hiint(root) < 0) {
                        dead = true;
                        if (lane == 0) {
                            s.fail = k0 + c;
                            atomicCAS(info, 0, kglob + k0 + c + 1);
                        }
                    }
                }
                if (!dead) {
                    if (lane > c) a = quot1(a, root, r);
                    else if (lane == c) a = root;
                    if (lane < kPB) s.col[c][lane] = a;
                    if (lane >= c && row < w) x[c * kLdP] = a;
                    if (lane == 0) { s.root[c] = root; s.rinv[c] = r; }
                }
                if (lane == 0) s.dead[c] = dead;
                __syncwarp();
                if (c < nb - 2) named_arrive(9 + (c & 1), 128);
                if (below > 0 && ((c & 1) || c == nb - 1)) named_arrive(1 + c / 2, 32 * (1 + below));
                if (c + 1 < nb) {
                    if (c > 0) named_sync(11 + ((c - 1) & 1), 128);      // column c + 1 has every earlier column's part
                    const double y = x[(c + 1) * kLdP];
                    a = dead ? y : fma(-a, s.col[c][c + 1], y);
                }
            }
        } else if (warp < 4) {
            // its helpers: the later columns of the same rows, a third each
            const int row = k0 + lane;
            double *x = s.t + k0 * kLdP + min(row, w - 1);
#pragma unroll 1
            for (int c = 0; c < nb - 2; ++c) {
                named_sync(9 + (c & 1), 128);
                if (!s.dead[c]) {
                    const double a = x[c * kLdP];
                    for (int q = c + 1 + warp; q < nb; q += 3) {
                        const double v = fma(-a, s.col[c][q], x[q * kLdP]);
                        if (lane >= q && row < w) x[q * kLdP] = v;
                    }
                }
                named_arrive(11 + (c & 1), 128);
            }
        } else if (warp >= 5 && warp < 5 + below) {
            // the rows below, one or two columns behind
            const int row = k0 + 32 * (warp - 4) + lane;
            const bool in = row < w;
            double *x = s.t + k0 * kLdP + (in ? row : w - 1);
#pragma unroll 1
            for (int c = 0; c < nb; ++c) {
                if ((c & 1) == 0) named_sync(1 + c / 2, 32 * (1 + below));      // columns c and c + 1 are ready
                if (s.dead[c]) continue;
                const double a = quot1(x[c * kLdP], s.root[c], s.rinv[c]);
                const double *col = s.col[c];
                if (in) x[c * kLdP] = a;
                for (int q0 = c + 1; q0 < nb; q0 += 4) {
                    double v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (q0 + q < nb) v[q] = fma(-a, col[q0 + q], x[(q0 + q) * kLdP]);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (q0 + q < nb && in) x[(q0 + q) * kLdP] = v[q];
                }
            }
        }
        __syncthreads();
        if (s.fail >= 0) break;
        // ---- the columns right of the block: 16 x 16 tiles on or below the
        // diagonal (two columns per FP64 instruction: tiles of 32 rows would
        // spend a third of them above it), round the warps
        const int c1 = k0 + kPB;
        if (c1 < w) {
            const int g = (w - c1 + 15) / 16;
            const int half = lane >> 4;
            for (int u = warp; u < g * (g + 1) / 2; u += kPotThreads / 32) {
                int ti = 0, tj = u;                                    // tile row, tile column
                while (tj > ti) { ++ti; tj -= ti; }
                const int r = c1 + ti * 16 + (lane & 15), j0 = c1 + tj * 16 + half;
                const int rr = min(r, w - 1);
                double acc[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[q] = s.t[min(j0 + 2 * q, w - 1) * kLdP + rr];
#pragma unroll 4
                for (int c = 0; c < kPB; ++c) {
                    const double *tc = s.t + (k0 + c) * kLdP;
                    const double l = tc[rr];
#pragma unroll
                    for (int q = 0; q < 8; ++q) acc[q] = fma(-l, tc[min(j0 + 2 * q, w - 1)], acc[q]);
                }
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (r < w && j0 + 2 * q <= r) s.t[(j0 + 2 * q) * kLdP + r] = acc[q];
            }
        }
        __syncthreads();
    }
    // Write back the lower triangle (columns past a breakdown keep their
    // partially updated values, as LAPACK leaves them).
    for (int k = warp; k < w; k += kPotThreads / 32)
        for (int r = lane; r < w; r += 32)
            if (r >= k) A[r + (size_t)k * lda] = s.t[k * kLdP + r];
}

// ---------------------------------------------------------------------------
// LU-3, CH-2 and LU-4: lines of X (rows in the right solves, columns in the
// left one) against the step's w x w triangle:
//   for k = 0..w-1:  x_k = x_k / M(k,k) (not LU-4);  x_j -= x_k M(k,j), j > k.
//   kRight  M = U00: M(k, j) = U[k + j ldm]      (a zero pivot divides nothing)
//   kChol   M = L00^T: M(k, j) = L[j + k ldm]
//   kLeft   M = L00^T, unit: the columns of A01
// Bound by the FP64 pipe: an FP64 instruction takes a quarter SM 64 clocks
// whatever its active lanes, so lines are spread over all SMs (the number per
// CTA is lines / SMs) and a line over LPR lanes, each holding every LPR-th
// element in registers: 8 lanes keep four lines per warp and the shuffle of x_k
// short; 16 where an SM has at most 8 lines, so that its four quarters still
// have a warp each.  LU's updates are a separately rounded multiply and
// subtract, and its quotients correctly rounded, in the oracle's order;
// Cholesky's are fused.
// ---------------------------------------------------------------------------
enum { kRight = 0, kChol = 1, kLeft = 2 };
constexpr int kLdM = kMaxV + 1;

// LU-3's quotient in full: a zero pivot divides nothing.
static __device__ __noinline__ double pivot_div(double x, double u) { return u != 0.0 ? __ddiv_rn(x, u) : x; }

// RN(x / u) with r = quot_recip(u).
__device__ __forceinline__ double quot_rn(double x, double u, double r) {
    double q = quot_from(x, u, r);
    if (quot_odd(x, r)) q = pivot_div(x, u);
    return q;
}

template <int LPR, int KIND>
__global__ void __launch_bounds__(512, 1)
k_panel_solve(double *__restrict__ X, int ldx, int lines, int per, int w, const double *__restrict__ M, int ldm,
              const int *skip) {
    if (skip != nullptr && *skip != 0) return;
    constexpr int NI = kMaxV / LPR;                // elements per lane
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *Ms = reinterpret_cast<double *>(smem_raw);      // Ms[k * kLdM + j] = M(k, j)
    double *rs = Ms + kMaxV * kLdM;                         // RN(1 / M(k, k)), 0: divide
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int sub = tid & (LPR - 1);
    const int line = blockIdx.x * per + tid / LPR;
    const bool in = tid / LPR < per && line < lines;
    double x[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int e = LPR * i + sub;
        x[i] = (in && e < w) ? (KIND == kLeft ? X[(size_t)e + (size_t)line * ldx] : X[(size_t)line + (size_t)e * ldx]) : 0.0;
    }
    for (int idx = tid; idx < kMaxV * w; idx += nthr) {
        const int a = idx & (kMaxV - 1), b = idx / kMaxV;   // a runs along the memory of the triangle
        if (KIND == kRight) {
            if (a <= b) Ms[a * kLdM + b] = M[a + (size_t)b * ldm];
        } else {
            if (a < w && a >= b) Ms[b * kLdM + a] = M[a + (size_t)b * ldm];
        }
    }
    __syncthreads();
    if (KIND != kLeft) {
        for (int k = tid; k < w; k += nthr) {
            const double u = Ms[k * kLdM + k];
            rs[k] = KIND == kRight ? quot_recip(u) : (exp_bits(u) - 723u <= 600u ? __drcp_rn(u) : 1.0 / u);
        }
        __syncthreads();
    }
#pragma unroll
    for (int kk = 0; kk < NI; ++kk) {
        if (kk * LPR >= w) break;
        const int kend = min(LPR, w - kk * LPR);
        for (int kl = 0; kl < kend; ++kl) {
            const int k = kk * LPR + kl;
            const double *m = Ms + k * kLdM + sub;
            double xk = __shfl_sync(0xffffffffu, x[kk], kl, LPR);
            if (KIND != kLeft) {
                const double u = Ms[k * kLdM + k];
                xk = KIND == kChol ? quot1(xk, u, rs[k]) : quot_rn(xk, u, rs[k]);
                if (sub == kl) x[kk] = xk;
            }
            if (sub > kl) {
                const double mk = m[kk * LPR];
                x[kk] = KIND == kChol ? fma(-xk, mk, x[kk]) : sub_rn(x[kk], mul_rn(xk, mk));
            }
#pragma unroll
            for (int i = kk + 1; i < NI; ++i) {
                const double mk = m[i * LPR];
                x[i] = KIND == kChol ? fma(-xk, mk, x[i]) : sub_rn(x[i], mul_rn(xk, mk));
            }
        }
    }
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int e = LPR * i + sub;
        if (in && e < w) (KIND == kLeft ? X[(size_t)e + (size_t)line * ldx] : X[(size_t)line + (size_t)e * ldx]) = x[i];
    }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
template <typename K>
static int set_smem(K kernel, size_t bytes) {
    CF_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    return CF_OK;
}

int launch_getf2_nopiv(double *A00, int lda, int w, int kglob, int *info, const double *lu, const int *lu_ok,
                       cudaStream_t st) {
    if (w <= 0) return CF_OK;
    const size_t smem = sizeof(double) * kLdT * kMaxV;
    int rc = set_smem(k_getf2_nopiv, smem);
    if (rc) return rc;
    k_getf2_nopiv<<<lu != nullptr ? 16 : 1, kPanelThreads, smem, st>>>(A00, lda, w, kglob, info, lu, lu_ok);
    CF_LAUNCH_CHECK();
    return CF_OK;
}

int launch_potf2(double *A00, int lda, int w, int kglob, int *info, cudaStream_t st) {
    if (w <= 0) return CF_OK;
    int rc = set_smem(k_potf2, sizeof(PotSmem));
    if (rc) return rc;
    k_potf2<<<1, kPotThreads, sizeof(PotSmem), st>>>(A00, lda, w, kglob, info);
    CF_LAUNCH_CHECK();
    return CF_OK;
}

template <int LPR, int KIND>
static int launch_panel_lpr(double *X, int ldx, int lines, int per, int w, const double *M, int ldm, const int *skip,
                            cudaStream_t st) {
    const size_t smem = sizeof(double) * (kMaxV * kLdM + kMaxV);
    int rc = set_smem(k_panel_solve<LPR, KIND>, smem);
    if (rc) return rc;
    const int threads = (int)align_up((size_t)per * LPR, 32);
    k_panel_solve<LPR, KIND><<<ceil_div(lines, per), threads, smem, st>>>(X, ldx, lines, per, w, M, ldm, skip);
    CF_LAUNCH_CHECK();
    return CF_OK;
}

template <int KIND>
static int launch_panel(double *X, int ldx, int lines, int w, const double *M, int ldm, const int *skip,
                        cudaStream_t st) {
    if (lines <= 0 || w <= 0) return CF_OK;
    const int per = ceil_div(lines, device_sm_count());
    if (per <= 8) return launch_panel_lpr<16, KIND>(X, ldx, lines, per, w, M, ldm, skip, st);
    return launch_panel_lpr<8, KIND>(X, ldx, lines, per < 64 ? per : 64, w, M, ldm, skip, st);
}

int launch_trsm_right_upper(double *X, int ldx, int rows, int w, const double *U, int ldu, bool trans_lower,
                            const int *skip_if_nonzero, cudaStream_t st) {
    return trans_lower ? launch_panel<kChol>(X, ldx, rows, w, U, ldu, skip_if_nonzero, st)
                       : launch_panel<kRight>(X, ldx, rows, w, U, ldu, skip_if_nonzero, st);
}

int launch_trsm_left_lower_unit(double *X, int ldx, int w, int cols, const double *L, int ldl, cudaStream_t st) {
    return launch_panel<kLeft>(X, ldx, cols, w, L, ldl, nullptr, st);
}

}  // namespace cf
