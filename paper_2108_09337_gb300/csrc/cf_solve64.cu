// cf_solve64.cu -- S-1: the FP64 triangular solves of cf_getrs / cf_potrs and
// the row order of a list of interchanges.
//
// A solve with an n x n triangle is a chain of n dependent steps; its bytes
// (4 n^2 per direction) and its 2 lanes of FP64 per clock and SM are far from
// binding for a few right-hand sides.  So the chain is what counts:
//   * the triangle is cut into super-blocks of 2048 rows.  (Up to some 200
//     right-hand sides; more go block by block over all of them.)  One thread-block
//     cluster per right-hand side solves a super-block; its rows beyond take
//     one launch over the whole GPU;
//   * inside the cluster, a solved block is written into every CTA's shared
//     memory (distributed shared memory, an mbarrier per block); no inverse is
//     formed, the operations are substitution's own.
// LU's factors (k_lu_solve64): blocks of 128 rows, a row per thread, and the
// operations on a row in one fixed order: per solved block an FMA chain over
// its 128 columns, subtracted as one value; in its own block a separately
// rounded multiply and subtract per column, a correctly rounded division.  The
// solution of an ill-conditioned system moves with any other order by as much
// as its error (1e-11 at n = 2048, 3e-9 at n = 8192 on uniform matrices), so
// every form of the solve keeps this one.
// Cholesky's (k_tri_solve64): blocks of 64 rows go round the eight CTAs, the
// products by all 256 threads, a block in one warp (two rows per lane, the
// pivot's value by shuffle), the quotients from reciprocals.
// The waits are inside a cluster, whose CTAs run at the same time by
// definition, and bounded.  No workspace: cf_potrs has none.
#include <cooperative_groups.h>

#include "cf_common.cuh"
#include "cf_kernels.cuh"
#include "cf_solve64.cuh"

namespace cg = cooperative_groups;

namespace cf {

__device__ int g_solve64_status = 0;       // 0 or CF_ERR_TIMEOUT

namespace sv {

constexpr int NB = 64;                 // rows of a block
constexpr int CL = 8;                  // CTAs of a cluster
constexpr int kSuper = 2048;           // rows of a super-block
constexpr int MAXB = kSuper / NB;      // blocks
constexpr int OWN = MAXB / CL;         // blocks of a CTA
constexpr int LDD = NB + 1;
constexpr int kThreads = 256;

struct Smem {
    double D[OWN][NB * LDD];           // diagonal blocks: D[k * LDD + r] = M(r, k)
    double rinv[OWN][NB];              // 1 / M(k, k)
    double xs[MAXB][NB];               // solved blocks, in solving order
    double x0[OWN][NB];                // right-hand side of the CTA's blocks
    double part[4 * NB];
    double pub[NB];
    uint64_t bar[MAXB];
    int dead;                          // a wait ran out
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

constexpr long long kSpin = 1ll << 17;      // polls: half a second (a poll that finds nothing takes 3.9 us)

// Waits (bounded) for a solved block; where one wait ran out (*dead) the CTA's
// others give up too, and the solve ends with X wrong and the status set.
__device__ __forceinline__ void wait_block(uint64_t *bar, volatile int *dead, long long limit) {
    for (long long i = 0; i < limit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(smem_u32(bar))
            : "memory");
        if (ok) return;
        if (i > 64) {
            if (*dead) return;
            __nanosleep(20);
        }
    }
    *dead = 1;
    atomicExch(&g_solve64_status, CF_ERR_TIMEOUT);
}

constexpr int LB = 128;                // rows of a block of k_lu_solve64
constexpr int LBLK = kSuper / LB;      // blocks: two per CTA
static_assert(LBLK == 2 * CL, "a half CTA owns one block");

struct LuSmem {
    double xs[LBLK][LB];               // solved blocks, in solving order
    uint64_t bar[LBLK][LB / 32];       // their 32-row parts
    int dead;                          // a wait ran out
};

// L y = b (FWD, unit lower) or U x = y with a super-block of the LU factors.
// Half a CTA (four warps, one per quarter of the SM) owns the t-th block solved.
// Bound by the chain: per block four 32-row parts one after the other, each 32
// steps of shuffle, multiply and subtract (U: and a quotient, five FP64
// operations), then the next part's 32 columns; the FMA chains of blocks solved
// earlier run beside it.  Both directions, 1 to 8 right-hand sides: n = 300 0.28
// ms, 2048 1.37 ms, 8192 6.4 ms (blocks of 64 rows in one warp with the sums in
// another order: 0.18, 0.80, 3.5; a launch per 128 rows and product: 1.52, 11.6,
// 48.5).
template <bool FWD>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kThreads)
k_lu_solve64(int n, const double *__restrict__ T, int ldt, double *__restrict__ X, int ldx, long long spin, int withhold) {
    __shared__ LuSmem s;
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, q = (tid & (LB - 1)) >> 5;      // q: part of the block
    const int nb = (n + LB - 1) / LB;
    const int t = (int)cl.block_rank() + CL * (tid / LB);                        // solving order
    const size_t ld = (size_t)ldt;
    double *xg = X + (size_t)blockIdx.y * ldx;
    auto row0 = [&](int b) { return (FWD ? b : nb - 1 - b) * LB; };
    if (tid < LBLK * (LB / 32))
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s.bar[0][0] + tid)) : "memory");
    if (tid == 0) {
        s.dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cl.sync();
    if (t < nb) {
        const int r0 = row0(t), row = r0 + 32 * q + lane;
        const bool live = row < n;
        const double *Tr = T + (live ? row : 0);
        // Chunks of 16 columns: 8 per solved block, then the block's own up to the
        // warp's part, in solving order; the next chunk is loaded ahead.
        const int own0 = 8 * t, last = own0 + 2 * (FWD ? q + 1 : LB / 32 - q);
        auto first_col = [&](int c) {
            if (c < own0) return row0(c >> 3) + 16 * (c & 7);
            return r0 + 16 * (FWD ? c - own0 : LB / 16 - 1 - (c - own0));
        };
        auto load = [&](int c, double (&v)[16]) {
            const int k0 = first_col(c);
#pragma unroll
            for (int a = 0; a < 16; ++a) v[a] = (live && k0 + a < n) ? Tr[(size_t)(k0 + a) * ld] : 0.0;
        };
        double x = live ? xg[row] : 0.0;
        const double u = (!FWD && live) ? Tr[(size_t)row * ld] : 1.0;
        const double r = FWD ? 0.0 : quot_recip(u);
        double cur[16], nxt[16];
        load(0, cur);
        double acc = 0.0;
        for (int c = 0; c < last; ++c) {
            if (c + 1 < last) load(c + 1, nxt);
            if (c < own0) {                                   // a block solved before: one FMA chain
                const int b = c >> 3, kk = c & 7;
                if ((kk & 1) == 0) wait_block(&s.bar[b][kk >> 1], &s.dead, spin);
#pragma unroll
                for (int a = 0; a < 16; ++a) acc = fma(cur[a], s.xs[b][16 * kk + a], acc);
                if (kk == 7) {
                    x -= acc;
                    acc = 0.0;
                }
            } else if (c < last - 2) {                        // a part of this block solved before
                const int k0 = first_col(c) - r0;
                if (((c - own0) & 1) == 0) wait_block(&s.bar[t][k0 >> 5], &s.dead, spin);
#pragma unroll
                for (int a = 0; a < 16; ++a) {
                    const int e = FWD ? a : 15 - a;
                    x = sub_rn(x, mul_rn(cur[e], s.xs[t][k0 + e]));
                }
            } else {                                          // its own part
#pragma unroll
                for (int a = 0; a < 16; ++a) {
                    const int e = FWD ? a : 15 - a;
                    const int kl = (first_col(c) - r0 + e) & 31;      // the lane whose row is the pivot
                    if (!FWD) {
                        double y = quot_from(x, u, r);
                        if (lane == kl) {
                            if (quot_odd(x, r)) y = div_call(x, u);
                            x = y;
                        }
                    }
                    const double xk = __shfl_sync(0xffffffffu, x, kl);
                    const double z = sub_rn(x, mul_rn(cur[e], xk));
                    if (FWD ? lane > kl : lane < kl) x = z;
                }
            }
#pragma unroll
            for (int a = 0; a < 16; ++a) cur[a] = nxt[a];
        }
        for (int p = 0; p < CL; ++p) cl.map_shared_rank(&s, p)->xs[t][32 * q + lane] = x;
        __syncwarp();
        if (lane < CL && !(withhold && t == 0)) {
            uint32_t remote;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(&s.bar[t][q])), "r"(lane));
            asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
        }
        if (live) xg[row] = x;
    }
    cl.sync();                          // no CTA leaves while others may still write into it
}

// X[r] -= T(r, block) Y(block) for the super-block's blocks of 128 columns in
// solving order (desc: the last one first), each as one FMA chain: a row per
// thread, one warp per CTA, so that a few thousand rows reach every SM.
__global__ void __launch_bounds__(32)
k_lu_rows_sub(int m, int len, const double *__restrict__ T, int ldt, const double *__restrict__ Y, double *__restrict__ X,
              int ldx, int desc) {
    __shared__ double ys[kSuper];
    const int row = blockIdx.x * 32 + threadIdx.x;
    const double *y = Y + (size_t)blockIdx.y * ldx;
    for (int k = threadIdx.x; k < kSuper; k += 32) ys[k] = k < len ? y[k] : 0.0;
    __syncwarp();
    const bool live = row < m;
    const double *t = T + (live ? row : 0);
    double *xp = X + (size_t)blockIdx.y * ldx + (live ? row : 0);
    const int nb = (len + LB - 1) / LB;
    auto first_col = [&](int c) { return (desc ? nb - 1 - (c >> 3) : c >> 3) * LB + 16 * (c & 7); };
    auto load = [&](int c, double (&v)[16]) {
        const int k0 = first_col(c);
#pragma unroll
        for (int a = 0; a < 16; ++a) v[a] = (live && k0 + a < len) ? t[(size_t)(k0 + a) * ldt] : 0.0;
    };
    double x = *xp, acc = 0.0, cur[16], nxt[16];
    load(0, cur);
    for (int c = 0; c < 8 * nb; ++c) {
        if (c + 1 < 8 * nb) load(c + 1, nxt);
        const double *yc = ys + first_col(c);
#pragma unroll
        for (int a = 0; a < 16; ++a) acc = fma(cur[a], yc[a], acc);
        if ((c & 7) == 7) {
            x -= acc;
            acc = 0.0;
        }
#pragma unroll
        for (int a = 0; a < 16; ++a) cur[a] = nxt[a];
    }
    if (live) *xp = x;
}

// MODE 2: lower, 3: transposed lower (M = T^T)
template <int MODE>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(kThreads, 1)
k_tri_solve64(int n, const double *__restrict__ T, int ldt, double *__restrict__ X, int ldx, long long spin, int withhold) {
    constexpr bool FWD = MODE == 2, TRANS = MODE == 3;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem &s = *reinterpret_cast<Smem *>(smem_raw);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = (n + NB - 1) / NB;
    const size_t ld = (size_t)ldt;
    double *x = X + (size_t)blockIdx.y * ldx;
    auto row0 = [&](int t) { return (FWD ? t : nb - 1 - t) * NB; };   // first row of the t-th block solved

    if (tid < MAXB) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s.bar[tid])) : "memory");
    if (tid == 0) {
        s.dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int t = rank, o = 0; t < nb; t += CL, ++o) {
        const int r0 = row0(t), nr = min(NB, n - r0);
        for (int e = tid; e < NB * NB; e += kThreads) {
            const int a = e & (NB - 1), b = e >> 6;                   // a runs along the memory
            const int r = TRANS ? b : a, k = TRANS ? a : b;
            const bool need = (FWD ? k <= r : k >= r) && r < nr && k < nr;
            double v = (r == k) ? 1.0 : 0.0;                          // rows past the end: identity
            if (need) v = TRANS ? T[(size_t)(r0 + k) + (size_t)(r0 + r) * ld] : T[(size_t)(r0 + r) + (size_t)(r0 + k) * ld];
            s.D[o][k * LDD + r] = v;
        }
        if (tid < NB) s.x0[o][tid] = tid < nr ? x[r0 + tid] : 0.0;
    }
    __syncthreads();
    for (int t = rank, o = 0; t < nb; t += CL, ++o)
        if (tid < NB) s.rinv[o][tid] = 1.0 / s.D[o][tid * LDD + tid];
    cl.sync();

    // Partial sums of the CTA's blocks.  Row r, k quarter q (TRANS: eight rows
    // of a warp, the lane's two k): every load of a tile is coalesced.
    constexpr int AR = TRANS ? 8 : 1;
    double acc[OWN][AR];
#pragma unroll
    for (int o = 0; o < OWN; ++o)
#pragma unroll
        for (int a = 0; a < AR; ++a) acc[o][a] = 0.0;

    auto load_tile = [&](int t, int j, double (&v)[16]) {             // block row t, block column j
        const int r0 = row0(t), c0 = row0(j);
        if (TRANS) {
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = r0 + warp * 8 + a, k = c0 + lane + 32 * h;
                    v[2 * a + h] = (r < n && k < n) ? T[(size_t)k + (size_t)r * ld] : 0.0;
                }
        } else {
            const int r = r0 + (tid & (NB - 1)), k0 = c0 + (tid >> 6) * 16;
#pragma unroll
            for (int a = 0; a < 16; ++a) v[a] = (r < n && k0 + a < n) ? T[(size_t)r + (size_t)(k0 + a) * ld] : 0.0;
        }
    };
    auto mac = [&](int t, int j, const double (&v)[16]) {
        const double *xj = s.xs[j];
        double sum[AR];
        if (TRANS) {
            const double x0 = xj[lane], x1 = xj[lane + 32];
#pragma unroll
            for (int a = 0; a < AR; ++a) sum[a] = fma(v[2 * a + 1], x1, v[2 * a] * x0);
        } else {
            const double *xq = xj + (tid >> 6) * 16;
            double s0 = 0.0, s1 = 0.0;                                // two chains
#pragma unroll
            for (int a = 0; a < 16; a += 2) {
                s0 = fma(v[a], xq[a], s0);
                s1 = fma(v[a + 1], xq[a + 1], s1);
            }
            sum[0] = s0 + s1;
        }
        const int o = t / CL;
#pragma unroll
        for (int q = 0; q < OWN; ++q)
            if (q == o) {
#pragma unroll
                for (int a = 0; a < AR; ++a) acc[q][a] += sum[a];
            }
    };
    // Block t: sum of the parts, substitution, result to every CTA.
    auto solve_block = [&](int t) {
        const int o = t / CL, r0 = row0(t);
        double v[AR];
#pragma unroll
        for (int q = 0; q < OWN; ++q)
            if (q == o) {
#pragma unroll
                for (int a = 0; a < AR; ++a) v[a] = acc[q][a];
            }
        if (TRANS) {
            // eight sums over the warp's lanes: halve the values with each exchange
            double w4[4], w2[2], w1;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const bool up = lane & 16;
                const double send = up ? v[a % AR] : v[(a + 4) % AR], keep = up ? v[(a + 4) % AR] : v[a % AR];
                w4[a] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
            }
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const bool up = lane & 8;
                const double send = up ? w4[a] : w4[a + 2], keep = up ? w4[a + 2] : w4[a];
                w2[a] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
            }
            {
                const bool up = lane & 4;
                const double send = up ? w2[0] : w2[1], keep = up ? w2[1] : w2[0];
                w1 = keep + __shfl_xor_sync(0xffffffffu, send, 4);
            }
            w1 += __shfl_xor_sync(0xffffffffu, w1, 2);
            w1 += __shfl_xor_sync(0xffffffffu, w1, 1);
            if ((lane & 3) == 0) s.part[warp * 8 + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = w1;
        } else {
            s.part[tid] = v[0];
        }
        __syncthreads();
        if (warp == 0) {
            double a, b;                                              // rows lane and lane + 32
            if (TRANS) {
                a = s.x0[o][lane] - s.part[lane];
                b = s.x0[o][lane + 32] - s.part[lane + 32];
            } else {
                a = s.x0[o][lane] - ((s.part[lane] + s.part[NB + lane]) + (s.part[2 * NB + lane] + s.part[3 * NB + lane]));
                b = s.x0[o][lane + 32] - ((s.part[lane + 32] + s.part[NB + lane + 32]) +
                                          (s.part[2 * NB + lane + 32] + s.part[3 * NB + lane + 32]));
            }
            const double *D = s.D[o];
#pragma unroll 8
            for (int q = 0; q < NB; ++q) {
                const int k = FWD ? q : NB - 1 - q;
                const bool low = FWD ? q < 32 : q >= 32;              // the pivot is in the lanes' first row
                double xk = __shfl_sync(0xffffffffu, low ? a : b, k & 31);
                {
                    // the quotient from the reciprocal, corrected by its exact remainder; a zero, and
                    // whatever leaves the normal numbers, by the division itself
                    const double d = D[k * LDD + k], r = s.rinv[o][k];
                    const double q0 = xk * r;
                    double q1 = fma(fma(-q0, d, xk), r, q0);
                    if (exp_bits(q0) - 100u >= 1900u || exp_bits(r) - 100u >= 1900u) q1 = div_call(xk, d);
                    xk = q1;
                }
                const double da = D[k * LDD + lane], db = D[k * LDD + lane + 32];
                if (FWD) {
                    if (low) a = lane == (k & 31) ? xk : (lane > k ? fma(-da, xk, a) : a);
                    b = (!low && lane == (k & 31)) ? xk : (lane + 32 > k ? fma(-db, xk, b) : b);
                } else {
                    if (!low) b = lane == (k & 31) ? xk : (lane + 32 < k ? fma(-db, xk, b) : b);
                    a = (low && lane == (k & 31)) ? xk : (lane < k ? fma(-da, xk, a) : a);
                }
            }
            s.pub[lane] = a;
            s.pub[lane + 32] = b;
            if (r0 + lane < n) x[r0 + lane] = a;
            if (r0 + lane + 32 < n) x[r0 + lane + 32] = b;
        }
        __syncthreads();
        {
            Smem *rs = cl.map_shared_rank(&s, warp);                  // warp q serves CTA q
            rs->xs[t][lane] = s.pub[lane];
            rs->xs[t][lane + 32] = s.pub[lane + 32];
            __syncwarp();
            if (lane == 0 && !(withhold && t == 0)) {
                uint32_t remote;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(&s.bar[t])), "r"(warp));
                asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
            }
        }
    };

    if (rank == 0) solve_block(0);
    // The CTA's tiles: for every solved block j, its own blocks t > j, nearest
    // first; the next tile's loads are in flight while the current one waits.
    auto first_own = [&](int j) { return j + 1 + ((rank - (j + 1)) % CL + CL) % CL; };
    int j = 0, t = first_own(0);
    while (j < nb - 1 && t >= nb) { ++j; t = first_own(j); }
    double cur[16], nxt[16];
    if (j < nb - 1) load_tile(t, j, cur);
    while (j < nb - 1) {
        int j2 = j, t2 = t + CL;
        while (j2 < nb - 1 && t2 >= nb) { ++j2; t2 = first_own(j2); }
        if (j2 < nb - 1) load_tile(t2, j2, nxt);
        wait_block(&s.bar[j], &s.dead, spin);
        mac(t, j, cur);
        if (t == j + 1) solve_block(t);
#pragma unroll
        for (int a = 0; a < 16; ++a) cur[a] = nxt[a];
        j = j2;
        t = t2;
    }
    cl.sync();                          // no CTA leaves while others may still write into it
}

// X[c] -= sum_k L[k + c ldl] Y[k], c < m, k < len, for nrhs columns: a warp per
// column of L, four right-hand sides at a time.
__global__ void __launch_bounds__(256)
k_gemv_t_sub(int m, int len, int nrhs, const double *__restrict__ L, int ldl, const double *__restrict__ Y, int ldy,
             double *__restrict__ X, int ldx) {
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (c >= m) return;
    const double *l = L + (size_t)c * ldl;
    for (int q0 = 0; q0 < nrhs; q0 += 4) {
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        const int nq = min(4, nrhs - q0);
#pragma unroll 4
        for (int k = lane; k < len; k += 32) {
            const double a = l[k];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (q < nq) acc[q] = fma(a, Y[(size_t)k + (size_t)(q0 + q) * ldy], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
            if (lane == 0 && q < nq) X[(size_t)c + (size_t)(q0 + q) * ldx] -= acc[q];
        }
    }
}

// ---------------------------------------------------------------------------
// ipiv (1-based interchanges) -> row order: perm[i] = original row now at i.
// The interchanges are a chain, but a chunk of 128 of them only permutes its own
// 128 positions and the at most 128 others it names: one warp per chunk plays it
// on labels (all chunks at once), then the chunks' permutations are applied in
// order.  Scratch: 6 bytes per row, the chunk's other positions (int) and the
// labels of its own and of the other positions (one byte each).
// ---------------------------------------------------------------------------
constexpr int CH = 128;
constexpr size_t kChunkBytes = 6 * CH;

__global__ void __launch_bounds__(32) k_ipiv_chunks(int n, const int *__restrict__ ipiv, unsigned char *scratch) {
    __shared__ int far_[CH];
    __shared__ unsigned char lab[2 * CH];
    const int lane = threadIdx.x, k0 = blockIdx.x * CH, cnt = min(CH, n - k0);
    for (int q = lane; q < 2 * CH; q += 32) lab[q] = (unsigned char)q;
    for (int q = lane; q < CH; q += 32) far_[q] = -1;
    int piv[CH / 32];
#pragma unroll
    for (int q = 0; q < CH / 32; ++q) piv[q] = lane + 32 * q < cnt ? ipiv[k0 + lane + 32 * q] - 1 : 0;
    __syncwarp();
    int nfar = 0;
#pragma unroll
    for (int q = 0; q < CH / 32; ++q)
        for (int e = 0; e < 32; ++e) {
            const int i = 32 * q + e;
            if (i >= cnt) break;
            const int p = __shfl_sync(0xffffffffu, piv[q], e);
            int slot = p - k0;
            if (slot < 0 || slot >= CH) {
                slot = -1;
#pragma unroll
                for (int h = 0; h < CH / 32; ++h) {
                    const unsigned hit = __ballot_sync(0xffffffffu, lane + 32 * h < nfar && far_[lane + 32 * h] == p);
                    if (hit && slot < 0) slot = CH + 32 * h + __ffs(hit) - 1;
                }
                if (slot < 0) {
                    if (lane == 0) far_[nfar] = p;
                    slot = CH + nfar++;
                    __syncwarp();
                }
            }
            if (lane == 0 && slot != i) {
                const unsigned char a = lab[i];
                lab[i] = lab[slot];
                lab[slot] = a;
            }
            __syncwarp();
        }
    unsigned char *out = scratch + (size_t)blockIdx.x * kChunkBytes;
    for (int q = lane; q < cnt; q += 32) {
        reinterpret_cast<int *>(out)[q] = far_[q];
        out[4 * cnt + q] = lab[q];
        out[5 * cnt + q] = lab[CH + q];
    }
}

__global__ void __launch_bounds__(1024) k_compose_perm(int n, const unsigned char *__restrict__ scratch, int *perm,
                                                       int use_smem) {
    extern __shared__ int sp[];
    int *p = use_smem ? sp : perm;
    for (int i = threadIdx.x; i < n; i += 1024) p[i] = i;
    const int nchunks = (n + CH - 1) / CH;
    const int q = threadIdx.x;
    __syncthreads();
    int pos = -1, src = -1;
    auto fetch = [&](int c) {           // this thread's place in chunk c and where its new content is
        const unsigned char *ch = scratch + (size_t)c * kChunkBytes;
        const int *far_ = reinterpret_cast<const int *>(ch);
        const int cnt = min(CH, n - c * CH);
        pos = src = -1;
        if (q < 2 * CH && (q & (CH - 1)) < cnt) {
            const int l = ch[(q < CH ? 4 : 5) * cnt + (q & (CH - 1))];
            if (l != q) {
                pos = q < CH ? c * CH + q : far_[q - CH];
                src = l < CH ? c * CH + l : far_[l - CH];
            }
        }
    };
    fetch(0);
    for (int c = 0; c < nchunks; ++c) {
        const int at = pos, v = src >= 0 ? p[src] : 0;
        __syncthreads();
        if (at >= 0) p[at] = v;
        if (c + 1 < nchunks) fetch(c + 1);
        __syncthreads();
    }
    if (use_smem)
        for (int i = threadIdx.x; i < n; i += 1024) perm[i] = p[i];
}

// Out[i, c] = In[perm[i], c]
__global__ void k_gather_rows(int n, int nrhs, const int *perm, const double *In, int ldi, double *Out, int ldo) {
    const size_t tot = (size_t)n * nrhs;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e % n), c = (int)(e / n);
        Out[(size_t)i + (size_t)c * ldo] = In[(size_t)perm[i] + (size_t)c * ldi];
    }
}

template <int MODE>
static int chol_mode(int n, int nrhs, const double *T, int ldt, double *X, int ldx, long long spin, int withhold,
                     cudaStream_t st) {
    constexpr bool FWD = MODE == 2;
    const size_t ld = (size_t)ldt;
    CF_CUDA_TRY(cudaFuncSetAttribute(k_tri_solve64<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)));
    const int ns = ceil_div(n, kSuper);
    for (int q = 0; q < ns; ++q) {
        const int k0 = (FWD ? q : ns - 1 - q) * kSuper;
        const int w = kSuper < n - k0 ? kSuper : n - k0;
        k_tri_solve64<MODE><<<dim3(CL, nrhs), kThreads, sizeof(Smem), st>>>(w, T + k0 + k0 * ld, ldt, X + k0, ldx, spin, withhold);
        CF_LAUNCH_CHECK();
        if (FWD) {
            const int r0 = k0 + w;
            const int rc = launch_residual_f64(n - r0, w, nrhs, T + r0 + k0 * ld, ldt, X + k0, ldx, X + r0, ldx, X + r0,
                                               ldx, st);
            if (rc) return rc;
        } else if (k0 > 0) {
            k_gemv_t_sub<<<ceil_div(k0, 8), 256, 0, st>>>(k0, w, nrhs, T + k0, ldt, X + k0, ldx, X, ldx);
            CF_LAUNCH_CHECK();
        }
    }
    return CF_OK;
}

template <bool FWD>
static int lu_mode(int n, int nrhs, const double *T, int ldt, double *X, int ldx, long long spin, int withhold,
                   cudaStream_t st) {
    const size_t ld = (size_t)ldt;
    const int ns = ceil_div(n, kSuper);
    for (int q = 0; q < ns; ++q) {
        const int k0 = (FWD ? q : ns - 1 - q) * kSuper;
        const int w = kSuper < n - k0 ? kSuper : n - k0;
        const int r0 = FWD ? k0 + w : 0, m = FWD ? n - r0 : k0;      // the rows beyond
        k_lu_solve64<FWD><<<dim3(CL, nrhs), kThreads, 0, st>>>(w, T + k0 + k0 * ld, ldt, X + k0, ldx, spin, withhold);
        CF_LAUNCH_CHECK();
        if (m <= 0) continue;
        k_lu_rows_sub<<<dim3(ceil_div(m, 32), nrhs), 32, 0, st>>>(m, w, T + r0 + k0 * ld, ldt, X + k0, X + r0, ldx,
                                                                 FWD ? 0 : 1);
        CF_LAUNCH_CHECK();
    }
    return CF_OK;
}

// ---------------------------------------------------------------------------
// Many right-hand sides: per block of 128 rows one left solve over all columns
// and one product over the whole GPU, with k_lu_solve64's order of operations.
// Its time hardly grows with their number, the clusters' does (every one reads
// the triangle and takes 8 CTAs).  Both directions, blocked / clusters, ms:
//   LU        n = 130: 128 rhs 0.72 / 0.66, 160 0.72 / 0.81; n = 300: 192 1.64 /
//             1.44, 256 1.64 / 1.91; n = 2048: 256 12.3 / 10.9, 320 12.0 / 12.7;
//             n = 8192: 256 71.6 / 66.7, 320 76.6 / 79.3, 512 96.5 / 127.9
//   Cholesky  n = 130: 64 0.99 / 0.94, 96 0.99 / 1.30; n = 300: 160 2.24 / 2.05,
//             192 2.25 / 2.43; n = 2048: 192 17.2 / 13.0, 256 17.2 / 18.0;
//             n = 8192: 192 83.3 / 75.5, 256 89.4 / 103.1
//
// X <- M^{-1} X with M = T (TRANS: T^T) of size w x w, lower (forward) or upper
// (backward), non-unit.  CTA: 64 columns, four lanes of one warp each.
// ---------------------------------------------------------------------------
constexpr int kCB = 64;
constexpr size_t kBlockSmem = sizeof(double) * ((size_t)kMaxV * kMaxV + (size_t)kCB * (kMaxV + 1));

template <bool LOWER, bool TRANS>
__global__ void __launch_bounds__(kThreads, 1)
k_block_solve(double *X, int ldx, int w, int cols, const double *__restrict__ T, int ldt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *Ms = reinterpret_cast<double *>(smem_raw);        // Ms[k * kMaxV + i] = M(i, k)
    double *Xs = Ms + kMaxV * kMaxV;                          // Xs[c * XLD + i]
    constexpr int XLD = kMaxV + 1;
    const int tid = threadIdx.x;
    const int c0 = blockIdx.x * kCB, nc = min(kCB, cols - c0);
    for (int e = tid; e < w * w; e += kThreads) {
        const int a = e % w, b = e / w;                       // a runs along the memory
        const int i = TRANS ? b : a, k = TRANS ? a : b;
        if (LOWER ? i >= k : i <= k) Ms[k * kMaxV + i] = T[(size_t)a + (size_t)b * ldt];
    }
    for (int e = tid; e < nc * w; e += kThreads) Xs[e / w * XLD + e % w] = X[(size_t)(e % w) + (size_t)(c0 + e / w) * ldx];
    __syncthreads();
    const int c = tid >> 2, q = tid & 3;
    if (c < nc) {
        double *x = Xs + c * XLD;
        const unsigned mask = 0xfu << (tid & 28);
        for (int s = 0; s < w; ++s) {
            const int k = LOWER ? s : w - 1 - s;
            if (q == 0) x[k] = div_rn(x[k], Ms[k * kMaxV + k]);
            __syncwarp(mask);
            const double xk = x[k];
            for (int i = LOWER ? k + 1 + q : q; i < (LOWER ? w : k); i += 4) x[i] = sub_rn(x[i], mul_rn(Ms[k * kMaxV + i], xk));
            __syncwarp(mask);
        }
    }
    __syncthreads();
    for (int e = tid; e < nc * w; e += kThreads) X[(size_t)(e % w) + (size_t)(c0 + e / w) * ldx] = Xs[e / w * XLD + e % w];
}

template <bool LOWER, bool TRANS>
static int block_solve(double *X, int ldx, int w, int cols, const double *T, int ldt, cudaStream_t st) {
    CF_CUDA_TRY(cudaFuncSetAttribute(k_block_solve<LOWER, TRANS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kBlockSmem));
    k_block_solve<LOWER, TRANS><<<ceil_div(cols, kCB), kThreads, kBlockSmem, st>>>(X, ldx, w, cols, T, ldt);
    CF_LAUNCH_CHECK();
    return CF_OK;
}

static int blocked_solve(int mode, int n, int nrhs, const double *T, int ldt, double *X, int ldx, cudaStream_t st) {
    const bool fwd = mode == 0 || mode == 2;
    const size_t ld = (size_t)ldt;
    const int nb = ceil_div(n, LB);
    for (int b = 0; b < nb; ++b) {
        const int k0 = (fwd ? b : nb - 1 - b) * LB, w = LB < n - k0 ? LB : n - k0;
        const double *D = T + k0 + k0 * ld;
        double *Y = X + k0;
        int rc = mode == 0   ? launch_trsm_left_lower_unit(Y, ldx, w, nrhs, D, ldt, st)
                 : mode == 1 ? block_solve<false, false>(Y, ldx, w, nrhs, D, ldt, st)
                 : mode == 2 ? block_solve<true, false>(Y, ldx, w, nrhs, D, ldt, st)
                             : block_solve<false, true>(Y, ldx, w, nrhs, D, ldt, st);
        if (rc) return rc;
        if (fwd)
            rc = launch_gemm_f64_sub(n - k0 - w, nrhs, w, D + w, ldt, Y, ldx, false, Y + w, ldx, false, nullptr, st);
        else if (mode == 1)
            rc = launch_gemm_f64_sub(k0, nrhs, w, T + k0 * ld, ldt, Y, ldx, false, X, ldx, false, nullptr, st);
        else
            rc = launch_gemm_f64_sub_at(k0, nrhs, w, T + k0, ldt, Y, ldx, X, ldx, st);
        if (rc) return rc;
    }
    return CF_OK;
}

}  // namespace sv

// Right-hand sides up to which a cluster takes each (measured above).
static int most_clusters(int mode, int n) { return mode < 2 ? (n > 256 ? 256 : 128) : (n > 256 ? 160 : 64); }

static int cluster_solve(int mode, int n, int nrhs, const double *T, int ldt, double *X, int ldx, long long spin,
                         int withhold, cudaStream_t st) {
    switch (mode) {
        case 0: return sv::lu_mode<true>(n, nrhs, T, ldt, X, ldx, spin, withhold, st);
        case 1: return sv::lu_mode<false>(n, nrhs, T, ldt, X, ldx, spin, withhold, st);
        case 2: return sv::chol_mode<2>(n, nrhs, T, ldt, X, ldx, spin, withhold, st);
        default: return sv::chol_mode<3>(n, nrhs, T, ldt, X, ldx, spin, withhold, st);
    }
}

int launch_tri_solve64(int mode, int n, int nrhs, const double *T, int ldt, double *X, int ldx, cudaStream_t st) {
    if (n <= 0 || nrhs <= 0) return CF_OK;
    if (mode < 0 || mode > 3) return CF_ERR_UNSUPPORTED;
    if (nrhs > most_clusters(mode, n)) return sv::blocked_solve(mode, n, nrhs, T, ldt, X, ldx, st);
    return cluster_solve(mode, n, nrhs, T, ldt, X, ldx, sv::kSpin, 0, st);
}

int launch_permute_rhs(int n, int nrhs, const int *ipiv, int *perm, const double *B, int ldb, double *T, cudaStream_t st) {
    // the chunks' lists lie in T until the rows are gathered into it
    const int nchunks = ceil_div(n, sv::CH);
    unsigned char *scratch = reinterpret_cast<unsigned char *>(T);
    sv::k_ipiv_chunks<<<nchunks, 32, 0, st>>>(n, ipiv, scratch);
    CF_LAUNCH_CHECK();
    const size_t smem = (size_t)n * sizeof(int) <= 200 * 1024 ? (size_t)n * sizeof(int) : 0;
    if (smem > 48 * 1024)
        CF_CUDA_TRY(cudaFuncSetAttribute(sv::k_compose_perm, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    sv::k_compose_perm<<<1, 1024, smem, st>>>(n, scratch, perm, smem != 0);
    CF_LAUNCH_CHECK();
    const size_t tot = (size_t)n * nrhs;
    const int blocks = tot < 1024 * 256 ? ceil_div((long long)tot, 256) : 1024;
    sv::k_gather_rows<<<blocks, 256, 0, st>>>(n, nrhs, perm, B, ldb, T, n);
    CF_LAUNCH_CHECK();
    return CF_OK;
}

int solve64_take_status(cudaStream_t st, int *status) {
    int h = 0;
    CF_CUDA_TRY(cudaMemcpyFromSymbolAsync(&h, g_solve64_status, sizeof(int), 0, cudaMemcpyDeviceToHost, st));
    CF_CUDA_TRY(cudaStreamSynchronize(st));
    if (h != 0) {
        const int zero = 0;
        CF_CUDA_TRY(cudaMemcpyToSymbolAsync(g_solve64_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st));
        CF_CUDA_TRY(cudaStreamSynchronize(st));
    }
    *status = h;
    return CF_OK;
}

}  // namespace cf

// Failure-detection test of the bounded waits, not part of the API: one direction
// of the cluster solves whose first block of every super-block is withheld from
// the others, so that each wait for it gives up after spin_limit polls (0: the
// usual number).
extern "C" int cf_tri_solve64_withheld(int mode, int n, int nrhs, const double *T, int ldt, double *X, int ldx,
                                       long long spin_limit, cudaStream_t stream) {
    if (mode < 0 || mode > 3) return -1;
    if (n < 1) return -2;
    if (nrhs < 1 || nrhs > 64) return -3;
    if (T == nullptr) return -4;
    if (ldt < n) return -5;
    if (X == nullptr) return -6;
    if (ldx < n) return -7;
    if (spin_limit < 0) return -8;
    return cf::cluster_solve(mode, n, nrhs, T, ldt, X, ldx, spin_limit > 0 ? spin_limit : cf::sv::kSpin, 1, stream);
}
