// cf_tourn.cu -- LU-1: TournPivot (Alg. 1; Sec. 7.3 "Tournament
// Pivoting" and "Pivoting in COnfLUX"; the pivot selection in the I/O-cost proof) and
// LU-2: the row interchanges that bring the winners to the top.
//
// GPU design.  One launch per level of the tree: a node (a leaf's rows, or the
// stacked winners of `arity` children, with their original panel values) is a
// thread-block cluster of 1 to 16 CTAs that hold its rows in shared memory in
// equal shares.  The elimination is bound by the FP64 pipe (an element's
// multiply and subtract take 128 clocks of a quarter SM per 32 lanes), so the
// cluster size is chosen to put a level on as many SMs as it has: 16 leaves of
// a 2048-row panel run on 128 SMs, 16 rows each.
//
// The elimination goes by blocks of 4 columns.  Inside a block only the rows'
// four entries move, in registers, one row per thread, and nothing but the
// candidates crosses warps and CTAs: per column each warp sends its best row's
// four entries (multipliers so far, then the values) and its position into
// every CTA's slots through distributed shared memory, counted by an mbarrier
// there; whoever has all slots picks the winner, divides, updates and sends the
// next.  No barrier over the CTA or the cluster is on this chain, and the warps
// without rows apply the block before to the other columns beside it.  At the
// block's end the CTA pulls the four pivot rows' other columns from their
// owners, brings them up to date among themselves and applies them to the next
// block's columns; always all four in the order of the columns, so that every
// element sees the operations of the column-by-column elimination.  The multipliers stay in
// place: the root's winners carry A00's LU, which the driver takes over
// (TournEpilogue::lu).
//
// Panels of 128 columns: 128 rows 0.28 ms, 2048 rows 1.08 ms, 8192 rows 1.60 ms
// (column by column, with a cluster barrier and the pivot row pulled per column:
// 0.32, 1.24, 1.80; one CTA per leaf, all levels in one launch: 0.88, 2.5, 3.2).
//
// Every elimination step uses separately rounded multiply and subtract and
// an IEEE division, in the same order as the FP64 oracle, so a tournament on
// the same panel bytes picks the same pivots bit for bit.
#include <cooperative_groups.h>

#include <atomic>
#include <climits>

#include "cf_common.cuh"
#include "cf_kernels.cuh"

namespace cg = cooperative_groups;

namespace cf {

constexpr int kTournThreads = 256;
constexpr int kTournMaxCluster = 16;

constexpr int kTB = 4;                           // columns of a block

struct TournSmem {
    // candidates of every CTA's warps, by column parity: the row's block entries,
    // then its stacked position (-1: none) as a double's bits
    alignas(16) double slot[2][32][kTB + 2];
    alignas(16) double stage[4][kTB + 2];        // a warp's candidate on its way out
    double pin[kTB][kTB];                        // the block's pivots: pin[u][t] = entry t of pivot u
    double U[kTB][kMaxV];                        // their other columns
    uint64_t bar[2];                             // all slots of a parity have arrived
    int act[2][kMaxV];                           // this CTA's rows still in the race, by block parity
    int rows[kMaxV];                             // panel row of each tile row
    int order[kMaxV];                            // stacked position of each pivot (CTA: modulo the cluster's size)
    int go[2][kTB];                              // pivot u is not zero, by block parity
    int nact[2];
    int out[4];                                  // rows a warp lost in the block
    int lab_at[2 * kMaxV];                       // root epilogue: swap simulation
    int where_[2 * kMaxV];
    int win[kMaxV];
    int cnt;
    int bad;
    int abort_flag;                              // 1: a wait in the cluster ran out
};

// Rank of a candidate as an unsigned key: |a| by its bits, NaN below every
// number but above "no candidate" (0), exactly as the oracle ranks it.
__device__ __forceinline__ unsigned long long piv_key(double a) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFull;
    return b > 0x7FF0000000000000ull ? 1ull : b + 2ull;
}

// Warp maximum of (key, smallest position); every lane gets the position (-1:
// none).  One lane usually has the largest upper word alone.
__device__ __forceinline__ int warp_best(unsigned long long key, int pos) {
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned tops = __ballot_sync(0xffffffffu, hi == mh);
    if (mh != 0u && (tops & (tops - 1u)) == 0u) return __shfl_sync(0xffffffffu, pos, __ffs(tops) - 1);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const bool top = hi == mh && lo == ml && key != 0;
    return (int)__reduce_min_sync(0xffffffffu, top ? (unsigned)pos : 0xffffffffu);
}

__device__ __forceinline__ void named_bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ int g_tourn_status = 0;               // 0 or CF_ERR_TIMEOUT

constexpr long long kTournSpin = 1ll << 17;      // polls: half a second (a poll that finds nothing takes 3.9 us)

// Waits (bounded) until the barrier's phase of this parity has completed; the
// writes of every arrival are then visible.  False where the wait, or any other
// of the cluster, ran out: the abort flags of all its CTAs are set then.
__device__ __forceinline__ bool tourn_wait(TournSmem &s, uint64_t *bar, uint32_t parity, long long limit) {
    volatile int *abort_flag = &s.abort_flag;
    for (long long i = 0; i < limit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"((uint32_t)__cvta_generic_to_shared(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if (i > 64) {
            if (*abort_flag) return false;
            __nanosleep(20);
        }
    }
    cg::cluster_group cl = cg::this_cluster();
    for (unsigned p = 0; p < cl.num_blocks(); ++p) *(volatile int *)cl.map_shared_rank(&s.abort_flag, p) = 1;
    atomicExch(&g_tourn_status, CF_ERR_TIMEOUT);
    return false;
}

// One phase more on the barrier: complete once `bytes` have arrived.
__device__ __forceinline__ void tourn_arm(uint64_t *bar, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(bar)),
                 "r"(bytes)
                 : "memory");
}
// Stores to a CTA of the cluster that count their bytes on its barrier: data and
// signal in one trip (a release after plain remote stores waits for them first).
__device__ __forceinline__ void st_async2(uint32_t dst, double a, double b, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(dst),
                 "l"(__double_as_longlong(a)), "l"(__double_as_longlong(b)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async1(uint32_t dst, double a, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
                 "l"(__double_as_longlong(a)), "r"(bar)
                 : "memory");
}
constexpr int kSlotBytes = 8 * (kTB + 1);

// Shared memory of the largest share (128 rows x 128 columns): the limit that
// is set for every launch, whatever the launch takes.
constexpr size_t kTournMaxSmem = ((sizeof(TournSmem) + 15) & ~(size_t)15) + sizeof(double) * (kMaxV + 1) * kMaxV;

struct TournLevel {
    const double *P;
    int ldp, m, w, h, arity, level, root;
    int cnt_below, off_below, off;               // nodes of the level below, first node indexes
    int per, ld;                                 // rows per CTA at most; leading dimension of the tile (odd)
    long long spin;                              // polls of a wait
    int withhold;                                // failure test: the first candidate of node 0 does not go out
};

// Root epilogue: LAPACK ipiv and the list of moved rows (relative positions)
// for bringing the winners, in pivot order, to positions 0..w-1.
__device__ void root_epilogue(TournSmem &s, int w, const TournEpilogue &ep) {
    // Home slot of a label: labels < w live in slot == label; the label of
    // a winner j with win[j] >= w lives in slot w + j.
    for (int q = threadIdx.x; q < 2 * w; q += kTournThreads) { s.lab_at[q] = q; s.where_[q] = q; }
    if (threadIdx.x == 0) s.cnt = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int j = 0; j < w; ++j) {
            const int hj = s.win[j] < w ? s.win[j] : w + j;
            const int ps = s.where_[hj];
            const int p = ps < w ? ps : s.win[ps - w];
            ep.ipiv[ep.k0 + j] = ep.k0 + p + 1;
            if (ps != j) {
                const int hx = s.lab_at[j];
                s.lab_at[j] = hj; s.where_[hj] = j;
                s.lab_at[ps] = hx; s.where_[hx] = ps;
            }
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 2 * w; q += kTournThreads) {
        const int hq = s.lab_at[q];
        if (hq == q) continue;
        const int at = atomicAdd(&s.cnt, 1);     // any order: the interchanges are applied as one gather
        ep.swap_dst[at] = q < w ? q : s.win[q - w];
        ep.swap_src[at] = hq < w ? hq : s.win[hq - w];
    }
    __syncthreads();
    if (threadIdx.x == 0) *ep.swap_cnt = s.cnt;
}

__global__ void __launch_bounds__(kTournThreads, 1)
k_tourn_level(TournLevel lv, TournWS ws, TournEpilogue ep) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TournSmem &s = *reinterpret_cast<TournSmem *>(smem_raw);
    double *tile = reinterpret_cast<double *>(smem_raw + ((sizeof(TournSmem) + 15) & ~(size_t)15));   // [column][row], ld odd
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), ncta = (int)cl.num_blocks();
    const int g = blockIdx.x / ncta;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int w = lv.w, ld = lv.ld;
    int *dst = ws.node_win + (size_t)(lv.off + g) * kMaxV;

    // ---- this CTA's rows: stacked positions rank, rank + ncta, ... (dealt out,
    // since the rows of one child tend to be chosen together)
    int total = 0, mine = 0;
    if (lv.level == 0) {
        total = min(lv.h, lv.m - g * lv.h);
        mine = total > rank ? (total - rank + ncta - 1) / ncta : 0;
        if (tid < mine) s.rows[tid] = g * lv.h + rank + tid * ncta;
    } else {
        const int child0 = g * lv.arity, nchild = min(lv.arity, lv.cnt_below - child0);
        if (nchild == 1) {                       // pass-through
            const int src = lv.off_below + child0, np = ws.node_cnt[src];
            if (rank == 0) {
                for (int j = tid; j < np; j += kTournThreads) dst[j] = ws.node_win[(size_t)src * kMaxV + j];
                if (tid == 0) ws.node_cnt[lv.off + g] = np;
            }
            return;
        }
        int at = -1, base = 0;
        const int want = rank + tid * ncta;
        for (int q = 0; q < nchild; ++q) {
            const int c = ws.node_cnt[lv.off_below + child0 + q];
            if (want >= base && want < base + c) at = (lv.off_below + child0 + q) * kMaxV + (want - base);
            base += c;
        }
        total = base;
        mine = total > rank ? (total - rank + ncta - 1) / ncta : 0;
        if (tid < mine) s.rows[tid] = ws.node_win[at];
    }
    if (tid < kMaxV) s.act[0][tid] = tid;
    const int npiv = min(total, w);
    const int nw = (lv.per + 31) / 32, nslots = nw * ncta;      // a slot per warp that has rows
    if (tid == 0) {
        s.nact[0] = mine;
        s.bad = s.abort_flag = 0;
        for (int b = 0; b < 2; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(&s.bar[b])),
                         "r"(1)
                         : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    for (int k = warp; k < w; k += kTournThreads / 32)
        for (int r = lane; r < mine; r += 32) tile[k * ld + r] = lv.P[(size_t)s.rows[r] + (size_t)k * lv.ldp];
    cl.sync();                                   // every CTA of the cluster is there before it is written to

    if (tid == 0)
        for (int b = 0; b < 2; ++b) tourn_arm(&s.bar[b], nslots * kSlotBytes);
    uint32_t phase = 0;                          // completed phases of the two barriers, bit per parity
    // Elements [first, last) by `step` of rows list[0 .. na) x columns k0 ..: less the
    // parts of the four pivots of block jb, in order.
    auto apply_block = [&](int jb, int par, const int *list, int na, int k0, int ncol, int first, int step) {
        const unsigned inv = na > 1 ? 0xFFFFFFFFu / (unsigned)na + 1u : 0u;
        unsigned gos = 0;
#pragma unroll
        for (int u = 0; u < kTB; ++u) gos |= s.go[par][u] ? 1u << u : 0u;
        for (int e = first; e < na * ncol; e += step) {
            const int c = na > 1 ? (int)__umulhi((unsigned)e, inv) : e;      // e / na
            const int r = list[e - c * na];
            const int k = k0 + c;
            double a = tile[k * ld + r], m[kTB], uk[kTB];
#pragma unroll
            for (int u = 0; u < kTB; ++u) {
                m[u] = tile[(jb + u) * ld + r];
                uk[u] = s.U[u][k];
            }
            if (gos == (1u << kTB) - 1u) {
#pragma unroll
                for (int u = 0; u < kTB; ++u) a = sub_rn(a, mul_rn(m[u], uk[u]));
            } else {
#pragma unroll
                for (int u = 0; u < kTB; ++u)
                    if (gos >> u & 1u) a = sub_rn(a, mul_rn(m[u], uk[u]));
            }
            tile[k * ld + r] = a;
        }
    };
    __syncthreads();
    for (int j0 = 0, cur = 0; j0 < npiv; j0 += kTB, cur ^= 1) {
        // Here the rows of act[cur] have every earlier block's part in this block's
        // columns, and all but the last block's in the columns right of it.
        const int cb = min(kTB, npiv - j0);
        const int nact = s.nact[cur];
        if (warp >= nw) {
            // ---- the last block's part, beside this block's chain
            if (j0 > 0)
                apply_block(j0 - kTB, cur ^ 1, s.act[cur], nact, j0 + kTB, w - j0 - kTB, tid - 32 * nw,
                            kTournThreads - 32 * nw);
        } else {
            // ---- the block's columns: this thread's row, its entries j0 .. j0 + 3
            bool live = tid < nact;
            const int row = live ? s.act[cur][tid] : 0;
            const int pos = rank + row * ncta;
            double x[kTB];
#pragma unroll
            for (int t = 0; t < kTB; ++t) x[t] = (live && j0 + t < w) ? tile[(j0 + t) * ld + row] : 0.0;
            bool lost = false;
#pragma unroll 1
            for (int u = 0; u <= cb; ++u) {
                double l = 0.0;
                if (u > 0) {
                    // ---- the winner of column j0 + u - 1, found by every warp alike
                    const int par = (j0 + u - 1) & 1;
                    const bool ok = __all_sync(0xffffffffu, tourn_wait(s, &s.bar[par], (phase >> par) & 1u, lv.spin));
                    phase ^= 1u << par;
                    // (armed again before this warp's next candidate goes out, which
                    // every sender of the next but one waits for)
                    if (tid == 0 && ok && !*(volatile int *)&s.abort_flag) tourn_arm(&s.bar[par], nslots * kSlotBytes);
                    const int best = lane < nslots ? (int)__double_as_longlong(s.slot[par][lane][kTB]) : -1;
                    const unsigned long long key = best >= 0 ? piv_key(s.slot[par][lane][u - 1]) : 0ull;
                    // (after a wait that ran out the slots hold anything: any row in range will do, the
                    // order is replaced at the end)
                    int gi = warp_best(key, best);
                    if (!ok || (unsigned)gi >= (unsigned)total) gi = j0 + u - 1;
                    const int at = max(__ffs(__ballot_sync(0xffffffffu, best == gi)) - 1, 0);
                    const double *pv = s.slot[par][at];
                    const double piv = pv[u - 1];
                    const bool go = !is_zero(piv);           // a zero pivot eliminates nothing
                    if (live && pos == gi) {
                        live = false;
                        lost = true;
                    }
                    if (warp == 0) {
                        if (lane < kTB) s.pin[u - 1][lane] = pv[lane];
                        if (lane == 0) {
                            s.order[j0 + u - 1] = gi;
                            s.go[cur][u - 1] = go;
                            if (!go) s.bad = 1;
                        }
                    }
                    // ---- multiplier (kept in the entry) and the later entries
                    if (live && go) {
                        double a = x[0];
#pragma unroll
                        for (int t = 1; t < kTB; ++t) a = t == u - 1 ? x[t] : a;
                        l = div_rn(a, piv);
#pragma unroll
                        for (int t = 0; t < kTB; ++t) x[t] = t == u - 1 ? l : x[t];
                        switch (u) {             // entries u .. 3
                            case 1: x[1] = sub_rn(x[1], mul_rn(l, pv[1])); [[fallthrough]];
                            case 2: x[2] = sub_rn(x[2], mul_rn(l, pv[2])); [[fallthrough]];
                            case 3: x[3] = sub_rn(x[3], mul_rn(l, pv[3])); [[fallthrough]];
                            default: break;
                        }
                    }
                    __syncwarp();
                }
                if (u == cb) break;
                // ---- this warp's candidate for column j0 + u, into every CTA's slots
                double a = x[0];
#pragma unroll
                for (int t = 1; t < kTB; ++t) a = t == u ? x[t] : a;
                const int best = warp_best(live ? piv_key(a) : 0ull, pos);
                if (best < 0 ? lane == 0 : (live && pos == best)) {
#pragma unroll
                    for (int t = 0; t < kTB; ++t) s.stage[warp][t] = x[t];
                    s.stage[warp][kTB] = __longlong_as_double((long long)best);
                }
                __syncwarp();
                const int par = (j0 + u) & 1;
                // lane = (CTA, half): asynchronous stores that count on the CTA's barrier
                {
                    const int cta = lane >> 1, half = lane & 1;
                    if (cta < ncta && !(lv.withhold && g == 0 && rank == 0 && warp == 0 && j0 + u == 0)) {
                        uint32_t dst, bar;
                        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                                     : "=r"(dst)
                                     : "r"((uint32_t)__cvta_generic_to_shared(&s.slot[par][rank * nw + warp][0])), "r"(cta));
                        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                                     : "=r"(bar)
                                     : "r"((uint32_t)__cvta_generic_to_shared(&s.bar[par])), "r"(cta));
                        const double *st = s.stage[warp];
                        st_async2(dst + 16 * half, st[2 * half], st[2 * half + 1], bar);
                        if (half == 0) st_async1(dst + 8 * kTB, st[kTB], bar);
                    }
                }
            }
            // ---- the rows back, the list without the chosen ones
            if (tid < nact) {
#pragma unroll
                for (int t = 0; t < kTB; ++t)
                    if (j0 + t < w) tile[(j0 + t) * ld + row] = x[t];
            }
            const unsigned gone = __ballot_sync(0xffffffffu, lost);
            if (lane == 0) s.out[warp] = __popc(gone);
            named_bar_sync(1, 32 * nw);
            int before = 0;
            for (int q = 0; q < warp; ++q) before += s.out[q];
            int all = 0;
            for (int q = 0; q < nw; ++q) all += s.out[q];
            if (tid < nact && !lost) s.act[cur ^ 1][tid - before - __popc(gone & ((1u << lane) - 1u))] = row;
            if (tid == 0) s.nact[cur ^ 1] = nact - all;
        }
        __syncthreads();
        const int k1 = j0 + kTB;                 // first column right of the block
        if (k1 >= w || k1 >= npiv) {
            if (lv.root && rank == 0 && ep.lu != nullptr && npiv == w)
                for (int e = tid; e < kTB * kTB; e += kTournThreads)
                    if (e / kTB < cb && j0 + e % kTB < w) ep.lu[(j0 + e / kTB) + (size_t)(j0 + e % kTB) * kMaxV] = s.pin[e / kTB][e % kTB];
            break;                               // no selection left
        }
        if (ncta > 1) cl.sync();                 // every CTA's rows have the last block's part
        // ---- the pivot rows' other columns, a column per thread: as they were at
        // the block's start, then each less the earlier ones' parts
        if (tid < w - k1) {
            const int k = k1 + tid;
            double v[kTB];
#pragma unroll
            for (int u = 0; u < kTB; ++u) {
                const int own = s.order[j0 + u] % ncta;
                v[u] = cl.map_shared_rank(tile, own)[(size_t)k * ld + s.order[j0 + u] / ncta];
            }
#pragma unroll
            for (int u = 1; u < kTB; ++u)
#pragma unroll
                for (int t = 0; t < u; ++t)
                    if (s.go[cur][t]) v[u] = sub_rn(v[u], mul_rn(s.pin[u][t], v[t]));
#pragma unroll
            for (int u = 0; u < kTB; ++u) s.U[u][k] = v[u];
            if (lv.root && rank == 0 && ep.lu != nullptr && npiv == w) {
#pragma unroll
                for (int u = 0; u < kTB; ++u) ep.lu[(j0 + u) + (size_t)k * kMaxV] = v[u];
            }
        }
        if (lv.root && rank == 0 && ep.lu != nullptr && npiv == w)
            for (int e = tid; e < kTB * kTB; e += kTournThreads)
                ep.lu[(j0 + e / kTB) + (size_t)(j0 + e % kTB) * kMaxV] = s.pin[e / kTB][e % kTB];
        __syncthreads();
        // ---- their part in the next block's columns (the rest goes beside its chain)
        apply_block(j0, cur, s.act[cur ^ 1], s.nact[cur ^ 1], k1, min(kTB, w - k1), tid, kTournThreads);
        __syncthreads();
    }
    __syncthreads();
    for (int j = tid; j < npiv; j += kTournThreads) {
        const int gi = s.order[j];
        if (gi % ncta == rank) {
            const int r = s.rows[gi / ncta];
            dst[j] = r;
            if (lv.root) ws.root_win[j] = r;
        }
    }
    if (rank == 0 && tid == 0) ws.node_cnt[lv.off + g] = npiv;
    if (lv.root && ep.lu != nullptr) {
        // A00's LU in pivot order: the multipliers of earlier blocks are with the
        // winners' rows, the rest was written block by block
        for (int j = warp; j < npiv; j += kTournThreads / 32) {
            if (s.order[j] % ncta != rank) continue;
            const int r = s.order[j] / ncta;
            for (int k = lane; k < j / kTB * kTB; k += 32) ep.lu[j + (size_t)k * kMaxV] = tile[k * ld + r];
        }
        if (rank == 0 && tid == 0) *ep.lu_ok = s.bad == 0 && npiv == w;
    }
    __threadfence();
    if (ncta > 1) cl.sync();                     // remote reads of the tiles and the winners' list are done
    else __syncthreads();
    if (s.abort_flag) {
        // A wait ran out: the CTAs may have followed different winners.  The first
        // rows instead, so that every list that others index with is whole; the
        // host learns of it from the status.  What is still on its way lands first.
        for (int j = rank + tid * ncta; j < npiv; j += kTournThreads * ncta) {
            dst[j] = s.rows[j / ncta];
            if (lv.root) ws.root_win[j] = s.rows[j / ncta];
        }
        if (lv.root && ep.lu != nullptr && rank == 0 && tid == 0) *ep.lu_ok = 0;
        __nanosleep(20000);
        __threadfence();
        cl.sync();
    }
    if (lv.root && rank == 0 && ep.ipiv != nullptr) {
        __syncthreads();
        for (int j = tid; j < npiv; j += kTournThreads) s.win[j] = __ldcg(ws.root_win + j);
        __syncthreads();
        root_epilogue(s, npiv, ep);
    }
}

// LU-2: gather the moved rows of every column (one warp per column) and the
// row order.  Reads all sources before writing any destination.
template <typename T>
__global__ void __launch_bounds__(256)
k_apply_swaps(T *__restrict__ A, int lda, int ncols, int k0, const int *swap_cnt, const int *swap_dst,
              const int *swap_src, int *perm) {
    __shared__ int sd[2 * kMaxV], ss[2 * kMaxV];
    const int cnt = *swap_cnt;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) { sd[e] = swap_dst[e]; ss[e] = swap_src[e]; }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int col = blockIdx.x * (blockDim.x >> 5) + warp;
    if (col < ncols) {
        T *c = A + (size_t)col * lda + k0;
        T v[2 * kMaxV / 32];
#pragma unroll
        for (int q = 0; q < 2 * kMaxV / 32; ++q) {
            const int e = lane + 32 * q;
            if (e < cnt) v[q] = c[ss[e]];
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2 * kMaxV / 32; ++q) {
            const int e = lane + 32 * q;
            if (e < cnt) c[sd[e]] = v[q];
        }
    } else if (col == ncols && perm != nullptr) {
        int *c = perm + k0;
        int v[2 * kMaxV / 32];
#pragma unroll
        for (int q = 0; q < 2 * kMaxV / 32; ++q) {
            const int e = lane + 32 * q;
            if (e < cnt) v[q] = c[ss[e]];
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2 * kMaxV / 32; ++q) {
            const int e = lane + 32 * q;
            if (e < cnt) c[sd[e]] = v[q];
        }
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
int make_tourn_plan(int m, int w, int h, int arity, TournPlan *plan) {
    if (m < 0 || w < 0 || w > kMaxV || h < 1 || h > 4 * kMaxV || arity < 2 || arity > 8) return CF_ERR_UNSUPPORTED;
    TournPlan p{};
    p.m = m; p.w = w; p.h = h; p.arity = arity;
    p.nleaves = m > 0 ? ceil_div(m, h) : 0;
    int c = p.nleaves, lv = 0, off = 0;
    while (true) {
        if (lv >= kMaxLevels) return CF_ERR_UNSUPPORTED;
        p.cnt[lv] = c; p.off[lv] = off; off += c; ++lv;
        if (c <= 1) break;
        c = (c + arity - 1) / arity;
    }
    p.nlevels = lv;
    p.total_nodes = off;
    *plan = p;
    return CF_OK;
}

size_t tourn_ws_bytes(int m, int h, int arity) {
    TournPlan p{};
    if (make_tourn_plan(m, 1, h, arity, &p) != CF_OK) return 0;
    Carver cv(nullptr);
    cv.take<int>((size_t)p.total_nodes * kMaxV);
    cv.take<int>(p.total_nodes);
    cv.take<int>(p.total_nodes);
    cv.take<int>(kMaxV);
    cv.take<int>(1);
    cv.take<int>(2 * kMaxV);
    cv.take<int>(2 * kMaxV);
    return cv.size();
}

// The counters are the FP32 tournaments', whose nodes climb the tree in one
// launch: zero before the first, left zero.  The FP64 one (a launch per level)
// has none.
int tourn_ws_carve(void *work, int m, int h, int arity, TournWS *ws, TournEpilogue *ep) {
    TournPlan p{};
    int st = make_tourn_plan(m, 1, h, arity, &p);
    if (st != CF_OK) return st;
    Carver cv(work);
    ws->node_win = cv.take<int>((size_t)p.total_nodes * kMaxV);
    ws->node_cnt = cv.take<int>(p.total_nodes);
    ws->counter = cv.take<int>(p.total_nodes);
    ws->root_win = cv.take<int>(kMaxV);
    ws->counter_bytes = sizeof(int) * (size_t)p.total_nodes;
    ep->swap_cnt = cv.take<int>(1);
    ep->swap_dst = cv.take<int>(2 * kMaxV);
    ep->swap_src = cv.take<int>(2 * kMaxV);
    return CF_OK;
}

// Largest cluster of the level kernel that the device takes: 16 (not
// portable) where some GPC has 16 SMs to give, else 8.
static int tourn_max_cluster() {
    constexpr int kDevs = 64;
    static std::atomic<int> cache[kDevs];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs) {
        cudaGetLastError();
        return 8;
    }
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    n = 8;
    if (cudaFuncSetAttribute(k_tourn_level, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kTournMaxCluster);
        cfg.blockDim = dim3(kTournThreads);
        cfg.dynamicSmemBytes = kTournMaxSmem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kTournMaxCluster;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaFuncSetAttribute(k_tourn_level, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTournMaxSmem) ==
                cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, k_tourn_level, &cfg) == cudaSuccess && clusters > 0)
            n = kTournMaxCluster;
    }
    cudaGetLastError();
    cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

static int run_tourn(const double *P, int ldp, int m, int w, int h, int arity, const TournWS &ws,
                     const TournEpilogue &ep, long long spin, bool withhold, cudaStream_t st) {
    if (h > kMaxV || arity > 8) return CF_ERR_UNSUPPORTED;      // a node has at most 8 x kMaxV rows
    TournPlan plan{};
    int rc = make_tourn_plan(m, w, h, arity, &plan);
    if (rc != CF_OK) return rc;
    if (m == 0 || w == 0) return CF_OK;
    const int sms = device_sm_count(), most = tourn_max_cluster();
    int rows = h < m ? h : m;                    // rows of the level's largest node
    for (int l = 0; l < plan.nlevels; ++l) {
        if (l > 0) {
            const int kids = arity < plan.cnt[l - 1] ? arity : plan.cnt[l - 1];
            rows = kids * (rows < w ? rows : w);
        }
        // as many CTAs per node as leave every CTA of the level an SM of its own,
        // down to 8 rows each
        int cta = ceil_div(rows, kMaxV) > 4 ? 8 : (ceil_div(rows, kMaxV) > 2 ? 4 : (rows > kMaxV ? 2 : 1));
        while (cta < most && 2ll * cta * plan.cnt[l] <= sms && ceil_div(rows, cta) > 8) cta *= 2;
        TournLevel lv{};
        lv.P = P;
        lv.ldp = ldp;
        lv.m = m;
        lv.w = w;
        lv.h = h;
        lv.arity = arity;
        lv.level = l;
        lv.root = l == plan.nlevels - 1;
        lv.cnt_below = l > 0 ? plan.cnt[l - 1] : 0;
        lv.off_below = l > 0 ? plan.off[l - 1] : 0;
        lv.off = plan.off[l];
        lv.per = ceil_div(rows, cta);
        lv.ld = lv.per | 1;
        if (ceil_div(lv.per, 32) * cta > 32) return CF_ERR_UNSUPPORTED;      // a slot per lane (1024 rows: 4 x 8, 2 x 16)
        lv.spin = spin;
        lv.withhold = withhold && l == 0;
        const size_t smem = align_up(sizeof(TournSmem), 16) + sizeof(double) * (size_t)lv.ld * w;
        // the attributes belong to the current device: set on every call
        CF_CUDA_TRY(cudaFuncSetAttribute(k_tourn_level, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTournMaxSmem));
        if (cta > 8) CF_CUDA_TRY(cudaFuncSetAttribute(k_tourn_level, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(plan.cnt[l] * cta);
        cfg.blockDim = dim3(kTournThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cta;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        CF_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_tourn_level, lv, ws, ep));
        count_launches(1);
    }
    return CF_OK;
}

int launch_tourn(const double *P, int ldp, int m, int w, int h, int arity, const TournWS &ws, const TournEpilogue &ep,
                 cudaStream_t st) {
    return run_tourn(P, ldp, m, w, h, arity, ws, ep, kTournSpin, false, st);
}

int tourn_take_status(cudaStream_t st, int *status) {
    int h = 0;
    CF_CUDA_TRY(cudaMemcpyFromSymbolAsync(&h, g_tourn_status, sizeof(int), 0, cudaMemcpyDeviceToHost, st));
    CF_CUDA_TRY(cudaStreamSynchronize(st));
    if (h != 0) {
        const int zero = 0;
        CF_CUDA_TRY(cudaMemcpyToSymbolAsync(g_tourn_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st));
        CF_CUDA_TRY(cudaStreamSynchronize(st));
    }
    *status = h;
    return CF_OK;
}

template <typename T>
int launch_apply_swaps(T *A, int lda, int ncols, int k0, const TournEpilogue &ep, int *perm, cudaStream_t st) {
    const int cols = ncols + (perm ? 1 : 0);
    if (cols == 0) return CF_OK;
    k_apply_swaps<T><<<ceil_div(cols, 8), 256, 0, st>>>(A, lda, ncols, k0, ep.swap_cnt, ep.swap_dst, ep.swap_src,
                                                          perm);
    CF_LAUNCH_CHECK();
    return CF_OK;
}

template int launch_apply_swaps<double>(double *, int, int, int, const TournEpilogue &, int *, cudaStream_t);
template int launch_apply_swaps<float>(float *, int, int, int, const TournEpilogue &, int *, cudaStream_t);

}  // namespace cf

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
extern "C" size_t cf_tourn_workspace_size(int m, int w, int leaf_h, int arity) {
    (void)w;
    (void)leaf_h;   // sized for the most leaves (h = 1), valid for every leaf height
    if (arity > 8) return 0;
    return cf::tourn_ws_bytes(m > 0 ? m : 1, 1, arity < 2 ? 2 : arity);
}

static int tourn_select_api(int m, int w, const double *panel, int ldp, int leaf_h, int arity, int *winners, void *work,
                            size_t lwork, long long spin, bool withhold, cudaStream_t stream) {
    using namespace cf;
    if (m < 0) return -1;
    if (w < 0 || w > kMaxV) return -2;
    if (m > 0 && w > 0 && panel == nullptr) return -3;
    if (ldp < (m > 1 ? m : 1)) return -4;
    if (leaf_h < 1 || leaf_h > kMaxV) return -5;
    if (arity < 2 || arity > 8) return -6;
    if (m == 0 || w == 0) return CF_OK;
    if (winners == nullptr) return -7;
    if (lwork < cf_tourn_workspace_size(m, w, leaf_h, arity) || work == nullptr) return CF_ERR_WORKSPACE;
    TournWS ws{};
    TournEpilogue ep{};
    int rc = tourn_ws_carve(work, m, 1, arity, &ws, &ep);
    if (rc != CF_OK) return rc;
    ep.ipiv = nullptr;
    ws.root_win = winners;
    return run_tourn(panel, ldp, m, w, leaf_h, arity, ws, ep, spin, withhold, stream);
}

extern "C" int cf_tourn_select(int m, int w, const double *panel, int ldp, int leaf_h, int arity, int *winners,
                               void *work, size_t lwork, cudaStream_t stream) {
    return tourn_select_api(m, w, panel, ldp, leaf_h, arity, winners, work, lwork, cf::kTournSpin, false, stream);
}

// Failure-detection test of the bounded waits, not part of the API: the first
// candidate of the first leaf is withheld, so that the wait for it gives up
// after spin_limit polls (0: the usual number).
extern "C" int cf_tourn_select_withheld(int m, int w, const double *panel, int ldp, int leaf_h, int arity, int *winners,
                                        long long spin_limit, void *work, size_t lwork, cudaStream_t stream) {
    if (spin_limit < 0) return -8;
    return tourn_select_api(m, w, panel, ldp, leaf_h, arity, winners, work, lwork,
                            spin_limit > 0 ? spin_limit : cf::kTournSpin, true, stream);
}
