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
// a 2048-row panel run on 128 SMs, 16 rows each.  Per column:
//   * the threads that own a row divide by the pivot, update the next column
//     and take its argmax (redux on the key's bits), which goes straight into
//     every CTA's slots through distributed shared memory;
//   * all threads update the other columns, element by element over the rows
//     still in the race (a list, so that chosen rows cost nothing);
//   * one cluster barrier; then every warp finds the winner from the slots and
//     pulls the pivot row from its owner while the multipliers are divided.
// The eliminated rows of the root's winners are A00's LU, which the root hands
// to the driver (TournEpilogue::lu).
//
// A 2048-row, 128-column panel: 1.0 ms for its three levels (2.5 with one CTA per
// leaf and all levels in one launch), an 8192-row one 1.9 (3.2).
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

struct TournSmem {
    double prow[kMaxV];                          // pivot row from the current column on
    double mult[kMaxV];                          // multiplier of each row
    double slotv[2][4 * kTournMaxCluster];       // candidates of every CTA's warps, by column parity
    int sloti[2][4 * kTournMaxCluster];          // their stacked positions (-1: none)
    int act[kMaxV];                              // this CTA's rows still in the race
    int rows[kMaxV];                             // panel row of each tile row
    int order[kMaxV];                            // stacked position of each pivot, and its CTA
    int own[kMaxV];
    int nact;
    int hole;                                    // place of the chosen row in act
    int lab_at[2 * kMaxV];                       // root epilogue: swap simulation
    int where_[2 * kMaxV];
    int win[kMaxV];
    int cnt;
    int bad;
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

// Shared memory of the largest share (128 rows x 128 columns): the limit that
// is set for every launch, whatever the launch takes.
constexpr size_t kTournMaxSmem = ((sizeof(TournSmem) + 15) & ~(size_t)15) + sizeof(double) * (kMaxV + 1) * kMaxV;

struct TournLevel {
    const double *P;
    int ldp, m, w, h, arity, level, root;
    int cnt_below, off_below, off;               // nodes of the level below, first node indexes
    int per, ld;                                 // rows per CTA at most; leading dimension of the tile (odd)
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

    // ---- this CTA's rows: stacked positions [rank * per, rank * per + mine)
    const int p0 = rank * lv.per;
    int total = 0, mine = 0;
    if (lv.level == 0) {
        total = min(lv.h, lv.m - g * lv.h);
        mine = max(0, min(lv.per, total - p0));
        if (tid < mine) s.rows[tid] = g * lv.h + p0 + tid;
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
        for (int q = 0; q < nchild; ++q) {
            const int c = ws.node_cnt[lv.off_below + child0 + q];
            if (p0 + tid >= base && p0 + tid < base + c)
                at = (lv.off_below + child0 + q) * kMaxV + (p0 + tid - base);
            base += c;
        }
        total = base;
        mine = max(0, min(lv.per, total - p0));
        if (tid < mine) s.rows[tid] = ws.node_win[at];
    }
    if (tid < kMaxV) s.act[tid] = tid;
    if (tid == 0) { s.nact = mine; s.bad = 0; }
    __syncthreads();
    for (int k = warp; k < w; k += kTournThreads / 32)
        for (int r = lane; r < mine; r += 32) tile[k * ld + r] = lv.P[(size_t)s.rows[r] + (size_t)k * lv.ldp];
    __syncthreads();
    const int npiv = min(total, w);
    const int nw = (lv.per + 31) / 32, nslots = nw * ncta;      // a slot per warp that has rows

    // Candidate of this warp's rows in one column, into every CTA's slots.
    auto publish = [&](int par, bool have, double a, int row) {
        const int best = warp_best(have ? piv_key(a) : 0ull, p0 + row);
        const unsigned owner = __ballot_sync(0xffffffffu, have && p0 + row == best);
        const double v = __shfl_sync(0xffffffffu, a, owner ? __ffs(owner) - 1 : 0);
        if (lane < ncta) {
            TournSmem *rs = cl.map_shared_rank(&s, lane);
            rs->slotv[par][rank * nw + warp] = v;
            rs->sloti[par][rank * nw + warp] = best;
        }
    };
    if (ncta > 1) cl.sync();                     // every CTA of the cluster runs before it is written to
    if (warp < nw) publish(0, tid < mine, tid < mine ? tile[tid] : 0.0, tid);

    for (int j = 0; j < npiv; ++j) {
        if (ncta > 1) cl.sync(); else __syncthreads();
        // ---- (1) the winner, found by every warp alike
        const int par = j & 1;
        int gi, owner;
        double piv;
        {
            int at = lane, pos = lane < nslots ? s.sloti[par][lane] : -1;
            double v = pos >= 0 ? s.slotv[par][lane] : 0.0;
            unsigned long long key = pos >= 0 ? piv_key(v) : 0ull;
            if (nslots > 32) {
                const int i1 = lane + 32 < nslots ? s.sloti[par][lane + 32] : -1;
                const double v1 = i1 >= 0 ? s.slotv[par][lane + 32] : 0.0;
                const unsigned long long k1 = i1 >= 0 ? piv_key(v1) : 0ull;
                if (k1 > key || (k1 == key && k1 != 0 && i1 < pos)) { key = k1; pos = i1; v = v1; at = lane + 32; }
            }
            gi = warp_best(key, pos);
            const int src = __ffs(__ballot_sync(0xffffffffu, pos == gi)) - 1;
            piv = __shfl_sync(0xffffffffu, v, src);
            owner = __shfl_sync(0xffffffffu, at / nw, src);
        }
        const bool go = !is_zero(piv);           // a zero pivot eliminates nothing
        const int lrow = gi - owner * lv.per;
        // ---- (2) pivot row from its owner; meanwhile the multipliers
        double pr = 0.0;
        const bool pull = tid < w - j;
        if (pull) {
            const double *src = ncta > 1 ? cl.map_shared_rank(tile, owner) : tile;
            pr = src[(size_t)(j + tid) * ld + lrow];
        }
        const int nact = s.nact;
        const bool mine_won = owner == rank;
        int row = -1;
        double l = 0.0;
        if (tid < nact) {
            row = s.act[tid];
            if (mine_won && row == lrow) {
                s.hole = tid;
                row = -1;
            }
            if (row >= 0 && go) {
                l = div_rn(tile[j * ld + row], piv);
                tile[j * ld + row] = l;
                s.mult[row] = l;
            }
        }
        if (pull) s.prow[j + tid] = pr;
        if (tid == 0) { s.order[j] = gi; s.own[j] = owner; }
        if (!go && tid == 0) s.bad = 1;
        __syncthreads();
        const int jn = j + 1;
        // ---- (3) the next column and its candidates; the chosen row leaves the list
        if (mine_won && tid == kTournThreads - 1) {
            s.act[s.hole] = s.act[nact - 1];
            s.nact = nact - 1;
        }
        if (warp < nw && jn < npiv) {
            double a = 0.0;
            if (row >= 0) {
                a = tile[jn * ld + row];
                if (go) {
                    a = sub_rn(a, mul_rn(l, s.prow[jn]));
                    tile[jn * ld + row] = a;
                }
            }
            publish(jn & 1, row >= 0, a, row);
        } else if (row >= 0 && jn < w && go) {       // the last pivot of a node with fewer rows than columns
            tile[jn * ld + row] = sub_rn(tile[jn * ld + row], mul_rn(l, s.prow[jn]));
        }
        __syncthreads();
        // ---- (4) the other columns
        if (go) {
            const int na = s.nact, tot = na * (w - jn - 1);
            const unsigned inv = na > 1 ? 0xFFFFFFFFu / (unsigned)na + 1u : 0u;
#pragma unroll 4
            for (int e = tid; e < tot; e += kTournThreads) {
                const int c = na > 1 ? (int)__umulhi((unsigned)e, inv) : e;      // e / na
                const int r = s.act[e - c * na];
                const int k = jn + 1 + c;
                tile[k * ld + r] = sub_rn(tile[k * ld + r], mul_rn(s.mult[r], s.prow[k]));
            }
        }
    }
    __syncthreads();
    for (int j = tid; j < npiv; j += kTournThreads) {
        const int gi = s.order[j];
        if (s.own[j] == rank) {
            const int r = s.rows[gi - rank * lv.per];
            dst[j] = r;
            if (lv.root) ws.root_win[j] = r;
        }
    }
    if (rank == 0 && tid == 0) ws.node_cnt[lv.off + g] = npiv;
    if (lv.root && ep.lu != nullptr) {
        // the winners' eliminated rows are the LU of A00 in pivot order
        for (int j = warp; j < npiv; j += kTournThreads / 32) {
            const int gi = s.order[j];
            if (s.own[j] != rank) continue;
            for (int k = lane; k < w; k += 32) ep.lu[j + (size_t)k * kMaxV] = tile[k * ld + (gi - rank * lv.per)];
        }
        if (rank == 0 && tid == 0) *ep.lu_ok = s.bad == 0 && npiv == w;
    }
    __threadfence();
    if (ncta > 1) cl.sync();                     // remote reads of the tiles and the winners' list are done
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

// Counters must be zero before the first tournament; the tournament leaves
// them zero.
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

int launch_tourn(const double *P, int ldp, int m, int w, int h, int arity, const TournWS &ws, const TournEpilogue &ep,
                 cudaStream_t st) {
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

extern "C" int cf_tourn_select(int m, int w, const double *panel, int ldp, int leaf_h, int arity, int *winners,
                               void *work, size_t lwork, cudaStream_t stream) {
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
    CF_CUDA_TRY(cudaMemsetAsync(ws.counter, 0, ws.counter_bytes, stream));
    ws.root_win = winners;
    return launch_tourn(panel, ldp, m, w, leaf_h, arity, ws, ep, stream);
}
