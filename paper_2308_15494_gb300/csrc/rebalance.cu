// Step (d): rebalancing (Sec. 6) in synchronous sub-rounds.  Per sub-round:
// every node of an overloaded block proposes its best-gain move into a block
// that stays within L_max (unconnected nodes: the lightest block, Sec. 6.1);
// proposals are ordered by the priority of Sec. 6.1 (g * c(u) for g >= 0,
// g / c(u) for g < 0, higher first, ties by node id) through an exact integer
// key; each source keeps the minimal prefix that removes its excess; each
// target admits the longest prefix that fits.  engine.cu runs the loop, from
// the host or as one CUDA graph whose condition k_reb_continue sets.
#include <cstddef>

#include "rebalance_team.cuh"

namespace upr {
namespace {

int sm_count_reb() {
    static int cnt = 0;
    if (!cnt) {
        int dev = 0;
        UPR_CUDA(cudaGetDevice(&dev));
        UPR_CUDA(cudaDeviceGetAttribute(&cnt, cudaDevAttrMultiProcessorCount, dev));
    }
    return cnt;
}

template <int G>
__global__ void __launch_bounds__(256) k_propose(const __grid_constant__ GraphDev g, const int32_t *__restrict__ list,
                                                 const int32_t *__restrict__ d_n1, const int32_t *__restrict__ part,
                                                 const int32_t *__restrict__ W, const __grid_constant__ RebalState st,
                                                 int32_t *__restrict__ prop_tgt, int32_t *__restrict__ prop_gain,
                                                 int32_t *__restrict__ flags) {
    propose_rows<G, 256>(g, list, *d_n1, part, W, st, prop_tgt, prop_gain, flags);
}

__device__ __forceinline__ int32_t int4_at(const int4 &x, int c) {
    return c == 0 ? x.x : c == 1 ? x.y : c == 2 ? x.z : x.w;
}

// Proposals of the listed nodes (the nodes of blocks overloaded when
// rebalancing started; those that left them are skipped).  Vectorised rows
// as in selection; room(b) = L_max - C[b] for an allowed target, -1 for an
// excluded one, so one comparison c <= room(b) tests validity.  With one
// graph the rooms are staged in shared memory; in a batch each node reads its
// graph's blocks from global memory.
template <int G, int CH, bool EXACT, bool BATCH, bool PACK = false>
__global__ void __launch_bounds__(256) k_propose_vec(const GraphDev g, const int32_t *__restrict__ list,
                                                     const int32_t *__restrict__ d_n1,
                                                     const int32_t *__restrict__ part, const int32_t *__restrict__ W,
                                                     RebalState st, int32_t *__restrict__ prop_tgt,
                                                     int32_t *__restrict__ prop_gain, int32_t *__restrict__ flags) {
    // EXACT: k == 4 * G * CH, every lane's four blocks exist.  The room of an
    // excluded block (which includes every overloaded block, so the node's own
    // block) is -1, so "c <= room" alone decides whether a block may receive
    // the node; room is clamped to 2^31 - 1 since c < 2^31.
    const int64_t n1 = *d_n1;
    if (n1 == 0) return;
    const int32_t k = g.k;
    extern __shared__ int32_t s_room[];
    int8_t *s_over = reinterpret_cast<int8_t *>(s_room + k);
    if (!BATCH) {
        for (int i = threadIdx.x; i < k; i += blockDim.x) {
            const int64_t room = st.Lb[i] - st.C[i];
            s_room[i] = st.excl[i] ? -1 : (int32_t)(room > 0x7fffffffLL ? 0x7fffffffLL : room);
            s_over[i] = st.over[i];
        }
        __syncthreads();
    }
    constexpr int kGroups = 256 / G;
    const int gid = threadIdx.x / G, gl = threadIdx.x % G;
    const int gbase = (threadIdx.x & 31) & ~(G - 1);
    // PACK (unit weights, one graph): a column's score is one integer,
    // (omega << kb) + (2^kb - 1 - b), whose maximum is the largest omega, ties
    // to the smaller block.  The second part is fixed for the launch, and -2^31
    // for a block without room for a node of weight 1: omega << kb is at most
    // 2^31 - 2^kb (gb + kb <= 31), so that such a score is negative and every
    // other one stays below 2^31; a score below 2^kb has omega = 0.  The
    // loop issues instructions rather than waits for rows (2.2 million rows of
    // 64 blocks, 0.6 of every issue slot at 3.7 TB/s), and this takes two per
    // column, where a mask of the allowed columns took six (with the same change to
    // the selection, 2^22 nodes, 64 blocks: 17.74 -> 17.52 ms)
    const int kb = st.pack_bits;
    const int32_t kmask = (1 << kb) - 1;
    int32_t cst[CH][4];
    if (PACK) {
#pragma unroll
        for (int j = 0; j < CH; j++)
#pragma unroll
            for (int cc = 0; cc < 4; cc++) {
                const int b = 4 * (gl + G * j) + cc;
                cst[j][cc] = (EXACT || b < k) && s_room[b] >= 1 ? kmask - b : INT32_MIN;
            }
    }
    for (int64_t base = (int64_t)blockIdx.x * kGroups; base < n1; base += (int64_t)gridDim.x * kGroups) {
        const int64_t i = base + gid;
        const int32_t v = i < n1 ? list[i] : 0;
        const int32_t ag = i < n1 ? part[v] : 0;
        const int32_t a = BATCH ? blk_local(g, ag) : ag, b0 = ag - a;
        const bool src = i < n1 && (BATCH ? st.over[ag] : s_over[a]);
        const int4 zero = make_int4(0, 0, 0, 0);
        int4 r[CH];
        // the row is loaded as soon as v is known, beside its block (a
        // listed node that is no longer a source ignores it)
        if (i < n1) {
            const int4 *row4 = reinterpret_cast<const int4 *>(W + (int64_t)v * k);
#pragma unroll
            for (int j = 0; j < CH; j++) {
                const int q = gl + G * j;
                r[j] = (EXACT || 4 * q < k) ? row4[q] : zero;
            }
        } else {
#pragma unroll
            for (int j = 0; j < CH; j++) r[j] = zero;
        }
        const int q4 = a >> 2;
        int32_t mine = 0;
#pragma unroll
        for (int j = 0; j < CH; j++)
            if (j == q4 / G) mine = int4_at(r[j], a & 3);
        const int32_t own = __shfl_sync(0xffffffffu, mine, gbase + (q4 % G));
        const int32_t c = src ? (g.vwgt ? g.vwgt[v] : 1) : 1;
        // best valid block: the largest omega(v, V_b) (gain = omega - own), ties to the smaller b
        int32_t bw = 0, bt = -1;
        if (PACK) {
            int32_t best = 0;
#pragma unroll
            for (int j = 0; j < CH; j++) {
#pragma unroll
                for (int cc = 0; cc < 4; cc++) {
                    best = max(best, (int4_at(r[j], cc) << kb) + cst[j][cc]);
                }
            }
            for (int o = G / 2; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
            if (src && best > kmask) { bw = best >> kb; bt = kmask - (best & kmask); }
        } else if (src) {
#pragma unroll
            for (int j = 0; j < CH; j++) {
#pragma unroll
                for (int cc = 0; cc < 4; cc++) {
                    const int b = 4 * (gl + G * j) + cc;
                    const int32_t w = int4_at(r[j], cc);
                    if ((!EXACT && b >= k) || w <= 0) continue;
                    int32_t room;
                    if (BATCH) {
                        const int64_t rm = st.Lb[b0 + b] - st.C[b0 + b];
                        room = st.excl[b0 + b] ? -1 : (int32_t)(rm > 0x7fffffffLL ? 0x7fffffffLL : rm);
                    } else {
                        room = s_room[b];
                    }
                    if (c > room) continue;
                    if (bt < 0 || w > bw) { bw = w; bt = b; }
                }
            }
        }
        int32_t id = bt;
        if (!PACK) group_argmax32<G>(bw, id);
        if (i < n1 && gl == 0) {
            int32_t tgt = src && id >= 0 ? b0 + id : -1;
            int32_t gain = bw - own;
            if (src && tgt < 0) {
                const int32_t light = st.light[BATCH ? blk_graph(g, ag) : 0];
                if (light >= 0) {
                    const int64_t lroom = st.Lb[light] - st.C[light];
                    if ((int64_t)c <= lroom) { tgt = light; gain = -own; }
                }
            }
            if (tgt >= 0) {
                prop_tgt[v] = tgt;
                prop_gain[v] = gain;
                if (st.lgain) { st.lgain[i] = gain; st.lsrc[i] = ag; }
            }
            flags[i] = tgt >= 0 ? 1 : 0;
        }
    }
}

// Proposals over the sparse table: G lanes per node walk the node's slots;
// the best valid block has the largest omega(v, V_b), ties to the smaller b.
template <int G>
__global__ void __launch_bounds__(256) k_propose_sparse(const GraphDev g, const int32_t *__restrict__ list,
                                                        const int32_t *__restrict__ d_n1,
                                                        const int32_t *__restrict__ part, RebalState st,
                                                        int32_t *__restrict__ prop_tgt, int32_t *__restrict__ prop_gain,
                                                        int32_t *__restrict__ flags) {
    const int64_t n1 = *d_n1;
    constexpr int kGroups = 256 / G;
    const int gid = threadIdx.x / G, gl = threadIdx.x % G;
    const SparseRows &sp = g.sp;
    for (int64_t base = (int64_t)blockIdx.x * kGroups; base < n1; base += (int64_t)gridDim.x * kGroups) {
        const int64_t i = base + gid;
        const int32_t v = i < n1 ? list[i] : 0;
        const int32_t ag = i < n1 ? part[v] : 0;
        const bool src = i < n1 && st.over[ag];
        const int32_t a = blk_local(g, ag), b0 = ag - a;
        int32_t bw = 0, bt = -1, own = 0;
        const int32_t c = src ? (g.vwgt ? g.vwgt[v] : 1) : 1;
        if (src) {
            own = sp_get(sp, v, a);
            for (int64_t q = sp.off[v] + gl; q < sp.off[v + 1]; q += G) {
                const int2 e = sp.slot[q];
                if (e.x == kEmpty || e.y <= 0) continue;
                const int32_t gb = b0 + e.x;
                if (st.excl[gb] || st.C[gb] + c > st.Lb[gb]) continue;
                if (bt < 0 || e.y > bw || (e.y == bw && e.x < bt)) { bw = e.y; bt = e.x; }
            }
        }
        int32_t id = bt;
        group_argmax32<G>(bw, id);
        if (i < n1 && gl == 0) {
            int32_t tgt = src && id >= 0 ? b0 + id : -1;
            int32_t gain = bw - own;
            if (src && tgt < 0) {
                const int32_t light = st.light[blk_graph(g, ag)];
                if (light >= 0 && (int64_t)c <= st.Lb[light] - st.C[light]) { tgt = light; gain = -own; }
            }
            if (tgt >= 0) {
                prop_tgt[v] = tgt;
                prop_gain[v] = gain;
                if (st.lgain) { st.lgain[i] = gain; st.lsrc[i] = ag; }
            }
            flags[i] = tgt >= 0 ? 1 : 0;
        }
    }
}

// ---- loop control.  One graph: one CTA each (K = k <= 4096).  A batch: a
// grid over the graphs, warp per graph; the last CTA to finish (ticket)
// updates the control block.
// The last CTA of a batch controller grid: true in thread 0 of that CTA.
__device__ __forceinline__ bool last_cta(RebalCtl *ctl) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_last) {
        __threadfence();
        return true;
    }
    return false;
}

__global__ void k_reb_init_batch(const int64_t *__restrict__ C, const int64_t *__restrict__ Lb, int32_t K,
                                 int8_t *__restrict__ excl, RebalCtl *__restrict__ ctl) {
    int any = 0;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < K; b += gridDim.x * blockDim.x) {
        const bool o = C[b] > Lb[b];
        excl[b] = o ? 1 : 0;
        any |= o;
    }
    if (__syncthreads_or(any) && threadIdx.x == 0) atomicOr(&ctl->flag, 1);
    if (last_cta(ctl)) {
        const int f = atomicAdd(&ctl->flag, 0);
        ctl->active = 0;
        ctl->stopped = f ? 0 : 1;
        ctl->light = -1;
        ctl->subrounds = 0;
        ctl->nR = 0;
        ctl->n1_active = 0;
        ctl->flag = 0;
        ctl->ticket = 0;
    }
}

// Batch form: warp per graph.
__global__ void k_reb_begin_batch(const int64_t *__restrict__ C, const int64_t *__restrict__ Lb, int32_t k,
                                  int32_t ng, const int8_t *__restrict__ excl, int8_t *__restrict__ over,
                                  int8_t *__restrict__ reject, const int32_t *__restrict__ d_n1,
                                  int32_t max_subrounds, RebalCtl *__restrict__ ctl, int32_t *__restrict__ light) {
    const int lane = threadIdx.x & 31;
    int any = 0;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < ng;
         g += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        int64_t bw = 0;
        int32_t bb = -1;
        for (int32_t j = lane; j < k; j += 32) {
            const int32_t b = (int32_t)g * k + j;
            const bool o = C[b] > Lb[b];
            over[b] = o ? 1 : 0;
            reject[b] = 0;
            any |= o;
            // lightest: smallest weight, ties to the smaller block (b grows with j)
            if (!excl[b] && (bb < 0 || C[b] < bw)) { bw = C[b]; bb = b; }
        }
        // argmin over the warp: negate weights for group_argmax (larger score wins, ties to smaller id)
        int64_t sc = -bw;
        group_argmax<32>(sc, bb);
        if (lane == 0) light[g] = bb;
    }
    if (__syncthreads_or(any) && threadIdx.x == 0) atomicOr(&ctl->flag, 1);
    if (last_cta(ctl)) {
        const int f = atomicAdd(&ctl->flag, 0);
        const int32_t h = ctl->subrounds + 1;
        const bool run = !ctl->stopped && f && h <= max_subrounds;
        ctl->active = run ? 1 : 0;
        if (!run) ctl->stopped = 1;
        if (run) ctl->subrounds = h;
        ctl->n1_active = run ? *d_n1 : 0;
        ctl->flag = 0;
        ctl->ticket = 0;
    }
}

__global__ void __launch_bounds__(256) k_reb_end(const int64_t *__restrict__ C, const int64_t *__restrict__ Lb,
                                                 int32_t K, int8_t *excl, int8_t *reject, int8_t *over,
                                                 const int32_t *__restrict__ d_na, const int32_t *__restrict__ d_n1,
                                                 int32_t max_subrounds, RebalCtl *ctl,
                                                 cudaGraphConditionalHandle cond) {
    end_subround(C, Lb, K, excl, reject, over, d_na, d_n1, max_subrounds, ctl, cond);
}

__global__ void k_reb_end_batch(const int64_t *__restrict__ C, const int64_t *__restrict__ Lb, int32_t K,
                                int8_t *__restrict__ excl, const int8_t *__restrict__ reject,
                                const int32_t *__restrict__ d_na, RebalCtl *__restrict__ ctl) {
    if (!ctl->active) return;                 // uniform over the grid: no CTA takes a ticket
    int grew = 0, over = 0;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < K; b += gridDim.x * blockDim.x) {
        if (reject[b] && !excl[b]) { excl[b] = 1; grew = 1; }
        if (C[b] > Lb[b]) over = 1;
    }
    if (__syncthreads_or(grew) && threadIdx.x == 0) atomicOr(&ctl->flag, 1);
    if (__syncthreads_or(over) && threadIdx.x == 0) atomicOr(&ctl->flag, 2);
    if (last_cta(ctl)) {
        const int f = atomicAdd(&ctl->flag, 0);
        const int32_t na = *d_na;
        ctl->nR += na;
        if ((na == 0 && !(f & 1)) || !(f & 2)) ctl->stopped = 1;
        ctl->flag = 0;
        ctl->ticket = 0;
    }
}

template <bool UNIT, bool RANK, bool WIDE>
__global__ void __launch_bounds__(team::kTT, 1) k_reb_team(const __grid_constant__ RebalTeam a) {
    __shared__ team::Smem s;
    extern __shared__ unsigned long long s_dyn[];
    reb_team_body<UNIT, RANK, WIDE>(a, s, s_dyn);
}

__global__ void __launch_bounds__(team::kTT, 1) k_reb_start(const __grid_constant__ RebalStart a) {
    __shared__ team::Smem s;
    reb_start_body(a, s);
}

}  // namespace

int rebalance_group(int k) {
    int G = k / 4;
    return G >= 32 ? 32 : G >= 16 ? 16 : G >= 8 ? 8 : k >= 4 ? 4 : 2;
}

void rebalance_propose_scalar_list(const GraphDev &g, const int32_t *list, const int32_t *d_n1, int64_t n1_max,
                                   const int32_t *part, const int32_t *W, RebalState st, int32_t *prop_tgt,
                                   int32_t *prop_gain, int32_t *flags, cudaStream_t s) {
    if (n1_max <= 0) return;
    const int G = rebalance_group(g.k);
    const int64_t groups = 256 / G;
    const int64_t blocks = std::min<int64_t>(ceil_div(n1_max, groups), (int64_t)sm_count_reb() * 16);
#define UPR_PROP(GG) k_propose<GG><<<(unsigned)blocks, 256, 0, s>>>(g, list, d_n1, part, W, st, prop_tgt, prop_gain, \
                                                                    flags)
    switch (G) {
        case 2: UPR_PROP(2); break;
        case 4: UPR_PROP(4); break;
        case 8: UPR_PROP(8); break;
        case 16: UPR_PROP(16); break;
        default: UPR_PROP(32); break;
    }
#undef UPR_PROP
    UPR_LAUNCH_CHECK();
}

namespace {

template <int G, int CH>
void launch_propose_vec(bool exact, bool batch, unsigned blocks, size_t shm, cudaStream_t s, const GraphDev &g,
                        const int32_t *list, const int32_t *d_n1, const int32_t *part, const int32_t *W,
                        const RebalState &st, int32_t *prop_tgt, int32_t *prop_gain, int32_t *flags) {
    // one full wave of CTAs at most (the kernel loops over the list)
    auto go = [&](auto kern) {
        kern<<<wave_grid((const void *)kern, 256, shm, blocks), 256, shm, s>>>(g, list, d_n1, part, W, st, prop_tgt,
                                                                             prop_gain, flags);
    };
    const bool pack = !batch && st.pack_bits > 0 && g.vwgt == nullptr;
    if constexpr (CH == 1 || (G == 32 && CH == 2)) {
        if (!exact) {
            if (batch) go(k_propose_vec<G, CH, false, true>);
            else if (pack) go(k_propose_vec<G, CH, false, false, true>);
            else go(k_propose_vec<G, CH, false, false>);
            return;
        }
    }
    if (batch) go(k_propose_vec<G, CH, true, true>);
    else if (pack) go(k_propose_vec<G, CH, true, false, true>);
    else go(k_propose_vec<G, CH, true, false>);
}

}  // namespace

void rebalance_propose_list(const GraphDev &g, const int32_t *list, const int32_t *d_n1, int64_t n1_max,
                            const int32_t *part, const int32_t *W, RebalState st, int32_t *prop_tgt,
                            int32_t *prop_gain, int32_t *flags, LaneCfg cfg, cudaStream_t s) {
    if (n1_max <= 0) return;
    const int k = g.k;
    const bool batch = g.ng > 1;
    if (g.sp.on()) {
        const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(n1_max, 256 / 8), (int64_t)sm_count_reb() * 8);
        k_propose_sparse<8><<<blocks, 256, 0, s>>>(g, list, d_n1, part, st, prop_tgt, prop_gain, flags);
        UPR_LAUNCH_CHECK();
        return;
    }
    const size_t shm = batch ? 0 : sizeof(int32_t) * (size_t)k + (size_t)k + 16;
    LaneCfg cands[3];
    if (lane_candidates(k, cands) > 0) {
        if (cfg.G <= 0) cfg = cands[0];
        const int G = cfg.G, CH = cfg.CH;
        const bool exact = k == 4 * G * CH;
        const int64_t groups = 256 / G;
        const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(n1_max, groups), (int64_t)sm_count_reb() * 8);
#define UPR_PVC(GG, CC)                                                                                        \
    if (G == GG && CH == CC) {                                                                                 \
        launch_propose_vec<GG, CC>(exact, batch, blocks, shm, s, g, list, d_n1, part, W, st, prop_tgt,         \
                                   prop_gain, flags);                                                          \
        UPR_LAUNCH_CHECK();                                                                                    \
        return;                                                                                                \
    }
        UPR_PVC(1, 1) UPR_PVC(2, 1) UPR_PVC(4, 1) UPR_PVC(8, 1) UPR_PVC(16, 1) UPR_PVC(32, 1)
        UPR_PVC(1, 2) UPR_PVC(2, 2) UPR_PVC(4, 2) UPR_PVC(8, 2) UPR_PVC(16, 2) UPR_PVC(32, 2)
        UPR_PVC(1, 4) UPR_PVC(2, 4) UPR_PVC(4, 4) UPR_PVC(8, 4) UPR_PVC(16, 4)
#undef UPR_PVC
        throw CudaError{cudaErrorInvalidValue, "rebalance_propose_list: unsupported lane schedule"};
    }
    rebalance_propose_scalar_list(g, list, d_n1, n1_max, part, W, st, prop_tgt, prop_gain, flags, s);
}

void rebalance_start_args(const GraphDev &g, RebalStart &a) {
    a.n = g.n;
    a.K = g.K();
    a.Lb = g.Lb;
    a.batch = g.ng > 1;
}

void rebalance_start(const GraphDev &g, RebalStart a, cudaStream_t s) {
    rebalance_start_args(g, a);
    launch_team(k_reb_start, a, a.team.size, s);
}

size_t rebalance_order_args(const GraphDev &g, RebalTeam &a) {
    a.K = g.K();
    a.kbits = 1;
    while ((1ll << a.kbits) < a.K) a.kbits++;
    a.vwgt = g.vwgt;
    a.Lb = g.Lb;
    // (weighted: the warps' block sums are 64-bit, 64 KB at K = 256)
    return a.K <= kRebRankK && g.vwgt ? sizeof(unsigned long long) * team::kTW * (size_t)a.K : 0;
}

void rebalance_order(const GraphDev &g, RebalTeam a, cudaStream_t s) {
    if (g.n <= 0) return;
    const size_t shm = rebalance_order_args(g, a);
    const bool rank = a.K <= kRebRankK, wide = 1 + a.gbits + 2 * a.cbits > 63;
    auto go = [&](auto kern) { launch_team(kern, a, a.team.size, s, shm); };
    if (!g.vwgt) {           // (unit weights: keys of at most 34 bits)
        if (rank) go(k_reb_team<true, true, false>);
        else go(k_reb_team<true, false, false>);
    } else if (wide) {
        if (rank) go(k_reb_team<false, true, true>);
        else go(k_reb_team<false, false, true>);
    } else {
        if (rank) go(k_reb_team<false, true, false>);
        else go(k_reb_team<false, false, false>);
    }
}

// Grid of a batch controller: warp per graph (begin) or thread per block.
inline unsigned ctl_grid(int64_t items) {
    return (unsigned)std::min<int64_t>(ceil_div(items > 0 ? items : 1, 256), (int64_t)sm_count_reb() * 2);
}

// The batch controllers count finished CTAs in ctl->ticket and collect a flag
// in ctl->flag; both are cleared before every such launch, so nothing
// depends on what the control block held before.
inline void clear_ticket(RebalCtl *ctl, cudaStream_t s) {
    static_assert(offsetof(RebalCtl, ticket) == offsetof(RebalCtl, flag) + sizeof(int32_t), "flag, ticket adjacent");
    UPR_CUDA(cudaMemsetAsync(&ctl->flag, 0, sizeof(int32_t) + sizeof(uint32_t), s));
}

void rebalance_init_batch(const GraphDev &g, const int64_t *C, int8_t *excl, RebalCtl *ctl, cudaStream_t s) {
    clear_ticket(ctl, s);
    k_reb_init_batch<<<ctl_grid(g.K()), 256, 0, s>>>(C, g.Lb, g.K(), excl, ctl);
    UPR_LAUNCH_CHECK();
}

void rebalance_begin_batch(const GraphDev &g, const int64_t *C, const int8_t *excl, int8_t *over, int8_t *reject,
                           const int32_t *d_n1, int32_t max_subrounds, RebalCtl *ctl, int32_t *light, cudaStream_t s) {
    clear_ticket(ctl, s);
    k_reb_begin_batch<<<ctl_grid((int64_t)g.ng * 32), 256, 0, s>>>(C, g.Lb, g.k, g.ng, excl, over, reject, d_n1,
                                                                   max_subrounds, ctl, light);
    UPR_LAUNCH_CHECK();
}

// The loop condition of the graph-resident rebalancing loop: run another
// sub-round while the loop has not stopped and sub-rounds are left.
__global__ void k_reb_continue(const RebalCtl *__restrict__ ctl, int32_t max_subrounds,
                               cudaGraphConditionalHandle handle) {
    if (threadIdx.x == 0)
        cudaGraphSetConditional(handle, (!ctl->stopped && ctl->subrounds < max_subrounds) ? 1u : 0u);
}

void rebalance_continue(const RebalCtl *ctl, int32_t max_subrounds, cudaGraphConditionalHandle handle,
                        cudaStream_t s) {
    k_reb_continue<<<1, 32, 0, s>>>(ctl, max_subrounds, handle);
    UPR_LAUNCH_CHECK();
}

void rebalance_end(const GraphDev &g, const int64_t *C, int8_t *excl, int8_t *reject, int8_t *over,
                   const int32_t *d_na, const int32_t *d_n1, int32_t max_subrounds, RebalCtl *ctl, cudaStream_t s,
                   cudaGraphConditionalHandle cond) {
    if (g.ng == 1) {
        k_reb_end<<<1, 256, 0, s>>>(C, g.Lb, g.K(), excl, reject, over, d_na, d_n1, max_subrounds, ctl, cond);
    } else {
        clear_ticket(ctl, s);
        k_reb_end_batch<<<ctl_grid(g.K()), 256, 0, s>>>(C, g.Lb, g.K(), excl, reject, d_na, ctl);
    }
    UPR_LAUNCH_CHECK();
}

}  // namespace upr
