// Step (c): the interleaved move sequence I of M and R_1..R_k (Sec. 4.4),
// merging of a node's two moves (Sec. 4.4 footnote), exact gains of I, the
// balanced prefixes and the best one (Alg. 1, Sec. 4.1).
//
// Interleaving in parallel.  Walking M, after each move into block b the
// sequential rule emits the shortest further prefix of R_b that brings b to
// L_max.  Blocks with R_b non-empty were overloaded when rebalancing started
// and never receive rebalancing moves, so b's weight at that point is
// D_b(i) - (weight of R_b already emitted), with D_b(i) the weight of b after
// M's first i moves.  Hence the emitted count after M move i is
// min(|R_b|, max over inflow events i' <= i of need_b(i')), need_b = the
// shortest prefix of R_b whose weight covers D_b - L_max.  Every move of M
// becomes two block events (-c at its source, +c at its target); events are
// sorted by block (stable, so M order within a block), D_b is a segmented
// sum and the running maximum of need a segmented max-scan.
//
// All list lengths (|M|, |R|, |I|) are read from device memory.
#include <climits>

#include "sequence_team.cuh"

namespace upr {
namespace {

// Exact gain of every move of I against the partition just before it (Sec.
// 4.4): warp per move, hubs (degree > kHubDegree) are left to the chunk kernel.
__global__ void k_gains_warp(const int64_t *__restrict__ xadj, const int32_t *__restrict__ adj,
                             const int32_t *__restrict__ adjw, const int32_t *__restrict__ I_node,
                             const int32_t *__restrict__ I_from, const int32_t *__restrict__ I_to,
                             const int32_t *__restrict__ d_nI, const int2 *__restrict__ pk, int32_t k, int32_t kmask,
                             int64_t *__restrict__ gain) {
    const int lane = threadIdx.x & 31;
    const int64_t nI = *d_nI;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nI;
         i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int32_t v = I_node[i];
        const uint32_t a = (uint32_t)blk_local(I_from[i], k, kmask), b = (uint32_t)blk_local(I_to[i], k, kmask);
        const int64_t e0 = xadj[v], e1 = xadj[v + 1];
        if (e1 - e0 > kHubDegree) {
            if (lane == 0) gain[i] = 0;
            continue;
        }
        long long acc = 0;
        for (int64_t e = e0 + lane; e < e1; e += 32) {
            const uint32_t bu = block_before(pk[adj[e]], i);
            const int32_t w = adjw ? adjw[e] : 1;
            acc += (bu == b ? w : 0) - (bu == a ? w : 0);
        }
        acc = warp_sum(acc);
        if (lane == 0) gain[i] = acc;
    }
}

// Exact gains of hub moves, one CTA per static chunk of a hub's adjacency:
// partial sums added to gain[i] (set to 0 by k_gains_warp) with 64-bit
// integer atomics, whose result does not depend on their order.
__global__ void __launch_bounds__(512) k_gains_hub_chunks(const HubChunk *__restrict__ chunks,
                                                          const int32_t *__restrict__ adj,
                                                          const int32_t *__restrict__ adjw,
                                                          const int2 *__restrict__ pk,
                                                          int64_t *__restrict__ gain) {
    __shared__ long long s_w[16];
    const HubChunk ch = chunks[blockIdx.x];
    const int2 me = pk[ch.v];
    const int32_t i = me.x;
    if (i == INT32_MAX) return;                  // this hub is not in I
    const uint32_t a = (uint32_t)me.y & 0xffffu, b = (uint32_t)me.y >> 16;
    long long acc = 0;
    for (int64_t e = ch.begin + threadIdx.x; e < ch.end; e += blockDim.x) {
        const uint32_t bu = block_before(pk[adj[e]], i);
        const int32_t w = adjw ? adjw[e] : 1;
        acc += (bu == b ? w : 0) - (bu == a ? w : 0);
    }
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += s_w[w];
        if (t) atomicAdd(reinterpret_cast<unsigned long long *>(&gain[i]), (unsigned long long)t);
    }
}

// number of blocks above L_max, per graph (out[0..ng) zeroed by the caller)
__global__ void k_count_over(const int64_t *__restrict__ C, const int64_t *__restrict__ Lb, int32_t K, int32_t k,
                             int32_t *__restrict__ out) {
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < K; b += gridDim.x * blockDim.x)
        if (C[b] > Lb[b]) atomicAdd(&out[b / k], 1);
}

__global__ void __launch_bounds__(team::kTT, 1) k_seq_build(const __grid_constant__ SeqBuild a) {
    __shared__ team::Smem s;
    seq_build_body(a, s);
}

__global__ void __launch_bounds__(team::kTT, 1) k_seq_best(const __grid_constant__ SeqBest a) {
    __shared__ team::Smem s;
    seq_best_body(a, s);
}

// per graph: best gain so far = 0 if the empty prefix is eligible, else "none"
__global__ void k_best_seg_init(const int32_t *__restrict__ over0, int32_t ng, long long *__restrict__ best_g,
                                long long *__restrict__ best_j) {
    UPR_FOR(g, ng) {
        best_g[g] = over0[g] == 0 ? 0 : LLONG_MIN;
        best_j[g] = LLONG_MAX;
    }
}

struct SegPoint { int32_t g; long long G; long long j; bool elig; };

// Prefix of length j = i - seg_beg + 1 of move i's graph: its gain and eligibility.
__device__ __forceinline__ SegPoint seg_point(int64_t i, const int32_t *I_node, const int32_t *gid,
                                              const int32_t *seg_beg, const int64_t *Gsum, const int32_t *diff,
                                              const int32_t *diff_excl, const int32_t *over0) {
    const int32_t g = gid[I_node[i]];
    const int32_t s = seg_beg[g];
    const long long G = Gsum[i] - (s > 0 ? Gsum[s - 1] : 0);
    const int32_t over = over0[g] + (diff_excl[i + 1] + diff[i + 1]) - (diff_excl[s] + diff[s]);
    return SegPoint{g, G, (long long)(i - s + 1), over == 0};
}

__global__ void k_best_seg_max(const int32_t *__restrict__ I_node, const int32_t *__restrict__ d_nI,
                               const int32_t *__restrict__ gid, const int32_t *__restrict__ seg_beg,
                               const int64_t *__restrict__ Gsum, const int32_t *__restrict__ diff,
                               const int32_t *__restrict__ diff_excl, const int32_t *__restrict__ over0,
                               long long *__restrict__ best_g) {
    const int64_t nI = *d_nI;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nI; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + threadIdx.x;
        int32_t key = -1;
        long long val = LLONG_MIN;
        if (i < nI) {
            const SegPoint p = seg_point(i, I_node, gid, seg_beg, Gsum, diff, diff_excl, over0);
            if (p.elig) { key = p.g; val = p.G; }
        }
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        long long m = val;
        for (unsigned r = peers; r; r &= r - 1) m = max(m, __shfl_sync(peers, val, __ffs(r) - 1));
        if (key >= 0 && (peers & ((1u << (threadIdx.x & 31)) - 1u)) == 0) atomicMax(&best_g[key], m);
    }
}

__global__ void k_best_seg_min(const int32_t *__restrict__ I_node, const int32_t *__restrict__ d_nI,
                               const int32_t *__restrict__ gid, const int32_t *__restrict__ seg_beg,
                               const int64_t *__restrict__ Gsum, const int32_t *__restrict__ diff,
                               const int32_t *__restrict__ diff_excl, const int32_t *__restrict__ over0,
                               const long long *__restrict__ best_g, long long *__restrict__ best_j) {
    const int64_t nI = *d_nI;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nI; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + threadIdx.x;
        int32_t key = -1;
        long long val = LLONG_MAX;
        if (i < nI) {
            const SegPoint p = seg_point(i, I_node, gid, seg_beg, Gsum, diff, diff_excl, over0);
            if (p.elig && p.G == best_g[p.g]) { key = p.g; val = p.j; }
        }
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        long long m = val;
        for (unsigned r = peers; r; r &= r - 1) m = min(m, __shfl_sync(peers, val, __ffs(r) - 1));
        if (key >= 0 && (peers & ((1u << (threadIdx.x & 31)) - 1u)) == 0) atomicMin(&best_j[key], m);
    }
}

// per graph: j* (the empty prefix wins ties), cut update; totals for the
// round statistics in tot[0..3) = (sum of j*, sum of gains, infeasible graphs)
__global__ void k_best_seg_final(const int32_t *__restrict__ over0, int32_t ng, long long *__restrict__ best_g,
                                 long long *__restrict__ best_j, long long *__restrict__ cut,
                                 int32_t *__restrict__ infeasible, unsigned long long *__restrict__ tot) {
    long long sj = 0, sg = 0, ninf = 0;
    UPR_FOR(g, ng) {
        long long G = best_g[g], j;
        if (G == LLONG_MIN) {
            infeasible[g] = 1;
            G = 0;
            j = 0;
            ninf++;
        } else {
            infeasible[g] = 0;
            j = (over0[g] == 0 && G == 0) ? 0 : best_j[g];
            cut[g] -= G;
        }
        best_g[g] = G;
        best_j[g] = j;
        sj += j;
        sg += G;
    }
    sj = warp_sum(sj);
    sg = warp_sum(sg);
    ninf = warp_sum(ninf);
    if ((threadIdx.x & 31) == 0) {
        if (sj) atomicAdd(&tot[0], (unsigned long long)sj);
        if (sg) atomicAdd(&tot[1], (unsigned long long)sg);
        if (ninf) atomicAdd(&tot[2], (unsigned long long)ninf);
    }
}

__global__ void k_apply_prefix_seg(const int32_t *__restrict__ I_node, const int32_t *__restrict__ I_from,
                                   const int32_t *__restrict__ I_to, const int32_t *__restrict__ d_nI,
                                   const int32_t *__restrict__ gid, const int32_t *__restrict__ seg_beg,
                                   const long long *__restrict__ best_j, const int32_t *__restrict__ vwgt,
                                   int32_t *__restrict__ part0, unsigned long long *__restrict__ C0, int32_t K) {
    extern __shared__ unsigned long long s_delta[];
    BlockDelta bd = make_block_delta(s_delta, K, C0);
    bd.init();
    const int64_t nI = *d_nI;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nI; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + threadIdx.x;
        int32_t a = -1, b = -1;
        long long c = 0;
        if (i < nI) {
            const int32_t v = I_node[i];
            const int32_t g = gid[v];
            if (i - seg_beg[g] < best_j[g]) {
                a = I_from[i];
                b = I_to[i];
                c = vwgt ? vwgt[v] : 1;
                part0[v] = b;
            }
        }
        bd.add(a, -c);
        bd.add(b, c);
    }
    bd.flush(C0);
}

// ---- carrying the gain table into the next round.  After rebalancing the
// table is W(P o M o R) = W(P o I); the next round starts from P o I^{j*},
// so the moves of I after the best prefix are undone in the table (delta
// updates), or the table is rebuilt when they touch many entries.
__device__ __forceinline__ bool rolled_back(const Rollback &rb, int64_t i) {
    if (!rb.gid) {
        const long long j = rb.best[1];
        return i >= (j < 0 ? 0 : j);
    }
    const int32_t g = rb.gid[rb.I_node[i]];
    return i - rb.seg_beg[g] >= rb.best_j[g];
}

__global__ void k_rollback_degsum(Rollback rb, const int64_t *__restrict__ xadj, unsigned long long *__restrict__ out) {
    const int64_t nI = *rb.d_nI;
    long long acc = 0;
    UPR_FOR(i, nI) {
        if (rolled_back(rb, i)) {
            const int32_t v = rb.I_node[i];
            acc += xadj[v + 1] - xadj[v];
        }
    }
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out, (unsigned long long)acc);
}

// warp per move of I; hubs are left to k_table_rollback_hubs
// (sparse rows: both blocks are keys of the row already, so nothing is inserted)
__global__ void k_table_rollback(Rollback rb, const int64_t *__restrict__ xadj, const int32_t *__restrict__ adj,
                                 const int32_t *__restrict__ adjw, int32_t k, int32_t kmask, int32_t *__restrict__ W,
                                 const int64_t *__restrict__ deg_sum, int64_t m, SparseRows sp) {
    if (*deg_sum * 4 >= m) return;          // the rebuild handles this case
    const int lane = threadIdx.x & 31;
    const int64_t nI = *rb.d_nI;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nI;
         i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        if (!rolled_back(rb, i)) continue;
        const int32_t v = rb.I_node[i];
        const int64_t e0 = xadj[v], e1 = xadj[v + 1];
        if (e1 - e0 > kHubDegree) continue;
        const int32_t a = blk_local(rb.I_to[i], k, kmask), b = blk_local(rb.I_from[i], k, kmask);
        for (int64_t e = e0 + lane; e < e1; e += 32) {
            const int32_t w = adjw ? adjw[e] : 1;
            if (sp.on()) {
                sp_sub(sp, adj[e], a, w);
                sp_add(sp, adj[e], b, w);
                continue;
            }
            int32_t *row = W + (int64_t)adj[e] * k;
            atomicSub(&row[a], w);
            atomicAdd(&row[b], w);
        }
    }
}

__global__ void __launch_bounds__(512) k_table_rollback_hubs(Rollback rb, const HubChunk *__restrict__ chunks,
                                                             const int2 *__restrict__ pk,
                                                             const int32_t *__restrict__ adj,
                                                             const int32_t *__restrict__ adjw, int32_t k,
                                                             int32_t kmask, int32_t *__restrict__ W,
                                                             const int64_t *__restrict__ deg_sum, int64_t m,
                                                             SparseRows sp) {
    if (*deg_sum * 4 >= m) return;
    const HubChunk ch = chunks[blockIdx.x];
    const int32_t i = pk[ch.v].x;
    if (i == INT32_MAX || !rolled_back(rb, i)) return;
    const int32_t a = blk_local(rb.I_to[i], k, kmask), b = blk_local(rb.I_from[i], k, kmask);
    for (int64_t e = ch.begin + threadIdx.x; e < ch.end; e += blockDim.x) {
        const int32_t w = adjw ? adjw[e] : 1;
        if (sp.on()) {
            sp_sub(sp, adj[e], a, w);
            sp_add(sp, adj[e], b, w);
            continue;
        }
        int32_t *row = W + (int64_t)adj[e] * k;
        atomicSub(&row[a], w);
        atomicAdd(&row[b], w);
    }
}

// The oscillation guard of Sec. 2: lock the nodes of the applied prefix whose
// move comes from rebalancing alone (an R move and no M move).
__global__ void k_guard_locks(Rollback rb, const int32_t *__restrict__ m_pos, const int32_t *__restrict__ r_to,
                              int8_t *__restrict__ locked) {
    const int64_t nI = *rb.d_nI;
    UPR_FOR(i, nI) {
        if (rolled_back(rb, i)) continue;
        const int32_t v = rb.I_node[i];
        if (m_pos[v] < 0 && r_to[v] >= 0) locked[v] = 1;
    }
}

// no candidate among the locked nodes
__global__ void k_guard_filter(const int8_t *__restrict__ locked, NodeList nl, Candidates cand) {
    const int64_t n = *nl.d_n;
    UPR_FOR(i, n) {
        if (!locked[nl.node[i]]) continue;
        cand.tgt[i] = -1;
        cand.s0[i] = 0;
        cand.gain[i] = 0;
    }
}

__global__ void k_reset_nodes(const int32_t *__restrict__ nodes, const int32_t *__restrict__ d_cnt,
                              int32_t *__restrict__ arr, int32_t val) {
    const int64_t cnt = *d_cnt;
    UPR_FOR(i, cnt) arr[nodes[i]] = val;
}

__global__ void k_fill_i32(int32_t *a, int64_t n, int32_t v) {
    UPR_FOR(i, n) a[i] = v;
}

}  // namespace

// ---------------------------------------------------------------- wrappers
void fill_i32(int32_t *a, int64_t n, int32_t v, cudaStream_t s) {
    if (n <= 0) return;
    k_fill_i32<<<grid_for(n), 256, 0, s>>>(a, n, v);
    UPR_LAUNCH_CHECK();
}

void reset_nodes(const int32_t *nodes, const int32_t *d_cnt, int64_t max, int32_t *arr, int32_t val, cudaStream_t s) {
    if (max <= 0) return;
    k_reset_nodes<<<grid_for(max), 256, 0, s>>>(nodes, d_cnt, arr, val);
    UPR_LAUNCH_CHECK();
}

void count_over(const GraphDev &g, const int64_t *C, int32_t *out, cudaStream_t s) {
    UPR_CUDA(cudaMemsetAsync(out, 0, sizeof(int32_t) * g.ng, s));
    k_count_over<<<grid_for(g.K()), 256, 0, s>>>(C, g.Lb, g.K(), g.k, out);
    UPR_LAUNCH_CHECK();
}

void seq_build_args(const GraphDev &g, SeqBuild &a) {
    a.n = g.n;
    a.k = g.k;
    a.kmask = g.kmask;
    a.K = g.K();
    a.ng = g.ng;
    a.vwgt = g.vwgt;
    a.gid = g.gid;
    a.xadj = g.xadj;
    a.Lb = g.Lb;
    a.kbits = a.ngbits = 1;
    while ((1ll << a.kbits) < a.K) a.kbits++;
    while ((1ll << a.ngbits) < a.ng) a.ngbits++;
}

void seq_build(const GraphDev &g, SeqBuild a, cudaStream_t s) {
    seq_build_args(g, a);
    launch_team(k_seq_build, a, a.team.size, s);
}

void seq_gains(const GraphDev &g, const int32_t *I_node, const int32_t *I_from, const int32_t *I_to,
               const int32_t *d_nI, int64_t max, const int2 *pk, int64_t *gain, const HubChunk *hub_chunks,
               int64_t n_chunks, cudaStream_t s) {
    // two waves of CTAs (moved nodes differ widely in degree)
    const unsigned blocks = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>(ceil_div(max * 32, 256), (int64_t)device_sm_count() * 16));
    k_gains_warp<<<blocks, 256, 0, s>>>(g.xadj, g.adj, g.adjw, I_node, I_from, I_to, d_nI, pk, g.k, g.kmask, gain);
    UPR_LAUNCH_CHECK();
    if (n_chunks > 0) {
        k_gains_hub_chunks<<<(unsigned)n_chunks, 512, 0, s>>>(hub_chunks, g.adj, g.adjw, pk, gain);
        UPR_LAUNCH_CHECK();
    }
}

void seq_best_args(const GraphDev &g, SeqBest &a) {
    a.K = g.K();
    a.vwgt = g.vwgt;
    a.gid = g.gid;
    a.xadj = g.xadj;
    a.Lb = g.Lb;
    a.kbits = 1;
    while ((1ll << a.kbits) < a.K) a.kbits++;
}

void seq_best(const GraphDev &g, SeqBest a, cudaStream_t s) {
    seq_best_args(g, a);
    launch_team(k_seq_best, a, a.team.size, s);
}

void table_rollback(const GraphDev &g, const Rollback &rb, int64_t max, const int2 *pk, int32_t *W,
                    const HubChunk *hub_chunks, int64_t n_chunks, int64_t *deg_sum, cudaStream_t s) {
    if (max <= 0) return;
    if (rb.gid) {           // (one graph: summed by k_seq_best)
        k_rollback_degsum<<<grid_for(max), 256, 0, s>>>(rb, g.xadj, (unsigned long long *)deg_sum);
        UPR_LAUNCH_CHECK();
    }
    const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(max * 32, 256), (int64_t)device_sm_count() * 16);
    k_table_rollback<<<blocks, 256, 0, s>>>(rb, g.xadj, g.adj, g.adjw, g.k, g.kmask, W, deg_sum, g.m,
                                                      g.sp);
    UPR_LAUNCH_CHECK();
    if (n_chunks > 0) {
        k_table_rollback_hubs<<<(unsigned)n_chunks, 512, 0, s>>>(rb, hub_chunks, pk, g.adj, g.adjw, g.k, g.kmask, W,
                                                                 deg_sum, g.m, g.sp);
        UPR_LAUNCH_CHECK();
    }
}

void guard_locks(const Rollback &rb, int64_t max, int64_t n, const int32_t *m_pos, const int32_t *r_to,
                 int8_t *locked, cudaStream_t s) {
    if (n > 0) UPR_CUDA(cudaMemsetAsync(locked, 0, (size_t)n, s));
    if (max <= 0) return;
    k_guard_locks<<<grid_for(max), 256, 0, s>>>(rb, m_pos, r_to, locked);
    UPR_LAUNCH_CHECK();
}

void guard_filter(const int8_t *locked, int64_t n_max, NodeList nl, Candidates cand, cudaStream_t s) {
    if (n_max <= 0) return;
    k_guard_filter<<<grid_for(n_max), 256, 0, s>>>(locked, nl, cand);
    UPR_LAUNCH_CHECK();
}

void seq_best_seg(const GraphDev &g, const int32_t *I_node, const int32_t *d_nI, int64_t max, const int32_t *seg_beg,
                  const int64_t *Gsum, const int32_t *diff, const int32_t *diff_excl, const int32_t *over0,
                  long long *best_g, long long *best_j, int64_t *cut, int32_t *infeasible, int64_t *tot,
                  cudaStream_t s) {
    UPR_CUDA(cudaMemsetAsync(tot, 0, 3 * sizeof(int64_t), s));
    k_best_seg_init<<<grid_for(g.ng), 256, 0, s>>>(over0, g.ng, best_g, best_j);
    UPR_LAUNCH_CHECK();
    if (max > 0) {
        k_best_seg_max<<<grid_for(max), 256, 0, s>>>(I_node, d_nI, g.gid, seg_beg, Gsum, diff, diff_excl, over0, best_g);
        UPR_LAUNCH_CHECK();
        k_best_seg_min<<<grid_for(max), 256, 0, s>>>(I_node, d_nI, g.gid, seg_beg, Gsum, diff, diff_excl, over0, best_g,
                                                     best_j);
        UPR_LAUNCH_CHECK();
    }
    k_best_seg_final<<<grid_for(g.ng), 256, 0, s>>>(over0, g.ng, best_g, best_j, (long long *)cut, infeasible,
                                                    (unsigned long long *)tot);
    UPR_LAUNCH_CHECK();
}

void seq_apply_prefix_seg(const GraphDev &g, const int32_t *I_node, const int32_t *I_from, const int32_t *I_to,
                          const int32_t *d_nI, int64_t max, const int32_t *seg_beg, const long long *best_j,
                          int32_t *part0, int64_t *C0, cudaStream_t s) {
    if (max <= 0) return;
    const int64_t blocks = std::min<int64_t>(ceil_div(max, 256), (int64_t)device_sm_count() * 4);
    k_apply_prefix_seg<<<(unsigned)blocks, 256, block_delta_smem(g.K()), s>>>(
        I_node, I_from, I_to, d_nI, g.gid, seg_beg, best_j, g.vwgt, part0, (unsigned long long *)C0, g.K());
    UPR_LAUNCH_CHECK();
}

}  // namespace upr
