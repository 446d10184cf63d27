// All rounds of a refinement call on a small graph in one launch: the steps of
// the round (engine.cu's run_round_once) by one CTA or one cluster, whose
// barriers stand where launches end, and the rebalancing loop on the device.
// Launched step by step, a round of a graph of 10^3 to 10^4 nodes is about
// seventeen launches and a wait of the host for every sub-round and round,
// most of its time outside the kernels' work.  In one launch the chains of
// dependent loads and barriers of a step bound it (some 100 us a round), and,
// with rows spread over warps, no longer the longest row.  Four rounds, default
// parameters, step by step -> here: Chung-Lu graphs of 1024 nodes (degree 8,
// 2 blocks) 0.66 -> 0.50 ms, 4096 (16, 8) 0.78 -> 0.61, 16384 (16, 8)
// 1.10 -> 0.98; geometric graphs of 1024, 4096 and 16384 nodes (8, 2)
// 0.61 -> 0.38, 0.68 -> 0.46 and 0.72 -> 0.51.
#pragma once

#include "rebalance_team.cuh"
#include "select_team.cuh"
#include "sequence_team.cuh"

namespace upr {
namespace {

// Rows of very different lengths, spread evenly: item i of [b, e) has the
// adjacency row of node(i) (negative: none).  A warp takes an item's row unless
// it is longer than kLongRow; those are noted, and the CTA's warps then take
// 128 entries of them each in turn.  part(i, e0, e1, whole) is called by a whole
// warp.  Rows of hubs (degree > kHubDegree) are left to the chunk loops.  With
// a warp per row whatever its length, 1024 nodes of mean degree 128 took
// 0.75 ms for four rounds, 0.54 with long rows spread.
constexpr int kLongRow = 512, kLongMax = 256;

struct LongRows {
    int cnt, item[kLongMax];
};
__device__ __forceinline__ LongRows &long_rows() {   // one array for all the loops
    __shared__ LongRows s_long;
    return s_long;
}

template <class Node, class Part>
__device__ __forceinline__ void for_rows(const GraphDev &g, int64_t b, int64_t e, Node node, Part part) {
    LongRows &rows = long_rows();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) rows.cnt = 0;
    __syncthreads();
    for (int64_t i = b + (blockIdx.x * team::kTW + warp); i < e; i += gridDim.x * team::kTW) {
        const int32_t v = node(i);
        const int64_t e0 = g.xadj[v], e1 = g.xadj[v + 1];
        if (e1 - e0 > kHubDegree) continue;
        if (e1 - e0 > kLongRow) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&rows.cnt, 1);
            at = __shfl_sync(0xffffffffu, at, 0);
            if (at < kLongMax) {
                if (lane == 0) rows.item[at] = (int)i;
                continue;
            }
        }
        part(i, e0, e1, true);
    }
    __syncthreads();
    const int cnt = min(rows.cnt, kLongMax);
    for (int j = 0; j < cnt; j++) {
        const int64_t i = rows.item[j];
        const int32_t v = node(i);
        const int64_t e0 = g.xadj[v], e1 = g.xadj[v + 1];
        for (int64_t q = e0 + 128 * warp; q < e1; q += 128 * team::kTW) part(i, q, min(q + 128, e1), false);
    }
    __syncthreads();
}

// W[u][from] -= w, W[u][to] += w for the neighbours u of the nodes i in
// [b, e) of a move list, four entries in flight per lane.
__device__ __forceinline__ void move_rows(const SmallRefine &a, const int32_t *nodes, const int32_t *from,
                                          const int32_t *to, int64_t b, int64_t e) {
    const GraphDev &g = a.g;
    const int lane = threadIdx.x & 31;
    for_rows(g, b, e, [&](int64_t i) { return nodes[i]; },
             [&](int64_t i, int64_t e0, int64_t e1, bool) {
                 const int32_t x = from[i], y = to[i];
                 for (int64_t q = e0 + lane; q < e1; q += 128) {
                     int32_t u[4], w[4];
#pragma unroll
                     for (int r = 0; r < 4; r++) {
                         u[r] = q + 32 * r < e1 ? g.adj[q + 32 * r] : -1;
                         w[r] = u[r] >= 0 ? (g.adjw ? g.adjw[q + 32 * r] : 1) : 0;
                     }
#pragma unroll
                     for (int r = 0; r < 4; r++) {
                         if (u[r] < 0) continue;
                         int32_t *row = a.W + (int64_t)u[r] * g.k;
                         atomicSub(&row[x], w[r]);
                         atomicAdd(&row[y], w[r]);
                     }
                 }
             });
}

// The same for moved hubs, a CTA per chunk: moved(v, &from, &to).
template <class Moved>
__device__ __forceinline__ void hub_rows(const SmallRefine &a, Moved moved) {
    const GraphDev &g = a.g;
    for (int64_t c = blockIdx.x; c < a.n_chunks; c += gridDim.x) {
        const HubChunk ch = a.chunks[c];
        int32_t x, y;
        if (!moved(ch.v, &x, &y)) continue;
        for (int64_t q = ch.begin + threadIdx.x; q < ch.end; q += team::kTT) {
            int32_t *row = a.W + (int64_t)g.adj[q] * g.k;
            const int32_t w = g.adjw ? g.adjw[q] : 1;
            atomicSub(&row[x], w);
            atomicAdd(&row[y], w);
        }
    }
}

// W = W(part0).
__device__ __forceinline__ void build_table(const SmallRefine &a) {
    const GraphDev &g = a.g;
    const int32_t *part = a.np.part0;
    const int lane = threadIdx.x & 31;
    UPR_TEAM_FOR(i, g.n * g.k) a.W[i] = 0;
    team::sync(a.team);
    for_rows(g, 0, g.n, [](int64_t v) { return (int32_t)v; },
             [&](int64_t v, int64_t e0, int64_t e1, bool) {
                 int32_t *row = a.W + v * g.k;
                 for (int64_t q = e0 + lane; q < e1; q += 128) {
                     int32_t p[4], w[4];
#pragma unroll
                     for (int r = 0; r < 4; r++) {
                         const int64_t x = q + 32 * r;
                         p[r] = x < e1 ? part[g.adj[x]] : -1;
                         w[r] = x < e1 && g.adjw ? g.adjw[x] : 1;
                     }
#pragma unroll
                     for (int r = 0; r < 4; r++)
                         if (p[r] >= 0) atomicAdd(&row[p[r]], w[r]);
                 }
             });
    for (int64_t c = blockIdx.x; c < a.n_chunks; c += gridDim.x) {
        const HubChunk ch = a.chunks[c];
        int32_t *row = a.W + (int64_t)ch.v * g.k;
        for (int64_t q = ch.begin + threadIdx.x; q < ch.end; q += team::kTT)
            atomicAdd(&row[part[g.adj[q]]], g.adjw ? g.adjw[q] : 1);
    }
    team::sync(a.team);
}

// Exact gains of I (as k_gains_warp and k_gains_hub_chunks).
__device__ __forceinline__ void exact_gains(const SmallRefine &a) {
    const GraphDev &g = a.g;
    const int lane = threadIdx.x & 31;
    const int64_t nI = *a.sq.dI;
    int64_t *gain = const_cast<int64_t *>(a.sb.gain);
    auto term = [&](int64_t q, int64_t i, uint32_t x, uint32_t y) -> long long {
        const uint32_t bu = block_before(a.sq.pk[g.adj[q]], i);
        const int32_t w = g.adjw ? g.adjw[q] : 1;
        return (bu == y ? w : 0) - (bu == x ? w : 0);
    };
    UPR_TEAM_FOR(i, nI) gain[i] = 0;          // (long and hub rows add their parts)
    team::sync(a.team);
    for_rows(g, 0, nI, [&](int64_t i) { return a.sq.I_node[i]; },
             [&](int64_t i, int64_t e0, int64_t e1, bool whole) {
                 const uint32_t x = (uint32_t)a.sq.I_from[i], y = (uint32_t)a.sq.I_to[i];
                 long long acc = 0;
                 for (int64_t q = e0 + lane; q < e1; q += 128) {
#pragma unroll
                     for (int r = 0; r < 4; r++)
                         if (q + 32 * r < e1) acc += term(q + 32 * r, i, x, y);
                 }
                 acc = warp_sum(acc);
                 if (lane != 0) return;
                 if (whole) gain[i] = acc;
                 else if (acc) atomicAdd(reinterpret_cast<unsigned long long *>(&gain[i]), (unsigned long long)acc);
             });
    team::sync(a.team);
    if (a.n_chunks == 0) return;
    for (int64_t c = blockIdx.x; c < a.n_chunks; c += gridDim.x) {
        const HubChunk ch = a.chunks[c];
        const int2 me = a.sq.pk[ch.v];
        if (me.x == INT32_MAX) continue;
        const uint32_t x = (uint32_t)me.y & 0xffffu, y = (uint32_t)me.y >> 16;
        long long acc = 0;
        for (int64_t q = ch.begin + threadIdx.x; q < ch.end; q += team::kTT) acc += term(q, me.x, x, y);
        acc = warp_sum(acc);
        if (lane == 0 && acc) atomicAdd(reinterpret_cast<unsigned long long *>(&gain[me.x]), (unsigned long long)acc);
    }
    team::sync(a.team);
}

template <bool UNIT, bool RANK>
__global__ void __launch_bounds__(team::kTT, 1) k_small_refine(const __grid_constant__ SmallRefine a) {
    __shared__ team::ClusterSmem s;
    extern __shared__ unsigned long long s_dyn[];
    const Team &t = a.team;
    const GraphDev &g = a.g;
    const int K = g.k;
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    long long ns[4] = {0, 0, 0, 0}, last = 0;
    auto lap = [&](int phase) {
        if (!first) return;
        long long now;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
        if (phase >= 0) ns[phase] += now - last;
        last = now;
    };
    lap(-1);
    if (a.build) build_table(a);
    lap(0);
    long long sum[6] = {0, 0, 0, 0, 0, 0}, infeasible = 0;
    for (int32_t r = 0; r < a.rounds; r++) {
        // ---- selection and M
        UPR_TEAM_FOR(i, K * kSlots) a.np.BW[i] = 0;
        team::sync(t);
        node_pass_body(a.np, r == 0 && a.np.cut_pending, s, s_dyn);
        team::sync(t);
        Penalty pen = a.so.pen;
        pen.F = a.F + (int64_t)r * kSlots;
        if (K >= 16) select_rows<8, team::kTT>(g, a.so.nl, a.np.part0, a.W, pen, a.so.cand);
        else select_rows<2, team::kTT>(g, a.so.nl, a.np.part0, a.W, pen, a.so.cand);
        team::sync(t);
        sel_order_body<team::Item32>(a.so, pen, s);
        team::sync(t);
        move_rows(a, a.so.M_node, a.so.M_from, a.so.M_to, 0, *a.so.d_moves);
        hub_rows(a, [&](int32_t v, int32_t *x, int32_t *y) {
            const int32_t p = a.so.m_pos[v];
            if (p < 0) return false;
            *x = a.so.M_from[p];
            *y = a.so.M_to[p];
            return true;
        });
        lap(1);
        // ---- rebalancing (the loop's state is in *ctl, which CTA 0 alone changes, between barriers)
        reb_start_body(a.rs, s);
        team::sync(t);
        while (*(volatile const int32_t *)&a.ctl->active) {
            const int64_t n1 = *(volatile const int32_t *)&a.ctl->n1_active;
            int32_t *tgt = const_cast<int32_t *>(a.rt.prop_tgt);
            if (K >= 16)
                propose_rows<8, team::kTT>(g, a.rt.list, n1, a.rt.part, a.W, a.st, tgt, a.prop_gain, a.flags);
            else
                propose_rows<2, team::kTT>(g, a.rt.list, n1, a.rt.part, a.W, a.st, tgt, a.prop_gain, a.flags);
            team::sync(t);
            const Appended app = reb_team_body<UNIT, RANK, false>(a.rt, s, s_dyn);
            team::sync(t);
            move_rows(a, a.rt.R_node, a.rt.R_from, a.rt.R_to, app.first, app.first + app.count);
            hub_rows(a, [&](int32_t v, int32_t *x, int32_t *y) {
                if (a.rt.r_to[v] < 0) return false;
                const int64_t p = a.rt.r_at[v];
                if (p < app.first || p >= app.first + app.count) return false;
                *x = a.rt.R_from[p];
                *y = a.rt.R_to[p];
                return true;
            });
            if (blockIdx.x == 0)
                end_subround(a.rs.C, a.rs.Lb, K, a.rs.excl, a.rs.reject, a.rs.over, a.rt.d_na, a.rt.d_np,
                             a.rs.max_subrounds, a.ctl, 0);
            team::sync(t);
        }
        lap(2);
        // ---- the sequence, its exact gains, the best prefix, the table of the next round
        seq_build_body(a.sq, s);
        team::sync(t);
        exact_gains(a);
        if (first) {
            sum[0] += *a.so.d_cand;
            sum[1] += *a.so.d_moves;
            sum[2] += a.ctl->nR;
            sum[3] += a.ctl->subrounds;
            sum[4] += *a.sq.dI;
        }
        seq_best_body(a.sb, s);
        team::sync(t);
        const int64_t kept = max(0ll, *(volatile const long long *)&a.sb.best[1]);
        if (first) {
            sum[5] += kept;
            infeasible += *(volatile const long long *)&a.sb.best[1] < 0;
        }
        move_rows(a, a.sq.I_node, a.sq.I_to, a.sq.I_from, kept, *a.sq.dI);
        hub_rows(a, [&](int32_t v, int32_t *x, int32_t *y) {
            const int32_t i = a.sq.pk[v].x;
            if (i == INT32_MAX || i < kept) return false;
            *x = a.sq.I_to[i];
            *y = a.sq.I_from[i];
            return true;
        });
        team::sync(t);
        lap(3);
    }
    if (first) {
        for (int i = 0; i < 6; i++) a.d[i] = sum[i];
        a.d[6] = 0;
        a.d[7] = infeasible;
        for (int i = 0; i < 4; i++) a.d[10 + i] = ns[i];
    }
    team::sync(t);        // no CTA leaves while another may still read its totals
}

}  // namespace

template <bool UNIT, bool RANK>
void small_form(SmallRefine a, cudaStream_t s) {
    size_t shm = node_pass_args(a.g, a.np, a.W, dynamic_smem((const void *)k_small_refine<UNIT, RANK>));
    select_order_args(a.g, a.so);
    rebalance_start_args(a.g, a.rs);
    shm = std::max(shm, rebalance_order_args(a.g, a.rt));
    seq_build_args(a.g, a.sq);
    seq_best_args(a.g, a.sb);
    launch_team(k_small_refine<UNIT, RANK>, a, a.team.size, s, shm);
}

}  // namespace upr
