// Step (b) in team launches (team.cuh): the node pass and the ordering of the
// candidates and of M, as device functions for the kernels of select.cu and the
// one-launch refinement of small graphs.
#pragma once

#include "team.cuh"

namespace upr {
namespace {

// (3/2)^s * c >= omega, exactly (p3 = the powers of 3, in shared memory).
__device__ __forceinline__ bool slot_ok(int s, uint64_t omega, uint64_t c, const uint64_t *p3) {
    if (s >= 0) return (u128)p3[s] * c >= ((u128)omega << s);
    return ((u128)c << (-s)) >= (u128)p3[-s] * omega;
}

// Smallest s in [kSlotLo, kSlotHi] with (3/2)^s >= omega / c (kSlotHi if none).
// A single-precision logarithm gives a first guess; the exact test, monotone
// in s, then moves it to the answer (one or two tests in practice).
__device__ __forceinline__ int slot_of(uint64_t omega, uint64_t c, const uint64_t *p3) {
    if (omega == 0) return kSlotLo;
    const float guess = (log2f((float)omega) - log2f((float)c)) * 1.7095113f;   // 1 / log2(3/2)
    int s = guess > (float)kSlotHi ? kSlotHi : guess < (float)kSlotLo ? kSlotLo : (int)ceilf(guess);
    while (s > kSlotLo && slot_ok(s - 1, omega, c, p3)) s--;
    while (s < kSlotHi && !slot_ok(s, omega, c, p3)) s++;
    return s;
}

// Penalty of moving weight cu into block b that would then exceed L_max by x;
// -1 = forbidden (no slot's cumulative weight covers x).
// An excess of exactly 1 (every overfilling move of a unit-weight node) takes
// the block's first non-empty slot without a search.
__device__ __forceinline__ int64_t penalty(const Penalty &p, int32_t b, int64_t x, int64_t cu) {
    if (x <= 0) return 0;
    int lo;
    if (x == 1) {
        lo = p.first[b];
        if (lo < 0) return -1;
    } else {
        const int64_t *row = p.PW + (int64_t)b * kSlots;
        if (row[kSlots - 1] < x) return -1;
        lo = 0;
        int hi = kSlots - 1;
        while (lo < hi) {
            int mid = (lo + hi) >> 1;
            if (row[mid] >= x) hi = mid; else lo = mid + 1;
        }
    }
    return (int64_t)(((u128)(uint64_t)cu * (uint64_t)p.F[lo]) >> kQ);
}

// (b1) in one team launch: availability, slots and bucket weights of every
// node, the bucket prefixes, the round-start cut when it is still unknown (the
// sum over the nodes of omega(I(v)) - omega(v, V_P(v)) is twice the cut, Sec.
// 2), and the list of the boundary nodes in node order, which the selection
// and the ordering work on (a node with all its neighbours in its own block
// has no block to move to).  The working partition and block weights start
// from the round's.  Bound by the gather of one table sector per node, four
// in flight per thread; 1024 threads share one histogram, where 256-thread
// CTAs fitted the weighted one of K = 256 (149 KB) only once per SM and took
// 298 us for 2^22 nodes with hashed rows.
constexpr int kSlotTable = 1024;

template <class Sm>
__device__ __forceinline__ void node_pass_body(const NodePass &a, bool cut_pending, Sm &s,
                                               unsigned long long *s_bw) {
    __shared__ uint64_t s_p3[41];                // 3^i (3^40 < 2^64)
    const Team &t = a.team;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int64_t n = a.n;
    const int bins = a.K * kSlots;
    unsigned int *s_bw32 = reinterpret_cast<unsigned int *>(s_bw);
    if (threadIdx.x < 41) {
        uint64_t p = 1;
        for (int i = 0; i < (int)threadIdx.x; i++) p *= 3;
        s_p3[threadIdx.x] = p;
    }
    // unit weights: the slots of the small omegas, computed once a CTA
    __shared__ int8_t s_slot[kSlotTable];
    if (!a.vwgt) {
        __syncthreads();
        for (int i = threadIdx.x; i < kSlotTable; i += team::kTT) s_slot[i] = (int8_t)slot_of((uint64_t)i, 1, s_p3);
    }
    if (a.use_shared)
        for (int i = threadIdx.x; i < (a.vwgt ? 2 : 1) * bins; i += team::kTT) s_bw32[i] = 0;
    UPR_TEAM_FOR(b, a.K) a.C[b] = a.C0[b];
    __syncthreads();
    const team::Seg g = team::warp_seg(n);
    long long cnt = 0, out_w = 0;      // boundary nodes; weight of the edges that leave the nodes' blocks
    int32_t cur = -1;                  // a batch: the graph out_w belongs to
    auto flush_cut = [&]() {
        out_w = warp_sum(out_w);
        if (lane == 0 && cur >= 0 && out_w) atomicAdd(reinterpret_cast<unsigned long long *>(&a.cut[cur]),
                                                      (unsigned long long)out_w);
        out_w = 0;
    };
    for (int64_t b0 = g.b; b0 < g.e; b0 += 128) {
        int32_t p[4], wi[4];
        int64_t own[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int64_t v = b0 + 32 * j + lane;
            p[j] = v < g.e ? a.part0[v] : 0;
            wi[j] = v < g.e ? a.wI[v] : 0;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int64_t v = b0 + 32 * j + lane;
            // an isolated node's row is zero: no gather
            own[j] = wi[j] == 0 ? 0
                     : a.sp.on() ? sp_get(a.sp, v, blk_local(p[j], a.k, a.kmask))
                                 : a.W[v * (int64_t)a.k + blk_local(p[j], a.k, a.kmask)];
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            if (b0 + 32 * j >= g.e) break;
            const int64_t v = b0 + 32 * j + lane;
            const bool in = v < g.e;
            if (in) {
                const int64_t c = a.vwgt ? a.vwgt[v] : 1;
                const bool av = (int64_t)a.t_den * own[j] >= (int64_t)a.t_num * (int64_t)wi[j];
                const int sl = !a.vwgt && own[j] < kSlotTable ? s_slot[own[j]]
                                                              : slot_of((uint64_t)own[j], (uint64_t)c, s_p3);
                if (av) {
                    const int at = p[j] * kSlots + (sl - kSlotLo);
                    if (!a.use_shared) atomicAdd(&a.BW[at], (unsigned long long)c);
                    else if (!a.vwgt) atomicAdd(&s_bw32[at], 1u);      // (a CTA's counts fit 32 bits)
                    else {       // 32-bit words with a carry: shared memory has no native 64-bit add
                        const unsigned int w = (unsigned int)c, old = atomicAdd(&s_bw32[2 * at], w);
                        if (old + w < old) atomicAdd(&s_bw32[2 * at + 1], 1u);
                    }
                }
                a.part[v] = p[j];
                a.own[v] = (int32_t)own[j];
                if (a.avail_out) a.avail_out[v] = av ? 1 : 0;
                if (a.slot_out) a.slot_out[v] = sl;
            }
            cnt += __popc(__ballot_sync(full, in && own[j] < wi[j]));
            const long long w = in ? (long long)wi[j] - own[j] : 0;
            if (!cut_pending || !a.gid) {
                out_w += w;
            } else {
                // nodes of one graph are contiguous: the warp keeps a running
                // sum until its graph changes
                const int32_t gi = in ? a.gid[v] : -1;
                const int32_t g0 = __shfl_sync(full, gi, 0);
                if (!__all_sync(full, gi == cur || gi < 0)) {
                    flush_cut();
                    cur = g0;
                    if (!__all_sync(full, gi == cur || gi < 0)) {       // several graphs in these 32 nodes
                        if (gi >= 0 && w) atomicAdd(reinterpret_cast<unsigned long long *>(&a.cut[gi]),
                                                    (unsigned long long)w);
                        continue;
                    }
                }
                out_w += w;
            }
        }
    }
    if (cut_pending && a.gid) flush_cut();
    const long long mine = team::publish<team::Sum>(t, s, 0, cnt);
    team::publish<team::Sum>(t, s, 1, team::warp_all<team::Sum>(out_w));     // (CTA barriers: the histogram is complete)
    if (a.use_shared)
        for (int i = threadIdx.x; i < bins; i += team::kTT) {
            const unsigned long long w = a.vwgt ? s_bw[i] : s_bw32[i];
            if (w) atomicAdd(&a.BW[i], w);
        }
    team::sync(t);
    long long all;
    int64_t pos = team::collect<team::Sum>(t, s, 0, &all) + mine;
    for (int64_t v0 = g.b; v0 < g.e; v0 += 32) {
        const int64_t v = v0 + lane;
        const bool f = v < g.e && a.own[v] < a.wI[v];
        const unsigned m = __ballot_sync(full, f);
        if (f) a.list[pos + __popc(m & ((1u << lane) - 1u))] = (int32_t)v;
        pos += __popc(m);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_list = (int32_t)all;
    if (cut_pending) {
        if (!a.gid) {
            long long twice;
            team::collect<team::Sum>(t, s, 1, &twice);
            if (blockIdx.x == 0 && threadIdx.x == 0) a.cut[0] = a.cut_in[0] = twice / 2;
        } else {
            UPR_TEAM_FOR(i, a.ng) a.cut[i] = a.cut_in[i] = a.cut[i] / 2;
        }
    }
    // the buckets' prefixes, a warp per block
    for (int64_t b = blockIdx.x * team::kTW + (threadIdx.x >> 5); b < a.K; b += (int64_t)gridDim.x * team::kTW) {
        long long run = 0;
        int first = -1;
        for (int l0 = 0; l0 < kSlots; l0 += 32) {
            const int l = l0 + lane;
            const long long inc = run + team::warp_incl<team::Sum>(l < kSlots ? (long long)a.BW[b * kSlots + l] : 0);
            if (l < kSlots) a.PW[b * kSlots + l] = inc;
            const unsigned some = __ballot_sync(full, l < kSlots && inc >= 1);
            if (first < 0 && some) first = l0 + __ffs(some) - 1;
            run = __shfl_sync(full, inc, 31);
        }
        if (lane == 0) a.first[b] = (int8_t)first;
    }
}

// Selection over a list, by CTAs of THREADS threads, G lanes per node: best
// target by (gain - penalty) among adjacent blocks, ties to the smaller block
// id; candidate iff the score is positive and v is a boundary node.
template <int G, int THREADS>
__device__ __forceinline__ void select_rows(const GraphDev &g, NodeList nl, const int32_t *__restrict__ part,
                                            const int32_t *__restrict__ W, const Penalty &pen, Candidates out) {
    const int64_t n = *nl.d_n;
    const int32_t k = g.k;
    constexpr int kGroups = THREADS / G;
    const int gid = threadIdx.x / G, gl = threadIdx.x % G;
    for (int64_t base = (int64_t)blockIdx.x * kGroups; base < n; base += (int64_t)gridDim.x * kGroups) {
        const int64_t i = base + gid;
        const bool active = i < n;
        const int64_t v = active ? nl.node[i] : 0;
        int64_t best = 0;
        int32_t bt = -1, bg = 0, b0 = 0;
        if (active) {
            const int32_t ag = part[v];
            const int32_t a = blk_local(g, ag);
            b0 = ag - a;
            const int32_t *row = W + v * (int64_t)k;
            const int32_t own = row[a];
            if (own < g.wI[v]) {
                const int64_t c = g.vwgt ? g.vwgt[v] : 1;
                for (int b = gl; b < k; b += G) {
                    const int32_t w = row[b];
                    if (b == a || w <= own) continue;         // (a gain of 0 or less is never a candidate's)
                    const int64_t gain = (int64_t)w - own;
                    const int32_t gb = b0 + b;
                    const int64_t p = penalty(pen, gb, pen.C[gb] + c - pen.Lb[gb], c);
                    if (p < 0) continue;
                    const int64_t sc = gain - p;
                    if (bt < 0 || sc > best) { best = sc; bt = b; bg = (int32_t)gain; }
                }
            }
        }
        int64_t s = best;
        int32_t id = bt;
        group_argmax<G>(s, id);
        // lanes own disjoint blocks, so exactly one lane holds the winner's gain
        const int32_t gsel = group_sum<G>((id >= 0 && bt == id) ? bg : 0);
        if (active && gl == 0) {
            const bool cand = id >= 0 && s > 0;
            out.tgt[i] = cand ? b0 + id : -1;
            out.s0[i] = cand ? (int32_t)s : 0;
            out.gain[i] = cand ? gsel : 0;
        }
    }
}

// ---- (b3) in one team launch: the candidates ordered by (target, score
// desc, id), the penalties with the inflow of better-ranked candidates, M
// ordered by (score desc, id) and applied.  One launch replaces about thirty
// (keys, radix passes of three launches each, scans, compactions), each 3 to
// 10 us for lists of 10^4 to 10^6 nodes, nearly all of it latency.
// Keys hold (largest - score), so their width follows the largest score that
// occurs, not the largest omega(I(v)): power-law graphs sort in two 8-bit
// passes where the bound asks for three.  The node's index in the boundary
// list is the sort's value and the kept scores go to an array by that index,
// so nothing is compacted.
template <class Item, class Sm>
__device__ __forceinline__ void sel_order_body(const SelOrder &a, const Penalty &pen, Sm &s) {
    const Team &t = a.team;
    const int lane = threadIdx.x & 31;
    const int64_t n = *a.nl.d_n;
    const Candidates &cd = a.cand;
    // the candidates' largest score
    uint32_t mx = 0;
    UPR_TEAM_FOR(i, n) {
        a.score[i] = 0;
        mx = max(mx, (uint32_t)cd.s0[i]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.deg_sum = 0;
    team::publish<team::Max>(t, s, 0, team::warp_all<team::Max>(mx));
    team::sync(t);
    long long top;
    team::collect<team::Max>(t, s, 0, &top);
    const int sbits = top > 0 ? team::bits_of((uint32_t)top - 1) : 0;
    using Key = typename Item::Key;
    int64_t cand;
    Item *bufA = reinterpret_cast<Item *>(a.bufA), *bufB = reinterpret_cast<Item *>(a.bufB);
    const Item *S = team::sort(
        t, s, n,
        [&](int64_t i, Item &it) {
            const int32_t tgt = cd.tgt[i], s0 = cd.s0[i];
            it.key = ((Key)tgt << sbits) | (Key)((uint32_t)top - (uint32_t)s0);
            it.val = (uint32_t)i;
            return tgt >= 0;
        },
        sbits + a.kbits, bufA, bufB, &cand);
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_cand = (int32_t)cand;

    // weight of the better-ranked candidates of the same target: the position
    // in the target's run with unit weights, a difference of prefix sums else
    const team::Seg g = team::warp_seg(cand);
    long long base = 0;
    if (a.vwgt) {
        long long x = 0;
        for (int64_t j = g.b + lane; j < g.e; j += 32) x += a.vwgt[a.nl.node[S[j].val]];
        const long long mine = team::publish<team::Sum>(t, s, 1, team::warp_all<team::Sum>(x));
        team::sync(t);
        long long all;
        base = team::collect<team::Sum>(t, s, 1, &all) + mine;
    }
    for (int64_t j0 = g.b; j0 < g.e; j0 += 32) {
        const int64_t j = j0 + lane;
        long long pre = j;
        if (a.vwgt) {
            const long long c = j < g.e ? a.vwgt[a.nl.node[S[j].val]] : 0;
            const long long inc = team::warp_incl<team::Sum>(c);
            pre = base + inc - c;
            base += __shfl_sync(0xffffffffu, inc, 31);
            if (j < g.e) a.c_excl[j] = pre;
        }
        if (j < g.e) {
            const Key tg = S[j].key >> sbits;
            if (j == 0 || (S[j - 1].key >> sbits) != tg) a.seg_base[tg] = pre;
        }
    }
    team::sync(t);
    uint32_t kept_top = 0;
    for (int64_t j0 = g.b + lane; j0 < g.e; j0 += 128) {
        Item it[4];
        int32_t gain[4];
        int64_t c[4], room[4], inflow[4];
#pragma unroll
        for (int r = 0; r < 4; r++)
            if (j0 + 32 * r < g.e) it[r] = S[j0 + 32 * r];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int64_t j = j0 + 32 * r;
            if (j >= g.e) continue;
            const int32_t tg = (int32_t)(it[r].key >> sbits);
            gain[r] = cd.gain[it[r].val];
            c[r] = a.vwgt ? a.vwgt[a.nl.node[it[r].val]] : 1;
            inflow[r] = (a.vwgt ? a.c_excl[j] : j) - a.seg_base[tg];
            room[r] = pen.Lb[tg] - pen.C[tg];
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            if (j0 + 32 * r >= g.e) continue;
            const int64_t p = penalty(pen, (int32_t)(it[r].key >> sbits), inflow[r] + c[r] - room[r], c[r]);
            const int64_t sc = (int64_t)gain[r] - p;
            if (p >= 0 && sc > 0) {
                a.score[it[r].val] = (int32_t)sc;
                kept_top = max(kept_top, (uint32_t)sc);
            }
        }
    }
    team::publish<team::Max>(t, s, 2, team::warp_all<team::Max>(kept_top));
    team::sync(t);
    long long ktop;
    team::collect<team::Max>(t, s, 2, &ktop);

    // M by (score desc, node id), applied
    int64_t cnt;
    using team::Item32;
    const Item32 *M = team::sort(
        t, s, n,
        [&](int64_t i, Item32 &it) {
            const int32_t sc = a.score[i];
            it.key = (uint32_t)ktop - (uint32_t)sc;
            it.val = (uint32_t)i;
            return sc > 0;
        },
        ktop > 0 ? team::bits_of((uint32_t)ktop - 1) : 0, reinterpret_cast<Item32 *>(a.bufA),
        reinterpret_cast<Item32 *>(a.bufB), &cnt);
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_moves = (int32_t)cnt;
    BlockDelta bd = make_block_delta(s.cnt64, a.K, reinterpret_cast<unsigned long long *>(a.C));
    bd.init();
    long long degs = 0;
    const team::Seg gm = team::warp_seg(cnt);
    for (int64_t p0 = gm.b; p0 < gm.e; p0 += 32) {
        const int64_t p = p0 + lane;
        int32_t from = -1, to = -1;
        long long c = 0;
        if (p < gm.e) {
            const Item32 it = M[p];
            const int32_t v = a.nl.node[it.val];
            from = a.part0[v];
            to = cd.tgt[it.val];
            c = a.vwgt ? a.vwgt[v] : 1;
            a.M_node[p] = v;
            a.M_from[p] = from;
            a.M_to[p] = to;
            a.M_score[p] = (int64_t)((uint32_t)ktop - it.key);
            a.m_pos[v] = (int32_t)p;
            a.part[v] = to;
            degs += a.xadj[v + 1] - a.xadj[v];
        }
        bd.add(from, -c);
        bd.add(to, c);
    }
    bd.flush(reinterpret_cast<unsigned long long *>(a.C));
    degs = warp_sum(degs);
    if (lane == 0 && degs) atomicAdd(reinterpret_cast<unsigned long long *>(a.deg_sum), (unsigned long long)degs);
}

}  // namespace
}  // namespace upr
