// Step (c) in team launches (team.cuh): the move sequence and its best prefix,
// as device functions for the kernels of sequence.cu and the one-launch
// refinement of small graphs.
#pragma once

#include "team.cuh"

namespace upr {
namespace {

__device__ __forceinline__ int64_t cw(const int32_t *vwgt, int32_t v) { return vwgt ? (int64_t)vwgt[v] : 1; }

// Exact gain of the i-th move of I: neighbours moved earlier in I count in
// their new block, all others in their round-start block.  Warp per move;
// hub moves (degree > kHubDegree) are left to k_gains_hub_chunks.
// Block of each node at every step of I, packed for one 8-byte gather per
// adjacency entry: x = the node's position in I (INT32_MAX when it does not
// move), y = (local block before its move) | (local block after it) << 16.
// Before step i a neighbour u is in its later block iff x < i (k_seq_build fills it).
__device__ __forceinline__ uint32_t block_before(int2 p, int64_t i) {
    const uint32_t code = (uint32_t)p.y;
    return p.x < i ? (code >> 16) : (code & 0xffffu);
}

// best prefix: max G(j) over eligible j (ties: smallest j); G(0) = 0, eligible(0) = (over0 == 0)
struct Best { long long g; long long j; };

__device__ __forceinline__ Best better(Best x, Best y) {
    if (x.j < 0) return y;
    if (y.j < 0) return x;
    if (y.g > x.g || (y.g == x.g && y.j < x.j)) return y;
    return x;
}

// ---- (c1) in one team launch (team.cuh): X = the interleaving of M and the
// R_b (or M then R), the merged sequence I, and the packed state of every node
// for the exact gains; a batch's I also sorted by graph.  One launch replaces
// about thirty.  R's entries and M's events are sorted by block together: R
// comes first in the input, so in every block's run its R_b precedes its
// events, and one sort, one scan and one walk serve both.
constexpr uint32_t kIsR = 1u << 31;       // in a sort key: an entry of R (blocks have at most 30 bits)

__device__ __forceinline__ uint32_t blk_of(uint32_t key) { return key & ~kIsR; }

// Move (v, to) of M or R at position x of X: its fate after merging (an R move
// of a node with an M move folds into the M move; a move back to the
// round-start block is dropped).
__device__ __forceinline__ void put_x(const SeqBuild &a, int64_t x, int32_t v, int32_t from, int32_t to, bool isr) {
    a.X_node[x] = v;
    a.X_from[x] = from;
    a.X_to[x] = to;
    int32_t fin = to;
    if (isr) {
        if (a.m_pos[v] >= 0) fin = -1;
    } else {
        const int32_t r = a.r_to[v];
        if (r >= 0) fin = r;
    }
    a.fin[x] = fin == a.part0[v] ? -1 : fin;
}

template <class Sm>
__device__ __forceinline__ void seq_build_body(const SeqBuild &a, Sm &s) {
    using team::Item32;
    const Team &t = a.team;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int64_t n = a.n, nM = *a.dM, nR = *a.dR, K = a.K;
    const int64_t nX = nM + nR;
    Item32 *A = reinterpret_cast<Item32 *>(a.bufA), *B = reinterpret_cast<Item32 *>(a.bufB);
    UPR_TEAM_FOR(u, n) {
        const uint32_t l = (uint32_t)blk_local(a.part0[u], a.k, a.kmask);
        a.pk[u] = make_int2(INT32_MAX, (int32_t)(l | (l << 16)));
    }
    if (a.append || nR == 0) {
        UPR_TEAM_FOR(i, nX) {
            const bool r = i >= nM;
            const int64_t j = r ? i - nM : i;
            put_x(a, i, r ? a.R_node[j] : a.M_node[j], r ? a.R_from[j] : a.M_from[j], r ? a.R_to[j] : a.M_to[j], r);
        }
    } else {
        UPR_TEAM_FOR(b, K) a.rbeg[b] = a.rend[b] = a.ebeg[b] = a.eend[b] = 0;
        // entries of R and events of M (2i = leave M_from[i], 2i + 1 = enter M_to[i]) by block
        int64_t L;
        const Item32 *S = team::sort(
            t, s, nR + 2 * nM,
            [&](int64_t i, Item32 &it) {
                if (i < nR) {
                    it.key = (uint32_t)a.R_from[i] | kIsR;
                    it.val = (uint32_t)i;
                } else {
                    const int64_t e = i - nR;
                    it.key = (uint32_t)((e & 1) ? a.M_to[e >> 1] : a.M_from[e >> 1]);
                    it.val = (uint32_t)e;
                }
                return true;
            },
            a.kbits, A, B, &L);
        const team::Seg g = team::warp_seg(L);
        // runs of every block, and the two prefix sums: weights of R's
        // entries, weight changes of M's events (each over its own kind)
        long long sr = 0, sd = 0;
        for (int64_t j = g.b + lane; j < g.e; j += 32) {
            const Item32 it = S[j];
            const uint32_t b = blk_of(it.key);
            const uint32_t kp = j > 0 ? S[j - 1].key : ~0u, kn = j + 1 < L ? S[j + 1].key : ~0u;
            if (it.key & kIsR) {
                if (kp != it.key) a.rbeg[b] = (int32_t)j;
                if (kn != it.key) a.rend[b] = (int32_t)(j + 1);
                const long long c = cw(a.vwgt, a.R_node[it.val]);
                a.ex[j] = c;
                sr += c;
            } else {
                if (kp != it.key) a.ebeg[b] = (int32_t)j;
                if (kn != it.key) a.eend[b] = (int32_t)(j + 1);
                const long long c = cw(a.vwgt, a.M_node[it.val >> 1]);
                const long long d = (it.val & 1) ? c : -c;
                a.ex[j] = d;
                sd += d;
            }
        }
        long long all;
        const long long mr = team::publish<team::Sum>(t, s, 0, team::warp_all<team::Sum>(sr));
        const long long md = team::publish<team::Sum>(t, s, 1, team::warp_all<team::Sum>(sd));
        team::sync(t);
        sr = team::collect<team::Sum>(t, s, 0, &all) + mr;
        sd = team::collect<team::Sum>(t, s, 1, &all) + md;
        for (int64_t j0 = g.b; j0 < g.e; j0 += 32) {
            const int64_t j = j0 + lane;
            const bool ok = j < g.e;
            const bool isr = ok && (S[j].key & kIsR);
            const long long x = ok ? a.ex[j] : 0;
            const long long ir = team::warp_incl<team::Sum>(isr ? x : 0), id = team::warp_incl<team::Sum>(isr ? 0 : x);
            if (ok) a.ex[j] = isr ? sr + ir - x : sd + id - x;
            sr += __shfl_sync(full, ir, 31);
            sd += __shfl_sync(full, id, 31);
        }
        team::sync(t);
        // need of every event that enters a block with R_b non-empty; packed
        // with the block, so that the running maximum restarts at each block
        long long mx = 0;
        for (int64_t j = g.b + lane; j < g.e; j += 32) {
            const Item32 it = S[j];
            const uint32_t b = blk_of(it.key);
            uint32_t need = 0;
            if (!(it.key & kIsR) && (it.val & 1)) {
                const int32_t r0 = a.rbeg[b], r1 = a.rend[b];
                if (r1 > r0) {
                    const int64_t Lmax = a.Lb[b];
                    const int64_t D = a.C0[b] + a.ex[j] + cw(a.vwgt, a.M_node[it.val >> 1]) - a.ex[a.ebeg[b]];
                    if (D > Lmax) {
                        // smallest x in [1, |R_b|] with D - (weight of R_b[0..x)) <= L_max, else |R_b|
                        const int64_t base = a.ex[r0], over = D - Lmax;
                        int lo = 1, hi = r1 - r0;
                        if (!a.vwgt) lo = (int)min((int64_t)hi, over);      // (unit weights: x = the excess)
                        else
                            while (lo < hi) {
                                const int mid = lo + ((hi - lo) >> 1);
                                if (over <= a.ex[r0 + mid] - base) hi = mid; else lo = mid + 1;
                            }
                        need = (uint32_t)lo;
                    }
                }
            }
            a.qmax[j] = need;
            mx = max(mx, (long long)(((uint64_t)b << 32) | need));
        }
        const long long mq = team::publish<team::Max>(t, s, 2, team::warp_all<team::Max>(mx));
        team::sync(t);
        mx = max(team::collect<team::Max>(t, s, 2, &all), mq);
        for (int64_t j0 = g.b; j0 < g.e; j0 += 32) {
            const int64_t j = j0 + lane;
            const bool ok = j < g.e;
            Item32 it{0, 0};
            if (ok) it = S[j];
            const uint32_t b = blk_of(it.key);
            const long long p = ok ? (long long)(((uint64_t)b << 32) | a.qmax[j]) : 0;
            const long long inc = max(mx, team::warp_incl<team::Max>(p));
            long long prev = __shfl_up_sync(full, inc, 1);
            if (lane == 0) prev = mx;
            mx = __shfl_sync(full, inc, 31);
            if (!ok) continue;
            const uint32_t after = (uint32_t)inc;
            a.qmax[j] = after;
            if (!(it.key & kIsR) && (it.val & 1)) {
                const uint32_t before = (uint32_t)(prev >> 32) == b ? (uint32_t)prev : 0u;
                a.emit[it.val >> 1] = (int32_t)(after - before);
            }
        }
        team::sync(t);
        // emissions before every M move; per block, what is left of R_b after M
        const team::Seg gm = team::warp_seg(nM), gk = team::warp_seg(K);
        long long se = 0, sl = 0;
        for (int64_t i = gm.b + lane; i < gm.e; i += 32) se += a.emit[i];
        for (int64_t b = gk.b + lane; b < gk.e; b += 32) {
            const int32_t f = a.eend[b] > a.ebeg[b] ? (int32_t)a.qmax[a.eend[b] - 1] : 0;
            a.qfin[b] = f;
            sl += (a.rend[b] - a.rbeg[b]) - f;
        }
        const long long me = team::publish<team::Sum>(t, s, 3, team::warp_all<team::Sum>(se));
        const long long ml = team::publish<team::Sum>(t, s, 4, team::warp_all<team::Sum>(sl));
        team::sync(t);
        long long emitted;
        se = team::collect<team::Sum>(t, s, 3, &emitted) + me;
        sl = team::collect<team::Sum>(t, s, 4, &all) + ml;
        for (int64_t i0 = gm.b; i0 < gm.e; i0 += 32) {
            const int64_t i = i0 + lane;
            const long long x = i < gm.e ? a.emit[i] : 0;
            const long long inc = team::warp_incl<team::Sum>(x);
            if (i < gm.e) {
                const int64_t p = i + se + inc - x;
                a.pos_m[i] = (int32_t)p;
                put_x(a, p, a.M_node[i], a.M_from[i], a.M_to[i], false);
            }
            se += __shfl_sync(full, inc, 31);
        }
        for (int64_t b0 = gk.b; b0 < gk.e; b0 += 32) {
            const int64_t b = b0 + lane;
            const long long x = b < gk.e ? (a.rend[b] - a.rbeg[b]) - a.qfin[b] : 0;
            const long long inc = team::warp_incl<team::Sum>(x);
            if (b < gk.e) a.left_excl[b] = (int32_t)(sl + inc - x);
            sl += __shfl_sync(full, inc, 31);
        }
        team::sync(t);
        // R's entries: after the event that emits them, or behind M in block
        // order (strided over the team: they lie in runs, a few segments hold
        // them all)
        UPR_TEAM_FOR(j, L) {
            const Item32 it = S[j];
            if (!(it.key & kIsR)) continue;
            const uint32_t b = blk_of(it.key), i = it.val;
            const uint32_t r = (uint32_t)(j - a.rbeg[b]);
            int64_t p;
            if ((int32_t)r < a.qfin[b]) {
                // first event of b with running max > r (an inflow event)
                const int first = a.ebeg[b];
                int lo = first, hi = a.eend[b] - 1;
                while (lo < hi) {
                    const int mid = lo + ((hi - lo) >> 1);
                    if (a.qmax[mid] > r) hi = mid; else lo = mid + 1;
                }
                const uint32_t before = lo == first ? 0u : a.qmax[lo - 1];
                p = (int64_t)a.pos_m[S[lo].val >> 1] + 1 + (r - before);
            } else {
                p = nM + emitted + a.left_excl[b] + (r - (uint32_t)a.qfin[b]);
            }
            put_x(a, p, a.R_node[i], a.R_from[i], a.R_to[i], true);
        }
    }
    team::sync(t);
    // the moves left after merging, in order: I
    const team::Seg gx = team::warp_seg(nX);
    long long keep = 0;
    for (int64_t x = gx.b + lane; x < gx.e; x += 32) keep += a.fin[x] >= 0;
    const long long mk = team::publish<team::Sum>(t, s, 5, team::warp_all<team::Sum>(keep));
    team::sync(t);
    long long nI;
    keep = team::collect<team::Sum>(t, s, 5, &nI) + mk;
    long long deg = 0;
    for (int64_t x0 = gx.b; x0 < gx.e; x0 += 32) {
        const int64_t x = x0 + lane;
        const int32_t to = x < gx.e ? a.fin[x] : -1;
        const unsigned kept = __ballot_sync(full, to >= 0);
        if (to >= 0) {
            const int64_t i = keep + __popc(kept & ((1u << lane) - 1u));
            const int32_t v = a.X_node[x], from = a.part0[v];
            a.I_node[i] = v;
            a.I_from[i] = from;
            a.I_to[i] = to;
            if (!a.gid) {
                const uint32_t lf = (uint32_t)blk_local(from, a.k, a.kmask), lo = (uint32_t)blk_local(to, a.k, a.kmask);
                a.pk[v] = make_int2((int32_t)i, (int32_t)(lf | (lo << 16)));
            }
            deg += a.xadj[v + 1] - a.xadj[v];
        }
        keep += __popc(kept);
    }
    deg = warp_sum(deg);
    if (lane == 0 && deg) atomicAdd(reinterpret_cast<unsigned long long *>(a.deg_sum), (unsigned long long)deg);
    UPR_TEAM_FOR(j, nI + 1) a.diff[j] = 0;
    auto lengths = [&] {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            *a.dX = (int32_t)nX;
            *a.dI = (int32_t)nI;
        }
    };
    if (!a.gid) {
        lengths();
        return;
    }
    // a batch: each graph's moves contiguous, in their own order
    UPR_TEAM_FOR(g, a.ng) a.seg_beg[g] = a.seg_end[g] = 0;
    team::sync(t);
    int64_t cnt;
    const Item32 *S = team::sort(
        t, s, nI,
        [&](int64_t i, Item32 &it) {
            it.key = (uint32_t)a.gid[a.I_node[i]];
            it.val = (uint32_t)i;
            return true;
        },
        a.ngbits, A, B, &cnt);
    UPR_TEAM_FOR(q, nI) {
        const Item32 it = S[q];
        const int32_t i = (int32_t)it.val, v = a.I_node[i], from = a.I_from[i], to = a.I_to[i];
        a.O_node[q] = v;
        a.O_from[q] = from;
        a.O_to[q] = to;
        const uint32_t lf = (uint32_t)blk_local(from, a.k, a.kmask), lo = (uint32_t)blk_local(to, a.k, a.kmask);
        a.pk[v] = make_int2((int32_t)q, (int32_t)(lf | (lo << 16)));
        if (q == 0 || S[q - 1].key != it.key) a.seg_beg[it.key] = (int32_t)q;
        if (q == nI - 1 || S[q + 1].key != it.key) a.seg_end[it.key] = (int32_t)(q + 1);
    }
    lengths();
}

// ---- (c2) after the exact gains, in one team launch: prefix gains, the
// number of overloaded blocks after every move (the moves' block events sorted
// by block, a segmented sum of their weights), and for one graph the best
// balanced prefix, applied, with the degree sum of the undone moves; the
// markers of M and R go back to "none" (unless the oscillation guard still
// needs them).  Replaces about twenty launches.
struct Segd { int head; long long sum; };         // a run boundary inside, the sum since the last one
__device__ __forceinline__ Segd seg_op(Segd x, Segd y) { return Segd{x.head | y.head, y.head ? y.sum : x.sum + y.sum}; }
__device__ __forceinline__ Segd seg_incl(Segd v) {
    for (int o = 1; o < 32; o <<= 1) {
        const Segd u{__shfl_up_sync(0xffffffffu, v.head, o), __shfl_up_sync(0xffffffffu, v.sum, o)};
        if ((threadIdx.x & 31) >= o) v = seg_op(u, v);
    }
    return v;
}
__device__ __forceinline__ Segd seg_at(Segd v, int lane) {
    return Segd{__shfl_sync(0xffffffffu, v.head, lane), __shfl_sync(0xffffffffu, v.sum, lane)};
}

template <class Sm>
__device__ __forceinline__ void seq_best_body(const SeqBest &a, Sm &s) {
    using team::Item32;
    const Team &t = a.team;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu;
    const int64_t nI = *a.dI;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.undone = 0;
    if (a.reset) {
        const int64_t nM = *a.dM, nR = *a.dR;
        UPR_TEAM_FOR(i, nM) a.m_pos[a.M_node[i]] = -1;
        UPR_TEAM_FOR(i, nR) a.r_to[a.R_node[i]] = -1;
    }
    const team::Seg gi = team::warp_seg(nI);
    long long sg = 0;
    for (int64_t i = gi.b + lane; i < gi.e; i += 32) sg += a.gain[i];
    const long long mg = team::publish<team::Sum>(t, s, 0, team::warp_all<team::Sum>(sg));
    int64_t nev;
    const Item32 *S = team::sort(
        t, s, 2 * nI,
        [&](int64_t e, Item32 &it) {
            it.key = (uint32_t)((e & 1) ? a.I_to[e >> 1] : a.I_from[e >> 1]);
            it.val = (uint32_t)e;
            return true;
        },
        a.kbits, reinterpret_cast<Item32 *>(a.bufA), reinterpret_cast<Item32 *>(a.bufB), &nev);
    long long all;
    sg = team::collect<team::Sum>(t, s, 0, &all) + mg;
    for (int64_t i0 = gi.b; i0 < gi.e; i0 += 32) {
        const int64_t i = i0 + lane;
        const long long inc = team::warp_incl<team::Sum>(i < gi.e ? a.gain[i] : 0);
        if (i < gi.e) a.Gsum[i] = sg + inc;
        sg += __shfl_sync(full, inc, 31);
    }
    // the weight of every event's block before it: a segmented sum over the
    // sorted events (per warp, per CTA, then over the CTAs)
    const team::Seg g = team::warp_seg(nev);
    auto event = [&](int64_t j) {
        const Item32 it = S[j];
        const long long c = cw(a.vwgt, a.I_node[it.val >> 1]);
        return Segd{j == 0 || S[j - 1].key != it.key, (it.val & 1) ? c : -c};
    };
    Segd acc{0, 0};
    for (int64_t j0 = g.b; j0 < g.e; j0 += 32) {
        const int64_t j = j0 + lane;
        acc = seg_op(acc, seg_at(seg_incl(j < g.e ? event(j) : Segd{0, 0}), 31));
    }
    __shared__ int s_head[team::kTW];
    if (lane == 0) { s.w[warp] = acc.sum; s_head[warp] = acc.head; }
    __syncthreads();
    const Segd winc = seg_incl(Segd{s_head[lane], s.w[lane]});
    Segd mine = seg_at(winc, warp > 0 ? warp - 1 : 0);
    if (warp == 0) mine = Segd{0, 0};
    if (threadIdx.x == team::kTT - 1) {
        team::put(t, s, 1, winc.sum);
        team::put(t, s, 2, winc.head);
    }
    team::sync(t);
    Segd carry{0, 0};
    for (int c0 = 0; c0 < (int)blockIdx.x; c0 += 32) {
        const int c = c0 + lane;
        Segd x{0, 0};
        if (c < (int)blockIdx.x)
            x = Segd{(int)team::get(t, s, 2, c), team::get(t, s, 1, c)};
        carry = seg_op(carry, seg_at(seg_incl(x), 31));
    }
    carry = seg_op(carry, mine);
    for (int64_t j0 = g.b; j0 < g.e; j0 += 32) {
        const int64_t j = j0 + lane;
        const bool ok = j < g.e;
        const Segd x = ok ? event(j) : Segd{0, 0};
        const Segd inc = seg_incl(x);
        const long long after_d = inc.head ? inc.sum : carry.sum + inc.sum;
        if (ok) {
            const Item32 it = S[j];
            const int64_t Lmax = a.Lb[it.key], after = a.C0[it.key] + after_d, before = after - x.sum;
            const int d = (after > Lmax ? 1 : 0) - (before > Lmax ? 1 : 0);
            if (d) atomicAdd(&a.diff[(it.val >> 1) + 1], d);
        }
        carry = seg_op(carry, seg_at(inc, 31));
    }
    team::sync(t);
    // overloaded blocks after every prefix
    const team::Seg gj = team::warp_seg(nI + 1);
    long long so = 0;
    for (int64_t j = gj.b + lane; j < gj.e; j += 32) so += a.diff[j];
    int over0 = 0;
    if (!a.gid) {
        if (threadIdx.x == 0) s.tot[0] = 0;
        __syncthreads();
        for (int b = threadIdx.x; b < a.K; b += team::kTT)
            if (a.C0[b] > a.Lb[b]) atomicAdd(&s.tot[0], 1);
    }
    const long long mo = team::publish<team::Sum>(t, s, 3, team::warp_all<team::Sum>(so));   // (a CTA barrier)
    over0 = s.tot[0];
    team::sync(t);
    so = team::collect<team::Sum>(t, s, 3, &all) + mo;
    Best best{0, -1};
    for (int64_t j0 = gj.b; j0 < gj.e; j0 += 32) {
        const int64_t j = j0 + lane;
        const long long x = j < gj.e ? a.diff[j] : 0;
        const long long inc = team::warp_incl<team::Sum>(x);
        if (j < gj.e) {
            a.diff_excl[j] = (int32_t)(so + inc - x);
            if (!a.gid && over0 + so + inc == 0) best = better(best, Best{j == 0 ? 0 : a.Gsum[j - 1], j});
        }
        so += __shfl_sync(full, inc, 31);
    }
    if (a.gid) return;          // (a batch: per graph, in kernels of their own)
    auto warp_best = [&](Best b) {
        for (int o = 16; o > 0; o >>= 1)
            b = better(b, Best{__shfl_xor_sync(full, b.g, o), __shfl_xor_sync(full, b.j, o)});
        return b;
    };
    best = warp_best(best);
    __shared__ long long s_j[team::kTW];
    if (lane == 0) { s.w[warp] = best.g; s_j[warp] = best.j; }
    __syncthreads();
    best = warp_best(Best{s.w[lane], s_j[lane]});
    if (threadIdx.x == 0) {
        team::put(t, s, 4, best.g);
        team::put(t, s, 5, best.j);
    }
    team::sync(t);
    best = Best{0, -1};
    for (int c = lane; c < (int)gridDim.x; c += 32)
        best = better(best, Best{team::get(t, s, 4, c), team::get(t, s, 5, c)});
    best = warp_best(best);
    // the prefix applied; the degrees of the moves after it
    BlockDelta bd = make_block_delta(s.cnt64, a.K, reinterpret_cast<unsigned long long *>(a.C0));
    bd.init();
    long long degs = 0;
    for (int64_t i0 = gi.b; i0 < gi.e; i0 += 32) {
        const int64_t i = i0 + lane;
        int32_t from = -1, to = -1;
        long long c = 0;
        if (i < gi.e) {
            const int32_t v = a.I_node[i];
            if (i < best.j) {
                from = a.I_from[i];
                to = a.I_to[i];
                c = cw(a.vwgt, v);
                a.part0[v] = to;
            } else {
                degs += a.xadj[v + 1] - a.xadj[v];
            }
        }
        bd.add(from, -c);
        bd.add(to, c);
    }
    bd.flush(reinterpret_cast<unsigned long long *>(a.C0));
    degs = warp_sum(degs);
    if (lane == 0 && degs) atomicAdd(reinterpret_cast<unsigned long long *>(a.undone), (unsigned long long)degs);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.best[0] = best.g;
        a.best[1] = best.j;
        *a.d_over0 = over0;
        if (best.j < 0) *a.d_infeasible = 1;
        else *a.cut -= best.g;
    }
}

// ---- batches: I sorted by graph (stable), then per-graph segments
// [seg_beg[g], seg_end[g]) of I; G_g(j) and eligibility are differences of
// the global prefix sums taken at the segment start.

}  // namespace
}  // namespace upr
