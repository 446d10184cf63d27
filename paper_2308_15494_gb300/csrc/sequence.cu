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

__global__ void __launch_bounds__(team::kTT, 1) k_seq_build(const SeqBuild a) {
    __shared__ team::Smem s;
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
        sr = team::collect<team::Sum>(t, 0, &all) + mr;
        sd = team::collect<team::Sum>(t, 1, &all) + md;
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
        mx = max(team::collect<team::Max>(t, 2, &all), mq);
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
        se = team::collect<team::Sum>(t, 3, &emitted) + me;
        sl = team::collect<team::Sum>(t, 4, &all) + ml;
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
    keep = team::collect<team::Sum>(t, 5, &nI) + mk;
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
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.dX = (int32_t)nX;
        *a.dI = (int32_t)nI;
    }
    if (!a.gid) return;
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

__global__ void __launch_bounds__(team::kTT, 1) k_seq_best(const SeqBest a) {
    __shared__ team::Smem s;
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
    sg = team::collect<team::Sum>(t, 0, &all) + mg;
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
        t.tot[1 * team::kTeamMax + blockIdx.x] = winc.sum;
        t.tot[2 * team::kTeamMax + blockIdx.x] = winc.head;
    }
    team::sync(t);
    Segd carry{0, 0};
    for (int c0 = 0; c0 < (int)blockIdx.x; c0 += 32) {
        const int c = c0 + lane;
        Segd x{0, 0};
        if (c < (int)blockIdx.x)
            x = Segd{(int)t.tot[2 * team::kTeamMax + c], t.tot[1 * team::kTeamMax + c]};
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
    so = team::collect<team::Sum>(t, 3, &all) + mo;
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
        t.tot[4 * team::kTeamMax + blockIdx.x] = best.g;
        t.tot[5 * team::kTeamMax + blockIdx.x] = best.j;
    }
    team::sync(t);
    best = Best{0, -1};
    for (int c = lane; c < (int)gridDim.x; c += 32)
        best = better(best, Best{t.tot[4 * team::kTeamMax + c], t.tot[5 * team::kTeamMax + c]});
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

void seq_build(const GraphDev &g, SeqBuild a, cudaStream_t s) {
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

void seq_best(const GraphDev &g, SeqBest a, cudaStream_t s) {
    a.K = g.K();
    a.vwgt = g.vwgt;
    a.gid = g.gid;
    a.xadj = g.xadj;
    a.Lb = g.Lb;
    a.kbits = 1;
    while ((1ll << a.kbits) < a.K) a.kbits++;
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
