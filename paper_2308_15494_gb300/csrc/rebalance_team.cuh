// Step (d) in team launches (team.cuh): the start of a round's rebalancing, a
// sub-round after its proposals and its end, as device functions for the
// kernels of rebalance.cu and the one-launch refinement of small graphs.
#pragma once

#include <type_traits>

#include "team.cuh"

namespace upr {
namespace {

// Start of the next sub-round of one graph (h = the number run so far + 1), by
// one CTA of any size: overloaded set, lightest allowed block, activity; with
// cond also the condition of a graph-resident loop, "this sub-round runs".
__device__ __forceinline__ void begin_subround(const int64_t *C, const int64_t *Lb, int32_t K, const int8_t *excl,
                                               int8_t *over, int8_t *reject, int32_t n1, int32_t max_subrounds,
                                               RebalCtl *ctl, cudaGraphConditionalHandle cond) {
    __shared__ long long s_bw[32];
    __shared__ int32_t s_bb[32];
    int64_t bw = 0;
    int32_t bb = -1;
    int any = 0;
    for (int b = threadIdx.x; b < K; b += blockDim.x) {
        const int64_t c = C[b];
        const bool o = c > Lb[b];
        over[b] = o ? 1 : 0;
        reject[b] = 0;
        any |= o;
        // lightest: smallest weight, ties to the smaller block
        if (!excl[b] && (bb < 0 || -c > bw)) { bw = -c; bb = b; }
    }
    any = __syncthreads_or(any);
    group_argmax<32>(bw, bb);
    if ((threadIdx.x & 31) == 0) { s_bw[threadIdx.x >> 5] = bw; s_bb[threadIdx.x >> 5] = bb; }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const bool in = threadIdx.x < blockDim.x >> 5;
    bw = in ? s_bw[threadIdx.x] : 0;
    bb = in ? s_bb[threadIdx.x] : -1;
    group_argmax<32>(bw, bb);
    if (threadIdx.x == 0) {
        const int32_t h = ctl->subrounds + 1;
        const bool run = !ctl->stopped && any && h <= max_subrounds;
        ctl->active = run ? 1 : 0;
        if (!run) ctl->stopped = 1;
        if (run) ctl->subrounds = h;
        ctl->light = bb;
        ctl->n1_active = run ? n1 : 0;
        if (cond) cudaGraphSetConditional(cond, run ? 1u : 0u);
    }
}

// End of a sub-round: targets that rejected a move are excluded from now on;
// stop when nothing was admitted and no target was newly excluded, or when no
// block is overloaded any more (the next sub-round would find nothing to do).
// One graph: the next sub-round begins in the same kernel.
__device__ __forceinline__ void end_subround(const int64_t *C, const int64_t *Lb, int32_t K, int8_t *excl,
                                             int8_t *reject, int8_t *over, const int32_t *d_na, const int32_t *d_n1,
                                             int32_t max_subrounds, RebalCtl *ctl, cudaGraphConditionalHandle cond) {
    const bool active = ctl->active != 0;
    int grew = 0, any = 0;
    if (active)
        for (int b = threadIdx.x; b < K; b += blockDim.x) {
            if (reject[b] && !excl[b]) { excl[b] = 1; grew = 1; }
            if (C[b] > Lb[b]) any = 1;
        }
    grew = __syncthreads_or(grew);
    any = __syncthreads_or(any);
    if (threadIdx.x == 0 && active) {
        const int32_t na = *d_na;
        ctl->nR += na;
        if ((na == 0 && !grew) || !any) ctl->stopped = 1;
    }
    __syncthreads();
    begin_subround(C, Lb, K, excl, over, reject, *d_n1, max_subrounds, ctl, cond);
}

// Proposals of the listed nodes in overloaded blocks, by CTAs of THREADS
// threads, G lanes per node: the best-gain block with room, else the lightest
// one.
template <int G, int THREADS>
__device__ __forceinline__ void propose_rows(const GraphDev &g, const int32_t *__restrict__ list, int64_t n1,
                                             const int32_t *__restrict__ part, const int32_t *__restrict__ W,
                                             const RebalState &st, int32_t *__restrict__ prop_tgt,
                                             int32_t *__restrict__ prop_gain, int32_t *__restrict__ flags) {
    const int32_t k = g.k;
    constexpr int kGroups = THREADS / G;
    const int gid = threadIdx.x / G, gl = threadIdx.x % G;
    for (int64_t base = (int64_t)blockIdx.x * kGroups; base < n1; base += (int64_t)gridDim.x * kGroups) {
        const int64_t i = base + gid;
        const int32_t v = i < n1 ? list[i] : 0;
        const int32_t ag = i < n1 ? part[v] : 0;
        const bool src = i < n1 && st.over[ag];
        const int32_t a = blk_local(g, ag), b0 = ag - a;
        int64_t best = 0;
        int32_t bt = -1;
        int32_t own = 0;
        int64_t c = 1;
        if (src) {
            const int32_t *row = W + (int64_t)v * k;
            own = row[a];
            c = g.vwgt ? g.vwgt[v] : 1;
            for (int b = gl; b < k; b += G) {
                const int32_t w = row[b];
                const int32_t gb = b0 + b;
                if (b == a || w <= 0 || st.excl[gb] || st.C[gb] + c > st.Lb[gb]) continue;
                const int64_t gain = (int64_t)w - own;
                if (bt < 0 || gain > best) { best = gain; bt = b; }
            }
        }
        int64_t s = best;
        int32_t id = bt;
        group_argmax<G>(s, id);
        if (i < n1 && gl == 0) {
            int32_t tgt = src && id >= 0 ? b0 + id : -1;
            int64_t gain = s;
            const int32_t light = src ? st.light[blk_graph(g, ag)] : -1;
            if (src && tgt < 0 && light >= 0 && st.C[light] + c <= st.Lb[light]) { tgt = light; gain = -(int64_t)own; }
            if (tgt >= 0) {
                prop_tgt[v] = tgt;
                prop_gain[v] = (int32_t)gain;
                if (st.lgain) { st.lgain[i] = (int32_t)gain; st.lsrc[i] = ag; }
            }
            flags[i] = tgt >= 0 ? 1 : 0;
        }
    }
}

// Ascending key = descending priority.  Class 0 (g >= 0): (2^(gb+cb) - 1) - g*c.
// Class 1 (g < 0): 2^(gb+2cb) + floor(|g| * 2^(2cb) / c), exact for c < 2^cb.
// Equal priorities give equal keys; the stable sort then keeps node order.
// The key has 1 + gb + 2cb bits; up to 63 it is one word (prio_key), above
// it the 128-bit form (prio_key_wide) is sorted as two words, low word first.
__device__ __forceinline__ uint64_t prio_key(int64_t g, uint64_t c, int gbits, int cbits) {
    const int S = 2 * cbits;
    if (g >= 0) return ((1ull << (gbits + cbits)) - 1ull) - (uint64_t)g * c;
    const uint64_t num = ((uint64_t)(-g)) << S;
    return (1ull << (gbits + S)) | (c == 1 ? num : num / c);     // unit weights need no division
}

__device__ __forceinline__ unsigned __int128 prio_key_wide(int64_t g, uint64_t c, int gbits, int cbits) {
    typedef unsigned __int128 u128;
    const int S = 2 * cbits;
    if (g >= 0) return (u128)(((1ull << (gbits + cbits)) - 1ull) - (uint64_t)g * c);     // gb + cb <= 62
    const u128 num = ((u128)(uint64_t)(-g)) << S;
    return ((u128)1 << (gbits + S)) | (c == 1 ? num : num / (u128)c);
}

// gain_only (the variant of Sec. 7.2): the priority is the gain alone, the
// key of weight 1 (g >= 0 first by g, then g < 0 by |g|: g descending).

// ---- prefilter of the proposals.  A source keeps the minimal prefix of its
// proposals (priority order) that covers its excess; that prefix is usually a
// few percent of them.  A coarse bin, non-decreasing in the key, splits each
// source's proposals into ranges: every proposal in a bin below the bin where
// the source's cumulative weight reaches the excess is in the prefix, none
// above it is, so only the proposals up to that bin need the exact ordering.
// Keeping them (in their order) and dropping the rest leaves every kept
// proposal with the same weight before it in its source's order.
// The bin of a proposal of gain g and weight c (c = 1 for the gain-only
// priority), from g and c directly so that it needs no key of any width.  It
// equals the bin of the key: class 0 keys bin by g*c (127 - g*c, larger values
// all in bin 0), class 1 keys by floor(|g| * 2^cb / c), the key's class-1
// part shifted right by cb (128 + that value, larger values all in bin 255).
__device__ __forceinline__ int prio_bin(int64_t g, uint64_t c, int cbits) {
    if (g >= 0) {
        const uint64_t v = (uint64_t)g * c;
        return 127 - (int)(v < 127ull ? v : 127ull);
    }
    const uint64_t r = (((uint64_t)(-g)) << cbits) / c;     // |g| < 2^31, cb <= 31
    return 128 + (int)(r < 127ull ? r : 127ull);
}

// ---- the ordered part of a sub-round in one team launch (team.cuh): the
// proposers compacted (they are the next sub-round's list), the prefilter, the
// kept proposals in priority order, the minimal prefix per source, the longest
// fitting prefix per target, R appended and the moves applied.
//
// The weight before a proposal in its source's (then its target's) order needs
// no sort by block when the blocks' counts fit a CTA's shared memory (RANK,
// K <= 256): every warp sums the weights per block of its segment of the
// priority order, and one barrier later walks the segment again from the sums
// of the segments before, exactly as a sort pass ranks its digits.  With more
// blocks (batches) the proposals are sorted by block, stably, instead.
// When every prefilter bin holds one key value among the kept proposals (with
// unit weights and gains of moderate size it does), sorting by the bin gives
// the key order in one pass; else the keys are sorted, less their smallest.
// Eight barriers in the common form; what bounds a sub-round is their latency
// and, in the first sub-rounds, the lists.  Per sub-round, against a kernel
// with thirteen barriers of 304 CTAs that scanned tile sums: R-MAT scale 18,
// k = 8 37 us (56 before), scale 22, k = 64 81 us (110 before).  It also stands
// for the forty launches a sub-round took with several graphs, more than 256
// blocks or some key widths (Chung-Lu n = 10^6, weights, k = 23: 6.6 -> 5.3 ms
// a refinement; 1024 graphs in one context 19.0 -> 16.4 ms).
constexpr int kHistSlots = 2048;
constexpr uint32_t kHistEmpty = 0xffffffffu;
constexpr unsigned long long kNoKey = ~0ull;
constexpr int kRankK = kRebRankK;

struct __align__(32) Item128 {
    using Key = unsigned __int128;
    unsigned __int128 key;
    uint32_t val, pad[3];
};

// The weight of this lane's group (equal digits) and of its earlier lanes.
template <bool UNIT>
__device__ __forceinline__ long long group_before(unsigned peers, long long c, long long *tot) {
    const int lane = threadIdx.x & 31;
    if (UNIT) {
        *tot = __popc(peers);
        return __popc(peers & ((1u << lane) - 1u));
    }
    long long before = 0, all = 0;
    for (unsigned m = peers; m; m &= m - 1) {
        const int l = __ffs(m) - 1;
        const long long x = __shfl_sync(peers, c, l);
        all += x;
        if (l < lane) before += x;
    }
    *tot = all;
    return before;
}

// One RANK step over the items [g.b, g.e) of this warp: visit(j, digit, before)
// for every item with digit(j) >= 0, before = the weight of the items of the
// same digit before it in the whole list.  step: 0 or 1, alternating (it picks
// the published totals' place).  One barrier inside.
template <bool UNIT, class Digit, class Weight, class Visit, class Sm>
__device__ __forceinline__ void rank_walk(const Team &t, Sm &s, void *dyn, const team::Seg &g, int K,
                                          int step, Digit digit, Weight weight, Visit visit) {
    unsigned long long *hist = t.hist64 + (int64_t)step * gridDim.x * K;
    using Row = typename std::conditional<UNIT, int, unsigned long long>::type;
    Row *rows = UNIT ? reinterpret_cast<Row *>(s.cnt()) : reinterpret_cast<Row *>(dyn);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    Row *row = rows + warp * K;
    for (int i = lane; i < K; i += 32) row[i] = 0;
    __syncwarp();
    for (int64_t j0 = g.b; j0 < g.e; j0 += 32) {
        const int64_t j = j0 + lane;
        const int d = j < g.e ? digit(j) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        long long tot;
        group_before<UNIT>(peers, UNIT || d < 0 ? 1 : weight(j), &tot);
        if (d >= 0 && (peers & lt) == 0) row[d] += (Row)tot;
        __syncwarp();
    }
    __syncthreads();
    for (int d = threadIdx.x; d < K; d += team::kTT) {
        unsigned long long run = 0;
#pragma unroll 8
        for (int w = 0; w < team::kTW; w++) {
            const Row c = rows[w * K + d];
            rows[w * K + d] = (Row)run;
            run += c;
        }
        if constexpr (Sm::kCluster) s.row64[step][d] = run;
        else hist[(int64_t)blockIdx.x * K + d] = run;
        s.rep[d] = 0;
    }
    team::sync(t);
    {
        const int d = threadIdx.x & (kRankK - 1);
        unsigned long long v = 0;
        if (d < K)
            for (int c = threadIdx.x / kRankK; c < (int)blockIdx.x; c += team::kTT / kRankK)
                if constexpr (Sm::kCluster) v += team::remote(&s.row64[step][d], c);
                else v += hist[(int64_t)c * K + d];
        if (v) atomicAdd(&s.rep[d], v);
    }
    __syncthreads();
    for (int64_t j0 = g.b; j0 < g.e; j0 += 32) {
        const int64_t j = j0 + lane;
        const int d = j < g.e ? digit(j) : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        long long tot;
        const long long in = group_before<UNIT>(peers, UNIT || d < 0 ? 1 : weight(j), &tot);
        Row at = 0;
        if (d >= 0) at = row[d];
        __syncwarp();
        if (d >= 0) {
            if ((peers & lt) == 0) row[d] = at + (Row)tot;
            visit(j, d, (int64_t)(s.rep[d] + (unsigned long long)at) + in);
        }
        __syncwarp();
    }
}

// The same by a sort (any K): the items with digit(j) >= 0 sorted by digit,
// visited in that order.
template <class Digit, class Weight, class Visit, class Sm>
__device__ __forceinline__ void sort_walk(const RebalTeam &a, Sm &s, int slot, int64_t n, Digit digit,
                                          Weight weight, Visit visit) {
    using team::Item32;
    const Team &t = a.team;
    const int lane = threadIdx.x & 31;
    int64_t cnt;
    const Item32 *S = team::sort(
        t, s, n,
        [&](int64_t j, Item32 &it) {
            const int d = digit(j);
            it.key = (uint32_t)d;
            it.val = (uint32_t)j;
            return d >= 0;
        },
        a.kbits, reinterpret_cast<Item32 *>(a.bufA), reinterpret_cast<Item32 *>(a.bufB), &cnt);
    const team::Seg g = team::warp_seg(cnt);
    long long base = 0;
    if (a.vwgt) {
        long long x = 0, all;
        for (int64_t q = g.b + lane; q < g.e; q += 32) x += weight(S[q].val);
        const long long mine = team::publish<team::Sum>(t, s, slot, team::warp_all<team::Sum>(x));
        team::sync(t);
        base = team::collect<team::Sum>(t, s, slot, &all) + mine;
    }
    for (int64_t q0 = g.b; q0 < g.e; q0 += 32) {
        const int64_t q = q0 + lane;
        long long pre = q;
        if (a.vwgt) {
            const long long c = q < g.e ? weight(S[q].val) : 0;
            const long long inc = team::warp_incl<team::Sum>(c);
            pre = base + inc - c;
            base += __shfl_sync(0xffffffffu, inc, 31);
            if (q < g.e) a.c_excl[q] = pre;
        }
        if (q < g.e && (q == 0 || S[q - 1].key != S[q].key)) a.seg_base[S[q].key] = pre;
    }
    team::sync(t);
    for (int64_t q = g.b + lane; q < g.e; q += 32) {
        const Item32 it = S[q];
        visit((int64_t)it.val, (int)it.key, (a.vwgt ? a.c_excl[q] : q) - a.seg_base[it.key]);
    }
}

struct Appended { int64_t first, count; };      // the sub-round's moves in R

template <bool UNIT, bool RANK, bool WIDE, class Sm>
__device__ __forceinline__ Appended reb_team_body(const RebalTeam &a, Sm &s, unsigned long long *s_dyn) {
    using team::Item32;
    using KeyItem = typename std::conditional<WIDE, Item128, team::Item64>::type;
    const Team &t = a.team;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;
    const int K = a.K;
    const int64_t n1 = *a.d_n1;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_na = 0;      // (until R is appended to)
    if (n1 == 0) {                           // (no sub-round runs, or nothing is listed)
        if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_np = *a.d_nk = *a.d_na = 0;
        return Appended{a.ctl->nR, 0};
    }
    auto weight_of = [&](int32_t v) -> uint64_t { return UNIT ? 1ull : (uint64_t)a.vwgt[v]; };
    auto bin_of = [&](int64_t gain, int32_t v) { return prio_bin(gain, a.gain_only ? 1ull : weight_of(v), a.cbits); };

    // ---- the proposers counted; their weight per (source, bin), summed in a
    // shared hash table first (it piles up on a few bins of each source)
    const team::Seg g1 = team::warp_seg(n1);
    {
        uint32_t *s_key = reinterpret_cast<uint32_t *>(s.cnt64);
        unsigned long long *s_val = s.cnt64 + kHistSlots / 2;
        if (a.hist) {
            for (int i = threadIdx.x; i < kHistSlots; i += team::kTT) { s_key[i] = kHistEmpty; s_val[i] = 0; }
            __syncthreads();
        }
        long long cnt = 0;
        for (int64_t i0 = g1.b; i0 < g1.e; i0 += 128) {
            bool f[4];
            uint32_t key[4];
            long long c[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int64_t i = i0 + 32 * q + lane;
                f[q] = false;
                if (i0 + 32 * q >= g1.e) break;
                f[q] = i < g1.e && a.flags[i] != 0;
                key[q] = kHistEmpty;
                c[q] = 1;
                if (a.hist && f[q]) {
                    const int32_t v = UNIT ? 0 : a.list[i];
                    c[q] = (long long)weight_of(v);
                    key[q] = (uint32_t)a.lsrc[i] * kPrioBins + bin_of(a.lgain[i], v);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if (i0 + 32 * q >= g1.e) break;
                cnt += __popc(__ballot_sync(full, f[q]));
                if (!a.hist) continue;
                const unsigned peers = __match_any_sync(full, key[q]);
                long long tot;
                group_before<UNIT>(peers, c[q], &tot);
                if (f[q] && (peers & lt) == 0) {
                    uint32_t h = (key[q] * 0x9E3779B1u) >> 21;          // 11 bits: kHistSlots
                    bool done = false;
                    for (int probe = 0; probe < 32 && !done; probe++) {
                        uint32_t at = *(volatile uint32_t *)&s_key[h];
                        if (at == kHistEmpty) {
                            at = atomicCAS(&s_key[h], kHistEmpty, key[q]);
                            if (at == kHistEmpty) at = key[q];
                        }
                        if (at == key[q]) {
                            atomicAdd(&s_val[h], (unsigned long long)tot);
                            done = true;
                        }
                        h = (h + 1) & (kHistSlots - 1);
                    }
                    if (!done) atomicAdd(&a.hist[key[q]], (unsigned long long)tot);   // crowded: straight there
                }
                __syncwarp();
            }
        }
        const long long mine = team::publish<team::Sum>(t, s, 0, cnt);         // (CTA barriers inside)
        if (a.hist)
            for (int i = threadIdx.x; i < kHistSlots; i += team::kTT)
                if (s_key[i] != kHistEmpty) atomicAdd(&a.hist[s_key[i]], s_val[i]);
        if (blockIdx.x == 0) {
            for (int i = threadIdx.x; i < kPrioBins; i += team::kTT) a.rep[i] = kNoKey;
            if (threadIdx.x == 0) *a.exact = 1;
        }
        team::sync(t);
        // ---- compacted in node order, and the cut bin of every source
        long long np;
        long long pos = team::collect<team::Sum>(t, s, 0, &np) + mine;
        for (int64_t i0 = g1.b; i0 < g1.e; i0 += 128) {
            bool f[4];
            int32_t v[4], src[4], gain[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int64_t i = i0 + 32 * q + lane;
                f[q] = i < g1.e && a.flags[i] != 0;
                if (i < g1.e) { v[q] = a.list[i]; src[q] = a.lsrc[i]; gain[q] = a.lgain[i]; }
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if (i0 + 32 * q >= g1.e) break;
                const unsigned m = __ballot_sync(full, f[q]);
                if (f[q]) {
                    const int64_t p = pos + __popc(m & lt);
                    a.list2[p] = v[q];
                    a.lsrc2[p] = src[q];
                    a.lgain2[p] = gain[q];
                }
                pos += __popc(m);
            }
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_np = (int32_t)np;
    }
    long long np;
    team::collect<team::Sum>(t, s, 0, &np);
    if (a.hist) {
        // a warp per overloaded source, eight bins per lane: the first bin
        // where the cumulative weight reaches the excess; the row is cleared
        for (int64_t b = blockIdx.x * team::kTW + (threadIdx.x >> 5); b < K; b += (int64_t)gridDim.x * team::kTW) {
            if (!a.over[b]) continue;
            unsigned long long *row = a.hist + b * kPrioBins + lane * 8;
            unsigned long long w[8], sum = 0;
#pragma unroll
            for (int i = 0; i < 8; i++) { w[i] = row[i]; row[i] = 0; sum += w[i]; }
            unsigned long long run = (unsigned long long)team::warp_incl<team::Sum>((long long)sum) - sum;
            const unsigned long long excess = (unsigned long long)(a.C[b] - a.Lb[b]);
            int first = kPrioBins - 1;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                run += w[i];
                if (run >= excess) first = min(first, lane * 8 + i);
            }
            for (int o = 16; o > 0; o >>= 1) first = min(first, __shfl_xor_sync(full, first, o));
            if (lane == 0) a.cut[b] = first;
        }
    }
    team::sync(t);

    // ---- the kept proposals in priority order.  First their bins counted for
    // a one-pass sort, and whether every bin holds one key value
    auto kept = [&](int64_t i, int32_t *v, int64_t *gain, int *bin) {
        *v = a.list2[i];
        *gain = a.lgain2[i];
        *bin = bin_of(*gain, *v);
        return !a.hist || *bin <= a.cut[a.lsrc2[i]];
    };
    auto key_weight = [&](int32_t v) { return a.gain_only ? 1ull : weight_of(v); };
    const team::Seg gp = team::warp_seg(np);
    if (threadIdx.x < kPrioBins) s.rep[threadIdx.x] = kNoKey;
    __shared__ int s_inexact;
    if (threadIdx.x == 0) s_inexact = 0;
    __syncthreads();
    unsigned long long hi = 0, lo = 0;       // largest key, and largest 2^63 - 1 - key
    team::sort_count<Item32>(
        t, s, np,
        [&](int64_t i, Item32 &it) {
            int32_t v;
            int64_t gain;
            int bin;
            const bool k = kept(i, &v, &gain, &bin);
            a.list[i] = v;
            it.key = (uint32_t)bin;
            if (!k) return false;
            if (WIDE) return true;
            const unsigned long long key = prio_key(gain, key_weight(v), a.gbits, a.cbits);
            hi = max(hi, key);
            lo = max(lo, 0x7fffffffffffffffull - key);
            unsigned long long r = *(volatile unsigned long long *)&s.rep[bin];
            if (r == kNoKey) {
                r = atomicCAS(&s.rep[bin], kNoKey, key);
                if (r == kNoKey) r = key;
            }
            if (r != key) s_inexact = 1;
            return true;
        },
        0, 8);
    team::publish<team::Max>(t, s, 1, team::warp_all<team::Max>((long long)hi));
    team::publish<team::Max>(t, s, 2, team::warp_all<team::Max>((long long)lo));
    if (!WIDE) {
        if (threadIdx.x < kPrioBins && s.rep[threadIdx.x] != kNoKey) {
            const unsigned long long r = atomicCAS(&a.rep[threadIdx.x], kNoKey, s.rep[threadIdx.x]);
            if (r != kNoKey && r != s.rep[threadIdx.x]) s_inexact = 1;
        }
        __syncthreads();
        if (threadIdx.x == 0 && s_inexact) *a.exact = 0;
    }
    team::sync(t);
    int64_t nk;
    const Item32 *S32 = nullptr;
    const KeyItem *SK = nullptr;
    if (!WIDE && *(volatile const int32_t *)a.exact != 0) {
        nk = team::sort_place<Item32>(
            t, s, np,
            [&](int64_t i, Item32 &it) {
                int32_t v;
                int64_t gain;
                int bin;
                const bool k = kept(i, &v, &gain, &bin);
                it.key = (uint32_t)bin;
                it.val = (uint32_t)v;
                return k;
            },
            0, 8, reinterpret_cast<Item32 *>(a.bufA));
        S32 = reinterpret_cast<const Item32 *>(a.bufA);
    } else {
        long long top, low;
        team::collect<team::Max>(t, s, 1, &top);
        team::collect<team::Max>(t, s, 2, &low);
        const unsigned long long kmin = WIDE ? 0 : 0x7fffffffffffffffull - (unsigned long long)low;
        const int bits = WIDE ? 1 + a.gbits + 2 * a.cbits : max(1, 64 - __clzll(top - (long long)kmin));
        SK = team::sort(
            t, s, np,
            [&](int64_t i, KeyItem &it) {
                int32_t v;
                int64_t gain;
                int bin;
                if (!kept(i, &v, &gain, &bin)) return false;
                if constexpr (WIDE) it.key = prio_key_wide(gain, key_weight(v), a.gbits, a.cbits);
                else it.key = prio_key(gain, key_weight(v), a.gbits, a.cbits) - kmin;
                it.val = (uint32_t)v;
                return true;
            },
            bits, reinterpret_cast<KeyItem *>(a.bufA), reinterpret_cast<KeyItem *>(a.bufB), &nk);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_nk = (int32_t)nk;
    const team::Seg g = team::warp_seg(nk);
    for (int64_t j = g.b + lane; j < g.e; j += 32) a.U[j] = S32 ? S32[j].val : SK[j].val;
    __syncwarp();
    if (!RANK) team::sync(t);                // (the sorts below read other segments and reuse the buffers)

    // ---- the minimal prefix per source: the weight before a proposal is
    // below the excess; at[j] = its target, or -1
    auto weight = [&](int64_t j) { return (long long)weight_of((int32_t)a.U[j]); };
    auto src_of = [&](int64_t j) { return a.part[a.U[j]]; };
    auto select = [&](int64_t j, int b, int64_t before) {
        a.at[j] = before < a.C[b] - a.Lb[b] ? a.prop_tgt[a.U[j]] : -1;
    };
    // ---- the longest fitting prefix per target
    auto tgt_of = [&](int64_t j) { return a.at[j]; };
    long long adm = 0;
    auto admit = [&](int64_t j, int b, int64_t before) {
        if (a.C[b] + before + weight(j) > a.Lb[b]) {
            a.at[j] = -1;
            a.reject[b] = 1;
        }
    };
    if constexpr (RANK) {
        rank_walk<UNIT>(t, s, s_dyn, g, K, 0, src_of, weight, select);
        rank_walk<UNIT>(t, s, s_dyn, g, K, 1, tgt_of, weight, admit);
    } else {
        sort_walk(a, s, 3, nk, src_of, weight, select);
        team::sync(t);
        sort_walk(a, s, 4, nk, tgt_of, weight, admit);
        team::sync(t);
    }
    // ---- the admitted, in priority order, appended to R and applied
    for (int64_t j = g.b + lane; j < g.e; j += 32) adm += a.at[j] >= 0;
    const long long mine = team::publish<team::Sum>(t, s, 5, team::warp_all<team::Sum>(adm));
    team::sync(t);
    long long na;
    const int64_t first = a.ctl->nR;
    int64_t pos = first + team::collect<team::Sum>(t, s, 5, &na) + mine;
    const int32_t subround = a.ctl->subrounds;
    BlockDelta bd = make_block_delta(s.cnt64, K, reinterpret_cast<unsigned long long *>(a.C));
    bd.init();
    for (int64_t j0 = g.b; j0 < g.e; j0 += 32) {
        const int64_t j = j0 + lane;
        const int32_t to = j < g.e ? a.at[j] : -1;
        const unsigned m = __ballot_sync(full, to >= 0);
        int32_t from = -1;
        long long c = 0;
        if (to >= 0) {
            const int32_t v = (int32_t)a.U[j];
            const int64_t p = pos + __popc(m & lt);
            from = a.part[v];
            c = (long long)weight_of(v);
            a.R_node[p] = v;
            a.R_from[p] = from;
            a.R_to[p] = to;
            a.R_sub[p] = subround;
            a.r_to[v] = to;
            a.r_at[v] = (int32_t)p;
            a.part[v] = to;
        }
        pos += __popc(m);
        if (m) {
            bd.add(from, -c);
            bd.add(to, c);
        }
    }
    bd.flush(reinterpret_cast<unsigned long long *>(a.C));
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_na = (int32_t)na;
    return Appended{first, na};
}

// ---- the start of a round's rebalancing: the nodes of the overloaded blocks,
// in node order, are the first list; the overloaded blocks are never targets.
// One graph (light == nullptr): CTA 0 also begins the first sub-round.
template <class Sm>
__device__ __forceinline__ void reb_start_body(const RebalStart &a, Sm &s) {
    const Team &t = a.team;
    const int lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.cond) cudaGraphSetConditional(a.cond, 0);    // (until it is known)
    const team::Seg g = team::warp_seg(a.n);
    long long cnt = 0;
    for (int64_t v = g.b + lane; v < g.e; v += 32) {
        const int32_t b = a.part[v];
        cnt += a.C[b] > a.Lb[b];
    }
    const long long mine = team::publish<team::Sum>(t, s, 0, team::warp_all<team::Sum>(cnt));
    team::sync(t);
    long long all;
    int64_t pos = team::collect<team::Sum>(t, s, 0, &all) + mine;
    for (int64_t v0 = g.b; v0 < g.e; v0 += 32) {
        const int64_t v = v0 + lane;
        bool f = false;
        if (v < g.e) {
            const int32_t b = a.part[v];
            f = a.C[b] > a.Lb[b];
        }
        const unsigned m = __ballot_sync(0xffffffffu, f);
        if (f) a.list[pos + __popc(m & ((1u << lane) - 1u))] = (int32_t)v;
        pos += __popc(m);
    }
    if (blockIdx.x != 0) return;
    if (threadIdx.x == 0) *a.d_list = (int32_t)all;
    if (a.batch) return;
    for (int b = threadIdx.x; b < a.K; b += team::kTT) a.excl[b] = a.C[b] > a.Lb[b] ? 1 : 0;
    if (threadIdx.x == 0) {
        a.ctl->stopped = 0;
        a.ctl->subrounds = 0;
        a.ctl->nR = 0;
        a.ctl->flag = 0;
        a.ctl->ticket = 0;
    }
    __syncthreads();
    begin_subround(a.C, a.Lb, a.K, a.excl, a.over, a.reject, (int32_t)all, a.max_subrounds, a.ctl, a.cond);
}

}  // namespace
}  // namespace upr
