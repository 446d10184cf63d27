// Step (b): rebalancing availability, slots and bucket weights (Alg. 1,
// Sec. 4.3), each boundary node's best move by gain minus penalty
// (Alg. 1), penalties with the inflow of better-ranked candidates,
// the global move order M (Sec. 4.4), and the application of M.
#include "team.cuh"

namespace upr {
namespace {

// 3^i for i = 0..40 (3^40 < 2^64).
__constant__ uint64_t c_pow3[41];

int sm_count_sel() {
    static int cnt = 0;
    if (!cnt) {
        int dev = 0;
        UPR_CUDA(cudaGetDevice(&dev));
        UPR_CUDA(cudaDeviceGetAttribute(&cnt, cudaDevAttrMultiProcessorCount, dev));
    }
    return cnt;
}

void ensure_pow3() {
    static int done_dev = -1;
    int dev = 0;
    UPR_CUDA(cudaGetDevice(&dev));
    if (done_dev == dev) return;
    uint64_t p[41];
    p[0] = 1;
    for (int i = 1; i <= 40; i++) p[i] = p[i - 1] * 3;
    UPR_CUDA(cudaMemcpyToSymbol(c_pow3, p, sizeof(p)));
    done_dev = dev;
}

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

__global__ void __launch_bounds__(team::kTT, 1) k_node_pass(const NodePass a) {
    __shared__ team::Smem s;
    __shared__ uint64_t s_p3[41];
    extern __shared__ unsigned long long s_bw[];
    const Team &t = a.team;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const int64_t n = a.n;
    const int bins = a.K * kSlots;
    unsigned int *s_bw32 = reinterpret_cast<unsigned int *>(s_bw);
    for (int i = threadIdx.x; i < 41; i += team::kTT) s_p3[i] = c_pow3[i];
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
            if (!a.cut_pending || !a.gid) {
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
    if (a.cut_pending && a.gid) flush_cut();
    const long long mine = team::publish<team::Sum>(t, s, 0, cnt);
    team::publish<team::Sum>(t, s, 1, team::warp_all<team::Sum>(out_w));     // (CTA barriers: the histogram is complete)
    if (a.use_shared)
        for (int i = threadIdx.x; i < bins; i += team::kTT) {
            const unsigned long long w = a.vwgt ? s_bw[i] : s_bw32[i];
            if (w) atomicAdd(&a.BW[i], w);
        }
    team::sync(t);
    long long all;
    int64_t pos = team::collect<team::Sum>(t, 0, &all) + mine;
    for (int64_t v0 = g.b; v0 < g.e; v0 += 32) {
        const int64_t v = v0 + lane;
        const bool f = v < g.e && a.own[v] < a.wI[v];
        const unsigned m = __ballot_sync(full, f);
        if (f) a.list[pos + __popc(m & ((1u << lane) - 1u))] = (int32_t)v;
        pos += __popc(m);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_list = (int32_t)all;
    if (a.cut_pending) {
        if (!a.gid) {
            long long twice;
            team::collect<team::Sum>(t, 1, &twice);
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

// The selection kernels work on a list of nodes (the boundary nodes in a
// round, the active nodes in label propagation) and write by list index.
// G lanes per node: best target by (gain - penalty) among adjacent blocks,
// ties to the smaller block id; candidate iff the score is positive and v is
// a boundary node.
template <int G>
__global__ void __launch_bounds__(256) k_select(const GraphDev g, NodeList nl, const int32_t *__restrict__ part,
                                                const int32_t *__restrict__ W, Penalty pen, Candidates out) {
    constexpr int kGroups = 256 / G;
    const int gid = threadIdx.x / G, gl = threadIdx.x % G;
    const int64_t n = *nl.d_n;
    const int32_t k = g.k;
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
                    if (b == a || w <= 0) continue;
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

__device__ __forceinline__ int32_t int4_get(const int4 &x, int c) {
    return c == 0 ? x.x : c == 1 ? x.y : c == 2 ? x.z : x.w;
}

// Vectorised form of k_select for k % 4 == 0, k <= 4*G*CH: lane gl of a group
// holds blocks [4(gl + G j), 4(gl + G j) + 4) of the row in one int4 per j.
// With one graph (BATCH false) the per-block slack L_max - C[b] and the
// factors F_r (and, when they fit, the bucket prefixes) are staged in shared
// memory; in a batch each node reads its own graph's blocks from global
// memory.  A move into a block with room for it costs no penalty and needs no
// search.
template <int G, int CH, bool EXACT, bool BATCH, bool PACK = false>
__global__ void __launch_bounds__(256) k_select_vec(const GraphDev g, NodeList nl, const int32_t *__restrict__ part,
                                                    const int32_t *__restrict__ W, Penalty pen, int smem_pw,
                                                    Candidates out) {
    // s_slack[b] = L_max - C[b] clamped to 2^31 - 1 (blocks start balanced, so
    // it is >= 0): a node of weight c < 2^31 overfills b iff c > s_slack[b],
    // and then x = c - s_slack[b] is exact.
    extern __shared__ int64_t s_mem[];
    const int64_t n = *nl.d_n;
    const int32_t k = g.k;
    int64_t *s_F = s_mem;
    int64_t *s_PW = s_mem + kSlots;
    int32_t *s_slack = reinterpret_cast<int32_t *>(s_mem + kSlots + (smem_pw ? (size_t)k * kSlots : 0));
    int8_t *s_first = reinterpret_cast<int8_t *>(s_slack + k);
    if (!BATCH)
        for (int i = threadIdx.x; i < k; i += blockDim.x) {
            const int64_t sl = pen.Lb[i] - pen.C[i];
            s_slack[i] = (int32_t)(sl > 0x7fffffffLL ? 0x7fffffffLL : sl);
            s_first[i] = pen.first[i];
        }
    for (int i = threadIdx.x; i < kSlots; i += blockDim.x) s_F[i] = pen.F[i];
    if (!BATCH && smem_pw)
        for (int i = threadIdx.x; i < k * kSlots; i += blockDim.x) s_PW[i] = pen.PW[i];
    __syncthreads();
    const int64_t *PW = (!BATCH && smem_pw) ? s_PW : pen.PW;
    constexpr int kGroups = 256 / G;
    const int gid = threadIdx.x / G, gl = threadIdx.x % G;
    const int gbase = (threadIdx.x & 31) & ~(G - 1);
    // PACK (unit weights, one graph): a node of weight 1 pays the same
    // penalty p(b) into block b wherever it comes from, so p(b) (-1:
    // forbidden) is fixed for the launch; the lane keeps, per column it
    // scores, a bit "allowed" and the constant (2^kb - 1 - b) - (p(b) << kb)
    const int kb = PACK ? pen.pack_bits : 0;
    const int32_t kmask = (1 << kb) - 1;
    int32_t *s_pen = reinterpret_cast<int32_t *>(s_first + ((k + 3) & ~3));
    uint32_t okm = 0;
    int32_t cst[CH][4];
    if (PACK) {
        for (int b = threadIdx.x; b < k; b += blockDim.x) {
            const int32_t sl = s_slack[b];
            int32_t p = 0;
            if (sl < 1) {
                const int64_t x = 1 - (int64_t)sl;
                int lo;
                if (x == 1) {
                    lo = s_first[b];
                } else {
                    const int64_t *row = PW + (int64_t)b * kSlots;
                    if (row[kSlots - 1] < x) {
                        lo = -1;
                    } else {
                        lo = 0;
                        int hi = kSlots - 1;
                        while (lo < hi) {
                            const int mid = (lo + hi) >> 1;
                            if (row[mid] >= x) hi = mid; else lo = mid + 1;
                        }
                    }
                }
                if (lo < 0) {
                    p = -1;
                } else {
                    // floor(1 * F / 2^Q); a penalty of at least 2^gb exceeds every gain
                    const uint64_t pp = (uint64_t)s_F[lo] >> kQ;
                    p = pp >= (1ull << pen.gbits) ? -1 : (int32_t)pp;
                }
            }
            s_pen[b] = p;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < CH; j++)
#pragma unroll
            for (int cc = 0; cc < 4; cc++) {
                const int b = 4 * (gl + G * j) + cc;
                const int32_t p = (EXACT || b < k) ? s_pen[b] : -1;
                if (p >= 0) okm |= 1u << (4 * j + cc);
                cst[j][cc] = (kmask - b) - (p >= 0 ? (p << kb) : 0);
            }
    }
    // (the next node's id is loaded one iteration ahead, so that a row's load
    // does not wait for it)
    const int64_t step = (int64_t)gridDim.x * kGroups;
    const int64_t i0 = (int64_t)blockIdx.x * kGroups + gid;
    int32_t vnext = i0 < n ? nl.node[i0] : 0;
    for (int64_t base = (int64_t)blockIdx.x * kGroups; base < n; base += step) {
        const int64_t i = base + gid;
        const bool active = i < n;
        const int64_t v = vnext;
        if (i + step < n) vnext = nl.node[i + step];
        int4 r[CH];
        int32_t a = 0, b0 = 0;
        const int4 zero = make_int4(0, 0, 0, 0);
        const int32_t wIv = active ? g.wI[v] : 0;
        if (active) {
            const int32_t ag = part[v];
            a = BATCH ? blk_local(g, ag) : ag;
            b0 = ag - a;
            const int4 *row4 = reinterpret_cast<const int4 *>(W + v * (int64_t)k);
#pragma unroll
            for (int j = 0; j < CH; j++) {
                const int q = gl + G * j;
                r[j] = (EXACT || 4 * q < k) ? __ldcs(row4 + q) : zero;
            }
        } else {
#pragma unroll
            for (int j = 0; j < CH; j++) r[j] = zero;
        }
        const int q4 = a >> 2;
        int32_t mine = 0;
#pragma unroll
        for (int j = 0; j < CH; j++)
            if (j == q4 / G) mine = int4_get(r[j], a & 3);
        const int32_t own = __shfl_sync(0xffffffffu, mine, gbase + (q4 % G));
        if (PACK) {
            int32_t pbest = 0;
            if (active && own < wIv) {
                const int32_t ownk = own << kb;
#pragma unroll
                for (int j = 0; j < CH; j++)
#pragma unroll
                    for (int cc = 0; cc < 4; cc++) {
                        const int32_t key = (int4_get(r[j], cc) << kb) - ownk + cst[j][cc];
                        pbest = max(pbest, ((okm >> (4 * j + cc)) & 1u) ? key : 0);
                    }
            }
            for (int o = G / 2; o > 0; o >>= 1) pbest = max(pbest, __shfl_xor_sync(0xffffffffu, pbest, o));
            if (active && gl == 0) {
                // a score >= 1 (key >= 2^kb) makes a candidate
                const bool cand = pbest >= (1 << kb);
                const int32_t b = kmask - (pbest & kmask);
                const int32_t sc = pbest >> kb;
                out.tgt[i] = cand ? b0 + b : -1;
                out.s0[i] = cand ? sc : 0;
                out.gain[i] = cand ? sc + s_pen[b] : 0;
            }
            continue;
        }
        // Only a positive score makes a candidate and the penalty is never
        // negative, so blocks with gain <= 0 (the own block among them) are
        // skipped and every score kept lies in [1, 2^31).
        int32_t best = 0;
        int32_t bt = -1, bg = 0;
        if (active && own < wIv) {
            const int32_t c = g.vwgt ? g.vwgt[v] : 1;
#pragma unroll
            for (int j = 0; j < CH; j++) {
#pragma unroll
                for (int cc = 0; cc < 4; cc++) {
                    const int b = 4 * (gl + G * j) + cc;
                    const int32_t w = int4_get(r[j], cc);
                    if ((!EXACT && b >= k) || w <= own) continue;
                    const int32_t gain = w - own;
                    int32_t sc = gain;
                    int32_t slack;
                    if (BATCH) {
                        const int64_t sl = pen.Lb[b0 + b] - pen.C[b0 + b];
                        slack = (int32_t)(sl > 0x7fffffffLL ? 0x7fffffffLL : sl);
                    } else {
                        slack = s_slack[b];
                    }
                    if (c > slack) {
                        const int64_t x = (int64_t)c - slack;
                        int lo;
                        if (x == 1) {                               // first non-empty slot
                            lo = BATCH ? pen.first[b0 + b] : s_first[b];
                            if (lo < 0) continue;                   // forbidden
                        } else {
                            const int64_t *row = PW + (int64_t)(b0 + b) * kSlots;
                            if (row[kSlots - 1] < x) continue;      // no slot covers the excess: forbidden
                            lo = 0;
                            int hi = kSlots - 1;
                            while (lo < hi) {
                                const int mid = (lo + hi) >> 1;
                                if (row[mid] >= x) hi = mid; else lo = mid + 1;
                            }
                        }
                        const int64_t p = (int64_t)(((u128)(uint64_t)c * (uint64_t)s_F[lo]) >> kQ);
                        if (p >= gain) continue;
                        sc = gain - (int32_t)p;
                    }
                    if (bt < 0 || sc > best) { best = sc; bt = b; bg = gain; }
                }
            }
        }
        int32_t sbest = best;
        int32_t id = bt;
        group_argmax32<G>(sbest, id);
        const int32_t gsel = group_sum<G>((id >= 0 && bt == id) ? bg : 0);
        if (active && gl == 0) {
            const bool cand = id >= 0 && sbest > 0;
            out.tgt[i] = cand ? b0 + id : -1;
            out.s0[i] = cand ? sbest : 0;
            out.gain[i] = cand ? gsel : 0;
        }
    }
}

// Selection over the sparse table: G lanes per node walk the node's slots
// (hash order, so ties compare block ids explicitly); penalties as in
// k_select_vec with the per-block values read from global memory.
template <int G>
__global__ void __launch_bounds__(256) k_select_sparse(const GraphDev g, NodeList nl,
                                                       const int32_t *__restrict__ part, Penalty pen,
                                                       Candidates out) {
    constexpr int kGroups = 256 / G;
    const int gid = threadIdx.x / G, gl = threadIdx.x % G;
    const int64_t n = *nl.d_n;
    const SparseRows &sp = g.sp;
    for (int64_t base = (int64_t)blockIdx.x * kGroups; base < n; base += (int64_t)gridDim.x * kGroups) {
        const int64_t i = base + gid;
        const bool active = i < n;
        const int64_t v = active ? nl.node[i] : 0;
        int32_t best = 0, bt = -1, bg = 0, b0 = 0;
        if (active) {
            const int32_t ag = part[v];
            const int32_t a = blk_local(g, ag);
            b0 = ag - a;
            const int32_t own = nl.own ? nl.own[v] : sp_get(sp, v, a);
            if (nl.own || own < g.wI[v]) {
                const int32_t c = g.vwgt ? g.vwgt[v] : 1;
                for (int64_t q = sp.off[v] + gl; q < sp.off[v + 1]; q += G) {
                    const int2 e = sp.slot[q];
                    if (e.x == kEmpty || e.y <= own) continue;      // gain <= 0 (the own block among them)
                    const int32_t b = e.x, gain = e.y - own;
                    const int64_t sl = pen.Lb[b0 + b] - pen.C[b0 + b];
                    const int32_t slack = (int32_t)(sl > 0x7fffffffLL ? 0x7fffffffLL : sl);
                    int32_t sc = gain;
                    if (c > slack) {
                        const int64_t x = (int64_t)c - slack;
                        int lo;
                        if (x == 1) {
                            lo = pen.first[b0 + b];
                            if (lo < 0) continue;
                        } else {
                            const int64_t *row = pen.PW + (int64_t)(b0 + b) * kSlots;
                            if (row[kSlots - 1] < x) continue;
                            lo = 0;
                            int hi = kSlots - 1;
                            while (lo < hi) {
                                const int mid = (lo + hi) >> 1;
                                if (row[mid] >= x) hi = mid; else lo = mid + 1;
                            }
                        }
                        const int64_t p = (int64_t)(((u128)(uint64_t)c * (uint64_t)pen.F[lo]) >> kQ);
                        if (p >= gain) continue;
                        sc = gain - (int32_t)p;
                    }
                    if (bt < 0 || sc > best || (sc == best && b < bt)) { best = sc; bt = b; bg = gain; }
                }
            }
        }
        int32_t sbest = best, id = bt;
        group_argmax32<G>(sbest, id);
        const int32_t gsel = group_sum<G>((id >= 0 && bt == id) ? bg : 0);
        if (active && gl == 0) {
            const bool cand = id >= 0 && sbest > 0;
            out.tgt[i] = cand ? b0 + id : -1;
            out.s0[i] = cand ? sbest : 0;
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
template <class Item>
__global__ void __launch_bounds__(team::kTT, 1) k_sel_order(const SelOrder a) {
    __shared__ team::Smem s;
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
    team::collect<team::Max>(t, 0, &top);
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
        base = team::collect<team::Sum>(t, 1, &all) + mine;
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
            room[r] = a.pen.Lb[tg] - a.pen.C[tg];
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            if (j0 + 32 * r >= g.e) continue;
            const int64_t p = penalty(a.pen, (int32_t)(it[r].key >> sbits), inflow[r] + c[r] - room[r], c[r]);
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
    team::collect<team::Max>(t, 2, &ktop);

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

void select_order(const GraphDev &g, SelOrder a, int gbits, cudaStream_t s) {
    if (g.n <= 0) return;
    a.K = g.K();
    a.vwgt = g.vwgt;
    a.xadj = g.xadj;
    a.kbits = 1;
    while ((1ll << a.kbits) < a.K) a.kbits++;
    // (scores are at most omega(I(v)), so they have at most gbits bits)
    if (gbits + a.kbits <= 32) launch_team(k_sel_order<team::Item32>, a, a.team.size, s);
    else launch_team(k_sel_order<team::Item64>, a, a.team.size, s);
}

void node_pass(const GraphDev &g, NodePass a, const int32_t *W, cudaStream_t s) {
    ensure_pow3();
    a.n = g.n;
    a.k = g.k;
    a.kmask = g.kmask;
    a.K = g.K();
    a.ng = g.ng;
    a.W = W;
    a.sp = g.sp;
    a.wI = g.wI;
    a.vwgt = g.vwgt;
    a.gid = g.gid;
    UPR_CUDA(cudaMemsetAsync(a.BW, 0, sizeof(int64_t) * a.K * kSlots, s));
    if (a.cut_pending && g.ng > 1) UPR_CUDA(cudaMemsetAsync(a.cut, 0, sizeof(int64_t) * g.ng, s));
    const size_t shm = (g.vwgt ? sizeof(unsigned long long) : sizeof(unsigned int)) * (size_t)a.K * kSlots;
    a.use_shared = shm <= 184 * 1024;            // (the team's own shared memory is static, 37 KB)
    launch_team(k_node_pass, a, a.team.size, s, a.use_shared ? shm : 0);
}

int select_group(int k) {
    int G = k / 4;
    return G >= 32 ? 32 : G >= 16 ? 16 : G >= 8 ? 8 : k >= 4 ? 4 : 2;
}

int lane_candidates(int32_t k, LaneCfg *out) {
    if (k % 4 != 0 || k > 256) return 0;
    int G = 1;
    while (G < 32 && 4 * G < k) G <<= 1;
    int CH = (k + 4 * G - 1) / (4 * G);
    int cnt = 0;
    out[cnt++] = LaneCfg{G, CH};
    // fewer lanes per node, more chunks per lane (exact fits only, at most 4 chunks)
    while (cnt < 3 && G > 1 && CH * 2 <= 4 && 4 * (G / 2) * (CH * 2) == k) {
        G /= 2;
        CH *= 2;
        out[cnt++] = LaneCfg{G, CH};
    }
    return cnt;
}

namespace {

template <int G, int CH>
void launch_select_vec(bool exact, bool batch, unsigned blocks, size_t shm, cudaStream_t s, const GraphDev &g,
                       NodeList nl, const int32_t *part, const int32_t *W, const Penalty &pen, int smem_pw,
                       Candidates out) {
    // one full wave of CTAs at most (the kernel loops over the nodes)
    auto go = [&](auto kern) {
        kern<<<wave_grid((const void *)kern, 256, shm, blocks), 256, shm, s>>>(g, nl, part, W, pen, smem_pw, out);
    };
    const bool pack = !batch && pen.pack_bits > 0 && g.vwgt == nullptr;
    if constexpr (CH == 1 || (G == 32 && CH == 2)) {
        if (!exact) {
            if (batch) go(k_select_vec<G, CH, false, true>);
            else if (pack) go(k_select_vec<G, CH, false, false, true>);
            else go(k_select_vec<G, CH, false, false>);
            return;
        }
    }
    if (batch) go(k_select_vec<G, CH, true, true>);
    else if (pack) go(k_select_vec<G, CH, true, false, true>);
    else go(k_select_vec<G, CH, true, false>);
}

}  // namespace

void select_moves(const GraphDev &g, NodeList nl, const int32_t *part, const int32_t *W, Penalty pen, Candidates out,
                  LaneCfg cfg, cudaStream_t s) {
    if (g.n == 0) return;
    const int k = g.k;
    const bool batch = g.ng > 1;
    if (g.sp.on()) {
        const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(g.n, 256 / 8), (int64_t)sm_count_sel() * 8);
        k_select_sparse<8><<<blocks, 256, 0, s>>>(g, nl, part, pen, out);
        UPR_LAUNCH_CHECK();
        return;
    }
    LaneCfg cands[3];
    if (lane_candidates(k, cands) > 0) {
        if (cfg.G <= 0) cfg = cands[0];
        const int G = cfg.G, CH = cfg.CH;
        const bool exact = k == 4 * G * CH;
        // the slot prefixes are read only for an excess x > 1, i.e. a node
        // weight c >= 2: with unit node weights they stay in global memory
        // and the smaller shared footprint lets more CTAs run
        const int smem_pw = !batch && g.vwgt && (size_t)k * kSlots * 8 <= 40 * 1024;
        const size_t shm = sizeof(int64_t) * ((size_t)kSlots + (smem_pw ? (size_t)k * kSlots : 0)) +
                           (batch ? 0 : (sizeof(int32_t) + 1) * k + sizeof(int32_t) * (k + 4));
        const int64_t groups = 256 / G;
        const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(g.n, groups), (int64_t)sm_count_sel() * 8);
#define UPR_SELC(GG, CC)                                                                                       \
    if (G == GG && CH == CC) {                                                                                 \
        launch_select_vec<GG, CC>(exact, batch, blocks, shm, s, g, nl, part, W, pen, smem_pw, out);            \
        UPR_LAUNCH_CHECK();                                                                                    \
        return;                                                                                                \
    }
        UPR_SELC(1, 1) UPR_SELC(2, 1) UPR_SELC(4, 1) UPR_SELC(8, 1) UPR_SELC(16, 1) UPR_SELC(32, 1)
        UPR_SELC(1, 2) UPR_SELC(2, 2) UPR_SELC(4, 2) UPR_SELC(8, 2) UPR_SELC(16, 2) UPR_SELC(32, 2)
        UPR_SELC(1, 4) UPR_SELC(2, 4) UPR_SELC(4, 4) UPR_SELC(8, 4) UPR_SELC(16, 4)
#undef UPR_SELC
        throw CudaError{cudaErrorInvalidValue, "select_moves: unsupported lane schedule"};
    }
    const int G = select_group(k);
    const int64_t groups = 256 / G;
    const int64_t blocks = std::min<int64_t>(ceil_div(g.n, groups), (int64_t)sm_count_sel() * 16);
#define UPR_SEL(GG) k_select<GG><<<(unsigned)blocks, 256, 0, s>>>(g, nl, part, W, pen, out)
    switch (G) {
        case 2: UPR_SEL(2); break;
        case 4: UPR_SEL(4); break;
        case 8: UPR_SEL(8); break;
        case 16: UPR_SEL(16); break;
        default: UPR_SEL(32); break;
    }
#undef UPR_SEL
    UPR_LAUNCH_CHECK();
}

}  // namespace upr
