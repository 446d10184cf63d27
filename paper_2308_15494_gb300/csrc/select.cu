// Step (b): rebalancing availability, slots and bucket weights (Alg. 1,
// Sec. 4.3), each boundary node's best move by gain minus penalty
// (Alg. 1), penalties with the inflow of better-ranked candidates,
// the global move order M (Sec. 4.4), and the application of M.
#include "select_team.cuh"

namespace upr {
namespace {

int sm_count_sel() {
    static int cnt = 0;
    if (!cnt) {
        int dev = 0;
        UPR_CUDA(cudaGetDevice(&dev));
        UPR_CUDA(cudaDeviceGetAttribute(&cnt, cudaDevAttrMultiProcessorCount, dev));
    }
    return cnt;
}

__global__ void __launch_bounds__(team::kTT, 1) k_node_pass(const __grid_constant__ NodePass a) {
    __shared__ team::Smem s;
    extern __shared__ unsigned long long s_bw[];
    node_pass_body(a, a.cut_pending != 0, s, s_bw);
}

template <class Item>
__global__ void __launch_bounds__(team::kTT, 1) k_sel_order(const __grid_constant__ SelOrder a) {
    __shared__ team::Smem s;
    sel_order_body<Item>(a, a.pen, s);
}

// The selection kernels work on a list of nodes (the boundary nodes in a
// round, the active nodes in label propagation) and write by list index.
template <int G>
__global__ void __launch_bounds__(256) k_select(const __grid_constant__ GraphDev g, NodeList nl,
                                                const int32_t *__restrict__ part, const int32_t *__restrict__ W,
                                                const __grid_constant__ Penalty pen, Candidates out) {
    select_rows<G, 256>(g, nl, part, W, pen, out);
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
    // scores, the constant (2^kb - 1 - b) - (p(b) << kb), or one so low that no
    // omega (omega << kb < 2^30) lifts it above another score.  The node's own
    // omega comes off the maximum instead of every column: two instructions a
    // column where a mask of the allowed ones took five (with the same change to
    // the proposals, 2^22 nodes, 64 blocks: 17.74 -> 17.52 ms)
    const int kb = PACK ? pen.pack_bits : 0;
    const int32_t kmask = (1 << kb) - 1;
    int32_t *s_pen = reinterpret_cast<int32_t *>(s_first + ((k + 3) & ~3));
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
                cst[j][cc] = p >= 0 ? (kmask - b) - (p << kb) : INT32_MIN;
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
                int32_t top = ownk;
#pragma unroll
                for (int j = 0; j < CH; j++)
#pragma unroll
                    for (int cc = 0; cc < 4; cc++) top = max(top, (int4_get(r[j], cc) << kb) + cst[j][cc]);
                pbest = top - ownk;
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

}  // namespace

void select_order_args(const GraphDev &g, SelOrder &a) {
    a.K = g.K();
    a.vwgt = g.vwgt;
    a.xadj = g.xadj;
    a.kbits = 1;
    while ((1ll << a.kbits) < a.K) a.kbits++;
}

void select_order(const GraphDev &g, SelOrder a, int gbits, cudaStream_t s) {
    if (g.n <= 0) return;
    select_order_args(g, a);
    // (scores are at most omega(I(v)), so they have at most gbits bits)
    if (gbits + a.kbits <= 32) launch_team(k_sel_order<team::Item32>, a, a.team.size, s);
    else launch_team(k_sel_order<team::Item64>, a, a.team.size, s);
}

size_t node_pass_args(const GraphDev &g, NodePass &a, const int32_t *W, size_t room) {
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
    const size_t shm = (g.vwgt ? sizeof(unsigned long long) : sizeof(unsigned int)) * (size_t)a.K * kSlots;
    a.use_shared = shm <= room;
    return a.use_shared ? shm : 0;
}

void node_pass(const GraphDev &g, NodePass a, const int32_t *W, cudaStream_t s) {
    const size_t shm = node_pass_args(g, a, W, std::min(kNodePassSmem, dynamic_smem((const void *)k_node_pass)));
    UPR_CUDA(cudaMemsetAsync(a.BW, 0, sizeof(int64_t) * a.K * kSlots, s));
    if (a.cut_pending && g.ng > 1) UPR_CUDA(cudaMemsetAsync(a.cut, 0, sizeof(int64_t) * g.ng, s));
    launch_team(k_node_pass, a, a.team.size, s, shm);
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
