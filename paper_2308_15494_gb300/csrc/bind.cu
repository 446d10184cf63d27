// Static schedules of a binding, built on the device from the packed row
// offsets (the hub chunks, the table build's tiles, the hashed rows' slot
// offsets and the hub list), in two passes over fixed segments of
// kSchedSegment nodes: one warp per segment counts, a one-CTA scan turns the
// counts into offsets and totals (read back to size the arena), and the same
// walk writes.  A segment boundary also ends a tile; rows are independent, so
// any such tiling gives the same table.  The walk takes 32 nodes at a time:
// prefix sums over the lanes, and one ballot per tile that ends among them
// (one thread per segment, node by node, waited for every offset: 0.61 and
// 0.56 ms for 2^19 nodes).
#include "prim.cuh"

namespace upr {
namespace {

using namespace prim;

struct SchedOut {
    HubChunk *chunks;
    TableTile *tiles;
    int64_t *sp_off;
    int32_t *hubs;
};
struct SchedCount { int64_t chunks, tiles, sp, hubs; };

__device__ __forceinline__ int64_t warp_incl_sum(int64_t v) {
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) >= o) v += u;
    }
    return v;
}

// Walks the nodes [v0, v1) of one segment with one warp: hub chunks (8192
// entries of one node of degree > kHubDegree), tiles (runs of consecutive
// nodes with at most tile_nodes rows, kTileEntries non-hub entries and, with
// hashed rows, kTileSlots non-hub slots, a hub closing its tile) and the
// hashed rows' slots (a power of two >= min(k, 2 deg) + 1, or min(k, deg) + 1
// with sp_mode 3).  base: this segment's first chunk, tile, slot and hub; with
// out == nullptr it only counts.  Offsets outside [0, m] or decreasing (an
// input the check rejects) count as empty rows.
__device__ __forceinline__ SchedCount sched_walk(const int64_t *__restrict__ x, int64_t m, int64_t v0, int64_t v1,
                                                 int tile_nodes, int sp_mode, int32_t k, const SchedOut *out,
                                                 SchedCount base) {
    constexpr int64_t kTileEntries = 4096;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    SchedCount c{0, 0, 0, 0};
    // the open tile: rows, entries and slots so far, its first node and entry
    int64_t rows = 0, ent = 0, slots = 0, tv = v0, te = 0;
    auto close = [&](int64_t v_end) {
        if (out && lane == 0) out->tiles[base.tiles + c.tiles] = TableTile{te, te + ent, (int32_t)tv, (int32_t)v_end};
        c.tiles++;
        rows = ent = slots = 0;
    };
    for (int64_t b = v0; b < v1; b += 32) {
        const int64_t v = b + lane;
        const bool in = v < v1;
        const int64_t e0 = in ? x[v] : 0, e1 = in ? x[v + 1] : 0;
        const int64_t d = (e0 < 0 || e1 < e0 || e1 > m) ? 0 : e1 - e0;
        const bool hub = d > kHubDegree;
        const unsigned hubs = __ballot_sync(full, hub);
        if (hubs) {
            const int64_t nc = hub ? (d + 8191) / 8192 : 0;
            const int64_t inc = warp_incl_sum(nc);
            if (out && hub) {
                out->hubs[base.hubs + c.hubs + __popc(hubs & ((1u << lane) - 1u))] = (int32_t)v;
                for (int64_t i = 0; i < nc; i++)
                    out->chunks[base.chunks + c.chunks + inc - nc + i] =
                        HubChunk{(int32_t)v, 0, e0 + i * 8192, min(e0 + (i + 1) * 8192, e0 + d)};
            }
            c.hubs += __popc(hubs);
            c.chunks += __shfl_sync(full, inc, 31);
        }
        int64_t cap = 0;
        if (sp_mode) {
            const int64_t want = min((int64_t)k, sp_mode == 3 ? d : 2 * d) + 1;
            cap = in ? (want <= 1 ? 1 : (int64_t)1 << (64 - __clzll(want - 1))) : 0;
            const int64_t inc = warp_incl_sum(cap);
            if (out && in) out->sp_off[v] = base.sp + c.sp + inc - cap;
            c.sp += __shfl_sync(full, inc, 31);
        }
        if (!tile_nodes) continue;
        const int64_t pe = warp_incl_sum(hub ? 0 : d), ps = warp_incl_sum(hub ? 0 : cap);
        const int last = (int)min((int64_t)32, v1 - b);
        int cur = 0;                       // the first lane whose node is in no tile yet
        while (cur < last) {
            const int64_t be = cur ? __shfl_sync(full, pe, cur - 1) : 0, bs = cur ? __shfl_sync(full, ps, cur - 1) : 0;
            if (rows == 0) {
                tv = b + cur;
                te = __shfl_sync(full, e0, cur);
            }
            const int64_t at = rows + lane - cur;        // rows of the tile when this lane's node is reached
            const bool stop = lane >= cur && lane < last &&
                              (at >= tile_nodes || (at > 0 && !hub && (ent + pe - be > kTileEntries ||
                                                                       slots + ps - bs > kTileSlots)));
            const unsigned sb = __ballot_sync(full, stop), hb = hubs & (full << cur);
            const int ls = sb ? __ffs(sb) - 1 : 32, lh = hb ? __ffs(hb) - 1 : 32;
            const int end = lh < ls ? lh + 1 : min(ls, last);       // lanes [cur, end) join the tile
            if (end > cur) {
                ent += __shfl_sync(full, pe, end - 1) - be;
                slots += __shfl_sync(full, ps, end - 1) - bs;
                rows += end - cur;
            }
            cur = end;
            if (lh < ls || ls < 32) close(b + cur);
        }
    }
    if (tile_nodes && rows) close(v1);
    return c;
}

// Per segment s: cnt[4 s + 0..3] = chunks, tiles, sparse slots, hubs.
__global__ void k_sched_count(const int64_t *__restrict__ x, int64_t n, int64_t m, int64_t nseg, int tile_nodes,
                              int sp_mode, int32_t k, int64_t *__restrict__ cnt) {
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= nseg) return;
    const int64_t v0 = s * kSchedSegment, v1 = min(n, v0 + kSchedSegment);
    const SchedCount c = sched_walk(x, m, v0, v1, tile_nodes, sp_mode, k, nullptr, SchedCount{0, 0, 0, 0});
    if ((threadIdx.x & 31) == 0) {
        cnt[4 * s + 0] = c.chunks;
        cnt[4 * s + 1] = c.tiles;
        cnt[4 * s + 2] = c.sp;
        cnt[4 * s + 3] = c.hubs;
    }
}

// Exclusive prefix of each of the four count columns in place, one CTA, a run
// of segments per thread; tot[0..3] = the totals.
__global__ void __launch_bounds__(kThreads) k_sched_scan(int64_t *__restrict__ cnt, int64_t nseg,
                                                         int64_t *__restrict__ tot) {
    __shared__ int64_t s_warp[kWarps];
    const int64_t per = (nseg + kThreads - 1) / kThreads;
    const int64_t a = min(nseg, (int64_t)threadIdx.x * per), b = min(nseg, a + per);
    for (int col = 0; col < 4; col++) {
        int64_t sum = 0, total;
        for (int64_t i = a; i < b; i++) sum += cnt[4 * i + col];
        int64_t run = block_exclusive<OpSum>(sum, s_warp, &total);
        for (int64_t i = a; i < b; i++) {
            const int64_t v = cnt[4 * i + col];
            cnt[4 * i + col] = run;
            run += v;
        }
        if (threadIdx.x == 0) tot[col] = total;
    }
}

__global__ void k_sched_write(const int64_t *__restrict__ x, int64_t n, int64_t m, int64_t nseg, int tile_nodes,
                              int sp_mode, int32_t k, const int64_t *__restrict__ off, SchedOut out) {
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= nseg) return;
    const int64_t v0 = s * kSchedSegment, v1 = min(n, v0 + kSchedSegment);
    const SchedCount c = sched_walk(x, m, v0, v1, tile_nodes, sp_mode, k, &out,
                                    SchedCount{off[4 * s + 0], off[4 * s + 1], off[4 * s + 2], off[4 * s + 3]});
    if (sp_mode && v1 == n && (threadIdx.x & 31) == 0) out.sp_off[n] = off[4 * s + 2] + c.sp;
}

// One graph's offsets: x[0] = 0, x[n] = m, non-decreasing; *bad = 1 otherwise.
__global__ void k_xadj_check(const int64_t *__restrict__ x, int64_t n, int64_t m, int32_t *__restrict__ bad) {
    UPR_FOR(v, n) if (x[v + 1] < x[v]) *bad = 1;
    if (blockIdx.x == 0 && threadIdx.x == 0 && (x[0] != 0 || x[n] != m)) *bad = 1;
}

// A batch's packed offsets: node j of graph i (noff[i] <= j < noff[i + 1])
// takes graph i's own offset raw[noff[i] + i + (j - noff[i])] plus eoff[i];
// out[n] = eoff[ng].  *bad = 1 unless each graph's offsets start at 0, end at
// its entry count and do not decrease.
__global__ void k_xadj_pack(const int64_t *__restrict__ raw, const int64_t *__restrict__ noff,
                            const int64_t *__restrict__ eoff, int32_t ng, int64_t n, int64_t *__restrict__ out,
                            int32_t *__restrict__ bad) {
    UPR_FOR(j, n) {
        int32_t lo = 0, hi = ng - 1;            // the last graph i with noff[i] <= j
        while (lo < hi) {
            const int32_t mid = (lo + hi + 1) >> 1;
            if (noff[mid] <= j) lo = mid; else hi = mid - 1;
        }
        const int64_t p = noff[lo] + lo + (j - noff[lo]);
        const int64_t a = raw[p], b = raw[p + 1];
        out[j] = a + eoff[lo];
        if (b < a) *bad = 1;
        if (j == noff[lo] && a != 0) *bad = 1;
        if (j + 1 == noff[lo + 1] && b != eoff[lo + 1] - eoff[lo]) *bad = 1;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = eoff[ng];
}

// Copies of many host arrays in one launch: the arrays are page-locked host
// memory, which the GPU reads directly; segment i moves len elements from
// src to dst + off (segments of at most kGatherChunk elements, one per CTA
// at a time, eight loads in flight per thread).
template <typename T>
__global__ void __launch_bounds__(256) k_gather_host(const HostSeg *__restrict__ segs, int64_t nseg,
                                                     T *__restrict__ dst) {
    for (int64_t i = blockIdx.x; i < nseg; i += gridDim.x) {
        const HostSeg sg = segs[i];
        const T *src = static_cast<const T *>(sg.src);
        T *out = dst + sg.off;
        for (int64_t b = 0; b < sg.len; b += 8 * 256) {
            T x[8];
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const int64_t e = b + u * 256 + threadIdx.x;
                if (e < sg.len) x[u] = src[e];
            }
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const int64_t e = b + u * 256 + threadIdx.x;
                if (e < sg.len) out[e] = x[u];
            }
        }
    }
}

}  // namespace

void gather_host(const HostSeg *d_segs, int64_t nseg, size_t elem, void *dst, cudaStream_t s) {
    if (nseg <= 0) return;
    const unsigned grid = (unsigned)std::min<int64_t>(nseg, (int64_t)device_sm_count() * 8);
    if (elem == 8) k_gather_host<int64_t><<<grid, 256, 0, s>>>(d_segs, nseg, static_cast<int64_t *>(dst));
    else k_gather_host<int32_t><<<grid, 256, 0, s>>>(d_segs, nseg, static_cast<int32_t *>(dst));
    UPR_LAUNCH_CHECK();
}

void xadj_pack(const int64_t *raw, const int64_t *noff, const int64_t *eoff, int32_t ng, int64_t n, int64_t *out,
               int32_t *bad, cudaStream_t s) {
    k_xadj_pack<<<grid_for(std::max<int64_t>(n, 1)), 256, 0, s>>>(raw, noff, eoff, ng, n, out, bad);
    UPR_LAUNCH_CHECK();
}

int64_t sched_segments(int64_t n) { return n > 0 ? ceil_div(n, kSchedSegment) : 0; }

void sched_count(const int64_t *xadj, int64_t n, int64_t m, int tile_nodes, int sp_mode, int32_t k, int64_t *cnt,
                 int64_t *tot, cudaStream_t s) {
    const int64_t nseg = sched_segments(n);
    if (nseg == 0) {
        UPR_CUDA(cudaMemsetAsync(tot, 0, 4 * sizeof(int64_t), s));
        return;
    }
    k_sched_count<<<(unsigned)ceil_div(nseg, 4), 128, 0, s>>>(xadj, n, m, nseg, tile_nodes, sp_mode, k, cnt);
    UPR_LAUNCH_CHECK();
    k_sched_scan<<<1, kThreads, 0, s>>>(cnt, nseg, tot);
    UPR_LAUNCH_CHECK();
}

void sched_write(const int64_t *xadj, int64_t n, int64_t m, int tile_nodes, int sp_mode, int32_t k,
                 const int64_t *off, HubChunk *chunks, TableTile *tiles, int64_t *sp_off, int32_t *hubs,
                 cudaStream_t s) {
    const int64_t nseg = sched_segments(n);
    if (nseg == 0) return;
    k_sched_write<<<(unsigned)ceil_div(nseg, 4), 128, 0, s>>>(xadj, n, m, nseg, tile_nodes, sp_mode, k, off,
                                                              SchedOut{chunks, tiles, sp_off, hubs});
    UPR_LAUNCH_CHECK();
}

void xadj_check(const int64_t *xadj, int64_t n, int64_t m, int32_t *bad, cudaStream_t s) {
    k_xadj_check<<<grid_for(std::max<int64_t>(n, 1)), 256, 0, s>>>(xadj, n, m, bad);
    UPR_LAUNCH_CHECK();
}

}  // namespace upr
