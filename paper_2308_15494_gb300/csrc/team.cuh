// Building blocks of the team kernels: one cooperative launch of P CTAs of
// 1024 threads (one CTA per SM at most) runs a whole chain of steps over
// ordered lists, separated by grid barriers, instead of one launch per step.
//
// A list of n items is cut into one contiguous segment per warp (CTA order,
// then warp order), so a scan needs one barrier: every warp sums its segment,
// the CTA publishes its total, and after the barrier every warp adds the
// totals before its CTA and the sums before it in its CTA.  A stable sort pass
// needs two: every warp counts the digits of its segment in its own row of
// shared memory, the CTA publishes its digit totals, and after the barrier
// the rows hold every warp's first position per digit, which the warp walks
// its segment with (ranks inside 32 items by __match_any_sync), without any
// CTA barrier.  What bounds these chains is latency: with lists of 10^4 to
// 10^6 items a step of its own launch takes 3 to 10 us, most of it launch,
// ramp and look-back; a step here is a few hundred cycles of work plus one
// barrier.  Three team launches a round (k_sel_order, k_seq_build, k_seq_best)
// stand for about ninety launches; per refinement, before and after: Chung-Lu
// n = 1024, k = 2, 4 rounds 1.68 and 0.96 ms; R-MAT scale 18, k = 8, 8 rounds
// 5.85 and 3.28 ms (785 and 209 launches); Chung-Lu n = 10^6 with weights,
// k = 23 10.0 and 6.6 ms; R-MAT scale 22, k = 64 22.0 and 20.1 ms.  In a round
// at scale 18 they take 43, 41 and 35 us.
#pragma once

#include "prim.cuh"

namespace upr {
namespace team {

constexpr int kTT = 1024;                // threads of a CTA
constexpr int kTW = kTT / 32;
constexpr int kTeamMax = 160;            // CTAs at most
constexpr int kTotSlots = 24;            // published per-CTA totals (one slot per scan of a kernel)
constexpr int kSortBins = 256;
constexpr int kMaxSpin = 1 << 22;        // polls before a barrier's wait gives up (about a second)
constexpr unsigned long long kBroken = 1ull << 63;     // in the arrival counter: a wait gave up

struct Smem {
    unsigned long long cnt64[kTW * kSortBins / 2];     // digit counts [kTW][bins], or block-weight changes
    int tot[kSortBins], bef[kSortBins];
    unsigned long long rep[kSortBins];
    long long w[kTW];
    static constexpr bool kCluster = false;            // the team's totals are in global memory
    __device__ __forceinline__ int *cnt() { return reinterpret_cast<int *>(cnt64); }
};
// Of a kernel whose teams are one CTA or one cluster: a CTA's totals for the
// team stay in its shared memory (a write and a read through the L2 cost about
// 1.2 us per step).  The kernels of larger teams are compiled without it: with
// both forms in one kernel and a test at each use, 2^18 nodes, 8 blocks took
// 2.88 ms instead of 2.77.
struct ClusterSmem : Smem {
    static constexpr bool kCluster = true;
    unsigned long long row64[2][kSortBins];            // block weights,
    int row[kSortBins];                                // digits,
    long long sums[kTotSlots];                         // and scans
};

constexpr int kClusterMax = 16;          // teams up to this size run as one cluster

// The team's barrier: a CTA barrier for one CTA, a cluster barrier for a
// cluster, else a grid barrier on an arrival counter that only grows: the
// barrier a CTA reaches with arrival number `old` ends when the count reaches
// the next multiple of the grid size.  (About 1.2 us with 152 CTAs.  Arriving
// without the old value, by a release reduction, took 0.15 us longer; an epoch
// word per CTA polled by a warp of every CTA 1 us longer.)
//
// Every wait on the counter is bounded.  One that gives up sets the counter's
// top bit, by an exchange that succeeds only while the barrier is incomplete:
// so every CTA passes a barrier or none does, and a CTA that meets the bit sets
// the error word and leaves the kernel, at this barrier and at the first one of
// every later launch (until the next binding clears the counter).  No step then
// runs on what another CTA has not published, and what a kernel writes behind
// its last barrier is there in full or not at all: the lengths that other
// kernels read are written there, and are 0 before.  (A sub-round's next list
// has its length earlier; it holds nodes either way.)
__device__ __forceinline__ void sync(const Team &t) {
    if (gridDim.x == 1) {
        __syncthreads();
        return;
    }
    if (gridDim.x <= kClusterMax) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        return;
    }
    __syncthreads();
    int broken = 0;
    if (threadIdx.x == 0) {
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        const unsigned long long old = atomicAdd(t.bar, 1ull);
        const unsigned long long target = (old / gridDim.x + 1) * gridDim.x;
        for (int it = 0;; it++) {
            unsigned long long v;
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(t.bar) : "memory");
            broken = (v & kBroken) != 0;
            if (broken || v >= target) break;
            // (the exchange fails only when another CTA has just arrived or given up)
            if (it >= kMaxSpin && atomicCAS(t.bar, v, v | kBroken) == v) {
                broken = 1;
                break;
            }
            if (it >= 16) __nanosleep(32);
        }
        if (broken) atomicOr(t.err, 2);
    }
    if (__syncthreads_or(broken)) asm volatile("exit;");
}

// A value of CTA c's shared memory (c in this team, a cluster).
template <typename T>
__device__ __forceinline__ T remote(const T *mine, int c) {
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "one word");
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(mine)), "r"(c));
    if constexpr (sizeof(T) == 4) {
        uint32_t v;
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
        return (T)v;
    } else {
        unsigned long long v;
        asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
        return (T)v;
    }
}

// A per-CTA value published in a slot, and CTA c's after a barrier.
template <class Sm>
__device__ __forceinline__ void put(const Team &t, Sm &s, int slot, long long v) {
    if constexpr (Sm::kCluster) s.sums[slot] = v;
    else t.tot[slot * kTeamMax + blockIdx.x] = v;
}
template <class Sm>
__device__ __forceinline__ long long get(const Team &t, const Sm &s, int slot, int c) {
    if constexpr (Sm::kCluster) return remote(&s.sums[slot], c);
    else return t.tot[slot * kTeamMax + c];
}

struct Seg { int64_t b, e; };

// This warp's segment of a list of n items (a multiple of 32 items long).
__device__ __forceinline__ Seg warp_seg(int64_t n) {
    const unsigned warps = gridDim.x * kTW;
    const int64_t per = ((n + warps - 1) / warps + 31) & ~(int64_t)31;
    const int64_t b = min(n, per * (int64_t)(blockIdx.x * kTW + (threadIdx.x >> 5)));
    return Seg{b, min(n, b + per)};
}

// The threads' stride loop of the whole team (work without an order).
#define UPR_TEAM_FOR(i, cnt)                                                                        \
    for (int64_t i = (int64_t)blockIdx.x * upr::team::kTT + threadIdx.x; i < (int64_t)(cnt);         \
         i += (int64_t)gridDim.x * upr::team::kTT)

struct Sum {
    __device__ __forceinline__ static long long id() { return 0; }
    __device__ __forceinline__ static long long op(long long a, long long b) { return a + b; }
};
struct Max {       // of values >= 0
    __device__ __forceinline__ static long long id() { return 0; }
    __device__ __forceinline__ static long long op(long long a, long long b) { return a > b ? a : b; }
};

template <class Op>
__device__ __forceinline__ long long warp_all(long long v) {
    for (int o = 16; o > 0; o >>= 1) v = Op::op(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
template <class Op>
__device__ __forceinline__ long long warp_incl(long long v) {
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) >= o) v = Op::op(u, v);
    }
    return v;
}

// Publishes the CTA's total of the warps' values x (equal in a warp's lanes)
// in the slot; returns the total of the warps before this one in the CTA.
template <class Op, class Sm>
__device__ __forceinline__ long long publish(const Team &t, Sm &s, int slot, long long x) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s.w[warp] = x;
    __syncthreads();
    const long long inc = warp_incl<Op>(s.w[lane]);
    const long long before = __shfl_sync(0xffffffffu, inc, warp > 0 ? warp - 1 : 0);
    if (threadIdx.x == kTT - 1) put(t, s, slot, inc);
    __syncthreads();
    return warp > 0 ? before : Op::id();
}

// After a barrier: the published totals of the CTAs before this one, and of all.
template <class Op, class Sm>
__device__ __forceinline__ long long collect(const Team &t, const Sm &s, int slot, long long *all) {
    const int lane = threadIdx.x & 31;
    if constexpr (Sm::kCluster)
        if (gridDim.x == 1) {
            *all = s.sums[slot];
            return Op::id();
        }
    long long b = Op::id(), a = Op::id();
    for (int c = lane; c < (int)gridDim.x; c += 32) {
        const long long v = get(t, s, slot, c);
        a = Op::op(a, v);
        if (c < (int)blockIdx.x) b = Op::op(b, v);
    }
    *all = warp_all<Op>(a);
    return warp_all<Op>(b);
}

// Sort items: an 8-byte pair while the keys have at most 32 bits.
struct __align__(8) Item32 {
    using Key = uint32_t;
    uint32_t key, val;
};
struct __align__(16) Item64 {
    using Key = uint64_t;
    uint64_t key;
    uint32_t val, pad;
};

// One stable pass on the key bits [shift, shift + bits) over the items that
// load(i, it) accepts, i < n, in two halves with a team barrier between them:
// sort_count counts the digits of the warps' segments, sort_place writes the
// items to out[0..count), returns count and ends with a barrier.
template <class Item, class Load, class Sm>
__device__ __forceinline__ void sort_count(const Team &t, Sm &s, int64_t n, Load load, int shift, int bits) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int bins = 1 << bits, mask = bins - 1;
    const Seg g = warp_seg(n);
    int *cnt = s.cnt() + warp * bins;
    for (int i = lane; i < bins; i += 32) cnt[i] = 0;
    if (threadIdx.x < kSortBins) { s.tot[threadIdx.x] = 0; s.bef[threadIdx.x] = 0; }
    __syncwarp();
    for (int64_t b = g.b; b < g.e; b += 128) {
        Item it[4];
        bool ok[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int64_t i = b + 32 * j + lane;
            ok[j] = i < g.e && load(i, it[j]);
        }
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (ok[j]) atomicAdd(&cnt[(int)(it[j].key >> shift) & mask], 1);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < bins; d += kTT) {
        int run = 0;
#pragma unroll 8
        for (int w = 0; w < kTW; w++) {
            const int c = s.cnt()[w * bins + d];
            s.cnt()[w * bins + d] = run;
            run += c;
        }
        if constexpr (Sm::kCluster) s.row[d] = run;
        else t.hist[blockIdx.x * bins + d] = run;
    }
}

template <class Item, class Load, class Sm>
__device__ __forceinline__ int64_t sort_place(const Team &t, Sm &s, int64_t n, Load load, int shift, int bits,
                                              Item *out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int mask = (1 << bits) - 1;
    const int bins = 1 << bits;
    const Seg g = warp_seg(n);
    int *cnt = s.cnt() + warp * bins;
    // first position of every digit: the totals of the smaller digits, and of
    // this digit in the CTAs before
    {
        const int d = threadIdx.x & mask;
        int tot = 0, bef = 0;
        for (int c = threadIdx.x >> bits; c < (int)gridDim.x; c += kTT >> bits) {
            int v;
            if constexpr (Sm::kCluster) v = remote(&s.row[d], c);
            else v = t.hist[c * bins + d];
            tot += v;
            if (c < (int)blockIdx.x) bef += v;
        }
        if (tot) atomicAdd(&s.tot[d], tot);
        if (bef) atomicAdd(&s.bef[d], bef);
    }
    __syncthreads();
    const int mine = threadIdx.x < kSortBins ? s.tot[threadIdx.x] : 0;
    const long long inc = warp_incl<Sum>(mine);
    if (lane == 31) s.w[warp] = inc;
    __syncthreads();
    const long long winc = warp_incl<Sum>(s.w[lane]);
    const long long wbef = __shfl_sync(0xffffffffu, winc, warp > 0 ? warp - 1 : 0);
    const int64_t count = __shfl_sync(0xffffffffu, winc, 31);
    if (threadIdx.x < kSortBins) s.bef[threadIdx.x] += (int)((warp > 0 ? wbef : 0) + inc - mine);
    __syncthreads();
    for (int64_t b = g.b; b < g.e; b += 128) {
        Item it[4];
        bool ok[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int64_t i = b + 32 * j + lane;
            ok[j] = i < g.e && load(i, it[j]);
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            if (b + 32 * j >= g.e) break;             // (uniform over the warp: short segments skip the rest)
            const int d = ok[j] ? (int)(it[j].key >> shift) & mask : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const int rank = __popc(peers & lt);
            int first = 0;
            if (ok[j]) first = cnt[d];
            __syncwarp();
            if (ok[j]) {
                out[s.bef[d] + first + rank] = it[j];
                if (rank == 0) cnt[d] = first + __popc(peers);
            }
            __syncwarp();
        }
    }
    sync(t);
    return count;
}

template <class Item, class Load, class Sm>
__device__ __forceinline__ int64_t sort_pass(const Team &t, Sm &s, int64_t n, Load load, int shift, int bits,
                                             Item *out) {
    sort_count<Item>(t, s, n, load, shift, bits);
    sync(t);
    return sort_place<Item>(t, s, n, load, shift, bits, out);
}

// Stable sort by the low `bits` key bits of the items load accepts; the
// result is returned (A or B), its length in *count.
template <class Item, class Load, class Sm>
__device__ __forceinline__ const Item *sort(const Team &t, Sm &s, int64_t n, Load load, int bits, Item *A, Item *B,
                                            int64_t *count) {
    const int passes = bits <= 8 ? 1 : (bits + 7) / 8;
    const int per = max(1, (bits + passes - 1) / passes);
    const int64_t cnt = sort_pass(t, s, n, load, 0, per, A);
    Item *src = A, *dst = B;
    for (int p = 1; p < passes; p++) {
        const Item *from = src;
        sort_pass<Item>(
            t, s, cnt, [from](int64_t i, Item &it) { it = from[i]; return true; }, p * per, min(per, bits - p * per),
            dst);
        Item *x = src; src = dst; dst = x;
    }
    *count = cnt;
    return src;
}

__device__ __forceinline__ int bits_of(uint32_t x) { return 32 - __clz((int)x); }

}  // namespace team

// CTAs of the team kernels of a binding of n nodes: one up to 2048 nodes (its
// barriers are __syncthreads), else one per 1024 nodes; up to kClusterMax of
// them as one cluster (its hardware barrier takes a fraction of the 1.2 us of a
// grid barrier), for graphs of up to 65536 nodes; beyond, at most one per SM.
// A cooperative launch starts only when all its CTAs fit at once, so
// contexts that refine side by side (the batches of a mixed context) share
// the SMs between them; with the whole GPU each, they would wait for one
// another at every launch (1024 Chung-Lu graphs in five batches: 18.0 ms at
// 30 CTAs each, 20.5 ms at 152; one batch alone: 18.0 ms at 152, 29.5 ms at 30).
// sms: the device's SMs, at most kTeamMax.
inline int team_size(int64_t n, int beside, int sms) {
    if (n <= 2048) return 1;
    const int64_t want = ceil_div(n, (int64_t)1024);
    if (n <= 65536) return (int)std::min<int64_t>(want, team::kClusterMax);
    return (int)std::min<int64_t>(std::max(team::kClusterMax + 1, sms / std::max(1, beside)), want);
}

template <typename Args>
inline void launch_team(void (*kern)(Args), const Args &a, int size, cudaStream_t s, size_t shm = 0) {
    if (shm > 0) kernel_setup((const void *)kern, -1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size);
    cfg.blockDim = dim3(team::kTT);
    cfg.dynamicSmemBytes = shm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    if (size > team::kClusterMax) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    } else {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)size;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        if (size > 8) UPR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    }
    cfg.attrs = attr;
    cfg.numAttrs = size > 1 ? 1 : 0;
    UPR_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
    UPR_LAUNCH_CHECK();
}

}  // namespace upr
