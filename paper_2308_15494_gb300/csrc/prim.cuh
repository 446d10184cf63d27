// Block-wide scan of 256-thread CTAs.
#pragma once

#include "kernels.h"

namespace upr {
namespace prim {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

struct OpSum {
    template <typename T> __device__ __forceinline__ static T apply(T a, T b) { return a + b; }
    template <typename T> __device__ __forceinline__ static T identity() { return T(0); }
};

// Block-wide exclusive scan of one value per thread; returns the exclusive
// prefix, *total receives the block aggregate.
template <typename Op, typename T>
__device__ __forceinline__ T block_exclusive(T v, T *s_warp, T *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc = Op::template apply<T>(u, inc);
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < kWarps ? s_warp[lane] : Op::template identity<T>();
        for (int o = 1; o < kWarps; o <<= 1) {
            T u = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w = Op::template apply<T>(u, w);
        }
        if (lane < kWarps) s_warp[lane] = w;   // inclusive over warps
    }
    __syncthreads();
    T warp_prefix = warp == 0 ? Op::template identity<T>() : s_warp[warp - 1];
    *total = s_warp[kWarps - 1];
    T excl = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) excl = Op::template identity<T>();
    __syncthreads();
    return Op::template apply<T>(warp_prefix, excl);
}

}  // namespace prim
}  // namespace upr
