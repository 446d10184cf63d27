// The grid barrier of the team launches (team.cuh) by itself, for inspection.
#include "team.cuh"

namespace upr {
namespace {

struct BarrierProbe {
    Team team;
    int absent;
    int32_t *passed;
};

__global__ void __launch_bounds__(team::kTT, 1) k_barrier_probe(const BarrierProbe a) {
    if ((int)(gridDim.x - blockIdx.x) <= a.absent) return;       // (never arrives)
    team::sync(a.team);
    if (threadIdx.x == 0) atomicAdd(a.passed, 1);
}

}  // namespace

bool barrier_probe(const Team &t, int absent, int32_t *passed, cudaStream_t s) {
    if (t.size <= team::kClusterMax || absent < 0 || absent >= t.size) return false;
    UPR_CUDA(cudaMemsetAsync(passed, 0, sizeof(int32_t), s));
    launch_team(k_barrier_probe, BarrierProbe{t, absent, passed}, t.size, s);
    return true;
}

}  // namespace upr
