// adjoint_plan.h -- which states an adjoint call keeps and where. Host code without CUDA.
#pragma once

#include <algorithm>
#include <cmath>

namespace lbmv {
namespace adj {

// Device bytes of states kept instead of recomputed, where they can be had.
constexpr long long kKeep = 512LL << 20;

// The device holds every state after f(0) (nothing is recomputed; the host keeps f(0)), or a
// whole segment of `every` states (every step recomputed once), or sub-segments of ceil(sqrt)
// of them, whose first states are kept on the host too while a segment is processed
// (recomputed twice). dense: the checkpoints and a whole segment on the device.
enum class Keep { all, segment, subsegment };

struct Plan {
    Keep keep;
    int K2;                  // states of a (sub-)segment on the device
    long long seg;           // states of the device's segment buffer
    long long device_ck;     // checkpoints on the device
    long long host_states;   // states in pinned host memory
};

inline Plan make_plan(Keep keep, bool dense, int nsteps, int every) {
    const int K = std::min(every, nsteps), nck = (nsteps - 1) / every + 1;
    const int K2 = keep == Keep::subsegment ? std::max(1, (int)std::ceil(std::sqrt((double)K))) : K;
    if (dense) return Plan{Keep::segment, K, K, nck, 0};
    if (keep == Keep::all) return Plan{keep, K, std::max(1, nsteps - 1), 0, 1};
    return Plan{keep, K2, K2, 0, (long long)nck + (keep == Keep::segment ? 0 : (K - 1) / K2 + 1)};
}

// Allocates what a call needs: the plan that recomputes least among those whose states take at
// most kKeep bytes; where the device does not have that much, the ones that take less in turn,
// down to sub-segments. allocate(plan) returns 0 (it has the memory), 1 (the device has not) or
// another error. Returns its last answer.
template <typename Allocate>
int allocate_plan(Plan& plan, bool dense, int nsteps, int every, long long state_bytes, Allocate allocate) {
    if (dense) return allocate(plan = make_plan(Keep::segment, true, nsteps, every));
    auto fits = [&](long long states) { return states * state_bytes <= kKeep; };
    int r = 1;
    if (fits(nsteps - 1LL)) r = allocate(plan = make_plan(Keep::all, false, nsteps, every));
    if (r == 1 && fits(std::min(every, nsteps))) r = allocate(plan = make_plan(Keep::segment, false, nsteps, every));
    if (r == 1) r = allocate(plan = make_plan(Keep::subsegment, false, nsteps, every));
    return r;
}

}  // namespace adj
}  // namespace lbmv
