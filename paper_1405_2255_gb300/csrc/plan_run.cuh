// plan_run.cuh -- how a P2P work plan gets its scratch (host only, no CUDA calls).
#pragma once
#include <stddef.h>

namespace gb3 {

enum PlanEnd {
    kPlanRan,
    kPlanTooLarge,  // beyond the plan's index ranges
    kPlanNoRoom,    // no memory for its scratch
    kPlanUnfit      // more than it had asked for (cannot be: the sizes follow from the lists)
};

// fixed: the scratch a plan needs to find out its size; run(parts) plans and computes and returns the bytes it
// needs (more than have(): nothing was computed; ~0: too large); grow(bytes) makes have() at least that, or
// returns an error.  parts: the pieces of small systems shared by several warps, which takes more
// scratch and indexes; without room for that they stay whole.
template <class Run, class Grow, class Have>
PlanEnd run_plan(size_t fixed, bool parts, Run run, Grow grow, Have have) {
    PlanEnd end = kPlanUnfit;
    for (int whole = parts ? 0 : 1; whole < 2; ++whole) {
        size_t need = fixed;
        end = kPlanUnfit;
        for (int attempt = 0; attempt < 2; ++attempt) {
            if (grow(need)) {
                end = kPlanNoRoom;
                break;
            }
            need = run(whole == 0);
            if (need == ~(size_t)0) {
                end = kPlanTooLarge;
                break;
            }
            if (need <= have()) return kPlanRan;
        }
    }
    return end;
}

}  // namespace gb3
