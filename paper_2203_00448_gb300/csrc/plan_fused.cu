// plan_fused.cu -- the launches of the fused pass (plan.cuh): live profile,
// greedy_by_size plan and its validation.
#include "plan.cuh"

namespace mp {

cudaError_t launch_plan_fused(const mp_batch& bt, int32_t policy, int64_t* profile, int64_t* peak_lb,
                              int64_t* offsets, int64_t* plan_peak, int32_t* verdict, int32_t* conflict,
                              int32_t* status, void* workspace, cudaStream_t stream) {
    if (grid_path(bt))
        return launch_grid_fused(bt, policy, profile, peak_lb, offsets, plan_peak, verdict, conflict, status,
                                 workspace, stream);
    const PlanOut out{policy, offsets, plan_peak, status, profile, peak_lb, verdict, conflict};
    return launch_any<true>(bt, out, workspace, stream);
}

}  // namespace mp
