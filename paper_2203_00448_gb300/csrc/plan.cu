// plan.cu -- host side of greedy_by_size (plan.cuh): workspace sizes and the
// launches of the planner alone.  The fused pass is in plan_fused.cu, so that
// the two sets of kernels compile in parallel.
#include "plan.cuh"

namespace mp {

// One workspace size serves both the planner and the fused entry point;
// batches of large traces take the grid-wide dataflow (grid.cu).
size_t plan_workspace_bytes(const mp_batch& bt) {
    return grid_path(bt) ? grid_workspace_bytes(bt) : plan_workspace(bt).total;
}

cudaError_t launch_plan(const mp_batch& bt, int32_t policy, int64_t* offsets, int64_t* plan_peak,
                        int32_t* status, void* workspace, cudaStream_t stream) {
    if (grid_path(bt)) return launch_grid_plan(bt, policy, offsets, plan_peak, status, workspace, -1, stream);
    const PlanOut out{policy, offsets, plan_peak, status, nullptr, nullptr, nullptr, nullptr};
    return launch_any<false>(bt, out, workspace, stream);
}

}  // namespace mp

#ifdef MP_TEST_HOOKS
// Test builds only: greedy_by_size as mp_plan_greedy_by_size, except that the
// member at alloc-order position hold_pos of trace hold_trace is never queued
// (the grid-wide planner for batches of a few large traces, the CTA tier's
// ready queue otherwise), so the planner's bounded waits run out and that
// trace reports MP_ETIMEOUT while the others are planned as usual.  With
// hold_trace kHoldBarrier a CTA of the grid-wide planner never arrives at the
// barriers between the stages that prepare a batch for its phases.
extern "C" __attribute__((visibility("default"))) mp_status mp_test_plan_hold(
    const mp_batch* batch, mp_fit_policy policy, int64_t* offsets, int64_t* plan_peak, int32_t* trace_status,
    void* workspace, size_t workspace_bytes, int32_t hold_trace, int32_t hold_pos, void* stream) {
    static const int32_t none[2] = {-1, -1};
    static int32_t held[2];
    if (batch == nullptr || workspace_bytes < mp::plan_workspace_bytes(*batch)) return MP_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (mp::grid_path(*batch)) {
        const int64_t slot = hold_trace == mp::kHoldBarrier ? mp::kHoldBarrier
                                                            : (int64_t)hold_trace * batch->max_tensors + hold_pos;
        return mp::launch_grid_plan(*batch, policy, offsets, plan_peak, trace_status, workspace, (int32_t)slot, st) ==
                       cudaSuccess
                   ? MP_OK
                   : MP_ECUDA;
    }
    held[0] = hold_trace;
    held[1] = hold_pos;
    cudaError_t e = cudaMemcpyToSymbol(mp::g_test_hold, held, sizeof(held));
    if (e == cudaSuccess) e = mp::launch_plan(*batch, policy, offsets, plan_peak, trace_status, workspace, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    const cudaError_t e2 = cudaMemcpyToSymbol(mp::g_test_hold, none, sizeof(none));
    return e == cudaSuccess && e2 == cudaSuccess ? MP_OK : MP_ECUDA;
}

// Test builds only: greedy_by_size, except that the member at alloc-order
// position hold_pos of trace hold_trace is never placed if a team of warps
// walks its chain (a trace placed in phases), so that the team's bounded waits
// run out.
extern "C" __attribute__((visibility("default"))) mp_status mp_test_plan_team_hold(
    const mp_batch* batch, mp_fit_policy policy, int64_t* offsets, int64_t* plan_peak, int32_t* trace_status,
    void* workspace, size_t workspace_bytes, int32_t hold_trace, int32_t hold_pos, void* stream) {
    if (batch == nullptr || workspace_bytes < mp::plan_workspace_bytes(*batch)) return MP_EINVAL;
    const int32_t none[2] = {-1, -1}, held[2] = {hold_trace, hold_pos};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemcpyToSymbol(mp::phases::g_test_team_hold, held, sizeof(held));
    if (e == cudaSuccess) e = mp::launch_plan(*batch, policy, offsets, plan_peak, trace_status, workspace, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    const cudaError_t e2 = cudaMemcpyToSymbol(mp::phases::g_test_team_hold, none, sizeof(none));
    return e == cudaSuccess && e2 == cudaSuccess ? MP_OK : MP_ECUDA;
}
#endif
