// step.cu -- the cold-started step kernels (every substep's solve starts from
// zero impulses) and the host entry points over all compiled shapes; the
// kernel itself is in step_kernel.cuh, its warm-started instances in
// step_warm.cu.
#include "step_kernel.cuh"

namespace ih {
bool step_variant_supported(int group, int cpl) {
#define IH_SUP(T, C) if (group == T && cpl == C) return true;
    IH_STEP_VARIANTS(IH_SUP)
#undef IH_SUP
    return false;
}

int step_variant_list(StepVariant *out, int cap) {
    int n = 0;
#define IH_LIST(T, C) if (n < cap) out[n] = StepVariant{T, C, 0, 0, false, 1}; ++n;
    IH_STEP_VARIANTS(IH_LIST)
#undef IH_LIST
    return n;
}

cudaError_t step_prepare(const StepVariant &v, int s_max, int c_max, bool warm, int clp_cap, int *blocks_per_sm) {
    return warm ? step_prepare_warm(v, s_max, c_max, clp_cap, blocks_per_sm)
                : prepare_w<false>(v, s_max, c_max, clp_cap, blocks_per_sm);
}

int step_stage_capacity(const StepVariant &v, int c_max) { return stage_capacity(v.lanes, c_max); }
bool step_has_first(const StepVariant &v, int c_max) {
    return v.lanes == 32 && v.per_sm == kFewBlocks && c_max > kSlots * 32;
}
int step_spill_rows(const StepVariant &v, int c_max) { return spill_rows(v.lanes, c_max); }

cudaError_t launch_step(const StepArgs &a, const StepVariant &v, int grid, int s_max, cudaStream_t s) {
    return a.cfg.warm ? launch_step_warm(a, v, grid, s_max, s) : launch_w<false>(a, v, grid, s_max, s);
}

}  // namespace ih
