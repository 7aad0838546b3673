// sw_devplan.cu -- the planner kernels (sw_plan.cuh), one block each.
#include "sw_plan.cuh"

namespace swgb {

__global__ void __launch_bounds__(kPlanThreads) k_plan_score(const ClassInfo *__restrict__ info, const PlanParams pp,
                                                             DevScorePlan *__restrict__ out,
                                                             int32_t *__restrict__ status)
{
    plan_score(info, pp, out, status);
}

__global__ void __launch_bounds__(kPlanThreads) k_plan_tb(const ClassInfo *__restrict__ info,
                                                          const TbClassInfo *__restrict__ ti,
                                                          const DevScorePlan *__restrict__ sp, const PlanParams pp,
                                                          DevTbPlan *__restrict__ out, int32_t *__restrict__ status)
{
    plan_tb(info, ti, sp, pp, out, status);
}

int launch_plan_score(const ClassInfo *info, const PlanParams &pp, DevScorePlan *out, int32_t *status,
                      cudaStream_t st)
{
    k_plan_score<<<1, kPlanThreads, 0, st>>>(info, pp, out, status);
    count_launch();
    return launch_status();
}

int launch_plan_tb(const ClassInfo *info, const TbClassInfo *ti, const DevScorePlan *sp, const PlanParams &pp,
                   DevTbPlan *out, int32_t *status, cudaStream_t st)
{
    k_plan_tb<<<1, kPlanThreads, 0, st>>>(info, ti, sp, pp, out, status);
    count_launch();
    return launch_status();
}

}  // namespace swgb
