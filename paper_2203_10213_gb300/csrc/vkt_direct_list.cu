// vkt_direct_list.cu -- the direct kernels of the listed modes with one float32 weight per tap
// (vkt_direct.cuh), and the choice between the listed modes.
#include "vkt_direct.cuh"

namespace vkt {

vktError launch_direct_listed(const Job& job, const float* w, int k, const Ctx& ctx, bool* taken)
{
    // k = 1 is one product; a float32 source has no bound on its values
    *taken = false;
    ListPlan plan;
    if (k < 3 || job.sfmt == FMT_F32 ||
        !make_list_plan(plan, k, w, job.sfmt, job.a0, job.a0lo, job.a1, job.a1lo))
        return VKT_NO_ERROR;
    *taken = true;
    if (plan.pair) return launch_direct_pair(job, w, k, ctx, plan);
    switch (k) {
    case 3:
        return dir::direct_small(job, ctx.sms) ? dir::launch_k<3, false, dir::M_LIST, 1>(job, w, ctx, &plan)
                                               : dir::launch_k<3, false, dir::M_LIST>(job, w, ctx, &plan);
    case 5: return dir::launch_k<5, false, dir::M_LIST>(job, w, ctx, &plan);
    case 7: return dir::launch_k<7, false, dir::M_LIST>(job, w, ctx, &plan);
    default: return dir::launch_k<9, false, dir::M_LIST>(job, w, ctx, &plan);
    }
}

}  // namespace vkt
