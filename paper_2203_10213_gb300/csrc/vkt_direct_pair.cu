// vkt_direct_pair.cu -- the direct kernels of the listed mode with high and low weights
// (vkt_direct.cuh).
#include "vkt_direct.cuh"

namespace vkt {

vktError launch_direct_pair(const Job& job, const float* w, int k, const Ctx& ctx, const ListPlan& plan)
{
    switch (k) {
    case 3: return dir::launch_k<3, false, dir::M_PAIR>(job, w, ctx, &plan);
    case 5: return dir::launch_k<5, false, dir::M_PAIR>(job, w, ctx, &plan);
    case 7: return dir::launch_k<7, false, dir::M_PAIR>(job, w, ctx, &plan);
    case 9: return dir::launch_k<9, false, dir::M_PAIR>(job, w, ctx, &plan);
    default: return VKT_ERROR_UNSUPPORTED;
    }
}

}  // namespace vkt
