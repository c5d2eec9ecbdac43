// vkt_walk3.cu -- the walking separable kernels of k = 3 (vkt_walk.cuh).
#include "vkt_walk.cuh"

namespace vkt {

vktError launch_walk_k3(const Job& job, const float* gx, const float* gy, const float* gz, const Ctx& ctx,
                        bool* taken)
{
    return launch_walk_k<3>(job, gx, gy, gz, ctx, taken);
}

}  // namespace vkt
