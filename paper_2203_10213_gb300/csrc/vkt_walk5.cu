// vkt_walk5.cu -- the walking separable kernels of k = 5 (vkt_walk.cuh).
#include "vkt_walk.cuh"

namespace vkt {

vktError launch_walk_k5(const Job& job, const float* gx, const float* gy, const float* gz, const Ctx& ctx,
                        bool* taken)
{
    return launch_walk_k<5>(job, gx, gy, gz, ctx, taken);
}

}  // namespace vkt
