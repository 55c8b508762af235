// vlb_step_bf16.cu -- time-step launches for populations stored in bfloat16, FP32 arithmetic.
#include "vlb_step.cuh"

namespace vlb {

cudaError_t launch_step_bf16(const vlb_sim *sim, int odd, cudaStream_t s) {
  return sim->mesh->md.q == 9 ? launch_step_t<9, __nv_bfloat16, float>(sim, odd, s)
                              : launch_step_t<19, __nv_bfloat16, float>(sim, odd, s);
}

}  // namespace vlb
