// vlb_step_f16.cu -- time-step launches for populations stored in IEEE half, FP32 arithmetic.
#include "vlb_step.cuh"

namespace vlb {

cudaError_t launch_step_f16(const vlb_sim *sim, int odd, cudaStream_t s) {
  return sim->mesh->md.q == 9 ? launch_step_t<9, __half, float>(sim, odd, s)
                              : launch_step_t<19, __half, float>(sim, odd, s);
}

}  // namespace vlb
