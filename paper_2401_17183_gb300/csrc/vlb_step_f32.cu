// vlb_step_f32.cu -- time-step launches for FP32 populations.
#include "vlb_step.cuh"

namespace vlb {

cudaError_t launch_step_f32(const vlb_sim *sim, int odd, cudaStream_t s) {
  return sim->mesh->md.q == 9 ? launch_step_t<9, float, float>(sim, odd, s)
                              : launch_step_t<19, float, float>(sim, odd, s);
}

}  // namespace vlb
