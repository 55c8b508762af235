// vlb_step.cu -- dispatch of the time step over storage types (FP64 here; the
// FP32, half and bfloat16 kernels are compiled in files of their own, in parallel).
#include "vlb_step.cuh"

namespace vlb {

cudaError_t launch_step_f32(const vlb_sim *sim, int odd, cudaStream_t s);
cudaError_t launch_step_f16(const vlb_sim *sim, int odd, cudaStream_t s);
cudaError_t launch_step_bf16(const vlb_sim *sim, int odd, cudaStream_t s);

cudaError_t launch_step(const vlb_sim *sim, int odd, cudaStream_t s) {
  switch (sim->p.precision) {
    case VLB_F64:
      return sim->mesh->md.q == 9 ? launch_step_t<9, double, double>(sim, odd, s)
                                  : launch_step_t<19, double, double>(sim, odd, s);
    case VLB_F32: return launch_step_f32(sim, odd, s);
    case VLB_F16: return launch_step_f16(sim, odd, s);
    default: return launch_step_bf16(sim, odd, s);
  }
}

}  // namespace vlb
