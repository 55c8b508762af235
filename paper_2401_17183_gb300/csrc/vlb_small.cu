// vlb_small.cu -- dispatch of the multi-step kernel for small meshes.
#include "vlb_small.cuh"

namespace vlb {

cudaError_t launch_steps_small(vlb_sim *sim, int64_t nsteps, int64_t *done, cudaStream_t s) {
  *done = 0;
  const vlb_mesh *m = sim->mesh;
  const int q = m->md.q;
  // us a step, one launch each / one launch for all: FP32 D2Q9 2,048 cells 4.2 / 2.4, 32,768
  // 4.2 / 2.8, 60,000 6.2 / 3.8; D3Q19 57,600 6.2 / 4.7 (plane), 8.2 / 5.1 (records per
  // cell); FP64 D2Q9 4,096 12.3 / 9.1, 32,768 18.5 / 16.8, alike from 60,000 on
  if (nsteps < 2 || m->ncell > kSmallCells) return cudaSuccess;
  auto go = [&](auto qt, auto tag) {
    constexpr int Q = decltype(qt)::value;
    using R = typename decltype(tag)::type;
    if constexpr (Q == 19) {
      if (sim->plane && m->extruded) return launch_small_t<Q, R, true, true>(sim, nsteps, done, s);
    }
    return sim->plane ? launch_small_t<Q, R, true, false>(sim, nsteps, done, s)
                      : launch_small_t<Q, R, false, false>(sim, nsteps, done, s);
  };
  auto lat = [&](auto tag) {
    return q == 9 ? go(std::integral_constant<int, 9>(), tag) : go(std::integral_constant<int, 19>(), tag);
  };
  if (q != 9 && q != 19) return cudaSuccess;
  if (sim->p.precision == VLB_F32) return lat(TypeTag<float>{});
  if (sim->p.precision == VLB_F64) return lat(TypeTag<double>{});
  return cudaSuccess;
}

}  // namespace vlb
