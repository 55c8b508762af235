// vlb_small.cuh -- many time steps of a small mesh in one launch. A mesh whose
// cells all fit on the device at once (one per thread) keeps its addresses and
// coefficient records from step to step and meets at a barrier over the blocks
// between steps, in place of a launch per step. Up to 16 blocks form one thread-block
// cluster and meet at its hardware barrier; more are launched cooperatively, so that
// every block is resident, and count themselves in global memory (that wait is bounded
// all the same). The arithmetic per cell is that of the step kernel, compiled apart: a
// compiler might contract a product and a sum otherwise, so the tests compare the two
// bit for bit in every form.
#pragma once

#include "vlb_step.cuh"

namespace vlb {

constexpr uint64_t kBarrierNs = 1000000000ull;

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// all blocks have arrived `target` times in total (counted from zero); false
// when that takes longer than kBarrierNs
__device__ __forceinline__ bool grid_barrier(unsigned *count, unsigned target) {
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    asm volatile("fence.acq_rel.gpu;\nred.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    uint64_t t0 = 0;
    for (unsigned spin = 0;; spin++) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
      if ((int)(v - target) >= 0) break;
      if ((spin & 255u) == 255u) {
        const uint64_t t = global_ns();
        if (t0 == 0) t0 = t;
        if (t - t0 > kBarrierNs) {
          ok = 0;
          break;
        }
      }
    }
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
  }
  return __syncthreads_and(ok);
}

// one cell's step: pull, collide, push (see step_tiles); populations are read
// past L1, which other SMs' writes do not reach
template <int Q, typename R, bool ODD, bool PLANE, bool EXT, typename RC>
__device__ __forceinline__ void small_cell(const StepArgs &a, const Addr<Q, int32_t> &ad, const RC &rc) {
  constexpr int D = Lat<Q>::D, H = Lat<Q>::H;
  using L = CoefLayout<Q>;
  R *f = static_cast<R *>(a.f);
  const int32_t cell = ad.cell;
  R N[Q], Np[Q];
#pragma unroll
  for (int av = 0; av < Q; av++) {
    const bool own = !ODD || av == 0 || ad.crosses(av, -1);
    N[av] = __ldcg(f + (own ? a.soff[av] + cell : a.soff[lat_opp<Q>(av)] + ad.nb(av, -1)));
  }
  CollideState<Q, R> cst;
  collide_cell<Q, R, true, false, PLANE || sizeof(R) == 8, RC, EXT>(N, rc, arg_r<R>(a.nref, a.nref_f),
                                                                    arg_r<R>(a.itau, a.itau_f),
                                                                    arg_r<R>(a.tol, a.tol_f), a.max_iter, Np, cst);
  if (!cst.conv) atomicOr(a.err, ERR_NOCONV);
  if (a.moving && ad.wall_cell()) {
    R uw[D], zero[D], gd[L::NS];
#pragma unroll
    for (int i = 0; i < D; i++) {
      if constexpr (!PLANE && sizeof(R) == 4)
        uw[i] = a.uw[(int64_t)cell * D + i];
      else
        uw[i] = rc[L::UW + i];
      zero[i] = R(0);
    }
#pragma unroll
    for (int i = 0; i < L::NS; i++) gd[i] = R(2) * rc[L::GH + i];
    EqParts<Q, R> ew;
    eq_parts<Q, R>(gd, uw, zero, ew);
    const R Jr2 = R(2) * rc[L::J] * cst.rho;
#pragma unroll
    for (int av = 1; av < Q; av++) {
      const int p = av <= H ? av : av - H;
      const R corr = Jr2 * lat_w<Q, R>(av) * eq_odd<Q, R>(ew, uw, p);
      const R nv = Np[av] - ((av <= H) ? corr : -corr);
      Np[av] = ad.crosses(av, 1) ? nv : Np[av];
    }
  }
#pragma unroll
  for (int av = 1; av < Q; av++) {
    const bool own = !ODD || ad.crosses(av, 1);
    f[own ? a.soff[lat_opp<Q>(av)] + cell : a.soff[av] + ad.nb(av, 1)] = Np[av];
  }
  f[cell] = Np[0];
}

// records a block keeps in shared memory: of its cells' columns (plane mode), or
// of its cells (FP64, with the rest state formed once a launch: 64 x 64 box 10.7 -> 9.8 us
// a step; an odd number of values against bank conflicts); FP32 records per cell stay in registers
template <int Q, typename R, bool PLANE>
struct SmallRecords {
  using L = CoefLayout<Q>;
  static constexpr int SRC = L::template stride<R, PLANE>();
  static constexpr int KEEP = PLANE ? L::SREST : SRC;            // values the step reads
  static constexpr int STRIDE = PLANE ? round4(KEEP) : (L::RW + L::H + 1) | 1;
  static size_t bytes(int T, int64_t nfast) {
    if (!PLANE) return sizeof(R) == 8 ? sizeof(R) * STRIDE * T : 0;
    return sizeof(R) * STRIDE * (size_t)((T - 1) / nfast + 2);
  }
};

// CLUSTER: all blocks form one thread-block cluster, whose barrier the hardware
// keeps; else they count themselves in global memory.
template <int Q, typename R, bool PLANE, bool EXT, int T, int MINB, bool CLUSTER>
__global__ void __launch_bounds__(T, MINB)
    k_steps_small(const __grid_constant__ StepArgs a, int32_t first, int32_t nsteps, unsigned *count) {
  constexpr bool CELLREC = !PLANE && sizeof(R) == 4;
  using SR = SmallRecords<Q, R, PLANE>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R *sm = reinterpret_cast<R *>(smem_raw);
  const int32_t c0 = (int32_t)blockIdx.x * T, ncell = (int32_t)a.ncell, cell = c0 + (int32_t)threadIdx.x;
  const bool live = cell < ncell;
  const Addr<Q, int32_t> ad = Addr<Q, int32_t>::linear(a.g, live ? cell : ncell - 1);
  using RC = typename std::conditional<CELLREC, CellRecord<Q>, PtrRecord<R>>::type;
  RC rc;
  if constexpr (CELLREC) {
    rc.load(static_cast<const float4 *>(a.coef), (int64_t)ad.cell);
    rc.form(a.cf.k6am, a.cf.kpe, a.cf.ktt);
  } else {
    const R *coef = static_cast<const R *>(a.coef);
    const int32_t nf = PLANE ? (int32_t)a.g.n[Lat<Q>::D - 1] : 1;
    const int32_t last = (c0 + T < ncell ? c0 + T : ncell) - 1;
    const int32_t r0 = c0 / nf, nrec = last / nf - r0 + 1;
    for (int32_t i = threadIdx.x; i < nrec * SR::KEEP; i += T) {
      const int32_t r = i / SR::KEEP, k = i - r * SR::KEEP;
      sm[r * SR::STRIDE + k] = coef[(int64_t)(r0 + r) * SR::SRC + k];
    }
    __syncthreads();
    rc.p = sm + (ad.cell / nf - r0) * SR::STRIDE;
    if constexpr (!PLANE && sizeof(R) == 8) {   // a thread's own cell
      using L = CoefLayout<Q>;
      double rr[Lat<Q>::H + 1], rw[Lat<Q>::H + 1], rsum;
      rest_state<Q>(rc, a.nref, rr, rw, rsum);
      R *const o = sm + (ad.cell - r0) * SR::STRIDE;
      __syncthreads();   // (threads past the last cell share its record)
#pragma unroll
      for (int q = 0; q <= Lat<Q>::H; q++) {
        o[L::RR + q] = rr[q];
        o[L::RW + q] = rw[q];
      }
      o[L::RR + Lat<Q>::H + 1] = rsum;
      __syncthreads();
    }
  }
#pragma unroll 1
  for (int32_t k = 0; k < nsteps; k++) {
    if constexpr (CELLREC) rc.opaque();
    if (live) {
      if ((first + k) & 1)
        small_cell<Q, R, true, PLANE, EXT, RC>(a, ad, rc);
      else
        small_cell<Q, R, false, PLANE, EXT, RC>(a, ad, rc);
    }
    if constexpr (CLUSTER) {
      __syncwarp();
      asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else if (k + 1 < nsteps && !grid_barrier(count, (unsigned)(k + 1) * gridDim.x)) {
      if (threadIdx.x == 0) atomicOr(a.err, ERR_BARRIER);
      return;
    }
  }
}

// Threads per block: FP32 128; FP64 one warp, so that as many SMs as possible
// share the FP64 operations.
template <typename R>
constexpr int small_threads() {
  return sizeof(R) == 8 ? 32 : 128;
}

// Blocks of one cluster: 16 at most (beyond 8 by permission)
constexpr int kClusterMax = 16;

// can a cluster of nblk blocks of this kernel run on the current device? (asked
// once per kernel, size, shared memory and device)
static bool cluster_fits(const void *kern, int nblk, int threads, size_t smem) {
  static std::mutex mu;
  static std::vector<std::tuple<const void *, int, size_t, int, bool>> cache;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  for (const auto &e : cache)
    if (std::get<0>(e) == kern && std::get<1>(e) == nblk && std::get<2>(e) == smem && std::get<3>(e) == dev)
      return std::get<4>(e);
  bool ok = smem <= 48 * 1024;
  if (ok && nblk > 8)
    ok = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  if (ok) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)nblk;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)nblk);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    ok = cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0;
  }
  if (!ok) cudaGetLastError();   // (a query that failed leaves no error behind)
  cache.emplace_back(kern, nblk, smem, dev, ok);
  return ok;
}

// One cluster over the whole mesh, T cells per block; *done = 0 when it does not fit.
template <int Q, typename R, bool PLANE, bool EXT, int T>
cudaError_t launch_cluster_t(vlb_sim *sim, int32_t first, int32_t n, int64_t *done, cudaStream_t s) {
  const vlb_mesh *m = sim->mesh;
  const size_t smem = SmallRecords<Q, R, PLANE>::bytes(T, m->md.n[m->md.dim - 1]);
  auto kern = k_steps_small<Q, R, PLANE, EXT, T, 1, true>;
  const int64_t nblk = (m->ncell + T - 1) / T;
  if (nblk > kClusterMax || !cluster_fits(reinterpret_cast<const void *>(kern), (int)nblk, T, smem)) return cudaSuccess;
  StepArgs a = make_step_args<Q>(sim, T);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)nblk;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)nblk);
  cfg.blockDim = dim3(T);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a, first, n, (unsigned *)nullptr);
  if (e == cudaSuccess) *done = n, sim->path = PATH_CLUSTER;
  return e;
}

// Advances the simulation by up to `nsteps` steps in one launch if its cells fit on the
// device at once; *done is the number of steps launched (0: take the step kernel).
template <int Q, typename R, bool PLANE, bool EXT>
cudaError_t launch_small_t(vlb_sim *sim, int64_t nsteps, int64_t *done, cudaStream_t s) {
  constexpr int T = small_threads<R>();
  constexpr int MINB = sizeof(R) == 8 ? 8 : Q == 9 ? 4 : 3;
  const vlb_mesh *m = sim->mesh;
  int32_t first = (int32_t)(sim->t & 1), n = (int32_t)(nsteps < kSmallSteps ? nsteps : kSmallSteps);
  *done = 0;
  if constexpr (sizeof(R) == 4) {
    // FP32 meshes of up to 16 blocks: one cluster (2,048 D2Q9 cells:
    // 1.29 us a step, against 2.43 with the counter in global memory; 4,096 cells 1.72)
    cudaError_t e = cudaSuccess;
    if (m->ncell <= kClusterMax * 128)
      e = launch_cluster_t<Q, R, PLANE, EXT, 128>(sim, first, n, done, s);
    else if (m->ncell <= kClusterMax * 256)
      e = launch_cluster_t<Q, R, PLANE, EXT, 256>(sim, first, n, done, s);
    if (e != cudaSuccess || *done > 0) return e;
  }
  const size_t smem = SmallRecords<Q, R, PLANE>::bytes(T, m->md.n[m->md.dim - 1]);
  auto kern = k_steps_small<Q, R, PLANE, EXT, T, MINB, false>;
  const int64_t nblk = (m->ncell + T - 1) / T;
  if (smem > 96 * 1024 || nblk > resident_blocks(reinterpret_cast<const void *>(kern), smem, T)) return cudaSuccess;
  StepArgs a = make_step_args<Q>(sim, T);
  unsigned *count = reinterpret_cast<unsigned *>(sim->d_err) + kBarrierWord;
  void *args[] = {&a, &first, &n, &count};
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(kern), dim3((unsigned)nblk), dim3(T), args, smem, s);
  if (e == cudaSuccess) *done = n, sim->path = PATH_COOPERATIVE;
  return e;
}

}  // namespace vlb
