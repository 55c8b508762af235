// vlb_nn_tc.cuh -- the warm-start network's 3x3 convolutions on the
// fifth-generation tensor cores (tcgen05): forward, gradient with respect to
// the input and gradient with respect to the weights.
//
// Operands are bfloat16 and accumulators FP32 in tensor memory. Gradients of
// activations are FP32: each is split into three bfloat16 planes (hi + mid + lo: all 24
// bits of a value of 2^-109 or more; below, the last ones are less than bfloat16's smallest
// value), and since the other operand of either
// gradient (weights, activations) is stored in bfloat16, the sum of the three
// planes' products is the product of the FP32 gradient.
//
// Shared-memory operands are in the no-swizzle K-major layout of core matrices
// (8 rows x 16 bytes): row r and 8-element K group k at k * LBO + r * 16 bytes
// (SBO = 128), so that threads holding consecutive rows store consecutive
// 16-byte pieces. LBO is the bytes of one K group, padded by 16 where threads
// with consecutive K groups store together.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "vlb_chain.cuh"

namespace nn {

using bf16 = __nv_bfloat16;

constexpr int kTcM = 128;                 // rows of one MMA
constexpr int kTcCh = 16;                 // channels per pipeline step of the convolution
constexpr int kTcKG = kTcCh * 9 / 8;      // its K groups of 8 (18: nine MMAs of K = 16)
constexpr int kTcABytes = kTcKG * kTcM * 16;
constexpr uint64_t kTcWaitNs = 1000000000ull;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// shared-memory matrix descriptor: start address, leading (K-direction) and
// stride (M/N-direction) byte offsets, all >> 4; the descriptor version bit
// (46); no swizzle
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo = 128) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         ((uint64_t)1 << 46);
}
// instruction descriptor: FP32 accumulators, bfloat16 A and B, both K-major,
// N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t kTcAmn = 1u << 15;   // A is M-contiguous (core matrices of 8 K rows x 8 M values)
__host__ __device__ constexpr uint32_t umma_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTcM >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate ? 1 : 0));
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// wait until the mbarrier has completed the phase of the given parity, at
// most kTcWaitNs; returns whether it did
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  uint32_t done = 0;
  uint64_t t0 = 0;
  while (true) {
    asm volatile("{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
                 : "=r"(done)
                 : "r"(bar), "r"(parity)
                 : "memory");
    if (done) return true;
    const uint64_t t = gtimer();
    if (t0 == 0) t0 = t;
    if (t - t0 > kTcWaitNs) return false;
  }
}
// the same by a whole warp, whose lanes get one answer and go on together: what follows a wait
// may be an instruction of the whole warp (.sync.aligned), also where the time limit ends some
// lanes' wait and not others'
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity));
}
__device__ __forceinline__ void cp16(uint32_t sdst, const void *gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sdst), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp16_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// 16 tensor-memory columns of the warp's 32 lanes
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr)
      : "memory");
}
// set-up and end of a block: two mbarriers, COLS tensor-memory columns
template <int COLS>
__device__ __forceinline__ uint32_t tc_begin(uint64_t *bar, uint32_t *tslot) {
  static_assert(COLS >= 32 && (COLS & (COLS - 1)) == 0, "tensor-memory columns: a power of two, at least 32");
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[1])));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 32) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)), "r"(COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return *tslot;
}
template <int COLS>
__device__ __forceinline__ void tc_end(uint32_t tmem) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS));
}

// half h1 of word a in the low, half h2 of word b in the high 16 bits
template <int H1, int H2>
__device__ __forceinline__ uint32_t pick2(uint32_t a, uint32_t b) {
  return __byte_perm(a, b, (H1 ? 0x32 : 0x10) | ((H2 ? 0x76 : 0x54) << 8));
}
// where value (channel c of 8, tap k) of a pixel of a pair sits: its word and
// half. EVENW: words hold (x-2, x-1), (x, x+1), (x+2, x+3) of each of the three
// rows; else one word per tap holds the tap of both pixels.
template <bool EVENW, int PX>
__device__ constexpr int a_word(int n) {
  return (n / 9) * 9 + (EVENW ? (n % 9) / 3 * 3 + ((n % 3) + PX == 0 ? 0 : (n % 3) + PX == 3 ? 2 : 1) : n % 9);
}
template <bool EVENW, int PX>
__device__ constexpr int a_half(int n) {
  // PX 0 reads x-1, x, x+1; PX 1 reads x, x+1, x+2
  return EVENW ? ((n % 3) + PX == 0 ? 1 : (n % 3) + PX == 1 ? 0 : (n % 3) + PX == 2 ? 1 : 0) : PX;
}
template <bool EVENW, int PX, int M>
__device__ __forceinline__ uint32_t a_pair(const uint32_t (&w)[72]) {
  return pick2<a_half<EVENW, PX>(2 * M), a_half<EVENW, PX>(2 * M + 1)>(w[a_word<EVENW, PX>(2 * M)],
                                                                       w[a_word<EVENW, PX>(2 * M + 1)]);
}
template <bool EVENW, int PX, int G>
__device__ __forceinline__ void a_store(const uint32_t (&w)[72], unsigned char *dst) {
  if constexpr (G < 9) {
    *reinterpret_cast<uint4 *>(dst + G * (kTcM * 16)) =
        make_uint4(a_pair<EVENW, PX, 4 * G>(w), a_pair<EVENW, PX, 4 * G + 1>(w), a_pair<EVENW, PX, 4 * G + 2>(w),
                   a_pair<EVENW, PX, 4 * G + 3>(w));
    a_store<EVENW, PX, G + 1>(w, dst);
  }
}

// 3x3 convolution (zero padding) of the forward pass as an implicit GEMM:
//   out[b][n][p] = act(bias[n] + sum_c sum_tap wp[n][c][tap] in[b][c][p + off_tap]),
// FP32 accumulators, K in the order (c, tap). grid (H W / 128, Co / NB, B),
// block 128. wp: weights in pipeline-step order [ceil(C/16)][18 K groups][Co][8]
// (k_pack_weights).
//
// Bounded by the chain of a step: 16 channels' loads, the 128 x 144 patch matrix (36 KB)
// stored by the threads, a barrier, and the nine MMAs that read it with NB x 144 weights; the
// shared-memory pipes are 17 to 41% busy, the issue slots 17 to 31%, with one or two
// blocks of four warps on an SM.
// A thread keeps a pixel pair (rows i and 64 + i of the tile, so that a warp's
// stores are consecutive) and 8 of the 16 channels: 9 aligned 32-bit loads per
// channel give the 18 taps of both pixels, and byte permutes place them; the
// loads of step j + 1 are in flight while step j's MMAs run, its weights come
// by asynchronous copies. Warm-start network (width 64, 32 x 64, batch 32): the
// ten layers take 208 us (one K = 16 step per barrier with a 16-bit gather per
// tap and channel: 1,470 us); the sums are in the same order, bit for bit.
template <int NB, bool RELU, bool EVENW>
__global__ void __launch_bounds__(128) k_conv3_mma(const bf16 *__restrict__ in, int64_t ibs, int C,
                                                   const bf16 *__restrict__ wp, int Co, const float *__restrict__ bias,
                                                   bf16 *__restrict__ out, int64_t obs, int H, int W, int *err) {
  vlb::chain_begin();
  static_assert(NB % 16 == 0 && NB >= 16 && NB <= 256, "MMA N for M = 128");
  constexpr int TCOLS = NB <= 32 ? 32 : NB <= 64 ? 64 : NB <= 128 ? 128 : 256;
  constexpr int BBytes = kTcKG * NB * 16;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, warp = tid >> 5, pr = tid & 63, half = tid >> 6;
  const int HW = H * W, p0 = blockIdx.x * kTcM, p = p0 + 2 * pr, n0 = blockIdx.y * NB, b = blockIdx.z;
  const int nch = (C + kTcCh - 1) / kTcCh;
  const uint32_t tmem = tc_begin<TCOLS>(bar, &tslot);
  const bf16 *inb = in + (int64_t)b * ibs + p;
  // which of the nine words (or, per pixel, taps) lie inside the image
  uint32_t ok0 = 0, ok1 = 0;
  {
    const int y = p / W, x = p - y * W;
    for (int r = 0; r < 3; r++)
      for (int t = 0; t < 3; t++) {
        const bool rv = y + r - 1 >= 0 && y + r - 1 < H;
        if constexpr (EVENW) {
          if (rv && (t == 0 ? x > 0 : t == 2 ? x + 2 < W : true)) ok0 |= 1u << (3 * r + t);
        } else {
          if (rv && x + t - 1 >= 0 && x + t - 1 < W) ok0 |= 1u << (3 * r + t);
          const int y1 = x + 1 < W ? y : y + 1, x1 = x + 1 < W ? x + 1 : 0;
          if (y1 + r - 1 >= 0 && y1 + r - 1 < H && x1 + t - 1 >= 0 && x1 + t - 1 < W) ok1 |= 1u << (3 * r + t);
        }
      }
  }
  uint32_t w[72];
  auto load_a = [&](int j) {
    const int c0 = j * kTcCh + half * 8;
    const bf16 *q = inb + (int64_t)c0 * HW;
    const uint32_t m0 = c0 < C ? ok0 : 0u, m1 = c0 < C ? ok1 : 0u;
#pragma unroll
    for (int c = 0; c < 8; c++, q += HW) {
#pragma unroll
      for (int k = 0; k < 9; k++) {
        uint32_t v = 0;
        if constexpr (EVENW) {
          if ((m0 >> k) & 1) v = *reinterpret_cast<const uint32_t *>(q + (k / 3 - 1) * W + 2 * (k % 3 - 1));
        } else {
          const int o = (k / 3 - 1) * W + k % 3 - 1;
          if ((m0 >> k) & 1) v = *reinterpret_cast<const unsigned short *>(q + o);
          if ((m1 >> k) & 1) v |= (uint32_t) * reinterpret_cast<const unsigned short *>(q + 1 + o) << 16;
        }
        w[c * 9 + k] = v;
      }
    }
  };
  unsigned char *const sB = sm + 2 * kTcABytes;
  auto load_b = [&](int j) {
    const bf16 *src = wp + ((int64_t)j * kTcKG * Co + n0) * 8;
    const uint32_t dst = smem_u32(sB + (j & 1) * BBytes);
    for (int i = tid; i < kTcKG * NB; i += 128) {
      const int kg = i / NB, n = i - kg * NB;
      cp16(dst + i * 16, src + ((int64_t)kg * Co + n) * 8);
    }
  };
  load_b(0);
  load_a(0);
  bool ok = true, late = false;
  int issued = 0;
  for (int j = 0; j < nch; j++) {
    const int s = j & 1;
    unsigned char *dst = sm + s * kTcABytes + half * 9 * (kTcM * 16);
    a_store<EVENW, 0, 0>(w, dst + pr * 16);
    a_store<EVENW, 1, 0>(w, dst + (64 + pr) * 16);
    if (j + 1 < nch) load_a(j + 1);
    cp16_wait_all();
    // the stores and copies above are read by the tensor cores (async proxy)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (__syncthreads_or(late)) {
      ok = false;
      break;
    }
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a0 = smem_u32(sm + s * kTcABytes), b0 = smem_u32(sB + s * BBytes);
      // a last step of 8 channels: K = 72, padded to five MMAs with zeros
      const int nm = C - j * kTcCh >= kTcCh ? 9 : 5;
      for (int m = 0; m < nm; m++)
        umma(tmem, umma_desc(a0 + m * 2 * (kTcM * 16), kTcM * 16), umma_desc(b0 + m * 2 * (NB * 16), NB * 16),
             umma_idesc(NB), j > 0 || m > 0);
      umma_commit(smem_u32(&bar[s]));
    }
    issued = j + 1;
    if (j + 1 < nch) {
      // step j - 1's MMAs have read the stage that step j + 1 fills
      if (j >= 1) late = !mbar_wait(smem_u32(&bar[s ^ 1]), ((j - 1) >> 1) & 1);
      if (!late) load_b(j + 1);
    }
  }
  cp16_wait_all();
  // the last MMA done (its commit also covers every earlier one)
  late = issued > 0 && !mbar_wait(smem_u32(&bar[(issued - 1) & 1]), ((issued - 1) >> 1) & 1);
  if (__syncthreads_or(late)) ok = false;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (ok) {
    // epilogue: warp w reads TMEM lanes 32w.. (row r: pixel 2 r or 2 (r - 64) + 1),
    // the tile is transposed in shared memory and written in 16-byte pieces
    bf16 *so = reinterpret_cast<bf16 *>(sm);
    const int r = tid, px = r < 64 ? 2 * r : 2 * (r - 64) + 1;
#pragma unroll 1
    for (int c0 = 0; c0 < NB; c0 += 16) {
      uint32_t v[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
      for (int u = 0; u < 16; u++) {
        float f = __uint_as_float(v[u]) + (bias ? bias[n0 + c0 + u] : 0.0f);
        if (RELU) f = fmaxf(f, 0.0f);
        so[(c0 + u) * kTcM + px] = __float2bfloat16_rn(f);
      }
    }
    __syncthreads();
    constexpr int PP = kTcM / 8;
    for (int i = tid; i < NB * PP; i += 128) {
      const int c = i / PP, k = i - c * PP;
      *reinterpret_cast<uint4 *>(out + (int64_t)b * obs + (int64_t)(n0 + c) * HW + p0 + k * 8) =
          *reinterpret_cast<const uint4 *>(so + c * kTcM + k * 8);
    }
  } else if (tid == 0) {
    atomicOr(err, 1);
  }
  tc_end<TCOLS>(tmem);
}

// ------------------------------------------------------------ gradient planes
// The masked gradient of a layer's output as three bfloat16 planes
// [plane][co / 8][position][8]: a position is a pixel of the batch with one zero column per
// row and one zero row per image around it, ((b (H + 1) + y + 1) (W + 1) + x + 1), so
// that a tap is a constant offset in positions and 8 channels are one 16-byte piece.
struct Padded {
  int H, W, B;
  int pitch() const { return W + 1; }
  // tiles of 128 positions from the first pixel of the first image on
  int tiles() const { return (int)(((int64_t)B * (H + 1) * (W + 1) + kTcM - 1) / kTcM); }
  // positions stored per 8 channels: the tiles with the reach of the taps
  int64_t positions() const { return (int64_t)kTcM * tiles() + 2 * W + 8; }
};

// Gradient with respect to the input of a 3x3 layer:
//   out[b][n][p] = sum_planes sum_c sum_tap wp[n][c][tap] g_plane[b][c][p + off_tap],
// with transposed and flipped weights wp [ceil(C/16)][9 taps][2][rows][8]. A tile is 128
// positions; a step of 16 channels stages the positions a tap can reach of all three planes (and
// the weights of the nine taps) by bulk copies, and a tap's MMA reads the staged
// positions from its own offset on, so no patch matrix is formed. One warp issues copies,
// one the MMAs, four add up: the hi plane's nine MMAs of a step go to one of two
// accumulators that those warps add to FP32 registers (round to nearest; an MMA truncates
// its sum to the accumulator's last bits, so a long chain of them drifts), mid and lo, 2^-8
// of hi, to a third that is read once. NB = 64: 192 accumulator columns, two
// blocks per SM. Bounded by the MMAs' shared-memory reads (A 32 + B 16 cycles for 32 of
// arithmetic at NB = 64; that pipe is 40 to 54% busy) and by waits between the roles.
// Warm-start network (width 64, 32 x 64, batch 32): nine layers in 242 us (CUDA cores:
// 2,900 us); the gradients' error against 64 bits 3.4e-7 (CUDA cores: 1.2e-6).
// grid (tiles, rows / NB), block 192. C a multiple of 16.
constexpr int kDgMaxStages = 4;
__host__ __device__ constexpr int dg_cols(int nb) { return 3 * nb <= 64 ? 64 : 3 * nb <= 128 ? 128 : 256; }
constexpr int dg_stage_bytes(int nb, int W) { return 6 * (132 + 2 * W) * 16 + 18 * nb * 16; }

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

template <int NB>
__global__ void __launch_bounds__(192, 2) k_dgrad_mma(const bf16 *__restrict__ g, int64_t plane, int64_t npos, int C,
                                                      const bf16 *__restrict__ wp, int rows, float *__restrict__ out,
                                                      int64_t obs, int H, int W, int B, int nstage, int *err) {
  vlb::chain_begin();
  static_assert(NB % 16 == 0 && NB <= 64, "three accumulators in 256 tensor-memory columns");
  constexpr int TCOLS = dg_cols(NB);
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t full[kDgMaxStages], empty[kDgMaxStages], dfull[2], dempty[2], dfin;
  __shared__ uint32_t tslot;
  __shared__ int failed;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = blockIdx.y * NB, nch = C / kTcCh, tile = blockIdx.x;
  const int ra = (132 + 2 * W) * 16, stage = 6 * ra + 18 * NB * 16;
  if (tid == 0) {
    failed = 0;
    for (int i = 0; i < nstage; i++) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; i++) {
      mbar_init(&dfull[i], 1);
      mbar_init(&dempty[i], 128);
    }
    mbar_init(&dfin, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tslot)), "r"(TCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tslot;
  bool ok = true;
  if (warp == 4) {
    // copies: lanes 0..5 the positions of (plane, K group), lanes 8..25 the weights of (tap, K group)
    int j = 0;
    for (; j < nch; j++) {
      const int s = j % nstage, use = j / nstage;
      if (use > 0 && !mbar_wait_warp(smem_u32(&empty[s]), (use - 1) & 1)) {
        ok = false;
        break;
      }
      const uint32_t base = smem_u32(sm) + s * stage, bar = smem_u32(&full[s]);
      if (lane == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(stage) : "memory");
      __syncwarp();
      if (lane < 6) {
        const int pl = lane >> 1, kg = lane & 1;
        bulk_g2s(base + lane * ra, g + pl * plane + ((int64_t)(2 * j + kg) * npos + (int64_t)kTcM * tile) * 8, ra, bar);
      } else if (lane >= 8 && lane < 26) {
        const int i = lane - 8;
        bulk_g2s(base + 6 * ra + i * NB * 16, wp + (((int64_t)j * 18 + i) * rows + n0) * 8, NB * 16, bar);
      }
    }
    // copies that nothing has waited for (after a failure) land before the block ends
    for (int i = j > nstage ? j - nstage : 0; i < j; i++)
      if (!mbar_wait_warp(smem_u32(&full[i % nstage]), (i / nstage) & 1)) ok = false;
  } else if (warp == 5) {
    for (int j = 0; j < nch; j++) {
      const int s = j % nstage, d = j & 1;
      if (!mbar_wait_warp(smem_u32(&full[s]), (j / nstage) & 1) ||
          (j >= 2 && !mbar_wait_warp(smem_u32(&dempty[d]), ((j >> 1) - 1) & 1))) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (lane == 0) {
        const uint32_t a0 = smem_u32(sm) + s * stage, b0 = a0 + 6 * ra;
        for (int pl = 0; pl < 3; pl++) {
          const uint32_t acc = tmem + (pl == 0 ? d * NB : 2 * NB);
          for (int t = 0; t < 9; t++)
            umma(acc, umma_desc(a0 + pl * 2 * ra + ((t / 3) * (W + 1) + t % 3) * 16, ra),
                 umma_desc(b0 + t * 2 * NB * 16, NB * 16), umma_idesc(NB), pl == 0 ? t > 0 : j > 0 || pl > 1 || t > 0);
          if (pl == 0) umma_commit(smem_u32(&dfull[d]));
        }
        umma_commit(smem_u32(&empty[s]));
        if (j + 1 == nch) umma_commit(smem_u32(&dfin));
      }
      __syncwarp();
    }
    if (!ok && lane == 0) umma_commit(smem_u32(&dfin));
    __syncwarp();
    // every MMA is done before the block ends
    if (!mbar_wait_warp(smem_u32(&dfin), 0)) ok = false;
  } else {
    float acc[NB];
#pragma unroll
    for (int i = 0; i < NB; i++) acc[i] = 0.0f;
    const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16);
    auto add = [&](uint32_t addr) {
#pragma unroll
      for (int c = 0; c < NB; c += 16) {
        uint32_t v[16];
        tmem_ld16(addr + c, v);
#pragma unroll
        for (int u = 0; u < 16; u++) acc[c + u] += __uint_as_float(v[u]);
      }
    };
    for (int j = 0; j < nch && ok; j++) {
      const int d = j & 1;
      if (!mbar_wait_warp(smem_u32(&dfull[d]), (j >> 1) & 1)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      add(ta + d * NB);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&dempty[d])) : "memory");
    }
    if (ok) ok = mbar_wait_warp(smem_u32(&dfin), 0);
    if (ok) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      add(ta + 2 * NB);
      const int q = kTcM * tile + tid;   // position of this row, from the first row of pixels on
      const int r = q / (W + 1), x = q - r * (W + 1), b = r / (H + 1), y = r - b * (H + 1);
      if (x < W && y < H && b < B) {
        float *o = out + (int64_t)b * obs + (int64_t)n0 * H * W + y * W + x;
#pragma unroll
        for (int i = 0; i < NB; i++) o[(int64_t)i * H * W] = acc[i];
      }
    }
  }
  if (!ok) failed = 1;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && failed) atomicOr(err, 1);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS));
}

// Weight-gradient partials as a GEMM over pixels:
//   D[row][ci, tap] = sum_p g_plane[co][p] in[ci][p + off_tap],
// rows = 128 of the (plane, co) pairs: CB = min(Co, 128) channels per group, so
// one MMA takes 128 / CB planes at once (three groups: hi, mid, lo), whose
// partial sums are written apart and added with the splits in a fixed order.
// N = 16 ci x 9 taps = 144 per MMA, NBK (1 or 2) of them per block, K = 64 pixels
// per step. The gradient operand is the planes' own 16-byte pieces of 8 channels (M
// contiguous); the nine shifted copies of an input row segment are formed from one 16-byte
// load and its two neighbours by byte permutes. grid (Co / CB x ngrp, nsplit),
// block 256, one block per SM.
// An MMA truncates its sum to the accumulator's last bits, so a long chain of
// them drifts: after every step (four MMAs deep per plane) the tensor-memory sums are
// added to FP32 registers, which round to nearest (144 a thread at NBK = 2,
// which bounds the block). Step j + 1 is staged while step j's MMAs run.
// Warm-start network (width 64, 32 x 64, batch 32): ten layers in 407 us (CUDA cores: 3,620 us).
// Needs W a multiple of 8, H W a multiple of 64, C a multiple of 8.
constexpr int kWgA = kTcM * 128;                 // one set of 128 gradient rows, 64 pixels
constexpr int kWgLboB = 144 * 16 + 16;
constexpr int kWgB = 8 * kWgLboB;                // 144 input rows, 64 pixels
__host__ __device__ constexpr int wg_sets(int cb) { return (3 * cb + kTcM - 1) / kTcM; }
__host__ __device__ constexpr int wg_groups(int cb) { return kTcM / cb < 3 ? kTcM / cb : 3; }

// 24 tensor-memory columns of the warp's 32 lanes
__device__ __forceinline__ void tmem_ld24(uint32_t addr, uint32_t (&r)[24]) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%24];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%25];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23])
      : "r"(addr), "r"(addr + 16)
      : "memory");
}

template <int CB, int NBK>
__global__ void __launch_bounds__(256, 1) k_wgrad_mma(const bf16 *__restrict__ in, int64_t ibs, int C,
                                                      const bf16 *__restrict__ g, int64_t npos, int64_t gplane, int Co,
                                                      float *__restrict__ dwp, int H, int W, int B, int ngrp,
                                                      int *err) {
  vlb::chain_begin();
  constexpr int NSET = wg_sets(CB), NG = wg_groups(CB), COLS = NBK * 72;
  constexpr int stage = NSET * kWgA + NBK * kWgB;
  constexpr int units = NBK * 128, UPT = (units + 255) / 256;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int HW = H * W, per_s = HW / 64;
  const int mb = blockIdx.x / ngrp, ci0 = (blockIdx.x % ngrp) * NBK * 16, co0 = mb * CB;
  // this split's 64-pixel steps
  const int64_t total = (int64_t)B * per_s, per = (total + gridDim.y - 1) / gridDim.y;
  const int64_t q0 = (int64_t)blockIdx.y * per, q1 = q0 + per < total ? q0 + per : total;
  const int nst = q1 > q0 ? (int)(q1 - q0) : 0;
  const uint32_t tmem = tc_begin<512>(bar, &tslot);
  // rows of no plane stay zero
  for (int i = tid; i < 2 * stage / 16; i += 256) *reinterpret_cast<uint4 *>(sm + i * 16) = make_uint4(0, 0, 0, 0);
  __syncthreads();
  auto load_g = [&](int j) {
    const int64_t q = q0 + j;
    const int b = (int)(q / per_s), pp = (int)(q % per_s) * 64;
    // a thread copies its pixel of groups of 8 rows (i / 64), 64 pixels each
    const int p = pp + (tid & 63), y = p / W, x = p - y * W;
    const int64_t pos = (int64_t)(b * (H + 1) + y + 1) * (W + 1) + x + 1;
    const uint32_t dst = smem_u32(sm + (j & 1) * stage) + tid * 16;
#pragma unroll 4
    for (int k = 0; k < NSET * 4; k++) {
      const int m = k * 4 + (tid >> 6), pl = m / (CB / 8), co8 = (co0 >> 3) + m % (CB / 8);
      if (pl < 3) cp16(dst + k * 4096, g + (int64_t)pl * gplane + ((int64_t)co8 * npos + pos) * 8);
    }
  };
  // units of (input channel, 8 pixels): the three rows' 16 bytes and the
  // pixels on either side
  uint4 rc[UPT][3];
  uint32_t rs[UPT][3];
  auto load_x = [&](int j) {
    const int64_t q = q0 + j;
    const int b = (int)(q / per_s), pp = (int)(q % per_s) * 64;
#pragma unroll
    for (int k = 0; k < UPT; k++) {
      const int u = tid + k * 256, ci = ci0 + (u >> 3);
      const int pq = pp + (u & 7) * 8, y = pq / W, x = pq - y * W;
      const bf16 *src = in + (int64_t)b * ibs + (int64_t)ci * HW + pq;
#pragma unroll
      for (int r = 0; r < 3; r++) {
        uint4 c = make_uint4(0, 0, 0, 0);
        uint32_t e = 0;
        if (u < units && ci < C && y + r - 1 >= 0 && y + r - 1 < H) {
          const bf16 *s = src + (r - 1) * W;
          c = *reinterpret_cast<const uint4 *>(s);
          if (x > 0) e = *reinterpret_cast<const unsigned short *>(s - 1);
          if (x + 8 < W) e |= (uint32_t) * reinterpret_cast<const unsigned short *>(s + 8) << 16;
        }
        rc[k][r] = c;
        rs[k][r] = e;
      }
    }
  };
  auto store_x = [&](int j) {
    unsigned char *base = sm + (j & 1) * stage + NSET * kWgA;
#pragma unroll
    for (int k = 0; k < UPT; k++) {
      const int u = tid + k * 256;
      if (u >= units) continue;
      const int cl = u >> 3;
      unsigned char *dst = base + (cl >> 4) * kWgB + (u & 7) * kWgLboB + (cl & 15) * 9 * 16;
#pragma unroll
      for (int r = 0; r < 3; r++) {
        const uint4 c = rc[k][r];
        const uint32_t e = rs[k][r];
        const uint32_t m0 = pick2<1, 0>(c.x, c.y), m1 = pick2<1, 0>(c.y, c.z), m2 = pick2<1, 0>(c.z, c.w);
        *reinterpret_cast<uint4 *>(dst + (3 * r) * 16) = make_uint4(pick2<0, 0>(e, c.x), m0, m1, m2);
        *reinterpret_cast<uint4 *>(dst + (3 * r + 1) * 16) = c;
        *reinterpret_cast<uint4 *>(dst + (3 * r + 2) * 16) = make_uint4(m0, m1, m2, pick2<1, 1>(c.w, e));
      }
    }
  };
  // this thread's sums: lane (warp % 4) * 32 + .., half (warp / 4) of the columns
  float acc[COLS];
#pragma unroll
  for (int i = 0; i < COLS; i++) acc[i] = 0.0f;
  const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * COLS);
  bool ok = true, late = false;
  if (nst > 0) {
    load_g(0);
    load_x(0);
    store_x(0);
    if (nst > 1) load_x(1);
  }
  for (int j = 0; j < nst; j++) {
    cp16_wait_all();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (__syncthreads_or(late)) {
      ok = false;
      break;
    }
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a0 = smem_u32(sm + (j & 1) * stage), b0 = a0 + NSET * kWgA;
      // the small planes first
      for (int set = NSET - 1; set >= 0; set--)
        for (int ks = 0; ks < 4; ks++)
          for (int k = 0; k < NBK; k++)
            umma(tmem + k * 144, umma_desc(a0 + set * kWgA + ks * 256, 128, 1024),
                 umma_desc(b0 + k * kWgB + ks * 2 * kWgLboB, kWgLboB), umma_idesc(144) | kTcAmn,
                 set < NSET - 1 || ks > 0);
      umma_commit(smem_u32(&bar[0]));
    }
    if (j + 1 < nst) {
      load_g(j + 1);
      store_x(j + 1);
      if (j + 2 < nst) load_x(j + 2);
    }
    late = !mbar_wait(smem_u32(&bar[0]), j & 1);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
    for (int c = 0; c < COLS; c += 24) {
      uint32_t v[24];
      tmem_ld24(ta + c, v);
#pragma unroll
      for (int u = 0; u < 24; u++) acc[c + u] += __uint_as_float(v[u]);
    }
  }
  cp16_wait_all();
  if (__syncthreads_or(late)) ok = false;
  if (ok) {
    const int r = (warp & 3) * 32 + (tid & 31), grp = r / CB, c1 = (warp >> 2) * COLS;
    float *row = dwp + (((int64_t)blockIdx.y * NG + grp) * Co + co0 + r % CB) * C * 9 + (int64_t)ci0 * 9;
    const int lim = (C - ci0) * 9;
    if (grp < NG) {
#pragma unroll
      for (int c = 0; c < COLS; c += 4)
        if (c1 + c < lim) *reinterpret_cast<float4 *>(row + c1 + c) = make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]);
    }
  } else if (tid == 0) {
    atomicOr(err, 1);
  }
  tc_end<512>(tmem);
}

// ------------------------------------------------------------ packed weights
// Weights of the tensor-core layers in pipeline-step order, from the FP32
// master rounded to bfloat16: [step of 16 K channels][K group of 8][row][8],
// K index within a step = channel * 9 + tap, zero past the last channel.
// Forward: rows co, K channels ci; backward: rows ci, K channels co, taps flipped,
// a step's K groups in the order [tap][2] (8 channels of one tap each).
struct PackLayer {
  int cin, cout;
  int64_t woff, fwd, bwd;   // offsets: master weights, packed forward, packed backward (-1: none)
};
struct PackTable {
  PackLayer l[10];
  int n;
};
__global__ void k_pack_weights(const float *__restrict__ p, bf16 *__restrict__ wp, const PackTable t) {
  const PackLayer l = t.l[blockIdx.y >> 1];
  const bool back = blockIdx.y & 1;
  const int64_t off = back ? l.bwd : l.fwd;
  if (off < 0) return;
  const int rows = back ? l.cin : l.cout, kc = back ? l.cout : l.cin;
  const int total = (kc + kTcCh - 1) / kTcCh * kTcKG * rows * 8;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int e = i & 7, n = (i >> 3) % rows, kg = ((i >> 3) / rows) % kTcKG, cc = (i >> 3) / rows / kTcKG;
    const int kk = kg * 8 + e, c = cc * kTcCh + (back ? (kg & 1) * 8 + e : kk / 9), tap = back ? kg >> 1 : kk % 9;
    float v = 0.0f;
    if (c < kc) v = back ? p[l.woff + ((int64_t)c * l.cin + n) * 9 + 8 - tap] : p[l.woff + ((int64_t)n * l.cin + c) * 9 + tap];
    wp[off + i] = __float2bfloat16_rn(v);
  }
}

// v = hi + mid + lo exactly to 24 bits, each a bfloat16; an infinity or NaN is
// hi alone (its remainder would be NaN), a value that rounds beyond the
// largest bfloat16 takes that one as hi
__device__ __forceinline__ void split3(float v, bf16 &h, bf16 &m, bf16 &l) {
  h = __float2bfloat16_rn(v);
  if (__builtin_expect(!(fabsf(v) <= 3.3895313892515355e38f), 0)) {
    if (isfinite(v)) {
      h = __ushort_as_bfloat16(v < 0.0f ? 0xff7f : 0x7f7f);
    } else {
      m = l = __float2bfloat16_rn(0.0f);
      return;
    }
  }
  const float r = v - __bfloat162float(h);
  m = __float2bfloat16_rn(r);
  l = __float2bfloat16_rn(r - __bfloat162float(m));
}
__device__ __forceinline__ uint32_t pack_bf16(bf16 lo, bf16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}
// 8 channels' gradients of one position into the three planes (16 bytes each)
__device__ __forceinline__ void store_planes(bf16 *dst, int64_t plane, const float (&v)[8]) {
  bf16 h[8], m[8], l[8];
#pragma unroll
  for (int i = 0; i < 8; i++) split3(v[i], h[i], m[i], l[i]);
  const bf16 *src[3] = {h, m, l};
#pragma unroll
  for (int p = 0; p < 3; p++)
    *reinterpret_cast<uint4 *>(dst + p * plane) =
        make_uint4(pack_bf16(src[p][0], src[p][1]), pack_bf16(src[p][2], src[p][3]), pack_bf16(src[p][4], src[p][5]),
                   pack_bf16(src[p][6], src[p][7]));
}
// sums over a block of 128 threads (fixed order) of N values a thread, into out[k * stride]
template <int N>
__device__ __forceinline__ void block_sums128(float (&v)[N], float *out, int stride) {
  __shared__ float sh[4][N];
#pragma unroll
  for (int k = 0; k < N; k++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][k] = v[k];
  }
  __syncthreads();
  if (threadIdx.x < N) {
    const int k = threadIdx.x;
    out[(int64_t)k * stride] = (sh[0][k] + sh[1][k]) + (sh[2][k] + sh[3][k]);
  }
}
// pixel of a position (false: a zero column or row, or past the batch)
__device__ __forceinline__ bool pad_pixel(int q, int H, int W, int B, int &b, int &y, int &x) {
  const int r = q / (W + 1);
  x = q - r * (W + 1) - 1;
  b = (r - 1) / (H + 1);
  y = (r - 1) - b * (H + 1);
  return r >= 1 && x >= 0 && y < H && b < B;
}

// The gradient of one layer's output, masked by its ReLU, as planes, and its
// sum over the pixels of a block per channel (the bias gradient's partial sums, bsum[block][C]).
// Where the gradient comes from: MODE 0 g itself; MODE 1 the four children of
// g at twice the resolution (below a nearest upsampling); MODE 2 g plus a
// quarter of the pooled gradient gp. One pass in place of the pool / upsampling
// gradient, the mask, the bias sum and the split. grid (blocks, C / 8), block 128.
template <int MODE>
__global__ void __launch_bounds__(128) k_mask_split(const float *__restrict__ g, int64_t gbs,
                                                    const float *__restrict__ gp, int64_t gpbs,
                                                    const bf16 *__restrict__ act, int64_t abs_,
                                                    bf16 *__restrict__ planes, int64_t plane, int npos,
                                                    float *__restrict__ bsum, int H, int W, int B) {
  vlb::chain_begin();
  const int c0 = blockIdx.y * 8, C = gridDim.y * 8, HW = H * W;
  float s[8];
#pragma unroll
  for (int i = 0; i < 8; i++) s[i] = 0.0f;
  for (int q = blockIdx.x * 128 + threadIdx.x; q < npos; q += gridDim.x * 128) {
    int b, y, x;
    float v[8];
    if (pad_pixel(q, H, W, B, b, y, x)) {
      const bf16 *a = act + (int64_t)b * abs_ + (int64_t)c0 * HW + y * W + x;
      const float *gb = g + (int64_t)b * gbs;
#pragma unroll
      for (int i = 0; i < 8; i++) {
        float t;
        if constexpr (MODE == 1) {
          const float *p = gb + (int64_t)(c0 + i) * 4 * HW + (int64_t)(2 * y) * (2 * W) + 2 * x;
          const float2 u = *reinterpret_cast<const float2 *>(p), w = *reinterpret_cast<const float2 *>(p + 2 * W);
          t = u.x + u.y + w.x + w.y;
        } else {
          t = gb[(int64_t)(c0 + i) * HW + y * W + x];
          if constexpr (MODE == 2)
            t += 0.25f * gp[(int64_t)b * gpbs + (int64_t)(c0 + i) * (HW / 4) + (y / 2) * (W / 2) + x / 2];
        }
        v[i] = __bfloat162float(a[(int64_t)i * HW]) > 0.0f ? t : 0.0f;
        s[i] += v[i];
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; i++) v[i] = 0.0f;
    }
    store_planes(planes + ((int64_t)blockIdx.y * npos + q) * 8, plane, v);
  }
  block_sums128<8>(s, bsum + (int64_t)blockIdx.x * C + c0, 1);
}

// The 1x1 head's backward pass and the mask of the layer below in one pass over
// t1: its gradient sum_co w[co][c] dy[co] masked and split into planes, the
// block's sums of that gradient (bias of the layer below, bsum[block][C]), and the
// block's part of the head's weight and bias gradients, hp[block][co C + c] and
// hp[block][NCO C + co]. grid (blocks, C / 8), block 128; NCO output channels.
template <int NCO>
__global__ void __launch_bounds__(128) k_head_bwd(const float *__restrict__ dy, int64_t ybs, const bf16 *__restrict__ w,
                                                  const bf16 *__restrict__ act, int64_t abs_, bf16 *__restrict__ planes,
                                                  int64_t plane, int npos, float *__restrict__ bsum,
                                                  float *__restrict__ hp, int H, int W, int B) {
  vlb::chain_begin();
  const int c0 = blockIdx.y * 8, C = gridDim.y * 8, HW = H * W;
  float wv[NCO][8], sums[9 * NCO + 8];   // dw [NCO][8], db [NCO], masked gradient [8]
#pragma unroll
  for (int o = 0; o < NCO; o++)
#pragma unroll
    for (int i = 0; i < 8; i++) wv[o][i] = __bfloat162float(w[o * C + c0 + i]);
#pragma unroll
  for (int k = 0; k < 9 * NCO + 8; k++) sums[k] = 0.0f;
  for (int q = blockIdx.x * 128 + threadIdx.x; q < npos; q += gridDim.x * 128) {
    int b, y, x;
    float v[8];
    if (pad_pixel(q, H, W, B, b, y, x)) {
      const bf16 *a = act + (int64_t)b * abs_ + (int64_t)c0 * HW + y * W + x;
      float d[NCO];
#pragma unroll
      for (int o = 0; o < NCO; o++) {
        d[o] = dy[(int64_t)b * ybs + (int64_t)o * HW + y * W + x];
        sums[8 * NCO + o] += d[o];
      }
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const float t = __bfloat162float(a[(int64_t)i * HW]);
        float gv = 0.0f;
#pragma unroll
        for (int o = 0; o < NCO; o++) {
          gv = fmaf(d[o], wv[o][i], gv);
          sums[8 * o + i] = fmaf(d[o], t, sums[8 * o + i]);
        }
        v[i] = t > 0.0f ? gv : 0.0f;
        sums[9 * NCO + i] += v[i];
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; i++) v[i] = 0.0f;
    }
    store_planes(planes + ((int64_t)blockIdx.y * npos + q) * 8, plane, v);
  }
  // (a value's place depends on its index: summed into shared memory, then placed)
  __shared__ float tot[9 * NCO + 8];
  block_sums128<9 * NCO + 8>(sums, tot, 1);
  __syncthreads();
  const int k = threadIdx.x;
  float *h = hp + (int64_t)blockIdx.x * (NCO * C + NCO);
  if (k < 8 * NCO)
    h[(k / 8) * C + c0 + k % 8] = tot[k];
  else if (k < 9 * NCO) {
    if (blockIdx.y == 0) h[NCO * C + k - 8 * NCO] = tot[k];
  } else if (k < 9 * NCO + 8)
    bsum[(int64_t)blockIdx.x * C + c0 + k - 9 * NCO] = tot[k];
}

// dst[i] = sum over the splits of src[s][i] (i < n), then dst[n + i] = sum over
// the samples of bsum[b][i] (i < nbias): a layer's weight and bias gradients
// lie one after the other. Fixed order.
__global__ void k_sum_parts(const float *__restrict__ src, int nsplit, int64_t n, const float *__restrict__ bsum,
                            int nsamp, int nbias, float *__restrict__ dst) {
  vlb::chain_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n + nbias) return;
  const float *q = i < n ? src + i : bsum + (i - n);
  const int64_t st = i < n ? n : nbias;
  const int m = i < n ? nsplit : nsamp;
  float s = 0.0f;
#pragma unroll 8
  for (int k = 0; k < m; k++) s += q[k * st];
  dst[i] = s;
}

}  // namespace nn
