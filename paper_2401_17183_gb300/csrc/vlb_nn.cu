// vlb_nn.cu -- the learned warm start (include/vlb_nn.h): a 2D U-Net with
// hand-written forward and backward kernels. Weights and activations are
// stored in FP32 or bfloat16 and every product is accumulated in FP32; the
// optimizer (Adam) works on an FP32 master copy of the parameters.
//
// Kernels: a tiled direct convolution (3x3, zero padding) that also
// serves the backward pass with respect to its input (with transposed,
// flipped weights), a tiled weight-gradient reduction with fixed-order
// split sums (deterministic), 2x2 average pooling, 2x nearest upsampling,
// the 1x1 head, ReLU masks, bias gradients, the mean-square loss and Adam.
// With bfloat16 storage the 3x3 layers run on the tensor cores, forward and
// backward, where they fit (vlb_nn_tc.cuh). Activations are NCHW with a
// batch stride, so a channel concatenation is a view into one buffer.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/vlb.h"
#include "../../include/vlb_nn.h"
#include "vlb_nn_tc.cuh"

namespace vlb {
int set_error(int code, const char *fmt, ...);
}

namespace nn {

constexpr int kTile = 16;   // output pixels per block side
constexpr int kCo = 16;     // output channels per block
constexpr int kCi = 8;      // input channels per chunk
constexpr int kThreads = kTile * kTile;

template <typename T>
__device__ __forceinline__ float ld(const T *p) {
  return static_cast<float>(*p);
}
template <>
__device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16 *p) {
  return __bfloat162float(*p);
}
template <typename T>
__device__ __forceinline__ T st(float x) {
  return static_cast<T>(x);
}
template <>
__device__ __forceinline__ __nv_bfloat16 st<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}

// ---------------------------------------------------------------- convolution
// out[b][co][p] = act(bias[co] + sum_ci sum_k w[co][ci][k] in[b][ci][p + off_k])
// in: channel stride H*W, batch stride ibs; out likewise with obs.
// grid (tiles of W x H, ceil(Co / kCo), B), block kThreads.
template <int K, typename TI, typename TW, typename TO, bool RELU>
__global__ void __launch_bounds__(kThreads) k_conv(const TI *__restrict__ in, int64_t ibs, const TW *__restrict__ w,
                                                   const float *__restrict__ bias, TO *__restrict__ out, int64_t obs,
                                                   int Ci, int Co, int H, int W) {
  constexpr int R = K / 2, TS = kTile + 2 * R;
  __shared__ float in_s[kCi][TS][TS];
  __shared__ __align__(16) float w_s[kCi][K * K][kCo];
  const int tilesx = (W + kTile - 1) / kTile;
  const int tx0 = (blockIdx.x % tilesx) * kTile, ty0 = (blockIdx.x / tilesx) * kTile;
  const int co0 = blockIdx.y * kCo, b = blockIdx.z;
  const int tx = threadIdx.x % kTile, ty = threadIdx.x / kTile;
  const int64_t HW = (int64_t)H * W;
  const TI *inb = in + b * ibs;
  float acc[kCo];
#pragma unroll
  for (int o = 0; o < kCo; o++) acc[o] = 0.0f;
  for (int c0 = 0; c0 < Ci; c0 += kCi) {
    for (int i = threadIdx.x; i < kCi * TS * TS; i += kThreads) {
      const int c = i / (TS * TS), r = i % (TS * TS), yy = ty0 - R + r / TS, xx = tx0 - R + r % TS;
      float v = 0.0f;
      if (c0 + c < Ci && yy >= 0 && yy < H && xx >= 0 && xx < W) v = ld(inb + (c0 + c) * HW + (int64_t)yy * W + xx);
      in_s[c][r / TS][r % TS] = v;
    }
    for (int i = threadIdx.x; i < kCi * K * K * kCo; i += kThreads) {
      const int o = i % kCo, k = (i / kCo) % (K * K), c = i / (kCo * K * K);
      float v = 0.0f;
      if (c0 + c < Ci && co0 + o < Co) v = ld(w + ((int64_t)(co0 + o) * Ci + c0 + c) * K * K + k);
      w_s[c][k][o] = v;
    }
    __syncthreads();
#pragma unroll 2
    for (int c = 0; c < kCi; c++)
#pragma unroll
      for (int k = 0; k < K * K; k++) {
        const float v = in_s[c][ty + k / K][tx + k % K];
        const float4 *wv = reinterpret_cast<const float4 *>(&w_s[c][k][0]);
#pragma unroll
        for (int q = 0; q < kCo / 4; q++) {
          const float4 x = wv[q];
          acc[4 * q] = fmaf(v, x.x, acc[4 * q]);
          acc[4 * q + 1] = fmaf(v, x.y, acc[4 * q + 1]);
          acc[4 * q + 2] = fmaf(v, x.z, acc[4 * q + 2]);
          acc[4 * q + 3] = fmaf(v, x.w, acc[4 * q + 3]);
        }
      }
    __syncthreads();
  }
  const int y = ty0 + ty, x = tx0 + tx;
  if (y >= H || x >= W) return;
  TO *ob = out + b * obs + (int64_t)y * W + x;
#pragma unroll
  for (int o = 0; o < kCo; o++) {
    if (co0 + o >= Co) break;
    float v = acc[o] + (bias ? bias[co0 + o] : 0.0f);
    if (RELU) v = fmaxf(v, 0.0f);
    ob[(int64_t)(co0 + o) * HW] = st<TO>(v);
  }
}

// wt[ci][co][k'] = w[co][ci][K*K - 1 - k'] (FP32): the weights of the
// backward pass with respect to the input
template <typename TW>
__global__ void k_transpose_flip(const TW *__restrict__ w, float *__restrict__ wt, int Ci, int Co, int KK) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)Ci * Co * KK) return;
  const int k = (int)(i % KK), co = (int)((i / KK) % Co), ci = (int)(i / ((int64_t)KK * Co));
  wt[i] = ld(w + ((int64_t)co * Ci + ci) * KK + (KK - 1 - k));
}

// Weight gradient partials: dwp[split][co][ci][k] = sum over this split's
// (sample, pixel tile) pairs of g[b][co][p] in[b][ci][p + off_k].
// grid (ceil(Co/16), ceil(Ci/8), nsplit), block 128: thread (co, ci).
template <int K, typename TI>
__global__ void __launch_bounds__(128) k_conv_dw(const TI *__restrict__ in, int64_t ibs, const float *__restrict__ g,
                                                 int64_t gbs, float *__restrict__ dwp, int Ci, int Co, int H, int W,
                                                 int B) {
  constexpr int R = K / 2, TS = kTile + 2 * R;
  __shared__ float g_s[16][kTile * kTile + 1];
  __shared__ float in_s[8][TS * TS + 1];
  const int co0 = blockIdx.x * 16, ci0 = blockIdx.y * 8;
  const int tco = threadIdx.x / 8, tci = threadIdx.x % 8;
  const int tilesx = (W + kTile - 1) / kTile, tilesy = (H + kTile - 1) / kTile;
  const int64_t HW = (int64_t)H * W;
  const int64_t nwork = (int64_t)B * tilesx * tilesy;
  float acc[K * K];
#pragma unroll
  for (int k = 0; k < K * K; k++) acc[k] = 0.0f;
  for (int64_t wk = blockIdx.z; wk < nwork; wk += gridDim.z) {
    const int b = (int)(wk / (tilesx * tilesy)), tl = (int)(wk % (tilesx * tilesy));
    const int tx0 = (tl % tilesx) * kTile, ty0 = (tl / tilesx) * kTile;
    for (int i = threadIdx.x; i < 16 * kTile * kTile; i += 128) {
      const int o = i / (kTile * kTile), p = i % (kTile * kTile), yy = ty0 + p / kTile, xx = tx0 + p % kTile;
      float v = 0.0f;
      if (co0 + o < Co && yy < H && xx < W) v = g[b * gbs + (co0 + o) * HW + (int64_t)yy * W + xx];
      g_s[o][p] = v;
    }
    for (int i = threadIdx.x; i < 8 * TS * TS; i += 128) {
      const int c = i / (TS * TS), r = i % (TS * TS), yy = ty0 - R + r / TS, xx = tx0 - R + r % TS;
      float v = 0.0f;
      if (ci0 + c < Ci && yy >= 0 && yy < H && xx >= 0 && xx < W) v = ld(in + b * ibs + (ci0 + c) * HW + (int64_t)yy * W + xx);
      in_s[c][r] = v;
    }
    __syncthreads();
    for (int p = 0; p < kTile * kTile; p++) {
      const float gv = g_s[tco][p];
      const int py = p / kTile, px = p % kTile;
#pragma unroll
      for (int k = 0; k < K * K; k++) acc[k] = fmaf(gv, in_s[tci][(py + k / K) * TS + px + k % K], acc[k]);
    }
    __syncthreads();
  }
  if (co0 + tco < Co && ci0 + tci < Ci) {
    float *o = dwp + (((int64_t)blockIdx.z * Co + co0 + tco) * Ci + ci0 + tci) * (K * K);
#pragma unroll
    for (int k = 0; k < K * K; k++) o[k] = acc[k];
  }
}

// dst[i] = sum_s src[s][i] in split order (deterministic)
__global__ void k_sum_splits(const float *__restrict__ src, int nsplit, int64_t n, float *__restrict__ dst) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float s = 0.0f;
  for (int k = 0; k < nsplit; k++) s += src[k * n + i];
  dst[i] = s;
}

// db[co] = sum_b sum_p g[b][co][p]; one block per channel, fixed-order tree
__global__ void k_bias_grad(const float *__restrict__ g, int64_t gbs, int64_t HW, int B, float *__restrict__ db) {
  __shared__ float sh[256];
  const int co = blockIdx.x;
  float s = 0.0f;
  for (int b = 0; b < B; b++)
    for (int64_t p = threadIdx.x; p < HW; p += 256) s += g[b * gbs + co * HW + p];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) db[co] = sh[0];
}

// g *= (act > 0) over C channels of B samples
template <typename TA>
__global__ void k_relu_mask(float *__restrict__ g, int64_t gbs, const TA *__restrict__ act, int64_t abs_, int64_t CHW,
                            int B) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= CHW * B) return;
  const int64_t b = i / CHW, r = i % CHW;
  if (!(ld(act + b * abs_ + r) > 0.0f)) g[b * gbs + r] = 0.0f;
}

// two neighbouring values of type T (the first at an even element offset)
template <typename T>
struct Pair;
template <>
struct Pair<float> {
  using V = float2;
  static __device__ __forceinline__ float2 f(V v) { return v; }
  static __device__ __forceinline__ V both(float x) { return make_float2(x, x); }
};
template <>
struct Pair<__nv_bfloat16> {
  using V = __nv_bfloat162;
  static __device__ __forceinline__ float2 f(V v) { return __bfloat1622float2(v); }
  static __device__ __forceinline__ V both(__nv_bfloat16 x) { return __nv_bfloat162(x, x); }
};

// 2x2 average pool: out [C][H/2][W/2] from in [C][H][W]; a block per channel
// and sample, so that no thread divides 64-bit indices (k_up likewise: 44 us
// -> 6 us for 16 MB written at width 64, 32 x 64, batch 32). Grid (C, B).
template <typename T>
__global__ void k_pool(const T *__restrict__ in, int64_t ibs, T *__restrict__ out, int64_t obs, int H, int W) {
  vlb::chain_begin();
  const int Ho = H / 2, Wo = W / 2, c = blockIdx.x, b = blockIdx.y;
  const T *p = in + (int64_t)b * ibs + (int64_t)c * H * W;
  T *o = out + (int64_t)b * obs + (int64_t)c * Ho * Wo;
  for (int i = threadIdx.x; i < Ho * Wo; i += blockDim.x) {
    const int y = i / Wo, x = i - y * Wo;
    const typename Pair<T>::V *q = reinterpret_cast<const typename Pair<T>::V *>(p + 2 * y * W + 2 * x);
    const float2 u = Pair<T>::f(q[0]), v = Pair<T>::f(q[W / 2]);
    o[i] = st<T>(0.25f * (u.x + u.y + v.x + v.y));
  }
}

// gradient of the pool: gin[..] += gout / 4 (gin FP32)
__global__ void k_pool_bwd(const float *__restrict__ gout, int64_t gobs, float *__restrict__ gin, int64_t gibs, int C,
                           int H, int W, int B) {
  const int64_t n = (int64_t)B * C * H * W;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int x = (int)(i % W), y = (int)((i / W) % H), c = (int)((i / ((int64_t)W * H)) % C);
  const int64_t b = i / ((int64_t)W * H * C);
  gin[b * gibs + (int64_t)c * H * W + (int64_t)y * W + x] +=
      0.25f * gout[b * gobs + (int64_t)c * (H / 2) * (W / 2) + (int64_t)(y / 2) * (W / 2) + x / 2];
}

// 2x nearest upsampling: out [C][2h][2w] from in [C][h][w], a pair of equal
// values per store. Grid (C, B).
template <typename T>
__global__ void k_up(const T *__restrict__ in, int64_t ibs, T *__restrict__ out, int64_t obs, int h, int w) {
  vlb::chain_begin();
  const int c = blockIdx.x, b = blockIdx.y;
  const T *p = in + (int64_t)b * ibs + (int64_t)c * h * w;
  typename Pair<T>::V *o = reinterpret_cast<typename Pair<T>::V *>(out + (int64_t)b * obs + (int64_t)c * 4 * h * w);
  for (int i = threadIdx.x; i < h * w; i += blockDim.x) {
    const int y = i / w, x = i - y * w;
    const typename Pair<T>::V v = Pair<T>::both(p[i]);
    o[2 * y * w + x] = v;
    o[(2 * y + 1) * w + x] = v;
  }
}

// The 1x1 head: out[b][co][p] = bias[co] + sum_c w[co][c] in[b][c][p], FP32 out,
// the channels in order for every output. Bounded by reading the input
// once; a thread takes two pixels and NCO outputs. grid (ceil(HW / 256), B,
// ceil(Co / NCO)), block 128; HW even.
template <typename T, typename TW, int NCO>
__global__ void __launch_bounds__(128) k_head(const T *__restrict__ in, int64_t ibs, const TW *__restrict__ w,
                                              const float *__restrict__ bias, float *__restrict__ out, int64_t obs,
                                              int C, int Co, int HW) {
  vlb::chain_begin();
  const int b = blockIdx.y, o0 = blockIdx.z * NCO, p = (blockIdx.x * 128 + threadIdx.x) * 2;
  if (p >= HW) return;
  const T *ib = in + (int64_t)b * ibs + p;
  float2 acc[NCO];
#pragma unroll
  for (int o = 0; o < NCO; o++) acc[o] = make_float2(0.f, 0.f);
#pragma unroll 8
  for (int c = 0; c < C; c++) {
    const float2 v = Pair<T>::f(*reinterpret_cast<const typename Pair<T>::V *>(ib + (int64_t)c * HW));
#pragma unroll
    for (int o = 0; o < NCO; o++) {
      const float wv = o0 + o < Co ? ld(w + (int64_t)(o0 + o) * C + c) : 0.0f;
      acc[o].x = fmaf(v.x, wv, acc[o].x);
      acc[o].y = fmaf(v.y, wv, acc[o].y);
    }
  }
#pragma unroll
  for (int o = 0; o < NCO; o++) {
    if (o0 + o >= Co) break;
    float *q = out + (int64_t)b * obs + (int64_t)(o0 + o) * HW + p;
    q[0] = acc[o].x + bias[o0 + o];
    q[1] = acc[o].y + bias[o0 + o];
  }
}

// gradient of the upsampling: gin[c][y][x] = sum of the four children (assigns)
__global__ void k_up_bwd(const float *__restrict__ gout, int64_t gobs, float *__restrict__ gin, int64_t gibs, int C,
                         int h, int w, int B) {
  const int64_t n = (int64_t)B * C * h * w;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int x = (int)(i % w), y = (int)((i / w) % h), c = (int)((i / ((int64_t)w * h)) % C);
  const int64_t b = i / ((int64_t)w * h * C);
  const float *p = gout + b * gobs + (int64_t)c * 4 * h * w + (int64_t)(2 * y) * (2 * w) + 2 * x;
  gin[b * gibs + (int64_t)c * h * w + (int64_t)y * w + x] = p[0] + p[1] + p[2 * w] + p[2 * w + 1];
}

template <typename TO>
__global__ void k_convert(const float *__restrict__ in, TO *__restrict__ out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = st<TO>(in[i]);
}

// dst[b][r] = src[b][r] (converted) for r < CHW: the input into its view
template <typename TO>
__global__ void k_convert_into(const float *__restrict__ src, int64_t sbs, TO *__restrict__ dst, int64_t dbs,
                               int64_t CHW, int B) {
  vlb::chain_begin();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= CHW * B) return;
  const int64_t b = i / CHW, r = i % CHW;
  dst[b * dbs + r] = st<TO>(src[b * sbs + r]);
}

// mean-square loss: partial sums per block and dy = 2 (y - t) / n
__global__ void k_mse(const float *__restrict__ y, const float *__restrict__ t, float *__restrict__ dy, int64_t n,
                      double *__restrict__ partial) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const float d = y[i] - t[i];
    dy[i] = 2.0f * d / (float)n;
    s += (double)d * d;
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                       int64_t n, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// He-uniform initial weights from SplitMix64 (counter = parameter index)
__global__ void k_init_params(float *p, int64_t off, int64_t n, float bound, uint64_t seed) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint64_t z = seed + 0x9E3779B97F4A7C15ull * (uint64_t)(off + i + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  const double u = (double)(z >> 11) * (1.0 / 9007199254740992.0);
  p[off + i] = (float)((2.0 * u - 1.0) * bound);
}

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace nn

// ------------------------------------------------------------------ host side
struct NNLayer {
  int cin, cout, k, h, w;  // input channels, output channels, kernel, grid at this layer
  int64_t woff, boff;       // offsets in the parameter vector
};

// an activation buffer (storage T) or gradient buffer (FP32) view
struct View {
  int64_t off;    // element offset of channel 0 in its buffer
  int64_t bs;     // batch stride (elements)
};

struct vlb_nn {
  int ci, co, width, H, W, maxb, storage;
  std::vector<NNLayer> L;
  int64_t np = 0;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // master params, grads, Adam moments
  void *pc = nullptr;        // compute copy of the parameters (bfloat16) or NULL
  void *act = nullptr;       // activations (storage type)
  float *gr = nullptr;       // gradients of activations (FP32)
  float *wt = nullptr;       // transposed weights (FP32), largest layer
  float *dwp = nullptr;      // weight-gradient split partials
  double *lossp = nullptr;
  int64_t act_n = 0, wt_n = 0, dwp_n = 0;
  int nsplit = 16;
  int *d_err = nullptr;      // set by a tensor-core kernel that gave up waiting
  int tc = 1;                // bfloat16 3x3 convolutions on the tensor cores where they fit
  // tensor-core layers: packed weights (forward and backward offsets per
  // layer, -1 where the layer does not fit), the planes of one layer's output
  // gradient and the bias and head gradients' partial sums
  nn::bf16 *wp = nullptr;
  nn::bf16 *planes = nullptr;
  float *bsum = nullptr, *hp = nullptr;
  int64_t wp_n = 0, planes_n = 0;
  int64_t fwd_off[11], bwd_off[11];
  int nsm = 152;
  // activation views (offsets in act / gr), per sample sizes
  View x_in, e1, c1, s1, p1, e2, c2, s2, p2, e3, b3, d2, t2, d1, t1;
};

namespace {

#define NN_CU(x)                                                                                  \
  do {                                                                                            \
    cudaError_t e_ = (x);                                                                         \
    if (e_ != cudaSuccess)                                                                        \
      return vlb::set_error(e_ == cudaErrorMemoryAllocation ? VLB_ENOMEM : VLB_ECUDA, "%s: %s", #x, \
                            cudaGetErrorString(e_));                                              \
  } while (0)

// the tensor-core form of a 3x3 layer (bfloat16 storage): Co a power of two
// in [16, 256], H * W a multiple of 128 (whole tiles of MMA rows; it also
// puts every view of the level on a multiple of 8 elements) and Ci a
// multiple of 8
inline bool tc_shape(const vlb_nn *n, const NNLayer &l) {
  const bool pow2 = l.cout >= 16 && l.cout <= 256 && (l.cout & (l.cout - 1)) == 0;
  return n->storage == VLB_NN_BF16 && l.k == 3 && pow2 && ((int64_t)l.h * l.w) % nn::kTcM == 0 && l.cin % 8 == 0;
}
// longest rows of the input gradient's tiles
constexpr int kDgMaxRow = 256;
// its backward pass: pixel groups of 8 within a row, the positions a tap
// reaches within a block's shared memory, positions in 32 bits
inline bool tc_bwd_shape(const vlb_nn *n, const NNLayer &l) {
  return tc_shape(n, l) && l.w % 8 == 0 && l.w <= kDgMaxRow &&
         (int64_t)n->maxb * (l.h + 1) * (l.w + 1) < ((int64_t)1 << 30);
}

// Rows of the weight operand per block: the patch matrix is formed once per
// block, so as many as fit, but fewer where that leaves SMs without a block
// (coarse grids, small batches)
inline int pick_nb(const vlb_nn *n, int co, int64_t tiles, int most) {
  const int cand[5] = {128, 64, 48, 32, 16};
  int nb = 16;
  for (int c : cand)
    if (c <= most && co % c == 0) {
      nb = c;
      if (tiles * (co / c) >= n->nsm * 2 / 3) break;
    }
  return nb;
}

// A launch chained to the kernel before it (every kernel launched so begins with
// chain_begin): one pass is 17 launches, its gradients another 45, of 5 to 30 us each.
template <typename... P, typename... A>
cudaError_t chain(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, A &&...args) {
  return vlb::launch_chained(kern, grid, block, smem, (cudaStream_t)0, std::forward<A>(args)...);
}

template <int NB, bool RELU, bool EVENW>
cudaError_t launch_conv_mma(const vlb_nn *n, const NNLayer &l, const nn::bf16 *in, int64_t ibs, const nn::bf16 *wp,
                            const float *bias, nn::bf16 *out, int64_t obs, int B) {
  constexpr int smem = 2 * nn::kTcABytes + 2 * nn::kTcKG * NB * 16;
  auto kern = nn::k_conv3_mma<NB, RELU, EVENW>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)((int64_t)l.h * l.w / nn::kTcM), (unsigned)(l.cout / NB), (unsigned)B);
  chain(kern, grid, dim3(128), smem, in, ibs, l.cin, wp, l.cout, bias, out, obs, l.h, l.w, n->d_err);
  return cudaGetLastError();
}
template <bool RELU>
cudaError_t conv_mma(const vlb_nn *n, const NNLayer &l, const nn::bf16 *in, int64_t ibs, const nn::bf16 *wp,
                     const float *bias, nn::bf16 *out, int64_t obs, int B) {
  auto go = [&](auto nb, auto even) {
    return launch_conv_mma<decltype(nb)::value, RELU, decltype(even)::value>(n, l, in, ibs, wp, bias, out, obs, B);
  };
  const std::true_type even;
  if (l.w % 2) return go(std::integral_constant<int, 16>(), std::false_type());   // rows of odd width: 16-bit gathers
  switch (pick_nb(n, l.cout, (int64_t)l.h * l.w / nn::kTcM * B, 128)) {
    case 128: return go(std::integral_constant<int, 128>(), even);
    case 64: return go(std::integral_constant<int, 64>(), even);
    case 32: return go(std::integral_constant<int, 32>(), even);
    default: return go(std::integral_constant<int, 16>(), even);
  }
}

// shared memory of a block of which an SM holds two
constexpr int kDgTwoBlocks = 112 * 1024;
template <int NB>
cudaError_t launch_dgrad(const vlb_nn *n, const NNLayer &l, int64_t plane, int64_t npos, const nn::bf16 *wp, float *out,
                         int64_t obs, int B, int tiles) {
  const int stage = nn::dg_stage_bytes(NB, l.w);
  // two blocks per SM where two stages of each fit
  int nst = kDgTwoBlocks / stage;
  nst = nst < 2 ? 2 : nst > nn::kDgMaxStages ? nn::kDgMaxStages : nst;
  auto kern = nn::k_dgrad_mma<NB>;
  // the limit belongs to the kernel, not to this launch: every call sets the same one, that of
  // the widest rows, or a thread with narrower rows would lower it under another's launch
  constexpr int widest = 2 * nn::dg_stage_bytes(NB, kDgMaxRow), most = widest > kDgTwoBlocks ? widest : kDgTwoBlocks;
  static_assert(most <= 227 * 1024, "shared memory of a block");
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e != cudaSuccess) return e;
  chain(kern, dim3((unsigned)tiles, (unsigned)(l.cin / NB)), dim3(192), nst * stage, n->planes, plane, npos, l.cout,
        wp, l.cin, out, obs, l.h, l.w, B, nst, n->d_err);
  return cudaGetLastError();
}

template <int CB, int NBK>
cudaError_t launch_wgrad_t(const NNLayer &l, const nn::bf16 *in, int64_t ibs, const nn::bf16 *g, int64_t npos,
                           int64_t plane, float *dwp, int ngrp, int nsplit, int B, int *err) {
  constexpr int smem = 2 * (nn::wg_sets(CB) * nn::kWgA + NBK * nn::kWgB);
  auto kern = nn::k_wgrad_mma<CB, NBK>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)(l.cout / CB * ngrp), (unsigned)nsplit);
  chain(kern, grid, dim3(256), smem, in, ibs, l.cin, g, npos, plane, l.cout, dwp, l.h, l.w, B, ngrp, err);
  return cudaGetLastError();
}
template <int CB>
cudaError_t launch_wgrad(const NNLayer &l, const nn::bf16 *in, int64_t ibs, const nn::bf16 *g, int64_t npos,
                         int64_t plane, float *dwp, int nb, int ngrp, int nsplit, int B, int *err) {
  return nb == 2 ? launch_wgrad_t<CB, 2>(l, in, ibs, g, npos, plane, dwp, ngrp, nsplit, B, err)
                 : launch_wgrad_t<CB, 1>(l, in, ibs, g, npos, plane, dwp, ngrp, nsplit, B, err);
}

template <typename T>
int conv(const vlb_nn *n, const NNLayer &l, const T *in, int64_t ibs, const void *w, const float *bias, void *out,
         int64_t obs, bool relu, int B) {
  if constexpr (std::is_same<T, __nv_bfloat16>::value) {
    const int64_t wo = n->fwd_off[&l - n->L.data()];
    if (n->tc && wo >= 0) {
      T *ob = static_cast<T *>(out);
      NN_CU(relu ? conv_mma<true>(n, l, in, ibs, n->wp + wo, bias, ob, obs, B)
                 : conv_mma<false>(n, l, in, ibs, n->wp + wo, bias, ob, obs, B));
      return VLB_OK;
    }
  }
  const dim3 grid((unsigned)(((l.w + nn::kTile - 1) / nn::kTile) * ((l.h + nn::kTile - 1) / nn::kTile)),
                  (unsigned)((l.cout + nn::kCo - 1) / nn::kCo), (unsigned)B);
  const bool bf = n->storage == VLB_NN_BF16;
  if (l.k == 3) {
    if (bf) {
      if (relu)
        nn::k_conv<3, T, __nv_bfloat16, T, true><<<grid, nn::kThreads>>>(
            in, ibs, (const __nv_bfloat16 *)w, bias, (T *)out, obs, l.cin, l.cout, l.h, l.w);
      else
        nn::k_conv<3, T, __nv_bfloat16, T, false><<<grid, nn::kThreads>>>(
            in, ibs, (const __nv_bfloat16 *)w, bias, (T *)out, obs, l.cin, l.cout, l.h, l.w);
    } else {
      if (relu)
        nn::k_conv<3, T, float, T, true><<<grid, nn::kThreads>>>(in, ibs, (const float *)w, bias, (T *)out, obs, l.cin,
                                                                  l.cout, l.h, l.w);
      else
        nn::k_conv<3, T, float, T, false><<<grid, nn::kThreads>>>(in, ibs, (const float *)w, bias, (T *)out, obs,
                                                                   l.cin, l.cout, l.h, l.w);
    }
  } else {
    // the 1x1 head writes FP32 outputs
    constexpr int NCO = 4;
    const int HW = l.h * l.w;
    const dim3 hg((unsigned)((HW + 255) / 256), (unsigned)B, (unsigned)((l.cout + NCO - 1) / NCO));
    if (bf)
      chain(nn::k_head<T, __nv_bfloat16, NCO>, hg, dim3(128), 0, in, ibs, (const __nv_bfloat16 *)w, bias,
            (float *)out, obs, l.cin, l.cout, HW);
    else
      chain(nn::k_head<T, float, NCO>, hg, dim3(128), 0, in, ibs, (const float *)w, bias, (float *)out, obs, l.cin,
            l.cout, HW);
  }
  NN_CU(cudaGetLastError());
  return VLB_OK;
}

// gradient with respect to the input of layer l: gin = conv(gout; w^T flipped)
int conv_bwd_data(vlb_nn *n, const NNLayer &l, const float *gout, int64_t gobs, float *gin, int64_t gibs, int B) {
  const int KK = l.k * l.k;
  const int64_t nw = (int64_t)l.cin * l.cout * KK;
  if (n->storage == VLB_NN_BF16)
    nn::k_transpose_flip<__nv_bfloat16><<<nn::nblk(nw), 256>>>((const __nv_bfloat16 *)n->pc + l.woff, n->wt, l.cin,
                                                                l.cout, KK);
  else
    nn::k_transpose_flip<float><<<nn::nblk(nw), 256>>>(n->p + l.woff, n->wt, l.cin, l.cout, KK);
  NN_CU(cudaGetLastError());
  const dim3 grid((unsigned)(((l.w + nn::kTile - 1) / nn::kTile) * ((l.h + nn::kTile - 1) / nn::kTile)),
                  (unsigned)((l.cin + nn::kCo - 1) / nn::kCo), (unsigned)B);
  if (l.k == 3)
    nn::k_conv<3, float, float, float, false><<<grid, nn::kThreads>>>(gout, gobs, n->wt, nullptr, gin, gibs, l.cout,
                                                                      l.cin, l.h, l.w);
  else
    nn::k_conv<1, float, float, float, false><<<grid, nn::kThreads>>>(gout, gobs, n->wt, nullptr, gin, gibs, l.cout,
                                                                      l.cin, l.h, l.w);
  NN_CU(cudaGetLastError());
  return VLB_OK;
}

// weight and bias gradients of layer l from its input (activations) and gout
template <typename T>
int conv_bwd_weight(vlb_nn *n, const NNLayer &l, const T *in, int64_t ibs, const float *gout, int64_t gobs, int B) {
  const int KK = l.k * l.k;
  const dim3 grid((unsigned)((l.cout + 15) / 16), (unsigned)((l.cin + 7) / 8), (unsigned)n->nsplit);
  if (l.k == 3)
    nn::k_conv_dw<3, T><<<grid, 128>>>(in, ibs, gout, gobs, n->dwp, l.cin, l.cout, l.h, l.w, B);
  else
    nn::k_conv_dw<1, T><<<grid, 128>>>(in, ibs, gout, gobs, n->dwp, l.cin, l.cout, l.h, l.w, B);
  NN_CU(cudaGetLastError());
  const int64_t nw = (int64_t)l.cout * l.cin * KK;
  nn::k_sum_splits<<<nn::nblk(nw), 256>>>(n->dwp, n->nsplit, nw, n->g + l.woff);
  NN_CU(cudaGetLastError());
  nn::k_bias_grad<<<l.cout, 256>>>(gout, gobs, (int64_t)l.h * l.w, B, n->g + l.boff);
  NN_CU(cudaGetLastError());
  return VLB_OK;
}

template <typename T>
int relu_mask(float *g, int64_t gbs, const T *act, int64_t abs_, int C, int H, int W, int B) {
  const int64_t chw = (int64_t)C * H * W;
  nn::k_relu_mask<T><<<nn::nblk(chw * B), 256>>>(g, gbs, act, abs_, chw, B);
  NN_CU(cudaGetLastError());
  return VLB_OK;
}

#define NN_TRY(x)          \
  do {                     \
    const int rc_ = (x);   \
    if (rc_) return rc_;   \
  } while (0)

// wait for the stream and report a tensor-core kernel that gave up waiting
int finish(vlb_nn *n, const char *what) {
  int err = 0;
  NN_CU(cudaMemcpy(&err, n->d_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (err) {
    cudaMemset(n->d_err, 0, sizeof(int));
    return vlb::set_error(VLB_ECUDA, "%s: a tensor-core convolution gave up waiting for its MMAs", what);
  }
  return VLB_OK;
}

template <typename T>
int forward_t(vlb_nn *n, const float *d_x, float *d_y, int B) {
  T *A = static_cast<T *>(n->act);
  const void *Wp = n->storage == VLB_NN_BF16 ? n->pc : (const void *)n->p;
  auto wp = [&](const NNLayer &l) -> const void * {
    return n->storage == VLB_NN_BF16 ? (const void *)((const __nv_bfloat16 *)Wp + l.woff)
                                     : (const void *)((const float *)Wp + l.woff);
  };
  const int w = n->width, H = n->H, W = n->W, H2 = H / 2, W2 = W / 2, H4 = H / 4, W4 = W / 4;
  const auto &L = n->L;
  // input in the storage type
  const int64_t chw = (int64_t)n->ci * H * W;
  chain(nn::k_convert_into<T>, dim3(nn::nblk(chw * B)), dim3(256), 0, d_x, chw, A + n->x_in.off, n->x_in.bs, chw, B);
  NN_CU(cudaGetLastError());
  NN_TRY(conv<T>(n, L[0], A + n->x_in.off, n->x_in.bs, wp(L[0]), n->p + L[0].boff, A + n->e1.off, n->e1.bs, true, B));
  NN_TRY(conv<T>(n, L[1], A + n->e1.off, n->e1.bs, wp(L[1]), n->p + L[1].boff, A + n->s1.off, n->s1.bs, true, B));
  chain(nn::k_pool<T>, dim3((unsigned)w, (unsigned)B), dim3(256), 0, A + n->s1.off, n->s1.bs, A + n->p1.off,
        n->p1.bs, H, W);
  NN_CU(cudaGetLastError());
  NN_TRY(conv<T>(n, L[2], A + n->p1.off, n->p1.bs, wp(L[2]), n->p + L[2].boff, A + n->e2.off, n->e2.bs, true, B));
  NN_TRY(conv<T>(n, L[3], A + n->e2.off, n->e2.bs, wp(L[3]), n->p + L[3].boff, A + n->s2.off, n->s2.bs, true, B));
  chain(nn::k_pool<T>, dim3((unsigned)(2 * w), (unsigned)B), dim3(128), 0, A + n->s2.off, n->s2.bs, A + n->p2.off,
        n->p2.bs, H2, W2);
  NN_CU(cudaGetLastError());
  NN_TRY(conv<T>(n, L[4], A + n->p2.off, n->p2.bs, wp(L[4]), n->p + L[4].boff, A + n->e3.off, n->e3.bs, true, B));
  NN_TRY(conv<T>(n, L[5], A + n->e3.off, n->e3.bs, wp(L[5]), n->p + L[5].boff, A + n->b3.off, n->b3.bs, true, B));
  // c2 = [up(b3), s2]: s2 already sits in its slice
  chain(nn::k_up<T>, dim3((unsigned)(4 * w), (unsigned)B), dim3(128), 0, A + n->b3.off, n->b3.bs, A + n->c2.off,
        n->c2.bs, H4, W4);
  NN_CU(cudaGetLastError());
  NN_TRY(conv<T>(n, L[6], A + n->c2.off, n->c2.bs, wp(L[6]), n->p + L[6].boff, A + n->d2.off, n->d2.bs, true, B));
  NN_TRY(conv<T>(n, L[7], A + n->d2.off, n->d2.bs, wp(L[7]), n->p + L[7].boff, A + n->t2.off, n->t2.bs, true, B));
  chain(nn::k_up<T>, dim3((unsigned)(2 * w), (unsigned)B), dim3(256), 0, A + n->t2.off, n->t2.bs, A + n->c1.off,
        n->c1.bs, H2, W2);
  NN_CU(cudaGetLastError());
  NN_TRY(conv<T>(n, L[8], A + n->c1.off, n->c1.bs, wp(L[8]), n->p + L[8].boff, A + n->d1.off, n->d1.bs, true, B));
  NN_TRY(conv<T>(n, L[9], A + n->d1.off, n->d1.bs, wp(L[9]), n->p + L[9].boff, A + n->t1.off, n->t1.bs, true, B));
  NN_TRY(conv<T>(n, L[10], A + n->t1.off, n->t1.bs, wp(L[10]), n->p + L[10].boff, d_y, (int64_t)n->co * H * W, false, B));
  return finish(n, "vlb_nn_forward");
}

// Where the gradient of a layer's output comes from: its own slot of the
// gradient buffer (mode 0), the four children of g below an upsampling
// (mode 1; h x w of the layer's own grid), or its slot plus the gradient gp
// of its 2x2 pool (mode 2)
struct GradSrc {
  int mode;
  View g, gp;
};

// blocks of the kernels that form a layer's planes, per 8 channels: about
// eight per SM over all of them (their partial sums are added one after another)
inline int plane_blocks(const vlb_nn *n, int c, int64_t npos) {
  const int64_t want = std::max<int64_t>(1, (int64_t)n->nsm * 8 / (c / 8));
  return (int)std::min<int64_t>(want, (npos + 127) / 128);
}

// Backward pass of one 3x3 layer: its weight and bias gradients and, unless
// gin is NULL, the gradient of its input. out: its output (activation and
// gradient slot). split: its output's gradient planes and bias sums are
// there already (from the head).
template <typename T>
int layer_backward(vlb_nn *n, int li, View in, View out, const GradSrc &src, const View *gin, bool split, int B) {
  const NNLayer &l = n->L[li];
  const T *A = static_cast<const T *>(n->act);
  float *G = n->gr;
  const int64_t hw = (int64_t)l.h * l.w;
  if constexpr (std::is_same<T, __nv_bfloat16>::value) {
    if (n->tc && n->bwd_off[li] >= 0) {
      const nn::Padded pad{l.h, l.w, B};
      const int64_t npos = pad.positions(), plane = npos * l.cout;
      const int blocks = plane_blocks(n, l.cout, npos);
      if (!split) {
        const dim3 grid((unsigned)blocks, (unsigned)(l.cout / 8));
        const T *act = A + out.off;
        auto launch = [&](auto kern) {
          chain(kern, grid, dim3(128), 0, G + src.g.off, src.g.bs, G + src.gp.off, src.gp.bs, act, out.bs, n->planes,
                plane, (int)npos, n->bsum, l.h, l.w, B);
        };
        if (src.mode == 0)
          launch(nn::k_mask_split<0>);
        else if (src.mode == 1)
          launch(nn::k_mask_split<1>);
        else
          launch(nn::k_mask_split<2>);
        NN_CU(cudaGetLastError());
      }
      // weights: groups of 32 or 16 input channels per block (the gradient rows
      // are read once per group), splits to fill the SMs
      const int cb = l.cout < 128 ? l.cout : 128, nci = (l.cin + 15) / 16;
      const int nb = nci % 2 == 0 ? 2 : 1, ngrp = nci / nb;
      const int64_t nw = (int64_t)l.cin * l.cout * 9, tiles = (int64_t)(l.cout / cb) * ngrp;
      int64_t nsplit = std::min<int64_t>(n->nsm / tiles, (int64_t)B * (hw / 64));
      nsplit = std::max<int64_t>(1, std::min<int64_t>(nsplit, n->dwp_n / (nw * nn::wg_groups(cb))));
      const T *x = A + in.off;
      const int nbk = nb, ng = ngrp, ns = (int)nsplit;
      switch (cb) {
        case 16: NN_CU(launch_wgrad<16>(l, x, in.bs, n->planes, npos, plane, n->dwp, nbk, ng, ns, B, n->d_err)); break;
        case 32: NN_CU(launch_wgrad<32>(l, x, in.bs, n->planes, npos, plane, n->dwp, nbk, ng, ns, B, n->d_err)); break;
        case 64: NN_CU(launch_wgrad<64>(l, x, in.bs, n->planes, npos, plane, n->dwp, nbk, ng, ns, B, n->d_err)); break;
        default: NN_CU(launch_wgrad<128>(l, x, in.bs, n->planes, npos, plane, n->dwp, nbk, ng, ns, B, n->d_err)); break;
      }
      chain(nn::k_sum_parts, dim3(nn::nblk(nw + l.cout)), dim3(256), 0, n->dwp, ns * nn::wg_groups(cb), nw, n->bsum,
            blocks, l.cout, n->g + l.woff);
      NN_CU(cudaGetLastError());
      if (gin) {
        float *o = G + gin->off;
        const nn::bf16 *wt = n->wp + n->bwd_off[li];
        const int tiles = pad.tiles();
        switch (pick_nb(n, l.cin, tiles, 64)) {
          case 64: NN_CU(launch_dgrad<64>(n, l, plane, npos, wt, o, gin->bs, B, tiles)); break;
          case 48: NN_CU(launch_dgrad<48>(n, l, plane, npos, wt, o, gin->bs, B, tiles)); break;
          case 32: NN_CU(launch_dgrad<32>(n, l, plane, npos, wt, o, gin->bs, B, tiles)); break;
          default: NN_CU(launch_dgrad<16>(n, l, plane, npos, wt, o, gin->bs, B, tiles)); break;
        }
      }
      return VLB_OK;
    }
  }
  if (src.mode == 1)
    nn::k_up_bwd<<<nn::nblk((int64_t)B * l.cout * hw), 256>>>(G + src.g.off, src.g.bs, G + out.off, out.bs, l.cout, l.h,
                                                              l.w, B);
  if (src.mode == 2)
    nn::k_pool_bwd<<<nn::nblk((int64_t)B * l.cout * hw), 256>>>(G + src.gp.off, src.gp.bs, G + out.off, out.bs, l.cout,
                                                                l.h, l.w, B);
  NN_CU(cudaGetLastError());
  NN_TRY(relu_mask<T>(G + out.off, out.bs, A + out.off, out.bs, l.cout, l.h, l.w, B));
  NN_TRY(conv_bwd_weight<T>(n, l, A + in.off, in.bs, G + out.off, out.bs, B));
  if (gin) NN_TRY(conv_bwd_data(n, l, G + out.off, out.bs, G + gin->off, gin->bs, B));
  return VLB_OK;
}

template <int NCO>
void launch_head_bwd(vlb_nn *n, const float *d_dy, int64_t ybs, int B) {
  const NNLayer &l = n->L[10];
  const int64_t npos = nn::Padded{l.h, l.w, B}.positions();
  chain(nn::k_head_bwd<NCO>, dim3((unsigned)plane_blocks(n, l.cin, npos), (unsigned)(l.cin / 8)), dim3(128), 0, d_dy,
        ybs, (const __nv_bfloat16 *)n->pc + l.woff, (const __nv_bfloat16 *)n->act + n->t1.off, n->t1.bs, n->planes,
        npos * l.cin, (int)npos, n->bsum, n->hp, l.h, l.w, B);
}

template <typename T>
int backward_t(vlb_nn *n, const float *d_dy, int B) {
  const T *A = static_cast<const T *>(n->act);
  float *G = n->gr;
  const auto &L = n->L;
  const int64_t ybs = (int64_t)n->co * n->H * n->W;
  // the head: every gradient slot below is written before it is read
  const bool head = n->tc && n->bwd_off[9] >= 0 && n->co <= 4;
  if (head) {
    switch (n->co) {
      case 1: launch_head_bwd<1>(n, d_dy, ybs, B); break;
      case 2: launch_head_bwd<2>(n, d_dy, ybs, B); break;
      case 3: launch_head_bwd<3>(n, d_dy, ybs, B); break;
      default: launch_head_bwd<4>(n, d_dy, ybs, B);
    }
    NN_CU(cudaGetLastError());
    const int64_t nw = (int64_t)n->co * L[10].cin + n->co;
    const int blocks = plane_blocks(n, L[10].cin, nn::Padded{n->H, n->W, B}.positions());
    chain(nn::k_sum_parts, dim3(nn::nblk(nw)), dim3(256), 0, n->hp, blocks, nw, nullptr, 0, 0, n->g + L[10].woff);
    NN_CU(cudaGetLastError());
  } else {
    NN_TRY(conv_bwd_weight<T>(n, L[10], A + n->t1.off, n->t1.bs, d_dy, ybs, B));
    NN_TRY(conv_bwd_data(n, L[10], d_dy, ybs, G + n->t1.off, n->t1.bs, B));
  }
  auto own = [](View v) { return GradSrc{0, v, v}; };
  // t1 = relu(conv(d1)), d1 = relu(conv(c1))
  NN_TRY(layer_backward<T>(n, 9, n->d1, n->t1, own(n->t1), &n->d1, head, B));
  NN_TRY(layer_backward<T>(n, 8, n->c1, n->d1, own(n->d1), &n->c1, false, B));
  // c1 = [up(t2), s1]: gradient of t2 from the first 2w channels; s1's part stays in its slice
  NN_TRY(layer_backward<T>(n, 7, n->d2, n->t2, GradSrc{1, n->c1, n->c1}, &n->d2, false, B));
  NN_TRY(layer_backward<T>(n, 6, n->c2, n->d2, own(n->d2), &n->c2, false, B));
  // c2 = [up(b3), s2]
  NN_TRY(layer_backward<T>(n, 5, n->e3, n->b3, GradSrc{1, n->c2, n->c2}, &n->e3, false, B));
  NN_TRY(layer_backward<T>(n, 4, n->p2, n->e3, own(n->e3), &n->p2, false, B));
  // p2 = pool(s2): adds to s2's gradient (its slice of c2)
  NN_TRY(layer_backward<T>(n, 3, n->e2, n->s2, GradSrc{2, n->s2, n->p2}, &n->e2, false, B));
  NN_TRY(layer_backward<T>(n, 2, n->p1, n->e2, own(n->e2), &n->p1, false, B));
  // p1 = pool(s1)
  NN_TRY(layer_backward<T>(n, 1, n->e1, n->s1, GradSrc{2, n->s1, n->p1}, &n->e1, false, B));
  NN_TRY(layer_backward<T>(n, 0, n->x_in, n->e1, own(n->e1), nullptr, false, B));
  return finish(n, "vlb_nn_backward");
}

int refresh_compute_copy(vlb_nn *n) {
  if (n->storage != VLB_NN_BF16) return VLB_OK;
  nn::k_convert<__nv_bfloat16><<<nn::nblk(n->np), 256>>>(n->p, (__nv_bfloat16 *)n->pc, n->np);
  NN_CU(cudaGetLastError());
  if (n->wp) {
    nn::PackTable t;
    t.n = 10;
    int most = 1;
    for (int i = 0; i < 10; i++) {
      const NNLayer &l = n->L[i];
      t.l[i] = nn::PackLayer{l.cin, l.cout, l.woff, n->fwd_off[i], n->bwd_off[i]};
      most = std::max(most, (std::max(l.cin, l.cout) + 15) / 16);
    }
    nn::k_pack_weights<<<dim3((unsigned)(most * 16), 20), 256>>>(n->p, n->wp, t);
    NN_CU(cudaGetLastError());
  }
  return VLB_OK;
}

}  // namespace

extern "C" {

int vlb_nn_create(int32_t in_ch, int32_t out_ch, int32_t width, int32_t H, int32_t W, int32_t max_batch,
                  int32_t storage, uint64_t seed, vlb_nn **out) {
  if (!out) return vlb::set_error(VLB_EINVAL, "vlb_nn_create: out is NULL");
  *out = nullptr;
  if (in_ch < 1 || out_ch < 1 || width < 1 || H < 4 || W < 4 || (H % 4) || (W % 4) || max_batch < 1 ||
      (storage != VLB_NN_F32 && storage != VLB_NN_BF16))
    return vlb::set_error(VLB_EINVAL, "vlb_nn_create: bad shape (H and W must be multiples of 4) or storage");
  vlb_nn *n = new (std::nothrow) vlb_nn();
  if (!n) return vlb::set_error(VLB_ENOMEM, "vlb_nn_create: host allocation");
  n->ci = in_ch;
  n->co = out_ch;
  n->width = width;
  n->H = H;
  n->W = W;
  n->maxb = max_batch;
  n->storage = storage;
  const int w = width, H2 = H / 2, W2 = W / 2, H4 = H / 4, W4 = W / 4;
  const int spec[11][5] = {{in_ch, w, 3, H, W},        {w, w, 3, H, W},          {w, 2 * w, 3, H2, W2},
                           {2 * w, 2 * w, 3, H2, W2},  {2 * w, 4 * w, 3, H4, W4}, {4 * w, 4 * w, 3, H4, W4},
                           {6 * w, 2 * w, 3, H2, W2},  {2 * w, 2 * w, 3, H2, W2}, {3 * w, w, 3, H, W},
                           {w, w, 3, H, W},            {w, out_ch, 1, H, W}};
  int64_t off = 0, wmax = 0, dwmax = 0;
  for (const auto &sp : spec) {
    NNLayer l{sp[0], sp[1], sp[2], sp[3], sp[4], 0, 0};
    l.woff = off;
    off += (int64_t)l.cin * l.cout * l.k * l.k;
    l.boff = off;
    off += l.cout;
    wmax = std::max<int64_t>(wmax, (int64_t)l.cin * l.cout * l.k * l.k);
    n->L.push_back(l);
  }
  dwmax = wmax;
  n->np = off;
  // activation layout per sample (elements), in one buffer with batch stride = per-sample total
  const int64_t HW = (int64_t)H * W, HW2 = (int64_t)H2 * W2, HW4 = (int64_t)H4 * W4;
  int64_t o = 0;
  auto take = [&](int64_t sz) {
    const int64_t r = o;
    o += sz;
    return r;
  };
  const int64_t x0 = take(in_ch * HW), e10 = take(w * HW), c10 = take(3 * w * HW), p10 = take(w * HW2),
                e20 = take(2 * w * HW2), c20 = take(6 * w * HW2), p20 = take(2 * w * HW4), e30 = take(4 * w * HW4),
                b30 = take(4 * w * HW4), d20 = take(2 * w * HW2), t20 = take(2 * w * HW2), d10 = take(w * HW),
                t10 = take(w * HW);
  const int64_t per = o;
  auto V = [&](int64_t off_) { return View{off_, per}; };
  n->x_in = V(x0);
  n->e1 = V(e10);
  n->c1 = V(c10);
  n->s1 = V(c10 + 2 * w * HW);   // s1 is the second slice of c1
  n->p1 = V(p10);
  n->e2 = V(e20);
  n->c2 = V(c20);
  n->s2 = V(c20 + 4 * w * HW2);  // s2 is the second slice of c2
  n->p2 = V(p20);
  n->e3 = V(e30);
  n->b3 = V(b30);
  n->d2 = V(d20);
  n->t2 = V(t20);
  n->d1 = V(d10);
  n->t1 = V(t10);
  n->act_n = per * max_batch;
  n->wt_n = wmax;
  n->dwp_n = dwmax * n->nsplit;
  const size_t es = storage == VLB_NN_BF16 ? 2 : 4;
  // tensor-core layers: packed weights and the largest layer's gradient planes
  auto steps = [](int c) { return (int64_t)((c + nn::kTcCh - 1) / nn::kTcCh) * nn::kTcKG * 8; };
  for (int i = 0; i < 11; i++) {
    const NNLayer &l = n->L[i];
    n->fwd_off[i] = n->bwd_off[i] = -1;
    if (tc_shape(n, l)) {
      n->fwd_off[i] = n->wp_n;
      n->wp_n += steps(l.cin) * l.cout;
    }
    // (the first layer's input gradient is not needed; its packed rows, 8 input
    // channels, would not fill an MMA, and its offset only marks the fit)
    if (tc_bwd_shape(n, l) && (i == 0 || l.cin % 16 == 0)) {
      n->bwd_off[i] = n->wp_n;
      n->wp_n += steps(l.cout) * l.cin;
      n->planes_n = std::max<int64_t>(n->planes_n, 3 * l.cout * nn::Padded{l.h, l.w, max_batch}.positions());
    }
  }
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n->nsm, cudaDevAttrMultiProcessorCount, dev);
  // partial sums: at most 64 nsm channels x blocks, and the blocks' head parts
  const int64_t bs_n = std::max<int64_t>(64 * (int64_t)n->nsm, 256),
                hp_n = std::max<int64_t>(1, (int64_t)n->nsm * 8 / std::max(1, w / 8)) * ((int64_t)out_ch * w + out_ch);
  cudaError_t e = cudaMalloc(&n->p, sizeof(float) * n->np);
  if (e == cudaSuccess && n->wp_n) e = cudaMalloc(&n->wp, sizeof(nn::bf16) * n->wp_n);
  if (e == cudaSuccess && n->planes_n) e = cudaMalloc(&n->planes, sizeof(nn::bf16) * n->planes_n);
  if (e == cudaSuccess && n->planes_n) e = cudaMalloc(&n->bsum, sizeof(float) * bs_n);
  if (e == cudaSuccess && n->planes_n)
    e = cudaMalloc(&n->hp, sizeof(float) * hp_n);
  if (e == cudaSuccess) e = cudaMalloc(&n->g, sizeof(float) * n->np);
  if (e == cudaSuccess) e = cudaMalloc(&n->m, sizeof(float) * n->np);
  if (e == cudaSuccess) e = cudaMalloc(&n->v, sizeof(float) * n->np);
  if (e == cudaSuccess && storage == VLB_NN_BF16) e = cudaMalloc(&n->pc, 2 * n->np);
  if (e == cudaSuccess) e = cudaMalloc(&n->act, es * n->act_n);
  if (e == cudaSuccess) e = cudaMalloc(&n->gr, sizeof(float) * n->act_n);
  if (e == cudaSuccess) e = cudaMalloc(&n->wt, sizeof(float) * n->wt_n);
  if (e == cudaSuccess) e = cudaMalloc(&n->dwp, sizeof(float) * n->dwp_n);
  if (e == cudaSuccess) e = cudaMalloc(&n->lossp, sizeof(double) * 1024);
  if (e == cudaSuccess) e = cudaMalloc(&n->d_err, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(n->d_err, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(n->g, 0, sizeof(float) * n->np);
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, sizeof(float) * n->np);
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, sizeof(float) * n->np);
  if (e == cudaSuccess) e = cudaMemset(n->p, 0, sizeof(float) * n->np);
  if (e == cudaSuccess) e = cudaMemset(n->act, 0, es * n->act_n);
  for (size_t i = 0; i < n->L.size() && e == cudaSuccess; i++) {
    const NNLayer &l = n->L[i];
    const int64_t nw = (int64_t)l.cin * l.cout * l.k * l.k;
    const float bound = (float)std::sqrt(6.0 / ((double)l.cin * l.k * l.k));
    nn::k_init_params<<<nn::nblk(nw), 256>>>(n->p, l.woff, nw, bound, seed);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    vlb_nn_destroy(n);
    return vlb::set_error(e == cudaErrorMemoryAllocation ? VLB_ENOMEM : VLB_ECUDA, "vlb_nn_create: %s",
                          cudaGetErrorString(e));
  }
  const int rc = refresh_compute_copy(n);
  if (rc) {
    vlb_nn_destroy(n);
    return rc;
  }
  *out = n;
  return VLB_OK;
}

int vlb_nn_num_params(const vlb_nn *n, int64_t *np) {
  if (!n || !np) return vlb::set_error(VLB_EINVAL, "vlb_nn_num_params: NULL argument");
  *np = n->np;
  return VLB_OK;
}

int vlb_nn_get_params(const vlb_nn *n, float *host) {
  if (!n || !host) return vlb::set_error(VLB_EINVAL, "vlb_nn_get_params: NULL argument");
  NN_CU(cudaMemcpy(host, n->p, sizeof(float) * n->np, cudaMemcpyDeviceToHost));
  return VLB_OK;
}

int vlb_nn_set_params(vlb_nn *n, const float *host) {
  if (!n || !host) return vlb::set_error(VLB_EINVAL, "vlb_nn_set_params: NULL argument");
  NN_CU(cudaMemcpy(n->p, host, sizeof(float) * n->np, cudaMemcpyHostToDevice));
  NN_TRY(refresh_compute_copy(n));
  NN_CU(cudaDeviceSynchronize());
  return VLB_OK;
}

int vlb_nn_set_tensor_cores(vlb_nn *n, int32_t enable) {
  if (!n) return vlb::set_error(VLB_EINVAL, "vlb_nn_set_tensor_cores: NULL net");
  n->tc = enable ? 1 : 0;
  return VLB_OK;
}

int vlb_nn_forward(vlb_nn *n, const float *d_x, float *d_y, int32_t batch) {
  if (!n || !d_x || !d_y || batch < 1 || batch > n->maxb)
    return vlb::set_error(VLB_EINVAL, "vlb_nn_forward: NULL argument or batch outside [1, max_batch]");
  return n->storage == VLB_NN_BF16 ? forward_t<__nv_bfloat16>(n, d_x, d_y, batch) : forward_t<float>(n, d_x, d_y, batch);
}

int vlb_nn_mse(vlb_nn *n, const float *d_y, const float *d_target, float *d_dy, int32_t batch, double *loss) {
  if (!n || !d_y || !d_target || !d_dy || !loss || batch < 1 || batch > n->maxb)
    return vlb::set_error(VLB_EINVAL, "vlb_nn_mse: NULL argument or bad batch");
  const int64_t cnt = (int64_t)batch * n->co * n->H * n->W;
  const int blocks = 1024;
  nn::k_mse<<<blocks, 256>>>(d_y, d_target, d_dy, cnt, n->lossp);
  NN_CU(cudaGetLastError());
  std::vector<double> h(blocks);
  NN_CU(cudaMemcpy(h.data(), n->lossp, sizeof(double) * blocks, cudaMemcpyDeviceToHost));
  double s = 0.0;
  for (double x : h) s += x;
  *loss = s / (double)cnt;
  return VLB_OK;
}

int vlb_nn_backward(vlb_nn *n, const float *d_dy, int32_t batch) {
  if (!n || !d_dy || batch < 1 || batch > n->maxb)
    return vlb::set_error(VLB_EINVAL, "vlb_nn_backward: NULL argument or bad batch");
  return n->storage == VLB_NN_BF16 ? backward_t<__nv_bfloat16>(n, d_dy, batch) : backward_t<float>(n, d_dy, batch);
}

int vlb_nn_get_grads(const vlb_nn *n, float *host) {
  if (!n || !host) return vlb::set_error(VLB_EINVAL, "vlb_nn_get_grads: NULL argument");
  NN_CU(cudaMemcpy(host, n->g, sizeof(float) * n->np, cudaMemcpyDeviceToHost));
  return VLB_OK;
}

int vlb_nn_adam(vlb_nn *n, float lr, float beta1, float beta2, float eps, int64_t t) {
  if (!n || t < 1) return vlb::set_error(VLB_EINVAL, "vlb_nn_adam: NULL net or t < 1");
  const float c1 = 1.0f - (float)std::pow((double)beta1, (double)t);
  const float c2 = 1.0f - (float)std::pow((double)beta2, (double)t);
  nn::k_adam<<<nn::nblk(n->np), 256>>>(n->p, n->g, n->m, n->v, n->np, lr, beta1, beta2, eps, c1, c2);
  NN_CU(cudaGetLastError());
  NN_TRY(refresh_compute_copy(n));
  NN_CU(cudaDeviceSynchronize());
  return VLB_OK;
}

void vlb_nn_destroy(vlb_nn *n) {
  if (!n) return;
  cudaDeviceSynchronize();
  cudaFree(n->p);
  cudaFree(n->g);
  cudaFree(n->m);
  cudaFree(n->v);
  if (n->pc) cudaFree(n->pc);
  cudaFree(n->act);
  cudaFree(n->gr);
  cudaFree(n->wt);
  cudaFree(n->dwp);
  cudaFree(n->lossp);
  if (n->d_err) cudaFree(n->d_err);
  if (n->wp) cudaFree(n->wp);
  if (n->planes) cudaFree(n->planes);
  if (n->bsum) cudaFree(n->bsum);
  if (n->hp) cudaFree(n->hp);
  delete n;
}

}  // extern "C"
