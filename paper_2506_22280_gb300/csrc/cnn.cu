// Weight-predictor CNN: a downsampled projection (128 x 128) and its gantry angle -> the projection's R
// low-rank temporal weights, used as the warm start of the per-projection weights of a reconstruction.
// (Not part of the paper; it learns the inverse of the forward model from pairs the forward model
// renders.)
//
// Network: four 3 x 3 convolutions of stride 2 and padding 1 (1 -> 32 -> 64 -> 128 -> 128 channels,
// 128^2 -> 64^2 -> 32^2 -> 16^2 -> 8^2), each followed by ReLU; the 8 x 8 x 128 features and
// (cos theta, sin theta) feed a 128-unit ReLU layer and a linear layer to R outputs.  Activations are
// NHWC.  With rows = output pixels and columns = (ky, kx, c) of the inputs they read, a convolution is a product with
// the transposed weight matrix W[Co][ky][kx][Ci], and every layer, forward and backward, one of three forms:
//   forward      Y[M][N]  = X[M][K] W[N][K]^T      (+ bias, ReLU)
//   data grad    dX[M][K] = dY[M][N] W[N][K]
//   weight grad  dW[N][K] = dY[M][N]^T X[M][K]     (split over M, partials summed in a fixed order)
// X is read in place, never written out.  The forward and backward run either in FP32 on the SIMT pipes (cnn_f32.cu)
// or, with DIGS_CNN_TENSOR_CORES, with the large products (the convolutions but the first, and the 8194-wide layer)
// on the tensor cores (cnn_tc.cu, cnn_conv.cu): BF16 activations, gradients and weights, FP32 accumulation; the R-wide
// output layer stays FP32.  Inference runs the tensor-core forward.
#include <cuda_bf16.h>

#include <algorithm>

#include "digs_internal.h"

namespace digs {

namespace {

constexpr int kConvs = 4;
constexpr int kCh[kConvs + 1] = {1, 32, 64, 128, 128};
constexpr int kFeat = 8 * 8 * 128;
constexpr int kFeatIn = kFeat + 2;
constexpr int kHid = 128;
constexpr int kMaxBatch = 1024;
constexpr int kFc2Blocks = 16;  // blocks of the output layer's weight gradient

struct ParamOffsets {
  size_t w[kConvs], b[kConvs], w1, b1, w2, b2, total;
};

ParamOffsets param_offsets(int R) {
  ParamOffsets o;
  size_t off = 0;
  for (int l = 0; l < kConvs; ++l) {
    o.w[l] = off;
    off += (size_t)kCh[l + 1] * 9 * kCh[l];
    o.b[l] = off;
    off += kCh[l + 1];
  }
  o.w1 = off;
  off += (size_t)kHid * kFeatIn;
  o.b1 = off;
  off += kHid;
  o.w2 = off;
  off += (size_t)R * kHid;
  o.b2 = off;
  off += R;
  o.total = off;
  return o;
}

size_t kdim(int l) { return (size_t)9 * kCh[l]; }

// Workspace of one batch: activations for the backward, gradients, split-K partials, BF16 copies.
struct CnnWs {
  float *h, *out, *dout, *dh, *part, *loss;
  CnnF32 f32;  // the FP32 path's activations, gradients and partial sums (cnn_f32.cu)
  CnnTc tc;  // the tensor-core path's BF16 activations, gradients and weight copies (cnn_tc.cu)
  size_t bytes;
};

CnnWs cnn_layout(void* base, int B, int R) {
  CnnWs w;
  size_t off = 0;
  char* p = (char*)base;
  auto take = [&](size_t bytes) -> char* {
    char* q = p ? p + off : nullptr;
    off += (bytes + 255) & ~(size_t)255;
    return q;
  };
  w.h = (float*)take((size_t)B * kHid * 4);
  w.out = (float*)take((size_t)B * R * 4 + 4);
  w.dout = (float*)take((size_t)B * R * 4 + 4);
  w.dh = (float*)take((size_t)B * kHid * 4);
  w.part = (float*)take((size_t)kFc2Blocks * R * (kHid + 1) * 4);  // output-layer weight-gradient partials
  w.loss = (float*)take(256);
  off += cnn_f32_layout(p ? p + off : nullptr, B, &w.f32);
  off += cnn_tc_layout(p ? p + off : nullptr, B, &w.tc);
  w.bytes = off;
  return w;
}

// The R-wide output layer, FP32: out[b][r] = b2[r] + sum_n h[b][n] W2[r][n], one warp per batch entry.
__global__ void __launch_bounds__(256) k_fc2_fwd(const float* __restrict__ h, const float* __restrict__ w2,
                                                 const float* __restrict__ b2, int B, int R, float* __restrict__ out) {
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (b >= B) return;  // whole warps
  float x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) x[q] = h[(size_t)b * kHid + lane + 32 * q];
  for (int r = 0; r < R; ++r) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) s = fmaf(x[q], w2[r * kHid + lane + 32 * q], s);
    s = warp_sum(s);
    if (lane == 0) out[(size_t)b * R + r] = s + b2[r];
  }
}

// Its parameter gradient, per block of batch entries (blockIdx.x selects entries b = blockIdx.x,
// blockIdx.x + gridDim.x, ...): part[block][r kHid + n] = sum_b dout[b][r] h[b][n] (threads n < kHid) and
// part[block][R kHid + r] = sum_b dout[b][r] (threads kHid + r); the blocks are added in order after.
__global__ void __launch_bounds__(kHid + 32) k_fc2_wgrad(const float* __restrict__ dout, const float* __restrict__ h,
                                                         int B, int R, float* __restrict__ part) {
  const int n = threadIdx.x;
  float acc[DIGS_MAX_R] = {0.f, 0.f, 0.f, 0.f};
  if (n < kHid) {
    for (int b = blockIdx.x; b < B; b += gridDim.x) {
      const float x = h[(size_t)b * kHid + n];
#pragma unroll
      for (int r = 0; r < DIGS_MAX_R; ++r)
        if (r < R) acc[r] = fmaf(dout[(size_t)b * R + r], x, acc[r]);
    }
    for (int r = 0; r < R; ++r) part[(size_t)blockIdx.x * (R * kHid + R) + r * kHid + n] = acc[r];
  } else if (n - kHid < R) {
    const int r = n - kHid;
    float t = 0.f;
    for (int b = blockIdx.x; b < B; b += gridDim.x) t += dout[(size_t)b * R + r];
    part[(size_t)blockIdx.x * (R * kHid + R) + R * kHid + r] = t;
  }
}

// dh[b][n] = [h[b][n] > 0] sum_r dout[b][r] W2[r][n]: the gradient of the dense layer's pre-activation.
// dh = dL/d(dense pre-activation), masked by the dense layer's ReLU; with dhb, also its BF16 copy (the
// tensor-core backward's operand).
__global__ void k_fc2_dh(const float* __restrict__ dout, const float* __restrict__ w2, const float* __restrict__ h,
                         int B, int R, float* __restrict__ dh, uint16_t* __restrict__ dhb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * kHid) return;
  const int b = i / kHid, n = i - b * kHid;
  float s = 0.f;
  for (int r = 0; r < R; ++r) s = fmaf(dout[(size_t)b * R + r], w2[r * kHid + n], s);
  const float v = h[i] <= 0.f ? 0.f : s;  // h is NaN where its kernels gave up waiting: so is dh then
  dh[i] = v;
  if (dhb) dhb[i] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
}

// out[i] (+)= sum_z part[z][i], z in a fixed order.
__global__ void k_sum_splits(const float* __restrict__ part, int splits, long long n, float* __restrict__ out,
                             int accumulate) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float s = accumulate ? out[i] : 0.f;
  for (int z = 0; z < splits; ++z) s += part[(size_t)z * n + i];
  out[i] = s;
}

unsigned grid_for(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 152LL * 32); }

// loss = mean (out - target)^2 over B x R; dout = 2 (out - target) / (B R).  One block.
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ out, const float* __restrict__ target, int n,
                                             float* __restrict__ dout, float* __restrict__ loss) {
  __shared__ float red[8];
  float s = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float r = out[i] - target[i];
    dout[i] = 2.f * r / (float)n;
    s = fmaf(r, r, s);
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int k = 0; k < 8; ++k) t += red[k];
    *loss = t / (float)n;
  }
}

// The network input [B][128][128] of a projection stack [B][nv][nu], times `scale`: the 2 x 2 means of
// 256 x 256 projections, or 128 x 128 projections as they are.
__global__ void k_downsample(const float* __restrict__ proj, int B, int nu, int nv, float scale,
                             float* __restrict__ img) {
  const int f = nu / 128;  // 2: 2 x 2 means of a 256 x 256 projection; 1: a 128 x 128 one, scaled
  const long long total = (long long)B * 128 * 128;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % 128), y = (int)((i / 128) % 128), b = (int)(i / (128LL * 128));
    const float* p = proj + ((size_t)b * nv + f * y) * nu + f * x;
    img[i] = f == 2 ? 0.25f * scale * (p[0] + p[1] + p[nu] + p[nu + 1]) : scale * p[0];
  }
}

// He-normal weights (std sqrt(2 / fan_in)) from a counter-based generator (splitmix64 of seed and index,
// Box-Muller), zero biases.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void k_init(float* __restrict__ p, long long n, unsigned long long seed, float std_dev, int is_bias) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (is_bias) { p[i] = 0.f; continue; }
    const unsigned long long r = splitmix64(seed ^ splitmix64((unsigned long long)i));
    const float u1 = ((float)(r >> 40) + 1.f) * (1.f / 16777217.f);          // (0, 1]
    const float u2 = (float)((r >> 16) & 0xFFFFFFull) * (1.f / 16777216.f);  // [0, 1)
    p[i] = std_dev * sqrtf(-2.f * logf(u1)) * cospif(2.f * u2);
  }
}

struct NetPtrs {
  const float *w[kConvs], *b[kConvs], *w1, *b1, *w2, *b2;
};

NetPtrs net_ptrs(const float* p, const ParamOffsets& o) {
  NetPtrs n;
  for (int l = 0; l < kConvs; ++l) {
    n.w[l] = p + o.w[l];
    n.b[l] = p + o.b[l];
  }
  n.w1 = p + o.w1;
  n.b1 = p + o.b1;
  n.w2 = p + o.w2;
  n.b2 = p + o.b2;
  return n;
}

#define CNN_TRY(...)                         \
  do {                                       \
    cudaError_t e__ = (__VA_ARGS__);         \
    if (e__ != cudaSuccess) return e__;      \
  } while (0)

CnnNet cnn_net(const NetPtrs& N) {
  CnnNet n;
  for (int l = 0; l < kConvs; ++l) {
    n.w[l] = N.w[l];
    n.b[l] = N.b[l];
  }
  n.w1 = N.w1;
  n.b1 = N.b1;
  return n;
}

// Forward keeping every activation in the workspace for the backward.  tc: the tensor-core path of
// cnn_tc.cu up to the dense layer's output (BF16 activations), else the FP32 SIMT GEMMs of cnn_f32.cu; the
// R-wide output layer is FP32 either way.
cudaError_t forward_f32(const NetPtrs& N, int R, const float* img, const float* cs, int B, const CnnWs& w,
                        bool tc, cudaStream_t st) {
  if (tc) {
    CNN_TRY(cnn_tc_forward(cnn_net(N), img, cs, B, w.tc, w.h, st));
  } else {
    CNN_TRY(cnn_f32_forward(cnn_net(N), img, cs, B, w.f32, w.h, st));
  }
  k_fc2_fwd<<<(B + 7) / 8, 256, 0, st>>>(w.h, N.w2, N.b2, B, R, w.out);
  note_launches(1);
  return cudaGetLastError();
}

// Backward of forward_f32 for dL/dout in w.dout; writes every parameter gradient to grad (layout as params).
cudaError_t backward_f32(const NetPtrs& N, const ParamOffsets& o, int R, int B, const CnnWs& w, float* grad,
                         bool tc, cudaStream_t st) {
  // output layer
  k_fc2_wgrad<<<kFc2Blocks, kHid + 32, 0, st>>>(w.dout, w.h, B, R, w.part);
  k_sum_splits<<<(R * kHid + R + 255) / 256, 256, 0, st>>>(w.part, kFc2Blocks, R * kHid + R, grad + o.w2, 0);
  k_fc2_dh<<<(B * kHid + 255) / 256, 256, 0, st>>>(w.dout, N.w2, w.h, B, R, w.dh, tc ? w.tc.dhb : nullptr);
  note_launches(3);
  CNN_TRY(cnn_colsum(w.dh, B, kHid, w.tc, grad + o.b1, st));
  CnnGrad g;
  for (int l = 0; l < kConvs; ++l) {
    g.w[l] = grad + o.w[l];
    g.b[l] = grad + o.b[l];
  }
  g.w1 = grad + o.w1;
  return tc ? cnn_tc_backward(B, w.tc, w.dh, g, st) : cnn_f32_backward(cnn_net(N), B, w.f32, w.tc, w.dh, g, st);
}

bool args_ok(int R, int B) { return R >= 1 && R <= DIGS_MAX_R && B >= 1 && B <= kMaxBatch; }

}  // namespace
}  // namespace digs

using namespace digs;

extern "C" {

size_t digs_cnn_params(int R) { return (R >= 1 && R <= DIGS_MAX_R) ? param_offsets(R).total : 0; }

size_t digs_cnn_workspace_size(int B, int R) { return args_ok(R, B) ? cnn_layout(nullptr, B, R).bytes : 0; }

digs_status digs_cnn_init(float* params, int R, unsigned long long seed, void* stream) {
  if (!params || R < 1 || R > DIGS_MAX_R) return DIGS_ERR_ARG;
  const ParamOffsets o = param_offsets(R);
  cudaStream_t st = (cudaStream_t)stream;
  auto init = [&](size_t off, long long n, int fan_in, int is_bias) {
    k_init<<<grid_for(n), 256, 0, st>>>(params + off, n, seed + off, sqrtf(2.f / (float)fan_in), is_bias);
    note_launches(1);
  };
  for (int l = 0; l < kConvs; ++l) {
    init(o.w[l], (long long)kCh[l + 1] * kdim(l), (int)kdim(l), 0);
    init(o.b[l], kCh[l + 1], 1, 1);
  }
  init(o.w1, (long long)kHid * kFeatIn, kFeatIn, 0);
  init(o.b1, kHid, 1, 1);
  init(o.w2, (long long)R * kHid, kHid, 0);
  init(o.b2, R, 1, 1);
  return cudaGetLastError() == cudaSuccess ? DIGS_OK : DIGS_ERR_CUDA;
}

digs_status digs_cnn_prepare_input(const float* proj, int B, int nu, int nv, float scale, float* img, void* stream) {
  if (!proj || !img || B < 1 || nu != nv || (nu != 256 && nu != 128)) return DIGS_ERR_ARG;
  k_downsample<<<grid_for((long long)B * 128 * 128), 256, 0, (cudaStream_t)stream>>>(proj, B, nu, nv, scale, img);
  note_launches(1);
  return cudaGetLastError() == cudaSuccess ? DIGS_OK : DIGS_ERR_CUDA;
}

digs_status digs_cnn_forward(const float* params, int R, const float* img, const float* cs, int B, float* w_out,
                             int flags, void* ws, size_t ws_bytes, void* stream) {
  if (!params || !img || !cs || !w_out || !ws || !args_ok(R, B)) return DIGS_ERR_ARG;
  const CnnWs w = cnn_layout(ws, B, R);
  if (w.bytes > ws_bytes) return DIGS_ERR_ARG;
  const ParamOffsets o = param_offsets(R);
  cudaStream_t st = (cudaStream_t)stream;
  const bool tc = (flags & DIGS_CNN_TENSOR_CORES) != 0;
  if (forward_f32(net_ptrs(params, o), R, img, cs, B, w, tc, st) != cudaSuccess) return DIGS_ERR_CUDA;
  if (cudaMemcpyAsync(w_out, w.out, (size_t)B * R * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return DIGS_ERR_CUDA;
  return DIGS_OK;
}

digs_status digs_cnn_backward(const float* params, int R, int B, const float* grad_w, float* grad_params, int flags,
                              void* ws, size_t ws_bytes, void* stream) {
  if (!params || !grad_w || !grad_params || !ws || !args_ok(R, B)) return DIGS_ERR_ARG;
  const CnnWs w = cnn_layout(ws, B, R);
  if (w.bytes > ws_bytes) return DIGS_ERR_ARG;
  const ParamOffsets o = param_offsets(R);
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(w.dout, grad_w, (size_t)B * R * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return DIGS_ERR_CUDA;
  const bool tc = (flags & DIGS_CNN_TENSOR_CORES) != 0;
  if (backward_f32(net_ptrs(params, o), o, R, B, w, grad_params, tc, st) != cudaSuccess)
    return DIGS_ERR_CUDA;
  return DIGS_OK;
}

digs_status digs_cnn_train_step(float* params, float* m, float* v, float* grad, int step, float lr, int R,
                                const float* img, const float* cs, const float* target, int B, float* loss_out,
                                int flags, void* ws, size_t ws_bytes, void* stream) {
  if (!params || !m || !v || !grad || !img || !cs || !target || !loss_out || !ws || step < 1 || !args_ok(R, B))
    return DIGS_ERR_ARG;
  const CnnWs w = cnn_layout(ws, B, R);
  if (w.bytes > ws_bytes) return DIGS_ERR_ARG;
  const ParamOffsets o = param_offsets(R);
  cudaStream_t st = (cudaStream_t)stream;
  const NetPtrs N = net_ptrs(params, o);
  const bool tc = (flags & DIGS_CNN_TENSOR_CORES) != 0;
  if (forward_f32(N, R, img, cs, B, w, tc, st) != cudaSuccess) return DIGS_ERR_CUDA;
  k_mse<<<1, 256, 0, st>>>(w.out, target, B * R, w.dout, loss_out);
  note_launches(1);
  if (backward_f32(N, o, R, B, w, grad, tc, st) != cudaSuccess) return DIGS_ERR_CUDA;
  AdamGroup g{params, grad, m, v, (long long)o.total, 0, 0, lr, lr};
  if (launch_adam(&g, 1, 0.9f, 0.999f, 1e-8f, step, nullptr, 0, st) != cudaSuccess) return DIGS_ERR_CUDA;
  return DIGS_OK;
}

digs_status digs_cnn_infer_bf16(const float* params, int R, const float* img, const float* cs, int B, float* w_out,
                                void* ws, size_t ws_bytes, void* stream) {
  if (!params || !img || !cs || !w_out || !ws || !args_ok(R, B)) return DIGS_ERR_ARG;
  const CnnWs w = cnn_layout(ws, B, R);
  if (w.bytes > ws_bytes) return DIGS_ERR_ARG;
  const ParamOffsets o = param_offsets(R);
  cudaStream_t st = (cudaStream_t)stream;
  const NetPtrs N = net_ptrs(params, o);
  if (cnn_tc_forward(cnn_net(N), img, cs, B, w.tc, w.h, st) != cudaSuccess) return DIGS_ERR_CUDA;
  k_fc2_fwd<<<(B + 7) / 8, 256, 0, st>>>(w.h, N.w2, N.b2, B, R, w_out);
  note_launches(1);
  if (cudaGetLastError() != cudaSuccess) return DIGS_ERR_CUDA;
  return DIGS_OK;
}

}  // extern "C"
