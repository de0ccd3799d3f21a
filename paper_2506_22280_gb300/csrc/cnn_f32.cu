// The weight-predictor CNN in FP32 on the SIMT pipes: the exact reference of the tensor-core path and the
// default mode of its forward and backward calls.
//
// Every contraction is one launch of one kernel template over BM x BN tiles of C, its operands read in place by
// loaders (the same three forms as the tensor-core path): the forward convolution gathers its im2col rows, the
// data gradient runs one GEMM per output-pixel parity class of the stride-2 convolution (no col2im), the
// weight gradient reduces over the pixels, split into partial sums that are added in a fixed order.  No
// im2col matrix is written (9/4 of a layer's input, written once and read twice before), and the ReLU masks
// are applied where a gradient is stored.
//
// Bound: FP32 FMAs (18.8 GFLOP per forward and backward at batch 64: 0.24 ms at the pipe's measured 38.6 T
// FMA/s).  A thread holds an 8 x 4 block of C: 32 FMAs per three 16-byte shared-memory reads, where the 4 x 4
// block read with scalar loads before issued one read for two FMAs.  The next K slice is in registers while
// the current one is multiplied.  Layers with few tiles split K until about two CTAs per SM have work (the
// dense layer's 64 x 128 outputs ran on two CTAs before: 1003 us of 3050).
// Forward and backward at batch 64: 3.00 -> 0.94 ms.
#include <algorithm>

#include "digs_internal.h"

namespace digs {
namespace {

constexpr int kCh[5] = {1, 32, 64, 128, 128};
constexpr int kEdge[5] = {128, 64, 32, 16, 8};
constexpr int kFeat = 8192, kFeatIn = kFeat + 2, kHid = 128;
constexpr int kBK = 16;

// ---- loaders: four consecutive elements of an operand, along K (kchunk) or along its row index (rchunk) ----
// kK says which: true for kchunk(row, k), false for rchunk(row, k) = X[row .. row + 3][k].

// Caller's arrays (parameters) need not lie on 16 bytes: vec says whether they do.
__device__ __forceinline__ float4 load4(const float* p, bool vec) {
  return vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}

struct PlainK {  // X[row][k] = p[row ld + k], any alignment and any K
  static constexpr bool kK = true;
  const float* p;
  int ld, rows, K;
  __device__ float4 kchunk(int row, int k) const {
    float v[4];
    const float* q = p + (size_t)row * ld + k;
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = row < rows && k + j < K ? q[j] : 0.f;
    return make_float4(v[0], v[1], v[2], v[3]);
  }
};

struct PlainR {  // X[row][k] = p[k ld + row]
  static constexpr bool kK = false;
  const float* p;
  int ld, rows, K;
  __device__ float4 rchunk(int row, int k) const {
    float v[4];
    const float* q = p + (size_t)k * ld + row;
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = row + j < rows && k < K ? q[j] : 0.f;
    return make_float4(v[0], v[1], v[2], v[3]);
  }
};

// im2col of a 3 x 3, stride-2, padding-1 convolution over NHWC input H x H x C (powers of two, C >= 4).
struct ConvGeom {
  const float* act;
  int H, lwo, lc, rows, cols;  // input edge; log2 output edge; log2 C; output pixels; 9 C
  __device__ float4 at(int p, int kk) const {
    if (p >= rows || kk >= cols) return make_float4(0.f, 0.f, 0.f, 0.f);
    const int tap = kk >> lc, c = kk & ((1 << lc) - 1), ky = tap / 3, kx = tap - 3 * ky;
    const int x = p & ((1 << lwo) - 1), y = (p >> lwo) & ((1 << lwo) - 1), b = p >> (2 * lwo);
    const int iy = 2 * y + ky - 1, ix = 2 * x + kx - 1;
    if (iy < 0 || iy >= H || ix < 0 || ix >= H) return make_float4(0.f, 0.f, 0.f, 0.f);
    return *reinterpret_cast<const float4*>(act + ((((size_t)b * H + iy) * H + ix) << lc) + c);
  }
};
struct ConvK {  // rows = output pixels, K = (tap, c)
  static constexpr bool kK = true;
  ConvGeom g;
  __device__ float4 kchunk(int row, int k) const { return g.at(row, k); }
};
struct ConvR {  // rows = (tap, c), K = output pixels
  static constexpr bool kK = false;
  ConvGeom g;
  __device__ float4 rchunk(int row, int k) const { return g.at(k, row); }
};

struct WeightK {  // W[co][9 C] by rows co
  static constexpr bool kK = true;
  const float* w;
  int rows, K;
  bool vec;
  __device__ float4 kchunk(int row, int k) const {
    return row < rows && k < K ? load4(w + (size_t)row * K + k, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};

// dY[pixel][co] with pixels as K (weight gradient).
struct DyR {
  static constexpr bool kK = false;
  const float* dy;
  int ld, K;
  __device__ float4 rchunk(int row, int k) const {
    return row < ld && k < K ? *reinterpret_cast<const float4*>(dy + (size_t)k * ld + row) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};

// The taps that reach the input pixels of parity class z = 2 py + px: ky = 1 (py = 0) or {0, 2}, likewise kx.
__device__ __forceinline__ int class_taps(int z) { return z == 0 ? 1 : (z == 3 ? 4 : 2); }
__device__ __forceinline__ void class_tap(int z, int t, int& ky, int& kx) {
  const int nx = (z & 1) ? 2 : 1, ty = t / nx, tx = t - ty * nx;
  ky = (z >> 1) ? 2 * ty : 1;
  kx = (z & 1) ? 2 * tx : 1;
}
struct ParityK {  // rows = (b, Y, X) of the class grid, K = (tap of the class, co)
  static constexpr bool kK = true;
  const float* dy;
  int lho, ln, rows;  // log2 output edge; log2 output channels
  __device__ float4 kchunk(int row, int k) const {
    const int z = blockIdx.z, t = k >> ln, co = k & ((1 << ln) - 1), Ho = 1 << lho;
    const int X = row & (Ho - 1), Y = (row >> lho) & (Ho - 1), b = row >> (2 * lho);
    int ky, kx;
    class_tap(z, t, ky, kx);
    const int y = (2 * Y + (z >> 1) + 1 - ky) >> 1, x = (2 * X + (z & 1) + 1 - kx) >> 1;
    if (row >= rows || y >= Ho || x >= Ho) return make_float4(0.f, 0.f, 0.f, 0.f);
    return *reinterpret_cast<const float4*>(dy + ((((((size_t)b << lho) + y) << lho) + x) << ln) + co);
  }
};
struct ClassWR {  // W[co][ky][kx][ci]: rows = ci, K = (tap of the class, co)
  static constexpr bool kK = false;
  const float* w;
  int ln, C;
  bool vec;
  __device__ float4 rchunk(int row, int k) const {
    const int t = k >> ln, co = k & ((1 << ln) - 1);
    int ky, kx;
    class_tap(blockIdx.z, t, ky, kx);
    return row < C ? load4(w + ((size_t)co * 9 + ky * 3 + kx) * C + row, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};

// ---- epilogues: one row's four consecutive columns --------------------------------------------------
struct EpiAct {  // out[row][col] = relu(v + bias[col]), rows of `ld` floats in groups (a group's rows at gld)
  float* out;
  const float* bias;
  int rows, cols, group, gld;
  __device__ void apply(int row, int col, const float v[4]) const {
    if (row >= rows) return;
    float* d = out + (size_t)(row / group) * gld + (size_t)(row % group) * cols + col;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (col + j < cols) d[j] = fmaxf(v[j] + bias[col + j], 0.f);
  }
};
struct EpiPart {  // partial sums of split blockIdx.z
  float* out;
  long long zstride;
  int rows, cols;
  __device__ void apply(int row, int col, const float v[4]) const {
    if (row >= rows) return;
    float* d = out + blockIdx.z * zstride + (size_t)row * cols + col;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (col + j < cols) d[j] = v[j];
  }
};
struct EpiDx {  // gradient of input pixel (2Y + py, 2X + px), masked by that layer's ReLU (C = cols channels)
  float* dx;
  const float* act;
  int lho, rows, cols;
  __device__ void apply(int row, int col, const float v[4]) const {
    if (row >= rows) return;
    const int z = blockIdx.z, Ho = 1 << lho, H = 2 * Ho;
    const int X = row & (Ho - 1), Y = (row >> lho) & (Ho - 1), b = row >> (2 * lho);
    const size_t at = (((size_t)b * H + 2 * Y + (z >> 1)) * H + 2 * X + (z & 1)) * cols + col;
    const float4 a = *reinterpret_cast<const float4*>(act + at);
    *reinterpret_cast<float4*>(dx + at) = make_float4(a.x > 0.f ? v[0] : 0.f, a.y > 0.f ? v[1] : 0.f,
                                                      a.z > 0.f ? v[2] : 0.f, a.w > 0.f ? v[3] : 0.f);
  }
};
struct EpiDfeat {  // dY of the last convolution [B][8192], masked by its ReLU output in feat [B][8194]
  float* dy;
  const float* feat;
  int rows;
  __device__ void apply(int row, int col, const float v[4]) const {
    if (row >= rows) return;
    const float* a = feat + (size_t)row * kFeatIn + col;
    *reinterpret_cast<float4*>(dy + (size_t)row * kFeat + col) =
        make_float4(a[0] > 0.f ? v[0] : 0.f, a[1] > 0.f ? v[1] : 0.f, a[2] > 0.f ? v[2] : 0.f, a[3] > 0.f ? v[3] : 0.f);
  }
};

// ---- the GEMM ---------------------------------------------------------------------------------------
// C(m, n) = sum over k of A(m, k) B(n, k).  Grid: (row tiles, column tiles, splits or parity classes).
// kchunk > 0: block z sums k in [z kchunk, (z + 1) kchunk), kchunk a multiple of the slice (or all of K);
// kchunk == 0: the whole K, class_k times the taps of parity class z.  Loaders give zeros past their K.
template <int BM, int BN>
struct Tile {
  static constexpr int kThreads = (BM / 8) * (BN / 4);  // 8 x 4 outputs each
};

template <int BM, int BN, class LA, class LB, class EP>
__global__ void __launch_bounds__(Tile<BM, BN>::kThreads) k_gemm_f32(const LA la, const LB lb, const EP ep, int K, int kchunk,
                                                                  int class_k) {
  constexpr int NT = Tile<BM, BN>::kThreads;
  constexpr int QA = BM * kBK / 4 / NT, QB = BN * kBK / 4 / NT;  // 16-byte chunks of a slice per thread
  static_assert(QA * NT * 4 == BM * kBK && QB * NT * 4 == BN * kBK, "whole chunks");
  __shared__ __align__(16) float As[2][kBK][BM + 4], Bs[2][kBK][BN + 4];
  const int tid = threadIdx.x, tx = tid % (BN / 4), ty = tid / (BN / 4);
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int kb = kchunk ? min(K, (int)blockIdx.z * kchunk) : 0;
  const int ke = kchunk ? min(K, kb + kchunk) : class_k * class_taps(blockIdx.z);
  float4 ra[QA], rb[QB];
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < QA; ++i) {
      const int q = tid + NT * i;
      if constexpr (LA::kK) ra[i] = la.kchunk(m0 + q % BM, k0 + (q / BM) * 4);
      else ra[i] = la.rchunk(m0 + (q % (BM / 4)) * 4, k0 + q / (BM / 4));
    }
#pragma unroll
    for (int i = 0; i < QB; ++i) {
      const int q = tid + NT * i;
      if constexpr (LB::kK) rb[i] = lb.kchunk(n0 + q % BN, k0 + (q / BN) * 4);
      else rb[i] = lb.rchunk(n0 + (q % (BN / 4)) * 4, k0 + q / (BN / 4));
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < QA; ++i) {
      const int q = tid + NT * i;
      const float v[4] = {ra[i].x, ra[i].y, ra[i].z, ra[i].w};
      if constexpr (LA::kK) {
#pragma unroll
        for (int j = 0; j < 4; ++j) As[buf][(q / BM) * 4 + j][q % BM] = v[j];
      } else {
        *reinterpret_cast<float4*>(&As[buf][q / (BM / 4)][(q % (BM / 4)) * 4]) = ra[i];
      }
    }
#pragma unroll
    for (int i = 0; i < QB; ++i) {
      const int q = tid + NT * i;
      const float v[4] = {rb[i].x, rb[i].y, rb[i].z, rb[i].w};
      if constexpr (LB::kK) {
#pragma unroll
        for (int j = 0; j < 4; ++j) Bs[buf][(q / BN) * 4 + j][q % BN] = v[j];
      } else {
        *reinterpret_cast<float4*>(&Bs[buf][q / (BN / 4)][(q % (BN / 4)) * 4]) = rb[i];
      }
    }
  };
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  if (kb < ke) {
    load(kb);
    store(0);
  }
  __syncthreads();
  int buf = 0;
  for (int k0 = kb; k0 < ke; k0 += kBK, buf ^= 1) {
    const bool more = k0 + kBK < ke;
    if (more) load(k0 + kBK);
#pragma unroll
    for (int k = 0; k < kBK; ++k) {
      float a[8], b[4];
      *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(&As[buf][k][ty * 8]);
      *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(&As[buf][k][ty * 8 + 4]);
      *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(&Bs[buf][k][tx * 4]);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) store(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) ep.apply(m0 + ty * 8 + i, n0 + tx * 4, acc[i]);
}

template <int BM, int BN, class LA, class LB, class EP>
cudaError_t gemm(const LA& la, const LB& lb, const EP& ep, int M, int N, int K, int gz, int kchunk, int class_k,
                 cudaStream_t st) {
  const dim3 grid((M + BM - 1) / BM, (N + BN - 1) / BN, gz);
  k_gemm_f32<BM, BN, LA, LB, EP><<<grid, Tile<BM, BN>::kThreads, 0, st>>>(la, lb, ep, K, kchunk, class_k);
  note_launches(1);
  return cudaGetLastError();
}

// First convolution (1 -> 32 channels) on FP32 images; the images are also kept (copy) for the backward.
__global__ void __launch_bounds__(256) k_conv0_f32(const float* __restrict__ img, const float* __restrict__ w,
                                                   const float* __restrict__ bias, int npix, float* __restrict__ out,
                                                   float* __restrict__ copy) {
  __shared__ float sw[32 * 9], sb[32];
  for (int i = threadIdx.x; i < 32 * 9; i += blockDim.x) sw[i] = w[i];
  if (threadIdx.x < 32) sb[threadIdx.x] = bias[threadIdx.x];
  __syncthreads();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npix) return;
  const int x = p & 63, y = (p >> 6) & 63, b = p >> 12;
  float xin[9];
#pragma unroll
  for (int t = 0; t < 9; ++t) {
    const int iy = 2 * y + t / 3 - 1, ix = 2 * x + t % 3 - 1;
    xin[t] = (iy >= 0 && iy < 128 && ix >= 0 && ix < 128) ? img[((size_t)b * 128 + iy) * 128 + ix] : 0.f;
  }
  float2* c = reinterpret_cast<float2*>(copy + ((size_t)b * 128 + 2 * y) * 128 + 2 * x);  // its taps 4, 5, 7, 8
  c[0] = make_float2(xin[4], xin[5]);
  c[64] = make_float2(xin[7], xin[8]);
  float4* d = reinterpret_cast<float4*>(out + (size_t)p * 32);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    float o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int co = 4 * q + j;
      float a = 0.f;  // the bias last, as every other layer's epilogue adds it
#pragma unroll
      for (int t = 0; t < 9; ++t) a = fmaf(sw[co * 9 + t], xin[t], a);
      o[j] = fmaxf(a + sb[co], 0.f);
    }
    d[q] = make_float4(o[0], o[1], o[2], o[3]);
  }
}

// The dense layer's two angle inputs: feat[b][8192 + j] = cs[b][j].
__global__ void k_feat_angles(float* __restrict__ feat, const float* __restrict__ cs, int B) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 2 * B) feat[(size_t)(i >> 1) * kFeatIn + kFeat + (i & 1)] = cs[i];
}

#define F32_TRY(...)                      \
  do {                                    \
    cudaError_t e__ = (__VA_ARGS__);      \
    if (e__ != cudaSuccess) return e__;   \
  } while (0)

bool on16(const void* p) { return ((uintptr_t)p & 15) == 0; }

// Splits of a K-long reduction over `tiles` CTAs: about four CTAs per SM, at least `least` of K each, partial
// sums of `n` outputs within `room` floats.
int splits_for(int tiles, long long K, int least, long long n, long long room) {
  long long z = std::min((4LL * 152 + tiles - 1) / tiles, std::max(1LL, K / least));
  return (int)std::max(1LL, std::min(z, room / n));
}
int chunk_of(long long K, int z) { return (int)(((K + z - 1) / z + kBK - 1) / kBK * kBK); }

// Gradients of the convolutions' outputs pass through two buffers in turn: layers 0 and 2 in dy[0], 1 and 3 in dy[1]
// (floats per image).
constexpr int out_floats(int l) { return kEdge[l + 1] * kEdge[l + 1] * kCh[l + 1]; }
constexpr int kDyFloats[2] = {out_floats(0), out_floats(1)};
static_assert(out_floats(2) <= kDyFloats[0] && out_floats(3) <= kDyFloats[1], "every layer's gradient fits its buffer");

struct Layer {
  int H, lwo, lc, ln, rows, N, K, C;
};
Layer layer(int l, int B) {
  Layer a;
  a.H = kEdge[l];
  a.lwo = l == 1 ? 5 : (l == 2 ? 4 : 3);
  a.lc = l == 1 ? 5 : (l == 2 ? 6 : 7);
  a.ln = l == 1 ? 6 : 7;
  a.rows = B * kEdge[l + 1] * kEdge[l + 1];
  a.N = kCh[l + 1];
  a.C = kCh[l];
  a.K = 9 * a.C;
  return a;
}

}  // namespace

size_t cnn_f32_layout(void* base, int B, CnnF32* t) {
  size_t off = 0;
  char* p = (char*)base;
  auto take = [&](size_t floats) -> float* {
    float* q = p ? (float*)(p + off) : nullptr;
    off += (floats * 4 + 255) & ~(size_t)255;
    return q;
  };
  CnnF32 w{};
  w.img = take((size_t)B * 128 * 128);
  for (int l = 0; l < 3; ++l) w.act[l] = take((size_t)B * kEdge[l + 1] * kEdge[l + 1] * kCh[l + 1]);
  w.feat = take((size_t)B * kFeatIn);
  for (int k = 0; k < 2; ++k) w.dy[k] = take((size_t)B * kDyFloats[k]);
  w.part_floats = std::max<long long>(16LL * B * kHid, 6LL << 20);
  w.part = take((size_t)w.part_floats);
  if (t) *t = w;
  return off;
}

cudaError_t cnn_f32_forward(const CnnNet& net, const float* img, const float* cs, int B, const CnnF32& t, float* h,
                            cudaStream_t st) {
  const int npix = B * 4096;
  k_conv0_f32<<<(npix + 255) / 256, 256, 0, st>>>(img, net.w[0], net.b[0], npix, t.act[0], t.img);
  note_launches(1);
  for (int l = 1; l < 4; ++l) {
    const Layer a = layer(l, B);
    const ConvK A{ConvGeom{t.act[l - 1], a.H, a.lwo, a.lc, a.rows, a.K}};
    const WeightK W{net.w[l], a.N, a.K, on16(net.w[l])};
    const EpiAct ep = l < 3 ? EpiAct{t.act[l], net.b[l], a.rows, a.N, 1 << 30, 0}
                            : EpiAct{t.feat, net.b[l], a.rows, a.N, 64, kFeatIn};
    // 128 rows where that leaves two CTAs per SM, else 64
    if ((a.rows / 128) * (a.N / 64) >= 304) F32_TRY((gemm<128, 64>(A, W, ep, a.rows, a.N, a.K, 1, a.K, 0, st)));
    else F32_TRY((gemm<64, 32>(A, W, ep, a.rows, a.N, a.K, 1, a.K, 0, st)));
  }
  k_feat_angles<<<(2 * B + 255) / 256, 256, 0, st>>>(t.feat, cs, B);
  note_launches(1);
  const int Z = splits_for(2 * ((B + 63) / 64), kFeatIn, 32, (long long)B * kHid, t.part_floats), kc = chunk_of(kFeatIn, Z);
  F32_TRY((gemm<64, 64>(PlainK{t.feat, kFeatIn, B, kFeatIn}, PlainK{net.w1, kFeatIn, kHid, kFeatIn},
                        EpiPart{t.part, (long long)B * kHid, B, kHid}, B, kHid, kFeatIn, Z, kc, 0, st)));
  return cnn_sum_splits(t.part, Z, (long long)B * kHid, net.b1, kHid, h, st);
}

cudaError_t cnn_f32_backward(const CnnNet& net, int B, const CnnF32& t, const CnnTc& tc, const float* dh, const CnnGrad& g,
                             cudaStream_t st) {
  // dense layer: dW1[n][f] = sum_b dh[b][n] feat[b][f]; dY of the last convolution
  F32_TRY((gemm<64, 64>(PlainR{dh, kHid, kHid, B}, PlainR{t.feat, kFeatIn, kFeatIn, B}, EpiPart{g.w1, 0, kHid, kFeatIn}, kHid,
                        kFeatIn, B, 1, B, 0, st)));
  float* dy = t.dy[1];
  F32_TRY((gemm<64, 64>(PlainK{dh, kHid, B, kHid}, PlainR{net.w1, kFeatIn, kFeat, kHid}, EpiDfeat{dy, t.feat, B}, B, kFeat, kHid,
                        1, kHid, 0, st)));
  for (int l = 3; l >= 1; --l) {
    const Layer a = layer(l, B);
    F32_TRY(cnn_colsum(dy, a.rows, a.N, tc, g.b[l], st));
    const ConvR X{ConvGeom{t.act[l - 1], a.H, a.lwo, a.lc, a.rows, a.K}};
    const int tiles = (a.N / 64) * ((a.K + 63) / 64);
    const int Z = splits_for(tiles, a.rows, 256, (long long)a.N * a.K, t.part_floats);
    F32_TRY((gemm<64, 64>(DyR{dy, a.N, a.rows}, X, EpiPart{t.part, (long long)a.N * a.K, a.N, a.K}, a.N, a.K, a.rows, Z,
                          chunk_of(a.rows, Z), 0, st)));
    F32_TRY(cnn_sum_splits(t.part, Z, (long long)a.N * a.K, nullptr, 1, g.w[l], st));
    float* dx = t.dy[(l - 1) & 1];
    const ParityK A{dy, a.lwo, a.ln, a.rows};
    const ClassWR W{net.w[l], a.ln, a.C, on16(net.w[l])};
    const EpiDx ep{dx, t.act[l - 1], a.lwo, a.rows, a.C};
    if (a.C == 32) F32_TRY((gemm<128, 32>(A, W, ep, a.rows, a.C, 0, 4, 0, a.N, st)));
    else if ((a.rows / 128) * (a.C / 64) * 4 >= 304) F32_TRY((gemm<128, 64>(A, W, ep, a.rows, a.C, 0, 4, 0, a.N, st)));
    else F32_TRY((gemm<64, 32>(A, W, ep, a.rows, a.C, 0, 4, 0, a.N, st)));
    dy = dx;
  }
  F32_TRY(cnn_colsum(dy, B * 4096, 32, tc, g.b[0], st));
  return cnn_conv0_dw_f32(dy, t.img, B, tc, g.w[0], st);
}

}  // namespace digs
