// The weight-predictor CNN on the tensor cores: forward (training and inference) and parameter gradient
// with BF16 operands and FP32 accumulation in tensor memory (tcgen05, sm_103a).
//
// Activations live in BF16, NHWC, exactly as the GEMMs consume them: the post-ReLU output of every
// convolution is rounded once by the epilogue that produces it (the rounding the tensor cores would
// apply anyway), its sign is the ReLU mask of the backward.  Convolutions 1 to 3 are in cnn_conv.cu; the first one
// has a single input channel (K = 9) and runs on the SIMT pipes with the same rounded operands.  The dense layer's
// three GEMMs are launches of one kernel template: 128 threads per CTA, looping over 128-row tiles of C; the four
// warps fill a ring of 2-4 stages of 64-deep K slices of A and B with 16-byte cp.async copies (zero-filled where an
// operand is padding), one thread issues the four 128 x 128 x 16 MMAs of a slice and commits them to the slice's
// mbarrier, and the accumulator goes through a per-role epilogue: feat W1^T (split K), the weight gradient
// (transposed stores) and the data gradient (the last convolution's ReLU mask, its BF16 rounding and per-CTA column
// sums for its bias gradient), the latter two with MN-major operands.
// Every mbarrier wait is bounded; a K-loop wait that gives up sets *status, and the CTA drains its own MMAs (default
// bound) and stores NaN for the tiles it owes before it frees its tensor memory.  Sums launched after that are NaN too
// (k_sum_z, k_colreduce_once), so that nothing computed from a result that is missing looks like one.
#include <cuda_bf16.h>

#include <algorithm>

#include "digs_internal.h"
#include "tcgen05.cuh"

namespace digs {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int kThr = 128;
constexpr int kBM = 128, kBN = 128, kBK = 64;

// ---- geometry of the network (cnn.cu holds the parameter layout) --------------------------------
constexpr int kCh[5] = {1, 32, 64, 128, 128};
constexpr int kEdge[5] = {128, 64, 32, 16, 8};
constexpr int kFeat = 8192, kFeatPitch = 8200, kHid = 128;

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ void unpack8(const uint4& u, float f[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

// 16-byte asynchronous copy global -> shared; src == nullptr fills the 16 bytes with zeros (no bytes read).
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, const void* valid_any) {
  const int n = src ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src ? src : valid_any), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// ---- operand loaders -------------------------------------------------------------------------------
// K-major loaders return the address of the 8 reduction elements [k, k + 8) of operand row `row`;
// MN-major loaders the address of the 8 row elements [mn, mn + 8) at reduction index k; nullptr where
// the operand is zero.

struct PlainK {  // X[row][k] = p[row * ld + k]
  const bf16* p;
  int ld, rows;
  __device__ const bf16* kchunk(int row, int k) const { return row < rows ? p + (size_t)row * ld + k : nullptr; }
};

struct PlainMN {  // X[mn][k] = p[k * ld + mn]
  const bf16* p;
  int ld, cols;
  __device__ const bf16* mnchunk(int mn, int k) const { return mn < cols ? p + (size_t)k * ld + mn : nullptr; }
};

// ---- epilogues ---------------------------------------------------------------------------------------
// apply(row, col0, v[16], scratch): the accumulator's row `row`, columns [col0, col0 + 16) of the CTA's tile
// (global indices); finish(scratch, ...) runs once per thread after all columns (all threads call it).

// FP32 rows of split z: part[z * zstride + row * ld + col].
struct EpiF32 {
  float* part;
  long long zstride;
  int rows, ld;
  __device__ void apply(int row, int col0, float v[16], float*) const {
    if (row >= rows) return;
    float4* d = reinterpret_cast<float4*>(part + blockIdx.z * zstride + (size_t)row * ld + col0);
#pragma unroll
    for (int q = 0; q < 4; ++q) d[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  }
  __device__ void finish(float*, int, int, int) const {}
};

// Transposed FP32 store of split z: out[z * zstride + col * ld + row] for row < rows (coalesced: the
// lanes of a warp hold consecutive rows).
struct EpiF32T {
  float* out;
  long long zstride;
  int rows, ld;
  __device__ void apply(int row, int col0, float v[16], float*) const {
    if (row >= rows) return;
    float* d = out + blockIdx.z * zstride + (size_t)col0 * ld + row;
#pragma unroll
    for (int j = 0; j < 16; ++j) d[(size_t)j * ld] = v[j];
  }
  __device__ void finish(float*, int, int, int) const {}
};

// Sum 16 per-lane values over the warp's 32 lanes by recursive halving (16 shuffles); lane l ends with
// the total of value 8 b4 + 4 b3 + 2 b2 + b1 (b_i = bit i of l).
__device__ __forceinline__ float warp_sum16(float v[16], int lane) {
#pragma unroll
  for (int half = 8, bit = 16; half >= 1; half >>= 1, bit >>= 1) {
    const bool hi = (lane & bit) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = hi ? v[i] : v[i + half], keep = hi ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}
__device__ __forceinline__ int sum16_col(int lane) {
  return 8 * ((lane >> 4) & 1) + 4 * ((lane >> 3) & 1) + 2 * ((lane >> 2) & 1) + ((lane >> 1) & 1);
}

// Gradient of the dense layer's input, rows b (batch entry) and columns f (feature, blockIdx.y selects
// 128 of them, i.e. one pixel's 128 channels of the last convolution):
// dY3[b][f] = dfeat[b][f] [act3[b][f] > 0] in BF16 (feat holds act3 in its first 8192 columns; the two
// angle inputs get no gradient), and the masked FP32 values summed per column over the CTA's rows into
// colpart[blockIdx.y * n_mt + mt][c] (the last convolution's bias gradient sums those rows).
struct EpiDfeat {
  bf16* dy3;
  const bf16* feat;  // [B][kFeatPitch]
  float* colpart;
  int nb;
  __device__ void apply(int row, int col0, float v[16], float* scratch) const {
    if (row < nb) {
      const uint4* a = reinterpret_cast<const uint4*>(feat + (size_t)row * kFeatPitch + col0);
      float m[16];
      unpack8(a[0], m);
      unpack8(a[1], m + 8);
      uint32_t w[8];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = m[j] > 0.f ? v[j] : 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) w[j] = pack2(v[2 * j], v[2 * j + 1]);
      uint4* d = reinterpret_cast<uint4*>(dy3 + (size_t)row * kFeat + col0);
      d[0] = make_uint4(w[0], w[1], w[2], w[3]);
      d[1] = make_uint4(w[4], w[5], w[6], w[7]);
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = 0.f;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float s = warp_sum16(v, lane);
    if ((lane & 1) == 0) scratch[warp * 128 + col0 - blockIdx.y * 128 + sum16_col(lane)] = s;
  }
  __device__ void finish(float* scratch, int tid, int mt, int n_mt) const {
    __syncthreads();
    if (tid < 128) {
      const float s = scratch[tid] + scratch[128 + tid] + scratch[256 + tid] + scratch[384 + tid];
      colpart[((size_t)blockIdx.y * n_mt + mt) * 128 + tid] = s;
    }
  }
};

// ---- the GEMM kernel -------------------------------------------------------------------------------
// S stages of (A, B) slices: 4 for long reductions, fewer where a CTA has only a few slices, so that more CTAs share
// an SM (three with two stages: 384 of the 512 tensor-memory columns).
template <int S>
struct Cfg {
  static constexpr int kA = kBM * kBK * 2;  // bytes of one A slice (16 KB)
  static constexpr int kB = kBN * kBK * 2;
  static constexpr int kStage = kA + kB;
  static constexpr int kScratch = 4 * kBN * 4;  // epilogue column sums [warp][kBN]
  static constexpr size_t kSmem = 1024 + (size_t)S * kStage + 128 + kScratch;
};

// Shared-memory byte offset of a 16-byte chunk: K-major (row, kc) of a ROWS x 64 slice; MN-major
// (mn chunk mc, k) of an MN x 64 slice.
__device__ __forceinline__ uint32_t off_k(int row, int kc) { return (uint32_t)(((row >> 3) * 8 + kc) * 128 + (row & 7) * 16); }
template <int MN>
__device__ __forceinline__ uint32_t off_mn(int mc, int k) {
  return (uint32_t)(((k >> 3) * (MN / 8) + mc) * 128 + (k & 7) * 16);
}

// Fills one operand slice: ROWS (MN extent) x 64 reduction elements starting at (r0, k0); the thread's
// chunks are q = tid + 128 i, laid out so that a warp's copies fill whole 128-byte core-matrix rows.
template <int ROWS, bool MN, class L>
__device__ __forceinline__ void fill(const L& ld, uint32_t sdst, int r0, int k0, int kend, const void* any) {
#pragma unroll
  for (int i = 0; i < ROWS / 16; ++i) {
    const int q = threadIdx.x + kThr * i;
    if constexpr (!MN) {
      const int row = (q & 7) | ((q >> 6) << 3), kc = (q >> 3) & 7;
      const int k = k0 + kc * 8;
      cp16(sdst + off_k(row, kc), k < kend ? ld.kchunk(r0 + row, k) : nullptr, any);
    } else {
      constexpr int G = ROWS / 8;
      const int rest = q >> 3, mc = rest & (G - 1), k = ((rest / G) << 3) | (q & 7);
      cp16(sdst + off_mn<ROWS>(mc, k), k0 + k < kend ? ld.mnchunk(r0 + mc * 8, k0 + k) : nullptr, any);
    }
  }
}

template <int ROWS, bool MN>
__device__ __forceinline__ uint64_t slice_desc(uint32_t a, int j) {
  if constexpr (!MN) return tc::smem_desc(a + j * 256, 128, 1024);
  return tc::smem_desc(a + j * 2 * (ROWS / 8) * 128, (ROWS / 8) * 128, 128);
}

// C tiles (128 x 128) of rows [mt 128, mt 128 + 128) for mt = blockIdx.x, blockIdx.x + gridDim.x, ...
// (n_mt row tiles in all), columns from blockIdx.y 128; blockIdx.z = split of the reduction (kchunk each).  The
// tensor memory and the mbarrier ring stay with the CTA across its tiles; g counts the slices issued so far, which
// selects the stage buffer (g mod S) and the mbarrier phase (g div S).
template <int kStages, bool AMN, bool BMN, class LA, class LB, class EP>
__global__ void __launch_bounds__(kThr, 1) k_cnn_gemm(const LA la, const LB lb, const EP ep, int n_mt, int K, int kchunk,
                                                      unsigned* status, unsigned wait_limit, const void* any) {
  using C = Cfg<kStages>;
  extern __shared__ unsigned char smem_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bar = (uint64_t*)(sm + kStages * C::kStage);
  uint32_t* tslot = (uint32_t*)(bar + kStages);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = blockIdx.y * kBN;
  const int kb = (int)min((long long)K, (long long)blockIdx.z * kchunk);
  const int ke = (int)min((long long)K, (long long)kb + kchunk);
  const int nk = ke > kb ? (ke - kb + kBK - 1) / kBK : 0;
  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < kStages; ++s) tc::mbar_init(bar + s, 1);
    tc::mbar_init_fence();
  }
  if (warp == 0) tc::tmem_alloc(tslot, kBN);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *tslot;
  const uint32_t sbase = tc::smem_u32(sm);
  constexpr uint32_t idesc = tc::idesc_bf16(kBM, kBN, AMN, BMN);
  float* scratch = reinterpret_cast<float*>((uint8_t*)bar + 128);  // the epilogue's column sums
  int ok = 1;
  unsigned g = 0;
  // the first S - 1 slices of a tile, into the stage buffers g, g + 1, ... (all free: no MMA in flight)
  auto prologue = [&](int m0) {
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
      if (s < nk) {
        const uint32_t sa = sbase + ((g + s) % kStages) * C::kStage;
        fill<kBM, AMN>(la, sa, m0, kb + s * kBK, ke, any);
        fill<kBN, BMN>(lb, sa + C::kA, n0, kb + s * kBK, ke, any);
      }
      cp_commit();
    }
  };
  int mt = blockIdx.x;
  if (mt < n_mt) prologue(mt * kBM);
  while (mt < n_mt) {
    const int m0 = mt * kBM;
    int issued = 0;
    for (int c = 0; c < nk; ++c) {
      cp_wait<kStages - 2>();     // this thread's copies of slice c have landed
      tc::fence_async_smem();     // ... and are visible to the tensor core
      ok = __syncthreads_and(ok);
      if (!ok) break;
      const unsigned gc = g + c;
      if (tid == 0) {
        tc::fence_after();
        const uint32_t sa = sbase + (gc % kStages) * C::kStage, sb = sa + C::kA;
#pragma unroll
        for (int j = 0; j < kBK / 16; ++j)
          tc::mma_bf16(tmem, slice_desc<kBM, AMN>(sa, j), slice_desc<kBN, BMN>(sb, j), idesc, (c > 0 || j > 0) ? 1u : 0u);
        tc::mma_commit(bar + gc % kStages);
      }
      issued = c + 1;
      const int nxt = c + kStages - 1;  // refills the buffer of slice c - 1 once its MMAs are done
      if (nxt < nk) {
        if (c >= 1) ok = ok && tc::mbar_wait(bar + (gc - 1) % kStages, ((gc - 1) / kStages) & 1u, wait_limit);
        if (ok) {
          const uint32_t sa = sbase + ((g + nxt) % kStages) * C::kStage;
          fill<kBM, AMN>(la, sa, m0, kb + nxt * kBK, ke, any);
          fill<kBN, BMN>(lb, sa + C::kA, n0, kb + nxt * kBK, ke, any);
        }
      }
      cp_commit();
    }
    cp_wait<0>();
    const unsigned gl = g + issued - 1;  // the last slice: its commit tracks all the tile's MMAs
    const bool drained = issued == 0 || tc::mbar_wait(bar + gl % kStages, (gl / kStages) & 1u, tc::kWaitLimit);
    ok = __syncthreads_and(ok && drained);
    tc::fence_after();
    g += issued;
    if (!ok) break;
    // the next tile's first copies go out now, so that they land while this tile's epilogue runs
    const int next = mt + gridDim.x;
    if (next < n_mt) prologue(next * kBM);
    const int row = m0 + warp * 32 + lane;
#pragma unroll 1
    for (int c0 = 0; c0 < kBN; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
      if (issued == 0) {
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = 0.f;
      }
      ep.apply(row, n0 + c0, v, scratch);
    }
    ep.finish(scratch, tid, mt, n_mt);
    // the accumulator and the scratch are free again before the next tile's MMAs
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    mt = next;
  }
  cp_wait<0>();
  if (!ok) {  // the same for the whole CTA
    for (; mt < n_mt; mt += gridDim.x)
#pragma unroll 1
      for (int c0 = 0; c0 < kBN; c0 += 16) {
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = __int_as_float(0x7fffffff);
        ep.apply(mt * kBM + warp * 32 + lane, n0 + c0, v, scratch);
      }
    if (tid == 0) atomicExch(status, 1u);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after();
    tc::tmem_dealloc(tmem, kBN);
  }
}

// ---- SIMT kernels and small steps --------------------------------------------------------------------

// ---- first convolution (1 -> 32 channels, 128^2 -> 64^2) ---------------------------------------------
// Both directions work on bands of kBandRows output rows of one image, whose input rows lie in shared memory as
// FP32 (columns -1 to 127; zeros outside the image).  Four lanes share an output pixel, 8 channels each: their
// weights (or their sums of the weight gradient) stay in 72 registers, a pixel's 9 inputs are broadcast reads, and
// a warp's 16-byte accesses of act0 and dY0 cover eight whole pixels in a row.
// What bounds them: 288 FMAs a pixel, then HBM.  With a thread per pixel the forward read a weight from shared
// memory for every FMA and stored 16 bytes per lane 64 bytes apart, and the gradient loaded nine inputs from global
// memory for 36 FMAs.  Batch 256: forward 33.6 -> 22.2 us, weight gradient 52.5 -> 23.3 us.
constexpr int kBandRows = 8, kBands = 64 / kBandRows, kBandIn = 2 * kBandRows + 1, kBandPitch = 132;

__device__ __forceinline__ void load4(const bf16* p, float d[4]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  d[0] = __uint_as_float(u.x << 16);
  d[1] = __uint_as_float(u.x & 0xFFFF0000u);
  d[2] = __uint_as_float(u.y << 16);
  d[3] = __uint_as_float(u.y & 0xFFFF0000u);
}
__device__ __forceinline__ void load4(const float* p, float d[4]) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  d[0] = u.x; d[1] = u.y; d[2] = u.z; d[3] = u.w;
}
__device__ __forceinline__ float to_float(bf16 x) { return __bfloat162float(x); }
__device__ __forceinline__ float to_float(float x) { return x; }

// A band's share of a thread (of 256): input rows 2 y0 - 1 ... 2 y0 + 15 of image b, 4 columns at a time.
struct BandPart {
  float v[3][4];
};
template <typename T>
__device__ __forceinline__ void fetch_band(const T* __restrict__ img, bool wide, int b, int y0, BandPart& o) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = threadIdx.x + 256 * k, iy = 2 * y0 - 1 + (i >> 5);
#pragma unroll
    for (int e = 0; e < 4; ++e) o.v[k][e] = 0.f;
    if (i >= kBandIn * 32 || iy < 0) continue;
    const T* p = img + ((size_t)b * 128 + iy) * 128 + (i & 31) * 4;
    if (wide) {
      load4(p, o.v[k]);
    } else {  // the caller's images need only be aligned to their elements
#pragma unroll
      for (int e = 0; e < 4; ++e) o.v[k][e] = to_float(p[e]);
    }
  }
}
// ... into s[row][4 + column] (s[row][3] = column -1 = 0); with ROUND rounded to BF16, and rows 2 y0 ... also stored
// to imgb (every row by one band).
template <bool ROUND>
__device__ __forceinline__ void put_band(BandPart& o, int b, int y0, float (*s)[kBandPitch], bf16* imgb) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = threadIdx.x + 256 * k, r = i >> 5, c = (i & 31) * 4;
    if (i >= kBandIn * 32) continue;
    float* v = o.v[k];
    if (ROUND) {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = bf16r(v[e]);
      if (r > 0)
        *reinterpret_cast<uint2*>(imgb + ((size_t)b * 128 + 2 * y0 - 1 + r) * 128 + c) =
            make_uint2(pack2(v[0], v[1]), pack2(v[2], v[3]));
    }
    *reinterpret_cast<float4*>(&s[r][4 + c]) = make_float4(v[0], v[1], v[2], v[3]);
  }
  if (threadIdx.x < kBandIn) s[threadIdx.x][3] = 0.f;
}
// The 9 inputs of output pixel (row r of the band, x).
__device__ __forceinline__ void taps9(const float (*s)[kBandPitch], int r, int x, float v[9]) {
#pragma unroll
  for (int ky = 0; ky < 3; ++ky) {
    v[3 * ky] = s[2 * r + ky][3 + 2 * x];
    const float2 u = *reinterpret_cast<const float2*>(&s[2 * r + ky][4 + 2 * x]);
    v[3 * ky + 1] = u.x;
    v[3 * ky + 2] = u.y;
  }
}

// act0[p][co] = relu(b[co] + sum over taps of r(w[co][tap]) r(img(tap))), r = BF16 rounding, stored in BF16 with the
// rounded input (imgb) for the backward.  Blocks stride over the n_bands bands, the next one's inputs on the way
// during the sums of the last.
__global__ void __launch_bounds__(256, 2) k_conv0_fwd(const float* __restrict__ img, const float* __restrict__ w,
                                                      const float* __restrict__ bias, int n_bands, bf16* __restrict__ out,
                                                      bf16* __restrict__ imgb) {
  __shared__ __align__(16) float s[2][kBandIn][kBandPitch];
  const int q = threadIdx.x & 3, x = threadIdx.x >> 2;
  const bool wide = ((uintptr_t)img & 15) == 0;
  int band = blockIdx.x;
  BandPart part;
  fetch_band(img, wide, band / kBands, band % kBands * kBandRows, part);
  float wr[8][9], br[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    br[j] = bias[q * 8 + j];
#pragma unroll
    for (int t = 0; t < 9; ++t) wr[j][t] = bf16r(w[(q * 8 + j) * 9 + t]);
  }
  for (int buf = 0; band < n_bands; buf ^= 1) {
    const int b = band / kBands, y0 = band % kBands * kBandRows;
    put_band<true>(part, b, y0, s[buf], imgb);
    __syncthreads();  // one a band: a buffer's readers have passed the next band's barrier before it is refilled
    band += gridDim.x;
    if (band < n_bands) fetch_band(img, wide, band / kBands, band % kBands * kBandRows, part);
#pragma unroll 1
    for (int r = 0; r < kBandRows; ++r) {
      float v[9], o[8];
      taps9(s[buf], r, x, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float a = br[j];
#pragma unroll
        for (int t = 0; t < 9; ++t) a = fmaf(wr[j][t], v[t], a);
        o[j] = fmaxf(a, 0.f);
      }
      *reinterpret_cast<uint4*>(out + (((size_t)b * 64 + y0 + r) * 64 + x) * 32 + q * 8) =
          make_uint4(pack2(o[0], o[1]), pack2(o[2], o[3]), pack2(o[4], o[5]), pack2(o[6], o[7]));
    }
  }
}

// Weight gradient: part[block][co * 9 + tap] = sum over the block's bands of dY0[p][co] img(tap), both of type T
// (BF16, or FP32 for the FP32 mode), blocks striding over the n_bands bands.  A thread's column of pixels adds up in
// its registers; the 64 columns are added at the end in a fixed order.
template <typename T>
__global__ void __launch_bounds__(256, 2) k_conv0_dw(const T* __restrict__ dy, const T* __restrict__ img, int n_bands,
                                                     float* __restrict__ part) {
  __shared__ __align__(16) float s[kBandIn][kBandPitch];
  const int q = threadIdx.x & 3, x = threadIdx.x >> 2, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float acc[8][9];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[j][t] = 0.f;
  constexpr int A = sizeof(T) == 2 ? 4 : 2, W = sizeof(T) / 2;  // rows of dY0 fetched ahead, 16-byte words of 8 channels
  for (int band = blockIdx.x; band < n_bands; band += gridDim.x) {
    const int b = band / kBands, y0 = band % kBands * kBandRows;
    const T* d0 = dy + (((size_t)b * 64 + y0) * 64 + x) * 32 + q * 8;
    uint4 cur[A][W], next[A][W];
    auto fetch = [&](uint4 (*u)[W], int r) {
#pragma unroll
      for (int k = 0; k < A; ++k)
#pragma unroll
        for (int e = 0; e < W; ++e) u[k][e] = __ldg(reinterpret_cast<const uint4*>(d0 + (size_t)(r + k) * 64 * 32) + e);
    };
    fetch(cur, 0);
    BandPart p;
    fetch_band(img, true, b, y0, p);
    __syncthreads();
    put_band<false>(p, b, y0, s, nullptr);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kBandRows; r += A) {
      if (r + A < kBandRows) fetch(next, r + A);
#pragma unroll
      for (int k = 0; k < A; ++k) {
        float d[8], v[9];
        if constexpr (W == 1) {
          unpack8(cur[k][0], d);
        } else {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            d[4 * e] = __uint_as_float(cur[k][e].x);
            d[4 * e + 1] = __uint_as_float(cur[k][e].y);
            d[4 * e + 2] = __uint_as_float(cur[k][e].z);
            d[4 * e + 3] = __uint_as_float(cur[k][e].w);
          }
        }
        taps9(s, r + k, x, v);
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int t = 0; t < 9; ++t) acc[j][t] = fmaf(d[j], v[t], acc[j][t]);
      }
#pragma unroll
      for (int k = 0; k < A; ++k)
#pragma unroll
        for (int e = 0; e < W; ++e) cur[k][e] = next[k][e];
    }
  }
  __syncthreads();
  float* red = &s[0][0];  // [warp][288] of four warps at a time (8 x 288 do not fit)
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      float a = acc[j][t];
      a += __shfl_xor_sync(0xffffffffu, a, 4);
      a += __shfl_xor_sync(0xffffffffu, a, 8);
      a += __shfl_xor_sync(0xffffffffu, a, 16);
      acc[j][t] = a;
    }
  float sum[2] = {0.f, 0.f};
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    if ((warp >> 2) == h && lane < 4) {
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int t = 0; t < 9; ++t) red[(warp & 3) * 288 + (q * 8 + j) * 9 + t] = acc[j][t];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int o = threadIdx.x + 256 * k;
      if (o < 288) sum[k] += (red[o] + red[288 + o]) + (red[576 + o] + red[864 + o]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < 2; ++k)
    if (threadIdx.x + 256 * k < 288) part[(size_t)blockIdx.x * 288 + threadIdx.x + 256 * k] = sum[k];
}

// out[c] = sum over the rows r < R of in[r * ld + c], in one launch: block (x, y) sums rows
// [y chunk, (y + 1) chunk) of the columns 32 x .. 32 x + 31 (strided over its 8 warps, then the warp sums
// in order) into part[y * cols + c]; the last block of column group x to finish (a ticket counter per
// group, reset by that block) then adds the gridDim.y partials in chunk order.  The result does not depend
// on which block finishes last, and no block waits for another.
__global__ void __launch_bounds__(256) k_colreduce_once(const float* __restrict__ in, int R, int cols, int ld,
                                                        int chunk, float* part, float* __restrict__ out,
                                                        unsigned* tickets, const unsigned* status) {
  __shared__ float red[8][32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  const int r0 = blockIdx.y * chunk, r1 = min(R, r0 + chunk);
  float s = 0.f;
  if (c < cols)
    for (int r = r0 + warp; r < r1; r += 8) s += in[(size_t)r * ld + c];
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && c < cols) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) t += red[k][lane];
    part[(size_t)blockIdx.y * cols + c] = t;
  }
  __threadfence();  // this block's partials are visible before its ticket is taken
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&tickets[blockIdx.x], 1u) == gridDim.y - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  s = 0.f;
  if (c < cols)
    for (int y = warp; y < (int)gridDim.y; y += 8) s += __ldcg(&part[(size_t)y * cols + c]);
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && c < cols) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) t += red[k][lane];
    if (status && *status) t = __int_as_float(0x7fffffff);
    out[c] = t;
  }
  if (threadIdx.x == 0) tickets[blockIdx.x] = 0u;
}

// out[i] = sum over z of part[z * n + i] (+ bias[i % nb] and ReLU when bias != nullptr), in a fixed order:
// 32 outputs per block, warp w adding the splits z = w, w + 8, ... in order (coalesced over the outputs),
// then the eight warp sums added in warp order.  NaN where a kernel of this pass gave up waiting (*status).
__global__ void __launch_bounds__(256) k_sum_z(const float* __restrict__ part, int Z, long long n,
                                               const float* __restrict__ bias, int nb, float* __restrict__ out,
                                               const unsigned* status) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long i = (long long)blockIdx.x * 32 + lane;
  float s = 0.f;
  if (i < n)
    for (int z = warp; z < Z; z += 8) s += part[(size_t)z * n + i];
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && i < n) {
    float t = red[0][lane];
#pragma unroll
    for (int w = 1; w < 8; ++w) t += red[w][lane];
    if (bias) t = fmaxf(t + bias[i % nb], 0.f);
    if (status && *status) t = __int_as_float(0x7fffffff);
    out[i] = t;
  }
}

// All of a forward's weight conversions to BF16 in one launch: job k covers the elements [start[k], start[k + 1])
// of a grid-stride loop.  Kind 0, rows: out[r][c] = BF16 of in[r][c] for c < b, 0 for b <= c < c_pitch
// (a rows, row pitch c).  Kind 1, the transposed weights of a convolution with N = a output and C = b input
// channels for its data gradient (Dx in cnn_conv.cu): rows of 64 output channels, in blocks of CC = min(C, 64) input
// channels, for each CC of the C the blocks of the four shifts (dy, dx) (for each 64 of the N): 4, 2, 2 and 1
// parity classes, the class (py, px) of a shift taking the tap ky = py ? 2 - 2 dy : 1, kx = px ? 2 - 2 dx : 1.
// *status is set to zero for the kernels that follow.
struct BfJob {
  const float* in;
  bf16* out;
  int kind, a, b, c;
};
struct BfJobs {
  BfJob job[8];
  long long start[9];
  int count;
};
__global__ void __launch_bounds__(256) k_to_bf16_jobs(const __grid_constant__ BfJobs J, unsigned* status) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *status = 0u;
  const long long total = J.start[J.count];
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    int k = 0;
    while (k + 1 < J.count && i >= J.start[k + 1]) ++k;
    const BfJob& jb = J.job[k];
    const long long e = i - J.start[k];
    float x;
    if (jb.kind == 0) {
      const int r = (int)(e / jb.c), c = (int)(e - (long long)r * jb.c);
      x = c < jb.b ? jb.in[(size_t)r * jb.b + c] : 0.f;
    } else {
      const int CC = min(jb.b, 64), H = jb.a / 64, row = (int)(e >> 6), chunk = row / (9 * H * CC);
      const int blk = row / CC - chunk * 9 * H, ci = chunk * CC + row % CC;
      const int shift = blk < 4 * H ? 0 : blk / (2 * H) - 1;  // blocks [0, 4H), [4H, 6H), [6H, 8H), [8H, 9H)
      const int nb = shift == 0 ? 4 : (shift == 3 ? 1 : 2), k2 = blk - (shift == 0 ? 0 : 2 + 2 * shift) * H;
      const int half = k2 / nb, pos = k2 % nb + (shift >= 2);
      const int cls = pos == 0 ? 1 : (pos == 1 ? 3 : (pos == 2 ? 2 : 0));
      const int ky = (cls >> 1) ? 2 - 2 * (shift >> 1) : 1, kx = (cls & 1) ? 2 - 2 * (shift & 1) : 1;
      x = jb.in[((size_t)(half * 64 + (int)(e & 63)) * 9 + ky * 3 + kx) * jb.b + ci];
    }
    jb.out[e] = __float2bfloat16_rn(x);
  }
}

// The dense layer's two angle inputs and zero padding: feat[b][8192 + j] = BF16 of (cos, sin, 0, ...).
__global__ void k_feat_tail(bf16* __restrict__ feat, const float* __restrict__ cs, int B) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * (kFeatPitch - kFeat)) return;
  const int b = i / (kFeatPitch - kFeat), j = i - b * (kFeatPitch - kFeat);
  feat[(size_t)b * kFeatPitch + kFeat + j] = __float2bfloat16_rn(j < 2 ? cs[2 * b + j] : 0.f);
}

unsigned grid_of(long long n) { return (unsigned)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152LL * 16)); }

// One GEMM launch: M rows of C in 128-row tiles, gy column tiles, gz splits.
template <int S, bool AMN, bool BMN, class LA, class LB, class EP>
cudaError_t gemm(const LA& la, const LB& lb, const EP& ep, int M, int K, int gy, int gz, int kchunk, const void* any,
                 unsigned* status, cudaStream_t st) {
  using C = Cfg<S>;
  auto kern = k_cnn_gemm<S, AMN, BMN, LA, LB, EP>;
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmem);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  if (M <= 0) return cudaSuccess;
  // row tiles per CTA: enough CTAs for every SM to hold as many as its shared memory allows, several
  // tiles each when there are more
  const int n_mt = (M + kBM - 1) / kBM;
  const long long per_sm = std::max(1, std::min(512 / kBN, (int)(227 * 1024 / C::kSmem)));
  const long long total = (long long)n_mt * gy * gz, target = 4LL * 152 * per_sm;
  const int per_cta = (int)std::max(1LL, (total + target - 1) / target);
  const int gx = (n_mt + per_cta - 1) / per_cta;
  kern<<<dim3(gx, gy, gz), kThr, C::kSmem, st>>>(la, lb, ep, n_mt, K, kchunk, status, loop_wait_limit(), any);
  note_launches(1);
  return cudaGetLastError();
}

#define TC_TRY(...)                       \
  do {                                    \
    cudaError_t e__ = (__VA_ARGS__);      \
    if (e__ != cudaSuccess) return e__;   \
  } while (0)

constexpr int kConv0Ctas = 2 * 152;  // two CTAs per SM (the registers of k_conv0_fwd and _dw)
constexpr int kColTickets = 64;      // colreduce ticket counters (column groups of 32)

int chunk_of(long long n, int z) { return (int)(((n + z - 1) / z + kBK - 1) / kBK * kBK); }

// out[c] = sum over r < R of in[r * ld + c] in a fixed order: row chunks of 64 summed into scratch by
// many blocks, then the chunk sums by one block per 32 columns (one pass when R <= 512).
// tickets: (cols + 31) / 32 counters, zero on entry (and left zero).
cudaError_t colreduce(const float* in, int R, int cols, int ld, float* out, float* scratch, unsigned* tickets,
                      const unsigned* status, cudaStream_t st) {
  const unsigned gx = (unsigned)((cols + 31) / 32);
  // at most 512 chunks: the last block adds their sums one after the other
  const int chunk = R <= 2048 ? 64 : std::max(128, (R + 511) / 512), nch = (R + chunk - 1) / chunk;
  k_colreduce_once<<<dim3(gx, nch), 256, 0, st>>>(in, R, cols, ld, chunk, scratch, out, tickets, status);
  note_launches(1);
  return cudaGetLastError();
}

// dW of the first convolution into out (32 x 9): at most kConv0Ctas partial sums in colpart, then added.
template <typename T>
cudaError_t conv0_dw(const T* dy, const T* img, int B, float* colpart, float* scratch, unsigned* tickets, float* out,
                     const unsigned* status, cudaStream_t st) {
  const int ctas = std::min(kConv0Ctas, B * kBands);
  k_conv0_dw<T><<<ctas, 256, 0, st>>>(dy, img, B * kBands, colpart);
  note_launches(1);
  return colreduce(colpart, ctas, 288, 288, out, scratch, tickets, status, st);
}

}  // namespace

// ---- host side -------------------------------------------------------------------------------------

size_t cnn_tc_layout(void* base, int B, CnnTc* t) {
  size_t off = 0;
  char* p = (char*)base;
  auto take = [&](size_t bytes) -> void* {
    void* q = p ? p + off : nullptr;
    off += (bytes + 255) & ~(size_t)255;
    return q;
  };
  CnnTc w{};
  w.imgb = (uint16_t*)take((size_t)B * 128 * 128 * 2);
  for (int l = 0; l < 3; ++l) w.act[l] = (uint16_t*)take((size_t)B * kEdge[l + 1] * kEdge[l + 1] * kCh[l + 1] * 2);
  w.feat = (uint16_t*)take((size_t)B * kFeatPitch * 2);
  w.dy[0] = (uint16_t*)take((size_t)B * 4096 * 32 * 2);  // dY of conv 2, then of conv 0
  w.dy[1] = (uint16_t*)take((size_t)B * 1024 * 64 * 2);  // dY of conv 1
  w.dy3 = (uint16_t*)take((size_t)B * kFeat * 2);
  w.dhb = (uint16_t*)take((size_t)B * kHid * 2);
  for (int l = 1; l < 4; ++l) {
    w.wb[l] = (uint16_t*)take((size_t)kCh[l + 1] * 9 * kCh[l] * 2);
    w.wt[l] = (uint16_t*)take((size_t)kCh[l + 1] * 9 * kCh[l] * 2);
  }
  w.wb[0] = w.wt[0] = nullptr;
  w.w1b = (uint16_t*)take((size_t)kHid * kFeatPitch * 2);
  w.part_floats = std::max<long long>(16LL * B * kHid, 5LL << 20);
  w.part = (float*)take((size_t)w.part_floats * 4);
  w.colpart_floats = std::max<long long>({1024LL * B, 8192LL * ((B + 127) / 128), (long long)kConv0Ctas * 288});
  w.colpart = (float*)take((size_t)w.colpart_floats * 4);
  w.tickets = (unsigned*)take(kColTickets * sizeof(unsigned));
  w.status = (unsigned*)take(sizeof(unsigned));
  if (t) *t = w;
  return off;
}

cudaError_t cnn_tc_forward(const CnnNet& net, const float* img, const float* cs, int B, const CnnTc& t, float* h,
                           cudaStream_t st) {
  // BF16 copies of the weights, row-major (forward) and transposed (data gradient): one
  // launch (the first convolution rounds the input images itself and stores their BF16 copy)
  BfJobs J{};
  long long at = 0;
  auto add = [&](const float* in, bf16* out, int kind, int a, int b, int c, long long n) {
    J.job[J.count] = BfJob{in, out, kind, a, b, c};
    J.start[J.count++] = at;
    at += n;
  };
  for (int l = 1; l < 4; ++l) {
    const int N = kCh[l + 1], Kl = 9 * kCh[l];
    add(net.w[l], (bf16*)t.wb[l], 0, N, Kl, Kl, (long long)N * Kl);
    add(net.w[l], (bf16*)t.wt[l], 1, N, kCh[l], 0, (long long)N * Kl);
  }
  add(net.w1, (bf16*)t.w1b, 0, kHid, kFeat + 2, kFeatPitch, (long long)kHid * kFeatPitch);
  J.start[J.count] = at;
  k_to_bf16_jobs<<<grid_of(at), 256, 0, st>>>(J, t.status);
  k_conv0_fwd<<<std::min(kConv0Ctas, B * kBands), 256, 0, st>>>(img, net.w[0], net.b[0], B * kBands, (bf16*)t.act[0],
                                                                (bf16*)t.imgb);
  note_launches(2);
  const void* any = t.wb[1];
  for (int l = 1; l < 4; ++l) {
    // the last convolution writes the dense layer's feature rows ((y, x, c) order, pitch 8200)
    const long long pitch = l == 3 ? kFeatPitch : (long long)kEdge[l + 1] * kEdge[l + 1] * kCh[l + 1];
    TC_TRY(cnn_conv_forward(l, t.act[l - 1], t.wb[l], net.b[l], B, l == 3 ? t.feat : t.act[l], pitch, t.status, st));
  }
  k_feat_tail<<<(B * (kFeatPitch - kFeat) + 255) / 256, 256, 0, st>>>((bf16*)t.feat, cs, B);
  note_launches(1);
  // dense layer: K = 8200 split 16 ways into FP32 partials, then summed with bias and ReLU
  const int Z = 16, kc = chunk_of(kFeatPitch, Z);
  const EpiF32 ep{t.part, (long long)B * kHid, B, kHid};
  TC_TRY((gemm<4, false, false>(PlainK{(const bf16*)t.feat, kFeatPitch, B}, PlainK{(const bf16*)t.w1b, kFeatPitch, kHid},
                                  ep, B, kFeatPitch, 1, Z, kc, any, t.status, st)));
  k_sum_z<<<(unsigned)(((long long)B * kHid + 31) / 32), 256, 0, st>>>(t.part, Z, (long long)B * kHid, net.b1, kHid, h, t.status);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t cnn_tc_backward(int B, const CnnTc& t, const float* dh, const CnnGrad& g, cudaStream_t st) {
  const void* any = t.wb[1];
  (void)dh;  // its BF16 copy t.dhb, written with it, is what the GEMMs read
  const cudaError_t ez = cudaMemsetAsync(t.tickets, 0, kColTickets * sizeof(unsigned), st);
  if (ez != cudaSuccess) return ez;
  // dense layer: dW1[n][f] = sum_b dh[b][n] feat[b][f] (rows f, both operands MN-major)
  TC_TRY((gemm<3, true, true>(PlainMN{(const bf16*)t.feat, kFeatPitch, kFeatPitch}, PlainMN{(const bf16*)t.dhb, kHid, kHid},
                                EpiF32T{g.w1, 0, kFeat + 2, kFeat + 2}, kFeatPitch, B, 1, 1, B, any, t.status, st)));
  // ... and dfeat[b][f] = sum_n dh[b][n] W1[n][f] (rows b, B MN-major) -> dY of the last convolution
  // (masked, BF16) and its per-channel column sums
  const int nmt = (B + kBM - 1) / kBM;
  TC_TRY((gemm<2, false, true>(PlainK{(const bf16*)t.dhb, kHid, B}, PlainMN{(const bf16*)t.w1b, kFeatPitch, kFeat},
                                    EpiDfeat{(bf16*)t.dy3, (const bf16*)t.feat, t.colpart, B}, B, kHid, kFeat / 128, 1,
                                    kHid, any, t.status, st)));
  TC_TRY(colreduce(t.colpart, (kFeat / 128) * nmt, 128, 128, g.b[3], t.part, t.tickets, t.status, st));
  // convolutions 3, 2, 1: weight gradient (split over pixels), then the data gradient of the layer below
  const uint16_t* dyl = t.dy3;
  for (int l = 3; l >= 1; --l) {
    const long long n = 9LL * kCh[l] * kCh[l + 1];
    const int Z = cnn_conv_dw_splits(l, B, t.part_floats);
    TC_TRY(cnn_conv_dw(l, t.act[l - 1], dyl, B, t.part, Z, t.status, st));
    k_sum_z<<<(unsigned)((n + 31) / 32), 256, 0, st>>>(t.part, Z, n, nullptr, 1, g.w[l], t.status);
    note_launches(1);
    // output dY of convolution l - 1 and its bias partials, a row per CTA
    uint16_t* dyo = l == 2 ? t.dy[1] : t.dy[0];
    TC_TRY(cnn_conv_dx(l, dyl, t.wt[l], t.act[l - 1], B, dyo, t.colpart, t.status, st));
    TC_TRY(colreduce(t.colpart, cnn_conv_dx_rows(l, B), kCh[l], kCh[l], g.b[l - 1], t.part, t.tickets, t.status, st));
    dyl = dyo;
  }
  // the first convolution's weight gradient on the SIMT pipes
  TC_TRY(conv0_dw((const bf16*)dyl, (const bf16*)t.imgb, B, t.colpart, t.part, t.tickets, g.w[0], t.status, st));
  return cudaGetLastError();
}

cudaError_t cnn_colsum(const float* dY, int M, int N, const CnnTc& t, float* out, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(t.tickets, 0, kColTickets * sizeof(unsigned), st);
  return e != cudaSuccess ? e : colreduce(dY, M, N, N, out, t.part, t.tickets, nullptr, st);
}

cudaError_t cnn_conv0_dw_f32(const float* dy, const float* img, int B, const CnnTc& t, float* out, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(t.tickets, 0, kColTickets * sizeof(unsigned), st);
  return e != cudaSuccess ? e : conv0_dw(dy, img, B, t.colpart, t.part, t.tickets, out, nullptr, st);
}

cudaError_t cnn_sum_splits(const float* part, int Z, long long n, const float* bias, int nb, float* out, cudaStream_t st) {
  k_sum_z<<<(unsigned)((n + 31) / 32), 256, 0, st>>>(part, Z, n, bias, nb, out, nullptr);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace digs
