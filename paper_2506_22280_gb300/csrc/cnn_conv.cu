// The weight predictor's 3 x 3, stride-2 convolutions 1 to 3 on the tensor cores (tcgen05, TMA, sm_103a):
// forward, data gradient and weight gradient, BF16 operands, FP32 accumulation in tensor memory.
//
// Every operand tile is a box of the activations as they lie in memory.  An input [B][H][H][C] is seen as
// [B][H/2][2][H/2][2 C]: tap (ky, kx) of the output pixels (b, y, x) then reads row parity ky != 1, column
// half kx != 1 and the pixel (y - (ky == 0), x - (kx == 0)), so that a tile of 128 output pixels is one box with
// unit steps whose out-of-range rows and columns (the padding) TMA fills with zeros.  Boxes are 64 channels
// (128 bytes, 128-byte swizzle) wide and serve as K-major operands (forward, data gradient) and as MN-major
// ones (weight gradient) alike.
//
// Forward: C[pixel][co], K = (tap, 64 channels); 32 input channels take (kx = 1, kx = 2) in one box, since these
// are the two halves of the same pixel pair, and kx = 0 as the upper half of the pair to the left.
// Data gradient: the input pixels (2Y + py, 2X + px) of the four parity classes need dY at (Y + dy, X + dx),
// dy <= py and dx <= px, only: four shifted boxes per tile of 128 pixels (Y, X) serve the nine (class, tap)
// products.  The classes' accumulators lie side by side in the order (0,1), (1,1), (1,0), (0,0), which
// makes the classes of every shift neighbours and each shift a single MMA of 4, 2, 2 or 1 blocks of columns.  The
// shifts run from (1, 1) to (0, 0): a class's taps in ascending order.
// The layer's activations (the ReLU mask) arrive by TMA in the buffers from which the masked gradient leaves.
// Weight gradient: dW[(tap, ci)][co], K = pixels; a CTA holds three 128-row tiles of (tap, ci) and reads dY once
// for them, its share of the pixels one 64-pixel box after another.
//
// What bounds them: the latency of a tile's chain of copies, MMAs and epilogue with one tile after another on an SM; at
// batch 256 HBM runs at 15 to 48 % of its peak, the L2 at 15 to 35 % and the tensor pipe at 13 to 39 %.  (Keeping
// layer 1's weights in shared memory, a third of its fill, changed nothing.)
// The form before this one gathered 16 bytes per thread and cp.async, with the address arithmetic of a tap for
// each, on the threads that also ran the epilogue, and stored 16 bytes per lane at a distance of 128.
// Launch times at batch 256, layers 1 / 2 / 3, before and now: forward 97 / 62 / 39 -> 29 / 18 / 12 us, data
// gradient 167 / 102 / 51 -> 34 / 28 / 18, weight gradient 103 / 67 / 35 -> 29 / 18 / 13; the training step, with the
// first layer's kernels, 978 -> 418 us, inference of 680 projections 745 -> 346 us.  The multiply-adds of every output
// element are added in the same order as before.
// One warp issues the copies, one the MMAs, four run the epilogue on the other half of the tensor memory; CTAs are
// persistent, one per SM (layer 1's forward two, 2.5 % of a training step).  Every wait is bounded: a role that gives
// up sets *status, waits for what it has in flight and leaves; the sums that follow are NaN (k_sum_z, k_colreduce_once).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "digs_internal.h"
#include "tcgen05.cuh"

namespace digs {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int kSms = 152;
constexpr int kThreads = 256;  // warp 0: copies, 1: MMAs, 2: tensor memory, 4-7: epilogue
constexpr int kSlice = 128 * 128;  // bytes of a box of 128 rows x 64 channels
constexpr int kChan[5] = {1, 32, 64, 128, 128};
constexpr int kSide[5] = {128, 64, 32, 16, 8};

// ---- PTX ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void load2(uint32_t dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
               "l"(m), "r"(tc::smem_u32(bar)), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void load4(uint32_t dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
      "l"(m), "r"(tc::smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void load5(uint32_t dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1, int c2, int c3,
                                      int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(
          dst),
      "l"(m), "r"(tc::smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}
__device__ __forceinline__ void store3(const CUtensorMap* m, uint32_t src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(m), "r"(src), "r"(c0),
               "r"(c1), "r"(c2)
               : "memory");
}
__device__ __forceinline__ void store5(const CUtensorMap* m, uint32_t src, int c0, int c1, int c2, int c3, int c4) {
  asm volatile("cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];" ::"l"(m), "r"(src),
               "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
               : "memory");
}
__device__ __forceinline__ void store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// 32 consecutive FP32 columns of this thread's accumulator lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// Matrix descriptor of a 128-byte-swizzled operand (layout type 2 in bits 61-63) whose boxes start on 1024-byte
// boundaries, 8-row groups 1024 bytes apart (SBO).  K-major: LBO unused, a K step of 16 is 32 bytes along the row.
// MN-major: LBO = distance between blocks of 64 M or N elements, a K step of 16 is two groups of 8 rows.
__device__ __forceinline__ uint64_t desc128(uint32_t addr, uint32_t lbo) {
  return tc::smem_desc(addr, lbo, 1024) | (2ull << 61);
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// Byte offset of 16-byte chunk c of row r in a swizzled box.
__device__ __forceinline__ uint32_t box_off(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

// ---- geometry of convolution L ----------------------------------------------------------------------
template <int L>
struct Geo {
  static constexpr int C = kChan[L], N = kChan[L + 1], H = kSide[L], Wo = kSide[L + 1];
  static constexpr int kImgs = Wo * Wo >= 128 ? 1 : 128 / (Wo * Wo);  // images of a tile of 128 pixels
  static constexpr int kRows = 128 / (Wo * kImgs);                    // their pixel rows in it
  static constexpr int kTiles = Wo / kRows;                           // tiles per image (group)
  static __device__ int img(int t) { return t / kTiles * kImgs; }
  static __device__ int row(int t) { return t % kTiles * kRows; }
  static int tiles(int B) { return (B + kImgs - 1) / kImgs * kTiles; }
};

// ---- forward ------------------------------------------------------------------------------------------
template <int L>
struct Fwd {
  using G = Geo<L>;
  static constexpr bool kMask = false;
  static constexpr int kCols = G::N, kSlices = G::C == 32 ? 6 : 9 * G::C / 64, kStages = L == 1 ? 3 : 5, kCtas = L == 1 ? 2 : 1;
  static constexpr int kBBytes = G::N * 128, kIoBoxes = G::N / 64, kIo = 1, kSums = 1;
  static __device__ uint32_t slice_bytes(int) { return kSlice + kBBytes; }
  static __device__ void load(const CUtensorMap* ma, const CUtensorMap* mb, uint64_t* bar, uint32_t sa, uint32_t sb,
                              int s, int t, int) {
    int c0, dx, py, dy, k;
    if constexpr (G::C == 32) {
      const int ky = s >> 1, pair = s & 1;
      c0 = 0; dx = pair - 1; py = ky != 1; dy = ky == 0 ? -1 : 0; k = ky * 96 + pair * 32;
    } else {
      constexpr int Hf = G::C / 64;
      const int tap = s / Hf, half = s % Hf, ky = tap / 3, kx = tap % 3;
      c0 = (kx != 1 ? G::C : 0) + half * 64; dx = kx == 0 ? -1 : 0; py = ky != 1; dy = ky == 0 ? -1 : 0;
      k = tap * G::C + half * 64;
    }
    load5(sa, ma, bar, c0, dx, py, G::row(t) + dy, G::img(t));
    load2(sb, mb, bar, k, 0);
  }
  static __device__ void mma(uint32_t tmem, uint32_t sa, uint32_t sb, int s) {
    constexpr uint32_t idesc = tc::idesc_bf16(128, G::N, false, false);
    const bool upper = G::C == 32 && !(s & 1);  // kx = 0: the box's upper 32 channels, the weights' first 32
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (upper && j >= 2) break;
      tc::mma_bf16(tmem, desc128(sa + (upper ? 64 : 0) + j * 32, 0), desc128(sb + j * 32, 0), idesc, (s > 0 || j > 0) ? 1u : 0u);
    }
  }
  // Bias, ReLU, one rounding to BF16.
  static __device__ void epilogue(uint32_t tmem, uint8_t* io, const float* bias, int r, float*) {
#pragma unroll
    for (int q = 0; q < G::N / 32; ++q) {
      float v[32];
      tmem_ld32(tmem + q * 32, v);
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = fmaxf(v[j] + bias[q * 32 + j], 0.f);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        *reinterpret_cast<uint4*>(io + (q >> 1) * kSlice + box_off(r, (q & 1) * 4 + c)) =
            make_uint4(pack2(v[8 * c], v[8 * c + 1]), pack2(v[8 * c + 2], v[8 * c + 3]), pack2(v[8 * c + 4], v[8 * c + 5]),
                       pack2(v[8 * c + 6], v[8 * c + 7]));
    }
  }
  static __device__ void load_io(const CUtensorMap*, uint64_t*, uint32_t, int, int) {}
  static __device__ void store_io(const CUtensorMap* m, uint32_t io, int t, int) {
#pragma unroll
    for (int q = 0; q < kIoBoxes; ++q) store3(m, io + q * kSlice, q * 64, G::row(t) * G::Wo, G::img(t));
  }
};

// ---- data gradient ------------------------------------------------------------------------------------
// blockIdx.y selects CC of the C input channels.  Weights: rows of 64 output channels, as k_to_bf16_jobs lays them out (kind 1).
template <int L>
struct Dx {
  using G = Geo<L>;
  static constexpr bool kMask = true;
  static constexpr int CC = G::C < 64 ? G::C : 64, Hf = G::N / 64;
  static constexpr int kCols = 4 * CC, kSlices = 4 * Hf, kStages = CC == 32 ? 4 : 3, kCtas = 1;
  static constexpr int kBBytes = 4 * CC * 128, kIoBoxes = 4 * CC / 64, kIo = CC == 32 ? 2 : 1, kSums = CC;
  static __device__ int blocks(int shift) { return shift == 0 ? 4 : (shift == 3 ? 1 : 2); }
  static __device__ int shift_of(int s) { return 3 - s / Hf; }  // 2 dy + dx, (1, 1) first
  static __device__ uint32_t slice_bytes(int s) { return kSlice + blocks(shift_of(s)) * CC * 128; }
  static __device__ void load(const CUtensorMap* ma, const CUtensorMap* mb, uint64_t* bar, uint32_t sa, uint32_t sb,
                              int s, int t, int chunk) {
    const int shift = shift_of(s), half = s % Hf, nb = blocks(shift);
    load4(sa, ma, bar, half * 64, shift & 1, G::row(t) + (shift >> 1), G::img(t));
    const int base = (shift == 0 ? 0 : 2 + 2 * shift) * Hf + half * nb + chunk * 9 * Hf;
    for (int i = 0; i < nb; ++i) load2(sb + i * CC * 128, mb, bar, 0, (base + i) * CC);
  }
  static __device__ void mma(uint32_t tmem, uint32_t sa, uint32_t sb, int s) {
    const int shift = shift_of(s), nb = blocks(shift);
    // [at, at + n) of the slice's column blocks, one K step
    auto step = [&](int at, int n, int j, uint32_t accumulate) {
      tc::mma_bf16(tmem + ((shift >= 2) + at) * CC, desc128(sa + j * 32, 0), desc128(sb + at * CC * 128 + j * 32, 0),
                   tc::idesc_bf16(128, CC * n, false, false), accumulate);
    };
    if (s % Hf == 0) {  // every shift but the first adds to classes begun before and begins one
      if (shift == 0) {
        step(0, 3, 0, 1);
        step(3, 1, 0, 0);
      } else {
        if (shift != 3) step(shift == 2 ? 0 : 1, 1, 0, 1);
        step(shift == 2 ? 1 : 0, 1, 0, 0);
      }
    } else {
      step(0, nb, 0, 1);
    }
#pragma unroll
    for (int j = 1; j < 4; ++j) step(0, nb, j, 1);
  }
  // Masked by the sign of the activation that the buffer holds, added to the thread's column sums (FP32), rounded
  // once to BF16 in the activation's place.
  static __device__ void epilogue(uint32_t tmem, uint8_t* io, const float*, int r, float* sums) {
#pragma unroll
    for (int pos = 0; pos < 4; ++pos) {
      constexpr int kClass[4] = {1, 3, 2, 0};
      const int cls = kClass[pos];
#pragma unroll
      for (int q = 0; q < CC / 32; ++q) {
        float v[32];
        tmem_ld32(tmem + pos * CC + q * 32, v);
        uint8_t* box = io + (CC == 32 ? cls >> 1 : cls) * kSlice;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint4* p = reinterpret_cast<uint4*>(box + box_off(r, (CC == 32 ? (cls & 1) : q) * 4 + c));
          const uint4 a = *p;
          const uint32_t w[4] = {a.x, a.y, a.z, a.w};
          uint32_t o[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float lo = __uint_as_float(w[i] << 16) > 0.f ? v[8 * c + 2 * i] : 0.f;
            const float hi = __uint_as_float(w[i] & 0xFFFF0000u) > 0.f ? v[8 * c + 2 * i + 1] : 0.f;
            sums[q * 32 + 8 * c + 2 * i] += lo;
            sums[q * 32 + 8 * c + 2 * i + 1] += hi;
            o[i] = pack2(lo, hi);
          }
          *p = make_uint4(o[0], o[1], o[2], o[3]);
        }
      }
    }
  }
  static __device__ void load_io(const CUtensorMap* m, uint64_t* bar, uint32_t io, int t, int chunk) {
    expect_tx(bar, kIoBoxes * kSlice);
#pragma unroll
    for (int q = 0; q < kIoBoxes; ++q) {
      if constexpr (CC == 32) load5(io + q * kSlice, m, bar, 0, 0, q, G::row(t), G::img(t));
      else load5(io + q * kSlice, m, bar, (q & 1) * G::C + chunk * 64, 0, q >> 1, G::row(t), G::img(t));
    }
  }
  static __device__ void store_io(const CUtensorMap* m, uint32_t io, int t, int chunk) {
#pragma unroll
    for (int q = 0; q < kIoBoxes; ++q) {
      if constexpr (CC == 32) store5(m, io + q * kSlice, 0, 0, q, G::row(t), G::img(t));
      else store5(m, io + q * kSlice, (q & 1) * G::C + chunk * 64, 0, q >> 1, G::row(t), G::img(t));
    }
  }
};

template <class P>
struct Smem {
  static constexpr int kStage = kSlice + P::kBBytes;
  static constexpr int kIoBytes = P::kIoBoxes * kSlice;
  static constexpr int kBars = 1024 + P::kStages * kStage + P::kIo * kIoBytes;  // from the aligned base: - 1024
  static constexpr size_t kBytes = kBars + 256 + 512;                          // barriers, bias
};

// Tiles blockIdx.x, blockIdx.x + gridDim.x, ... of 128 rows.  Double-buffered accumulator (2 kCols columns).
template <class P>
__global__ void __launch_bounds__(kThreads, P::kCtas)
    k_conv(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, const __grid_constant__ CUtensorMap mio,
           const __grid_constant__ CUtensorMap mout, const float* __restrict__ bias, float* __restrict__ colpart, int colpitch,
           int n_tiles, unsigned* status, unsigned limit) {
  using S = Smem<P>;
  constexpr int kSt = P::kStages;
  extern __shared__ unsigned char smem_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* io = sm + kSt * S::kStage;
  uint64_t* full = (uint64_t*)(io + P::kIo * S::kIoBytes);
  uint64_t *empty = full + kSt, *tfull = empty + kSt, *tempty = tfull + 2, *iofull = tempty + 2, *ioempty = iofull + 2,
           *drain = ioempty + 2;
  uint32_t* slot = (uint32_t*)(drain + 1);
  float* sbias = (float*)((uint8_t*)full + 256);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, chunk = blockIdx.y;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSt; ++s) {
      tc::mbar_init(full + s, 1);
      tc::mbar_init(empty + s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(tfull + s, 1);
      tc::mbar_init(tempty + s, 4);
      tc::mbar_init(iofull + s, 1);
      tc::mbar_init(ioempty + s, 1);
    }
    tc::mbar_init(drain, 1);
    tc::mbar_init_fence();
  }
  if (!P::kMask && threadIdx.x < P::kCols) sbias[threadIdx.x] = bias[threadIdx.x];
  if (warp == 2) tc::tmem_alloc(slot, 2 * P::kCols);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *slot, sbase = tc::smem_u32(sm), iobase = tc::smem_u32(io);
  bool ok = true;
  if (warp == 0) {
    if (lane == 0) {
      unsigned g = 0, i = 0;  // slices and activation tiles issued
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        for (int s = 0; s < P::kSlices; ++s, ++g) {
          const unsigned st = g % kSt;
          if (g >= kSt && !(ok = tc::mbar_wait(empty + st, (g / kSt - 1) & 1u, limit))) break;
          expect_tx(full + st, P::slice_bytes(s));
          const uint32_t sa = sbase + st * S::kStage;
          P::load(&ma, &mb, full + st, sa, sa + kSlice, s, t, chunk);
        }
        if (P::kMask && ok) {  // the activations of the tile, once its buffer has been stored from
          const unsigned b = i % P::kIo;
          if (i >= P::kIo && !(ok = tc::mbar_wait(ioempty + b, (i / P::kIo - 1) & 1u, limit))) break;
          P::load_io(&mio, iofull + b, iobase + b * S::kIoBytes, t, chunk);
          ++i;
        }
      }
      // every copy has landed before the CTA may leave
      for (unsigned k = g > kSt ? g - kSt : 0; k < g; ++k) tc::mbar_wait(full + k % kSt, (k / kSt) & 1u, tc::kWaitLimit);
      for (unsigned k = i > P::kIo ? i - P::kIo : 0; k < i; ++k)
        tc::mbar_wait(iofull + k % P::kIo, (k / P::kIo) & 1u, tc::kWaitLimit);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      unsigned g = 0, i = 0;
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++i) {
        if (i >= 2 && !(ok = tc::mbar_wait(tempty + (i & 1), (i / 2 - 1) & 1u, limit))) break;
        tc::fence_after();
        for (int s = 0; s < P::kSlices; ++s, ++g) {
          const unsigned st = g % kSt;
          if (!(ok = tc::mbar_wait(full + st, (g / kSt) & 1u, limit))) break;
          tc::fence_after();
          const uint32_t sa = sbase + st * S::kStage;
          P::mma(tmem + (i & 1) * P::kCols, sa, sa + kSlice, s);
          tc::mma_commit(empty + st);
        }
        if (ok) tc::mma_commit(tfull + (i & 1));
      }
      tc::mma_commit(drain);
      tc::mbar_wait(drain, 0, tc::kWaitLimit);
    }
  } else if (warp >= 4) {
    const int r = threadIdx.x - 128, w = warp - 4;
    float sums[P::kSums];
#pragma unroll
    for (int j = 0; j < P::kSums; ++j) sums[j] = 0.f;
    unsigned i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
      const unsigned b = i % P::kIo;
      ok = tc::mbar_wait(tfull + (i & 1), (i / 2) & 1u, limit);
      if (P::kMask) ok = ok && tc::mbar_wait(iofull + b, (i / P::kIo) & 1u, limit);
      if (!P::kMask && r == 0) store_wait_read();  // the staging buffer has been read
      ok = __all_sync(0xffffffffu, ok);
      int all;  // the four warps leave together
      asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.and.pred q, 1, 128, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                   : "=r"(all)
                   : "r"((int)ok)
                   : "memory");
      ok = all != 0;
      if (!ok) break;
      tc::fence_after();
      P::epilogue(tmem + (i & 1) * P::kCols + ((uint32_t)(w * 32) << 16), io + b * S::kIoBytes, sbias, r, sums);
      tc::fence_before();
      tc::fence_async_smem();
      __syncwarp();
      if (lane == 0) arrive(tempty + (i & 1));
      epilogue_sync();
      if (r == 0) {
        P::store_io(&mout, iobase + b * S::kIoBytes, t, chunk);
        store_commit();
        if (P::kMask) {
          store_wait_read();
          arrive(ioempty + b);
        }
      }
    }
    if (r == 0) store_wait();
    if (P::kMask && ok) {  // column sums of the CTA's rows, in row order (the stage buffers are idle by now)
      float* red = reinterpret_cast<float*>(sm);
#pragma unroll
      for (int j = 0; j < P::kSums; ++j) red[r * (P::kSums + 1) + j] = sums[j];
      epilogue_sync();
      if (r < P::kSums) {
        float a[4] = {0.f, 0.f, 0.f, 0.f};
        for (int k = 0; k < 32; ++k)
#pragma unroll
          for (int q = 0; q < 4; ++q) a[q] += red[(q * 32 + k) * (P::kSums + 1) + r];
        colpart[(size_t)blockIdx.x * colpitch + chunk * P::kSums + r] = (a[0] + a[1]) + (a[2] + a[3]);
      }
    }
  }
  if (!ok) atomicExch(status, 1u);
  __syncthreads();
  if (warp == 2) {
    tc::fence_after();
    tc::tmem_dealloc(tmem, 2 * P::kCols);
  }
}

// ---- weight gradient ----------------------------------------------------------------------------------
// blockIdx.x: three of the 128-row tiles of (tap, ci); blockIdx.y: a share of the 64-pixel boxes, per_split each.
// A tile is two boxes of 64 channels: with C = 32 the pixel pairs x - 1 and x (its first 32 rows, the lower half of
// the left pair, belong to no tap), else blocks of 64 of the 9 C rows.
template <int L>
struct Dw {
  using G = Geo<L>;
  static constexpr int kBox = 64 * 128;  // bytes of 64 pixels x 64 channels
  static constexpr int kBoxes = G::C == 32 ? 6 : 9 * G::C / 64, kGroups = (kBoxes + 5) / 6;
  static constexpr int kBBoxes = G::N / 64, kStages = 3, kStage = (6 + kBBoxes) * kBox;
  static constexpr int kImgSlices = G::Wo * G::Wo / 64, kRows = 64 / G::Wo;
  static constexpr int kCols = G::N == 64 ? 256 : 512;
  static constexpr size_t kBytes = 1024 + (size_t)kStages * kStage + 128;
};

template <int L>
__global__ void __launch_bounds__(kThreads, 1)
    k_conv_dw(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, float* __restrict__ part,
              int n_slices, int per_split, unsigned* status, unsigned limit) {
  using P = Dw<L>;
  using G = Geo<L>;
  constexpr int kSt = P::kStages;
  extern __shared__ unsigned char smem_raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(sm + kSt * P::kStage);
  uint64_t *empty = full + kSt, *done = empty + kSt;
  uint32_t* slot = (uint32_t*)(done + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int box0 = blockIdx.x * 6, nbox = min(6, P::kBoxes - box0);
  const int s0 = min(n_slices, (int)blockIdx.y * per_split), ns = min(per_split, n_slices - s0);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSt; ++s) {
      tc::mbar_init(full + s, 1);
      tc::mbar_init(empty + s, 1);
    }
    tc::mbar_init(done, 1);
    tc::mbar_init_fence();
  }
  if (warp == 2) tc::tmem_alloc(slot, P::kCols);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *slot, sbase = tc::smem_u32(sm);
  bool ok = true;
  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      for (; g < ns; ++g) {
        const int st = g % kSt, s = s0 + g, b = s / P::kImgSlices, y = s % P::kImgSlices * P::kRows;
        if (g >= kSt && !(ok = tc::mbar_wait(empty + st, (g / kSt - 1) & 1u, limit))) break;
        expect_tx(full + st, (nbox + P::kBBoxes) * P::kBox);
        const uint32_t sa = sbase + st * P::kStage;
        for (int k = 0; k < nbox; ++k) {
          const int q = box0 + k;
          if constexpr (G::C == 32) {
            const int ky = q >> 1;
            load5(sa + k * P::kBox, &ma, full + st, 0, (q & 1) - 1, ky != 1, y - (ky == 0), b);
          } else {
            constexpr int Hf = G::C / 64;
            const int tap = q / Hf, ky = tap / 3, kx = tap % 3;
            load5(sa + k * P::kBox, &ma, full + st, (kx != 1 ? G::C : 0) + q % Hf * 64, -(kx == 0), ky != 1, y - (ky == 0), b);
          }
        }
        for (int k = 0; k < P::kBBoxes; ++k) load2(sa + (6 + k) * P::kBox, &mb, full + st, k * 64, s * 64);
      }
      for (int k = max(0, g - kSt); k < g; ++k) tc::mbar_wait(full + k % kSt, (k / kSt) & 1u, tc::kWaitLimit);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = tc::idesc_bf16(128, G::N, true, true);
      for (int g = 0; g < ns; ++g) {
        const int st = g % kSt;
        if (!(ok = tc::mbar_wait(full + st, (g / kSt) & 1u, limit))) break;
        tc::fence_after();
        const uint32_t sa = sbase + st * P::kStage;
        for (int m = 0; 2 * m < nbox; ++m)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            tc::mma_bf16(tmem + m * G::N, desc128(sa + 2 * m * P::kBox + j * 2048, P::kBox),
                         desc128(sa + 6 * P::kBox + j * 2048, P::kBox), idesc, (g > 0 || j > 0) ? 1u : 0u);
        tc::mma_commit(empty + st);
      }
      tc::mma_commit(done);
      if (!tc::mbar_wait(done, 0, tc::kWaitLimit)) ok = false;
    }
  }
  if (!ok) atomicExch(status, 1u);
  __syncthreads();  // all MMAs are done (their commit was waited for)
  tc::fence_after();
  if (warp >= 4) {
    constexpr int kK = 9 * G::C, kTile = G::C == 32 ? 96 : 128;
    const int r = threadIdx.x - 128, w = warp - 4;
    for (int m = 0; 2 * m < nbox; ++m) {
      const int k = (blockIdx.x * 3 + m) * kTile + r - (128 - kTile);
      const bool valid = r >= 128 - kTile && k < kK;
      float* out = part + (size_t)blockIdx.y * G::N * kK + k;
#pragma unroll 1
      for (int q = 0; q < G::N / 32; ++q) {
        float v[32];
        tmem_ld32(tmem + m * G::N + q * 32 + ((uint32_t)(w * 32) << 16), v);
        if (valid)
#pragma unroll
          for (int j = 0; j < 32; ++j) out[(size_t)(q * 32 + j) * kK] = ns > 0 ? v[j] : 0.f;
        __syncwarp();
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 2) {
    tc::fence_after();
    tc::tmem_dealloc(tmem, P::kCols);
  }
}

// ---- host side ----------------------------------------------------------------------------------------
typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static const EncodeFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return (EncodeFn)p;
  }();
  return fn;
}

// A BF16 tensor of `rank` dimensions (innermost first; strides of the others in elements), boxes of 64 channels.
struct Dims {
  cuuint64_t n[5], stride[5];
  cuuint32_t box[5];
};
bool encode(CUtensorMap* m, const void* p, int rank, const Dims& d) {
  cuuint64_t bytes[4];
  const cuuint32_t ones[5] = {1, 1, 1, 1, 1};
  for (int k = 1; k < rank; ++k) bytes[k - 1] = d.stride[k] * 2;
  const EncodeFn fn = encode_fn();
  return fn && fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(p), d.n, bytes, d.box, ones,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// The parity view of convolution L's input, boxes of `rows` output rows of `imgs` images.
template <int L>
bool input_map(CUtensorMap* m, const void* p, int B, int rows, int imgs) {
  using G = Geo<L>;
  constexpr cuuint64_t C = G::C, H = G::H;
  return encode(m, p, 5, Dims{{2 * C, H / 2, 2, H / 2, (cuuint64_t)B}, {1, 2 * C, H * C, 2 * H * C, H * H * C},
                              {64, (cuuint32_t)G::Wo, 1, (cuuint32_t)rows, (cuuint32_t)imgs}});
}
bool matrix_map(CUtensorMap* m, const void* p, long long cols, long long rows, int box_rows) {
  return encode(m, p, 2, Dims{{(cuuint64_t)cols, (cuuint64_t)rows}, {1, (cuuint64_t)cols}, {64, (cuuint32_t)box_rows}});
}

template <class P>
cudaError_t launch(const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& io, const CUtensorMap& out, const float* bias,
                   float* colpart, int tiles, int gx, int gy, unsigned* status, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(k_conv<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem<P>::kBytes);
  if (e != cudaSuccess) return e;
  k_conv<P><<<dim3(gx, gy), kThreads, Smem<P>::kBytes, st>>>(a, b, io, out, bias, colpart, P::G::C, tiles, status, loop_wait_limit());
  note_launches(1);
  return cudaGetLastError();
}

template <int L>
cudaError_t forward(const uint16_t* act, const uint16_t* w, const float* bias, int B, uint16_t* out, long long pitch,
                    unsigned* status, cudaStream_t st) {
  using G = Geo<L>;
  CUtensorMap a, b, o;
  constexpr cuuint64_t px = G::Wo * G::Wo;
  if (!input_map<L>(&a, act, B, G::kRows, G::kImgs) || !matrix_map(&b, w, 9 * G::C, G::N, G::N) ||
      !encode(&o, out, 3, Dims{{G::N, px, (cuuint64_t)B}, {1, G::N, (cuuint64_t)pitch}, {64, 128 / G::kImgs, G::kImgs}}))
    return cudaErrorInvalidValue;
  const int tiles = G::tiles(B);
  return launch<Fwd<L>>(a, b, o, o, bias, nullptr, tiles, std::min(tiles, Fwd<L>::kCtas * kSms), 1, status, st);
}

template <int L>
cudaError_t data_gradient(const uint16_t* dy, const uint16_t* wt, const uint16_t* act, int B, uint16_t* dx, float* colpart,
                          int gx, unsigned* status, cudaStream_t st) {
  using G = Geo<L>;
  using P = Dx<L>;
  CUtensorMap a, b, m, o;
  constexpr cuuint64_t N = G::N, W = G::Wo;
  if (!encode(&a, dy, 4, Dims{{N, W, W, (cuuint64_t)B}, {1, N, N * W, N * W * W}, {64, (cuuint32_t)W, G::kRows, G::kImgs}}) ||
      !matrix_map(&b, wt, 64, 9LL * G::C * (G::N / 64), P::CC) || !input_map<L>(&m, act, B, G::kRows, G::kImgs) ||
      !input_map<L>(&o, dx, B, G::kRows, G::kImgs))
    return cudaErrorInvalidValue;
  return launch<P>(a, b, m, o, nullptr, colpart, G::tiles(B), gx, G::C / P::CC, status, st);
}

template <int L>
cudaError_t weight_gradient(const uint16_t* act, const uint16_t* dy, int B, float* part, int Z, unsigned* status,
                            cudaStream_t st) {
  using G = Geo<L>;
  using P = Dw<L>;
  CUtensorMap a, b;
  const long long px = (long long)B * G::Wo * G::Wo;
  if (!input_map<L>(&a, act, B, P::kRows, 1) || !matrix_map(&b, dy, G::N, px, 64)) return cudaErrorInvalidValue;
  const cudaError_t e = cudaFuncSetAttribute(k_conv_dw<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P::kBytes);
  if (e != cudaSuccess) return e;
  const int n = (int)(px / 64);
  k_conv_dw<L><<<dim3(P::kGroups, Z), kThreads, P::kBytes, st>>>(a, b, part, n, (n + Z - 1) / Z, status, loop_wait_limit());
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t cnn_conv_forward(int l, const uint16_t* act, const uint16_t* w, const float* bias, int B, uint16_t* out,
                             long long pitch, unsigned* status, cudaStream_t st) {
  if (l == 1) return forward<1>(act, w, bias, B, out, pitch, status, st);
  if (l == 2) return forward<2>(act, w, bias, B, out, pitch, status, st);
  return forward<3>(act, w, bias, B, out, pitch, status, st);
}

int cnn_conv_dx_rows(int l, int B) {
  const int tiles = l == 1 ? Geo<1>::tiles(B) : (l == 2 ? Geo<2>::tiles(B) : Geo<3>::tiles(B));
  return std::min(tiles, kSms / (l == 3 ? Geo<3>::C / Dx<3>::CC : 1));
}

cudaError_t cnn_conv_dx(int l, const uint16_t* dy, const uint16_t* wt, const uint16_t* act, int B, uint16_t* dx,
                        float* colpart, unsigned* status, cudaStream_t st) {
  const int gx = cnn_conv_dx_rows(l, B);
  if (l == 1) return data_gradient<1>(dy, wt, act, B, dx, colpart, gx, status, st);
  if (l == 2) return data_gradient<2>(dy, wt, act, B, dx, colpart, gx, status, st);
  return data_gradient<3>(dy, wt, act, B, dx, colpart, gx, status, st);
}

int cnn_conv_dw_splits(int l, int B, long long part_floats) {
  const long long slices = (long long)B * kSide[l + 1] * kSide[l + 1] / 64;
  // 304 (tile of 128 rows, split) pairs, at least four boxes per split.  The line is that of the gathering kernels
  // before: the same splits give the same sums, bit for bit, and so the same rounded weights after a step.
  const int tiles = (9 * kChan[l] + 127) / 128;
  long long z = (2 * kSms + tiles - 1) / tiles;
  z = std::min(z, std::max(1LL, slices / 4));
  z = std::min(z, std::max(1LL, part_floats / (9LL * kChan[l] * kChan[l + 1])));
  const long long per = (slices + z - 1) / z;
  return (int)((slices + per - 1) / per);
}

cudaError_t cnn_conv_dw(int l, const uint16_t* act, const uint16_t* dy, int B, float* part, int Z, unsigned* status,
                        cudaStream_t st) {
  if (l == 1) return weight_gradient<1>(act, dy, B, part, Z, status, st);
  if (l == 2) return weight_gradient<2>(act, dy, B, part, Z, status, st);
  return weight_gradient<3>(act, dy, B, part, Z, status, st);
}

}  // namespace digs
