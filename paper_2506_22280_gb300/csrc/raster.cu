// Tile rasteriser of the X-ray transform (Sec. 3.1, Eq. 1, 3-4) and its backward pass.
//
// Per pixel, with (dx, dy) its offset from the projected mean:
//   num = n00 dx^2 + n01x2 dx dy + n11 dy^2,  t = 1 + wn0 dx + wn1 dy,  D = t^2 + kappa num,  E = num / D,
// and the pixel takes V = amp |X - s| D^-1/2 exp(-E/2) when E <= cutoff^2.  The constant k = -log2(e)/2
// is folded into num, so that k E is directly the argument of the SFU's exp2; D^-1/2 is the SFU's
// reciprocal square root.  Pixels are taken two at a time in packed FP32x2 arithmetic
// (fma/mul/add.rn.f32x2).
//
// Forward: a warp owns two 8 x 8 blocks, side by side, of a (projection, tile), each lane two pixels of both with
// their sums in registers; the warps of a CTA share its pixels and split its sorted Gaussian list.  A warp takes
// 32 records at a time, one per lane, writes an entry for every block whose pixels the record's cutoff ellipse
// can reach, and sweeps each block's entries, four per step, in list order: no canvas, no atomics, sums that do
// not depend on timing.  CTAs start in order of decreasing list length.
// What bounds it: instruction issue (69 % of cycles), about 26 instructions per entry and block of 64 pixels (FMA pipe
// 61 % busy, SFU 38 %), then loading and testing the records.  One block per warp made every block load and
// test the whole list by itself: a third of the time.  128 thorax projections (100k Gaussians, 256^2):
// 5.37 -> 4.70 ms; 16: 0.79 -> 0.60; 8 of 500k Gaussians on 512^2: 5.0 -> 4.1; 16 of 2,000 on 64^2:
// 0.045 -> 0.023.
//
// Backward: needs no tile lists.  One half-warp per (projection, Gaussian) record (the two records of a warp of
// similar box size) sweeps the record's pixel box in 16-column slices, reading g = dL/dI * |X - s| from the
// projection-sized image (L1/L2 resident).  Narrow slices (w <= 8): lane l owns column (l mod w), starts at row
// (l div w) and takes the row pair (r, r + s), s = 16 div w, stepping 2s rows; wider slices: the column pair
// (c, c + ceil(w/2)) of row (l div ceil(w/2)), stepping s = 16 div ceil(w/2) rows.  Each lane accumulates the value
// and six moments per pixel of its pair; a slice adds them to twelve (dx, dy)-moments, the half-warp reduces those with
// a 12-shuffle recursive halving and twelve lanes write them to the record's slot (no atomics).
// What bounds it: the FMA pipe (packed arithmetic takes two of its cycles; 65 % busy) and the instructions per
// record around the sweep (a third of the time).  128 thorax projections (100k Gaussians, 256^2), with the
// ranking of the records: 8.81 -> 7.67 ms; 16 of 2,000 on 64^2: 0.035 -> 0.029; 64 of four scans of 30k to 200k,
// whose missing records are no longer visited: 5.17 -> 3.97.
//
// Loss: per-warp partials of the squared residuals from the forward, summed in two fixed-order levels.
#include <algorithm>

#include "digs_internal.h"

namespace digs {

constexpr float kNegHalfLog2e = -0.5f * DIGS_LOG2E;


// ---- packed FP32x2: the two pixels of a lane's pair in one register pair ------------------------
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pack(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f2 f2_dup(float x) { return f2_pack(x, x); }
__device__ __forceinline__ void f2_unpack(f2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// The SFU's 2^x and 1/sqrt(x) (PTX ex2.approx / rsqrt.approx, flushing subnormals: the arguments here
// are in [-9, 0] and near 1).
__device__ __forceinline__ float sfu_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sfu_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ f2 f2_exp2(f2 x) {
  float a, b;
  f2_unpack(x, a, b);
  return f2_pack(sfu_exp2(a), sfu_exp2(b));
}
__device__ __forceinline__ f2 f2_rsqrt(f2 x) {
  float a, b;
  f2_unpack(x, a, b);
  return f2_pack(sfu_rsqrt(a), sfu_rsqrt(b));
}

// ---- lane layouts (forward and backward) ---------------------------------------------------------

// Lane layout of a box slice w <= LPR pixels wide for a group of LPR lanes (16 or 32) sharing one
// record, per w: cw | s << 6 | m << 12, where cw is the number of lane columns, s the rows covered per
// pass and m = ceil(1024 / cw), so that (l * m) >> 10 = l / cw exactly for l < 32 (cw <= 16).
// w <= LPR/2: lane l takes column l mod w and the row pair (r, r + s), s = LPR div w, stepping 2s rows.
// LPR/2 < w <= LPR: the column pair (c, c + ceil(w/2)), stepping s = LPR div ceil(w/2) rows.
template <int LPR>
struct LaneTable {
  int v[LPR + 1];
  constexpr LaneTable() : v() {
    for (int w = 1; w <= LPR; ++w) {
      const int cw = w <= LPR / 2 ? w : (w + 1) / 2;
      v[w] = cw | ((LPR / cw) << 6) | (((1024 + cw - 1) / cw) << 12);
    }
  }
};
__constant__ LaneTable<16> kLanes16 = LaneTable<16>();
__constant__ LaneTable<32> kLanes32 = LaneTable<32>();

struct HalfLanes {
  int c, r0, pdx, pdy, ystep;
  bool active, col2;
};
template <int LPR>
__device__ __forceinline__ HalfLanes group_lanes(int w, int h, int hl) {
  const int t = LPR == 16 ? kLanes16.v[w] : kLanes32.v[w];
  const int cw = t & 63, s = (t >> 6) & 63, m = t >> 12;
  const int q = (hl * m) >> 10;
  const bool rows = w <= LPR / 2;
  HalfLanes L;
  L.c = hl - q * cw;
  L.r0 = q;
  L.pdx = rows ? 0 : cw;
  L.pdy = rows ? s : 0;
  L.ystep = rows ? 2 * s : s;
  L.active = q < s && q < h;
  L.col2 = L.c + L.pdx < w;
  return L;
}

// ---- forward ------------------------------------------------------------------------------------

// A CTA takes 16 x 16 pixels of a (projection, tile) (tiles of 32 pixels: four CTAs share a list), or a tile of
// 8 x 8; tiles in the order `order` gives.  A warp owns `blocks` of its 8 x 8 blocks and every `splits`-th batch of the
// list; lane l owns the pixels (l mod 8, l div 8) and (l mod 8, l div 8 + 4) of each block and keeps their sums
// in registers.
template <int TS>
struct FwdCfg {
  static constexpr int blocks = TS == 8 ? 1 : 2;
  static constexpr int groups = TS == 8 ? 1 : 4 / blocks;  // warps that share the CTA's blocks
  // Four splits whatever the launch, so that a projection's sums, and its bits, do not depend on the views beside it.
  // They cut the longest chain of work in launches of few CTAs (two against four splits: 16 views of 64^2 29 against
  // 23 us); where a launch has many waves, two would do (a forward of 128 thorax projections, tiles of 8, 16 and 32
  // pixels: 6.91, 6.06 and 6.41 ms with one or two splits, 7.08, 6.02 and 6.63 with four).
  static constexpr int splits = 4;
  static constexpr int warps = groups * splits;
  static constexpr int subs = TS == 32 ? 4 : 1;        // CTAs per tile
  static constexpr int threads = 32 * warps;
  static constexpr int batch = 32;                     // records a warp takes at a time: one per lane
  static constexpr int step = splits * batch;          // from one of a warp's batches to its next
  // CTAs per SM that the registers are held to: 24 warps of 80 registers (one block per warp: 32 of 64).
  static constexpr int min_ctas = (blocks == 1 ? 32 : 24) / warps;
};

// A record as the pixel loops read it: with k = -log2(e) / 2 and sg = |amp| (1 when |amp| lies outside
// [2^-40, 2^40]),
//   (k n00 / sg^2, k n01x2 / sg^2, k n11 / sg^2, wn0 / sg), (wn1 / sg, kappa / k, amp / sg, -xc), (-yc, 1 / sg, 0, 0).
// The loop then forms the exp2 argument k E = k num / D directly; num and t scaled by 1 / sg^2 and 1 / sg scale D by
// 1 / sg^2 and leave E unchanged, so the SFU's rsqrt of the scaled D is sg D^-1/2 (amp / sg, i.e. the sign of amp,
// multiplies both pixels of a lane at once).
struct FwdEntry {
  float4 q[3];
};
__device__ __forceinline__ FwdEntry scale_record(const float4& a, const float4& b, const float4& c) {
  const float mag = fabsf(c.x);
  const bool fold = mag >= 0x1p-40f && mag <= 0x1p40f;
  const float s1 = fold ? __frcp_rn(mag) : 1.f, s2 = s1 * s1;
  FwdEntry e;
  e.q[0] = make_float4(kNegHalfLog2e * a.z * s2, kNegHalfLog2e * a.w * s2, kNegHalfLog2e * b.x * s2, b.y * s1);
  e.q[1] = make_float4(b.z * s1, b.w * (1.f / kNegHalfLog2e), fold ? copysignf(1.f, c.x) : c.x, -a.x);
  e.q[2] = make_float4(-a.y, s1, 0.f, 0.f);
  return e;
}

// Whether the 8 x 8 pixel block whose centre lies at (X, Y) from the projected mean can hold a pixel with
// E <= c2: E = num / D with D <= Dmax over the record's box, and lim = c2 Dmax (with a small margin, from the
// set-up), so no pixel qualifies when min over the block of the quadratic form num exceeds lim.  The minimum
// of a positive definite form over a rectangle lies on one of the two edges that face its centre (or on a
// line through the centre, where the rectangle spans it), and on such a line it is a clamped one-dimensional
// minimum; a centre inside the block gives zero.  A culled block's entries would only have added zeros.
// sy = -n01 / n11 and sx = -n01 / n00 (n01x2 = 2 n01) from approximate divisions: they move the clamped
// minimisers by a few ulps, far inside the margin.
__device__ __forceinline__ bool ellipse_meets(float n00, float n01x2, float n11, float sx, float sy, float lim, float X,
                                              float Y) {
  const float X0 = X - 3.5f, X1 = X + 3.5f, Y0 = Y - 3.5f, Y1 = Y + 3.5f;
  const float ex = fminf(fmaxf(0.f, X0), X1), ey = fminf(fmaxf(0.f, Y0), Y1);
  const float dy = fminf(fmaxf(sy * ex, Y0), Y1), dx = fminf(fmaxf(sx * ey, X0), X1);
  const float qx = fmaf(ex, fmaf(n00, ex, n01x2 * dy), n11 * dy * dy);
  const float qy = fmaf(ey, fmaf(n11, ey, n01x2 * dx), n00 * dx * dx);
  return !(fminf(qx, qy) > lim);
}

// One entry at the lane's two pixels, x and YY = (y, y + 4): their exp2 arguments k E (a pair counts where
// k E >= c2 k), and V / |X - s| as r 2^(k E).  The form is evaluated about the mean, whose offset is formed first:
// expanded about a block's centre instead it costs two operations fewer per entry, but its terms cancel near the mean
// of a small Gaussian (root mean square error of E in FP32, about the mean and about the block's centre: 1e-7 and
// 2.2e-7 at a sigma of 2.8 pixels, 6e-7 at 1, 6e-6 at 0.3, 5e-5 at 0.1).
struct FwdPair {
  float ra, rb, ea, eb;
};
__device__ __forceinline__ FwdPair fwd_pair(const float4* en, float x, f2 YY) {
  const float4 q0 = en[0], q1 = en[1], q2 = en[2];
  // the lane's two pixels share their column: its terms are formed once
  const float dx = x + q1.w;
  float p, bq;
  f2_unpack(f2_mul(f2_pack(q0.x, q0.y), f2_dup(dx)), p, bq);
  const float aq = p * dx, tq = fmaf(q0.w, dx, q2.y);
  const f2 DY = f2_add(YY, f2_dup(q2.x));
  const f2 NUM = f2_fma(DY, f2_fma(f2_dup(q0.z), DY, f2_dup(bq)), f2_dup(aq));  // k num / sg^2
  const f2 T = f2_fma(f2_dup(q1.x), DY, f2_dup(tq));                             // t / sg
  const f2 D = f2_fma(T, T, f2_mul(f2_dup(q1.y), NUM));                          // D / sg^2
  const f2 RS = f2_rsqrt(D);                                                     // sg D^-1/2
  const f2 ARG = f2_mul(NUM, f2_mul(RS, RS));                                    // k E
  FwdPair r;
  f2_unpack(f2_mul(RS, f2_dup(q1.z)), r.ra, r.rb);
  f2_unpack(ARG, r.ea, r.eb);
  return r;
}

// Each warp walks the tile's list a batch at a time, one record per lane (in registers, loaded while the batch
// before it is swept).  A lane tests its record against the warp's blocks and writes the entry of each block
// that it meets; a ballot's prefix count gives the entry its place, packed and in list order, in the block's
// table.  The warp then sweeps each block's table in order, four entries per step (independent dependency
// chains, summed in list order): no canvas, no atomics, no CTA barrier.
template <int TS, bool COUNT>
__global__ void __launch_bounds__(FwdCfg<TS>::threads, FwdCfg<TS>::min_ctas) k_raster_fwd(
    const float4* __restrict__ grec, const uint32_t* __restrict__ srid, const uint2* __restrict__ ranges,
    const uint32_t* __restrict__ order, const __grid_constant__ ViewsParam views, int tiles_x, int T, int nu, int nv,
    float* __restrict__ proj, const float* __restrict__ meas, float* __restrict__ dldi,
    float* __restrict__ loss_part, float c2, float inv_count, unsigned long long* __restrict__ counters) {
  using C = FwdCfg<TS>;
  constexpr int NB = C::blocks;
  __shared__ float4 tables[C::warps][NB][C::batch * 3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int group = warp % C::groups, split = warp / C::groups;
  const uint32_t bt = order[blockIdx.x / C::subs];  // heaviest (projection, tile) lists first
  const int sub = blockIdx.x % C::subs;
  const int b = (int)(bt / (uint32_t)T), tile = (int)(bt % (uint32_t)T);
  // first pixel of the warp's first block; block q lies 8 (q mod 2) pixels to the right and 8 (q div 2) below
  const int gx = (tile % tiles_x) * TS + (sub & 1) * 16 + (NB == 1 ? (group & 1) * 8 : 0);
  const int gy = (tile / tiles_x) * TS + (sub >> 1) * 16 + (NB == 1 ? group >> 1 : group) * 8;
  const float cx = (float)gx + 3.5f, cy = (float)gy + 3.5f;  // its centre
  const float xl = (float)(gx + (lane & 7)), yl = (float)(gy + (lane >> 3));  // the lane's pixel of that block
  const uint2 rg = ranges[(size_t)b * T + tile];
  const float c2k = c2 * kNegHalfLog2e;
  float s[NB][2];
#pragma unroll
  for (int q = 0; q < NB; ++q) s[q][0] = s[q][1] = 0.f;
  unsigned n_box = 0, n_cut = 0;
  // lane l's record of the next batch, and the record id one batch further ahead
  const uint32_t first = rg.x + split * C::batch;
  uint32_t rid = first + lane < rg.y ? srid[first + lane] : 0u;
  float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra, rc = ra;
  auto fetch = [&](uint32_t k0) {
    if (k0 + lane < rg.y) {
      const float4* src = grec + (size_t)rid * DIGS_REC_F4;
      ra = __ldg(src);
      rb = __ldg(src + 1);
      rc = __ldg(src + 2);
    }
    const uint32_t kn = k0 + C::step + lane;
    rid = kn < rg.y ? srid[kn] : 0u;
  };
  if (first < rg.y) fetch(first);
  for (uint32_t k0 = first; k0 < rg.y; k0 += C::step) {
    const float X = cx - ra.x, Y = cy - ra.y;
    const bool some = k0 + lane < rg.y;  // else the lane holds a record of the batch before, or none
    const float sy = __fdividef(-0.5f * ra.w, rb.x), sx = __fdividef(-0.5f * ra.w, ra.z);
    const FwdEntry r = scale_record(ra, rb, rc);
    int cnt[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      if (COUNT && some) {
        const int bx = __float_as_int(rc.y), by = __float_as_int(rc.z);
        const int qx = gx + (q & 1) * 8, qy = gy + (q >> 1) * 8;
        const int x0 = max(bx & 0xffff, qx), x1 = min(bx >> 16, qx + 7);
        const int y0 = max(by & 0xffff, qy), y1 = min(by >> 16, qy + 7);
        if (x0 <= x1 && y0 <= y1) n_box += (unsigned)((x1 - x0 + 1) * (y1 - y0 + 1));
      }
      const float Xq = X + (float)((q & 1) * 8), Yq = Y + (float)((q >> 1) * 8);
      const bool meets = some && ellipse_meets(ra.z, ra.w, rb.x, sx, sy, rc.w, Xq, Yq);
      const unsigned mask = __ballot_sync(0xffffffffu, meets);
      if (meets) {
        float4* e = &tables[warp][q][__popc(mask & ((1u << lane) - 1u)) * 3];
#pragma unroll
        for (int k = 0; k < 3; ++k) e[k] = r.q[k];
      }
      cnt[q] = __popc(mask);
    }
    __syncwarp();
    fetch(k0 + C::step);  // arrives while this batch is swept
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const float4* e = tables[warp][q];
      const float x = xl + (float)((q & 1) * 8), y = yl + (float)((q >> 1) * 8);
      const f2 YY = f2_pack(y, y + 4.f);
      // n entries from e: all evaluated (independent dependency chains), then accumulated in list order
      auto sweep = [&](int n) {
        FwdPair v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k < n) v[k] = fwd_pair(e + k * 3, x, YY);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k < n) {
            const bool ia = v[k].ea >= c2k, ib = v[k].eb >= c2k;
            const float va = sfu_exp2(v[k].ea), vb = sfu_exp2(v[k].eb);
            s[q][0] = ia ? fmaf(v[k].ra, va, s[q][0]) : s[q][0];
            s[q][1] = ib ? fmaf(v[k].rb, vb, s[q][1]) : s[q][1];
            if (COUNT) n_cut += (unsigned)ia + (unsigned)ib;
          }
        e += n * 3;
      };
#pragma unroll 1
      for (int k = cnt[q] >> 2; k > 0; --k) sweep(4);
      if (cnt[q] & 2) sweep(2);
      if (cnt[q] & 1) sweep(1);
    }
    __syncwarp();
  }
  {  // the splits' sums, added in split order by the first
    float* part = reinterpret_cast<float*>(&tables[0][0][0]);  // [warp][block][2][32]
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      part[((warp * NB + q) * 2) * 32 + lane] = s[q][0];
      part[((warp * NB + q) * 2 + 1) * 32 + lane] = s[q][1];
    }
    __syncthreads();
    if (split == 0) {
#pragma unroll
      for (int q = 0; q < NB; ++q)
#pragma unroll
        for (int z = 1; z < C::splits; ++z) {
          s[q][0] += part[(((z * C::groups + group) * NB + q) * 2) * 32 + lane];
          s[q][1] += part[(((z * C::groups + group) * NB + q) * 2 + 1) * 32 + lane];
        }
    }
  }
  const ViewC& v = views.v[b];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    if (split != 0) break;
    const int px = gx + (q & 1) * 8 + (lane & 7);
    float lsum = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int y = gy + (q >> 1) * 8 + (lane >> 3) + 4 * h;
      if (px < nu && y < nv) {
        const float lp = pixel_ray_length(v, (float)px, (float)y);
        const float I = s[q][h] * lp;
        const size_t idx = ((size_t)b * nv + y) * nu + px;
        if (proj) proj[idx] = I;
        if (meas) {
          const float res = I - meas[idx];
          lsum = fmaf(res, res, lsum);
          if (dldi) dldi[idx] = 2.f * res * inv_count * lp;  // dL/dI * |X - s|, what the backward consumes
        }
      }
    }
    if (loss_part) {  // one partial per 8 x 8 block
      lsum = warp_sum(lsum);
      if (lane == 0) loss_part[(((size_t)b * T + tile) * C::subs + sub) * (C::groups * NB) + group * NB + q] = lsum;
    }
  }
  if (COUNT) {
    unsigned c = n_cut, nb = n_box;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      c += __shfl_xor_sync(0xffffffffu, c, o);
      nb += __shfl_xor_sync(0xffffffffu, nb, o);
    }
    if (lane == 0 && (nb | c)) {
      atomicAdd(counters, (unsigned long long)nb);
      atomicAdd(counters + 1, (unsigned long long)c);
    }
  }
}

// ---- backward: one half-warp per (projection, Gaussian) record, over the record's whole pixel box ----


// Adds the lane's share of a record's twelve pixel moments: with A = (g V / amp) / D and k E the exp2 argument,
//   Sv[0] = sum g V / amp, Sv[1..5] = sum A (dx, dx^2, dy, dx dy, dy^2) and Sv[6..11] = sum A k E (1, dx, dx^2, dy, ...),
// (dx, dy) the pixel's offset from the projected mean.  With B = A (E - 1): dL/dnum = (amp / 2) (kappa B - A),
// dL/dt = amp B t, dL/dkappa = (amp / 2) B num and g V / amp = A D, and t, num and D are polynomials of degree two
// in (dx, dy), so the ten sums of the record's gradient and sum A follow from these twelve with per-record constants:
// pair_adjoint forms them, once per record, instead of every lane of the sweep once per slice of the box.  (The density's
// gradient is Sv[0] alone.  Taken from sum A and the others it costs an addition per pair fewer, 3 %, and carries the
// rounding of 1 / D and back: 3.7 % further from FP64 in the thorax's steps.)
// gp points at g = dL/dI * |X - s| of the lane's first pixel in the projection image (row pitch nu); (dx1, dy1)
// is that pixel's offset.  A lane's pixel keeps its column, so the loop accumulates the six dy-moments and sum g V / amp
// alone (21 packed operations per pixel pair).
__device__ __forceinline__ void bwd_box_pixels(const Rec& R0, const HalfLanes& B, int h, float dx1, float dy1,
                                               const float* __restrict__ gp, int nu, float c2, float Sv[12]) {
  // k = -log2(e) / 2 is folded into the quadratic form: NUM = k num, ARG = k E (the exp2 argument)
  const f2 DX = f2_pack(dx1, dx1 + (float)B.pdx);
  const f2 AQ = f2_mul(f2_mul(f2_dup(kNegHalfLog2e * R0.n00), DX), DX);
  const f2 BQ = f2_mul(f2_dup(kNegHalfLog2e * R0.n01x2), DX);
  const f2 T0 = f2_fma(f2_dup(R0.wn0), DX, f2_dup(1.f));
  const f2 N11 = f2_dup(kNegHalfLog2e * R0.n11), WN1 = f2_dup(R0.wn1);
  const f2 KAPK = f2_dup(R0.kappa * (1.f / kNegHalfLog2e)), STEP = f2_dup((float)B.ystep);
  const f2 C2K = f2_dup(c2 * kNegHalfLog2e);
  const int pstep = B.ystep * nu, d2 = B.pdy * nu + B.pdx, hb = B.col2 ? h - B.pdy : 0;
  f2 DY = f2_pack(dy1, dy1 + (float)B.pdy);
  f2 G0 = f2_dup(0.f), A0 = G0, A1 = G0, A2 = G0, E0 = G0, E1 = G0, E2 = G0;
  for (int r = B.r0; r < h; r += B.ystep, DY = f2_add(DY, STEP), gp += pstep) {
    const f2 NUM = f2_fma(DY, f2_fma(N11, DY, BQ), AQ);
    const f2 T = f2_fma(WN1, DY, T0);
    const f2 D = f2_fma(T, T, f2_mul(KAPK, NUM));
    // E <= cutoff^2 taken as num <= c2 D (D > 0), i.e. k num >= k c2 D: known before the SFU work, so
    // the two loads of dL/dI are in flight while it runs
    const f2 LIM = f2_mul(C2K, D);
    float na, nb, la, lb;
    f2_unpack(NUM, na, nb);
    f2_unpack(LIM, la, lb);
    const float ga = (na >= la) ? __ldg(gp) : 0.f;
    const float gb = (r < hb && nb >= lb) ? __ldg(gp + d2) : 0.f;  // partner in the box
    const f2 RS = f2_rsqrt(D);
    const f2 INVD = f2_mul(RS, RS);
    const f2 ARG = f2_mul(NUM, INVD);
    const f2 BV = f2_mul(RS, f2_exp2(ARG));                            // V / amp
    const f2 GA = f2_mul(f2_pack(ga, gb), BV);                         // g V / amp
    const f2 AL = f2_mul(GA, INVD);                                    // A
    const f2 AE = f2_mul(AL, ARG);                                     // A k E
    const f2 DY2 = f2_mul(DY, DY);
    G0 = f2_add(G0, GA);
    A0 = f2_add(A0, AL);
    A1 = f2_fma(AL, DY, A1);
    A2 = f2_fma(AL, DY2, A2);
    E0 = f2_add(E0, AE);
    E1 = f2_fma(AE, DY, E1);
    E2 = f2_fma(AE, DY2, E2);
  }
  auto add = [&](int q, f2 v) {
    float lo, hi;
    f2_unpack(v, lo, hi);
    Sv[q] += lo + hi;
  };
  const f2 AX = f2_mul(A0, DX), EX = f2_mul(E0, DX);
  add(0, G0);
  add(1, AX);
  add(2, f2_mul(AX, DX));
  add(3, A1);
  add(4, f2_mul(A1, DX));
  add(5, A2);
  add(6, E0);
  add(7, EX);
  add(8, f2_mul(EX, DX));
  add(9, E1);
  add(10, f2_mul(E1, DX));
  add(11, E2);
}

// Sum twelve per-lane values over each group of LPR lanes and store them to out[0..11]: first over each
// half-warp (lanes hl = 0..15), then, for LPR = 32, across the two halves.
// Recursive halving, 6 + 3 + 2 + 1 shuffles: after the xor-8 exchange a lane holds six values, after xor-4
// three, after xor-2 two (or one and a pad), after xor-1 one, the value 6 b3 + 3 b2 + 2 b1 + b0 (b_k = bit k
// of hl) where 2 b1 + b0 < 3.
template <int LPR>
__device__ __forceinline__ void group_reduce_store12(const float v[12], float* out, int hl, bool store) {
  const unsigned full = 0xffffffffu;
  float a[6];
  {
    const bool hi = (hl & 8) != 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const float keep = hi ? v[6 + j] : v[j], send = hi ? v[j] : v[6 + j];
      a[j] = keep + __shfl_xor_sync(full, send, 8);
    }
  }
  float b[3];
  {
    const bool hi = (hl & 4) != 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float keep = hi ? a[3 + j] : a[j], send = hi ? a[j] : a[3 + j];
      b[j] = keep + __shfl_xor_sync(full, send, 4);
    }
  }
  float c0, c1;
  {
    const bool hi = (hl & 2) != 0;
    const float k0 = hi ? b[2] : b[0], k1 = hi ? 0.f : b[1];
    const float s0 = hi ? b[0] : b[2], s1 = hi ? b[1] : 0.f;
    c0 = k0 + __shfl_xor_sync(full, s0, 2);
    c1 = k1 + __shfl_xor_sync(full, s1, 2);
  }
  const bool hi = (hl & 1) != 0;
  float d = (hi ? c1 : c0) + __shfl_xor_sync(full, hi ? c0 : c1, 1);
  if (LPR == 32) d += __shfl_xor_sync(full, d, 16);
  const int local = 2 * ((hl >> 1) & 1) + (hl & 1);
  if (store && (LPR == 16 || (threadIdx.x & 16) == 0) && local < 3)
    out[((hl & 8) ? 6 : 0) + ((hl & 4) ? 3 : 0) + local] = d;
}

// One group of LPR lanes (16: two records per warp, 32: one) per (projection, Gaussian) record: the twelve
// moments over every pixel of the record's box, reduced over the group and written to grec[record].  Nothing is
// written for culled records: the chain does not read those.
//
// A warp takes ranks of one group of 32 consecutive records of a projection.  The two records of a warp are
// swept in lockstep, for as many passes as the longer needs, so the warp first ranks the group by sweep cost
// (box pixels / 32, written by the set-up; 0: culled; ties in index order; bit-sliced ballots) and sweeps
// records of adjacent ranks together; the culled ones rank first and are skipped.  Ranking in the sweeping
// warps themselves replaced a kernel that wrote the ranks to memory (0.076 ms of 128 projections) and two
// dependent loads per record.
// WR rounds of 32 / LPR records per warp and W warps per CTA: one warp that takes the whole group, in a CTA of its
// own, whose place is free for the next as soon as it ends (eight warps in a CTA wait for the longest: 8.05
// against 7.5 ms for 128 thorax projections); where that leaves too few warps, a quarter of the group each (and
// each quarter's warp ranks the group again, about 45 instructions).
// The next rounds' records are copied to shared memory by cp.async (double buffer) while one is swept.
// 28 warps of 72 registers per SM (25 of 80: the same); with 64 registers (32 warps) the loop spills and recomputes
// its lane layout.
// counts.n[b]: records of projection b that exist (its scan's Gaussians); N: record stride of a projection.
// Grid: (ceil(warps / W), P), warps = ceil(N / 32) * 32 / (WR * (32 / LPR)).
struct ViewCounts {
  int n[DIGS_MAX_VIEWS];
};
template <int LPR, int WR, int W>
__global__ void __launch_bounds__(32 * W, 28 / W) k_raster_bwd(const float4* __restrict__ rec,
                                                               const uint8_t* __restrict__ cost,
                                                               const __grid_constant__ ViewCounts counts, int N, int nu,
                                                               int nv, const float* __restrict__ gpix, float c2,
                                                               float* __restrict__ grec) {
  constexpr int kPer = 32 / LPR;             // records per round
  constexpr int kSplits = 32 / (kPer * WR);  // warps per group of 32 records
  __shared__ __align__(16) float4 sbuf[W][2][kPer][DIGS_REC_F4];
  __shared__ uint8_t order[W][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, hl = lane & (LPR - 1), half = lane / LPR;
  const int b = blockIdx.y, nb = counts.n[b];
  const int gw = blockIdx.x * W + warp;
  const int n0 = gw / kSplits * 32, r0 = gw % kSplits * (kPer * WR);  // the group's first record, the warp's first rank
  if (n0 >= nb) return;  // whole warps
  rec += (size_t)b * N * DIGS_REC_F4;
  grec += (size_t)b * N * (DIGS_PARTIAL_F4 * 4);
  const float* gimg = gpix + (size_t)b * nv * nu;
  const unsigned key = n0 + lane < nb ? (unsigned)cost[(size_t)b * N + n0 + lane] : 0u;
  const int dead = __popc(__ballot_sync(0xffffffffu, key == 0u));
  unsigned lt = 0u, eq = 0xffffffffu;  // lanes with a smaller key; lanes whose key agrees so far
#pragma unroll
  for (int bit = 7; bit >= 0; --bit) {
    const unsigned one = (key >> bit) & 1u;
    const unsigned m = __ballot_sync(0xffffffffu, one);
    if (one) {
      lt |= eq & ~m;
      eq &= m;
    } else {
      eq &= ~m;
    }
  }
  order[warp][__popc(lt) + __popc(eq & ((1u << lane) - 1u))] = (uint8_t)lane;
  __syncwarp();
  const int of_rank = order[warp][lane];  // the record of rank `lane`
  const int i0 = max(0, (dead - r0) / kPer);  // the first round with a live record
  auto fetch = [&](int i) {  // one commit group per call and thread, empty or not
    if (i < WR) {
      const int rank = r0 + i * kPer + half, n = n0 + __shfl_sync(0xffffffffu, of_rank, rank);
      // not for a dead rank: its lane may lie past the projection's records
      if (rank >= dead && hl < DIGS_REC_F4) cp_async16(&sbuf[warp][i & 1][half][hl], rec + (unsigned)n * DIGS_REC_F4 + hl);
    }
    cp_async_commit();
  };
  fetch(i0);
  fetch(i0 + 1);
#pragma unroll 1
  for (int i = i0; i < WR; ++i) {
    cp_async_wait_but_one();  // this round's copies have landed (the next one's may still be in flight)
    __syncwarp();
    const int rank = r0 + i * kPer + half;
    const bool live = rank >= dead;
    float Sv[12];
#pragma unroll
    for (int q = 0; q < 12; ++q) Sv[q] = 0.f;
    if (live) {
      const Rec R0 = load_rec(sbuf[warp][i & 1][half]);
      const int x0 = R0.bx & 0xffff, x1 = R0.bx >> 16, y0 = R0.by & 0xffff, y1 = R0.by >> 16;
      const int w = x1 - x0 + 1, h = y1 - y0 + 1;
      for (int cx = 0; cx < w; cx += LPR) {  // boxes wider than LPR pixels: LPR-column slices
        const HalfLanes B = group_lanes<LPR>(min(LPR, w - cx), h, hl);
        if (B.active) {
          const int px = x0 + cx + B.c, py = y0 + B.r0;
          const float* gp = gimg + (unsigned)(py * nu + px);
          bwd_box_pixels(R0, B, h, (float)px - R0.xc, (float)py - R0.yc, gp, nu, c2, Sv);
        }
      }
    }
    const int n = n0 + __shfl_sync(0xffffffffu, of_rank, rank);
    group_reduce_store12<LPR>(Sv, grec + (unsigned)n * (DIGS_PARTIAL_F4 * 4), lane & 15, live);
    __syncwarp();  // every lane has read this buffer before it is refilled
    fetch(i + 2);
  }
  cp_async_wait_all();
}

// g = dL/dI * |X - s| for every pixel (the per-pixel factor of the line integral, applied once).
__global__ void __launch_bounds__(256) k_gpix(const float* __restrict__ grad_proj, const __grid_constant__ ViewsParam views,
                                              int nu, int nv, float* __restrict__ gpix) {
  const int b = blockIdx.y;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nu * nv) return;
  const size_t idx = (size_t)b * nu * nv + p;
  gpix[idx] = grad_proj[idx] * pixel_ray_length(views.v[b], (float)(p % nu), (float)(p / nu));
}

template <int TS>
static cudaError_t fwd_launch(const Workspace& ws, const ViewsParam& views, float c2, float* proj, const float* meas,
                              float* dldi, float inv_count, bool count, cudaStream_t st) {
  using C = FwdCfg<TS>;
  const unsigned grid = (unsigned)ws.T * (unsigned)ws.P * C::subs;
  float* lp = meas ? ws.loss_part : nullptr;
  if (count)
    k_raster_fwd<TS, true><<<grid, C::threads, 0, st>>>(ws.rec, ws.srid, ws.ranges, ws.order, views, ws.tiles_x, ws.T,
                                                        ws.nu, ws.nv, proj, meas, dldi, lp, c2, inv_count, ws.counters);
  else
    k_raster_fwd<TS, false><<<grid, C::threads, 0, st>>>(ws.rec, ws.srid, ws.ranges, ws.order, views, ws.tiles_x, ws.T,
                                                         ws.nu, ws.nv, proj, meas, dldi, lp, c2, inv_count, ws.counters);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_raster_fwd(const Workspace& ws, const ViewsParam& views, float c2, float* proj, const float* meas,
                              float* dldi, float inv_count, cudaStream_t st) {
  if (ws.P <= 0) return cudaSuccess;
  const bool count = meas == nullptr;  // pair statistics are gathered by plain projections only
#define DIGS_FWD(TS) return fwd_launch<TS>(ws, views, c2, proj, meas, dldi, inv_count, count, st)
  switch (ws.tile) {
    case 8: DIGS_FWD(8);
    case 16: DIGS_FWD(16);
    case 32: DIGS_FWD(32);
  }
#undef DIGS_FWD
  return cudaErrorInvalidValue;
}

cudaError_t launch_raster_bwd(const Workspace& ws, const ScanTable& sc, const ViewsParam& views, float c2, const float* grad_proj,
                              cudaStream_t st) {
  if (ws.P <= 0 || ws.n <= 0) return cudaSuccess;
  if (grad_proj) {  // else ws.dldi already holds dL/dI * |X - s| (written by the step's forward)
    dim3 g((ws.nu * ws.nv + 255) / 256, ws.P);
    k_gpix<<<g, 256, 0, st>>>(grad_proj, views, ws.nu, ws.nv, ws.dldi);
    note_launches(1);
  }
  ViewCounts counts;
  for (int b = 0; b < ws.P; ++b) counts.n[b] = sc.off[views.v[b].scan + 1] - sc.off[views.v[b].scan];
  const int G = (ws.n + 31) / 32;
#define DIGS_BWD(LPR, WR, W)                                                                        \
  k_raster_bwd<LPR, WR, W><<<dim3((G * (LPR / WR) + W - 1) / W, ws.P), 32 * W, 0, st>>>(            \
      ws.rec, ws.bcost, counts, ws.n, ws.nu, ws.nv, ws.dldi, c2, (float*)ws.grec)
  // A warp per group of 32 records from 8192 groups on, four below: 1000 groups 0.037 / 0.027 ms, 7300 0.117 / 0.111,
  // 12500 0.260 / 0.258, 50000 0.949 / 0.987, 400000 7.36 / 7.79.  One record per warp (32 lanes): always four
  // warps per group (1000 groups 0.043 / 0.031, 50000 1.28 / 1.16).  (Taken without the sum of g V, which adds 3 % to each.)
  if (ws.bwd_lanes == 32) DIGS_BWD(32, 8, 4);
  else if ((long long)G * ws.P > 8192) DIGS_BWD(16, 16, 1);
  else DIGS_BWD(16, 4, 4);
#undef DIGS_BWD
  note_launches(1);
  return cudaGetLastError();
}

// Sum of n partials in a fixed order: a block sums `chunk` consecutive values in one pass of its threads
// (strided), reduced by shuffles and through shared memory.  With more than one block, each block's sum
// replaces the first value of its own chunk (read only by that block) and one block then sums those.
__device__ __forceinline__ float block_sum_strided(const float* __restrict__ part, long long i0, long long i1,
                                                   long long stride) {
  __shared__ float red[32];
  float s = 0.f;
  for (long long i = i0 + (long long)threadIdx.x * stride; i < i1; i += (long long)blockDim.x * stride) s += part[i];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  float t = 0.f;
  if (threadIdx.x < 32) {
    t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    t = warp_sum(t);
  }
  return t;  // valid in thread 0
}

__global__ void __launch_bounds__(256) k_loss_partial(float* __restrict__ part, long long n, long long chunk) {
  const long long i0 = (long long)blockIdx.x * chunk, i1 = min(n, i0 + chunk);
  const float t = block_sum_strided(part, i0, i1, 1);
  __syncthreads();  // every thread has read its values before the chunk's first one is replaced
  if (threadIdx.x == 0) part[i0] = t;
}

__global__ void __launch_bounds__(1024) k_loss_reduce(const float* __restrict__ part, long long n, long long stride,
                                                      float* out, float scale) {
  const float t = block_sum_strided(part, 0, n, stride);
  if (threadIdx.x == 0) out[0] = t * scale;
}

cudaError_t launch_loss_reduce(float* part, int n, float* out, float scale, cudaStream_t st) {
  // part holds per-warp sums of squared residuals; out[0] = scale * their sum (part is overwritten)
  constexpr long long kChunk = 2048;
  if (n <= 4 * kChunk) {
    k_loss_reduce<<<1, 1024, 0, st>>>(part, n, 1, out, scale);
    note_launches(1);
  } else {
    const long long blocks = (n + kChunk - 1) / kChunk;
    k_loss_partial<<<(unsigned)blocks, 256, 0, st>>>(part, n, kChunk);
    k_loss_reduce<<<1, 1024, 0, st>>>(part, n, kChunk, out, scale);
    note_launches(2);
  }
  return cudaGetLastError();
}

}  // namespace digs
