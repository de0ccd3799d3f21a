// Evaluation volumes at one time point: the attenuation volume of the deformed cloud (Eq. 3 with the warp
// of Eq. 7-8), for image metrics, and the displacement field D(x, t) - x = sum_r w_r u_r(x) (Eq. 9-10),
// for motion metrics.
#include <math.h>

#include "digs_internal.h"
#include "ffd.cuh"
#include "setup.cuh"

namespace digs {
namespace {

struct GridC {
  int nx, ny, nz;
  float origin[3], spacing[3];
};

// Deformed mean and Jacobian of 32 Gaussians per CTA, then their voxels.
//
// Set-up: warp r of the CTA's four evaluates rank r of the FFD at each mean (lane = Gaussian); the ranks meet
// in shared memory, and one thread per Gaussian adds them in rank order (as the projector does) and forms its
// precision P = A^T A, voxel box (half extents cutoff sqrt(Sigma'_ii)) and density.  One warp per Gaussian
// doing all of it with identical lanes took longer than the voxels did.
// Sweep: a warp per Gaussian, a lane per (x, y) column of the box, 32 columns at a time: all lanes walk z
// together, so the x and y terms of E leave the loop and a voxel costs five FP32 operations, its test, and,
// where E <= cutoff^2, one exponential and one float atomic (several Gaussians share voxels).  Lanes over
// x and (y, z) rows instead left a third of them idle (boxes are about 11 wide): 0.41 ms against 0.22.
// The sums are bound by issue, then by the atomics.  No scratch memory: the records live in shared memory.
// 100k Gaussians into 128^3 voxels of 2 mm: 2.22 -> 0.22 ms.
constexpr int kVoxWarps = 4;

// 2^x by the SFU; SUB: with subnormal results, which cost instructions and come up beyond E = 2 ln 2^126 only.
template <bool SUB>
__device__ __forceinline__ float exp2_sfu(float x) {
  float y;
  if (SUB)
    asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  else
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// *p += v where E <= c2, without a branch around the one instruction.
__device__ __forceinline__ void add_within(float* p, float v, float E, float c2) {
  asm volatile("{\n .reg .pred q;\n setp.le.f32 q, %2, %3;\n @q red.global.add.f32 [%0], %1;\n}" ::"l"(p), "f"(v), "f"(E),
               "f"(c2)
               : "memory");
}

struct VoxRec {
  float mu[3], P[6], rho;
  int lo[3], ext[3];  // ext[0] = 0: nothing to add
};

// WIDE: cutoffs whose values reach below 2^-126 and grids of more than 2^24 layers (layer numbers no longer exact in
// FP32); otherwise z is counted in FP32, one conversion per voxel fewer.
constexpr float kWideC2 = 174.f;  // 2 ln 2^126 = 174.67, with room for rounding
constexpr int kWideLayers = 1 << 24;
template <int R, bool WIDE>
__global__ void __launch_bounds__(32 * kVoxWarps) k_voxelize(GaussPtrs g, LatticeC L, const float* __restrict__ phi,
                                                             const float* __restrict__ w, GridC G, float c2,
                                                             float* __restrict__ vol) {
  __shared__ float part[R][12][32];
  __shared__ VoxRec rec[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = blockIdx.x * 32 + lane;
  const bool valid = n < g.n;
  float mu0[3] = {0.f, 0.f, 0.f};
  if (valid) {
#pragma unroll
    for (int c = 0; c < 3; ++c) mu0[c] = g.mu0[3 * n + c];
    if (warp < R) {
      float U[1][3], dU[1][9];
      ffd_eval_point<1>(phi + (size_t)warp * L.nx * L.ny * L.nz * 3, L, mu0, U, dU);
#pragma unroll
      for (int c = 0; c < 3; ++c) part[warp][c][lane] = U[0][c];
#pragma unroll
      for (int c = 0; c < 9; ++c) part[warp][3 + c][lane] = dU[0][c];
    }
  }
  __syncthreads();
  if (warp == 0) {
    VoxRec r;
    r.ext[0] = 0;
    if (valid) {
      float K[9] = {1.f, 0.f, 0.f, 0.f, 1.f, 0.f, 0.f, 0.f, 1.f};
#pragma unroll
      for (int c = 0; c < 3; ++c) r.mu[c] = mu0[c];
#pragma unroll
      for (int k = 0; k < R; ++k) {
        const float wk = w[k];
#pragma unroll
        for (int c = 0; c < 3; ++c) r.mu[c] = fmaf(wk, part[k][c][lane], r.mu[c]);
#pragma unroll
        for (int c = 0; c < 9; ++c) K[c] = fmaf(wk, part[k][3 + c][lane], K[c]);
      }
      float s[3], q[4], Rm[9], Ki[9], A[9];
#pragma unroll
      for (int c = 0; c < 3; ++c) s[c] = g.scale[3 * n + c];
#pragma unroll
      for (int c = 0; c < 4; ++c) q[c] = g.quat[4 * n + c];
      const float qn = rsqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
#pragma unroll
      for (int c = 0; c < 4; ++c) q[c] *= qn;
      quat_to_R(q, Rm);
      if (inv3(K, Ki) > DIGS_FOLD_EPS) {  // folded Gaussians are dropped, as in the projector
        const float inv_s[3] = {1.f / s[0], 1.f / s[1], 1.f / s[2]};
        make_A(inv_s, Rm, Ki, A);
        const int ij[6][2] = {{0, 0}, {1, 1}, {2, 2}, {0, 1}, {0, 2}, {1, 2}};
#pragma unroll
        for (int e = 0; e < 6; ++e) {
          const int a = ij[e][0], b = ij[e][1];
          r.P[e] = A[a] * A[b] + A[3 + a] * A[3 + b] + A[6 + a] * A[6 + b];
        }
        r.rho = g.rho[n];
        const int dims[3] = {G.nx, G.ny, G.nz};
        bool some = true;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          float v = 0.f;  // Sigma'_ii, Sigma' = M M^T with M = K R S
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const float m = (K[3 * i] * Rm[k] + K[3 * i + 1] * Rm[3 + k] + K[3 * i + 2] * Rm[6 + k]) * s[k];
            v = fmaf(m, m, v);
          }
          const float half = sqrtf(c2 * v);
          r.lo[i] = max(0, (int)ceilf((r.mu[i] - half - G.origin[i]) / G.spacing[i]));
          r.ext[i] = min(dims[i] - 1, (int)floorf((r.mu[i] + half - G.origin[i]) / G.spacing[i])) - r.lo[i] + 1;
          some = some && r.ext[i] > 0;
        }
        if (!some) r.ext[0] = 0;
      }
    }
    rec[lane] = r;
  }
  __syncthreads();
#pragma unroll 1
  for (int q = warp; q < 32; q += kVoxWarps) {
    const VoxRec r = rec[q];
    const int ex = r.ext[0], ey = r.ext[1], ez = r.ext[2];
    if (ex == 0) continue;
    const float mx = r.mu[0], my = r.mu[1], mz = r.mu[2], rho = r.rho;
    const size_t plane = (size_t)G.ny * G.nx;
    const int sy = 32 / ex, sx = 32 - sy * ex;  // a step of 32 columns (x, y), x fastest
    int y = lane / ex, x = lane - y * ex;
    const unsigned steps = (unsigned)(((long long)ex * ey + 31) >> 5);
    for (unsigned c0 = 0; c0 < steps; ++c0) {
      if (y < ey) {
        const int i = r.lo[0] + x, j = r.lo[1] + y;
        const float dx = G.origin[0] + i * G.spacing[0] - mx;
        const float dy = G.origin[1] + j * G.spacing[1] - my;
        float* p = vol + ((size_t)r.lo[2] * G.ny + j) * G.nx + i;
        float k = (float)r.lo[2];
#pragma unroll 4
        for (int z = 0; z < ez; ++z, p += plane, k = WIDE ? (float)(r.lo[2] + z) : k + 1.f) {
          const float dz = G.origin[2] + k * G.spacing[2] - mz;
          const float E = r.P[0] * dx * dx + r.P[1] * dy * dy + r.P[2] * dz * dz +
                          2.f * (r.P[3] * dx * dy + r.P[4] * dx * dz + r.P[5] * dy * dz);
          add_within(p, rho * exp2_sfu<WIDE>(-0.5f * E * DIGS_LOG2E), E, c2);
        }
      }
      x += sx;
      y += sy;
      if (x >= ex) {
        x -= ex;
        ++y;
      }
    }
  }
}

template <int R>
__global__ void __launch_bounds__(128) k_dvf(LatticeC L, const float* __restrict__ phi, const float* __restrict__ w,
                                             GridC G, float* __restrict__ out) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nv = (long long)G.nx * G.ny * G.nz;
  if (v >= nv) return;
  const int i = (int)(v % G.nx), j = (int)((v / G.nx) % G.ny), k = (int)(v / ((long long)G.nx * G.ny));
  const float x[3] = {G.origin[0] + i * G.spacing[0], G.origin[1] + j * G.spacing[1], G.origin[2] + k * G.spacing[2]};
  float U[R][3], dU[R][9];
  ffd_eval_point<R>(phi, L, x, U, dU);
  float d[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float wr = w[r];
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = fmaf(wr, U[r][c], d[c]);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) out[3 * v + c] = d[c];
}

// The displacement field row by row: the field is separable, so on a plane of voxels (fixed z) the four lattice
// layers and the ranks collapse once per node column,
//   T[j][i] = sum_n3 B_n3(z) sum_r w_r phi_r[f_z + n3][j][i],
// along an x row of it the four node rows collapse once, S[i] = sum_m B_m(y) T[f_y + m][i], and a voxel is four
// taps of S.  A CTA takes xs voxels of ys consecutive rows of one plane: its threads form T and S for the nodes
// those voxels reach, then write the rows element by element (thread = (voxel, component): contiguous stores).
// xs and ys are as large as the node tables allow (kDvfNodesX, kDvfNodesY).  One thread per voxel reading its
// 64 nodes was bound by those loads: 128^3 voxels of 2 mm, R = 3, 16 mm lattice: 185 -> 15.5 us.
constexpr int kDvfX = 128, kDvfRows = 16, kDvfNodesX = 64, kDvfNodesY = 24;

template <int R>
__global__ void __launch_bounds__(3 * kDvfX) k_dvf_rows(LatticeC L, const float* __restrict__ phi,
                                                        const float* __restrict__ w, GridC G, int xs, int ys,
                                                        float* __restrict__ out) {
  __shared__ float T[kDvfNodesY][kDvfNodesX * 3];
  __shared__ float S[kDvfRows][kDvfNodesX * 3];
  __shared__ float Bx[4][kDvfX], By[4][kDvfRows];
  __shared__ int fx[kDvfX], fy[kDvfRows];
  const int i0 = blockIdx.x * xs, nx = min(xs, G.nx - i0);
  const int j0 = blockIdx.y * ys, ny = min(ys, G.ny - j0);
  auto cell = [&](int a, int i, float& t) {  // first of the four nodes along axis a at voxel index i
    const float p = (G.origin[a] + i * G.spacing[a] - L.origin[a]) * L.inv_h[a];
    const float fl = floorf(p);
    t = p - fl;
    return (int)fl - 1;
  };
  float t;
  const int bx = cell(0, i0, t), wx = min(cell(0, i0 + nx - 1, t) + 4 - bx, kDvfNodesX);
  const int by = cell(1, j0, t), wy = min(cell(1, j0 + ny - 1, t) + 4 - by, kDvfNodesY);
  const int tid = threadIdx.x;
  if (tid < nx) {
    float B[4];
    fx[tid] = (cell(0, i0 + tid, t) - bx) * 3;
    bspline4(t, B);
#pragma unroll
    for (int l = 0; l < 4; ++l) Bx[l][tid] = B[l];
  } else if (tid >= kDvfX && tid - kDvfX < ny) {
    const int q = tid - kDvfX;
    float B[4];
    fy[q] = cell(1, j0 + q, t) - by;
    bspline4(t, B);
#pragma unroll
    for (int l = 0; l < 4; ++l) By[l][q] = B[l];
  }
  const size_t rank_stride = (size_t)L.nx * L.ny * L.nz * 3;
  for (int z = blockIdx.z; z < G.nz; z += gridDim.z) {
    float Bz[4];
    const int fz = cell(2, z, t);
    bspline4(t, Bz);
    for (int e = tid; e < wy * wx * 3; e += blockDim.x) {
      const int q = e / (wx * 3), ic = e - q * (wx * 3), i = bx + ic / 3, j = by + q;
      float s = 0.f;
      if (i >= 0 && i < L.nx && j >= 0 && j < L.ny) {
        const float* p = phi + ((size_t)j * L.nx + i) * 3 + ic % 3;
#pragma unroll
        for (int n3 = 0; n3 < 4; ++n3) {
          const int k = fz + n3;
          if (k < 0 || k >= L.nz) continue;
          const float* d = p + (size_t)k * L.ny * L.nx * 3;
          float v = 0.f;
#pragma unroll
          for (int r = 0; r < R; ++r) v = fmaf(w[r], __ldg(d + r * rank_stride), v);
          s = fmaf(Bz[n3], v, s);
        }
      }
      T[q][ic] = s;
    }
    __syncthreads();
    for (int e = tid; e < ny * wx * 3; e += blockDim.x) {
      const int q = e / (wx * 3), ic = e - q * (wx * 3), f = fy[q];
      S[q][ic] = fmaf(By[0][q], T[f][ic], fmaf(By[1][q], T[f + 1][ic], fmaf(By[2][q], T[f + 2][ic], By[3][q] * T[f + 3][ic])));
    }
    __syncthreads();
    if (tid < nx * 3) {
      const int x = tid / 3, at = fx[x] + tid - 3 * x;
      const float b0 = Bx[0][x], b1 = Bx[1][x], b2 = Bx[2][x], b3 = Bx[3][x];
      float* o = out + (((size_t)z * G.ny + j0) * G.nx + i0) * 3 + tid;
      for (int q = 0; q < ny; ++q) {
        const float* s = &S[q][at];
        o[(size_t)q * G.nx * 3] = fmaf(b0, s[0], fmaf(b1, s[3], fmaf(b2, s[6], b3 * s[9])));
      }
    }
    __syncthreads();  // T and S are free for the next plane
  }
}

// Voxels of a row (*xs) and rows (*ys) per CTA of k_dvf_rows, or false where k_dvf serves: voxels more than 10^6
// lattice cells from the origins (nearer, a cell number's FP32 error is below 1/8, so n voxels of d cells reach
// at most (n - 1) d + 6 nodes), and grids so coarse that a CTA would write fewer than 16 voxels of a row.
bool dvf_by_rows(const GridC& G, const LatticeC& L, int* xs, int* ys) {
  const int dims[3] = {G.nx, G.ny, G.nz};
  for (int a = 0; a < 3; ++a) {
    const double p0 = (double)G.origin[a] * L.inv_h[a], p1 = p0 + (double)(dims[a] - 1) * G.spacing[a] * L.inv_h[a];
    if (!(fabs(p0) < 1e6) || !(fabs(p1) < 1e6) || !(fabs((double)L.origin[a] * L.inv_h[a]) < 1e6)) return false;
  }
  const double dx = (double)G.spacing[0] * L.inv_h[0], dy = (double)G.spacing[1] * L.inv_h[1];
  const double mx = (kDvfNodesX - 6) / dx + 1, my = (kDvfNodesY - 6) / dy + 1;
  *xs = mx < kDvfX ? (int)mx : kDvfX;
  *ys = my < kDvfRows ? (int)my : kDvfRows;
  return *xs >= 16 && (G.ny + *ys - 1) / *ys <= 65535;
}

bool make_grid(const DigsGrid* g, GridC& G) {
  if (!g || g->nx < 1 || g->ny < 1 || g->nz < 1) return false;
  G.nx = g->nx; G.ny = g->ny; G.nz = g->nz;
  for (int a = 0; a < 3; ++a) {
    if (!(g->spacing[a] > 0.f) || !isfinite(g->spacing[a]) || !isfinite(g->origin[a])) return false;
    G.origin[a] = g->origin[a];
    G.spacing[a] = g->spacing[a];
  }
  return true;
}

bool make_lat(const DigsLattice* lat, LatticeC& L) {
  if (!lat || lat->R < 1 || lat->R > DIGS_MAX_R || lat->nx < 1 || lat->ny < 1 || lat->nz < 1) return false;
  for (int a = 0; a < 3; ++a) {
    if (!(lat->spacing[a] > 0.f) || !isfinite(lat->spacing[a]) || !isfinite(lat->origin[a])) return false;
    L.origin[a] = lat->origin[a];
    L.inv_h[a] = 1.f / lat->spacing[a];
  }
  L.nx = lat->nx; L.ny = lat->ny; L.nz = lat->nz; L.R = lat->R;
  return true;
}

}  // namespace
}  // namespace digs

using namespace digs;

extern "C" {

digs_status digs_voxelize(const DigsGaussians* g, const DigsLattice* lat, const float* phi, const float* w,
                          const DigsGrid* grid, const DigsOpts* opts, float* vol, void* stream) {
  LatticeC L;
  GridC G;
  if (!g || !phi || !w || !vol || g->n < 0 || !make_lat(lat, L) || !make_grid(grid, G)) return DIGS_ERR_ARG;
  if (g->n > 0 && (!g->mu0 || !g->scale || !g->quat || !g->rho)) return DIGS_ERR_ARG;
  const float cut = opts ? opts->cutoff : 3.5f;
  if (!(cut >= 0.f) || !isfinite(cut)) return DIGS_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemsetAsync(vol, 0, (size_t)G.nx * G.ny * G.nz * sizeof(float), st) != cudaSuccess) return DIGS_ERR_CUDA;
  if (g->n == 0) return DIGS_OK;
  GaussPtrs gp{g->mu0, g->scale, g->quat, g->rho, g->n};
  const unsigned blocks = (unsigned)((g->n + 31LL) / 32);
  const bool wide = cut * cut > kWideC2 || G.nz > kWideLayers;
#define DIGS_VOX(RR)                                                                              \
  if (wide) k_voxelize<RR, true><<<blocks, 32 * kVoxWarps, 0, st>>>(gp, L, phi, w, G, cut * cut, vol); \
  else k_voxelize<RR, false><<<blocks, 32 * kVoxWarps, 0, st>>>(gp, L, phi, w, G, cut * cut, vol)
  switch (L.R) {
    case 1: DIGS_VOX(1); break;
    case 2: DIGS_VOX(2); break;
    case 3: DIGS_VOX(3); break;
    case 4: DIGS_VOX(4); break;
  }
#undef DIGS_VOX
  note_launches(1);
  return cudaGetLastError() == cudaSuccess ? DIGS_OK : DIGS_ERR_CUDA;
}

digs_status digs_dvf(const DigsLattice* lat, const float* phi, const float* w, const DigsGrid* grid, float* dvf,
                     void* stream) {
  LatticeC L;
  GridC G;
  if (!phi || !w || !dvf || !make_lat(lat, L) || !make_grid(grid, G)) return DIGS_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const long long nv = (long long)G.nx * G.ny * G.nz;
  const unsigned blocks = (unsigned)((nv + 127) / 128);
  int xs = 1, ys = 1;
  const bool by_rows = dvf_by_rows(G, L, &xs, &ys);
  const dim3 rows((unsigned)((G.nx + xs - 1) / xs), (unsigned)((G.ny + ys - 1) / ys), (unsigned)(G.nz < 65535 ? G.nz : 65535));
#define DIGS_DVF(RR)                                                                      \
  if (by_rows) k_dvf_rows<RR><<<rows, 3 * kDvfX, 0, st>>>(L, phi, w, G, xs, ys, dvf);    \
  else k_dvf<RR><<<blocks, 128, 0, st>>>(L, phi, w, G, dvf)
  switch (L.R) {
    case 1: DIGS_DVF(1); break;
    case 2: DIGS_DVF(2); break;
    case 3: DIGS_DVF(3); break;
    case 4: DIGS_DVF(4); break;
  }
#undef DIGS_DVF
  note_launches(1);
  return cudaGetLastError() == cudaSuccess ? DIGS_OK : DIGS_ERR_CUDA;
}

}  // extern "C"
