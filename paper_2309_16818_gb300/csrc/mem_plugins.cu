// Post-processing plugins that read map layers already on the GPU and produce
// new layers (Sec. III-D): surface normals of the elevation layer (Table I
// "normal calculation") and the PCA layer of a feature layer (the plugin of
// the post-processing figure that turns feature layers into a PCA layer).
//
// Normals: one thread per logical cell; slopes from central differences of
// the valid neighbours (one-sided where one is missing), as fixed float32
// sequences, so the result does not depend on the launch.
//
// PCA: per map, over the cells where the layer is observed,
//   1. mean: blocks take fixed cell ranges, warps take rows with their lanes over
//      the channels; the block sums (float32) are added in a fixed order in float64;
//   2. covariance of (f - mean): blocks take fixed cell ranges and stage centred
//      rows in shared memory; each thread accumulates an 8 x 8 tile of the upper
//      triangle of the C x C matrix with float32 FMAs; the partial matrices are
//      added in a fixed order in float64;
//   3. eigenvectors: one block runs cyclic Jacobi sweeps (round-robin pairs,
//      C/2 disjoint rotations at a time) in float32 shared memory until the
//      off-diagonal mass is at the float32 rounding level of the matrix
//      (at most 20 sweeps), then sorts the
//      eigenvalues and signs each kept vector so that its largest-magnitude
//      component is positive;
//   4. projection of every observed cell on the kept vectors, four lanes a cell.
#include <math.h>

#include <algorithm>
#include <vector>

#include "mem_host.h"

namespace memk {

// ---------------------------------------------------------------------------
// normals

__device__ __forceinline__ bool axis_slope(float hm, bool va, float ha, bool vb, float hb, float res, float& g) {
  if (va && vb) {
    g = __fdiv_rn(__fsub_rn(hb, ha), __fmul_rn(2.0f, res));
    return true;
  }
  if (vb) {
    g = __fdiv_rn(__fsub_rn(hb, hm), res);
    return true;
  }
  if (va) {
    g = __fdiv_rn(__fsub_rn(hm, ha), res);
    return true;
  }
  return false;
}

__global__ void __launch_bounds__(256) k_normals(MapDev md, int map, int rx, int ry, float* __restrict__ out,
                                                 uint8_t* __restrict__ ok) {
  const int W = md.W;
  const int ix = blockIdx.x * 16 + threadIdx.x, iy = blockIdx.y * 16 + threadIdx.y;
  if (ix >= W || iy >= W) return;
  const u32 base = (u32)map * md.W2;
  auto g_of = [&](int x, int y) {
    int px = x + rx;
    if (px >= W) px -= W;
    int py = y + ry;
    if (py >= W) py -= W;
    return base + (u32)py * (u32)W + (u32)px;
  };
  const int64_t j = (int64_t)iy * W + ix;
  float n0 = 0.f, n1 = 0.f, n2 = 0.f;
  bool good = false;
  const u32 g = g_of(ix, iy);
  if (md.flags[g] & kFlagValid) {
    const float hm = md.h[g];
    const bool vl = ix > 0 && (md.flags[g_of(ix - 1, iy)] & kFlagValid);
    const bool vr = ix + 1 < W && (md.flags[g_of(ix + 1, iy)] & kFlagValid);
    const bool vd = iy > 0 && (md.flags[g_of(ix, iy - 1)] & kFlagValid);
    const bool vu = iy + 1 < W && (md.flags[g_of(ix, iy + 1)] & kFlagValid);
    float gx, gy;
    if (axis_slope(hm, vl, vl ? md.h[g_of(ix - 1, iy)] : 0.f, vr, vr ? md.h[g_of(ix + 1, iy)] : 0.f, md.res, gx) &&
        axis_slope(hm, vd, vd ? md.h[g_of(ix, iy - 1)] : 0.f, vu, vu ? md.h[g_of(ix, iy + 1)] : 0.f, md.res, gy)) {
      const float q = __fmaf_rn(gx, gx, __fmaf_rn(gy, gy, 1.0f));
      const float inv = __fdiv_rn(1.0f, __fsqrt_rn(q));
      n0 = __fmul_rn(-gx, inv);
      n1 = __fmul_rn(-gy, inv);
      n2 = inv;
      good = true;
    }
  }
  out[3 * j] = n0;
  out[3 * j + 1] = n1;
  out[3 * j + 2] = n2;
  if (ok) ok[j] = good ? 1 : 0;
}

// ---------------------------------------------------------------------------
// PCA

constexpr int kPcaMaxC = 128;      // channels of a PCA input layer
constexpr int kPcaRows = 64;       // centred rows staged at a time by the covariance blocks
constexpr int kPcaBlocks = 2;      // blocks per SM of the mean and covariance kernels
constexpr int kPcaMaxComp = 8;

struct PcaArgs {
  int map, layer, C, n_comp, blocks;
  const void* data;  // the layer's values [cells][S]
  int S, dtype;
  u32 obs_bit;
  double* mean_part;  // [blocks][C + 1] (sums, then the count)
  float* cov_part;    // [blocks][64][tiles] (element of the tile, tile)
  float* mean;        // [C]
  float* cov;         // [C][C]
  float* vecs;        // [n_comp][C]
  float* vals;        // [n_comp]
  float* proj;        // [W2][n_comp] (logical order)
  float* info;        // optional: [n_comp] values, [n_comp][C] vectors, [C] mean
};

__device__ __forceinline__ float layer_val(const void* data, int dtype, int64_t off) {
  if (dtype == MEM_BF16) return __bfloat162float(((const __nv_bfloat16*)data)[off]);
  if (dtype == MEM_F16) return __half2float(((const __half*)data)[off]);
  return ((const float*)data)[off];
}

// four consecutive values of a row, 16-byte (float32) or 8-byte (16-bit) aligned
__device__ __forceinline__ float4 layer_val4(const void* data, int dtype, int64_t off) {
  if (dtype == MEM_F32) return *reinterpret_cast<const float4*>((const float*)data + off);
  const uint2 q = *reinterpret_cast<const uint2*>((const uint16_t*)data + off);
  const float2 a = dtype == MEM_BF16 ? __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x))
                                     : __half22float2(*reinterpret_cast<const __half2*>(&q.x));
  const float2 b = dtype == MEM_BF16 ? __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y))
                                     : __half22float2(*reinterpret_cast<const __half2*>(&q.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// the fixed cell range of block b of `blocks` over W2 cells
__device__ __forceinline__ void block_range(u32 W2, int b, int blocks, u32& c0, u32& c1) {
  c0 = (u32)(((uint64_t)W2 * b) / blocks);
  c1 = (u32)(((uint64_t)W2 * (b + 1)) / blocks);
}

// A warp takes 32 cells' flags at a time and adds the observed rows, kMeanU of them
// in flight, its lanes over the channels (lane, lane + 32, ...): whole lines, where a
// thread per (cell, channel) with four cells in flight was bound by its chain of
// loads (64 float32 channels of 500 x 500 cells: 63 -> 16 us).
constexpr int kMeanU = 8;

__global__ void __launch_bounds__(256) k_pca_mean(MapDev md, PcaArgs a) {
  constexpr int T = kPcaMaxC / 32;
  __shared__ float part[8][kPcaMaxC + 1];
  u32 c0, c1;
  block_range(md.W2, blockIdx.x, a.blocks, c0, c1);
  const u32 base = (u32)a.map * md.W2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float sum[T];
#pragma unroll
  for (int t = 0; t < T; ++t) sum[t] = 0.f;
  u32 cnt = 0;
  for (u32 p0 = c0 + warp * 32; p0 < c1; p0 += 256) {
    u32 m = __ballot_sync(0xffffffffu, p0 + lane < c1 && (md.flags[base + p0 + lane] & a.obs_bit));
    cnt += __popc(m);
    while (m) {
      float v[kMeanU][T];
#pragma unroll
      for (int u = 0; u < kMeanU; ++u) {
        const int r = __ffs(m) - 1;  // -1 when none is left
        m &= m - 1;
#pragma unroll
        for (int t = 0; t < T; ++t) {
          const int c = lane + 32 * t;
          v[u][t] = (r >= 0 && c < a.C) ? layer_val(a.data, a.dtype, (int64_t)(base + p0 + r) * a.S + c) : 0.f;
        }
      }
#pragma unroll
      for (int u = 0; u < kMeanU; ++u)
#pragma unroll
        for (int t = 0; t < T; ++t) sum[t] += v[u][t];
    }
  }
#pragma unroll
  for (int t = 0; t < T; ++t)
    if (lane + 32 * t < a.C) part[warp][lane + 32 * t] = sum[t];
  if (lane == 0) part[warp][a.C] = (float)cnt;  // below 2^24 for every block of a map of 2^28 cells
  __syncthreads();
  for (int c = threadIdx.x; c <= a.C; c += 256) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += (double)part[w][c];
    a.mean_part[(int64_t)blockIdx.x * (a.C + 1) + c] = t;
  }
}

// The blocks' sums in a fixed order: 1024 / 32 groups of blocks per column side by
// side, then the groups (one thread per column walking every block took 135 us).
__global__ void __launch_bounds__(1024) k_pca_mean_final(PcaArgs a) {
  __shared__ double part[32][33];
  __shared__ double tot[kPcaMaxC + 1];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  for (int cb = 0; cb <= a.C; cb += 32) {
    const int c = cb + lane;
    double s = 0.0;
    if (c <= a.C)
#pragma unroll 8
      for (int b = grp; b < a.blocks; b += 32) s += a.mean_part[(int64_t)b * (a.C + 1) + c];
    part[grp][lane] = s;
    __syncthreads();
    if (grp == 0 && c <= a.C) {
      double t = 0.0;
      for (int g = 0; g < 32; ++g) t += part[g][lane];
      tot[c] = t;
      a.mean_part[(int64_t)a.blocks * (a.C + 1) + c] = t;  // totals after the partials
    }
    __syncthreads();
  }
  const double n = tot[a.C];
  for (int c = threadIdx.x; c < a.C; c += blockDim.x) a.mean[c] = n > 0.0 ? (float)(tot[c] / n) : 0.f;
}

// Partial covariance sums of one block's cells. The C x C matrix is cut into 8 x 8
// tiles; the tiles on and above the diagonal, nt (nt + 1) / 2 with nt = ceil(C / 8),
// are the matrix. A thread owns one of them for every `groups`-th staged row
// (groups = the times the tiles fit 256 threads, at most 8): 64 FMAs for four
// 16-byte reads of a row, half the products of the full matrix. FP32 FMAs bound it
// (64 channels of 175k cells: 0.4 G FMAs); 100 -> 48 us against 4 x 4 tiles of the
// full matrix fed by scalar reads. Rows are staged four channels per thread and load,
// kCovU loads in flight (scalar staging loads took 111 us). A group's sums are added to the others' in group
// order.
constexpr int kCovU = 4;

__global__ void __launch_bounds__(256) k_pca_cov(MapDev md, PcaArgs a, int nt, int tiles, int groups) {
  extern __shared__ __align__(16) float xs[];  // [kPcaRows][ld], then reused for the groups' sums [tiles][64]
  const int Cp = nt * 8, ld = Cp + 4;
  __shared__ u32 wcnt[8];
  __shared__ u32 list[256];
  __shared__ __align__(16) float sm[kPcaMaxC];
  if (threadIdx.x < a.C) sm[threadIdx.x] = a.mean[threadIdx.x];
  for (int e = threadIdx.x; e < kPcaRows * ld; e += 256) xs[e] = 0.f;  // the columns past C stay 0
  u32 c0, c1;
  block_range(md.W2, blockIdx.x, a.blocks, c0, c1);
  const u32 base = (u32)a.map * md.W2;
  const int grp = threadIdx.x / tiles, tile = threadIdx.x - grp * tiles;
  const bool on = grp < groups;
  int ti = 0, tj = tile;  // row-major over the upper triangle
  while (tj >= nt - ti) {
    tj -= nt - ti;
    ++ti;
  }
  tj += ti;
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[i][k] = 0.f;
  for (u32 p0 = c0; p0 < c1; p0 += 256) {
    // list the observed cells of the next 256 (in cell order), then stage them kPcaRows at a time
    const u32 p = p0 + threadIdx.x;
    const bool obs = p < c1 && (md.flags[base + p] & a.obs_bit);
    const u32 bal = __ballot_sync(0xffffffffu, obs);
    if ((threadIdx.x & 31) == 0) wcnt[threadIdx.x >> 5] = __popc(bal);
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < 8; ++w) {
      before += w < (int)(threadIdx.x >> 5) ? (int)wcnt[w] : 0;
      total += (int)wcnt[w];
    }
    if (obs) list[before + __popc(bal & ((1u << (threadIdx.x & 31)) - 1u))] = p;
    __syncthreads();
    for (int r0 = 0; r0 < total; r0 += kPcaRows) {
      const int nr = min(kPcaRows, total - r0);
      if ((a.C & 3) == 0) {  // rows (S = C values) then start on 16-byte (8-byte) boundaries
        const int C4 = a.C >> 2;
        for (int e0 = threadIdx.x; e0 < nr * C4; e0 += 256 * kCovU) {
          float4 v[kCovU];
#pragma unroll
          for (int u = 0; u < kCovU; ++u) {
            const int e = e0 + u * 256, r = e / C4;
            if (e < nr * C4) v[u] = layer_val4(a.data, a.dtype, (int64_t)(base + list[r0 + r]) * a.S + 4 * (e - r * C4));
          }
#pragma unroll
          for (int u = 0; u < kCovU; ++u) {
            const int e = e0 + u * 256, r = e / C4, c = 4 * (e - r * C4);
            if (e >= nr * C4) continue;
            const float4 m = *reinterpret_cast<const float4*>(sm + c);
            *reinterpret_cast<float4*>(xs + r * ld + c) = make_float4(
                __fsub_rn(v[u].x, m.x), __fsub_rn(v[u].y, m.y), __fsub_rn(v[u].z, m.z), __fsub_rn(v[u].w, m.w));
          }
        }
      } else {
#pragma unroll 4
        for (int e = threadIdx.x; e < nr * a.C; e += 256) {
          const int r = e / a.C, c = e - r * a.C;
          xs[r * ld + c] = __fsub_rn(layer_val(a.data, a.dtype, (int64_t)(base + list[r0 + r]) * a.S + c), sm[c]);
        }
      }
      __syncthreads();
      if (on)
        for (int r = grp; r < nr; r += groups) {
          const float4* xa = reinterpret_cast<const float4*>(xs + r * ld + ti * 8);
          const float4* xb = reinterpret_cast<const float4*>(xs + r * ld + tj * 8);
          const float4 a0 = xa[0], a1 = xa[1], b0 = xb[0], b1 = xb[1];
          const float va[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
          const float vb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[i][k] = __fmaf_rn(va[i], vb[k], acc[i][k]);
        }
      __syncthreads();
    }
  }
  for (int g = 0; g < groups; ++g) {  // the groups' sums in group order
    if (on && grp == g) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          float* d = xs + (i * 8 + k) * tiles + tile;  // consecutive threads, consecutive words
          *d = g ? *d + acc[i][k] : acc[i][k];
        }
    }
    __syncthreads();
  }
  float* out = a.cov_part + (int64_t)blockIdx.x * tiles * 64;
  for (int e = threadIdx.x; e < tiles * 64; e += 256) out[e] = xs[e];
}

// The partial matrices in a fixed order, in float64: 8 groups of blocks per element
// side by side, then the groups (one thread per element walking every block: 106 -> 12 us).
__global__ void __launch_bounds__(256) k_pca_cov_final(PcaArgs a, int nt, int tiles) {
  __shared__ double part[8][33];
  const double n = a.mean_part[(int64_t)a.blocks * (a.C + 1) + a.C];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (e < tiles * 64)
#pragma unroll 8
    for (int b = grp; b < a.blocks; b += 8) s += (double)a.cov_part[(int64_t)b * tiles * 64 + e];
  part[grp][lane] = s;
  __syncthreads();
  if (grp != 0 || e >= tiles * 64) return;
  double t = 0.0;
  for (int g = 0; g < 8; ++g) t += part[g][lane];
  const float v = n > 0.0 ? (float)(t / n) : 0.f;
  const int ik = e / tiles, tile = e - ik * tiles;
  int ti = 0, tj = tile;
  while (tj >= nt - ti) {
    tj -= nt - ti;
    ++ti;
  }
  tj += ti;
  const int row = ti * 8 + ik / 8, col = tj * 8 + ik % 8;
  if (row < a.C && col < a.C) {
    a.cov[row * a.C + col] = v;
    a.cov[col * a.C + row] = v;
  }
}

// Cyclic Jacobi with round-robin pairs on the C x C covariance (C padded to an
// even n with a zero row and column), in shared memory; one block of 1024.
// A step rotates n / 2 disjoint pairs: A <- J^T A J falls apart into the 2 x 2
// blocks (pair, pair), so a thread applies both sides to its block at once; then
// warp 0 finds the next step's angles while the others bring V up to date (two
// barriers a step; the pairs of step t are computed from t; a warp per row of
// blocks, so no divisions). Bound by the latency of its steps; with the sides one
// after the other, V with them and the round-robin order moved along by one
// thread (four barriers a step) 64 channels took 609 us, now 314 us and 34 us for
// the corrections of three vectors (5e-8 from the float64 vectors, 3e-6 to 1e-5 without).
// the angles of step `step`: round-robin, position 0 holds row 0, position i >= 1 row
// 1 + (i - 1 - step) mod (n - 1); pair m: positions m and n - 1 - m. By one warp.
__device__ __forceinline__ void jacobi_angles(const float* A, int ld, int n, int step, float4* rot) {
  for (int m = threadIdx.x & 31; m < n / 2; m += 32) {
    int i1 = m - 1 - step, i2 = n - 2 - m - step;
    if (i1 < 0) i1 += n - 1;
    if (i2 < 0) i2 += n - 1;
    int p = m == 0 ? 0 : 1 + i1, q = 1 + i2;
    if (p > q) {
      const int t = p;
      p = q;
      q = t;
    }
    const float apq = A[p * ld + q], app = A[p * ld + p], aqq = A[q * ld + q];
    float c = 1.f, s = 0.f;
    if (apq != 0.f) {
      const float tau = (aqq - app) / (2.f * apq);
      const float t = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
      c = 1.f / sqrtf(1.f + t * t);
      s = t * c;
    }
    rot[m] = make_float4(c, s, __int_as_float(p), __int_as_float(q));
  }
}

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Kept eigenvector k (column `sel` of V) by the whole block: the rotations leave it with
// float32 rounding of several hundred steps, a few 1e-6; one first-order correction with the
// covariance itself (its product with v in float64), v += sum_j (u_j . r) / (lambda - lambda_j) u_j with the
// residual r = A v - lambda v, squares that error. Directions whose eigenvalue is as good as
// equal (a coefficient of 1 % or more) are left alone. Then normalised, signed by its
// largest-magnitude component (the smaller index first on ties) and written, with its
// Rayleigh quotient as the eigenvalue.
__device__ void refine_vector(const float* A, const float* V, int ld, int n, const PcaArgs& a, int sel, int k) {
  __shared__ double s_v[kPcaMaxC], s_r[kPcaMaxC], s_lam, s_scale;
  __shared__ float s_f[kPcaMaxC], s_c[kPcaMaxC];  // the residual and the coefficients: float32 carries a correction
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, C = a.C;
  for (int i = threadIdx.x; i < C; i += blockDim.x) s_v[i] = (double)V[i * ld + sel];
  __syncthreads();
  for (int i = warp; i < C; i += 32) {  // A v
    double y = 0.0;
    for (int j = lane; j < C; j += 32) y = fma((double)a.cov[i * C + j], s_v[j], y);
    y = warp_sum_d(y);
    if (lane == 0) s_r[i] = y;
  }
  __syncthreads();
  if (warp == 0) {
    double vy = 0.0, vv = 0.0;
    for (int i = lane; i < C; i += 32) {
      vy = fma(s_v[i], s_r[i], vy);
      vv = fma(s_v[i], s_v[i], vv);
    }
    vy = warp_sum_d(vy);
    vv = warp_sum_d(vv);
    if (lane == 0) s_lam = vv > 0.0 ? vy / vv : 0.0;
  }
  __syncthreads();
  const double lam = s_lam;
  for (int i = threadIdx.x; i < C; i += blockDim.x) s_f[i] = (float)(s_r[i] - lam * s_v[i]);
  __syncthreads();
  for (int j = warp; j < n; j += 32) {  // u_j . r
    float d = 0.f;
    for (int i = lane; i < C; i += 32) d = fmaf(V[i * ld + j], s_f[i], d);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if (lane == 0) {
      const float gap = (float)lam - A[j * (ld + 1)];
      s_c[j] = j != sel && fabsf(d) < 0.01f * fabsf(gap) ? d / gap : 0.f;
    }
  }
  __syncthreads();
  for (int i = warp; i < C; i += 32) {
    float x = 0.f;
    for (int j = lane; j < n; j += 32) x = fmaf(s_c[j], V[i * ld + j], x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) s_r[i] = s_v[i] + (double)x;
  }
  __syncthreads();
  if (warp == 0) {
    double vv = 0.0, mv = -1.0;
    int mi = C;
    for (int i = lane; i < C; i += 32) {
      vv = fma(s_r[i], s_r[i], vv);
      const double v = (double)(float)fabs(s_r[i]);
      if (v > mv) {
        mv = v;
        mi = i;
      }
    }
    vv = warp_sum_d(vv);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, mv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
      if (ov > mv || (ov == mv && oi < mi)) {
        mv = ov;
        mi = oi;
      }
    }
    if (lane == 0) {
      const double inv = vv > 0.0 ? 1.0 / sqrt(vv) : 1.0;
      s_scale = mi < C && s_r[mi] < 0.0 ? -inv : inv;
      a.vals[k] = (float)lam;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < C; i += blockDim.x) a.vecs[k * C + i] = (float)(s_r[i] * s_scale);
  __syncthreads();
}

__global__ void __launch_bounds__(1024) k_pca_eig(PcaArgs a) {
  extern __shared__ float sm[];
  const int C = a.C, n = (C + 1) & ~1;
  float* A = sm;                 // [n][n + 1]
  float* V = A + n * (n + 1);    // [n][n + 1]
  float4* rot = reinterpret_cast<float4*>(((uintptr_t)(V + n * (n + 1)) + 15) & ~(uintptr_t)15);  // [2][n / 2] cosine, sine, rows p < q
  __shared__ float s_off, s_tot;
  const int ld = n + 1, h = n / 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, k = e - i * n;
    A[i * ld + k] = (i < C && k < C) ? a.cov[i * C + k] : 0.f;
    V[i * ld + k] = i == k ? 1.f : 0.f;
  }
  __syncthreads();
  __shared__ float red[2][32];
  __shared__ int s_sel[kPcaMaxComp];
  // converged when the off-diagonal mass is at the float32 rounding level of the matrix
  const float conv = (4.f * n * 5.96e-8f) * (4.f * n * 5.96e-8f);
  for (int sweep = 0; sweep < 20; ++sweep) {
    float off = 0.f, tot = 0.f;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
      const int i = e / n, k = e - i * n;
      const float v = A[i * ld + k] * A[i * ld + k];
      tot += v;
      if (i != k) off += v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if ((threadIdx.x & 31) == 0) {
      red[0][threadIdx.x >> 5] = off;
      red[1][threadIdx.x >> 5] = tot;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      float o2 = 0.f, t2 = 0.f;
      for (int w = 0; w < 32; ++w) {
        o2 += red[0][w];
        t2 += red[1][w];
      }
      s_off = o2;
      s_tot = t2;
    }
    __syncthreads();
    if (!(s_off > conv * s_tot)) break;
    if (warp == 0) jacobi_angles(A, ld, n, 0, rot);
    __syncthreads();
    for (int step = 0; step < n - 1; ++step) {
      const float4* ro = rot + (step & 1) * h;
      for (int m1 = warp; m1 < h; m1 += 32) {  // A: rows of pair m1 first, then columns of pair m2
        const float4 r1 = ro[m1];
        float* rp = A + __float_as_int(r1.z) * ld;
        float* rq = A + __float_as_int(r1.w) * ld;
        for (int m2 = lane; m2 < h; m2 += 32) {
          const float4 r2 = ro[m2];
          const int p2 = __float_as_int(r2.z), q2 = __float_as_int(r2.w);
          const float app = rp[p2], apq = rp[q2], aqp = rq[p2], aqq = rq[q2];
          const float bpp = r1.x * app - r1.y * aqp, bqp = r1.y * app + r1.x * aqp;
          const float bpq = r1.x * apq - r1.y * aqq, bqq = r1.y * apq + r1.x * aqq;
          rp[p2] = r2.x * bpp - r2.y * bpq;
          rp[q2] = r2.y * bpp + r2.x * bpq;
          rq[p2] = r2.x * bqp - r2.y * bqq;
          rq[q2] = r2.y * bqp + r2.x * bqq;
        }
      }
      __syncthreads();
      if (warp == 0) {
        if (step + 1 < n - 1) jacobi_angles(A, ld, n, step + 1, rot + ((step + 1) & 1) * h);
      } else {
        for (int m2 = lane; m2 < h; m2 += 32) {  // V <- V J
          const float4 r2 = ro[m2];
          const int p2 = __float_as_int(r2.z), q2 = __float_as_int(r2.w);
          for (int k = warp - 1; k < n; k += 31) {
            float* vr = V + k * ld;
            const float vp = vr[p2], vq = vr[q2];
            vr[p2] = r2.x * vp - r2.y * vq;
            vr[q2] = r2.y * vp + r2.x * vq;
          }
        }
      }
      __syncthreads();
    }
  }
  // the n_comp largest eigenvalues (the smaller index first on ties), by one warp
  if (warp == 0) {
    u32 taken = 0;  // bit j: diagonal entry lane + 32 j is used
    for (int k = 0; k < a.n_comp; ++k) {
      float bv = -INFINITY;
      int bi = n;
      for (int j = 0; lane + 32 * j < C; ++j) {
        const float v = A[(lane + 32 * j) * (ld + 1)];
        if (!((taken >> j) & 1u) && (bi == n || v > bv)) {
          bv = v;
          bi = lane + 32 * j;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (oi < n && (bi == n || ov > bv || (ov == bv && oi < bi))) {
          bv = ov;
          bi = oi;
        }
      }
      if ((bi & 31) == lane) taken |= 1u << (bi >> 5);
      if (lane == 0) {
        s_sel[k] = bi;
        a.vals[k] = bv;
      }
    }
  }
  __syncthreads();
  for (int k = 0; k < a.n_comp; ++k) refine_vector(A, V, ld, n, a, s_sel[k], k);
  __syncthreads();
  if (a.info) {
    for (int k = threadIdx.x; k < a.n_comp; k += blockDim.x) a.info[k] = a.vals[k];
    for (int e = threadIdx.x; e < a.n_comp * C; e += blockDim.x) a.info[a.n_comp + e] = a.vecs[e];
    for (int c = threadIdx.x; c < C; c += blockDim.x) a.info[a.n_comp + a.n_comp * C + c] = a.mean[c];
  }
}

// Four lanes per cell, four channels per lane and load (one channel where the row length
// is not a multiple of 4), added over the lanes at the end: a thread per cell walked its row
// alone, one 4-byte load at a time (64 channels, 500 x 500 cells: 62 -> 21 us).
__global__ void __launch_bounds__(256) k_pca_project(MapDev md, PcaArgs a, int rx, int ry) {
  __shared__ __align__(16) float sv[kPcaMaxComp][kPcaMaxC], sm[kPcaMaxC];
  for (int e = threadIdx.x; e < a.n_comp * a.C; e += blockDim.x) sv[e / a.C][e % a.C] = a.vecs[e];
  for (int c = threadIdx.x; c < a.C; c += blockDim.x) sm[c] = a.mean[c];
  __syncthreads();
  const int W = md.W, sub = threadIdx.x & 3;
  const bool vec = (a.C & 3) == 0;  // rows (S = C values) then start on 16-byte (8-byte) boundaries
  for (u32 j0 = (blockIdx.x * blockDim.x + threadIdx.x) / 4; j0 - (threadIdx.x & 31) / 4 < md.W2;
       j0 += gridDim.x * blockDim.x / 4) {  // the same count for every lane of a warp
    const u32 j = min(j0, md.W2 - 1);
    const int ix = (int)(j % (u32)W), iy = (int)(j / (u32)W);
    int px = ix + rx;
    if (px >= W) px -= W;
    int py = iy + ry;
    if (py >= W) py -= W;
    const u32 g = (u32)a.map * md.W2 + (u32)py * (u32)W + (u32)px;
    float out[kPcaMaxComp];
#pragma unroll
    for (int k = 0; k < kPcaMaxComp; ++k) out[k] = 0.f;
    if (md.flags[g] & a.obs_bit) {
      if (vec) {
#pragma unroll 4
        for (int c = 4 * sub; c < a.C; c += 16) {
          const float4 v = layer_val4(a.data, a.dtype, (int64_t)g * a.S + c);
          const float4 m = *reinterpret_cast<const float4*>(sm + c);
          const float x[4] = {__fsub_rn(v.x, m.x), __fsub_rn(v.y, m.y), __fsub_rn(v.z, m.z), __fsub_rn(v.w, m.w)};
#pragma unroll
          for (int k = 0; k < kPcaMaxComp; ++k)
            if (k < a.n_comp) {
              const float4 w = *reinterpret_cast<const float4*>(&sv[k][c]);
              out[k] = __fmaf_rn(x[0], w.x, out[k]);
              out[k] = __fmaf_rn(x[1], w.y, out[k]);
              out[k] = __fmaf_rn(x[2], w.z, out[k]);
              out[k] = __fmaf_rn(x[3], w.w, out[k]);
            }
        }
      } else {
        for (int c = sub; c < a.C; c += 4) {
          const float x = __fsub_rn(layer_val(a.data, a.dtype, (int64_t)g * a.S + c), sm[c]);
#pragma unroll
          for (int k = 0; k < kPcaMaxComp; ++k)
            if (k < a.n_comp) out[k] = __fmaf_rn(x, sv[k][c], out[k]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kPcaMaxComp; ++k) {
      if (k >= a.n_comp) break;
      out[k] += __shfl_xor_sync(0xffffffffu, out[k], 1);
      out[k] += __shfl_xor_sync(0xffffffffu, out[k], 2);
      if (sub == (k & 3) && j0 < md.W2) a.proj[(int64_t)j * a.n_comp + k] = out[k];
    }
  }
}

}  // namespace memk

// ---------------------------------------------------------------------------
// host

namespace memh {
using namespace memk;

cudaError_t launch_normals(Map* m, int map_index, float* out, uint8_t* ok, cudaStream_t st) {
  dim3 blk(16, 16), grd((m->md.W + 15) / 16, (m->md.W + 15) / 16);
  k_normals<<<grd, blk, 0, st>>>(m->md, map_index, m->ring[2 * map_index], m->ring[2 * map_index + 1], out, ok);
  return cudaGetLastError();
}

// scratch of the PCA plugin, owned by the map (grown on demand, outside graphs)
cudaError_t launch_pca(Map* m, int map_index, int layer, int n_comp, float* proj, float* info, cudaStream_t st) {
  const LayerDev& L = m->Lh[layer];
  const int C = L.C;
  const int nt = (C + 7) / 8, tiles = nt * (nt + 1) / 2;  // 8 x 8 tiles of the upper triangle
  const int groups = std::max(1, std::min(8, 256 / tiles));
  const int blocks = m->n_sm * kPcaBlocks;
  const size_t need = sizeof(double) * (size_t)(blocks + 1) * (C + 1) + sizeof(float) * (size_t)blocks * tiles * 64 +
                      sizeof(float) * ((size_t)C * C + C + (size_t)kPcaMaxComp * (C + 1)) + 1024;
  if (need > m->pca_cap) {
    cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    if (m->pca_buf) cudaFree(m->pca_buf);
    m->pca_buf = nullptr;
    m->pca_cap = 0;
    e = cudaMalloc(&m->pca_buf, need);
    if (e != cudaSuccess) return e;
    m->pca_cap = need;
  }
  char* p = (char*)m->pca_buf;
  PcaArgs a;
  a.map = map_index;
  a.layer = layer;
  a.C = C;
  a.n_comp = n_comp;
  a.blocks = blocks;
  a.data = L.data;
  a.S = L.S;
  a.dtype = L.dtype;
  a.obs_bit = 2u << layer;
  a.mean_part = (double*)p;
  p += sizeof(double) * (size_t)(blocks + 1) * (C + 1);
  a.cov_part = (float*)p;
  p += sizeof(float) * (size_t)blocks * tiles * 64;
  a.cov = (float*)p;
  p += sizeof(float) * (size_t)C * C;
  a.mean = (float*)p;
  p += sizeof(float) * (size_t)C;
  a.vecs = (float*)p;
  p += sizeof(float) * (size_t)kPcaMaxComp * C;
  a.vals = (float*)p;
  a.proj = proj;
  a.info = info;
  k_pca_mean<<<blocks, 256, 0, st>>>(m->md, a);
  k_pca_mean_final<<<1, 1024, 0, st>>>(a);
  const int n = (C + 1) & ~1;
  // a staged block of rows, reused for the tiles' sums
  const size_t csm = sizeof(float) * std::max((size_t)kPcaRows * (nt * 8 + 4), (size_t)tiles * 64);
  const size_t esm = sizeof(float) * (2 * (size_t)n * (n + 1) + 4 * n) + 32;
  static bool attr[128] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 128 && !attr[dev]) {
    cudaError_t e = cudaFuncSetAttribute(k_pca_eig, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(sizeof(float) * (2 * 128 * 129 + 4 * 128) + 32));
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  k_pca_cov<<<blocks, 256, csm, st>>>(m->md, a, nt, tiles, groups);
  k_pca_cov_final<<<tiles * 2, 256, 0, st>>>(a, nt, tiles);
  k_pca_eig<<<1, 1024, esm, st>>>(a);
  k_pca_project<<<m->n_sm * 4, 256, 0, st>>>(m->md, a, m->ring[2 * map_index], m->ring[2 * map_index + 1]);
  return cudaGetLastError();
}

}  // namespace memh

extern "C" mem_status mem_compute_normals(mem_map* mm, int32_t map_index, float* normals, uint8_t* ok,
                                          void* stream) {
  if (!mm || !normals) return memh::api_fail(MEM_ERR_ARG, "NULL argument");
  memh::Map* m = memh::map_of(mm);
  if (map_index < 0 || map_index >= m->cfg.n_maps) return memh::api_fail(MEM_ERR_ARG, "map_index out of range");
  cudaError_t e = memh::launch_normals(m, map_index, normals, ok, (cudaStream_t)stream);
  if (e != cudaSuccess) return memh::api_cuda_fail(e, "normals launch");
  return MEM_OK;
}

extern "C" mem_status mem_pca_layer(mem_map* mm, int32_t map_index, int32_t layer, int32_t n_comp, float* proj,
                                    float* info, void* stream) {
  if (!mm || !proj) return memh::api_fail(MEM_ERR_ARG, "NULL argument");
  memh::Map* m = memh::map_of(mm);
  if (map_index < 0 || map_index >= m->cfg.n_maps) return memh::api_fail(MEM_ERR_ARG, "map_index out of range");
  if (layer < 0 || layer >= m->cfg.n_layers) return memh::api_fail(MEM_ERR_ARG, "layer out of range");
  if (m->cfg.layers[layer].rule == MEM_RULE_CLASSMAX) return memh::api_fail(MEM_ERR_ARG, "a class-max layer has no features");
  const int C = m->cfg.layers[layer].channels;
  if (C < 1 || C > memk::kPcaMaxC) return memh::api_fail(MEM_ERR_ARG, "PCA takes layers of 1..%d channels", memk::kPcaMaxC);
  if (n_comp < 1 || n_comp > memk::kPcaMaxComp || n_comp > C)
    return memh::api_fail(MEM_ERR_ARG, "n_comp in [1, min(%d, channels)]", memk::kPcaMaxComp);
  cudaError_t e = memh::launch_pca(m, map_index, layer, n_comp, proj, info, (cudaStream_t)stream);
  if (e != cudaSuccess) return memh::api_cuda_fail(e, "PCA launch");
  return MEM_OK;
}
