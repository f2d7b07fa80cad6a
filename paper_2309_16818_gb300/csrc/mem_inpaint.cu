// Diffusion (harmonic) inpainting of map crops: every unknown cell takes the
// mean of its in-crop 4-neighbours (zero-flux border), known cells stay fixed,
// i.e. the discrete Laplace equation with the known cells as boundary values.
//
// A crop that fits the shared memory of a cluster of up to 8 CTAs is solved by
// k_inpaint_sor_cluster (its rows split over the cluster, boundary rows written
// into the neighbours' shared memory); larger crops by k_inpaint_sor, one
// thread block per crop working in global memory (L2-resident).
// Unknown cells start from the mean of the crop's known cells; the sweeps stop
// when the largest update of a full sweep falls below `tol` or after
// `max_iters` sweeps.
//
// Over-relaxation factor: SOR with the optimal factor for the Jacobi spectral
// radius mu of the unknown region, omega = 2 / (1 + sqrt(1 - mu^2)), shrinks
// the error by omega - 1 per sweep (the classical red-black SOR theory of
// consistently ordered matrices). The shared-memory kernel bounds mu per crop
// from d, the largest Euclidean distance from an unknown cell to the nearest
// known cell (zero-flux crop borders mirror the region, so they do not bound
// it): a strip of width 2 d has the smallest Laplacian eigenvalue
// (pi / (2 d))^2, so mu <= 1 - (pi / (2 d))^2 / 4 is taken, which errs towards
// over-relaxation, where the rate degrades only linearly. The factor is capped
// at that of a square crop with fixed borders, sized by its longer side (the
// factor the global-memory kernel uses for every crop).
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "mem_host.h"

namespace cg = cooperative_groups;

namespace memk {

constexpr int kInpThreads = 1024;

__device__ __forceinline__ float block_max(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) red[32] = v;
  }
  __syncthreads();
  const float r = red[32];
  __syncthreads();
  return r;
}

__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[32] = v;
  }
  __syncthreads();
  const float r = red[32];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(kInpThreads) k_inpaint_sor(int H, int W, const float* __restrict__ hin,
                                                             const uint8_t* __restrict__ known,
                                                             float* __restrict__ hout, float omega, float tol,
                                                             int max_iters, int* iters_out) {
  __shared__ float red[33];
  const int64_t base = (int64_t)blockIdx.x * H * W;
  const float* in = hin + base;
  const uint8_t* kn = known + base;
  float* h = hout + base;
  const int n = H * W;
  // initial guess: known values, unknown cells at the mean of the known ones
  float s = 0.f, c = 0.f;
  for (int j = threadIdx.x; j < n; j += blockDim.x)
    if (kn[j]) {
      s += in[j];
      c += 1.f;
    }
  s = block_sum(s, red);
  c = block_sum(c, red);
  const float mean = c > 0.f ? s / c : 0.f;
  for (int j = threadIdx.x; j < n; j += blockDim.x) h[j] = kn[j] ? in[j] : mean;
  __syncthreads();
  int it = 0;
  for (; it < max_iters; ++it) {
    float dmax = 0.f;
    for (int color = 0; color < 2; ++color) {
      for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int y = j / W, x = j - y * W;
        if (((x + y) & 1) != color || kn[j]) continue;
        float sum = 0.f;
        int m = 0;
        if (x > 0) sum += h[j - 1], ++m;
        if (x + 1 < W) sum += h[j + 1], ++m;
        if (y > 0) sum += h[j - W], ++m;
        if (y + 1 < H) sum += h[j + W], ++m;
        if (m == 0) continue;  // a 1 x 1 crop keeps its starting value
        const float old = h[j];
        const float d = sum / (float)m - old;
        h[j] = fmaf(omega, d, old);
        dmax = fmaxf(dmax, fabsf(d));
      }
      __syncthreads();
    }
    dmax = block_max(dmax, red);
    if (dmax < tol) {
      ++it;
      break;
    }
  }
  if (threadIdx.x == 0 && iters_out) iters_out[blockIdx.x] = it;
}

// The same red-black SOR with the crop held in shared memory: a thread-block
// cluster of CL CTAs owns one crop, CTA r its band of rows [r H / CL,
// (r + 1) H / CL). Each colour is stored packed: cell (x, y) of colour
// c = (x + y) & 1 sits at index k = x >> 1 of row y of array c. With p = (y + c) & 1
// (so x = 2k + p), its four neighbours (colour 1 - c) are k - 1 + p and k + p of the
// same row and k of the rows above and below. A band has a row above and one below
// it: the neighbouring bands' boundary rows, which their CTAs write there
// (distributed shared memory) whenever they update them, or zeros outside the crop;
// rows are padded with zeros to a multiple of 4 with at least one zero, which also
// stand for the cells left and right of the crop.
//
// A sweep visits only groups of four cells that hold an unknown cell. They are
// listed once (the known cells never change): groups of four unknown cells off the
// crop's border by their row's parity p, whose update needs no masks and selects,
// and the others; the threads share a list out evenly, a warp's groups mostly side
// by side (no bank conflicts). A group costs five shared-memory reads and one write,
// all of them local. The largest update of a sweep goes to a word of every CTA by
// warp maxima and atomics (the bits of non-negative floats order as integers) before
// the barrier that ends the sweep. Bound by the two barriers of a sweep and the latency
// between them.
// Before: every group of every row, the neighbours' rows read remotely, and three
// block barriers for the maximum. 256 crops of 256 x 256, 27 % unknown, 207 sweeps on
// average: 7.66 -> 5.10 ms (a sweep of the 152 SMs' 76 crops 5.9 -> 4.4 us, the set-up 0.47 -> 0.17 ms
// of a round); 6 crops of 200 x 136, one CTA each: 1.25 -> 0.46 ms.
constexpr int kSorSmemMax = 224 * 1024;  // of 227 KB, with the static arrays
constexpr int kSorThreads = 1024;

__host__ __device__ constexpr int sor_stride(int W) { return ((W + 1) / 2 + 4) / 4 * 4; }  // floats per row, one zero at least

// list word: offset of the group in 16-byte units | unknown cells << 16 | p << 20 | the crop's
// edges that it lies at: top, bottom, left, right (bits 21..24) | cells up to the right edge << 25
static_assert(kSorThreads <= 1024, "a warp reads one word of every warp");
constexpr u32 kSorP = 1u << 20, kSorTop = 1u << 21, kSorBottom = 1u << 22, kSorLeft = 1u << 23, kSorRight = 1u << 24;

// the update of four cells from the group of the other colour beside them, above and below
template <int P>
__device__ __forceinline__ void sor_sums(const float* O, int off, int Ws, float m[4]) {
  const float4 o4 = *reinterpret_cast<const float4*>(O + off);
  const float4 u4 = *reinterpret_cast<const float4*>(O + off - Ws);
  const float4 d4 = *reinterpret_cast<const float4*>(O + off + Ws);
  const float side = P ? O[off + 4] : O[off - 1];
  m[0] = (((P ? o4.x : side) + (P ? o4.y : o4.x)) + u4.x) + d4.x;
  m[1] = (((P ? o4.y : o4.x) + (P ? o4.z : o4.y)) + u4.y) + d4.y;
  m[2] = (((P ? o4.z : o4.y) + (P ? o4.w : o4.z)) + u4.z) + d4.z;
  m[3] = (((P ? o4.w : o4.z) + (P ? side : o4.w)) + u4.w) + d4.w;
}

// where a band's first and last rows also live: the rows around the neighbouring bands
struct SorHalo {
  float *up, *dn;  // (of the colour), null at the crop's border
  int Ws, last;    // floats per row, offset of the band's last row
  __device__ __forceinline__ void put(int off, float4 v) const {
    if (up && off < 2 * Ws) *reinterpret_cast<float4*>(up + off - Ws) = v;
    if (dn && off >= last) *reinterpret_cast<float4*>(dn + off - last) = v;
  }
};

// one group of four unknown cells with four neighbours each, of a row of parity P
template <int P>
__device__ __forceinline__ float4 sor_full(const float* C, const float* O, int off, int Ws, float omega, float& dmax) {
  const float4 c4 = *reinterpret_cast<const float4*>(C + off);
  float m[4], cv[4] = {c4.x, c4.y, c4.z, c4.w};
  sor_sums<P>(O, off, Ws, m);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float d = fmaf(m[j], 0.25f, -cv[j]);  // the quarter is exact
    cv[j] = fmaf(omega, d, cv[j]);
    dmax = fmaxf(dmax, fabsf(d));
  }
  return make_float4(cv[0], cv[1], cv[2], cv[3]);
}

// one other group: some cells known, outside the crop or with q < 4 neighbours (the mean of q
// neighbours is a multiplication by 1 / q and one correction, which rounds like the division)
__device__ __forceinline__ float4 sor_rest(const float* C, const float* O, u32 w, int off, int Ws, float omega,
                                           float& dmax) {
  const float4 c4 = *reinterpret_cast<const float4*>(C + off);
  float m[4], cv[4] = {c4.x, c4.y, c4.z, c4.w};
  if (w & kSorP) sor_sums<1>(O, off, Ws, m);
  else sor_sums<0>(O, off, Ws, m);
  const int q0 = 4 - ((w & kSorTop) ? 1 : 0) - ((w & kSorBottom) ? 1 : 0);
  const int jr = (w & kSorRight) ? (int)(w >> 25) : 4;  // the cell at the right edge
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int q = q0 - (j == 0 && (w & kSorLeft) ? 1 : 0) - (j == jr ? 1 : 0);
    const float fq = (float)q, rq = q == 4 ? 0.25f : q == 3 ? 1.f / 3.f : q == 2 ? 0.5f : 1.f;
    float a = m[j] * rq;
    a = fmaf(fmaf(-fq, a, m[j]), rq, a);
    const float d = q ? a - cv[j] : 0.f;  // a 1 x 1 crop keeps its starting value
    if ((w >> (16 + j)) & 1u) {
      cv[j] = fmaf(omega, d, cv[j]);
      dmax = fmaxf(dmax, fabsf(d));
    }
  }
  return make_float4(cv[0], cv[1], cv[2], cv[3]);
}

// One colour of a sweep over the band's list: n[0] other groups, then n[1] and n[2] full groups
// of parity 0 and 1. One loop over all of them: a thread has one or two groups, and its
// chain of shared-memory reads and additions, not the instructions, is what a sweep takes.
template <bool HALO>
__device__ __forceinline__ float sor_color(float* C, const float* O, const u32* li, int n0, int n1, int n2, int Ws,
                                           float omega, const SorHalo& halo) {
  float dmax = 0.f;
  const int n = n0 + n1 + n2;
  for (int i = threadIdx.x; i < n; i += kSorThreads) {
    const u32 w = li[i];
    const int off = 4 * (int)(w & 0xffffu);
    const float4 v = i < n0 ? sor_rest(C, O, w, off, Ws, omega, dmax)
                            : (i < n0 + n1 ? sor_full<0>(C, O, off, Ws, omega, dmax)
                                           : sor_full<1>(C, O, off, Ws, omega, dmax));
    *reinterpret_cast<float4*>(C + off) = v;
    if (HALO) halo.put(off, v);
  }
  return dmax;
}

__global__ void __launch_bounds__(kSorThreads) k_inpaint_sor_cluster(int H, int W, int CL,
                                                                     const float* __restrict__ hin,
                                                                     const uint8_t* __restrict__ known,
                                                                     float* __restrict__ hout, float omega, float tol,
                                                                     int max_iters, int* iters_out) {
  cg::cluster_group cl = cg::this_cluster();
  const int r = (int)cl.block_rank();
  const int crop = blockIdx.x / CL;
  const int y0 = (int)((int64_t)H * r / CL), y1 = (int)((int64_t)H * (r + 1) / CL);
  const int rows = y1 - y0;
  const int rows_max = (H + CL - 1) / CL;
  const int Ws = sor_stride(W), Ws4 = Ws / 4;
  const int plane = (rows_max + 2) * Ws;  // floats of one colour: row above, rows, row below
  extern __shared__ __align__(16) float sh[];
  u32* list = (u32*)(sh + 2 * plane);  // [colour][rows_max * Ws4]
  __shared__ float red[33];
  __shared__ float s_part[3];
  __shared__ u32 s_max[2][8][kSorThreads / 32];  // largest updates (bits) of even and odd sweeps, of every CTA's warps
  __shared__ int s_n[2][3];    // per colour: other groups, groups of four unknown cells of parity 0, 1
  __shared__ int s_pos[2][3];  // next word of each in the list
  __shared__ int s_best;   // largest squared distance found so far
  __shared__ int s_y0[9];  // first row of every band, and H
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto barrier = [&]() {
    if (CL == 1) __syncthreads();
    else cl.sync();
  };
  const int64_t crop0 = (int64_t)crop * H * W, base = crop0 + (int64_t)y0 * W;
  // 0. the squared largest distance of an unknown cell to a known cell: first, per row of
  //    the band, the distance along the row (kFar: none) from the row's known bits, in the
  //    heights' shared memory (free until they are loaded); then per unknown cell of the band
  //    the exact Euclidean distance over the column (rows of the other bands read from their
  //    CTAs), scanning outwards until no closer known cell can remain
  constexpr int kFar = 0x3fff;
  uint16_t* gd = reinterpret_cast<uint16_t*>(sh);  // [rows][W]
  const int nw = (W + 31) / 32;
  u32* bits = reinterpret_cast<u32*>(sh + plane);  // known bits [rows][nw], in the other half of that memory
  {
    if (threadIdx.x <= CL) s_y0[threadIdx.x] = (int)((int64_t)H * threadIdx.x / CL);
    if (threadIdx.x == 0) s_best = 0;
#pragma unroll 4
    for (int i = warp; i < rows * nw; i += kSorThreads / 32) {
      const int ly = i / nw, x = (i - ly * nw) * 32 + lane;
      const u32 m = __ballot_sync(0xffffffffu, x < W && known[base + (int64_t)ly * W + x]);
      if (lane == 0) bits[i] = m;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < rows * W; j += kSorThreads) {
      const int ly = j / W, x = j - ly * W;
      const u32* row = bits + ly * nw;
      int d = kFar;
      u32 m = row[x >> 5] & (0xffffffffu >> (31 - (x & 31)));  // at x and to the left
      for (int w = x >> 5;;) {
        if (m) {
          d = min(d, x - (w * 32 + 31 - __clz(m)));
          break;
        }
        if (--w < 0 || x - (w * 32 + 31) >= d) break;
        m = row[w];
      }
      m = row[x >> 5] & (0xffffffffu << (x & 31));  // at x and to the right
      for (int w = x >> 5;;) {
        if (m) {
          d = min(d, w * 32 + __ffs(m) - 1 - x);
          break;
        }
        if (++w >= nw || w * 32 - x >= d) break;
        m = row[w];
      }
      gd[j] = (uint16_t)d;
    }
  }
  barrier();
  {
    // cells that can no longer exceed the block's largest distance so far stop early (s_best is
    // a lower bound that only grows, so an old value read here is only less tight)
    for (int j = threadIdx.x; j < rows * W; j += kSorThreads) {
      const int g0 = gd[j];
      int best = g0 * g0;
      int known_best = *(volatile int*)&s_best;
      if (best <= known_best) continue;  // among them every known cell
      const int ly = j / W, x = j - ly * W;
      const int y = y0 + ly;
      int qu = r, qd = r, ys = y0, ye = y1;  // the bands the two scans are in, their first and end rows
      const uint16_t *pu = gd + j, *pd = gd + j;
      for (int k = 1; k * k < best && best > known_best; ++k) {
        const bool up = y - k >= 0, dn = y + k < H;
        if (!up && !dn) break;
        if (up) {
          if (y - k < ys) {
            --qu;
            ys = s_y0[qu];
            pu = cl.map_shared_rank(gd, qu) + (s_y0[qu + 1] - 1 - ys) * W + x;
          } else {
            pu -= W;
          }
          const int g = *pu;
          best = min(best, g * g + k * k);
        }
        if (dn) {
          if (y + k >= ye) {
            ++qd;
            ye = s_y0[qd + 1];
            pd = cl.map_shared_rank(gd, qd) + x;
          } else {
            pd += W;
          }
          const int g = *pd;
          best = min(best, g * g + k * k);
        }
      }
      if (best > known_best) atomicMax(&s_best, best);
    }
    __syncthreads();
    if (threadIdx.x == 0) s_part[2] = (float)s_best;
  }
  // 1. mean of the known heights and the crop's over-relaxation factor
  float s = 0.f, c = 0.f;
#pragma unroll 4
  for (int j = threadIdx.x; j < rows * W; j += kSorThreads)
    if (known[base + j]) {
      s += hin[base + j];
      c += 1.f;
    }
  s = block_sum(s, red);
  c = block_sum(c, red);
  if (threadIdx.x == 0) {
    s_part[0] = s;
    s_part[1] = c;
  }
  if (threadIdx.x < 6) s_n[threadIdx.x / 3][threadIdx.x % 3] = 0;
  barrier();  // every band's distances are read too; the heights may overwrite them
  float S = 0.f, Cn = 0.f, D2 = 0.f;
  for (int q = 0; q < CL; ++q) {
    const float* pp = cl.map_shared_rank(s_part, q);
    S += pp[0];
    Cn += pp[1];
    D2 = fmaxf(D2, pp[2]);
  }
  const float mean = Cn > 0.f ? S / Cn : 0.f;
  {  // the crop's over-relaxation factor from the distance bound (at least one cell apart)
    const float d = fmaxf(sqrtf(D2), 1.f);
    const float a = 3.14159265f / (2.f * d);
    const float lq = 0.25f * a * a;  // 1 - mu
    omega = fminf(omega, 2.f / (1.f + sqrtf(lq * (2.f - lq))));
  }
  // 2. the lists of groups with unknown cells, counted, then written by warps over consecutive
  //    groups (which group has which place changes nothing: a colour's updates are independent)
  const int groups = rows * Ws4;
  for (int pass = 0; pass < 2; ++pass) {
    for (int col = 0; col < 2; ++col)
      for (int e0 = warp * 32; e0 < groups; e0 += kSorThreads) {
        const int e = e0 + lane, ly = e / Ws4, k0 = (e - ly * Ws4) * 4, y = y0 + ly, p = (y + col) & 1;
        u32 unknown = 0;
        if (e < groups && 2 * k0 < W) {
          const u32 kb = bits[ly * nw + (k0 >> 4)] >> (2 * k0 & 31);  // cells 2 k0 .. 2 k0 + 7 of the row
#pragma unroll
          for (int j = 0; j < 4; ++j)
            unknown |= (2 * (k0 + j) + p < W && !((kb >> (2 * j + p)) & 1u)) ? 1u << j : 0u;
        }
        // the crop's edges at the group (the right one: its cell (W - 1 - p) / 2 - k0, if that cell has the
        // parity of the last column)
        const int jr = (W - 1 - p) / 2 - k0;
        u32 edge = (y == 0 ? kSorTop : 0u) | (y == H - 1 ? kSorBottom : 0u) | (k0 == 0 && p == 0 ? kSorLeft : 0u);
        if (((W - 1 - p) & 1) == 0 && jr >= 0 && jr < 4) edge |= kSorRight | (u32)jr << 25;
        const int kind = unknown == 0 ? -1 : (unknown == 15u && !edge) ? 1 + p : 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const u32 bal = __ballot_sync(0xffffffffu, kind == q);
          if (bal == 0) continue;
          int at = 0;
          if (lane == 0) at = atomicAdd(pass ? &s_pos[col][q] : &s_n[col][q], __popc(bal));
          at = __shfl_sync(0xffffffffu, at, 0);
          if (pass && kind == q)
            list[col * rows_max * Ws4 + at + __popc(bal & ((1u << lane) - 1u))] =
                (u32)(e + Ws4) | unknown << 16 | (p ? kSorP : 0u) | edge;
        }
      }
    __syncthreads();
    if (pass == 0 && threadIdx.x < 2) {
      const int* n = s_n[threadIdx.x];
      s_pos[threadIdx.x][0] = 0;
      s_pos[threadIdx.x][1] = n[0];
      s_pos[threadIdx.x][2] = n[0] + n[1];
    }
    __syncthreads();
  }
  // both colours of the band and the rows around it: unknown cells start at the mean, cells
  // outside the crop are 0
  for (int i = threadIdx.x; i < 2 * (rows + 2) * Ws4; i += kSorThreads) {
    const int col = i >= (rows + 2) * Ws4, e = i - col * (rows + 2) * Ws4;
    const int ly = e / Ws4 - 1, k0 = (e - (ly + 1) * Ws4) * 4, y = y0 + ly;
    const int p = (y + col) & 1;
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int x = 2 * (k0 + j) + p;
      const bool in = y >= 0 && y < H && x < W;
      const int64_t at = crop0 + (int64_t)y * W + x;
      v[j] = in ? (known[at] ? hin[at] : mean) : 0.f;
    }
    *reinterpret_cast<float4*>(sh + col * plane + 4 * e) = make_float4(v[0], v[1], v[2], v[3]);
  }
  // the halo rows of the neighbouring bands that this band's first and last rows are
  float* up_halo = r > 0 ? cl.map_shared_rank(sh, r - 1) + (y0 - (int)((int64_t)H * (r - 1) / CL) + 1) * Ws : nullptr;
  float* dn_halo = r + 1 < CL ? cl.map_shared_rank(sh, r + 1) : nullptr;
  barrier();
  // 3. sweeps
  int it = 0;
  for (; it < max_iters; ++it) {
    float dmax = 0.f;
#pragma unroll 1
    for (int color = 0; color < 2; ++color) {
      float* C = sh + color * plane;
      const float* O = sh + (1 - color) * plane;
      const u32* li = list + color * rows_max * Ws4;
      const SorHalo halo = {up_halo ? up_halo + color * plane : nullptr, dn_halo ? dn_halo + color * plane : nullptr, Ws,
                            rows * Ws};
      const int n0 = s_n[color][0], n1 = s_n[color][1], n2 = s_n[color][2];
      dmax = fmaxf(dmax, CL > 1 ? sor_color<true>(C, O, li, n0, n1, n2, Ws, omega, halo)
                                : sor_color<false>(C, O, li, n0, n1, n2, Ws, omega, halo));
      if (color == 1) {  // the warp's largest update of the sweep, to every CTA
        const u32 m = __reduce_max_sync(0xffffffffu, __float_as_uint(dmax));
        if (lane < CL) (CL == 1 ? &s_max[0][0][0] : cl.map_shared_rank(&s_max[0][0][0], lane))[((it & 1) * 8 + r) * (kSorThreads / 32) + warp] = m;
      }
      barrier();  // this colour's values (and the sweep's maxima) are final for every CTA
    }
    // every warp takes the maximum of the same words; they are next written two sweeps later,
    // after two more barriers
    u32 m = 0;
    for (int q = 0; q < CL; ++q) m = max(m, lane < kSorThreads / 32 ? s_max[it & 1][q][lane] : 0u);
    if (__uint_as_float(__reduce_max_sync(0xffffffffu, m)) < tol) {
      ++it;
      break;
    }
  }
  for (int j = threadIdx.x; j < rows * W; j += kSorThreads) {
    const int ly = j / W, x = j - ly * W;
    hout[base + j] = sh[((x + y0 + ly) & 1) * plane + (ly + 1) * Ws + (x >> 1)];
  }
  if (r == 0 && threadIdx.x == 0 && iters_out) iters_out[crop] = it;
  barrier();  // no CTA leaves while another may still write its shared memory
}

}  // namespace memk

// shared memory of a CTA: two colours of its rows and the rows around them, the lists of groups
static size_t sor_smem(int H, int W, int cl) {
  const size_t rows = (H + cl - 1) / cl, ws = memk::sor_stride(W);
  return 4 * (2 * (rows + 2) * ws + 2 * rows * (ws / 4));  // the rows' distances and known bits fit in the colours
}
// cluster size for a crop held in shared memory: the fewest CTAs (1..8) whose bands of rows
// fit kSorSmemMax (fewer CTAs: fewer rows written across CTAs and cheaper barriers; measured
// faster than two CTAs per SM); 0 when none does. (A group's offset then fits 13 bits.)
static int sor_cluster_size(int H, int W) {
  for (int cl = 1; cl <= 8 && cl <= H; ++cl)
    if (sor_smem(H, W, cl) <= (size_t)memk::kSorSmemMax) return cl;
  return 0;
}

extern "C" mem_status mem_inpaint_diffusion(int32_t n_crops, int32_t H, int32_t W, const float* h_in,
                                            const uint8_t* known, float* h_out, float tol,
                                            int32_t max_iters, int32_t* iters_out, void* stream) {
  if (n_crops < 0 || H < 1 || W < 1 || (int64_t)H * W > (1 << 24))
    return memh::api_fail(MEM_ERR_ARG, "bad crop shape");
  if (n_crops > 0 && (!h_in || !known || !h_out)) return memh::api_fail(MEM_ERR_ARG, "NULL argument");
  if (!(tol > 0.f) || max_iters < 1) return memh::api_fail(MEM_ERR_ARG, "tol > 0 and max_iters >= 1");
  if (n_crops == 0) return MEM_OK;
  // optimal over-relaxation of a square crop with fixed borders on the longer side (the
  // shared-memory kernel lowers it per crop from the crop's unknown region)
  const int L = H > W ? H : W;
  const float omega = (float)(2.0 / (1.0 + sin(M_PI / (double)(L + 1))));
  const int CL = sor_cluster_size(H, W);
  cudaError_t e = cudaSuccess;
  if (CL > 0) {
    const size_t smem = sor_smem(H, W, CL);
    static bool attr[128] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 128 && !attr[dev]) {
      e = cudaFuncSetAttribute(memk::k_inpaint_sor_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               memk::kSorSmemMax);
      if (e != cudaSuccess) return memh::api_cuda_fail(e, "inpaint attribute");
      attr[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_crops * CL));
    cfg.blockDim = dim3(memk::kSorThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)CL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, memk::k_inpaint_sor_cluster, H, W, CL, h_in, known, h_out, omega, tol,
                           max_iters, iters_out);
  } else {
    memk::k_inpaint_sor<<<n_crops, memk::kInpThreads, 0, (cudaStream_t)stream>>>(
        H, W, h_in, known, h_out, omega, tol, max_iters, iters_out);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return memh::api_cuda_fail(e, "inpaint launch");
  return MEM_OK;
}

// ---------------------------------------------------------------------------
// Inputs of the inpainting network per crop: the mean of the known heights
// (float64 sums over a fixed assignment of cells to threads and a fixed reduction
// tree, so every run gives the same bits), then per cell
//   x3 = (fill - mean, hidden, known ? logvar_known : 0),  hidden = !known.
// A cluster of kPrepCl CTAs per crop, each with an even share of its cells and
// kPrepU of them per thread in flight; the CTAs' sums meet through distributed shared
// memory. A few crops leave most SMs idle, and an SM adds only a few float64 values
// per clock, so one block per crop was what a call took (6 crops of 200 x 136: 58.7 us
// with 256 threads and one cell at a time, 48.8 us with 1024 threads and eight, now 13.3 us).
namespace memk {

constexpr int kPrepThreads = 512, kPrepU = 8, kPrepCl = 8;

__global__ void __cluster_dims__(kPrepCl, 1, 1) __launch_bounds__(kPrepThreads)
    k_unet_prepare(int64_t P, const float* __restrict__ h, const uint8_t* __restrict__ known,
                   const float* __restrict__ fill, float* __restrict__ x3, uint8_t* __restrict__ hidden,
                   float* __restrict__ mean_out, float logvar_known) {
  cg::cluster_group cl = cg::this_cluster();
  const int r = (int)cl.block_rank();
  const int crop = blockIdx.x / kPrepCl;
  const int64_t base = (int64_t)crop * P;
  const int64_t q0 = P * r / kPrepCl, q1 = P * (r + 1) / kPrepCl;
  double s = 0.0;
  int c = 0;  // fewer than 2^31 cells
  for (int64_t p0 = q0 + threadIdx.x; p0 < q1; p0 += kPrepU * kPrepThreads) {
    uint8_t k[kPrepU];
    float v[kPrepU];
#pragma unroll
    for (int u = 0; u < kPrepU; ++u) {
      const int64_t p = p0 + u * kPrepThreads;
      k[u] = p < q1 ? known[base + p] : 0;
      v[u] = p < q1 ? h[base + p] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kPrepU; ++u)
      if (k[u]) {
        s += (double)v[u];
        ++c;
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  __shared__ double red[kPrepThreads / 32];
  __shared__ int redc[kPrepThreads / 32];
  __shared__ double s_sum;
  __shared__ int s_cnt;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    red[warp] = s;
    redc[warp] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double S = 0.0;
    int Cn = 0;
    for (int w = 0; w < kPrepThreads / 32; ++w) {
      S += red[w];
      Cn += redc[w];
    }
    s_sum = S;
    s_cnt = Cn;
  }
  cl.sync();
  double S = 0.0;
  int Cn = 0;
  for (int q = 0; q < kPrepCl; ++q) {
    S += *cl.map_shared_rank(&s_sum, q);
    Cn += *cl.map_shared_rank(&s_cnt, q);
  }
  const float mean = (float)(S / (double)(Cn > 1 ? Cn : 1));
  if (r == 0 && threadIdx.x == 0 && mean_out) mean_out[crop] = mean;
  for (int64_t p0 = q0 + threadIdx.x; p0 < q1; p0 += kPrepU * kPrepThreads) {
    uint8_t k[kPrepU];
    float v[kPrepU];
#pragma unroll
    for (int u = 0; u < kPrepU; ++u) {
      const int64_t p = p0 + u * kPrepThreads;
      k[u] = p < q1 ? known[base + p] : 0;
      v[u] = p < q1 ? fill[base + p] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kPrepU; ++u) {
      const int64_t p = p0 + u * kPrepThreads;
      if (p >= q1) continue;
      float* o = x3 + 3 * (base + p);
      o[0] = __fsub_rn(v[u], mean);
      o[1] = k[u] ? 0.f : 1.f;
      o[2] = k[u] ? logvar_known : 0.f;
      hidden[base + p] = k[u] ? 0 : 1;
    }
  }
  cl.sync();  // no CTA leaves while another may still read its sums
}

}  // namespace memk

extern "C" mem_status mem_unet_prepare(int32_t n_crops, int32_t H, int32_t W, const float* h_in,
                                       const uint8_t* known, const float* fill, float* x3, uint8_t* hidden,
                                       float* mean_out, void* stream) {
  if (!h_in || !known || !fill || !x3 || !hidden) return memh::api_fail(MEM_ERR_ARG, "NULL argument");
  if (n_crops < 1 || H < 1 || W < 1 || (int64_t)H * W >= (1ll << 31))
    return memh::api_fail(MEM_ERR_ARG, "bad crop shape");
  // observed cells carry variance 1e-4 m^2: 0.1 ln(1e-4) (hidden cells: 0)
  const float logvar_known = (float)(0.1 * log(1e-4));
  const int64_t P = (int64_t)H * W;
  constexpr int32_t most = INT32_MAX / memk::kPrepCl;  // crops of a launch
  for (int32_t c0 = 0; c0 < n_crops; c0 += std::min(most, n_crops - c0)) {
    const int64_t o = c0 * P;
    memk::k_unet_prepare<<<std::min(most, n_crops - c0) * memk::kPrepCl, memk::kPrepThreads, 0, (cudaStream_t)stream>>>(
        P, h_in + o, known + o, fill + o, x3 + 3 * o, hidden + o, mean_out ? mean_out + c0 : nullptr, logvar_known);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return memh::api_cuda_fail(e, "prepare launch");
  return MEM_OK;
}
