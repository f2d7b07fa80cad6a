// Image association and fusion (Sec. III-B, Fig. 2): every valid cell is
// projected at its elevation into a pinhole camera; a cell is visible iff
// every valid cell on the Bresenham line from the camera's cell to it lies
// strictly below the ray from the camera to the cell (equality occludes).
// Visible cells fuse their pixel with the layer rules (one observation).
//
// Two kernels: the cells that need a visibility walk are listed for the whole
// map; then a warp takes four listed cells, tests the cells of their lines with
// eight lanes each, and fuses the visible ones with the same lanes spread over
// the channels (pixel rows and layer rows read and written in whole sectors).
#include "mem_host.h"

namespace memk {

// the cells an image call lists for a visibility walk (capacity W * W)
struct ImgList {
  u32* n;         // listed cells
  u32* cell;      // y << 16 | x
  float* hz;      // the cell's height
  int32_t* pix;   // its pixel
};

struct ImgParams {
  float R[9], t[3];  // map-centre frame -> optical camera frame
  float fx, fy, cx, cy;
  float hc;          // camera height
  int sx, sy;        // camera cell (clamped into the map)
  int H, Wi;
  int map_index, ring_x, ring_y;
  int n_src;
  SrcDev src[kMaxSources];
};

__device__ __forceinline__ u32 phys(const MapDev& md, int rx, int ry, int x, int y) {
  int px = x + rx;
  if (px >= md.W) px -= md.W;
  int py = y + ry;
  if (py >= md.W) py -= md.W;
  return (u32)py * (u32)md.W + (u32)px;
}

// Whether the cells of the integer Bresenham line from the camera cell (sx, sy)
// to (ex, ey), both ends excluded, all lie below the ray height
//   ray = h_cam + t (h_cell - h_cam),  t = ((q - s).(e - s)) / |e - s|^2
// for the warp's four lines at once (kLineLanes lanes per line, LineWalk; kWalkU
// cells per lane in flight; lines with on == false are skipped). The ray height is
// first estimated with a reciprocal of |e - s|^2 (relative error of t below
// 2^-22), and only where the estimate lies within a bound of the cell's height is
// the exact sequence (correctly rounded division, fma) taken, so every decision
// equals the exact one. A line stops after the 32 cells that hold an occluder.
//
// A line's loads depend on nothing but its ends, so the lanes issue them side by
// side; with one thread per line (four cells at a time) the few lines of 200-300
// cells set the kernel's length, at 7 % of the warp slots.
constexpr int kWalkU = 4;

__device__ __forceinline__ bool walk_visible(const MapDev& md, u32 base, int rx, int ry, int sx, int sy,
                                             int ex, int ey, float hz, float hc, bool on) {
  const int lane = threadIdx.x & 31;
  const u32 mine = ((1u << kLineLanes) - 1u) << (lane & ~(kLineLanes - 1));  // the lanes of this line
  LineWalk lw(sx, sy, ex, ey, lane & (kLineLanes - 1));
  const int dxs = ex - sx, dys = ey - sy;
  const float den = (float)(dxs * dxs + dys * dys);
  const float rden = __frcp_rn(den);
  const float dh = __fsub_rn(hz, hc);
  const float tol = 4e-6f * (fabsf(dh) + fabsf(hc) + 1.f);
  bool visible = on;
  for (int k0 = 1;; k0 += kWalkU * kLineLanes) {
    const bool more = visible && k0 < lw.n;
    if (!__any_sync(0xffffffffu, more)) break;
    int qx[kWalkU], qy[kWalkU];
    u32 fl[kWalkU];
    float hq[kWalkU];
#pragma unroll
    for (int u = 0; u < kWalkU; ++u) {
      const bool act = lw.next(qx[u], qy[u]) && visible;
      const u32 q = base + phys(md, rx, ry, act ? qx[u] : sx, act ? qy[u] : sy);
      fl[u] = act ? md.flags[q] : 0u;
      hq[u] = act ? __ldg(md.h + q) : 0.f;
    }
    bool any = false;
#pragma unroll
    for (int u = 0; u < kWalkU; ++u) {
      if (!(fl[u] & kFlagValid)) continue;
      const int num = (qx[u] - sx) * dxs + (qy[u] - sy) * dys;
      const float est = hq[u] - __fmaf_rn(__fmul_rn((float)num, rden), dh, hc);
      bool occ = est > 0.f;
      if (fabsf(est) <= tol + 4e-6f * fabsf(hq[u])) {  // near the ray: the exact sequence
        const float tq = __fdiv_rn((float)num, den);
        occ = hq[u] >= __fmaf_rn(tq, dh, hc);
      }
      any |= occ;
    }
    const u32 hit = __ballot_sync(0xffffffffu, any);  // every lane takes part, also those of finished lines
    if (hit & mine) visible = false;
  }
  return visible;
}

constexpr int kImgU = 3;  // layers of a source with their old values in flight

// four (nc < 4: fewer) consecutive stored values of a layer; `vec`: the offset is a multiple of 4
__device__ __forceinline__ void ld_layer4(const LayerDev& L, int64_t off, int nc, bool vec, float o[4]) {
  if (vec) {
    if (L.dtype == MEM_F32) {
      const float4 q = *reinterpret_cast<const float4*>((const float*)L.data + off);
      o[0] = q.x; o[1] = q.y; o[2] = q.z; o[3] = q.w;
    } else {
      const uint2 q = *reinterpret_cast<const uint2*>((const uint16_t*)L.data + off);
      const float2 a = L.dtype == MEM_BF16 ? __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x))
                                           : __half22float2(*reinterpret_cast<const __half2*>(&q.x));
      const float2 b = L.dtype == MEM_BF16 ? __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y))
                                           : __half22float2(*reinterpret_cast<const __half2*>(&q.y));
      o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (k < nc) o[k] = ld_layer(L, off + k);
}
__device__ __forceinline__ void st_layer4(const LayerDev& L, int64_t off, int nc, bool vec, const float n[4]) {
  if (vec) {
    if (L.dtype == MEM_F32) {
      *reinterpret_cast<float4*>((float*)L.data + off) = make_float4(n[0], n[1], n[2], n[3]);
    } else {
      uint2 q;
      if (L.dtype == MEM_BF16) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(n[0], n[1]), b = __floats2bfloat162_rn(n[2], n[3]);
        q = make_uint2(*reinterpret_cast<const u32*>(&a), *reinterpret_cast<const u32*>(&b));
      } else {
        const __half2 a = __floats2half2_rn(n[0], n[1]), b = __floats2half2_rn(n[2], n[3]);
        q = make_uint2(*reinterpret_cast<const u32*>(&a), *reinterpret_cast<const u32*>(&b));
      }
      *reinterpret_cast<uint2*>((uint16_t*)L.data + off) = q;
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (k < nc) st_layer(L, off + k, n[k]);
}

// Fuse the warp's four cells (those with `on`), each by the kLineLanes lanes that
// walked its line: pixel p into cell g, four channels per lane, 32 at a time, so
// that the four cells share the instructions (with the whole warp on one cell at a
// time and one channel per lane the kernel was bound by issue). A source's values and the old values
// and prior variances of up to kImgU of its layers are loaded before the first of
// them is stored: a source costs one round trip to memory and not one per layer
// and chunk. Sources go in order: a layer may be fed by several sources of an
// image. Every lane runs every shuffle, with or without a cell.
__device__ __forceinline__ void fuse_pixels(const LayerDev* sL, u32* flags, const ImgParams& ip, int64_t g,
                                            int64_t p, u32 fl, bool on) {
  const int sub = threadIdx.x & (kLineLanes - 1);
  for (int q = 0; q < ip.n_src; ++q) {
    const SrcDev& s = ip.src[q];
    float best = -INFINITY;  // class max over the source's channels
    int bid = 0x7fffffff;
    for (int cb = 0; cb < s.C; cb += 4 * kLineLanes) {
      const int c0 = cb + 4 * sub;
      const int nc = on ? min(4, s.C - c0) : 0;
      const bool vec = nc == 4 && (s.C & 3) == 0;  // rows and layers (S = C) start on multiples of 4
      float v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = -INFINITY;
      if (nc > 0) {
        if (s.topk) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (k < nc) v[k] = src_val(s, p, c0 + k);
        } else {
          ld_src4(s, p, c0, v);
        }
      }
      for (int b0 = 0; b0 < s.n_layers; b0 += kImgU) {
        float old[kImgU][4], s02[kImgU];
#pragma unroll
        for (int u = 0; u < kImgU; ++u) {
          s02[u] = 0.f;
#pragma unroll
          for (int k = 0; k < 4; ++k) old[u][k] = 0.f;
          if (b0 + u >= s.n_layers || nc <= 0) continue;
          const int l = s.layers[b0 + u];
          const LayerDev& L = sL[l];
          if (L.rule == MEM_RULE_CLASSMAX || L.rule == MEM_RULE_LATEST || !(fl & (2u << l))) continue;
          if (L.rule == MEM_RULE_GAUSS) s02[u] = L.gvar[g];
          ld_layer4(L, g * L.S + c0, nc, vec, old[u]);
        }
#pragma unroll
        for (int u = 0; u < kImgU; ++u) {
          if (b0 + u >= s.n_layers || nc <= 0) continue;
          const int l = s.layers[b0 + u];
          const LayerDev& L = sL[l];
          if (L.rule == MEM_RULE_CLASSMAX) continue;
          const RuleCoef co = rule_coef(L, 1.f, 1.f, (fl & (2u << l)) != 0, s02[u]);
          float nv[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) nv[k] = rule_value(L, old[u][k], v[k], co);
          st_layer4(L, g * L.S + c0, nc, vec, nv);
        }
      }
      if (s.has_classmax) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k < nc && v[k] > best) {
            best = v[k];
            bid = c0 + k;
          }
      }
    }
    if (s.has_classmax) {
#pragma unroll
      for (int o = kLineLanes / 2; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bid, o);
        if (ov > best || (ov == best && oi < bid)) {
          best = ov;
          bid = oi;
        }
      }
    }
    __syncwarp();  // every lane read the prior variances
    if (on && sub < s.n_layers) {  // a lane per layer (at most 8): class max, the new Gaussian variance
      const int l = s.layers[sub];
      const LayerDev& L = sL[l];
      if (L.rule == MEM_RULE_CLASSMAX) {
        *reinterpret_cast<float2*>((float*)L.data + g * 2) =
            make_float2(best == -INFINITY ? -1.f : (float)bid, best);
      } else if (L.rule == MEM_RULE_GAUSS) {
        const bool obs = (fl & (2u << l)) != 0;
        L.gvar[g] = rule_coef(L, 1.f, 1.f, obs, obs ? L.gvar[g] : 0.f).var_new;
      }
    }
    __syncwarp();
    for (int b = 0; b < s.n_layers; ++b) fl |= 2u << s.layers[b];
  }
  if (on && sub == 0) flags[g] = fl;
}
static_assert(kLineLanes >= MEM_MAX_SOURCE_LAYERS, "a lane per layer of a source");

// 1. Listing: a block takes a 16 x 16 tile of cells, every thread projects
// its cell; the cells that are valid, in front of the camera and inside the
// image are appended to one list for the whole map (a warp's cells together,
// so neighbouring cells stay neighbours in the list); the others are done.
__global__ void __launch_bounds__(256) k_image_list(MapDev md, ImgParams ip, ImgList li, uint8_t* __restrict__ vis,
                                                    int32_t* __restrict__ pix) {
  const int W = md.W;
  const u32 base = (u32)ip.map_index * md.W2;
  const int lane = (threadIdx.y * 16 + threadIdx.x) & 31;
  const int ix = blockIdx.x * 16 + threadIdx.x;
  const int iy = blockIdx.y * 16 + threadIdx.y;
  bool listed = false;
  float hz = 0.f;
  int32_t px = -1;
  if (ix < W && iy < W) {
    const u32 g = base + phys(md, ip.ring_x, ip.ring_y, ix, iy);
    if (md.flags[g] & kFlagValid) {
      const float xc = __fmul_rn(__fadd_rn((float)(ix - W / 2), 0.5f), md.res);
      const float yc = __fmul_rn(__fadd_rn((float)(iy - W / 2), 0.5f), md.res);
      hz = md.h[g];
      const float Xc = __fmaf_rn(ip.R[0], xc, __fmaf_rn(ip.R[1], yc, __fmaf_rn(ip.R[2], hz, ip.t[0])));
      const float Yc = __fmaf_rn(ip.R[3], xc, __fmaf_rn(ip.R[4], yc, __fmaf_rn(ip.R[5], hz, ip.t[1])));
      const float Zc = __fmaf_rn(ip.R[6], xc, __fmaf_rn(ip.R[7], yc, __fmaf_rn(ip.R[8], hz, ip.t[2])));
      if (Zc > md.z_near) {
        const float u = __fmaf_rn(ip.fx, __fdiv_rn(Xc, Zc), ip.cx);
        const float v = __fmaf_rn(ip.fy, __fdiv_rn(Yc, Zc), ip.cy);
        const float fu = floorf(__fadd_rn(u, 0.5f));
        const float fv = floorf(__fadd_rn(v, 0.5f));
        if (fu >= 0.f && fu < (float)ip.Wi && fv >= 0.f && fv < (float)ip.H) {
          listed = true;
          px = (int32_t)((int64_t)fv * ip.Wi + (int64_t)fu);
        }
      }
    }
    if (!listed) {
      const int64_t j = (int64_t)iy * W + ix;
      if (vis) vis[j] = 0;
      if (pix) pix[j] = -1;
    }
  }
  const u32 bal = __ballot_sync(0xffffffffu, listed);
  u32 k0 = 0;
  if (lane == 0 && bal) k0 = atomicAdd(li.n, (u32)__popc(bal));
  k0 = __shfl_sync(0xffffffffu, k0, 0);
  if (listed) {
    const u32 k = k0 + (u32)__popc(bal & ((1u << lane) - 1u));
    li.cell[k] = ((u32)iy << 16) | (u32)ix;
    li.hz[k] = hz;
    li.pix[k] = px;
  }
}

// 2. Visibility and fusion: every warp of the grid takes listed cells in turn.
// The cell's flags, its pixel's rows and its layers' rows are asked for before
// the walk, which hides their way from memory. Each cell is fused on its own, so the
// list's order does not change a result.
constexpr int kImgBlocks = 8;  // blocks of 128 threads per SM (56-64 registers a thread)

__global__ void __launch_bounds__(128, kImgBlocks) k_image_walk_fuse(MapDev md, const __grid_constant__ ImgParams ip,
                                                                     ImgList li, uint8_t* __restrict__ vis,
                                                                     int32_t* __restrict__ pix) {
  __shared__ LayerDev sL[kMaxLayers];
  if (threadIdx.x < md.n_layers) sL[threadIdx.x] = md.L[threadIdx.x];
  __syncthreads();
  const int W = md.W;
  const u32 base = (u32)ip.map_index * md.W2;
  const int n = (int)*li.n;
  const int lane = threadIdx.x & 31;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  constexpr int kLines = 32 / kLineLanes;
  const int sub = lane & (kLineLanes - 1);
  for (int i0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kLines; i0 < n; i0 += nwarps * kLines) {
    const int i = i0 + lane / kLineLanes;
    const bool on = i < n;
    const u32 c = on ? li.cell[i] : 0u;
    const float hz = on ? li.hz[i] : 0.f;
    const int32_t px = on ? li.pix[i] : 0;
    const int ix = (int)(c & 0xffffu), iy = (int)(c >> 16);
    const u32 g = base + phys(md, ip.ring_x, ip.ring_y, ix, iy);
    const u32 fl = on ? md.flags[g] : 0u;
    for (int q = 0; q < ip.n_src && on; ++q) {
      const SrcDev& s = ip.src[q];
      const int es = s.dtype == MEM_F32 ? 4 : (s.dtype == MEM_U8 ? 1 : 2);
      const int row = s.topk ? 8 * s.topk : s.C * es;
      for (int o = sub * 128; o < row; o += kLineLanes * 128) prefetch_l2((const char*)s.data + (int64_t)px * row + o);
      for (int b = 0; b < s.n_layers; ++b) {
        const LayerDev& L = sL[s.layers[b]];
        const int lrow = L.S * (L.dtype == MEM_F32 ? 4 : 2);
        if (L.rule != MEM_RULE_LATEST)
          for (int o = sub * 128; o < lrow; o += kLineLanes * 128)
            prefetch_l2((const char*)L.data + (int64_t)g * lrow + o);
      }
    }
    const bool visible = walk_visible(md, base, ip.ring_x, ip.ring_y, ip.sx, ip.sy, ix, iy, hz, ip.hc, on);
    if (on && sub == 0) {
      const int64_t j = (int64_t)iy * W + ix;
      if (vis) vis[j] = visible ? 1 : 0;
      if (pix) pix[j] = visible ? px : -1;
    }
    if (ip.n_src > 0 && __any_sync(0xffffffffu, visible)) fuse_pixels(sL, md.flags, ip, g, px, fl, visible);
  }
}

}  // namespace memk

namespace memh {
using namespace memk;

cudaError_t launch_image_fuse(Map* m, int map_index, const MapCall& mc, int H, int Wi, int n_src,
                              const SrcDev* src, const float K[4], uint8_t* vis, int32_t* pix,
                              cudaStream_t st) {
  const MapDev& md = m->md;
  ImgParams ip;
  for (int k = 0; k < 9; ++k) ip.R[k] = mc.R[k];
  for (int k = 0; k < 3; ++k) ip.t[k] = mc.t[k];
  ip.fx = K[0];
  ip.fy = K[1];
  ip.cx = K[2];
  ip.cy = K[3];
  // camera cell, clamped into the map; camera height
  const float res = md.res;
  const float half = (float)(md.W / 2);
  float qx = floorf(mc.cam_x / res), qy = floorf(mc.cam_y / res);
  if (!(qx >= -half)) qx = -half;
  if (!(qx <= half - 1.0f)) qx = half - 1.0f;
  if (!(qy >= -half)) qy = -half;
  if (!(qy <= half - 1.0f)) qy = half - 1.0f;
  ip.sx = (int)qx + md.W / 2;
  ip.sy = (int)qy + md.W / 2;
  ip.hc = mc.cam_h;
  ip.H = H;
  ip.Wi = Wi;
  ip.map_index = map_index;
  ip.ring_x = mc.ring_x;
  ip.ring_y = mc.ring_y;
  ip.n_src = n_src;
  for (int q = 0; q < n_src; ++q) ip.src[q] = src[q];
  // the list (one map's cells at most), allocated on the first call
  const size_t need = sizeof(u32) * (4 + 3 * (size_t)md.W2);
  if (need > m->img_cap) {
    cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    if (m->img_buf) cudaFree(m->img_buf);
    m->img_buf = nullptr;
    m->img_cap = 0;
    e = cudaMalloc(&m->img_buf, need);
    if (e != cudaSuccess) return e;
    m->img_cap = need;
  }
  ImgList li;
  li.n = (u32*)m->img_buf;
  li.cell = li.n + 4;
  li.hz = (float*)(li.cell + md.W2);
  li.pix = (int32_t*)(li.hz + md.W2);
  ProfScope ps(m, kProfImage, st);
  cudaError_t e = cudaMemsetAsync(li.n, 0, sizeof(u32), st);
  if (e != cudaSuccess) return e;
  dim3 blk(16, 16), grd((md.W + 15) / 16, (md.W + 15) / 16);
  k_image_list<<<grd, blk, 0, st>>>(md, ip, li, vis, pix);
  k_image_walk_fuse<<<m->n_sm * kImgBlocks, 128, 0, st>>>(md, ip, li, vis, pix);
  return cudaGetLastError();
}

}  // namespace memh
