// Map building of the tracking pyramid (Sec. IV-D coarse-to-fine scheme; the
// inputs of Eq. 3 and Eq. 4).
//
//   pyramid      level-0 depth / intensity of the live map set from the frame's images,
//                and level l from level l-1: depth = mean of the 2x2 samples > 0 (0 if
//                none), intensity = 2x2 mean
//   normals      n = normalise((v(x+1,y) - v) x (v(x,y+1) - v)), facing the camera,
//                invalid (stored as 0) on the last row / column or next to an invalid
//                depth; v = d K^-1 [u, v, 1]^T; written with the depth as pack A
//   gradient     central-difference intensity gradient, zero on the one-pixel border;
//                written with the intensity as pack B
//
// Depth and intensity are FP32 planes; the packs (packs.cuh) hold FP32 or, with
// DRI_FP16_MAPS, FP16 normals and gradients.
// The batched kernels cover the images of every slot of a plan in one launch; the
// pair kernel serves the allocation-free entry, the single-image gradient kernel an
// uploaded reference.
#include <cuda_fp16.h>

#include "dri_internal.h"
#include "packs.cuh"

namespace dri {

namespace {

// A coarser pixel's depth from the finer 2x2 block, in its row-major order, and its intensity.
__device__ __forceinline__ float depth_mean(float a0, float a1, float b0, float b1) {
  float s = 0.f;
  int n = 0;
  if (a0 > 0.f) { s += a0; ++n; }
  if (a1 > 0.f) { s += a1; ++n; }
  if (b0 > 0.f) { s += b0; ++n; }
  if (b1 > 0.f) { s += b1; ++n; }
  return n ? s / (float)n : 0.f;
}
__device__ __forceinline__ float inten_mean(float a0, float a1, float b0, float b1) {
  return ((a0 + a1) + (b0 + b1)) * 0.25f;
}

// Level-0 copy and every coarser level of one 64 x 32 tile: a block's tile covers whole
// blocks of 8 x 8 pixels, so the levels (at most four) need nothing from outside it.  A
// thread takes 2 x 4 pixels and their two level-1 pixels; pairs of lanes make a level-2
// pixel, a level-3 pixel goes through shared memory.  Each image is read once and every
// level written once (18.5 bytes per pixel at three levels; a copy and a pass per level
// moved 28.5).  With the merged maps below, 64 x 640x480: 4542 -> 4469 us per frame.
__global__ void __launch_bounds__(256) k_pyramid_batch(const BatchArgs a) {
  const int i = batch_slot(a, blockIdx.x);
  const int slot = a.slot0 + i;
  const SlotDyn& d = batch_dyn(a, slot);
  if (d.mode == kSlotIdle) return;
  const SlotStatic& st = a.slots[slot];
  const int levels = st.levels;
  int w = st.tp[0].g.w, h = st.tp[0].g.h;
  const int cs = 1 - st.tp[0].ctrl->ref_index;
  const int t = blockIdx.x - __ldg(a.start + i);
  const int gx = (w + kCopyTileW - 1) / kCopyTileW;
  const int lane = threadIdx.x, ty = threadIdx.y, tx0 = t % gx, ty0 = t / gx;
  int x = tx0 * kCopyTileW + 2 * lane, y = ty0 * kCopyTileH + 4 * ty;
  float dv[4][2], iv[4][2];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    dv[r][0] = dv[r][1] = iv[r][0] = iv[r][1] = 0.f;
    if (y + r < h && x < w) {
      const float* sd = d.src_depth + (int64_t)(y + r) * d.pitch + x;
      const float* si = d.src_inten + (int64_t)(y + r) * d.pitch + x;
      if (x + 1 < w && (((uintptr_t)sd | (uintptr_t)si) & 7) == 0) {
        const float2 a2 = __ldg(reinterpret_cast<const float2*>(sd)), b2 = __ldg(reinterpret_cast<const float2*>(si));
        dv[r][0] = a2.x; dv[r][1] = a2.y;
        iv[r][0] = b2.x; iv[r][1] = b2.y;
      } else {
        dv[r][0] = __ldg(sd);
        iv[r][0] = __ldg(si);
        if (x + 1 < w) {
          dv[r][1] = __ldg(sd + 1);
          iv[r][1] = __ldg(si + 1);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (y + r < h && x < w) {
      float* od = st.tp[0].m.depth[cs] + (int64_t)(y + r) * w + x;
      float* oi = st.tp[0].m.inten[cs] + (int64_t)(y + r) * w + x;
      if ((w & 1) == 0) {            // rows of even width keep the pairs 8-byte aligned
        *reinterpret_cast<float2*>(od) = make_float2(dv[r][0], dv[r][1]);
        *reinterpret_cast<float2*>(oi) = make_float2(iv[r][0], iv[r][1]);
      } else {
        od[0] = dv[r][0];
        oi[0] = iv[r][0];
        if (x + 1 < w) {
          od[1] = dv[r][1];
          oi[1] = iv[r][1];
        }
      }
    }
  if (levels < 2) return;
  w >>= 1, h >>= 1, x >>= 1, y >>= 1;
  float d1[2], i1[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    d1[j] = depth_mean(dv[2 * j][0], dv[2 * j][1], dv[2 * j + 1][0], dv[2 * j + 1][1]);
    i1[j] = inten_mean(iv[2 * j][0], iv[2 * j][1], iv[2 * j + 1][0], iv[2 * j + 1][1]);
    if (x < w && y + j < h) {
      st.tp[1].m.depth[cs][(int64_t)(y + j) * w + x] = d1[j];
      st.tp[1].m.inten[cs][(int64_t)(y + j) * w + x] = i1[j];
    }
  }
  if (levels < 3) return;
  w >>= 1, h >>= 1, x >>= 1, y >>= 1;
  float d2[2], i2[2];                // the right neighbour's
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    d2[j] = __shfl_down_sync(0xffffffffu, d1[j], 1);
    i2[j] = __shfl_down_sync(0xffffffffu, i1[j], 1);
  }
  const float dd = depth_mean(d1[0], d2[0], d1[1], d2[1]), ii = inten_mean(i1[0], i2[0], i1[1], i2[1]);
  if ((lane & 1) == 0 && x < w && y < h) {
    st.tp[2].m.depth[cs][(int64_t)y * w + x] = dd;
    st.tp[2].m.inten[cs][(int64_t)y * w + x] = ii;
  }
  if (levels < 4) return;
  __shared__ float s_d[8][16], s_i[8][16];
  if ((lane & 1) == 0) {
    s_d[ty][lane >> 1] = dd;
    s_i[ty][lane >> 1] = ii;
  }
  __syncthreads();
  if (ty == 0) {
    w >>= 1, h >>= 1;
    const int cx = lane & 7, cy = lane >> 3, px = tx0 * (kCopyTileW / 8) + cx, py = ty0 * (kCopyTileH / 8) + cy;
    if (px < w && py < h) {
      const float *a0 = &s_d[2 * cy][2 * cx], *b0 = &s_d[2 * cy + 1][2 * cx];
      const float *p0 = &s_i[2 * cy][2 * cx], *q0 = &s_i[2 * cy + 1][2 * cx];
      st.tp[3].m.depth[cs][(int64_t)py * w + px] = depth_mean(a0[0], a0[1], b0[0], b0[1]);
      st.tp[3].m.inten[cs][(int64_t)py * w + px] = inten_mean(p0[0], p0[1], q0[0], q0[1]);
    }
  }
}

__device__ __forceinline__ void pyr_down_px(const LevelMaps& fine, const LevelMaps& coarse, int cs,
                                            int wf, int wc, int x, int y) {
  const float* D = fine.depth[cs];
  const float* I = fine.inten[cs];
  const int64_t i0 = (int64_t)(2 * y) * wf + 2 * x;
  const int64_t i1 = i0 + wf;
  const int64_t o = (int64_t)y * wc + x;
  coarse.depth[cs][o] = depth_mean(__ldg(D + i0), __ldg(D + i0 + 1), __ldg(D + i1), __ldg(D + i1 + 1));
  coarse.inten[cs][o] = inten_mean(__ldg(I + i0), __ldg(I + i0 + 1), __ldg(I + i1), __ldg(I + i1 + 1));
}

template <typename T>
__device__ __forceinline__ void normal_px(const LevelMaps& m, int set, const LevelGeom& g,
                                          float dmin, float dmax, int x, int y) {
  const float* D = m.depth[set];
  const int o = y * g.w + x;
  const float d0 = __ldg(D + o);
  float nx = 0.f, ny = 0.f, nz = 0.f;
  if (x + 1 < g.w && y + 1 < g.h) {
    const float d1 = __ldg(D + o + 1);
    const float d2 = __ldg(D + o + g.w);
    const bool ok = d0 >= dmin && d0 <= dmax && d1 >= dmin && d1 <= dmax && d2 >= dmin && d2 <= dmax;
    if (ok) {
      const float rx = ((float)x - g.cx) * g.ifx;
      const float ry = ((float)y - g.cy) * g.ify;
      const float rx1 = ((float)(x + 1) - g.cx) * g.ifx;
      const float ry2 = ((float)(y + 1) - g.cy) * g.ify;
      // forward differences of v = d * ray, written so no large terms cancel; every
      // product and sum is spelled out (fmaf / __fmul_rn) so that no kernel this is
      // inlined into contracts it differently: all map kernels give identical bits
      const float e1 = d1 - d0, e2 = d2 - d0;
      const float ax = fmaf(e1, rx1, __fmul_rn(d0, g.ifx)), ay = __fmul_rn(e1, ry), az = e1;
      const float bx = __fmul_rn(e2, rx), by = fmaf(e2, ry2, __fmul_rn(d0, g.ify)), bz = e2;
      float cx = fmaf(ay, bz, -__fmul_rn(az, by));
      float cy = fmaf(az, bx, -__fmul_rn(ax, bz));
      float cz = fmaf(ax, by, -__fmul_rn(ay, bx));
      const float n2 = fmaf(cx, cx, fmaf(cy, cy, __fmul_rn(cz, cz)));
      if (n2 > 0.f) {
        const float inv = rsqrtf(n2);
        cx = __fmul_rn(cx, inv);
        cy = __fmul_rn(cy, inv);
        cz = __fmul_rn(cz, inv);
        if (fmaf(cx, rx, fmaf(cy, ry, cz)) > 0.f) {   // sign of n . v (v = d0 * ray, d0 > 0)
          cx = -cx;
          cy = -cy;
          cz = -cz;
        }
        nx = cx;
        ny = cy;
        nz = cz;
      }
    }
  }
  Packs<T>::store_a(m.packA[set], o, nx, ny, nz, d0);
}

template <typename T>
__device__ __forceinline__ void gradient_px(const LevelMaps& m, int set, int w, int h, int x, int y) {
  const float* I = m.inten[set];
  const int o = y * w + x;
  float gx = 0.f, gy = 0.f;
  if (x > 0 && y > 0 && x + 1 < w && y + 1 < h) {
    gx = 0.5f * (__ldg(I + o + 1) - __ldg(I + o - 1));
    gy = 0.5f * (__ldg(I + o + w) - __ldg(I + o - w));
  }
  Packs<T>::store_b(m.packB[set], o, __ldg(I + o), gx, gy, __ldg(m.depth[set] + o));
}

// Block -> (slot, 32 x 8 kMapRows tile of the slot's level-`a.level` image):
// the thread's column x and first row y (its rows are y, y + 8, ...); false for
// an idle slot.  w, h: the level's size.
__device__ __forceinline__ bool map_tile(const BatchArgs& a, int* slot, int* x, int* y, int* w,
                                         int* h) {
  const int i = batch_slot(a, blockIdx.x);
  *slot = a.slot0 + i;
  if (batch_dyn(a, *slot).mode == kSlotIdle) return false;
  const LevelGeom& g = a.slots[*slot].tp[a.level].g;
  const int t = blockIdx.x - __ldg(a.start + i);
  const int gx = (g.w + kMapTileW - 1) / kMapTileW;
  *x = (t % gx) * kMapTileW + threadIdx.x;
  *y = (t / gx) * kMapTileH * kMapRows + threadIdx.y;
  *w = g.w;
  *h = g.h;
  return true;
}

// Normals (pack A) and intensity gradients (pack B) of the frame's own map set, which is
// the live frame now and becomes the reference at the frame end (launched before it).
// One pass reads depth and intensity for both: 40 bytes per pixel; as two kernels 44,
// and the captured gradient kernels of a large batch ran after the Gauss-Newton loop
// instead of beside it (64 x 640x480: 150 us at the frame's end).
template <typename T>
__global__ void __launch_bounds__(256) k_maps_batch(const BatchArgs a) {
  int slot, x, y, w, h;
  if (!map_tile(a, &slot, &x, &y, &w, &h) || x >= w) return;
  const TrackParams& tp = a.slots[slot].tp[a.level];
  const int cs = 1 - tp.ctrl->ref_index;
#pragma unroll
  for (int k = 0; k < kMapRows; ++k, y += kMapTileH)
    if (y < h) {
      normal_px<T>(tp.m, cs, tp.g, tp.depth_min, tp.depth_max, x, y);
      gradient_px<T>(tp.m, cs, w, h, x, y);
    }
}

// Both images' normal maps and the reference's gradient map of the allocation-free
// pair entry in one launch (as three, with a one-thread kernel of FP64 set-up in
// front, their launches and that thread's chain were two thirds of the call).
template <typename T>
__global__ void __launch_bounds__(256) k_pair_maps(LevelMaps m, LevelGeom g, float dmin, float dmax,
                                                   PairBegin b, uint8_t* __restrict__ flags) {
  grid_dep_launch();             // the pixel kernel waits for this grid's end itself
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    const int t = threadIdx.y * 32 + threadIdx.x;
    for (int i = t; i < b.ncounters; i += 256) b.counters[i] = 0u;
    if (t < 12) b.ctrl->xf_icp[t] = b.xf_icp[t];
    else if (t < 24) b.ctrl->xf_rgb[t - 12] = b.xf_rgb[t - 12];
    else if (t == 24) {
      b.ctrl->status = 0;
      b.ctrl->ref_index = 0;
      b.ctrl->margin_acc[0] = b.ctrl->margin_acc[1] = 0u;
    }
  }
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = blockIdx.y * 8 + threadIdx.y;
  if (x >= g.w || y >= g.h) return;
  normal_px<T>(m, 0, g, dmin, dmax, x, y);
  normal_px<T>(m, 1, g, dmin, dmax, x, y);
  gradient_px<T>(m, 0, g.w, g.h, x, y);
  if (flags) flags[y * g.w + x] = 0;
}

template <typename T>
__global__ void k_gradient(LevelMaps m, const Ctrl* __restrict__ ctrl, int w, int h) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= w || y >= h) return;
  gradient_px<T>(m, ctrl->ref_index, w, h, x, y);
}


// ---- uploaded reference (a model prediction rendered at T_ref) ----
// Level 0: per pixel, the vertex and normal moved into the reference camera in
// FP64 (v = R^T (V - r), n = R^T N); a zero normal means no surface (depth 0);
// the normal is kept where the depth is in [dmin, dmax].
template <typename T>
__global__ void k_ref_level0(LevelMaps m, const Ctrl* __restrict__ ctrl, LevelGeom g, float dmin,
                             float dmax, RefUpload up) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= g.w || y >= g.h) return;
  const int set = ctrl->ref_index;
  const int64_t src = (int64_t)y * up.pitch + x;
  const float* V = up.V + 3 * src;
  const float* N = up.N + 3 * src;
  const double vx = (double)__ldg(V) - up.r[0], vy = (double)__ldg(V + 1) - up.r[1],
               vz = (double)__ldg(V + 2) - up.r[2];
  const double nx = __ldg(N), ny = __ldg(N + 1), nz = __ldg(N + 2);
  const bool surf = nx != 0.0 || ny != 0.0 || nz != 0.0;
  const double* R = up.R;
  const float d = surf ? (float)(R[2] * vx + R[5] * vy + R[8] * vz) : 0.f;
  const bool keep = surf && d >= dmin && d <= dmax;
  const float cx = keep ? (float)(R[0] * nx + R[3] * ny + R[6] * nz) : 0.f;
  const float cy = keep ? (float)(R[1] * nx + R[4] * ny + R[7] * nz) : 0.f;
  const float cz = keep ? (float)(R[2] * nx + R[5] * ny + R[8] * nz) : 0.f;
  const int o = y * g.w + x;
  m.depth[set][o] = d;
  m.inten[set][o] = __ldg(up.I + src);
  Packs<T>::store_a(m.packA[set], o, cx, cy, cz, d);
}

// Level l from l - 1 of the reference set: depth (mean of the samples > 0) and
// intensity as for a live frame, the normal as the mean of the non-zero normals
// of the 2x2 block, renormalised, kept where the level's depth is in range.
template <typename T>
__global__ void k_ref_down(LevelMaps fine, LevelMaps coarse, const Ctrl* __restrict__ ctrl, int wf,
                           int wc, int hc, float dmin, float dmax) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= wc || y >= hc) return;
  const int set = ctrl->ref_index;
  pyr_down_px(fine, coarse, set, wf, wc, x, y);
  const int o = y * wc + x;
  const float d = coarse.depth[set][o];
  float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int f = (2 * y + (k >> 1)) * wf + 2 * x + (k & 1);
    const float4 n = Packs<T>::load_a(fine.packA[set], fine.depth[set], f);
    sx += n.x;                                   // zero normals add nothing
    sy += n.y;
    sz += n.z;
  }
  const float n2 = fmaf(sx, sx, fmaf(sy, sy, __fmul_rn(sz, sz)));
  float nx = 0.f, ny = 0.f, nz = 0.f;
  if (n2 > 0.f && d >= dmin && d <= dmax) {
    const float inv = rsqrtf(n2);
    nx = __fmul_rn(sx, inv);
    ny = __fmul_rn(sy, inv);
    nz = __fmul_rn(sz, inv);
  }
  Packs<T>::store_a(coarse.packA[set], o, nx, ny, nz, d);
}

__global__ void k_ref_pose(Ctrl* __restrict__ ctrl, RefUpload up) {
  const int i = threadIdx.x;
  if (i < 9) ctrl->Rref[i] = up.R[i];
  if (i < 3) ctrl->rref[i] = up.r[i];
}

inline dim3 grid2(int w, int h, dim3 b) { return dim3((w + b.x - 1) / b.x, (h + b.y - 1) / b.y); }

}  // namespace

cudaError_t launch_pyramid_batch(const BatchArgs& a, int blocks, cudaStream_t s) {
  k_pyramid_batch<<<blocks, dim3(32, 8), 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_maps_batch(const BatchArgs& a, int blocks, bool fp16, cudaStream_t s) {
  if (fp16) k_maps_batch<__half><<<blocks, dim3(kMapTileW, kMapTileH), 0, s>>>(a);
  else k_maps_batch<float><<<blocks, dim3(kMapTileW, kMapTileH), 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_pair_maps(const LevelMaps& m, const LevelGeom& g, float dmin, float dmax, bool fp16,
                             const PairBegin& begin, uint8_t* flags, cudaStream_t s) {
  const dim3 b(32, 8);
  if (fp16) k_pair_maps<__half><<<grid2(g.w, g.h, b), b, 0, s>>>(m, g, dmin, dmax, begin, flags);
  else k_pair_maps<float><<<grid2(g.w, g.h, b), b, 0, s>>>(m, g, dmin, dmax, begin, flags);
  return cudaGetLastError();
}

}  // namespace dri

namespace dri {

cudaError_t launch_upload_reference(const LevelMaps* m, const LevelGeom* g, int levels, Ctrl* ctrl,
                                    float dmin, float dmax, bool fp16, const RefUpload& up,
                                    cudaStream_t s) {
  const dim3 b(32, 8);
  if (fp16) k_ref_level0<__half><<<grid2(g[0].w, g[0].h, b), b, 0, s>>>(m[0], ctrl, g[0], dmin, dmax, up);
  else k_ref_level0<float><<<grid2(g[0].w, g[0].h, b), b, 0, s>>>(m[0], ctrl, g[0], dmin, dmax, up);
  for (int l = 1; l < levels; ++l) {
    const dim3 gr = grid2(g[l].w, g[l].h, b);
    if (fp16) k_ref_down<__half><<<gr, b, 0, s>>>(m[l - 1], m[l], ctrl, g[l - 1].w, g[l].w, g[l].h, dmin, dmax);
    else k_ref_down<float><<<gr, b, 0, s>>>(m[l - 1], m[l], ctrl, g[l - 1].w, g[l].w, g[l].h, dmin, dmax);
  }
  for (int l = 0; l < levels; ++l) {
    if (fp16) k_gradient<__half><<<grid2(g[l].w, g[l].h, b), b, 0, s>>>(m[l], ctrl, g[l].w, g[l].h);
    else k_gradient<float><<<grid2(g[l].w, g[l].h, b), b, 0, s>>>(m[l], ctrl, g[l].w, g[l].h);
  }
  k_ref_pose<<<1, 32, 0, s>>>(ctrl, up);
  return cudaGetLastError();
}

}  // namespace dri
