// Linearisation of one image pair with no allocation of any kind.
//
// Who needs this: code that may not call cudaMalloc / cudaFree when it runs --
// for example a host framework that owns all device memory and forbids
// allocation inside its per-frame callback, a real-time thread that must not
// block in the allocator, or work recorded while a CUDA stream capture is
// active (allocation calls are illegal there).  Creating a tracking stream
// allocates (its workspace, pinned staging, events), so such code cannot use
// the stream API on the fly.  This entry point takes the caller's device images
// and a caller-owned device output and keeps every intermediate it needs (the
// normal and gradient maps, the pixel kernel's per-block partial sums and its
// completion counter, the per-call transforms, the per-pixel flag bytes before
// they are copied to the caller) in one file-scope static device
// array, held until the process exits.  The array is device memory of the
// library's module: the CUDA runtime reserves it when it loads the module on a
// device, which with lazy module loading (the default since CUDA 12.2) happens
// at the first call made with that device current, so that first call itself
// reserves about 4 MB; later calls reserve nothing.
//
// Limits and rules:
//  * at most kNoallocMaxPixels = 320 * 240 pixels per image; larger images are
//    rejected with DRI_EINVAL before anything is launched;
//  * the static array is shared by every call on a device and keeps the last
//    call's contents; each call re-initialises what must start at zero (the
//    fold counters and the status word) before its kernels run;
//  * calls whose GPU work overlaps (different streams or host threads, without
//    ordering between them) race on the array: order them on one stream;
//  * the device address of the array is looked up once per device, on the first
//    call made with that device current (cudaGetSymbolAddress); make that first
//    call before any stream capture begins.
#include <cmath>
#include <cstring>
#include <mutex>

#include "dri_internal.h"

namespace dri {
namespace {

constexpr int kNoallocMaxW = 320;
constexpr int kNoallocMaxH = 240;
constexpr int64_t kNoallocMaxPixels = (int64_t)kNoallocMaxW * kNoallocMaxH;
constexpr size_t kAlignNA = 256;
constexpr size_t na_align(size_t v) { return (v + kAlignNA - 1) / kAlignNA * kAlignNA; }

constexpr int64_t kPlane = (kNoallocMaxPixels + 63) / 64 * 64;
constexpr size_t kOffCtrl = 0;
constexpr size_t kOffPackA0 = na_align(kOffCtrl + sizeof(Ctrl));       // reference normals + depth
constexpr size_t kOffPackA1 = na_align(kOffPackA0 + kPlane * 16);         // live normals + depth
constexpr size_t kOffPackB = na_align(kOffPackA1 + kPlane * 16);          // reference intensity + gradient
// one row per thread: at most ceil(320/32) * ceil(240/4) blocks
constexpr int kNoallocMaxBlocks = ((kNoallocMaxW + kTrackThreadsX - 1) / kTrackThreadsX) *
                                  ((kNoallocMaxH + kTrackRows - 1) / kTrackRows);
constexpr int kNoallocMaxGroups = (kNoallocMaxBlocks + kFoldGroup - 1) / kFoldGroup;
constexpr size_t kOffCounters = na_align(kOffPackB + kPlane * 16);
constexpr size_t kOffPartials = na_align(kOffCounters + (1 + kNoallocMaxGroups) * sizeof(uint32_t));
constexpr size_t kOffGPartials = na_align(kOffPartials + (size_t)kNoallocMaxBlocks * kSumsAll * sizeof(double));
// per-pixel flag bytes, or-ed in by 32-bit words, then copied to the caller's buffer
constexpr size_t kOffFlags = na_align(kOffGPartials + (size_t)kNoallocMaxGroups * kSumsAll * sizeof(double));
constexpr size_t kNoallocBytes = na_align(kOffFlags + (size_t)kPlane);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
void* g_scratch_addr[kMaxDevices] = {};

// Rotation matrix of a unit quaternion, and the pixel kernel's transform
// (A^T B - I, A^T d) in FP32 exactly as the stream path rounds it.
void quat_to_rot_h(const double* q, double* R) {
  const double w = q[0], x = q[1], y = q[2], z = q[3];
  R[0] = 1 - 2 * (y * y + z * z); R[1] = 2 * (x * y - w * z);     R[2] = 2 * (x * z + w * y);
  R[3] = 2 * (x * y + w * z);     R[4] = 1 - 2 * (x * x + z * z); R[5] = 2 * (y * z - w * x);
  R[6] = 2 * (x * z - w * y);     R[7] = 2 * (y * z + w * x);     R[8] = 1 - 2 * (x * x + y * y);
}
void transform_h(const double* A, const double* B, const double* d, float* xf) {
  for (int i = 0; i < 3; ++i) {
    for (int j = 0; j < 3; ++j) {
      const double m = A[i] * B[j] + A[3 + i] * B[3 + j] + A[6 + i] * B[6 + j];
      xf[3 * i + j] = (float)(m - (i == j ? 1.0 : 0.0));
    }
    xf[9 + i] = (float)(A[i] * d[0] + A[3 + i] * d[1] + A[6 + i] * d[2]);
  }
}

// A state the kernels can use: finite, with a non-zero orientation quaternion.
bool usable_state(const dri_state& s) {
  double nq = 0.0;
  for (int i = 0; i < 4; ++i) nq += s.q_WC[i] * s.q_WC[i];
  if (!(nq > 0.0) || !std::isfinite(nq)) return false;
  for (int i = 0; i < 3; ++i)
    if (!std::isfinite(s.r_WC[i]) || !std::isfinite(s.v_I[i]) || !std::isfinite(s.bg[i]) ||
        !std::isfinite(s.ba[i]))
      return false;
  for (int i = 0; i < 4; ++i)
    if (!std::isfinite(s.q_IW[i])) return false;
  return true;
}

DState dstate_of(const dri_state& s) {
  DState d;
  for (int i = 0; i < 3; ++i) {
    d.r[i] = s.r_WC[i];
    d.v[i] = s.v_I[i];
    d.bg[i] = s.bg[i];
    d.ba[i] = s.ba[i];
  }
  double nq = 0, ng = 0;
  for (int i = 0; i < 4; ++i) {
    nq += s.q_WC[i] * s.q_WC[i];
    ng += s.q_IW[i] * s.q_IW[i];
  }
  nq = sqrt(nq);
  ng = sqrt(ng);
  for (int i = 0; i < 4; ++i) {
    d.q[i] = s.q_WC[i] / nq;
    d.qg[i] = ng > 0 ? s.q_IW[i] / ng : (i == 0 ? 1.0 : 0.0);
  }
  return d;
}

// Device address of the static array for the current device, looked up once.
int scratch_address(unsigned char** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return DRI_ECUDA;
  if (dev < 0 || dev >= kMaxDevices) return DRI_EINVAL;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || p == nullptr) return DRI_ECUDA;
    g_scratch_addr[dev] = p;
  }
  *out = static_cast<unsigned char*>(g_scratch_addr[dev]);
  return DRI_OK;
}

}  // namespace
}  // namespace dri

using namespace dri;

extern "C" int dri_linearise_pair_noalloc(const dri_stream_config* cfg, const float* ref_depth,
                                          const float* ref_intensity, const float* live_depth,
                                          const float* live_intensity, const dri_state* x_ref,
                                          const dri_state* x0, const dri_state* x1,
                                          dri_linearisation* out, uint8_t* flags, void* cuda_stream) {
  if (!cfg || !ref_depth || !ref_intensity || !live_depth || !live_intensity || !x_ref || !x0 ||
      !x1 || !out)
    return DRI_EINVAL;
  if (cfg->width < 8 || cfg->height < 8 || cfg->width > kNoallocMaxW || cfg->height > kNoallocMaxH ||
      (int64_t)cfg->width * cfg->height > kNoallocMaxPixels)
    return DRI_EINVAL;
  if (!(cfg->fx > 0) || !(cfg->fy > 0) || !(cfg->sigma_I > 0) || !(cfg->sigma_d > 0) ||
      !(cfg->depth_max > cfg->depth_min) || !(cfg->icp_dist_thr > 0) ||
      !(cfg->icp_angle_thr_deg > 0) || !(cfg->icp_angle_thr_deg < 90))
    return DRI_EINVAL;
  if ((cfg->precision_flags & ~(DRI_FP16_MAPS | DRI_FP32_PARTIALS)) != 0 ||
      !(cfg->occlusion_thr >= 0.0) || !std::isfinite(cfg->occlusion_thr) ||
      (cfg->icp_depth_weight != 0 && cfg->icp_depth_weight != 1))
    return DRI_EINVAL;
  if (!usable_state(*x_ref) || !usable_state(*x0) || !usable_state(*x1)) return DRI_EINVAL;
  const bool fp16 = (cfg->precision_flags & DRI_FP16_MAPS) != 0;
  const bool fp32p = (cfg->precision_flags & DRI_FP32_PARTIALS) != 0;
  unsigned char* base = nullptr;
  const int r = scratch_address(&base);
  if (r != DRI_OK) return r;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Ctrl* ctrl = reinterpret_cast<Ctrl*>(base + kOffCtrl);

  LevelGeom g = level_geom(*cfg, 0);
  LevelMaps m;
  std::memset(&m, 0, sizeof(m));
  m.depth[0] = const_cast<float*>(ref_depth);      // set 0: reference
  m.inten[0] = const_cast<float*>(ref_intensity);
  m.depth[1] = const_cast<float*>(live_depth);     // set 1: live frame
  m.inten[1] = const_cast<float*>(live_intensity);
  m.packA[0] = base + kOffPackA0;
  m.packA[1] = base + kOffPackA1;
  m.packB[0] = base + kOffPackB;
  m.packB[1] = base + kOffPackB;                    // the live set's pack B is never read

  uint32_t* counters = reinterpret_cast<uint32_t*>(base + kOffCounters);
  // transforms of the pixel kernel from (x_ref, x0, x1), as the stream path computes them
  const DState dref = dstate_of(*x_ref), d0 = dstate_of(*x0), d1 = dstate_of(*x1);
  PairBegin begin;
  PairEnd end;
  double R1[9], dr[3];
  quat_to_rot_h(dref.q, end.Rref);
  quat_to_rot_h(d0.q, end.R0);
  quat_to_rot_h(d1.q, R1);
  for (int i = 0; i < 3; ++i) dr[i] = d1.r[i] - dref.r[i];
  transform_h(end.Rref, R1, dr, begin.xf_icp);
  for (int i = 0; i < 3; ++i) dr[i] = d1.r[i] - d0.r[i];
  transform_h(end.R0, R1, dr, begin.xf_rgb);
  begin.ctrl = ctrl;
  begin.counters = counters;
  begin.ncounters = 1 + kNoallocMaxGroups;
  end.W_icp = 1.0 / (cfg->sigma_d * cfg->sigma_d);
  end.W_rgb = 1.0 / (cfg->sigma_I * cfg->sigma_I);
  end.out = out;
  const float dmin = (float)cfg->depth_min, dmax = (float)cfg->depth_max;
  uint8_t* fl = flags ? base + kOffFlags : nullptr;
  if (launch_pair_maps(m, g, dmin, dmax, fp16, begin, fl, s) != cudaSuccess) return DRI_ECUDA;

  TrackParams p;
  std::memset(&p, 0, sizeof(p));
  p.g = g;
  p.m = m;
  p.ctrl = ctrl;
  p.partials = base + kOffPartials;
  p.gpartials = base + kOffGPartials;
  p.counters = counters;
  p.flags = fl;
  p.ppt = 1;
  p.nblocks = track_mixed_blocks(g.w, g.h, 1);
  if (p.nblocks > kNoallocMaxBlocks) return DRI_EINVAL;
  p.depth_min = dmin;
  p.depth_max = dmax;
  p.icp_dist2 = (float)(cfg->icp_dist_thr * cfg->icp_dist_thr);
  p.icp_cos = (float)std::cos(cfg->icp_angle_thr_deg * 3.14159265358979323846 / 180.0);
  p.occ_thr = (float)cfg->occlusion_thr;
  p.icp_dw = cfg->icp_depth_weight;
  if (launch_track(p, end, fp16, fp32p, s) != cudaSuccess) return DRI_ECUDA;
  if (flags && cudaMemcpyAsync(flags, p.flags, (size_t)g.w * g.h, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return DRI_ECUDA;
  return DRI_OK;
}
