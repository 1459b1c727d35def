// libdrr kernels: pose/ray setup, incremental Siddon traversal (forward,
// fused pose Jacobian, pose-gradient re-trace, back-projection), the
// deterministic pose-gradient reduction and volume ingest.
//
// Paper: Gopalakrishnan & Golland, arXiv 2208.12737.
//   Eq. (2)  radiologic path length E = |p-s| sum (a_{m+1}-a_m) V[midpoint voxel]
//   Eq. (3)  plane crossings a_x(i) = (b_x + i dX - s_x) / (p_x - s_x)
//   Sec. 2.2 Siddon-Jacobs: the next crossing is the minimum over the axes of
//            each axis' next plane, iterated until the ray leaves the volume
//   Sec. 2.3 entry/exit clip a_min / a_max
//   Sec. 2.4 pose parameterisation and differentiation w.r.t. the pose
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "drr_internal.cuh"

namespace drr {
namespace {

enum Mode : int { kFwd = 0, kFwdJac = 1, kPoseGrad = 2, kBackproject = 3, kCount = 4, kGeoGrad = 5 };

template <int DT>
struct Voxel;
template <>
struct Voxel<kF32> {
  static __device__ __forceinline__ float load(const void* base, int off) {
    return __ldg(static_cast<const float*>(base) + off);
  }
};
template <>
struct Voxel<kBF16> {
  static __device__ __forceinline__ float load(const void* base, int off) {
    const unsigned short u = __ldg(static_cast<const unsigned short*>(base) + off);
    return __uint_as_float(static_cast<unsigned int>(u) << 16);
  }
};
template <>
struct Voxel<kF16> {
  static __device__ __forceinline__ float load(const void* base, int off) {
    return __half2float(__ldg(static_cast<const __half*>(base) + off));
  }
};

// Bounds-checked build (-DDRR_CHECK_BOUNDS=1, a separate library built for
// tests): every voxel gather is checked against the padded volume and every
// back-projection add of a live segment against the gradient volume, but for
// segments shorter than the rounding of their ends (walk_backproject); a check
// that fails sets a bit of a device-wide fault word (read and cleared by
// drr_stream_check, which then returns DRR_ERR_DEVICE) and skips the access.
// The product build has no checks: the zero padding keeps every gather of the
// walk in bounds, which the checked build verifies on the parity workloads.
#ifndef DRR_CHECK_BOUNDS
#define DRR_CHECK_BOUNDS 0
#endif
enum FaultBits : unsigned int { kFaultGather = 1u, kFaultBackproject = 2u };
#if DRR_CHECK_BOUNDS
__device__ unsigned int g_fault_word = 0u;
#endif
template <int DT>
__device__ __forceinline__ float gather(const VolumeDev& vd, int off) {
#if DRR_CHECK_BOUNDS
  if (static_cast<unsigned long long>(static_cast<long long>(off)) >= static_cast<unsigned long long>(vd.elems)) {
    atomicOr(&g_fault_word, kFaultGather);
    return 0.f;
  }
#endif
  return Voxel<DT>::load(vd.data, off);
}

// The voxel d elements after offset off: base_d is the volume's base moved by d
// elements (kept in registers, so the second gather of a pair costs no offset
// addition).
template <int DT>
__device__ __forceinline__ float gather_at(const VolumeDev& vd, const void* base_d, int off, int d) {
#if DRR_CHECK_BOUNDS
  return gather<DT>(vd, off + d);
#else
  return Voxel<DT>::load(base_d, off);
#endif
}
template <int DT>
__device__ __forceinline__ const void* base_after(const VolumeDev& vd, int d) {
  return static_cast<const char*>(vd.data) + static_cast<int64_t>(d) * (DT == kF32 ? 4 : 2);
}

// x_a for a runtime axis index without indexing a register array (which
// would move the array to local memory).
template <class T>
__device__ __forceinline__ T pick3(int a, T x0, T x1, T x2) {
  return a == 0 ? x0 : (a == 1 ? x1 : x2);
}

// Programmatic dependent launch (sm_90 and later).  The pose-setup, walk and
// gradient-reduction kernels are launched with programmatic stream
// serialization, so each can be scheduled while the kernel before it in the
// stream is still finishing.  grid_dep_wait() blocks until that kernel has
// completed and its writes are visible; each of these kernels calls it before
// its first global-memory access (read or write).  grid_dep_release() lets the
// next kernel in the stream be scheduled early; its blocks then wait in their
// own grid_dep_wait().  Both are no-ops for a kernel launched without the
// attribute.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_release() { asm volatile("griddepcontrol.launch_dependents;" :::); }

// ---------------------------------------------------------------------------
// Pose -> frame (Sec. 2.4).  R = Rz(eta0) Ry(eta1) Rx(eta2).
// ---------------------------------------------------------------------------
// World-space frame of one pose: source s, pixel (0,0) centre p00, the
// per-column and per-row pixel steps ew, eh (all FP64), and optionally R and
// the sines / cosines of the three angles.  R = Rz Ry Rx written out.
__device__ void pose_frame(const float* pose, const DetDev& det, double s[3], double p00[3], double ew[3],
                           double eh[3], double sc_out[3], double pc00_out[3], double* R_out /*9 or null*/,
                           float* sincos_out /*6 or null: sz, cz, sy, cy, sx, cx*/) {
  double sz, cz, sy, cy, sx, cx;
  sincos(static_cast<double>(pose[0]), &sz, &cz);
  sincos(static_cast<double>(pose[1]), &sy, &cy);
  sincos(static_cast<double>(pose[2]), &sx, &cx);
  const double szsy = sz * sy, czsy = cz * sy;
  const double R[9] = {cz * cy, fma(czsy, sx, -sz * cx), fma(czsy, cx, sz * sx),
                       sz * cy, fma(szsy, sx, cz * cx),  fma(szsy, cx, -cz * sx),
                       -sy,     cy * sx,                 cy * cx};
  const double rho = 0.5 * static_cast<double>(det.sdr);
  const double pw = -0.5 * static_cast<double>(det.W - 1) * static_cast<double>(det.dw);
  const double ph = -0.5 * static_cast<double>(det.H - 1) * static_cast<double>(det.dh);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double t = static_cast<double>(pose[3 + a]);
    s[a] = fma(rho, R[3 * a], t);                                              // R (rho, 0, 0) + t
    p00[a] = fma(ph, R[3 * a + 2], fma(pw, R[3 * a + 1], fma(-rho, R[3 * a], t)));  // R pc00 + t
    ew[a] = static_cast<double>(det.dw) * R[3 * a + 1];                         // R (0, dw, 0)
    eh[a] = static_cast<double>(det.dh) * R[3 * a + 2];                         // R (0, 0, dh)
  }
  sc_out[0] = rho;
  sc_out[1] = sc_out[2] = 0.0;
  pc00_out[0] = -rho;
  pc00_out[1] = pw;
  pc00_out[2] = ph;
  if (R_out) {
#pragma unroll
    for (int i = 0; i < 9; ++i) R_out[i] = R[i];
  }
  if (sincos_out) {
    sincos_out[0] = static_cast<float>(sz);
    sincos_out[1] = static_cast<float>(cz);
    sincos_out[2] = static_cast<float>(sy);
    sincos_out[3] = static_cast<float>(cy);
    sincos_out[4] = static_cast<float>(sx);
    sincos_out[5] = static_cast<float>(cx);
  }
}

__device__ void mul3f(const float* A, const float* B, float* C) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) C[3 * r + c] = fmaf(A[3 * r], B[c], fmaf(A[3 * r + 1], B[3 + c], A[3 * r + 2] * B[6 + c]));
}

__device__ void apply3f(const float* A, const float* x, float* y) {
#pragma unroll
  for (int r = 0; r < 3; ++r) y[r] = fmaf(A[3 * r], x[0], fmaf(A[3 * r + 1], x[1], A[3 * r + 2] * x[2]));
}

// FP32 chain-rule terms of one angle j of a pose (dR/d eta_j applied to s_c, p_c -
// s_c and the pixel steps), from the FP32-rounded sines and cosines: they are
// stored as FP32.  One lane per angle: dR_j is the product of the three rotations
// with the j-th replaced by its derivative.
__device__ void chain_terms(int j, const float cs[6], double rho, double pw, double ph, const DetDev& det, PoseGeom* g) {
  const float sz = cs[0], cz = cs[1], sy = cs[2], cy = cs[3], sx = cs[4], cx = cs[5];
  const bool d0 = j == 0, d1 = j == 1, d2 = j == 2;
  // [c -s; s c] or its derivative [-s -c; c -s], embedded in the rotation's plane
  const float zc = d0 ? -sz : cz, zs = d0 ? cz : sz, z1 = d0 ? 0.f : 1.f;
  const float yc = d1 ? -sy : cy, ys = d1 ? cy : sy, y1 = d1 ? 0.f : 1.f;
  const float xc = d2 ? -sx : cx, xs = d2 ? cx : sx, x1 = d2 ? 0.f : 1.f;
  const float Z[9] = {zc, -zs, 0.f, zs, zc, 0.f, 0.f, 0.f, z1};
  const float Y[9] = {yc, 0.f, ys, 0.f, y1, 0.f, -ys, 0.f, yc};
  const float X[9] = {x1, 0.f, 0.f, 0.f, xc, -xs, 0.f, xs, xc};
  float T[9], dR[9];
  mul3f(Z, Y, T);
  mul3f(T, X, dR);
  // angular velocity of the angle in the world frame, dR_j R^T x = omega_j x x:
  // rz turns about e_z, ry about Rz e_y, rx about Rz Ry e_x
  g->Om[j][0] = d0 ? 0.f : (d1 ? -sz : cz * cy);
  g->Om[j][1] = d0 ? 0.f : (d1 ? cz : sz * cy);
  g->Om[j][2] = d0 ? 1.f : (d1 ? 0.f : -sy);
  const float q[3] = {static_cast<float>(-2.0 * rho), static_cast<float>(pw), static_cast<float>(ph)};
  const float vw[3] = {0.f, det.dw, 0.f};
  const float vh[3] = {0.f, 0.f, det.dh};
  apply3f(dR, q, g->Q[j]);
  apply3f(dR, vw, g->Wv[j]);
  apply3f(dR, vh, g->Hv[j]);
}

// Per-pose geometry in the volume's voxel units plus the chain-rule terms,
// computed by a whole warp and written to *g.  The three FP64 sine/cosine pairs
// run in lanes 0-2 and the per-axis terms in lanes 0-2: FP64 issue is narrow on
// this GPU, and spreading the serial FP64 work over lanes shortens the kernel.
// The arithmetic per value is that of pose_frame.
__device__ void warp_pose_geom(const float* pose, const DetDev& det, const VolumeDev& vd, PoseGeom* g) {
  constexpr unsigned int kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  double sv = 0.0, cv = 1.0;
  if (lane < 3) sincos(static_cast<double>(pose[lane]), &sv, &cv);
  const double sz = __shfl_sync(kFull, sv, 0), cz = __shfl_sync(kFull, cv, 0);
  const double sy = __shfl_sync(kFull, sv, 1), cy = __shfl_sync(kFull, cv, 1);
  const double sx = __shfl_sync(kFull, sv, 2), cx = __shfl_sync(kFull, cv, 2);
  const double szsy = sz * sy, czsy = cz * sy;
  const double R[9] = {cz * cy, fma(czsy, sx, -sz * cx), fma(czsy, cx, sz * sx),
                       sz * cy, fma(szsy, sx, cz * cx),  fma(szsy, cx, -cz * sx),
                       -sy,     cy * sx,                 cy * cx};
  const double rho = 0.5 * static_cast<double>(det.sdr);
  const double pw = -0.5 * static_cast<double>(det.W - 1) * static_cast<double>(det.dw);
  const double ph = -0.5 * static_cast<double>(det.H - 1) * static_cast<double>(det.dh);
  if (lane < 3) {
    const int a = lane;
    const double r0 = pick3(a, R[0], R[3], R[6]), r1 = pick3(a, R[1], R[4], R[7]), r2 = pick3(a, R[2], R[5], R[8]);
    const double t = static_cast<double>(pose[3 + a]);
    const double s = fma(rho, r0, t);                                  // R (rho, 0, 0) + t
    const double p00 = fma(ph, r2, fma(pw, r1, fma(-rho, r0, t)));     // R pc00 + t
    const double ew = static_cast<double>(det.dw) * r1;                 // R (0, dw, 0)
    const double eh = static_cast<double>(det.dh) * r2;                 // R (0, 0, dh)
    const double dl = static_cast<double>(pick3(a, vd.delta[0], vd.delta[1], vd.delta[2])), rd = 1.0 / dl;
    const int na = pick3(a, vd.n[0], vd.n[1], vd.n[2]);
    const double lo = -0.5 * static_cast<double>(na) * dl;  // b_a: volume centred at the origin
    const double u0 = (s - lo) * rd;
    const double un = static_cast<double>(na) - u0;
    g->u0[a] = u0;
    g->un[a] = un;
    g->u0f[a] = static_cast<float>(u0);
    g->unf[a] = static_cast<float>(un);
    g->g00[a] = (p00 - s) * rd;
    g->gw[a] = ew * rd;
    g->gh[a] = eh * rd;
  }
  // columns of R (R e_x, R e_y, R e_z) for the detector-parameter chain
#pragma unroll
  for (int i = 0; i < 9; ++i)
    if (lane == i) g->Rc[i % 3][i / 3] = static_cast<float>(R[i]);
  if (lane < 3) {
    const float cs[6] = {static_cast<float>(sz), static_cast<float>(cz), static_cast<float>(sy),
                         static_cast<float>(cy), static_cast<float>(sx), static_cast<float>(cx)};
    g->t[lane] = pose[3 + lane];
    chain_terms(lane, cs, rho, pw, ph, det, g);
  }
  if (lane == 3) {
    g->hc = 0.5f * static_cast<float>(det.H - 1);
    g->wc = 0.5f * static_cast<float>(det.W - 1);
  }
}

// One warp (block) per pose.
__global__ void __launch_bounds__(32) pose_setup_kernel(const float* __restrict__ poses, int B, DetDev det,
                                                        VolumeDev vd, PoseGeom* __restrict__ out) {
  grid_dep_wait();
  grid_dep_release();
  const int b = blockIdx.x;
  // the walk kernels' tile counters live in the slot after the last pose
  if (b == 0 && threadIdx.x < kLaunchCounters) reinterpret_cast<unsigned int*>(out + B)[threadIdx.x] = 0u;
  if (b >= B) return;
  warp_pose_geom(poses + 6 * b, det, vd, out + b);
}

__global__ void ray_setup_kernel(const float* __restrict__ poses, int B, DetDev det, float* __restrict__ rays) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t npix = static_cast<int64_t>(det.H) * det.W;
  if (i >= npix * B) return;
  const int b = static_cast<int>(i / npix);
  const int q = static_cast<int>(i % npix);
  const int h = q / det.W, w = q % det.W;
  double s[3], p00[3], ew[3], eh[3], sc[3], pc00[3];
  pose_frame(poses + 6 * b, det, s, p00, ew, eh, sc, pc00, nullptr, nullptr);
  float* r = rays + 6 * i;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r[a] = static_cast<float>(s[a]);
    r[3 + a] = static_cast<float>(fma(static_cast<double>(h), eh[a], fma(static_cast<double>(w), ew[a], p00[a])));
  }
}

// ---------------------------------------------------------------------------
// One ray: the FP64 clip and entry (Sec. 2.3) of the rays that slab_setup cannot
// decide, and of the segment count.
// ---------------------------------------------------------------------------
struct RayResult {
  float F;     // E
  float J[6];  // dE/d eta (only for the Jacobian modes)
};

// Per-ray state after the FP64 setup, for exact_rays, backproject_exact and the
// segment count (mode kCount).
//
// Crossing parameters are fixed point: alpha measured from the entry is held
// as a 32.32 number in units of span / 2^24 (span = alpha_max - alpha_min), so
// the high word of every crossing inside the ray lies in [0, 2^24] and the
// exit is exactly 2^24; every value the walk forms stays below 2^58.  Each
// axis' crossings form the arithmetic sequence first + k * delta (Eq. 3),
// advanced by exact 64-bit additions: ordering is exact to 2^-56 of the span
// and segment lengths are exact integers, so the FP32 arithmetic is confined
// to the accumulation of length x density.  (A high word below 2^24 converts
// to FP32 exactly; see fix_to_float.)
struct RaySetup {
  int nseg;                  // segments = plane crossings + 1 (0: the ray misses)
  int off;                   // element offset of the entry voxel (padded layout)
  int ient[3];               // entry voxel index per axis
  int cnt[3];                // plane crossings per axis between the entry and exit voxels
  int step[3];               // signed element stride per axis
  int ea, xa;                // axis of the entry / exit plane, -1 when clamped to alpha = 0 / 1
  unsigned long long A0[3];  // first crossing per axis (32.32 fixed point)
  unsigned long long D[3];   // fixed-point distance between consecutive planes
  float unit;                // alpha per high-word unit: span / 2^24
  double amin;               // absolute alpha of the entry
  float d[3];                // p - s in mm
};

constexpr unsigned int kExitUnits = 1u << 24;              // the exit, in high-word units
constexpr unsigned long long kFixMax = 1ull << 56;         // fixed-point value of the exit
constexpr unsigned long long kNoCrossing64 = 1ull << 58;  // beyond any crossing of the ray
constexpr double kFixScale = 72057594037927936.0;          // 2^56: fixed-point value of alpha = span

// Reciprocal of a double to ~1e-14 relative: an FP32 seed refined by one FP64
// Newton step (a full FP64 division costs several times more on the FP64 pipe,
// which is narrow on this GPU).  Exact division outside the FP32 seed's range.
__device__ __forceinline__ double rcp_fast(double x) {
  const float xf = static_cast<float>(x);
  const float ax = fabsf(xf);
  if (!(ax > 1e-30f && ax < 1e30f)) return 1.0 / x;
  const double r = static_cast<double>(__frcp_rn(xf));
  return fma(r, fma(-x, r, 1.0), r);
}

// floor of a double: in FP32 unless the value is within 2^-10 of an integer
// (or too large for FP32 to resolve that), where FP64 decides.
__device__ __forceinline__ int floor_fast(double x) {
  const float xf = static_cast<float>(x);
  const float fl = floorf(xf);
  const float fr = xf - fl;
  if (fabsf(xf) < 4096.f && fr > 9.765625e-4f && fr < 1.f - 9.765625e-4f) return static_cast<int>(fl);
  return static_cast<int>(floor(x));
}

// FP64 clip (Sec. 2.3, clamped to [0, 1]).  The faces the ray enters and leaves
// through are found in FP32 (in FP64 where FP32 cannot tell them apart);
// alpha_min / alpha_max are then evaluated in FP64 on those faces.  Returns 1
// for a hit, 0 when the ray misses, -1 for non-finite geometry.
struct RayClip {
  double g[3], rg[3];  // direction in voxel units and its reciprocals (0 for a parallel axis)
  float gf[3];
  double amin, amax;
  int ea, xa;  // axis of the entry / exit plane, -1 when clamped to alpha = 0 / 1
};
__device__ __forceinline__ int clip_ray(const PoseGeom& pg, int h, int w, RayClip& c) {
  double* g = c.g;
  float* gf = c.gf;
  double* rg = c.rg;
  bool finite = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    g[a] = fma(static_cast<double>(h), pg.gh[a], fma(static_cast<double>(w), pg.gw[a], pg.g00[a]));
    gf[a] = static_cast<float>(g[a]);
    finite = finite && isfinite(gf[a]) && isfinite(pg.u0f[a]);
  }
  if (!finite) return -1;
  // faces in FP32; a choice that FP32 cannot make safely -- the runner-up
  // crossing (or the clamp at alpha 0 / 1) within 2^-20 of the chosen one, four
  // times the FP32 error of these products, or a hit test that close -- is
  // made again in FP64.  That matters where the clipped span is a small part of
  // alpha (a small volume far from the source): there an FP32 tie moves the
  // entry by a visible share of the span.
  float lof = 0.f, hif = 1.f, lo2 = -1.f, hi2 = 2.f;  // chosen and runner-up entry / exit
  int ea = -1, xa = -1;
  bool hit = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (g[a] != 0.0) {
      const float rf = __frcp_rn(gf[a]);
      const float t0 = -pg.u0f[a] * rf, t1 = pg.unf[a] * rf;
      const float lo = fminf(t0, t1), hi = fmaxf(t0, t1);
      if (lo > lof) { lo2 = lof; lof = lo; ea = a; } else lo2 = fmaxf(lo2, lo);
      if (hi < hif) { hi2 = hif; hif = hi; xa = a; } else hi2 = fminf(hi2, hi);
    } else if (!(pg.u0[a] >= 0.0 && pg.un[a] > 0.0)) {
      hit = false;
    }
  }
  if (!hit) return 0;
  const float tol = 9.5367431640625e-7f * fmaxf(fabsf(lof), fabsf(hif)) + 1e-30f;  // 2^-20
  const bool exact = lof - lo2 < tol || hi2 - hif < tol || fabsf(hif - lof) < tol;
  if (!exact && !(lof < hif)) return 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) rg[a] = g[a] != 0.0 ? rcp_fast(g[a]) : 0.0;
  // entry / exit faces: plane 0 when the ray runs up the axis, plane n otherwise
  double amin = 0.0, amax = 1.0;
  if (exact) {
    ea = xa = -1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (g[a] != 0.0) {
        const double en = (g[a] > 0.0 ? -pg.u0[a] : pg.un[a]) * rg[a];
        const double ex = (g[a] > 0.0 ? pg.un[a] : -pg.u0[a]) * rg[a];
        if (en > amin) { amin = en; ea = a; }
        if (ex < amax) { amax = ex; xa = a; }
      }
    }
  } else {
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // static indices: the arrays stay in registers
      if (a == ea) amin = (g[a] > 0.0 ? -pg.u0[a] : pg.un[a]) * rg[a];
      if (a == xa) amax = (g[a] > 0.0 ? pg.un[a] : -pg.u0[a]) * rg[a];
    }
  }
  if (!(amin < amax)) return 0;
  c.ea = ea;
  c.xa = xa;
  c.amin = amin;
  c.amax = amax;
  return 1;
}

// Voxels in which the ray enters and leaves along one axis (entry and exit
// positions ue, ux in voxel units).
__device__ __forceinline__ void axis_voxels(const RayClip& c, int a, int n, double ue, double ux, int& i0, int& i1) {
  const bool up = c.g[a] > 0.0;
  if (a == c.ea) i0 = up ? 0 : n - 1;
  else i0 = up ? floor_fast(ue) : -floor_fast(-ue) - 1;
  if (a == c.xa) i1 = up ? n - 1 : 0;
  else i1 = up ? -floor_fast(-ux) - 1 : floor_fast(ux);
  i0 = min(max(i0, 0), n - 1);
  i1 = min(max(i1, 0), n - 1);
}

// The exact crossing sequences of one ray (the fixed-point form of RaySetup),
// from the FP64 clip.  Returns as clip_ray.
__device__ __forceinline__ int ray_setup(const VolumeDev& vd, const PoseGeom& pg, int h, int w, RaySetup& r) {
  r.nseg = 0;
  RayClip c;
  const int hit = clip_ray(pg, h, w, c);
  if (hit <= 0) return hit;
  const double* g = c.g;
  const double* rg = c.rg;
  r.ea = c.ea;
  r.xa = c.xa;
  r.amin = c.amin;
  const double span = c.amax - c.amin;
  const double to_fix = kFixScale * rcp_fast(span);  // fixed-point units per unit of alpha
  r.unit = static_cast<float>(span) * (1.f / static_cast<float>(kExitUnits));
  int total = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int n = vd.n[a];
    r.d[a] = c.gf[a] * vd.delta[a];
    const double ue = fma(c.amin, g[a], pg.u0[a]);
    if (g[a] == 0.0) {
      r.ient[a] = min(max(static_cast<int>(floor(pg.u0[a])), 0), n - 1);
      r.cnt[a] = 0;
      r.A0[a] = kNoCrossing64;
      r.D[a] = 0ull;
      r.step[a] = vd.stride[a];
      continue;
    }
    const bool up = g[a] > 0.0;
    int i0, i1;
    axis_voxels(c, a, n, ue, fma(c.amax, g[a], pg.u0[a]), i0, i1);
    r.ient[a] = i0;
    r.cnt[a] = max(up ? i1 - i0 : i0 - i1, 0);
    total += r.cnt[a];
    const double plane = static_cast<double>(up ? i0 + 1 : i0);
    // first crossing, kept within [0, span] (rounding can put it a hair outside)
    const double f = fmax((plane - ue) * rg[a], 0.0);
    r.A0[a] = r.cnt[a] > 0 ? min(__double2ull_rz(f * to_fix), kFixMax) : kNoCrossing64;
    // plane spacing, saturated at the span: an axis whose planes are farther
    // apart has at most one crossing, and one step past it stays below 2^57
    r.D[a] = min(__double2ull_rz(fabs(rg[a]) * to_fix), kFixMax);
    r.step[a] = up ? vd.stride[a] : -vd.stride[a];
  }
  r.nseg = total + 1;
  r.off = vd.origin + r.ient[0] * vd.stride[0] + r.ient[1] * vd.stride[1] + r.ient[2] * vd.stride[2];
  return 1;
}

// ---------------------------------------------------------------------------
// Fixed-point crossing sequences.  The exact positions are first + k * delta in
// 64-bit; the back-projection's per-segment arithmetic runs in FP32 on positions
// measured from a nearby origin, recomputed exactly at the start of every chunk
// of crossings, so local positions stay below ~chunk plane gaps and carry 2^-24
// of the chunk.  Positions are in fixed-point high-word units (span / 2^24).
// ---------------------------------------------------------------------------
#ifndef DRR_FWD_MINB
#define DRR_FWD_MINB 4
#endif
#ifndef DRR_BP_MINB
#define DRR_BP_MINB 4
#endif
#ifndef DRR_JAC_MINB
#define DRR_JAC_MINB 3
#endif
constexpr float kTwoM32 = 2.3283064365386963e-10f;  // 2^-32

__device__ __forceinline__ unsigned long long fix_at(unsigned long long A0, unsigned long long D, unsigned int k) {
  return A0 + static_cast<unsigned long long>(k) * D;
}

// FP32 value (high-word units) of a signed 32.32 fixed-point number, from two
// 32-bit conversions (a 64-bit conversion would run on the FP64 pipe, which is
// narrow on this GPU).  For |d| < 2^56 -- every position within a ray, every
// plane spacing -- the high word converts exactly, so the result carries one
// rounding (2^-24 relative) plus at most 2^-25 units from the low word.
__device__ __forceinline__ float fix_to_float(long long d) {
  return fmaf(static_cast<float>(static_cast<unsigned int>(d)), kTwoM32, static_cast<float>(static_cast<int>(d >> 32)));
}

// Next crossings of two axes, l * delta + x0 each, in one packed two-lane FP32
// FMA (each lane rounded as fmaf rounds it, so the results are the same);
// -DDRR_PACKED_XY=0 issues two scalar FMAs.
#ifndef DRR_PACKED_XY
#define DRR_PACKED_XY 1
#endif
__device__ __forceinline__ void next_xy(float& tx, float& ty, float lx, float ly, float dx, float dy, float x0,
                                        float y0) {
#if DRR_PACKED_XY
  const float2 t = __ffma2_rn(make_float2(lx, ly), make_float2(dx, dy), make_float2(x0, y0));
  tx = t.x;
  ty = t.y;
#else
  tx = fmaf(lx, dx, x0);
  ty = fmaf(ly, dy, y0);
#endif
}

// Local FP32 position of an exact position relative to O.
__device__ __forceinline__ float local_pos(unsigned long long x, unsigned long long O) {
  return fix_to_float(static_cast<long long>(x - O));
}

// ---------------------------------------------------------------------------
// Slab walk (Eq. 2 by the crossings of each axis on their own; the crossings
// are those of Eq. 3, Sec. 2.2).  With the axis of the largest direction
// component as the dominant one, its planes cut the ray into slabs of equal
// length, and
//   E = sum over slabs V[voxel the slab is entered in] * slab length
//     + sum over the minor axes' crossings (V after - V before) * (slab end - crossing),
// so nothing has to be merged in order: each axis' crossings are one counted
// loop, whose iterations are independent (the loads of several are in flight
// at once) and need no minimum, no ordering compares and no carried weights.
// The pose Jacobian's per-axis sums (Sec. 2.4) of w = V before - V after and of
// w times its position are those of the two minor loops; the dominant axis'
// follow from sum w = 0 and sum w alpha = F over all crossings.
// Measured (fused forward + Jacobian kernel, FP32, CUDA events): 16-pose CT
// batch, 512x512x133 and 200x200, 0.559 -> 0.421 ms against the walk that merged
// the axes' crossings in order (429 -> 259 M warp instructions); 150x141 on 256^3
// split over the warps of a tile, 0.067 -> 0.042 ms.  What bounds it now is the L1
// data pipe (81 % busy): the dominant loop's gathers touch ~15 lines each (rays of
// a tile at one plane x = const of an x-fastest volume), ~5 wavefronts.  Taking
// 2 x 4 rays and 4 planes per gather (35 instead of 50 M wavefronts but more L2
// sectors, 0.469 ms), the three loops interleaved in chunks (0.505), and a second
// copy of the volume with another fastest axis (17 M wavefronts, but every
// gather an L2 access and 0.74 GB from DRAM: 0.446) were slower.  The forward
// alone keeps the merged walk: it gathers once per segment, the slab walk once
// per slab and twice per minor crossing (0.391 ms when the merged one took 0.366; it
// takes 0.344 now).
//
// Coordinates run in the ray's direction on every axis, from the entry voxel's
// lower plane: q_a in [0, 1] at the entry, crossing k of axis a at q_a = 1 + k.
// Positions are 32.32 fixed point.  Slot 2 is the dominant axis, 0 and 1 the
// others (by decreasing direction).  The voxel that a crossing lies in is read
// off the integer parts of the other axes' coordinates at it; the two views of
// a pair of crossings (each in the other's loop) agree unless the pair is closer
// than the rounding of these coordinates.  A minor loop's smallest fractional
// distance to a plane is tracked against a bound on that rounding (SlabRay::t0,
// t1), piece by piece, and settle_pairs puts the pairs below it in exact order.
//
// The loops are cut into up to kPieces pieces of whole plane ranges, the same
// planes for the warp's 32 rays (so rays of one tile gather from the same plane
// at a time), and the pieces' sums are added in order: the split kernel, whose
// warps take different pieces, gives the same bits.
// ---------------------------------------------------------------------------
// Measured in one run (us; lone 150x141 on 256^3, CT batch, 4 poses of 509x451 on 512x512x300 BF16):
// pieces of 32 planes, 8 of them, 8 slabs and 4 minor crossings in flight 42 / 428 / 618;
// pieces of 16 or 64 the same; 4 pieces 43 / 426 / 605, but twice as many planes to look
// through for a pair (settle_pairs) and half the warps of a split tile idle; 4 slabs in
// flight 42 / 464 / 655, 16 41 / 421 / 622; 2 minor crossings 43 / 454 / 678, 8 43 / 443 / 647.
#ifndef DRR_PIECE_LEN
#define DRR_PIECE_LEN 32
#endif
#ifndef DRR_PIECES
#define DRR_PIECES 8
#endif
constexpr int kPieces = DRR_PIECES, kPieceLen = DRR_PIECE_LEN;
#ifndef DRR_SLAB_UNROLL
#define DRR_SLAB_UNROLL 8
#endif
#ifndef DRR_MINOR_UNROLL
#define DRR_MINOR_UNROLL 4
#endif
constexpr int kSlabUnroll = DRR_SLAB_UNROLL, kMinorUnroll = DRR_MINOR_UNROLL;  // loop iterations in flight
using u32 = unsigned int;
using u64 = unsigned long long;

// Per-ray values that only the ray's end needs, parked in shared memory while
// the loops run.
enum ParkSlot : int {
  kPkD = 0,       // p - s in mm (3)
  kPkE = 3,       // the entry point (3); the detector-parameter mode keeps 1 - 2 amin and amin here
  kPkF0 = 6,      // alpha from the entry to the first crossing of slots 0, 1 (2)
  kPkRg = 8,      // alpha per plane of slots 0, 1 (2)
  kPkSpan = 10,   // alpha_max - alpha_min
  kPkMm = 11,     // path length of a slab, a float-float (2)
  kPkCount = 13
};
struct Park {
  float v[kPkCount][kThreads];
};
// Per-ray values that the forward walk needs only where a chunk starts.
struct FwdPark {
  u64 x0[2][kThreads], dx[2][kThreads];  // slots 0, 1: q_2 at crossing 0 and its step (32.32)
  u64 y0[2][kThreads], dy[2][kThreads];  // q_0, q_1 at dominant crossing 0 and their steps (24.40)
};
struct NoPark {};
template <int MODE>
struct ParkFor {
  using type = std::conditional_t<MODE == kFwdJac || MODE == kPoseGrad || MODE == kGeoGrad, Park,
                                  std::conditional_t<MODE == kFwd || MODE == kBackproject, FwdPark, NoPark>>;
};

struct SlabRay {
  int cnt[3];      // crossings per slot
  int i0[3];       // entry voxel index per slot, counted in the ray's direction
  int off;         // element offset of the entry voxel (padded layout)
  int step[3];     // signed element stride per slot
  u32 axes;        // 2 bits each: real axis of slots 0, 1, 2; slot of the entry / exit plane, 3 when clamped to alpha = 0 / 1
  __device__ __forceinline__ int axis(int slot) const { return (axes >> (2 * slot)) & 3u; }
  __device__ __forceinline__ int entry_slot() const { return (axes >> 6) & 3u; }
  __device__ __forceinline__ int exit_slot() const { return (axes >> 8) & 3u; }
  u64 Y, Z;        // q_0, q_1 at dominant crossing 0 and their step per dominant crossing
  u32 dy, dz;
  u64 mX, mdX;     // slot 0's crossing 0: q_2 and q_1 (both + t0) and their steps
  u64 mZ;
  u32 mdz;
  u64 lX, ldX;     // slot 1's crossing 0: q_2 and q_0 (both + t1) and their steps
  u64 lY, ldY;
  u32 t0, t1;      // rounding bounds (and biases) of the minor loops' coordinates
  float w1;        // 1 - q_2 at the entry: the first slab's share inside the ray (a ray inside one slab: its length)
  float rest;      // share of the last slab beyond the exit (0 then)
  bool exact;      // to be summed by exact_rays
  // the forward walk only
  u64 qx;          // q_2 at the exit
  float start;     // q_2 at the entry
  float r0, r1;    // slabs per plane of slots 0, 1
  float len;       // |p - s| in mm
  float rg2;       // alpha per dominant plane
};

// A lane without a ray to walk takes part with no crossings.
__device__ __forceinline__ void slab_idle(const VolumeDev& vd, SlabRay& s) {
  s = SlabRay{};
  s.off = vd.origin;
}

// x * m / 2^32 for a 32.32 number m and a fraction x (0.32), rounded down.
__device__ __forceinline__ u64 mul_frac(u32 x, u64 m) {
  return static_cast<u64>(x) * static_cast<u32>(m >> 32) + __umulhi(x, static_cast<u32>(m));
}

// ---------------------------------------------------------------------------
// Float-float arithmetic (unevaluated sums h + l of two FP32 numbers, ~2^-46
// relative; Dekker 1971, Knuth TAOCP 2, with FMA products).  The per-ray setup
// needs ~2^-36 of a voxel; this GPU issues FP64 at 1/64 of the FP32 rate, and
// ~75 FP64 operations per ray took longer than the walk itself (277 us of an
// empty walk of the 16-pose CT batch).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 ff_sum(float a, float b) {  // exact a + b
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t)));
}
__device__ __forceinline__ float2 ff_norm(float h, float l) {  // |h| >= |l|
  const float s = __fadd_rn(h, l);
  return make_float2(s, __fsub_rn(l, __fsub_rn(s, h)));
}
__device__ __forceinline__ float2 ff_add(float2 a, float2 b) {
  const float2 s = ff_sum(a.x, b.x);
  return ff_norm(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 ff_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  const float e = __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.x, -p)));
  return ff_norm(p, e);
}
__device__ __forceinline__ float2 ff_rcp(float2 a) {  // 1e-30 < |a| < 1e30
  const float r = __frcp_rn(a.x);
  const float e = __fmaf_rn(-a.y, r, __fmaf_rn(-a.x, r, 1.f));
  return ff_norm(r, __fmul_rn(r, e));
}
// A sum kept as value + error: exact but for the rounding of the error.
struct Sum2 {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float2 r = ff_sum(s, x);
    s = r.x;
    e = __fadd_rn(e, r.y);
  }
  __device__ __forceinline__ void add(Sum2 x) {
    add(x.s);
    e = __fadd_rn(e, x.e);
  }
  __device__ __forceinline__ void add_product(float x, float y) {
    const float p = __fmul_rn(x, y);
    add(p);
    e = __fadd_rn(e, __fmaf_rn(x, y, -p));
  }
  // (an infinite or NaN s is the plain sum's; its error is NaN)
  __device__ __forceinline__ float value() const { return isfinite(s) ? __fadd_rn(s, e) : s; }
  __device__ __forceinline__ double value64() const {
    return isfinite(s) ? static_cast<double>(s) + static_cast<double>(e) : static_cast<double>(s);
  }
  // Total over the warp, the same in every lane (a fixed butterfly).
  __device__ __forceinline__ void warp_sum() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      add(Sum2{__shfl_xor_sync(0xffffffffu, s, o), __shfl_xor_sync(0xffffffffu, e, o)});
  }
};
// a times c, rounded once (to its last bit or so).
__device__ __forceinline__ float ff_scaled(const Sum2& a, float2 c) {
  const float p = __fmul_rn(a.s, c.x);
  if (!isfinite(p)) return p;
  return __fadd_rn(p, __fadd_rn(__fmaf_rn(a.s, c.x, -p), __fmaf_rn(a.s, c.y, __fmul_rn(a.e, c.x))));
}
// x as the unevaluated sum of two FP32 numbers.
__device__ __forceinline__ float2 ff_from(double x) {
  const float h = static_cast<float>(x);
  return make_float2(h, static_cast<float>(x - static_cast<double>(h)));
}

// A pose's FP64 geometry as float-float pairs, for the per-ray setup.
struct GeomFF {
  float2 u0[3], un[3], g00[3], gw[3], gh[3];
};
// From the pose's geometry in shared memory, by a warp (or the first warp of a
// block) after the geometry's copy; the caller synchronises.
__device__ __forceinline__ void geom_ff(const PoseGeom& pg, GeomFF& gf) {
  static_assert(sizeof(GeomFF) == 15 * sizeof(float2), "one pair per FP64 value");
  const int lane = threadIdx.x & 31;
  if (lane < 15) reinterpret_cast<float2*>(&gf)[lane] = ff_from(reinterpret_cast<const double*>(&pg)[lane]);
}
// x in [0, 2^31) as 32.32 fixed point; a negative x (rounding) gives 0.
__device__ __forceinline__ u64 ff_fix(float2 x) {
  if (x.x < 0.f) return 0ull;
  const float fl = floorf(x.x);
  const u64 v = (static_cast<u64>(__float2uint_rz(fl)) << 32) + __float2uint_rz((x.x - fl) * 4294967296.f);
  const long long lo = static_cast<long long>(__float2int_rn(x.y * 4294967296.f));
  const long long r = static_cast<long long>(v) + lo;
  return r < 0 ? 0ull : static_cast<u64>(r);
}
// x <= 1 as a 32-bit fraction (1 becomes 1 - 2^-32).
__device__ __forceinline__ u32 ff_frac(float2 x) {
  const u64 v = static_cast<u64>(__float2uint_rz(x.x * 4294967296.f)) +
                static_cast<u64>(static_cast<long long>(__float2int_rn(x.y * 4294967296.f)));
  return v >> 32 ? (static_cast<long long>(v) < 0 ? 0u : 0xffffffffu) : static_cast<u32>(v);
}
// x in [0, 1] times 2^40.
__device__ __forceinline__ u64 ff_fix40(float2 x) {
  const float h = x.x * 65536.f, a = floorf(h);
  const u64 v = (static_cast<u64>(__float2uint_rz(a)) << 24) + __float2uint_rz((h - a) * 16777216.f);
  const long long r = static_cast<long long>(v) + __float2int_rn(x.y * 1099511627776.f);
  return r < 0 ? 0ull : static_cast<u64>(r);
}
__device__ __forceinline__ float fix_float(u64 x) {  // 32.32 fixed point to FP32
  return fmaf(static_cast<float>(static_cast<u32>(x)), kTwoM32, static_cast<float>(static_cast<u32>(x >> 32)));
}

// The ray's slab form.  Returns 1 for a hit, 0 for a miss, -1 for non-finite
// geometry.  All in FP32 / float-float / fixed point; where that cannot decide
// (faces, end voxels or end counts closer than its rounding) s.exact is set and
// exact_rays decides in FP64.
template <int MODE>
__device__ __forceinline__ int slab_setup(const VolumeDev& vd, const PoseGeom& pg, const GeomFF& gf, int h,
                                          int w, SlabRay& s, typename ParkFor<MODE>::type* park) {
  constexpr bool kFwdOnly = MODE == kFwd;
  const int t = threadIdx.x;
  float d[3];
  float2 g[3];
  if (w < (1 << 24) && h < (1 << 24)) {
    const float fw = static_cast<float>(w), fh = static_cast<float>(h);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float p = __fmul_rn(fw, gf.gw[a].x), q = __fmul_rn(fh, gf.gh[a].x);
      const float pe = __fmaf_rn(fw, gf.gw[a].y, __fmaf_rn(fw, gf.gw[a].x, -p));
      const float qe = __fmaf_rn(fh, gf.gh[a].y, __fmaf_rn(fh, gf.gh[a].x, -q));
      const float2 u = ff_sum(p, q), v = ff_sum(gf.g00[a].x, u.x);
      g[a] = ff_norm(v.x, __fadd_rn(__fadd_rn(v.y, u.y), __fadd_rn(__fadd_rn(pe, qe), gf.g00[a].y)));
    }
  } else {
#pragma unroll
    for (int a = 0; a < 3; ++a)
      g[a] = ff_from(fma(static_cast<double>(h), pg.gh[a], fma(static_cast<double>(w), pg.gw[a], pg.g00[a])));
  }
  // faces in FP32; a choice that FP32 cannot make safely -- the runner-up
  // crossing (or the clamp at alpha 0 / 1) within 2^-20 of the chosen one, four
  // times the FP32 error of these products, or a hit test that close -- is left
  // to exact_rays.  That matters where the clipped span is a small part of alpha
  // (a small volume far from the source): there an FP32 tie moves the entry by
  // a visible share of the span.
  float lof = 0.f, hif = 1.f, lo2 = -1.f, hi2 = 2.f;  // chosen and runner-up entry / exit
  int ea = -1, xa = -1;
  bool finite = true, hit = true, unsafe = false;
  float2 ar[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    finite = finite && isfinite(g[a].x) && isfinite(gf.u0[a].x);
    d[a] = g[a].x * vd.delta[a];
    if constexpr (!kFwdOnly) park->v[kPkD + a][t] = d[a];
    if (g[a].x != 0.f) {
      ar[a] = ff_rcp(make_float2(fabsf(g[a].x), g[a].x < 0.f ? -g[a].y : g[a].y));
      unsafe = unsafe || fabsf(g[a].x) < 1e-20f;
      const float rf = copysignf(ar[a].x, g[a].x);
      const float t0 = -gf.u0[a].x * rf, t1 = gf.un[a].x * rf;
      const float lo = fminf(t0, t1), hi = fmaxf(t0, t1);
      if (lo > lof) { lo2 = lof; lof = lo; ea = a; } else lo2 = fmaxf(lo2, lo);
      if (hi < hif) { hi2 = hif; hif = hi; xa = a; } else hi2 = fminf(hi2, hi);
    } else {
      ar[a] = make_float2(0.f, 0.f);
      if (!(pg.u0[a] >= 0.0 && pg.un[a] > 0.0)) hit = false;
    }
  }
  if (!finite) return -1;
  if (!hit) return 0;
  const float tol = 9.5367431640625e-7f * fmaxf(fabsf(lof), fabsf(hif)) + 1e-30f;  // 2^-20
  unsafe = unsafe || lof - lo2 < tol || hi2 - hif < tol || fabsf(hif - lof) < tol;
  const float L = sqrtf(fmaf(d[2], d[2], fmaf(d[1], d[1], d[0] * d[0])));
  if (unsafe) {
    slab_idle(vd, s);
    s.exact = true;
    s.len = L;
    return 1;
  }
  if (!(lof < hif)) return 0;
  s.len = L;
  // slots: 2 the largest direction component, 1 the smallest
  float2 ag[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) ag[a] = make_float2(fabsf(g[a].x), g[a].x < 0.f ? -g[a].y : g[a].y);
  const auto more = [](float2 x, float2 y) { return x.x > y.x || (x.x == y.x && x.y > y.y); };
  const int a2 = more(ag[2], ag[0]) && more(ag[2], ag[1]) ? 2 : (more(ag[1], ag[0]) ? 1 : 0);
  const int p = a2 == 0 ? 1 : 0, q = a2 == 2 ? 1 : 2;
  const bool pq = !more(pick3(q, ag[0], ag[1], ag[2]), pick3(p, ag[0], ag[1], ag[2]));
  const int ax[3] = {pq ? p : q, pq ? q : p, a2};
  const auto slot_of = [&](int a) { return a < 0 ? 3u : (a == ax[0] ? 0u : (a == ax[1] ? 1u : 2u)); };
  s.axes = static_cast<u32>(ax[0] | ax[1] << 2 | ax[2] << 4) | slot_of(ea) << 6 | slot_of(xa) << 8;
  float2 sg[3], sr[3], U[3], N[3];  // direction, its reciprocal, source and far face (in the ray's direction), per slot
  int n[3];
  bool up[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    sg[k] = pick3(ax[k], ag[0], ag[1], ag[2]);
    sr[k] = pick3(ax[k], ar[0], ar[1], ar[2]);
    n[k] = pick3(ax[k], vd.n[0], vd.n[1], vd.n[2]);
    up[k] = !(pick3(ax[k], g[0].x, g[1].x, g[2].x) < 0.f);
    const float2 u = pick3(ax[k], gf.u0[0], gf.u0[1], gf.u0[2]), v = pick3(ax[k], gf.un[0], gf.un[1], gf.un[2]);
    U[k] = up[k] ? u : v;
    N[k] = up[k] ? v : u;
    const int st = pick3(ax[k], vd.stride[0], vd.stride[1], vd.stride[2]);
    s.step[k] = up[k] ? st : -st;
  }
  float2 amin = make_float2(0.f, 0.f), amax = make_float2(1.f, 0.f);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (ea == ax[k]) amin = ff_mul(make_float2(-U[k].x, -U[k].y), sr[k]);
    if (xa == ax[k]) amax = ff_mul(N[k], sr[k]);
  }
  // float-float rounding of positions, in 2^-32 voxel
  const float far = fmaxf(fmaxf(fabsf(gf.u0[0].x) + fabsf(gf.un[0].x), fabsf(gf.u0[1].x) + fabsf(gf.un[1].x)),
                          fabsf(gf.u0[2].x) + fabsf(gf.un[2].x)) * 2.44140625e-4f;
  const u32 te = static_cast<u32>(fminf(far, 1e8f)) + 4u;
  bool exact = far > 1e8f;
  // entry voxel and fraction per axis
  u32 E[3];
  s.off = vd.origin;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float uef = 0.f;
    if (ea == ax[k]) {
      E[k] = 0u;
      s.i0[k] = 0;
    } else {
      const float2 ue = ff_add(U[k], ff_mul(amin, sg[k]));
      uef = ue.x;
      const u64 f = min(ff_fix(ue), (static_cast<u64>(n[k]) << 32) - 1ull);
      E[k] = static_cast<u32>(f);
      s.i0[k] = static_cast<int>(f >> 32);
      if (sg[k].x != 0.f) {
        if (E[k] + te < 2u * te) exact = true;
      } else {  // parallel: the voxel as exact_rays finds it (half open, also for a ray in a voxel plane)
        s.i0[k] = min(max(static_cast<int>(floor(pick3(ax[k], pg.u0[0], pg.u0[1], pg.u0[2]))), 0), n[k] - 1);
      }
    }
    // element offset of the entry voxel: counted from the far end where the ray runs down
    s.off += s.step[k] * (up[k] ? s.i0[k] : s.i0[k] - (n[k] - 1));
    if constexpr (!kFwdOnly && MODE != kGeoGrad) {
      // the entry point in world coordinates (volume centred at the origin)
      const float dl = pick3(ax[k], vd.delta[0], vd.delta[1], vd.delta[2]), half = 0.5f * static_cast<float>(n[k]);
      const float e = up[k] ? fmaf(uef, dl, -half * dl) : fmaf(-uef, dl, half * dl);
      if (ax[k] == 0) park->v[kPkE][t] = e;
      else if (ax[k] == 1) park->v[kPkE + 1][t] = e;
      else park->v[kPkE + 2][t] = e;
    }
  }
  const float2 r02 = ff_mul(sg[0], sr[2]), r12 = ff_mul(sg[1], sr[2]);
  s.dy = ff_frac(r02);
  s.dz = ff_frac(r12);
  s.mdz = ff_frac(ff_mul(sg[1], sr[0]));
  const float2 r20 = ff_mul(sg[2], sr[0]), r21 = ff_mul(sg[2], sr[1]), r01 = ff_mul(sg[0], sr[1]);
  // exit: coordinate along the dominant axis, then the counts
  u64 qx = static_cast<u64>(n[2] - s.i0[2]) << 32;
  s.cnt[2] = n[2] - 1 - s.i0[2];
  s.rest = 0.f;
  if (xa != ax[2]) {
    const float2 ux = ff_add(U[2], ff_mul(amax, sg[2]));
    const u64 base = static_cast<u64>(s.i0[2]) << 32, f = ff_fix(ux);
    qx = min(f > base + E[2] ? f - base : static_cast<u64>(E[2]), qx - 1ull);
    s.cnt[2] = static_cast<int>(qx >> 32);
    const u32 fr = static_cast<u32>(qx);
    s.rest = static_cast<float>(0u - fr) * kTwoM32;
    if (fr == 0u) s.rest = 1.f;
    if (!kFwdOnly && fr + te < 2u * te) exact = true;
  }
  const float dom = static_cast<float>(s.cnt[2]) + 16.f + far;
  const u32 tx = static_cast<u32>(fminf(dom, 2e8f));
  const u64 len = qx - E[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int most = n[k] - 1 - s.i0[k];
    if (sg[k].x == 0.f) {
      s.cnt[k] = 0;
    } else if (xa == ax[k]) {
      s.cnt[k] = most;
    } else {
      const u32 sl = k == 0 ? s.dy : s.dz;
      const u64 f = static_cast<u64>(E[k]) + static_cast<u64>(static_cast<u32>(len >> 32)) * sl +
                    __umulhi(static_cast<u32>(len), sl);
      s.cnt[k] = min(static_cast<int>(f >> 32), most);
      if (!kFwdOnly && static_cast<u32>(f) + tx < 2u * tx) exact = true;
    }
  }
  s.rg2 = sr[2].x;
  if constexpr (kFwdOnly) {
    // positions along a minor axis whose planes lie more than 2^16 slabs apart
    // would lose more than FP32 keeps of them
    s.exact = exact || (s.cnt[0] > 0 && !(r20.x < 65536.f)) || (s.cnt[1] > 0 && !(r21.x < 65536.f)) || n[2] >= (1 << 23);
    if (s.exact) s.cnt[0] = s.cnt[1] = s.cnt[2] = 0;
    // a ray inside one slab (it clips a corner, or the volume is one slab thick) is
    // measured from its entry: its lengths would carry 2^-24 of the slab otherwise,
    // which may be a visible share of them
    const u64 origin = s.cnt[2] == 0 ? E[2] : 0ull;
    s.qx = qx - origin;
    s.start = s.cnt[2] == 0 ? 0.f : static_cast<float>(E[2]) * kTwoM32;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const bool any = s.cnt[k] > 0;
      const float2 r = k == 0 ? r20 : r21;
      const u64 dx = ff_fix(any ? r : make_float2(0.f, 0.f)), dy = ff_fix40(k == 0 ? r02 : r12);
      park->dx[k][t] = dx;
      park->x0[k][t] = any ? E[2] - origin + (dx - mul_frac(E[k], dx)) : static_cast<u64>(1u << 30) << 32;  // none: beyond any exit
      park->dy[k][t] = dy;
      park->y0[k][t] = (static_cast<u64>(E[k]) << 8) + (dy - mul_frac(E[2], dy));
      (k == 0 ? s.r0 : s.r1) = any ? r.x : 0.f;
    }
    return 1;
  }
  // rounding bounds in 2^-32: a minor crossing's own coordinates err by at most
  // ~cnt + 3, the dominant loop's view of it by ~cnt_2 + 3 of its plane spacings
  // (twice that where the start was pulled back below)
  const float t0 = fmaf(2.f * dom, r20.x, static_cast<float>(s.cnt[0]) + 16.f + far);
  const float t1 = fmaf(2.f * dom, r21.x, static_cast<float>(s.cnt[1]) + 16.f + far);
  // an axis whose planes lie more than 2^16 slabs apart, or a bound that is no
  // longer small, goes to exact_rays
  if (s.cnt[0] > 0 && !(r20.x < 65536.f && t0 < 2.68435456e8f)) exact = true;
  if (s.cnt[1] > 0 && !(r21.x < 65536.f && t1 < 2.68435456e8f)) exact = true;
  s.exact = exact;
  if (exact) s.cnt[0] = s.cnt[1] = s.cnt[2] = 0;
  s.t0 = s.cnt[0] > 0 ? static_cast<u32>(t0) : 0u;
  s.t1 = s.cnt[1] > 0 ? static_cast<u32>(t1) : 0u;
  s.mdX = ff_fix(r20.x < 65536.f ? r20 : make_float2(0.f, 0.f));
  s.ldX = ff_fix(r21.x < 65536.f ? r21 : make_float2(0.f, 0.f));
  s.ldY = ff_fix(r21.x < 65536.f ? r01 : make_float2(0.f, 0.f));
  s.Y = static_cast<u64>(E[0]) + (s.dy - __umulhi(E[2], s.dy));
  s.Z = static_cast<u64>(E[1]) + (s.dz - __umulhi(E[2], s.dz));
  // a ray inside one slab is measured from its entry, as the forward walk's
  const bool inside = s.cnt[2] == 0;
  const u64 from = inside ? 0ull : static_cast<u64>(E[2]);
  s.mX = from + (s.mdX - mul_frac(E[0], s.mdX)) + s.t0;
  s.mZ = static_cast<u64>(E[1]) + (s.mdz - __umulhi(E[0], s.mdz)) + s.t0;
  s.lX = from + (s.ldX - mul_frac(E[1], s.ldX)) + s.t1;
  s.lY = E[0] + (s.ldY - mul_frac(E[1], s.ldY)) + s.t1;
  if (s.cnt[2] > 0) {
    // no minor plane beyond the exit is counted at the last dominant crossing:
    // where rounding would, the start is pulled back by the excess
    const u64 m = static_cast<u64>(s.cnt[2] - 1);
    const u64 ey = s.Y + m * s.dy, ly = static_cast<u64>(s.cnt[0] + 1) << 32;
    if (ey >= ly) s.Y -= min(s.Y, ey - ly + 1ull);
    const u64 ez = s.Z + m * s.dz, lz = static_cast<u64>(s.cnt[1] + 1) << 32;
    if (ez >= lz) s.Z -= min(s.Z, ez - lz + 1ull);
  }
  s.w1 = inside ? fix_float(len) : (E[2] == 0u ? 1.f : static_cast<float>(0u - E[2]) * kTwoM32);
  if (inside) s.rest = 0.f;
  if constexpr (!kFwdOnly) {
    if (MODE == kGeoGrad) {
      park->v[kPkE][t] = (1.f - 2.f * amin.x) - 2.f * amin.y;
      park->v[kPkE + 1][t] = amin.x;
    }
    park->v[kPkF0][t] = (E[0] == 0u ? 1.f : static_cast<float>(0u - E[0]) * kTwoM32) * sr[0].x;
    park->v[kPkF0 + 1][t] = (E[1] == 0u ? 1.f : static_cast<float>(0u - E[1]) * kTwoM32) * sr[1].x;
    park->v[kPkRg][t] = sr[0].x;
    park->v[kPkRg + 1][t] = sr[1].x;
    park->v[kPkSpan][t] = fix_float(len) * sr[2].x;
    // the path length of a slab as float-float: the roundings of an FP32 product of
    // length and alpha per slab were a third of a pixel's error
    const auto side = [&](int k) { return pick3(ax[k], vd.delta[0], vd.delta[1], vd.delta[2]); };
    Sum2 sq;
    sq.add_product(side(2), side(2));
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float2 r = k == 0 ? r02 : r12;
      const float x = __fmul_rn(r.x, side(k)), xl = __fmaf_rn(r.y, side(k), __fmaf_rn(r.x, side(k), -x));
      sq.add_product(x, x);
      sq.e = __fmaf_rn(__fadd_rn(x, x), xl, sq.e);
    }
    const float root = __fsqrt_rn(sq.s);
    const float2 mm = sq.s > 1e-24f && sq.s < 1e30f
                          ? make_float2(root, __fadd_rn(__fmaf_rn(-root, root, sq.s), sq.e) * __fdividef(0.5f, root))
                          : make_float2(L * sr[2].x, 0.f);
    park->v[kPkMm][t] = mm.x;
    park->v[kPkMm + 1][t] = mm.y;
  }
  return 1;
}

// ---------------------------------------------------------------------------
// Forward walk (Eq. 2 with the crossings of Eq. 3 taken in order, Sec. 2.2):
// each step takes the smallest of the three axes' next crossings.  The steps run
// in chunks of the same number of crossings for the warp's 32 rays.  Inside a
// chunk positions are FP32 slab coordinates q_2 from the last dominant plane
// before it: the dominant axis' crossings are whole numbers, the minor ones l r +
// x0, so they err by 2^-24 of a chunk.  A chunk starts from counts of crossings
// per axis alone, in exact (32.32 fixed point) order, and its last segment ends
// at the exact position of its last crossing; where FP32 took a chunk's last
// crossings in another order (they are then closer than 2^-24 of a chunk) the
// counts are corrected.  So the chunks are independent: they are added in order
// whoever walks them, and the split kernel's warps, which take different chunks
// of a ray, give the same bits as one warp walking through.
//
// What bounds it: one gather per segment, 4.4 wavefronts each on the L1 data
// pipe (68 % busy), and ~18 warp instructions per segment (issue slots 62 %).
// Measured (CUDA events): 16-pose CT batch, 512x512x133 and 200x200, 0.366 ->
// 0.344 ms against the walk with an FP64 ray setup; one 128x128 pose on 256^3, split
// over the warps of a tile, 0.069 -> 0.028.  Chunks that begin at a dominant
// plane instead of keeping step, 8 / 4 / 2 / 1 per ray: 0.377 / 0.358 / 0.350 /
// 0.340 (rays that wait for each other at a plane x = const touch 15 cache lines
// per gather, rays in step 13), and a whole ray in one FP32 frame is too inexact
// for the smallest volumes.
// ---------------------------------------------------------------------------
#ifndef DRR_FWD_UNROLL
#define DRR_FWD_UNROLL 12  // a multiple of 3: the voxel registers of the two-ahead pipeline rotate without moves
#endif
constexpr int kFwdUnroll = DRR_FWD_UNROLL;
#ifndef DRR_CHUNKS
#define DRR_CHUNKS 8
#endif
constexpr int kChunks = DRR_CHUNKS;  // most chunks of a ray

// One step in predicated PTX: an = min(tx, ty, tz); the axis it belongs to
// (dominant before middle before least on ties) steps: the dominant position + 1
// or the minor axis' crossing counter + 1, and the voxel offset by its stride.
__device__ __forceinline__ float walk_step(float& tx, float ty, float tz, float& ly, float& lz, int& off, int sx, int sy,
                                           int sz) {
  float an;
  asm("{\n\t"
      ".reg .pred px, py, pxy;\n\t"
      "min.f32 %0, %1, %5;\n\t"
      "min.f32 %0, %0, %6;\n\t"
      "setp.eq.f32 px, %1, %0;\n\t"
      "setp.eq.and.f32 py, %5, %0, !px;\n\t"
      "or.pred pxy, px, py;\n\t"
      "@px add.f32 %1, %1, 0f3F800000;\n\t"
      "@py add.f32 %2, %2, 0f3F800000;\n\t"
      "@!pxy add.f32 %3, %3, 0f3F800000;\n\t"
      "@px add.s32 %4, %4, %7;\n\t"
      "@py add.s32 %4, %4, %8;\n\t"
      "@!pxy add.s32 %4, %4, %9;\n\t"
      "}"
      : "=&f"(an), "+f"(tx), "+f"(ly), "+f"(lz), "+r"(off)
      : "f"(ty), "f"(tz), "r"(sx), "r"(sy), "r"(sz));
  return an;
}

// Crossings taken per slot, and the exact positions around them: the last one
// taken (at), and the next one of each slot (beyond every crossing where there
// is none).
struct Counts {
  int k[3];
};
constexpr u64 kNever = 1ull << 62;
struct Around {
  u64 at, next[3];
  bool ordered;  // every crossing taken precedes every other (ties: slot 2, 0, 1)
};
__device__ __forceinline__ Around around(const SlabRay& s, const FwdPark* park, const Counts& c) {
  const int t = threadIdx.x;
  Around r;
  u64 last[3];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const u64 dx = park->dx[k][t], x = park->x0[k][t] + static_cast<u64>(static_cast<u32>(c.k[k])) * dx;
    r.next[k] = c.k[k] < s.cnt[k] ? x : kNever;
    last[k] = c.k[k] > 0 ? x - dx : 0ull;
  }
  last[2] = static_cast<u64>(static_cast<u32>(c.k[2])) << 32;
  r.next[2] = c.k[2] < s.cnt[2] ? last[2] + (1ull << 32) : kNever;
  if (c.k[2] == 0) last[2] = 0ull;
  r.at = max(max(last[0], last[1]), last[2]);
  r.ordered = c.k[0] <= s.cnt[0] && c.k[1] <= s.cnt[1] && c.k[2] <= s.cnt[2] && last[2] <= min(r.next[0], r.next[1]) &&
              last[0] <= r.next[1] && last[1] < r.next[0] && max(last[0], last[1]) < r.next[2];
  return r;
}

// The counts after n crossings in exact order, from a dominant crossing before.
__device__ __forceinline__ Counts counts_after(const SlabRay& s, const FwdPark* park, int n) {
  const int t = threadIdx.x;
  const int total = s.cnt[0] + s.cnt[1] + s.cnt[2];
  Counts c{{0, 0, 0}};
  int left = n;
  int a = static_cast<int>(static_cast<float>(n) * static_cast<float>(s.cnt[2]) / static_cast<float>(max(total, 1))) - 1;
  a = min(a, s.cnt[2]);
  while (a > 0) {
    const u64 X = static_cast<u64>(static_cast<u32>(a)) << 32;  // dominant crossing a - 1
    int m[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {  // minor crossings before it
      const u64 x0 = park->x0[k][t], dx = park->dx[k][t];
      m[k] = min(static_cast<int>((park->y0[k][t] + static_cast<u64>(static_cast<u32>(a - 1)) * park->dy[k][t]) >> 40), s.cnt[k]);
      while (m[k] > 0 && x0 + static_cast<u64>(static_cast<u32>(m[k] - 1)) * dx >= X) --m[k];
      while (m[k] < s.cnt[k] && x0 + static_cast<u64>(static_cast<u32>(m[k])) * dx < X) ++m[k];
    }
    const int d = n - (a + m[0] + m[1]);
    if (d >= 0) {
      c = Counts{{m[0], m[1], a}};
      left = d;
      break;
    }
    a += d;  // too far: at least as many dominant crossings back
  }
  for (; left > 0; --left) {
    const Around r = around(s, park, c);
    if (r.next[2] <= r.next[0] && r.next[2] <= r.next[1]) ++c.k[2];
    else if (r.next[0] <= r.next[1]) ++c.k[0];
    else ++c.k[1];
  }
  return c;
}

// Crossings per chunk, for the warp's 32 rays.  The FP32 error of a position grows
// with the chunk's share of the ray: an eighth keeps 2e-5 of the image maximum /
// 1000 on 64-voxel volumes (a whole ray in one frame: 3.8e-5), and chunks of 121
// crossings on 512-voxel ones (quarters of those rays, 1 to 3 % faster, do not).
__device__ __forceinline__ int chunk_steps(const SlabRay& s) {
  const int most = __reduce_max_sync(0xffffffffu, s.cnt[0] + s.cnt[1] + s.cnt[2]);
  constexpr int kBlock = kChunks * kFwdUnroll;
  return max((most + kBlock - 1) / kBlock, most > 512 ? 120 / kFwdUnroll : 1) * kFwdUnroll + 1;
}

// Chunks [q0, q1) of the ray, `size` crossings each, chunk q's sum to sink(q, sum);
// the last chunk goes on to the exit.
template <int DT, class Sink>
__device__ __forceinline__ void walk_forward(const VolumeDev& vd, const SlabRay& s, const FwdPark* park, int size, int q0,
                                             int q1, Sink sink) {
  const int total = s.cnt[0] + s.cnt[1] + s.cnt[2];
  if (q0 > 0 && q0 * size >= total) return;
  Counts c = q0 > 0 ? counts_after(s, park, q0 * size) : Counts{{0, 0, 0}};
  Around ar = around(s, park, c);
  int off = s.off + c.k[0] * s.step[0] + c.k[1] * s.step[1] + c.k[2] * s.step[2];
  float v = gather<DT>(vd, off);
  int todo = total - q0 * size;  // crossings from here on
  float ac = s.start;
  for (int q = q0; q < q1; ++q) {
    const u64 O = static_cast<u64>(static_cast<u32>(c.k[2])) << 32;  // the last dominant plane
    if (q > 0) ac = fix_to_float(static_cast<long long>(ar.at - O));
    const float x0 = fix_to_float(static_cast<long long>(ar.next[0] - O)),
                x1 = fix_to_float(static_cast<long long>(ar.next[1] - O));
    const int n = min(todo, size);
    float acc = 0.f;
    if (n > 0) {
      float tx = 1.f, ty = x0, tz = x1, ly = 0.f, lz = 0.f;
#define DRR_FSTEP(an)                                                                   \
  const float an = walk_step(tx, ty, tz, ly, lz, off, s.step[2], s.step[0], s.step[1]); \
  next_xy(ty, tz, ly, lz, s.r0, s.r1, x0, x1);
      DRR_FSTEP(a1)
      float an1 = a1;
      float v1 = gather<DT>(vd, off);
#pragma unroll kFwdUnroll
      for (int i = 1; i < n; ++i) {
        DRR_FSTEP(an2)
        const float v2 = gather<DT>(vd, off);
        acc = fmaf(an1 - ac, v, acc);
        ac = an1;
        an1 = an2;
        v = v1;
        v1 = v2;
      }
#undef DRR_FSTEP
      todo -= n;
      c.k[2] += static_cast<int>(tx) - 1;
      c.k[0] += static_cast<int>(ly);
      c.k[1] += static_cast<int>(lz);
      ar = around(s, park, c);
      if (!ar.ordered) {  // FP32 took the chunk's last crossings in another order
        c = counts_after(s, park, total - todo);
        ar = around(s, park, c);
        off = s.off + c.k[0] * s.step[0] + c.k[1] * s.step[1] + c.k[2] * s.step[2];
        v1 = gather<DT>(vd, off);
      }
      const float at = fix_to_float(static_cast<long long>(ar.at - O));
      acc = fmaf(at - ac, v, acc);  // the segment that ends at the chunk's last crossing, exact end
      ac = at;
      v = v1;
    }
    if (todo == 0) {  // the segment up to the exit
      sink(q, fmaf(fix_to_float(static_cast<long long>(s.qx - ar.at)), v, acc));  // (no crossing: from the entry, 0)
      return;
    }
    sink(q, acc);
  }
}

// The loops are cut into np pieces: piece p takes of each slot the planes
// [p, p + 1) * len counted from the warp's first entry plane (sh: this ray's
// entry plane in that count).
struct Pieces {
  int sh, len;
};
struct Plan {
  Pieces slot[3];
  int np;
};
__device__ __forceinline__ Plan plan_pieces(const SlabRay& s) {
  constexpr u32 kAll = 0xffffffffu;
  Plan pl;
  int total[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int base = __reduce_min_sync(kAll, s.cnt[k] > 0 ? s.i0[k] : 0x7fffffff);
    pl.slot[k].sh = s.cnt[k] > 0 ? s.i0[k] - base : 0;
    total[k] = __reduce_max_sync(kAll, s.cnt[k] > 0 ? pl.slot[k].sh + s.cnt[k] : 0);
  }
  pl.np = min(max((total[2] + kPieceLen - 1) / kPieceLen, 1), kPieces);
  // whole unrolled blocks per piece
  pl.slot[0].len = ((total[0] + pl.np - 1) / pl.np + kMinorUnroll - 1) / kMinorUnroll * kMinorUnroll;
  pl.slot[1].len = ((total[1] + pl.np - 1) / pl.np + kMinorUnroll - 1) / kMinorUnroll * kMinorUnroll;
  pl.slot[2].len = ((total[2] + pl.np - 1) / pl.np + kSlabUnroll - 1) / kSlabUnroll * kSlabUnroll;
  return pl;
}
// First crossing of piece p.
__device__ __forceinline__ int piece_start(const Pieces& pc, int p, int cnt) {
  return min(max(p * pc.len - pc.sh, 0), cnt);
}

// Pieces [p0, p1) of the sum of the voxels entered at dominant crossings; piece
// p's sum goes to sink(p, sum).  A block of kSlabUnroll voxels is added as a tree:
// a homogeneous tissue has few voxel values, and a running FP32 sum rounds each of
// them the same way on every ray, a common error of a DRR's pixels that does not
// average out of their sums (the pose gradient).
template <int DT, class Sink>
__device__ __forceinline__ void dominant_loop(const VolumeDev& vd, const SlabRay& s, const Pieces& pc, int p0, int p1,
                                              Sink sink) {
  int m = piece_start(pc, p0, s.cnt[2]);
  const u64 Y = s.Y + static_cast<u64>(static_cast<u32>(m)) * s.dy;
  const u64 Z = s.Z + static_cast<u64>(static_cast<u32>(m)) * s.dz;
  u32 fy = static_cast<u32>(Y), fz = static_cast<u32>(Z);
  int off = s.off + (m + 1) * s.step[2] + static_cast<int>(Y >> 32) * s.step[0] + static_cast<int>(Z >> 32) * s.step[1];
  const int st = s.step[2], st0 = st + s.step[0], s1 = s.step[1];
#pragma unroll 1
  for (int p = p0; p < p1; ++p) {
    const int end = piece_start(pc, p + 1, s.cnt[2]);
    float S = 0.f;
    const auto block = [&](auto whole) {
      float v[kSlabUnroll];
#pragma unroll
      for (int j = 0; j < kSlabUnroll; ++j) {
        v[j] = 0.f;
        if (whole || m + j < end) {
          v[j] = gather<DT>(vd, off);
          fy += s.dy;
          fz += s.dz;
          off += (fy < s.dy ? st0 : st) + (fz < s.dz ? s1 : 0);
        }
      }
#pragma unroll
      for (int o = kSlabUnroll / 2; o > 0; o >>= 1) {
#pragma unroll
        for (int j = 0; j < o; ++j) v[j] += v[j + o];
      }
      S += v[0];
    };
    for (; m + kSlabUnroll <= end; m += kSlabUnroll) block(std::true_type{});
    if (m < end) {
      block(std::false_type{});
      m = end;
    }
    sink(p, S);
  }
}

// Sums over one minor axis' crossings of a piece, w = V after - V before: g = sum
// w, c = sum w f (f: biased fraction of the slab at the crossing, times 2^32), h =
// sum w k (k from the piece's first crossing); near: the smallest biased fraction.
struct MinorSums {
  float g, c, h;
  u32 near;
};
#define DRR_MINOR_BLOCK(ON, ADVANCE)                                   \
  {                                                                    \
    float v0[kU], v1[kU];                                              \
    u32 f[kU];                                                         \
    _Pragma("unroll") for (int j = 0; j < kU; ++j) {                   \
      v0[j] = v1[j] = 0.f;                                             \
      f[j] = static_cast<u32>(X);                                      \
      if (ON) {                                                        \
        const int o = OFFSET;                                          \
        v0[j] = gather<DT>(vd, o);                                     \
        v1[j] = gather_at<DT>(vd, after, o, sk);                       \
        r.near = min(r.near, min(f[j], NEAR));                         \
        ADVANCE                                                        \
      }                                                                \
    }                                                                  \
    _Pragma("unroll") for (int j = 0; j < kU; ++j) {                   \
      const float w = v1[j] - v0[j];                                   \
      r.g += w;                                                        \
      r.c = fmaf(w, static_cast<float>(f[j]), r.c);                    \
      r.h = fmaf(w, kf + static_cast<float>(j), r.h);                  \
    }                                                                  \
    kf += static_cast<float>(kU);                                      \
  }
#define DRR_MINOR_PIECES(CNT, ADVANCE)                                 \
  _Pragma("unroll 1") for (int p = p0; p < p1; ++p) {                  \
    const int end = piece_start(pc, p + 1, CNT);                       \
    MinorSums r{0.f, 0.f, 0.f, 0xffffffffu};                           \
    float kf = 0.f;                                                    \
    for (; k + kU <= end; k += kU) DRR_MINOR_BLOCK(true, ADVANCE)      \
    if (k < end) {                                                     \
      DRR_MINOR_BLOCK(k + j < end, ADVANCE)                            \
      k = end;                                                         \
    }                                                                  \
    sink(p, r);                                                        \
  }

// Slot 0: the slab (q_2) advances by at least one plane per crossing, slot 1's
// coordinate by at most one.
template <int DT, class Sink>
__device__ __forceinline__ void middle_loop(const VolumeDev& vd, const SlabRay& s, const Pieces& pc, int p0, int p1,
                                            Sink sink) {
  constexpr int kU = kMinorUnroll;
  int k = piece_start(pc, p0, s.cnt[0]);
  u64 X = s.mX + static_cast<u64>(static_cast<u32>(k)) * s.mdX;
  const u64 Z = s.mZ + static_cast<u64>(static_cast<u32>(k)) * s.mdz;
  u32 fz = static_cast<u32>(Z);
  const int sk = s.step[0], sx = s.step[2], st = sk + s.step[1];
  int o1 = s.off + k * sk + static_cast<int>(Z >> 32) * s.step[1];
  const void* after = base_after<DT>(vd, sk);
#define OFFSET (o1 + static_cast<int>(X >> 32) * sx)
#define NEAR fz
  DRR_MINOR_PIECES(s.cnt[0], X += s.mdX; fz += s.mdz; o1 += fz < s.mdz ? st : sk;)
#undef OFFSET
#undef NEAR
}

// Slot 1: both other coordinates may advance by several planes per crossing.
template <int DT, class Sink>
__device__ __forceinline__ void least_loop(const VolumeDev& vd, const SlabRay& s, const Pieces& pc, int p0, int p1,
                                           Sink sink) {
  constexpr int kU = kMinorUnroll;
  int k = piece_start(pc, p0, s.cnt[1]);
  u64 X = s.lX + static_cast<u64>(static_cast<u32>(k)) * s.ldX;
  u64 Y = s.lY + static_cast<u64>(static_cast<u32>(k)) * s.ldY;
  const int sk = s.step[1], sx = s.step[2], sy = s.step[0];
  int o1 = s.off + k * sk;
  const void* after = base_after<DT>(vd, sk);
#define OFFSET (o1 + static_cast<int>(X >> 32) * sx + static_cast<int>(Y >> 32) * sy)
#define NEAR static_cast<u32>(Y)
  DRR_MINOR_PIECES(s.cnt[1], X += s.ldX; Y += s.ldY; o1 += sk;)
#undef OFFSET
#undef NEAR
}
#undef DRR_MINOR_PIECES
#undef DRR_MINOR_BLOCK

// Whole-ray sums of one minor axis' pieces, added in piece order.
struct MinorTotals {
  float g = 0.f, c = 0.f, h = 0.f;
  // first: the piece's first crossing (h counts from the ray's)
  __device__ __forceinline__ void add(float pg, float pc, float ph, int first) {
    g += pg;
    c += pc;
    h += fmaf(static_cast<float>(first), pg, ph);
  }
  __device__ __forceinline__ float3 value() const { return make_float3(g, c, h); }
};
struct SlabTotals {
  Sum2 S;
  float3 minor[2];  // g, c, h of slots 0 and 1
};

// What the ray's end takes from the walk: E; with the Jacobian
// the per-axis crossing sums G = sum w, A = sum w alpha (w = V before - V
// after, alpha from the entry; A of the dominant axis is not used), and the
// parts of the clamped end points (Gc, Ac), which belong to no axis.
struct JacSums {
  float E, G[3], A[3], Gc, Ac;
  int dom;
};
// exact_rays' answer: the sums and the ray's entry in world coordinates, amin
// and 1 - 2 amin.
struct ExactRay {
  JacSums q;
  float e[3], amin, c;
};

// Crossings of an axis (first one at A, spacing D, cnt of them) that precede
// position pos: those at a smaller position, and with `tie` those at the same one.
// The FP32 quotient is off by less than one (cnt below 2^20; checked by the caller
// through `loop`), so three candidates decide, without a branch.
__device__ __forceinline__ int count_before(u64 pos, bool tie, u64 A, u64 D, int cnt, float rd, bool loop) {
  const u64 lim = pos + (tie ? 1ull : 0ull);  // crossings below it count
  const int est = lim > A ? static_cast<int>(fix_to_float(static_cast<long long>(lim - A)) * rd) : 0;
  int n = max(min(est, cnt) - 1, 0);
  if (loop) {
    while (n < cnt && fix_at(A, D, static_cast<u32>(n)) < lim) ++n;
    while (n > 0 && fix_at(A, D, static_cast<u32>(n - 1)) >= lim) --n;
    return n;
  }
  const u64 x = fix_at(A, D, static_cast<u32>(n));
  return n + (n < cnt && x < lim) + (n + 1 < cnt && x + D < lim) + (n + 2 < cnt && x + 2ull * D < lim);
}

// The rays of `mask` (lanes of the warp, each lane's pixel in h, w) in exact
// crossing order: positions as 64-bit fixed point, ties to the lower axis, after
// an FP64 clip.  Out of line, for the rays whose faces or ends slab_setup could not
// tell and those whose sum is not finite.  All 32 lanes share one ray's crossings: a
// crossing's place in the order needs only its position (the other axes'
// crossings before it are counted), so nothing is serial; one lane walking such
// a ray alone took ~250 us of dependent gathers, and the kernel waited for it.
template <int DT>
__device__ __noinline__ void exact_rays(const VolumeDev& vd, const PoseGeom& pg, u32 mask, int h, int w,
                                        ExactRay* out) {
  constexpr u32 kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  for (; mask; mask &= mask - 1u) {
    const int L = __ffs(static_cast<int>(mask)) - 1;
    const int hh = __shfl_sync(kAll, h, L), ww = __shfl_sync(kAll, w, L);
    ExactRay x{};
    RaySetup r;
    if (ray_setup(vd, pg, hh, ww, r) > 0) {  // the same for all lanes
      JacSums& q = x.q;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double g = fma(static_cast<double>(hh), pg.gh[a], fma(static_cast<double>(ww), pg.gw[a], pg.g00[a]));
        x.e[a] = fmaf(static_cast<float>(fma(r.amin, g, pg.u0[a])), vd.delta[a],
                      -0.5f * static_cast<float>(vd.n[a]) * vd.delta[a]);
      }
      x.amin = static_cast<float>(r.amin);
      x.c = static_cast<float>(1.0 - 2.0 * r.amin);
      if (r.cnt[1] > r.cnt[0]) q.dom = 1;
      if (r.cnt[2] > max(r.cnt[0], r.cnt[1])) q.dom = 2;
      const bool many = max(max(r.cnt[0], r.cnt[1]), r.cnt[2]) >= (1 << 20);
      float rd[3];
      u64 first = kFixMax;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        rd[a] = 1.f / fix_to_float(static_cast<long long>(r.D[a]));
        if (r.cnt[a] > 0) first = min(first, r.A0[a]);
      }
      const float vfirst = gather<DT>(vd, r.off);
      const float vl =
          gather<DT>(vd, r.off + r.cnt[0] * r.step[0] + r.cnt[1] * r.step[1] + r.cnt[2] * r.step[2]);
      float F = lane == 0 ? fix_to_float(static_cast<long long>(first)) * vfirst : 0.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;
        float G = 0.f, A = 0.f;
#pragma unroll 4
        for (int k = lane; k < r.cnt[a]; k += 32) {
          const u64 pos = fix_at(r.A0[a], r.D[a], static_cast<u32>(k));
          const int nb = count_before(pos, b < a, r.A0[b], r.D[b], r.cnt[b], rd[b], many);
          const int nc = count_before(pos, c < a, r.A0[c], r.D[c], r.cnt[c], rd[c], many);
          const int off = r.off + k * r.step[a] + nb * r.step[b] + nc * r.step[c];
          const float vb = gather<DT>(vd, off), va = gather<DT>(vd, off + r.step[a]);
          u64 next = kFixMax;  // the end of the segment after the crossing
          if (k + 1 < r.cnt[a]) next = min(next, pos + r.D[a]);
          if (nb < r.cnt[b]) next = min(next, fix_at(r.A0[b], r.D[b], static_cast<u32>(nb)));
          if (nc < r.cnt[c]) next = min(next, fix_at(r.A0[c], r.D[c], static_cast<u32>(nc)));
          F = fmaf(fix_to_float(static_cast<long long>(next - pos)), va, F);
          const float wgt = vb - va;
          G += wgt;
          A = fmaf(wgt, fix_to_float(static_cast<long long>(pos)), A);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          G += __shfl_xor_sync(kAll, G, o);
          A += __shfl_xor_sync(kAll, A, o);
        }
        q.G[a] = G;
        q.A[a] = A;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) F += __shfl_xor_sync(kAll, F, o);
      q.E = F * r.unit * sqrtf(fmaf(r.d[2], r.d[2], fmaf(r.d[1], r.d[1], r.d[0] * r.d[0])));
      const float ex = static_cast<float>(kExitUnits);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (a == r.ea) q.G[a] -= vfirst;  // entry crossing: weight 0 - V first, at 0
        if (a == r.xa) {                  // exit crossing: weight V last - 0
          q.G[a] += vl;
          q.A[a] = fmaf(vl, ex, q.A[a]);
        }
        q.A[a] *= r.unit;
      }
      q.Gc = (r.ea < 0 ? -vfirst : 0.f) + (r.xa < 0 ? vl : 0.f);
      q.Ac = r.xa < 0 ? vl * ex * r.unit : 0.f;
      const float rest = pick3(q.dom, q.G[1] + q.G[2], q.G[0] + q.G[2], q.G[0] + q.G[1]) + q.Gc;
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (a == q.dom) q.G[a] = -rest;  // the sum of all crossing weights is 0
    }
    if (lane == L) *out = x;
  }
}

// Pairs of crossings that the loops' coordinates cannot order (closer than t0 / t1),
// put in order by their FP64 positions (ties to the lower axis, as exact_rays), and
// the voxels that the loops took wrongly corrected in the sums: those before and
// after a minor crossing, and the one entered at a dominant plane.  near: the pieces
// with such a pair (bit p: slot 0, bit 8 + p: slot 1), which alone are gone through
// again, without gathers but for the pairs.  On a generic pose 1 ray in 2000 has a
// pair, on axis-aligned ones up to half of them do, with ~3 each.  Such rays summed
// again one after another (exact_rays) took 8 times as long as the walk.  Measured
// with Jacobian, 16 poses of 256x256 at 1 mm on 256^3: no rotation 3335 -> 637 us, a
// quarter turn 1937 -> 540, generic poses 397 -> 390; CT batch unrotated 586 -> 341.
// Of the first, 300 are the walk, 70 the second setup, 95 looking for the pairs; with
// FP64 positions compared pair by pair it took 160 more.
template <int DT>
__device__ __forceinline__ void settle_pairs(const VolumeDev& vd, const PoseGeom& pg, int h, int w, const SlabRay& s,
                                             const Plan& pl, u32 near, SlabTotals& T) {
  static_assert(kPieces <= 8, "8 bits per slot");
  // alpha of each slot's crossing 0 and per plane, from FP64 to 2^-62: integers, since the
  // pairs of a tile's rays are settled one by one and FP64 is narrow on this GPU
  using i64 = long long;
  i64 A[3], D[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int a = s.axis(k);
    const double g = fabs(fma(static_cast<double>(h), pg.gh[a], fma(static_cast<double>(w), pg.gw[a], pg.g00[a])));
    double r = rcp_fast(g);
    r = fma(r, fma(-g, r, 1.0), r);
    const double U = s.step[k] > 0 ? pg.u0[a] : pg.un[a];  // the source, in the ray's direction
    constexpr double kOne = 4611686018427387904.0;         // 2^62
    A[k] = s.cnt[k] > 0 ? static_cast<i64>((static_cast<double>(s.i0[k] + 1) - U) * r * kOne) : 0;
    D[k] = s.cnt[k] > 0 ? static_cast<i64>(r * kOne) : 0;
  }
  const auto pos = [&](int k, int i) { return A[k] + static_cast<i64>(i) * D[k]; };
  const auto before = [&](int a, i64 pa, int b, i64 pb) { return pa < pb || (pa == pb && s.axis(a) < s.axis(b)); };
  // crossings of slot k before position P of slot a, n by the loops, where the n-th is near P
  const auto settled = [&](int k, int n, int a, i64 P) {
    return n < 1 ? 0 : (n > s.cnt[k] ? s.cnt[k] : (before(k, pos(k, n - 1), a, P) ? n : n - 1));
  };
  const auto offset = [&](int k0, int k1, int k2) { return s.off + k0 * s.step[0] + k1 * s.step[1] + k2 * s.step[2]; };
  float3 d[2] = {make_float3(0.f, 0.f, 0.f), make_float3(0.f, 0.f, 0.f)};
  // crossing k of slot a (0 or 1): its slab n2 and voxel at `was` by the loops, m2 and `is` in order
  const auto correct = [&](int a, int k, u32 f, int was, int is, int slabs) {
    if (was == is) return;
    const float wo = gather<DT>(vd, was + s.step[a]) - gather<DT>(vd, was);
    const float wn = gather<DT>(vd, is + s.step[a]) - gather<DT>(vd, is);
    d[a].x += wn - wo;
    d[a].y += fmaf(wn - wo, static_cast<float>(f), wn * (static_cast<float>(slabs) * 4294967296.f));
    d[a].z = fmaf(wn - wo, static_cast<float>(k), d[a].z);
  };
  const auto X0 = [&](int k) { return s.mX + static_cast<u64>(static_cast<u32>(k)) * s.mdX; };
  const auto X1 = [&](int j) { return s.lX + static_cast<u64>(static_cast<u32>(j)) * s.ldX; };
  const auto at_plane = [&](u64 X, u32 t, int q) { return static_cast<u32>(X) < 2u * t && static_cast<int>(X >> 32) == q; };
  // counts by the loops at dominant crossing q - 1, and the voxel entered there with k0, k1 in order
  const auto Y2 = [&](int q) { return static_cast<int>((s.Y + static_cast<u64>(static_cast<u32>(q - 1)) * s.dy) >> 32); };
  const auto Z2 = [&](int q) { return static_cast<int>((s.Z + static_cast<u64>(static_cast<u32>(q - 1)) * s.dz) >> 32); };
  const auto enter = [&](int q, int n0, int n1, int k0, int k1) {
    if (n0 != k0 || n1 != k1) T.S.add(gather<DT>(vd, offset(k0, k1, q)) - gather<DT>(vd, offset(n0, n1, q)));
  };
  for (u32 m = near & 0xffu; m; m &= m - 1u) {
    const int p = __ffs(static_cast<int>(m)) - 1, end = piece_start(pl.slot[0], p + 1, s.cnt[0]);
    int k = piece_start(pl.slot[0], p, s.cnt[0]);
    u64 X = X0(k), Z = s.mZ + static_cast<u64>(static_cast<u32>(k)) * s.mdz;
    for (; k < end; ++k, X += s.mdX, Z += s.mdz) {
      const bool nx = static_cast<u32>(X) < 2u * s.t0, nz = static_cast<u32>(Z) < 2u * s.t0;
      if (!nx && !nz) continue;
      const int n2 = static_cast<int>(X >> 32), n1 = static_cast<int>(Z >> 32);
      const i64 P = pos(0, k);
      const int m2 = nx ? settled(2, n2, 0, P) : n2, m1 = nz ? settled(1, n1, 0, P) : n1;
      correct(0, k, static_cast<u32>(X), offset(k, n1, n2), offset(k, m1, m2), n2 - m2);
      if (nx && n2 >= 1 && n2 <= s.cnt[2]) {
        const int k0 = Y2(n2), k1 = Z2(n2);
        const i64 Q = pos(2, n2 - 1);
        int j1 = k1;
        for (int j = max(k1 - 1, 0); j <= k1 && j < s.cnt[1]; ++j)
          if (at_plane(X1(j), s.t1, n2)) j1 = before(1, pos(1, j), 2, Q) ? j + 1 : j;
        enter(n2, k0, k1, before(0, P, 2, Q) ? k + 1 : k, j1);
      }
    }
  }
  for (u32 m = near >> 8; m; m &= m - 1u) {
    const int p = __ffs(static_cast<int>(m)) - 1, end = piece_start(pl.slot[1], p + 1, s.cnt[1]);
    int j = piece_start(pl.slot[1], p, s.cnt[1]);
    u64 X = X1(j), Y = s.lY + static_cast<u64>(static_cast<u32>(j)) * s.ldY;
    for (; j < end; ++j, X += s.ldX, Y += s.ldY) {
      const bool nx = static_cast<u32>(X) < 2u * s.t1, ny = static_cast<u32>(Y) < 2u * s.t1;
      if (!nx && !ny) continue;
      const int n2 = static_cast<int>(X >> 32), n0 = static_cast<int>(Y >> 32);
      const i64 P = pos(1, j);
      const int m2 = nx ? settled(2, n2, 1, P) : n2, m0 = ny ? settled(0, n0, 1, P) : n0;
      correct(1, j, static_cast<u32>(X), offset(n0, j, n2), offset(m0, j, m2), n2 - m2);
      if (nx && n2 >= 1 && n2 <= s.cnt[2]) {
        const int k0 = Y2(n2), k1 = Z2(n2);
        bool done = false;  // with slot 0's crossing near the same plane
        for (int k = max(k0 - 1, 0); k <= k0 && k < s.cnt[0]; ++k) done = done || at_plane(X0(k), s.t0, n2);
        if (!done) enter(n2, k0, k1, k0, before(1, P, 2, pos(2, n2 - 1)) ? j + 1 : j);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    T.minor[a].x += d[a].x;
    T.minor[a].y += d[a].y;
    T.minor[a].z += d[a].z;
  }
}

// From the pieces' totals to the ray's sums (see the section comment).
// Called by all 32 lanes of a warp; live: the lane has a ray.
template <int MODE, int DT>
__device__ __forceinline__ void slab_finish(const VolumeDev& vd, const PoseGeom& pg, int h, int w, bool live,
                                            const SlabRay& s, const SlabTotals& T, Park* park, JacSums& out) {
  const int t = threadIdx.x;
  const float v1 = gather<DT>(vd, s.off);
  const float vl = gather<DT>(vd, s.off + s.cnt[0] * s.step[0] + s.cnt[1] * s.step[1] + s.cnt[2] * s.step[2]);
  // sum w (1 - f), f the unbiased fraction; inside one slab, sum w (length - f) (its
  // 1 - f and rest would be two numbers near a slab that cancel to the length)
  const float to = s.cnt[2] == 0 ? s.w1 : 1.f;
  const float g0 = T.minor[0].x, g1 = T.minor[1].x;
  const float b0 = static_cast<float>(s.t0) * kTwoM32, b1 = static_cast<float>(s.t1) * kTwoM32;
  Sum2 sum = T.S;
  sum.add(fmaf(-kTwoM32, T.minor[0].y, fmaf(b0, g0, to * g0)));
  sum.add(fmaf(-kTwoM32, T.minor[1].y, fmaf(b1, g1, to * g1)));
  sum.add_product(v1, s.w1);
  sum.add_product(-s.rest, vl);
  const float F = sum.value();
  // a sum that is not finite (an infinite or NaN voxel) is taken segment by segment instead
  const bool exact = live && (s.exact || !(fabsf(F) <= 3.0e38f));
  const u32 mask = __ballot_sync(0xffffffffu, exact);
  if (mask) {
    ExactRay x;
    exact_rays<DT>(vd, pg, mask, h, w, &x);
    if (exact) {
      out = x.q;
      if (MODE != kGeoGrad) {
#pragma unroll
        for (int a = 0; a < 3; ++a) park->v[kPkE + a][t] = x.e[a];
      } else {
        park->v[kPkE][t] = x.c;
        park->v[kPkE + 1][t] = x.amin;
      }
      return;
    }
  }
  out.E = ff_scaled(sum, make_float2(park->v[kPkMm][t], park->v[kPkMm + 1][t]));
  float G0 = -g0, G1 = -g1;
  float A0 = -fmaf(park->v[kPkRg][t], T.minor[0].z, park->v[kPkF0][t] * g0);
  float A1 = -fmaf(park->v[kPkRg + 1][t], T.minor[1].z, park->v[kPkF0 + 1][t] * g1);
  const float ex = vl * park->v[kPkSpan][t];
  // entry crossing: weight 0 - V first at alpha 0; exit crossing: V last - 0 at the span
  float Gc = 0.f, Ac = 0.f;
  const int es = s.entry_slot(), xs = s.exit_slot(), ax0 = s.axis(0), ax1 = s.axis(1);
  if (es == 3) Gc -= v1;
  if (es == 0) G0 -= v1;
  if (es == 1) G1 -= v1;
  if (xs == 3) { Gc += vl; Ac = ex; }
  if (xs == 0) { G0 += vl; A0 += ex; }
  if (xs == 1) { G1 += vl; A1 += ex; }
  out.dom = s.axis(2);
#pragma unroll
  for (int a = 0; a < 3; ++a) {  // static indices: the arrays stay in registers
    out.G[a] = a == ax0 ? G0 : (a == ax1 ? G1 : -(G0 + G1 + Gc));  // sum of all crossing weights is 0
    out.A[a] = a == ax0 ? A0 : (a == ax1 ? A1 : 0.f);              // the dominant axis is handled through R
  }
  out.Gc = Gc;
  out.Ac = Ac;
}

// The same where lanes of the warp have pairs of crossings to settle (valid: the lane
// has a pixel).  The rays are set up again, out of line, rather than kept through the
// loops.
template <int MODE, int DT>
__device__ __noinline__ void settled_finish(const VolumeDev& vd, const PoseGeom& pg, const GeomFF& gf, int h, int w,
                                            bool valid, u32 near, SlabTotals& T, Park* park, JacSums* out) {
  SlabRay s;
  const int rs = valid ? slab_setup<MODE>(vd, pg, gf, h, w, s, park) : 0;
  if (rs <= 0) slab_idle(vd, s);
  const Plan pl = plan_pieces(s);  // as the loops had it
  if (near) settle_pairs<DT>(vd, pg, h, w, s, pl, near, T);
  slab_finish<MODE, DT>(vd, pg, h, w, rs > 0, s, T, park, *out);
}
template <int MODE, int DT>
__device__ __forceinline__ void finish_ray(const VolumeDev& vd, const PoseGeom& pg, const GeomFF& gf, int h, int w,
                                           bool valid, int rs, const SlabRay& s, const SlabTotals& T, u32 near,
                                           Park* park, JacSums& out) {
  if (__any_sync(0xffffffffu, near != 0u)) {
    SlabTotals t = T;
    JacSums x;
    settled_finish<MODE, DT>(vd, pg, gf, h, w, valid, near, t, park, &x);
    out = x;
  } else {
    slab_finish<MODE, DT>(vd, pg, h, w, rs > 0, s, T, park, out);
  }
}

// dE/d eta for one ray from the crossing sums (Sec. 2.4 with the voxel lookup
// held fixed).  With d = p - s, L = |d|, absolute alphas A_abs = A + amin G:
//   dE/dt_a = dE/ds_a + dE/dp_a = -L G_a / d_a
//   dE/dp_a = d_a F / L - L A_abs_a / d_a
// and for the dominant axis the second line is rearranged with
// A_abs = F - R (R = the other axes' and the clamped points' A_abs) into
//   dE/dp_a = (L R - F (L^2 - d_a^2) / L) / d_a,
// which has no cancellation for rays nearly along that axis.
//   dE/d eta_j = dE/dt . (dR_j s_c) + dE/dp . (dR_j (p_c - s_c)).
// gt = dE/dt, gp = dE/dp in world units.
__device__ __forceinline__ void ray_world_grads(const float d[3], const JacSums& s, float gt[3], float q[3]) {
  const float L2 = fmaf(d[2], d[2], fmaf(d[1], d[1], d[0] * d[0]));
  const float L = sqrtf(L2);
  const float F = s.E / L;  // in units of alpha
  float R = s.Ac;  // position sums relative to the entry
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (a != s.dom) R += s.A[a];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (d[a] != 0.f) {
      const float Ld = L / d[a];
      gt[a] = -s.G[a] * Ld;
      if (a == s.dom) {
        float D = 0.f;
#pragma unroll
        for (int b = 0; b < 3; ++b)
          if (b != a) D = fmaf(d[b], d[b], D);
        q[a] = (L * R - F * D / L) / d[a];
      } else {
        q[a] = d[a] * F / L - s.A[a] * Ld;
      }
    } else {
      gt[a] = 0.f;
      q[a] = 0.f;
    }
  }
}

__device__ __forceinline__ void pose_jacobian(const float d[3], const JacSums& s, const PoseGeom& pg,
                                              const float e[3], int h, int w, float scale, float J[6]) {
  float gt[3], q[3];
  ray_world_grads(d, s, gt, q);
  // an angle moves the entry point e by omega_j x (e - t): its term is
  // gt . (omega_j x (e - t)) = omega_j . ((e - t) x gt)
  const float x0 = e[0] - pg.t[0], x1 = e[1] - pg.t[1], x2 = e[2] - pg.t[2];
  const float c0 = fmaf(x1, gt[2], -x2 * gt[1]), c1 = fmaf(x2, gt[0], -x0 * gt[2]), c2 = fmaf(x0, gt[1], -x1 * gt[0]);
  const float fw = static_cast<float>(w), fh = static_cast<float>(h);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    float acc = fmaf(pg.Om[j][0], c0, fmaf(pg.Om[j][1], c1, pg.Om[j][2] * c2));
#pragma unroll
    for (int a = 0; a < 3; ++a) acc = fmaf(q[a], fmaf(fh, pg.Hv[j][a], fmaf(fw, pg.Wv[j][a], pg.Q[j][a])), acc);
    J[j] = acc * scale;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) J[3 + a] = gt[a] * scale;
}

// dE/d(sdr, dh, dw) for one ray: the detector parameters (the paper notes the
// generator also differentiates with respect to the source-to-detector
// distance 2 rho and the pixel spacing, Sec. 3.2).  With s = R (rho,0,0) + t,
// rho = sdr / 2, p = R (-rho, (w - wc) dw, (h - hc) dh) + t and dE/ds = gt - gp:
//   dE/dsdr = (dE/ds - dE/dp) . R e_x / 2,
//   dE/ddh  = (h - hc) dE/dp . R e_z,   dE/ddw = (w - wc) dE/dp . R e_y.
__device__ __forceinline__ void geometry_jacobian(const float d[3], const JacSums& s, const PoseGeom& pg, float am,
                                                  float c, int h, int w, float scale, float J[3]) {
  float gt[3], q[3];
  ray_world_grads(d, s, gt, q);
  // am = amin, c = 1 - 2 amin; dE/dp = q + amin gt; dE/ds - dE/dp = gt - 2 dE/dp = (1 - 2 amin) gt - 2 q
  float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float gp = fmaf(am, gt[a], q[a]);
    a0 = fmaf(fmaf(c, gt[a], -2.f * q[a]), pg.Rc[0][a], a0);
    a1 = fmaf(gp, pg.Rc[2][a], a1);
    a2 = fmaf(gp, pg.Rc[1][a], a2);
  }
  J[0] = 0.5f * a0 * scale;
  J[1] = (static_cast<float>(h) - pg.hc) * a1 * scale;
  J[2] = (static_cast<float>(w) - pg.wc) * a2 * scale;
}

// Back-projection adds of one warp step, merged down each column of the warp's
// TW x (32 / TW) pixel tile: the lanes of one column (pixels h, h+1, ... at the
// same w) whose rays are in the same voxel at this step add once, through the
// first lane of each run of equal addresses, the run's sum found by a segmented
// suffix scan over the column.  The L2 serves every lane's atomic as its own
// sector operation, so each lane merged away is one L2 operation less; rays a
// pixel apart along h often share a voxel (2.5 mm CT slices against 0.7 mm
// pixels at the isocentre).  Addresses at or beyond nvox add nothing.
#ifndef DRR_BP_MERGE_ROWS
#define DRR_BP_MERGE_ROWS 8  // runs are merged within aligned groups of this many rows (a power of two)
#endif
template <int TW>
__device__ __forceinline__ void red_column_merged(float* __restrict__ gvol, unsigned int addr, float v,
                                                  unsigned int nvox, int lane) {
  constexpr unsigned int kAll = 0xffffffffu;
  constexpr int TH = 32 / TW;
  constexpr int kRows = DRR_BP_MERGE_ROWS < TH ? DRR_BP_MERGE_ROWS : TH;
  const int hrow = lane / TW;
  const unsigned int a_dn = __shfl_down_sync(kAll, addr, TW);
  bool lk = (hrow + 1) % kRows != 0 && a_dn == addr;  // the pixel below adds to the same voxel
  const unsigned int first = __ballot_sync(kAll, lk);
  unsigned int lkm = first;
  float s = v;
#pragma unroll
  for (int d = 1; d < kRows; d *= 2) {
    // s: the run's sum over rows hrow .. hrow + d - 1; lk: the run goes on past them
    const float s_dn = __shfl_down_sync(kAll, s, d * TW);
    if (lk) s += s_dn;
    if (2 * d < kRows) {
      lk = lk && ((lkm >> ((lane + d * TW) & 31)) & 1u);
      lkm = __ballot_sync(kAll, lk);
    }
  }
  // the first row of each run within its group adds
  const bool head = hrow % kRows == 0 || !((first >> ((lane - TW) & 31)) & 1u);
  if (head && addr < nvox) atomicAdd(gvol + addr, s);
}

// Segments of the rays of `mask` in exact crossing order, as exact_rays finds them
// (all 32 lanes share one ray's crossings; the segment after each crossing is
// added), for the rays that slab_setup leaves to FP64.
__device__ __noinline__ void backproject_exact(const VolumeDev& vd, const PoseGeom& pg, u32 mask, int h, int w, float g,
                                               float* __restrict__ gvol) {
  constexpr u32 kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const u32 nvox = static_cast<u32>(vd.n[0] * vd.n[1] * vd.n[2]);
  for (; mask; mask &= mask - 1u) {
    const int L = __ffs(static_cast<int>(mask)) - 1;
    const int hh = __shfl_sync(kAll, h, L), ww = __shfl_sync(kAll, w, L);
    const float gg = __shfl_sync(kAll, g, L);
    RaySetup r;
    if (ray_setup(vd, pg, hh, ww, r) <= 0) continue;  // the same for all lanes
    const float s = gg * sqrtf(fmaf(r.d[2], r.d[2], fmaf(r.d[1], r.d[1], r.d[0] * r.d[0]))) * r.unit;
    const bool many = max(max(r.cnt[0], r.cnt[1]), r.cnt[2]) >= (1 << 20);
    const auto add = [&](int ix, int iy, int iz, u64 len) {
      const u32 lin = static_cast<u32>(ix + vd.n[0] * (iy + vd.n[1] * iz));
#if DRR_CHECK_BOUNDS
      if (lin >= nvox) atomicOr(&g_fault_word, kFaultBackproject);
#endif
      if (lin < nvox) atomicAdd(gvol + lin, s * fix_to_float(static_cast<long long>(len)));
    };
    float rd[3];
    int sg[3];
    u64 first = kFixMax;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      rd[a] = 1.f / fix_to_float(static_cast<long long>(r.D[a]));
      sg[a] = r.step[a] > 0 ? 1 : -1;
      if (r.cnt[a] > 0) first = min(first, r.A0[a]);
    }
    if (lane == 0) add(r.ient[0], r.ient[1], r.ient[2], first);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;
      for (int k = lane; k < r.cnt[a]; k += 32) {
        const u64 pos = fix_at(r.A0[a], r.D[a], static_cast<u32>(k));
        const int nb = count_before(pos, b < a, r.A0[b], r.D[b], r.cnt[b], rd[b], many);
        const int nc = count_before(pos, c < a, r.A0[c], r.D[c], r.cnt[c], rd[c], many);
        u64 next = kFixMax;  // the end of the segment after the crossing
        if (k + 1 < r.cnt[a]) next = min(next, pos + r.D[a]);
        if (nb < r.cnt[b]) next = min(next, fix_at(r.A0[b], r.D[b], static_cast<u32>(nb)));
        if (nc < r.cnt[c]) next = min(next, fix_at(r.A0[c], r.D[c], static_cast<u32>(nc)));
        int i[3];
        i[a] = r.ient[a] + (k + 1) * sg[a];
        i[b] = r.ient[b] + nb * sg[b];
        i[c] = r.ient[c] + nc * sg[c];
        add(i[0], i[1], i[2], next - pos);
      }
    }
  }
}

// Back-projection walk: grad_V[voxel] += g L (a_{m+1} - a_m), the transpose of
// the forward map V -> E (Eq. 2 is linear in V), into an unpadded (nz, ny, nx)
// FP32 volume.  The crossings are those of the forward walk, in chunks from exact
// counts (walk_forward).  All 32 lanes step together, since their adds are merged
// across lanes, and a ray starts at the step that is its entry voxel's level, the
// sum of the voxel indexes counted along the ray: every step adds one to it, so
// rays of the tile that pass through a voxel do so at the same step, and their
// adds merge.  A waiting ray takes dominant crossings before its entry; lengths
// are clipped to [entry, exit], so those before and after the ray add nothing.
// gL: g |p - s| alpha per dominant plane; nseg = 0: a lane without a ray.
//
// What bounds it: the L2's tag stage, 81 % busy with the adds (each lane's add is a
// sector operation of its own), so the merging decides.  12 poses of 181x217 on
// 200x216x180 voxels, forward + both gradients: 960 -> 930 us with this walk against
// one with an FP64 ray setup whose rays all started at the first step (this kernel
// 370 us); without the waiting 955 to 980; 3 blocks per SM 950, tiles of 2 x 16
// pixels 927, of 4 x 8 932.
// Waiting costs steps where a tile's rays enter at far levels (pixels many voxels
// apart, whose rays share no voxels anyway): such tiles, more than an eighth longer
// with it, do without.
#ifndef DRR_BP_WAIT_SHARE
#define DRR_BP_WAIT_SHARE 8
#endif
constexpr int kBpWaitShare = DRR_BP_WAIT_SHARE;
__device__ __forceinline__ void walk_backproject(const VolumeDev& vd, const SlabRay& s, const FwdPark* park, int nseg,
                                                 float gL, float* __restrict__ gvol, int lane) {
  constexpr u32 kAll = 0xffffffffu;
  const int size = chunk_steps(s);
  // unsigned index arithmetic: a lane before its entry or past its exit keeps stepping (wrapping) without adding
  const u32 nx = static_cast<u32>(vd.n[0]), nxy = nx * static_cast<u32>(vd.n[1]);
  const u32 nvox = static_cast<u32>(vd.n[0] * vd.n[1] * vd.n[2]);
  u32 st[3], entry = 0u;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int ax = s.axis(k);
    const u32 u = pick3(ax, 1u, nx, nxy);
    const bool up = s.step[k] > 0;
    entry += u * static_cast<u32>(up ? s.i0[k] : pick3(ax, vd.n[0], vd.n[1], vd.n[2]) - 1 - s.i0[k]);
    st[k] = up ? u : 0u - u;
  }
  const int level = s.i0[0] + s.i0[1] + s.i0[2];
  const int first = __reduce_min_sync(kAll, nseg > 0 ? level : 0x7fffffff);
  int wait = nseg > 0 ? level - first : 0;
  int nmax = __reduce_max_sync(kAll, wait + nseg);
  const int longest = __reduce_max_sync(kAll, nseg);
  if (nmax > longest + longest / kBpWaitShare) {
    wait = 0;
    nmax = longest;
  }
  const int total = nseg - 1;
  Counts c{{0, 0, 0}};
  float ac = s.start;
  u32 lin = entry;
  for (int m = 0; m < nmax;) {  // warp-uniform
    const int n = min(nmax - m, size);
    const int before = max(wait - m, 0);  // steps until the entry
    float x0 = 1e9f, x1 = 1e9f, xe = 0.f, lo = 0.f;
    u64 O = 0ull;
    if (m < wait + nseg) {
      const Around ar = around(s, park, c);
      O = static_cast<u64>(static_cast<u32>(c.k[2])) << 32;
      x0 = local_pos(ar.next[0], O);
      x1 = local_pos(ar.next[1], O);
      xe = local_pos(s.qx, O);
      lo = m <= wait ? s.start : local_pos(ar.at, O);
      lin = entry + static_cast<u32>(c.k[0]) * st[0] + static_cast<u32>(c.k[1]) * st[1] +
            (static_cast<u32>(c.k[2]) - static_cast<u32>(before)) * st[2];
    }
    ac = lo;
    float tx = static_cast<float>(1 - before), ty = x0, tz = x1, ly = 0.f, lz = 0.f;
    int sl = static_cast<int>(lin);
    int live = m - wait;  // the ray's segment of the next step
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const u32 at = static_cast<u32>(sl);
      const float an = walk_step(tx, ty, tz, ly, lz, sl, static_cast<int>(st[2]), static_cast<int>(st[0]),
                                 static_cast<int>(st[1]));
      next_xy(ty, tz, ly, lz, s.r0, s.r1, x0, x1);
      const float end = fminf(fmaxf(an, lo), xe);
      const bool on = static_cast<u32>(live) < static_cast<u32>(nseg);
#if DRR_CHECK_BOUNDS
      // Crossings closer than the positions' rounding may come in another order at the exit, with a
      // segment beyond it that is dropped: two positions l r + x0 (three roundings each, 2^-23 of the
      // position in all) apart by less, and the fixed-point ends by their own 2^-32 of a plane.
      const float tie = fmaf(2.384185791015625e-7f, fmaxf(fabsf(end), fabsf(ac)),
                             fmaf(9.313225746154785e-10f, s.r0 + s.r1, 5.9604644775390625e-8f));  // 2^-22, 2^-30, 2^-24
      if (on && at >= nvox && end - ac > tie) atomicOr(&g_fault_word, kFaultBackproject);
#endif
      red_column_merged<kBpTileW>(gvol, on ? at : 0xffffffffu, gL * (end - ac), nvox, lane);
      ac = end;
      ++live;
    }
    m += n;
    if (m > wait && m < wait + nseg) {
      c.k[2] += static_cast<int>(tx) - 1;
      c.k[0] += static_cast<int>(ly);
      c.k[1] += static_cast<int>(lz);
      // FP32 took the chunk's last crossings in another order
      if (!around(s, park, c).ordered) c = counts_after(s, park, m - wait);
    }
  }
}

// One warp's back-projection of its tile: every lane takes part in the walk,
// with nseg = 0 where its pixel is outside the detector, its upstream gradient
// is zero, the ray misses the volume or the geometry is not finite.
__device__ __forceinline__ void backproject_tile_ray(const VolumeDev& vd, const PoseGeom& pg, const GeomFF& gf, int h,
                                                     int w, bool active, float g, float* __restrict__ gvol,
                                                     FwdPark* park, int lane) {
  SlabRay s;
  const int rs = active ? slab_setup<kFwd>(vd, pg, gf, h, w, s, park) : 0;
  const bool exact = rs > 0 && s.exact;
  const u32 mask = __ballot_sync(0xffffffffu, exact);
  if (mask) backproject_exact(vd, pg, mask, h, w, g, gvol);
  if (rs <= 0 || exact) slab_idle(vd, s);
  const int nseg = rs > 0 && !exact ? s.cnt[0] + s.cnt[1] + s.cnt[2] + 1 : 0;
  walk_backproject(vd, s, park, nseg, nseg > 0 ? g * s.len * s.rg2 : 0.f, gvol, lane);
}

// The ray's outputs from its sums.
template <int MODE>
__device__ __forceinline__ void ray_outputs(const VolumeDev& vd, const PoseGeom& pg, int h, int w, const JacSums& q,
                                            const Park* park, RayResult& res) {
  const int t = threadIdx.x;
  const float d[3] = {park->v[kPkD][t], park->v[kPkD + 1][t], park->v[kPkD + 2][t]};
  res.F = q.E * vd.out_scale;
  if (MODE != kGeoGrad) {
    const float e[3] = {park->v[kPkE][t], park->v[kPkE + 1][t], park->v[kPkE + 2][t]};
    pose_jacobian(d, q, pg, e, h, w, vd.out_scale, res.J);
  } else {
    geometry_jacobian(d, q, pg, park->v[kPkE + 1][t], park->v[kPkE][t], h, w, vd.out_scale, res.J);
  }
}

// The DRR value from the sum of a ray's chunks (all 32 lanes call; rs as
// slab_setup returned it).
template <int DT>
__device__ __forceinline__ float forward_finish(const VolumeDev& vd, const PoseGeom& pg, int h, int w, int rs,
                                                const SlabRay& s, float F) {
  const bool exact = rs > 0 && (s.exact || !(fabsf(F) <= 3.0e38f));  // a voxel that is not finite: segment by segment
  const u32 mask = __ballot_sync(0xffffffffu, exact);
  F *= s.rg2 * s.len;
  if (mask) {
    ExactRay x;
    exact_rays<DT>(vd, pg, mask, h, w, &x);
    if (exact) F = x.q.E;
  }
  return rs < 0 ? __int_as_float(0x7fffffff) : (rs > 0 ? F * vd.out_scale : 0.f);
}

// The rays of one warp tile (all 32 lanes call; a lane outside the detector
// passes valid = false).
template <int MODE, int DT>
__device__ __forceinline__ void trace_tile(const VolumeDev& vd, const PoseGeom& pg, const GeomFF& gf, int h, int w, bool valid,
                                           typename ParkFor<MODE>::type* park, RayResult& res) {
  res.F = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) res.J[k] = 0.f;
  if constexpr (MODE == kFwd) {
    SlabRay s;
    const int rs = valid ? slab_setup<kFwd>(vd, pg, gf, h, w, s, park) : 0;
    if (rs <= 0) slab_idle(vd, s);
    const int size = chunk_steps(s);
    float F = 0.f;
    if (rs > 0) walk_forward<DT>(vd, s, park, size, 0, kChunks, [&](int, float acc) { F += acc; });
    res.F = forward_finish<DT>(vd, pg, h, w, rs, s, F);
  } else {
    SlabRay s;
    const int rs = valid ? slab_setup<MODE>(vd, pg, gf, h, w, s, park) : 0;
    if (rs <= 0) slab_idle(vd, s);
    u32 near = 0u;
    SlabTotals T;
    const Plan pl = plan_pieces(s);
    {
      MinorTotals m;
      least_loop<DT>(vd, s, pl.slot[1], 0, pl.np, [&](int p, const MinorSums& r) {
        near |= r.near < 2u * s.t1 ? 0x100u << p : 0u;
        m.add(r.g, r.c, r.h, piece_start(pl.slot[1], p, s.cnt[1]));
      });
      T.minor[1] = m.value();
    }
    {
      MinorTotals m;
      middle_loop<DT>(vd, s, pl.slot[0], 0, pl.np, [&](int p, const MinorSums& r) {
        near |= r.near < 2u * s.t0 ? 1u << p : 0u;
        m.add(r.g, r.c, r.h, piece_start(pl.slot[0], p, s.cnt[0]));
      });
      T.minor[0] = m.value();
    }
    dominant_loop<DT>(vd, s, pl.slot[2], 0, pl.np, [&](int, float S) { T.S.add(S); });
    JacSums q;
    finish_ray<MODE, DT>(vd, pg, gf, h, w, valid, rs, s, T, near, park, q);
    if (rs < 0) {  // non-finite geometry (e.g. a NaN pose): NaN out, no walk
      res.F = __int_as_float(0x7fffffff);
#pragma unroll
      for (int k = 0; k < 6; ++k) res.J[k] = res.F;
    } else if (rs > 0) {
      ray_outputs<MODE>(vd, pg, h, w, q, park, res);
    }
  }
}

// Persistent walk kernel: each warp claims 8x4-pixel tiles (pose-major order)
// from a per-launch counter until the batch runs out, so no warp slot idles
// while a slower warp of its block finishes, and the grid is exactly what the
// GPU holds at once.  A warp copies its pose's geometry to its own shared slot
// when the pose changes.  Pose-gradient mode writes one partial sum of g . J
// per tile, so the result does not depend on which warp took which tile.
template <int MODE, int DT>
__global__ void __launch_bounds__(kThreads, MODE == kFwdJac || MODE == kPoseGrad || MODE == kGeoGrad ? DRR_JAC_MINB
                                            : MODE == kBackproject                                   ? DRR_BP_MINB
                                                                                                     : DRR_FWD_MINB)
    siddon_kernel(VolumeDev vd, DetDev det, const PoseGeom* __restrict__ pgs, int B, unsigned int* __restrict__ counter,
                  float* __restrict__ out, float* __restrict__ jac, const float* __restrict__ gin,
                  float* __restrict__ partials, float* __restrict__ gvol) {
  __shared__ PoseGeom spg[kThreads / 32];
  constexpr bool kBp = MODE == kBackproject;
  constexpr bool kSlab = !std::is_same_v<typename ParkFor<MODE>::type, NoPark>;
  __shared__ typename ParkFor<MODE>::type ws;
  __shared__ GeomFF sgf[kSlab ? kThreads / 32 : 1];
  grid_dep_wait();
  grid_dep_release();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int TW = kBp ? kBpTileW : kWarpTileW, TH = 32 / TW;
  const int twx = (det.W + TW - 1) / TW;
  const int per_pose = twx * ((det.H + TH - 1) / TH);
  const unsigned int total = static_cast<unsigned int>(per_pose) * static_cast<unsigned int>(B);
  const size_t npix = static_cast<size_t>(det.H) * det.W;
  PoseGeom& pg = spg[warp];
  int cur = -1;
  for (;;) {
    unsigned int tile = 0u;
    if (lane == 0) tile = atomicAdd(counter, 1u);
    tile = __shfl_sync(0xffffffffu, tile, 0);  // also: every lane is done with the previous tile
    if (tile >= total) break;
    const int b = static_cast<int>(tile / static_cast<unsigned int>(per_pose));
    const int tin = static_cast<int>(tile) - b * per_pose;
    if (b != cur) {
      const unsigned int* src = reinterpret_cast<const unsigned int*>(pgs + b);
      unsigned int* dst = reinterpret_cast<unsigned int*>(&pg);
      for (int i = lane; i < static_cast<int>(sizeof(PoseGeom) / 4); i += 32) dst[i] = src[i];
      __syncwarp();
      if (kSlab) {
        geom_ff(pg, sgf[warp]);
        __syncwarp();
      }
      cur = b;
    }
    const int ty = tin / twx, tx = tin - ty * twx;
    const int h = ty * TH + lane / TW, w = tx * TW + lane % TW;
    const bool valid = (w < det.W) && (h < det.H);
    const size_t pix = static_cast<size_t>(h) * det.W + w;
    float gsc = 0.f;
    if (valid && (MODE == kPoseGrad || MODE == kGeoGrad || kBp)) gsc = gin[b * npix + pix];
    if constexpr (kBp) {
      backproject_tile_ray(vd, pg, sgf[warp], h, w, valid && gsc != 0.f, gsc, gvol, &ws, lane);
    } else if constexpr (MODE == kCount) {
      RaySetup rs;
      if (valid) reinterpret_cast<int*>(out)[b * npix + pix] = ray_setup(vd, pg, h, w, rs) > 0 ? rs.nseg : 0;
    } else {
      RayResult r;
      trace_tile<MODE, DT>(vd, pg, sgf[kSlab ? warp : 0], h, w, valid, &ws, r);
      if (MODE == kFwd || MODE == kFwdJac) {
        if (valid) {
          out[b * npix + pix] = r.F;
          if (MODE == kFwdJac) {
#pragma unroll
            for (int k = 0; k < 6; ++k) jac[(static_cast<size_t>(b) * 6 + k) * npix + pix] = r.J[k];
          }
        }
      } else {
        constexpr int nc = MODE == kPoseGrad ? 6 : 3;  // pose or detector parameters
        float c[nc];
#pragma unroll
        for (int k = 0; k < nc; ++k) {
          c[k] = gsc * r.J[k];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) c[k] += __shfl_xor_sync(0xffffffffu, c[k], o);
        }
        if (lane == 0) {
#pragma unroll
          for (int k = 0; k < nc; ++k) partials[(static_cast<size_t>(b) * per_pose + tin) * nc + k] = c[k];
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Split walk for launches too small to fill the GPU (modes kFwd and kFwdJac): a
// block of K warps takes
// one warp tile (8x4 pixels, pose-major); every warp sets up the tile's 32 rays
// and sums its share of the loops' pieces, which it parks in shared memory, and
// the first warp adds each ray's pieces in piece order and finishes the rays.
// The sums and their order are trace_tile's, so the results are the same bits.
// ---------------------------------------------------------------------------
template <int MODE, int DT, int K>
__global__ void __launch_bounds__(32 * K) siddon_split_kernel(VolumeDev vd, DetDev det, const PoseGeom* __restrict__ pgs,
                                                              int B, unsigned int* __restrict__ counter,
                                                              float* __restrict__ out, float* __restrict__ jac) {
  __shared__ PoseGeom pg;
  __shared__ GeomFF gf;
  __shared__ typename ParkFor<MODE>::type park;  // indexed by threadIdx.x (< 32 K)
  struct Piece {
    float S[32];
    float3 minor[MODE == kFwd ? 1 : 2][32];
    unsigned char near[MODE == kFwd ? 1 : 2][32];
  };
  __shared__ Piece piece[MODE == kFwd ? kChunks : kPieces];
  __shared__ unsigned int tile_s;
  grid_dep_wait();
  grid_dep_release();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int twx = (det.W + kWarpTileW - 1) / kWarpTileW;
  const int per_pose = twx * ((det.H + kWarpTileH - 1) / kWarpTileH);
  const unsigned int total = static_cast<unsigned int>(per_pose) * static_cast<unsigned int>(B);
  const size_t npix = static_cast<size_t>(det.H) * det.W;
  int cur = -1;
  for (;;) {
    if (threadIdx.x == 0) tile_s = atomicAdd(counter, 1u);
    __syncthreads();  // also: the block is done with the previous tile
    const unsigned int tile = tile_s;
    if (tile >= total) break;
    const int b = static_cast<int>(tile / static_cast<unsigned int>(per_pose));
    const int tin = static_cast<int>(tile) - b * per_pose;
    if (b != cur) {
      const unsigned int* src = reinterpret_cast<const unsigned int*>(pgs + b);
      unsigned int* dst = reinterpret_cast<unsigned int*>(&pg);
      for (int i = threadIdx.x; i < static_cast<int>(sizeof(PoseGeom) / 4); i += 32 * K) dst[i] = src[i];
      __syncthreads();
      if (warp == 0) geom_ff(pg, gf);
      cur = b;
    }
    __syncthreads();
    const int ty = tin / twx, tx = tin - ty * twx;
    const int h = ty * kWarpTileH + lane / kWarpTileW, w = tx * kWarpTileW + lane % kWarpTileW;
    const bool valid = (w < det.W) && (h < det.H);
    SlabRay s;
    const int rs = valid ? slab_setup<MODE>(vd, pg, gf, h, w, s, &park) : 0;
    if (rs <= 0) slab_idle(vd, s);
    RayResult r;
    if constexpr (MODE == kFwd) {
      const int size = chunk_steps(s), total = s.cnt[0] + s.cnt[1] + s.cnt[2];
      if (rs > 0)
        walk_forward<DT>(vd, s, &park, size, (kChunks * warp + K - 1) / K, (kChunks * (warp + 1) + K - 1) / K,
                         [&](int q, float acc) { piece[q].S[lane] = acc; });
      __syncthreads();
      if (warp == 0) {
        float F = 0.f;
        if (rs > 0)
          for (int q = 0; q == 0 || q * size < total; ++q) F += piece[q].S[lane];
        r.F = forward_finish<DT>(vd, pg, h, w, rs, s, F);
      }
    } else {
      const Plan pl = plan_pieces(s);
      // this warp's share of the pieces
      const int p0 = pl.np * warp / K, p1 = pl.np * (warp + 1) / K;
      least_loop<DT>(vd, s, pl.slot[1], p0, p1, [&](int p, const MinorSums& r) {
        piece[p].near[1][lane] = r.near < 2u * s.t1;
        piece[p].minor[1][lane] = make_float3(r.g, r.c, r.h);
      });
      middle_loop<DT>(vd, s, pl.slot[0], p0, p1, [&](int p, const MinorSums& r) {
        piece[p].near[0][lane] = r.near < 2u * s.t0;
        piece[p].minor[0][lane] = make_float3(r.g, r.c, r.h);
      });
      dominant_loop<DT>(vd, s, pl.slot[2], p0, p1, [&](int p, float S) { piece[p].S[lane] = S; });
      __syncthreads();
      if (warp == 0) {
        r.F = rs < 0 ? __int_as_float(0x7fffffff) : 0.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) r.J[k] = r.F;
        SlabTotals T;
        MinorTotals m[2];
        u32 near = 0u;
        for (int p = 0; p < pl.np; ++p) {
          near |= static_cast<u32>(piece[p].near[0][lane]) << p | static_cast<u32>(piece[p].near[1][lane]) << (8 + p);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float3 q = piece[p].minor[k][lane];
            m[k].add(q.x, q.y, q.z, piece_start(pl.slot[k], p, s.cnt[k]));
          }
          T.S.add(piece[p].S[lane]);
        }
        T.minor[0] = m[0].value();
        T.minor[1] = m[1].value();
        JacSums q;
        finish_ray<kFwdJac, DT>(vd, pg, gf, h, w, valid, rs, s, T, near, &park, q);
        if (rs > 0) ray_outputs<kFwdJac>(vd, pg, h, w, q, &park, r);
      }
    }
    if (warp == 0 && valid) {
      const size_t pix = static_cast<size_t>(h) * det.W + w;
      out[b * npix + pix] = r.F;
      if (MODE == kFwdJac) {
#pragma unroll
        for (int k = 0; k < 6; ++k) jac[(static_cast<size_t>(b) * 6 + k) * npix + pix] = r.J[k];
      }
    }
  }
}

// Pose gradient from a stored Jacobian in one launch (Sec. 2.4, chain rule:
// dL/d eta = sum over pixels of dL/dE * dE/d eta).  One thread-block cluster
// per pose: block r of the cluster sums g * J over the r-th of kJacCluster
// contiguous shares of the pose's pixels (as FP32 value + error with exact
// products: FP64 arithmetic is narrow on this GPU, and where the sum cancels to a
// small component, plain FP32 totals left 1e-8 of sum |g J| in it), writes its six
// sums into a row of block 0's shared memory through the cluster's distributed
// shared memory, and block 0 adds the rows in rank order in FP64.  Every sum has a fixed order, so the result is
// bitwise reproducible, and no partial sums leave the chip.
constexpr int kJacCluster = 8;  // blocks per pose (the portable cluster size)
#ifndef DRR_JAC_THREADS
#define DRR_JAC_THREADS 512
#endif
// Threads per block: two 512-thread blocks share an SM, so a cluster spans 4
// SMs and ~38 clusters run at once (1024-thread blocks allowed 15 at once: a
// 16-pose batch took two waves, 16.8 us).
constexpr int kJacThreads = DRR_JAC_THREADS;

__device__ __forceinline__ void jac_fma4(Sum2 c[6], const float4 gv, const float* __restrict__ jb, int npix, int i) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 jv = __ldcs(reinterpret_cast<const float4*>(jb + static_cast<size_t>(k) * npix) + i);
    c[k].add_product(gv.x, jv.x);
    c[k].add_product(gv.y, jv.y);
    c[k].add_product(gv.z, jv.z);
    c[k].add_product(gv.w, jv.w);
  }
}

__global__ void __cluster_dims__(kJacCluster, 1, 1) __launch_bounds__(kJacThreads)
    jac_grad_kernel(const float* __restrict__ gin, const float* __restrict__ jac, int npix, int vec,
                    float* __restrict__ grad) {
  static_assert(kJacThreads % 32 == 0 && kJacThreads <= 32 * 32, "the block sum takes one warp sum per lane");
  __shared__ float2 wsum[kJacThreads / 32][6];
  __shared__ double rows[kJacCluster][6];  // filled in block 0 only
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned int rank = cluster.block_rank();
  const int b = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  grid_dep_wait();
  grid_dep_release();
  const float* gb = gin + static_cast<size_t>(b) * npix;
  const float* jb = jac + static_cast<size_t>(b) * 6 * npix;
  Sum2 c[6];
  if (vec) {  // npix % 4 == 0 and 16-byte aligned planes: float4 loads
    const int nv = npix >> 2;
    const int lo = static_cast<int>(static_cast<int64_t>(nv) * rank / kJacCluster);
    const int hi = static_cast<int>(static_cast<int64_t>(nv) * (rank + 1) / kJacCluster);
#pragma unroll 1
    for (int i = lo + threadIdx.x; i < hi; i += kJacThreads)
      jac_fma4(c, __ldcs(reinterpret_cast<const float4*>(gb) + i), jb, npix, i);
  } else {
    const int lo = static_cast<int>(static_cast<int64_t>(npix) * rank / kJacCluster);
    const int hi = static_cast<int>(static_cast<int64_t>(npix) * (rank + 1) / kJacCluster);
    constexpr int kU = 4;  // pixels in flight per thread (154 us for 4 poses of 509x451 with one, 42 with FP32 sums)
#pragma unroll 1
    for (int p = lo + threadIdx.x; p < hi; p += kU * kJacThreads) {
      float gv[kU], jv[kU][6];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int q = p + u * kJacThreads;
        gv[u] = q < hi ? __ldcs(gb + q) : 0.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) jv[u][k] = q < hi ? __ldcs(jb + static_cast<size_t>(k) * npix + q) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
#pragma unroll
        for (int k = 0; k < 6; ++k) c[k].add_product(gv[u], jv[u][k]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) c[k].warp_sum();
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 6; ++k) wsum[warp][k] = make_float2(c[k].s, c[k].e);
  }
  __syncthreads();
  // every block of the cluster is running (its shared memory exists) before any
  // block writes into block 0's
  cluster.sync();
  if (warp == 0) {  // lane q holds warp q's sums; a fixed butterfly adds them
    double mine = 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      Sum2 t;
      if (lane < kJacThreads / 32) t = Sum2{wsum[lane][k].x, wsum[lane][k].y};
      t.warp_sum();
      if (lane == k) mine = t.value64();
    }
    if (lane < 6) cluster.map_shared_rank(&rows[0][0], 0)[rank * 6 + lane] = mine;
  }
  cluster.sync();  // rows complete; no block exits while its row is still being written
  if (rank == 0 && threadIdx.x < 6) {
    double t = 0.0;
    for (int r = 0; r < kJacCluster; ++r) t += rows[r][threadIdx.x];
    grad[6 * b + threadIdx.x] = static_cast<float>(t);
  }
}

// Fixed-order sum of one pose's per-tile partial sums (nt tiles, ncol values each,
// tile-major) to FP64 accuracy: thread t adds tiles t, t + kFinThreads, ... in
// order (one coalesced pass for all columns), each warp's sums are combined by a
// fixed shuffle tree, and thread k adds the warps' sums of column k in warp order.
// The order depends only on nt, so the result is bitwise reproducible, and the
// server and the direct calls, which both finish through here, agree bit for
// bit.  Called by all threads of the block.  The sums run as value + error pairs
// of FP32 (exact but for the rounding of the error, ~2^-46 of the sum) up to the
// warps' totals: as FP64 additions they bounded the kernel (15 us for 3 poses of
// 2720 tiles; this GPU issues FP64 at 1/64 of the FP32 rate).
constexpr int kFinThreads = 256;

__device__ __forceinline__ void sum_pose_partials(const float* __restrict__ p, int nt, int ncol,
                                                  float* __restrict__ out) {
  __shared__ double wsum[kFinThreads / 32][6];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  Sum2 s[6];
#pragma unroll 4
  for (int c = t; c < nt; c += kFinThreads) {
    const float* row = p + static_cast<size_t>(c) * ncol;
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (k < ncol) s[k].add(row[k]);
  }
  bool finite = true;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    s[k].warp_sum();
    finite = finite && isfinite(s[k].s);
    if (lane == 0) wsum[warp][k] = s[k].value64();
  }
  if (__syncthreads_or(!finite)) {  // infinite partial sums, or sums beyond FP32's range: again in FP64
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      double x = 0.0;
      for (int c = t; k < ncol && c < nt; c += kFinThreads) x += static_cast<double>(p[static_cast<size_t>(c) * ncol + k]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) wsum[warp][k] = x;
    }
    __syncthreads();
  }
  if (t < ncol) {
    double a = 0.0;
#pragma unroll
    for (int w = 0; w < kFinThreads / 32; ++w) a += wsum[w][t];
    out[t] = static_cast<float>(a);
  }
  __syncthreads();  // wsum is reused by the block's next pose
}

__global__ void __launch_bounds__(kFinThreads) pose_grad_finalize_kernel(const float* __restrict__ partials, int nblk,
                                                                         int ncol, float* __restrict__ grad) {
  grid_dep_wait();
  const int b = blockIdx.x;
  sum_pose_partials(partials + static_cast<size_t>(b) * nblk * ncol, nblk, ncol, grad + static_cast<size_t>(ncol) * b);
}

// ---------------------------------------------------------------------------
// Volume ingest: HU -> attenuation, storage conversion, padded layout.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float source_value(const void* src, int src_dtype, int64_t i, float mu_water) {
  if (src_dtype == 3) {  // int16 HU: mu = max(0, mu_water (1 + HU/1000))
    const float hu = static_cast<float>(static_cast<const short*>(src)[i]);
    return fmaxf(0.f, mu_water * (1.f + hu / 1000.f));
  }
  return static_cast<const float*>(src)[i];
}

__global__ void abs_max_kernel(const void* __restrict__ src, int src_dtype, int64_t count, float mu_water,
                               unsigned int* __restrict__ out_bits) {
  float m = 0.f;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < count;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    m = fmaxf(m, fabsf(source_value(src, src_dtype, i, mu_water)));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out_bits, __float_as_uint(m));
}

// Padded voxel (pi, pj, pk) is written at pi stride_x + pj stride_y + pk stride_z,
// whichever axis the layout makes fastest; the padding is zero.  A warp takes rows
// (pj, pk) of the padded volume, kIngestAhead lanes' worth of x at a time, so that
// many loads are in flight per lane.  Measured: 200x216x180 FP32 31 -> 12.8 us
// (4.9 TB/s), 512x512x133 HU 147 -> 111 us (bound there by the division and the
// 2-byte loads), against a block of 256 threads per row segment and one voxel per
// thread, which was bound by starting 40,000 to 200,000 short blocks.
constexpr int kIngestAhead = 8;
__global__ void __launch_bounds__(256) ingest_kernel(const void* __restrict__ src, int src_dtype, float mu_water,
                                                     VolumeDev vd, void* __restrict__ dst, float scale) {
  const int px = vd.n[0] + 2, py = vd.n[1] + 2;
  const int64_t rows = static_cast<int64_t>(py) * (vd.n[2] + 2);
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  for (int64_t r = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps) {
    const int pk = static_cast<int>(r / py), pj = static_cast<int>(r - static_cast<int64_t>(pk) * py);
    const int j = pj - 1, k = pk - 1;
    const bool in = j >= 0 && k >= 0 && j < vd.n[1] && k < vd.n[2];
    const int64_t row = (static_cast<int64_t>(k) * vd.n[1] + j) * vd.n[0];
    const int64_t e0 = static_cast<int64_t>(pj) * vd.stride[1] + static_cast<int64_t>(pk) * vd.stride[2];
    for (int base = lane; base < px; base += 32 * kIngestAhead) {
      float v[kIngestAhead];
#pragma unroll
      for (int q = 0; q < kIngestAhead; ++q) {
        const int i = base + 32 * q - 1;
        v[q] = in && i >= 0 && i < vd.n[0] ? source_value(src, src_dtype, row + i, mu_water) : 0.f;
      }
#pragma unroll
      for (int q = 0; q < kIngestAhead; ++q) {
        const int pi = base + 32 * q;
        if (pi >= px) break;
        const int64_t e = static_cast<int64_t>(pi) * vd.stride[0] + e0;
        if (vd.dtype == kF32) {
          static_cast<float*>(dst)[e] = v[q];
        } else if (vd.dtype == kBF16) {
          static_cast<__nv_bfloat16*>(dst)[e] = __float2bfloat16_rn(v[q]);
        } else {
          static_cast<__half*>(dst)[e] = __float2half_rn(v[q] * scale);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Serving tick kernels: one launch each covers every admitted request.
// ---------------------------------------------------------------------------
// Index of the request whose [start, next start) range holds `i` (starts ascending).
__device__ __forceinline__ int find_request(const ServeRequest* reqs, int nreq, int i, bool by_tile) {
  int lo = 0, hi = nreq - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    const int st = by_tile ? reqs[mid].tile_start : reqs[mid].pose_start;
    if (st <= i) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// One warp (block) per pose, grid-stride over the tick's poses.  A pose index
// that decodes outside its request (an inconsistent tick table) sets the
// request's status word and is skipped.
__global__ void __launch_bounds__(32) serve_setup_kernel(const ServeHeader* __restrict__ hdr,
                                                         const ServeRequest* __restrict__ reqs,
                                                         unsigned int* __restrict__ status) {
  const int nreq = hdr->nreq, total = hdr->total_poses;
  for (int i = blockIdx.x; i < total; i += gridDim.x) {
    const int r = find_request(reqs, nreq, i, false);
    const int b = i - reqs[r].pose_start;
    if (b < 0 || b >= reqs[r].B) {  // uniform in the warp
      if (threadIdx.x == 0) atomicOr(status + r, kServePoseRange);
      continue;
    }
    warp_pose_geom(reqs[r].poses + 6 * b, reqs[r].det, reqs[r].vd, reqs[r].geom + b);
  }
}

template <int MODE>
__device__ __forceinline__ void serve_trace(const VolumeDev& vd, const PoseGeom& pg, const GeomFF& gf, int h, int w, bool valid,
                                            typename ParkFor<MODE>::type* park, RayResult& r) {
  switch (vd.dtype) {
    case kF32: trace_tile<MODE, kF32>(vd, pg, gf, h, w, valid, park, r); break;
    case kBF16: trace_tile<MODE, kBF16>(vd, pg, gf, h, w, valid, park, r); break;
    default: trace_tile<MODE, kF16>(vd, pg, gf, h, w, valid, park, r); break;
  }
}

// Persistent walk: warps claim 8x4-pixel tiles of any request (numbered per
// request as in siddon_kernel, pose-major) until the tick's tiles run out, so
// a small request spreads over many SMs.  Render-only tiles run the forward
// walk, gradient tiles the Jacobian walk with the warp's sum of g . J written
// per tile; a warp copies its request's record and pose geometry to its own
// shared slots when they change.
__global__ void __launch_bounds__(kThreads, 3) serve_walk_kernel(const ServeHeader* __restrict__ hdr,
                                                                 const ServeRequest* __restrict__ reqs,
                                                                 unsigned int* __restrict__ status,
                                                                 int* __restrict__ counter) {
  __shared__ PoseGeom spg[kThreads / 32];
  __shared__ ServeRequest sreq[kThreads / 32];
  __shared__ GeomFF sgf[kThreads / 32];
  __shared__ struct {  // apart: at any time a block's warps may walk tiles of both kinds
    ParkFor<kPoseGrad>::type grad;
    ParkFor<kFwd>::type fwd;
  } park;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nreq = hdr->nreq, total = hdr->total_tiles;
  ServeRequest& sr = sreq[warp];
  PoseGeom& pg = spg[warp];
  int cur_r = -1, cur_b = -1;
  for (;;) {
    int t = 0;
    if (lane == 0) t = atomicAdd(counter, 1);
    t = __shfl_sync(0xffffffffu, t, 0);  // also: every lane is done with the previous tile
    if (t >= total) break;
    const int r = find_request(reqs, nreq, t, true);
    if (r != cur_r) {
      const unsigned int* src = reinterpret_cast<const unsigned int*>(reqs + r);
      unsigned int* dst = reinterpret_cast<unsigned int*>(&sr);
      for (int i = lane; i < static_cast<int>(sizeof(ServeRequest) / 4); i += 32) dst[i] = src[i];
      __syncwarp();
      cur_r = r;
      cur_b = -1;
    }
    const int per_pose = pose_tiles(sr.det);
    const int local = t - sr.tile_start;
    const int b = local / per_pose;
    if (b < 0 || b >= sr.B) {  // the tick table's tile ranges, checked (uniform in the warp)
      if (lane == 0) atomicOr(status + r, kServeTileRange);
      continue;
    }
    const int tin = local - b * per_pose;
    if (b != cur_b) {
      const unsigned int* src = reinterpret_cast<const unsigned int*>(sr.geom + b);
      unsigned int* dst = reinterpret_cast<unsigned int*>(&pg);
      for (int i = lane; i < static_cast<int>(sizeof(PoseGeom) / 4); i += 32) dst[i] = src[i];
      __syncwarp();
      geom_ff(pg, sgf[warp]);
      __syncwarp();
      cur_b = b;
    }
    const int twx = (sr.det.W + kWarpTileW - 1) / kWarpTileW;
    const int ty = tin / twx, tx = tin - ty * twx;
    const int h = ty * kWarpTileH + lane / kWarpTileW, w = tx * kWarpTileW + lane % kWarpTileW;
    const bool valid = (w < sr.det.W) && (h < sr.det.H);
    const size_t npix = static_cast<size_t>(sr.det.H) * sr.det.W;
    const size_t pix = static_cast<size_t>(h) * sr.det.W + w;
    const bool want_grad = sr.grad != nullptr;
    RayResult res;
    float gsc = 0.f;
    if (want_grad) {
      if (valid) gsc = sr.grad[b * npix + pix];
      serve_trace<kPoseGrad>(sr.vd, pg, sgf[warp], h, w, valid, &park.grad, res);
    } else {
      serve_trace<kFwd>(sr.vd, pg, sgf[warp], h, w, valid, &park.fwd, res);
    }
    if (valid) sr.out[b * npix + pix] = res.F;
    if (want_grad) {  // uniform across the warp: one partial per tile, as a direct render_backward
      float c[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        c[k] = gsc * res.J[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c[k] += __shfl_xor_sync(0xffffffffu, c[k], o);
      }
      if (lane == 0) {
        const size_t slot = static_cast<size_t>(b) * per_pose + tin;
#pragma unroll
        for (int k = 0; k < 6; ++k) sr.partials[slot * 6 + k] = c[k];
      }
    }
  }
}

// Each gradient request's pose gradients from its per-tile partials: one block
// per pose, summed in the fixed order of sum_pose_partials.
__global__ void __launch_bounds__(kFinThreads) serve_finalize_kernel(const ServeHeader* __restrict__ hdr,
                                                                     const ServeRequest* __restrict__ reqs) {
  const int nreq = hdr->nreq, total = hdr->total_poses;
  for (int i = blockIdx.x; i < total; i += gridDim.x) {
    const int r = find_request(reqs, nreq, i, false);
    const ServeRequest& q = reqs[r];
    if (q.grad == nullptr) continue;  // uniform across the block
    const int b = i - q.pose_start;
    if (b < 0 || b >= q.B) continue;  // flagged by serve_setup_kernel (same decode)
    const int nt = pose_tiles(q.det);
    sum_pose_partials(q.partials + static_cast<size_t>(b) * nt * 6, nt, 6, q.grad_pose + 6 * b);
  }
}

// Launch with programmatic stream serialization (the kernel must begin with
// grid_dep_wait()); -DDRR_PDL=0 launches plainly.
#ifndef DRR_PDL
#define DRR_PDL 1
#endif
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_smem(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                            Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = DRR_PDL ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t stream, Args... args) {
  return launch_pdl_smem(kernel, grid, block, 0, stream, args...);
}

int grid_for(int64_t n, int threads) {
  int64_t g = (n + threads - 1) / threads;
  if (g > 152 * 64) g = 152 * 64;
  return static_cast<int>(g < 1 ? 1 : g);
}

// Blocks of one walk-kernel instance that fit on the device at once (cached per device).
template <int MODE, int DT>
int resident_blocks() {
  constexpr int kMaxDev = 64;
  static std::atomic<int> cache[kMaxDev] = {};  // calls from several host threads may race to fill it
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) dev = 0;
  int v = cache[dev].load(std::memory_order_relaxed);
  if (v == 0) {
    int sms = 0, per_sm = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, siddon_kernel<MODE, DT>, kThreads, 0);
    v = (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
    cache[dev].store(v, std::memory_order_relaxed);
  }
  return v;
}

// The split kernel with K warps per tile: the blocks of it the device holds at
// once (cached per device).
template <int MODE, int DT, int K>
int split_resident_blocks() {
  constexpr int kMaxDev = 64;
  static std::atomic<int> cache[kMaxDev] = {};  // calls from several host threads may race to fill it
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 0;
  int v = cache[dev].load(std::memory_order_relaxed);
  if (v == 0) {
    int sms = 0, per_sm = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, siddon_split_kernel<MODE, DT, K>, 32 * K, 0) !=
        cudaSuccess) {
      cudaGetLastError();
      v = -1;
    } else {
      v = per_sm > 0 ? sms * per_sm : -1;
    }
    cache[dev].store(v, std::memory_order_relaxed);
  }
  return v > 0 ? v : 0;
}

template <int MODE, int DT, int K>
cudaError_t launch_split(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B, unsigned int* counter,
                         float* out, float* jac, cudaStream_t stream) {
  const int64_t tiles = static_cast<int64_t>(pose_tiles(det)) * B;
  const int grid = static_cast<int>(std::min<int64_t>(tiles, split_resident_blocks<MODE, DT, K>()));
  return launch_pdl(siddon_split_kernel<MODE, DT, K>, dim3(grid), dim3(32 * K), stream, vd, det, pg, B, counter, out,
                    jac);
}

// Warps per ray (per warp tile) for a render launch: 8 or 4 when the split
// kernel's resident blocks can take every tile of the launch at once (the
// whole-ray walk would leave most of the GPU idle, latency-bound on few warps),
// 1 otherwise.
template <int MODE, int DT>
int split_lanes(const DetDev& det, int B) {
  const int64_t tiles = static_cast<int64_t>(pose_tiles(det)) * B;
  if (tiles <= split_resident_blocks<MODE, DT, 8>()) return 8;
  if (tiles <= split_resident_blocks<MODE, DT, 4>()) return 4;
  return 1;
}

template <int MODE, int DT>
cudaError_t launch_siddon_dt(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B, unsigned int* counter,
                             float* out, float* jac, const float* gin, float* partials, float* gvol,
                             cudaStream_t stream, int lanes = 1) {
  if constexpr (MODE == kFwd || MODE == kFwdJac) {
    if (lanes == 8) return launch_split<MODE, DT, 8>(vd, det, pg, B, counter, out, jac, stream);
    if (lanes == 4) return launch_split<MODE, DT, 4>(vd, det, pg, B, counter, out, jac, stream);
  }
  const int64_t tiles = static_cast<int64_t>(pose_tiles(det)) * B;
  const int64_t want = (tiles + kThreads / 32 - 1) / (kThreads / 32);
  const int grid = static_cast<int>(std::min<int64_t>(want, resident_blocks<MODE, DT>()));
  return launch_pdl(siddon_kernel<MODE, DT>, dim3(grid), dim3(kThreads), stream, vd, det, pg, B, counter, out, jac, gin,
                    partials, gvol);
}

template <int MODE>
cudaError_t launch_siddon(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B, float* out, float* jac,
                          const float* gin, float* partials, float* gvol, cudaStream_t stream, int lanes = 1) {
  // one counter per walk kind, so a geometry can serve one launch of each
  const int slot = MODE == kPoseGrad ? 1 : (MODE == kBackproject ? 2 : (MODE == kGeoGrad ? 3 : 0));
  unsigned int* counter = reinterpret_cast<unsigned int*>(const_cast<PoseGeom*>(pg) + B) + slot;
  switch (vd.dtype) {
    case kF32:
      return launch_siddon_dt<MODE, kF32>(vd, det, pg, B, counter, out, jac, gin, partials, gvol, stream, lanes);
    case kBF16:
      return launch_siddon_dt<MODE, kBF16>(vd, det, pg, B, counter, out, jac, gin, partials, gvol, stream, lanes);
    default:
      return launch_siddon_dt<MODE, kF16>(vd, det, pg, B, counter, out, jac, gin, partials, gvol, stream, lanes);
  }
}

// ---------------------------------------------------------------------------
// Comparison baseline: the plain FP32 forward path.  The textbook incremental
// Siddon-Jacobs walk (Sec. 2.2, Eq. 2-3) entirely in FP32: one thread per ray
// in 16x16 blocks, FP32 clip (Sec. 2.3), each axis' next crossing advanced by
// repeated FP32 addition, the voxel of the first segment from its midpoint.
// It is what the product walk is measured against; its rounding drift is
// why the product walk anchors its crossings in fixed point.
// ---------------------------------------------------------------------------
template <int DT>
__global__ void __launch_bounds__(256) plain_fp32_kernel(VolumeDev vd, DetDev det, const PoseGeom* __restrict__ pgs,
                                                         float* __restrict__ out) {
  const int w = blockIdx.x * 16 + (threadIdx.x & 15), h = blockIdx.y * 16 + (threadIdx.x >> 4), b = blockIdx.z;
  if (w >= det.W || h >= det.H) return;
  const PoseGeom& pg = pgs[b];
  float u0[3], g[3], amin = 0.f, amax = 1.f;
  bool hit = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    u0[a] = pg.u0f[a];
    g[a] = static_cast<float>(pg.g00[a]) + static_cast<float>(w) * static_cast<float>(pg.gw[a]) +
           static_cast<float>(h) * static_cast<float>(pg.gh[a]);
    if (g[a] != 0.f) {
      const float t0 = -u0[a] / g[a], t1 = (static_cast<float>(vd.n[a]) - u0[a]) / g[a];
      amin = fmaxf(amin, fminf(t0, t1));
      amax = fminf(amax, fmaxf(t0, t1));
    } else if (!(u0[a] >= 0.f && u0[a] < static_cast<float>(vd.n[a]))) {
      hit = false;
    }
  }
  float acc = 0.f;
  if (hit && amin < amax) {
    float an[3], da[3];
    int idx[3], st[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float ue = u0[a] + amin * g[a];
      if (g[a] > 0.f) {
        an[a] = (floorf(ue) + 1.f - u0[a]) / g[a];
        da[a] = 1.f / g[a];
        st[a] = 1;
      } else if (g[a] < 0.f) {
        an[a] = (ceilf(ue) - 1.f - u0[a]) / g[a];
        da[a] = -1.f / g[a];
        st[a] = -1;
      } else {
        an[a] = 2.f;
        da[a] = 0.f;
        st[a] = 0;
      }
    }
    const float first = fminf(fminf(fminf(an[0], an[1]), an[2]), amax);
    const float am = 0.5f * (amin + first);
#pragma unroll
    for (int a = 0; a < 3; ++a) idx[a] = static_cast<int>(floorf(u0[a] + am * g[a]));
    // scalar copies: the walk indexes no register array
    float ax = an[0], ay = an[1], az = an[2];
    int ix = idx[0], iy = idx[1], iz = idx[2];
    float al = amin;
    for (int guard = 0; guard < 4 * (vd.n[0] + vd.n[1] + vd.n[2]) + 8 && al < amax; ++guard) {
      const float nx = fminf(fminf(fminf(ax, ay), az), amax);
      if (ix >= 0 && ix < vd.n[0] && iy >= 0 && iy < vd.n[1] && iz >= 0 && iz < vd.n[2])
        acc += (nx - al) * Voxel<DT>::load(vd.data, vd.origin + ix * vd.stride[0] + iy * vd.stride[1] +
                                                         iz * vd.stride[2]);
      al = nx;
      const bool sx = ax == nx, sy = !sx && ay == nx, sz = !sx && !sy;
      if (sx) { ix += st[0]; ax += da[0]; }
      if (sy) { iy += st[1]; ay += da[1]; }
      if (sz) { iz += st[2]; az += da[2]; }
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) g[a] *= vd.delta[a];
  out[(static_cast<size_t>(b) * det.H + h) * det.W + w] = acc * sqrtf(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]) *
                                                          vd.out_scale;
}

// The comparison server's central differences (see launch_plain_fd_finish).
__global__ void plain_fd_finish_kernel(const float* __restrict__ E13, int B, int npix, float h_rot, float h_trans,
                                       float* __restrict__ out, float* __restrict__ jac) {
  const int64_t n = static_cast<int64_t>(B) * npix;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int b = static_cast<int>(i / npix);
    const int p = static_cast<int>(i - static_cast<int64_t>(b) * npix);
    const float* e = E13 + static_cast<size_t>(b) * 13 * npix + p;
    out[i] = e[0];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float h2 = 2.f * (k < 3 ? h_rot : h_trans);
      jac[(static_cast<size_t>(b) * 6 + k) * npix + p] = (e[static_cast<size_t>(1 + 2 * k) * npix] -
                                                          e[static_cast<size_t>(2 + 2 * k) * npix]) / h2;
    }
  }
}

}  // namespace

cudaError_t read_and_clear_fault(unsigned int* bits) {
  *bits = 0u;
#if DRR_CHECK_BOUNDS
  cudaError_t e = cudaMemcpyFromSymbol(bits, g_fault_word, sizeof(unsigned int));
  if (e != cudaSuccess) return e;
  const unsigned int zero = 0u;
  if (*bits) e = cudaMemcpyToSymbol(g_fault_word, &zero, sizeof(unsigned int));
  return e;
#else
  return cudaSuccess;
#endif
}

bool bounds_checked() { return DRR_CHECK_BOUNDS != 0; }

cudaError_t launch_plain_fd_finish(const float* E13, int B, int npix, float h_rot, float h_trans, float* out,
                                   float* jac, cudaStream_t stream) {
  plain_fd_finish_kernel<<<grid_for(static_cast<int64_t>(B) * npix, 256), 256, 0, stream>>>(E13, B, npix, h_rot,
                                                                                          h_trans, out, jac);
  return cudaGetLastError();
}

cudaError_t launch_render_plain_fp32(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B, float* out,
                                     cudaStream_t stream) {
  dim3 grid((det.W + 15) / 16, (det.H + 15) / 16, B);
  switch (vd.dtype) {
    case kF32: plain_fp32_kernel<kF32><<<grid, 256, 0, stream>>>(vd, det, pg, out); break;
    case kBF16: plain_fp32_kernel<kBF16><<<grid, 256, 0, stream>>>(vd, det, pg, out); break;
    default: plain_fp32_kernel<kF16><<<grid, 256, 0, stream>>>(vd, det, pg, out); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_pose_setup(const float* poses, int B, const DetDev& det, const VolumeDev* vd, PoseGeom* out,
                              cudaStream_t stream) {
  return launch_pdl(pose_setup_kernel, dim3(B), dim3(32), stream, poses, B, det, *vd, out);
}

cudaError_t launch_ray_setup(const float* poses, int B, const DetDev& det, float* rays, cudaStream_t stream) {
  const int64_t n = static_cast<int64_t>(B) * det.H * det.W;
  ray_setup_kernel<<<static_cast<unsigned int>((n + 255) / 256), 256, 0, stream>>>(poses, B, det, rays);
  return cudaGetLastError();
}

namespace {
template <int MODE>
int mode_split_lanes(const VolumeDev& vd, const DetDev& det, int B) {
  switch (vd.dtype) {
    case kF32: return split_lanes<MODE, kF32>(det, B);
    case kBF16: return split_lanes<MODE, kBF16>(det, B);
    default: return split_lanes<MODE, kF16>(det, B);
  }
}
}  // namespace

int render_split_lanes(const VolumeDev& vd, const DetDev& det, int B, bool jacobian) {
  return jacobian ? mode_split_lanes<kFwdJac>(vd, det, B) : mode_split_lanes<kFwd>(vd, det, B);
}

cudaError_t launch_render(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B, float* out, float* jac,
                          cudaStream_t stream, int lanes) {
  if (jac) return launch_siddon<kFwdJac>(vd, det, pg, B, out, jac, nullptr, nullptr, nullptr, stream, lanes);
  return launch_siddon<kFwd>(vd, det, pg, B, out, nullptr, nullptr, nullptr, nullptr, stream, lanes);
}

cudaError_t launch_pose_grad_walk(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B,
                                  const float* grad_drr, float* partials, cudaStream_t stream) {
  return launch_siddon<kPoseGrad>(vd, det, pg, B, nullptr, nullptr, grad_drr, partials, nullptr, stream);
}

cudaError_t launch_pose_grad_from_jacobian(const DetDev& det, int B, const float* grad_drr, const float* jac,
                                           float* grad_pose, cudaStream_t stream) {
  const int npix = det.H * det.W;
  const int vec = (npix % 4 == 0) && (reinterpret_cast<uintptr_t>(grad_drr) % 16 == 0) &&
                  (reinterpret_cast<uintptr_t>(jac) % 16 == 0);
  return launch_pdl(jac_grad_kernel, dim3(kJacCluster, B), dim3(kJacThreads), stream, grad_drr, jac, npix, vec,
                    grad_pose);
}

cudaError_t launch_count_segments(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B, int* counts,
                                  cudaStream_t stream) {
  return launch_siddon<kCount>(vd, det, pg, B, reinterpret_cast<float*>(counts), nullptr, nullptr, nullptr, nullptr,
                               stream);
}

cudaError_t launch_pose_grad_finalize(const float* partials, int B, int nblk, float* grad_pose, cudaStream_t stream) {
  return launch_pdl(pose_grad_finalize_kernel, dim3(B), dim3(kFinThreads), stream, partials, nblk, 6, grad_pose);
}

cudaError_t launch_geometry_grad(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B,
                                 const float* grad_drr, float* partials, float* grad_geometry, cudaStream_t stream) {
  cudaError_t e = launch_siddon<kGeoGrad>(vd, det, pg, B, nullptr, nullptr, grad_drr, partials, nullptr, stream);
  if (e != cudaSuccess) return e;
  return launch_pdl(pose_grad_finalize_kernel, dim3(B), dim3(kFinThreads), stream, static_cast<const float*>(partials),
                    pose_tiles(det), 3, grad_geometry);
}

cudaError_t launch_backproject(const VolumeDev& vd, const DetDev& det, const PoseGeom* pg, int B,
                               const float* grad_drr, float* grad_vol, cudaStream_t stream) {
  return launch_siddon<kBackproject>(vd, det, pg, B, nullptr, nullptr, grad_drr, nullptr, grad_vol, stream);
}

int serve_walk_grid(int device) {
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, serve_walk_kernel, kThreads, 0);
  return max(1, sms * max(per_sm, 1));
}

cudaError_t launch_serve_tick(const ServeHeader* hdr, const ServeRequest* reqs, unsigned int* status, int* counter,
                              int max_poses, int walk_grid, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), stream);
  if (e != cudaSuccess) return e;
  // setup and finalize stride over the tick's poses: one block per pose up to
  // the walk's grid, so that a small tick does not pay for thousands of idle blocks
  const int aux = max(1, min(max_poses, walk_grid));
  serve_setup_kernel<<<aux, 32, 0, stream>>>(hdr, reqs, status);
  serve_walk_kernel<<<walk_grid, kThreads, 0, stream>>>(hdr, reqs, status, counter);
  serve_finalize_kernel<<<aux, kFinThreads, 0, stream>>>(hdr, reqs);
  return cudaGetLastError();
}

cudaError_t launch_abs_max(const void* src, int src_dtype, int64_t count, float mu_water, unsigned int* out_bits,
                           cudaStream_t stream) {
  abs_max_kernel<<<grid_for(count, 256), 256, 0, stream>>>(src, src_dtype, count, mu_water, out_bits);
  return cudaGetLastError();
}

cudaError_t launch_ingest(const void* src, int src_dtype, float mu_water, const VolumeDev& vd, void* dst, float scale,
                          cudaStream_t stream) {
  const int64_t rows = (static_cast<int64_t>(vd.n[1]) + 2) * (static_cast<int64_t>(vd.n[2]) + 2);
  const int grid = static_cast<int>(std::min<int64_t>((rows + 7) / 8, 152 * 8));  // a warp per row, 8 blocks per SM
  ingest_kernel<<<grid, 256, 0, stream>>>(src, src_dtype, mu_water, vd, dst, scale);
  return cudaGetLastError();
}

}  // namespace drr
