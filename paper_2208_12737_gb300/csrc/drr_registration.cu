// Registration support (Sec. 3.2 of the paper: slice-to-volume registration by
// gradient descent on the negative zero-normalised cross-correlation between a
// moving DRR and a fixed image): the ZNCC loss with its image gradient, and an
// Adam step on the pose parameters.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "drr.h"
#include "drr_internal.cuh"

namespace {

// One thread-block cluster per image pair; block r takes the r-th contiguous
// share of the pixels.  What bounded one block per pair was FP64 arithmetic (15
// operations per pixel at 1/64 of the FP32 rate), on one SM per pair.  Per thread
// the sums now run in FP32 with exact products, kept as value + error (Knuth /
// Dekker), and only the threads' partial sums are added in FP64; the image gradient
// is evaluated the same way from FP64 coefficients.  The errors are added in FP32:
// a sum of 2^20 pixels is good to ~2^-43, and a variance to as much of the mean
// square.  Images whose mean square is above kZWide variances (where that would reach
// FP32's bits: 1.7e-5 at a mean of 10^4 deviations) are taken in FP64.  Measured
// (call with gradient, CUDA events): one 256x256 pair 306 -> 19 us, 64 pairs 308 -> 29
// us, 8 pairs of 1024x1024 4400 -> 146 us; 256 pairs of 200x200 without gradient 212 ->
// 64 us, 4096 of them 2770 -> 907 us (two thirds of that the FP64 sums of the partial
// sums and the closing scalars).
constexpr int kZThreads = 256;
constexpr int kZCluster = 8;  // the portable cluster size
constexpr int kZSums = 5;     // sum I, I^2, F, F^2, I F
constexpr double kZWide = 128.0;

struct Acc {  // s + e, an unevaluated sum
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float x) {  // exact but for the rounding of e
    const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z)));
    s = t;
  }
  __device__ __forceinline__ void add_product(float x, float y) {
    const float p = __fmul_rn(x, y);
    add(p);
    e = __fadd_rn(e, __fmaf_rn(x, y, -p));
  }
};

struct Coefficients {  // d loss / dI = A F + B I + C, each h + l
  float Ah, Al, Bh, Bl, Ch, Cl;
};

__device__ __forceinline__ float loss_gradient(const Coefficients& q, float a, float b) {
  const float p = __fmul_rn(q.Ah, b), r = __fmul_rn(q.Bh, a);
  Acc t;
  t.s = p;
  t.e = __fmaf_rn(q.Al, b, __fmaf_rn(q.Ah, b, -p));
  t.add(r);
  t.e = __fadd_rn(t.e, __fmaf_rn(q.Bl, a, __fmaf_rn(q.Bh, a, -r)));
  t.add(q.Ch);
  return __fadd_rn(t.s, __fadd_rn(t.e, q.Cl));
}

__device__ __forceinline__ void split(double x, float& h, float& l) {
  h = static_cast<float>(x);
  l = static_cast<float>(x - static_cast<double>(h));
}

// Calls f(i, I_i, F_i) for this thread's pixels of [lo, hi), in order; vec: in
// aligned groups of four (lo and hi are then multiples of 4).
template <class Fn>
__device__ __forceinline__ void each_pixel(const float* __restrict__ I, const float* __restrict__ F, int lo, int hi,
                                           bool vec, Fn f) {
  if (vec) {
    for (int i = lo + 4 * static_cast<int>(threadIdx.x); i < hi; i += 4 * kZThreads) {
      const float4 a = *reinterpret_cast<const float4*>(I + i), b = *reinterpret_cast<const float4*>(F + i);
      f(i, a.x, b.x);
      f(i + 1, a.y, b.y);
      f(i + 2, a.z, b.z);
      f(i + 3, a.w, b.w);
    }
  } else {
    for (int i = lo + static_cast<int>(threadIdx.x); i < hi; i += kZThreads) f(i, I[i], F[i]);
  }
}

// With population statistics and c = I - mean(I), s = sqrt(mean(c^2)),
// I^ = c / (s + eps) (same for the fixed image F):
//   zncc = mean(I^ F^),  loss = -zncc,
//   d zncc / dI_j = (F^_j - zncc c_j / s) / (N (s + eps)).
// fixed_stride: elements between consecutive fixed images (0: one fixed image for all).
__global__ void __cluster_dims__(kZCluster, 1, 1) __launch_bounds__(kZThreads)
    zncc_kernel(const float* __restrict__ moving, const float* __restrict__ fixed, size_t fixed_stride, int npix,
                float eps, bool vec, float* __restrict__ loss, float* __restrict__ grad) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank()), pair = static_cast<int>(blockIdx.x / kZCluster);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // a block's shared memory may be written by another only once that block runs:
  // every block says so here, and the first remote write below waits for all
  cluster.barrier_arrive();
  __shared__ double part[kZSums][kZThreads];
  __shared__ float range[2][kZThreads / 32];
  __shared__ double rows[kZCluster][kZSums + 2];  // every block's sums and largest magnitudes (I, F)
  __shared__ Coefficients coef;
  __shared__ int again;
  __shared__ double coef64[3];
  const float* I = moving + static_cast<size_t>(pair) * npix;
  const float* F = fixed + static_cast<size_t>(pair) * fixed_stride;
  const int unit = vec ? 4 : 1, n = npix / unit;
  const int lo = static_cast<int>(static_cast<int64_t>(n) * rank / kZCluster) * unit;
  const int hi = static_cast<int>(static_cast<int64_t>(n) * (rank + 1) / kZCluster) * unit;
  // products and coefficients of images far from 1 in magnitude would leave the
  // range of FP32: such images (and images that are not finite) are taken in FP64
  int wide = 0;
  double v[kZSums];  // the pair's sums (thread 0)
  for (;; ++wide) {
    float mi = 0.f, mf = 0.f;
    if (!wide) {
      Acc s[kZSums];
      each_pixel(I, F, lo, hi, vec, [&](int, float a, float b) {
        s[0].add(a);
        s[1].add_product(a, a);
        s[2].add(b);
        s[3].add_product(b, b);
        s[4].add_product(a, b);
        mi = fmaxf(mi, fabsf(a));
        mf = fmaxf(mf, fabsf(b));
      });
#pragma unroll
      for (int k = 0; k < kZSums; ++k) {
        part[k][t] = static_cast<double>(s[k].s) + static_cast<double>(s[k].e);
        if (!isfinite(s[k].s) || !isfinite(s[k].e)) mi = __int_as_float(0x7f800000);
      }
    } else {
      double s[kZSums] = {0.0, 0.0, 0.0, 0.0, 0.0};
      each_pixel(I, F, lo, hi, vec, [&](int, float x, float y) {
        const double a = x, b = y;
        s[0] += a;
        s[1] += a * a;
        s[2] += b;
        s[3] += b * b;
        s[4] += a * b;
      });
#pragma unroll
      for (int k = 0; k < kZSums; ++k) part[k][t] = s[k];
    }
    // (the bits of numbers that are not negative are in the numbers' order)
    const unsigned int ri = __reduce_max_sync(0xffffffffu, __float_as_uint(mi)),
                       rf = __reduce_max_sync(0xffffffffu, __float_as_uint(mf));
    if (lane == 0) {
      range[0][warp] = __uint_as_float(ri);
      range[1][warp] = __uint_as_float(rf);
    }
    __syncthreads();
    if (!wide) cluster.barrier_wait();  // (the second pass: the sync at the end of the first)
    if (warp < kZSums) {  // warp k: the block's sum k, in a fixed order
      double x = 0.0;
#pragma unroll
      for (int q = 0; q < kZThreads / 32; ++q) x += part[warp][32 * q + lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      // to every block of the cluster (one of its lanes each)
      if (lane < kZCluster) cluster.map_shared_rank(&rows[0][0], lane)[rank * (kZSums + 2) + warp] = x;
    } else if (warp < kZSums + 2 && lane < kZCluster) {
      float x = 0.f;
#pragma unroll
      for (int q = 0; q < kZThreads / 32; ++q) x = fmaxf(x, range[warp - kZSums][q]);
      cluster.map_shared_rank(&rows[0][0], lane)[rank * (kZSums + 2) + warp] = static_cast<double>(x);
    }
    cluster.sync();  // every block's rows are complete in every block
    if (t == 0) {    // the same in every block
#pragma unroll
      for (int k = 0; k < kZSums; ++k) {
        double x = 0.0;
#pragma unroll
        for (int r = 0; r < kZCluster; ++r) x += rows[r][k];
        v[k] = x;
      }
      double li = 0.0, lf = 0.0;  // the images' largest magnitudes
#pragma unroll
      for (int r = 0; r < kZCluster; ++r) {
        li = fmax(li, rows[r][kZSums]);
        lf = fmax(lf, rows[r][kZSums + 1]);
      }
      const auto fits = [](double m) { return m == 0.0 || (m > 1e-8 && m < 1e10); };
      // mean square x^2 <= kZWide (x^2 - mean^2), with n = npix: q n <= kZWide (q n - m m)
      const auto spread = [&](double m, double q) {
        const double qn = q * static_cast<double>(npix);
        return qn <= kZWide * (qn - m * m);
      };
      again = !(fits(li) && fits(lf) && spread(v[0], v[1]) && spread(v[2], v[3]));
    }
    __syncthreads();
    if (wide || !again) break;
    cluster.sync();  // all blocks have read the rows before they are written again
  }
  if (t == 0 && (grad || rank == 0)) {  // every block needs the coefficients, one the loss
    const double inv = 1.0 / static_cast<double>(npix);
    const double mi = v[0] * inv, mf = v[2] * inv;
    const double si = sqrt(fmax(v[1] * inv - mi * mi, 0.0)), sf = sqrt(fmax(v[3] * inv - mf * mf, 0.0));
    const double ri = 1.0 / (si + eps), rf = 1.0 / (sf + eps);
    const double zncc = (v[4] * inv - mi * mf) * ri * rf;
    if (rank == 0 && loss) loss[pair] = static_cast<float>(-zncc);
    const double k1 = -inv * ri;  // d loss = -d zncc
    const double A = k1 * rf, B = si > 0.0 ? -k1 * zncc / si : 0.0;
    split(A, coef.Ah, coef.Al);
    split(B, coef.Bh, coef.Bl);
    split(-(A * mf + B * mi), coef.Ch, coef.Cl);
    coef64[0] = A;
    coef64[1] = B;
    coef64[2] = -(A * mf + B * mi);
  }
  cluster.sync();  // no block exits while its rows may still be written; coef is set
  if (!grad) return;
  const Coefficients q = coef;
  float* g = grad + static_cast<size_t>(pair) * npix;
  if (wide) {
    each_pixel(I, F, lo, hi, vec, [&](int i, float a, float b) {
      g[i] = static_cast<float>(fma(coef64[0], static_cast<double>(b), fma(coef64[1], static_cast<double>(a), coef64[2])));
    });
  } else if (vec) {
    for (int i = lo + 4 * t; i < hi; i += 4 * kZThreads) {
      const float4 a = *reinterpret_cast<const float4*>(I + i), b = *reinterpret_cast<const float4*>(F + i);
      *reinterpret_cast<float4*>(g + i) = make_float4(loss_gradient(q, a.x, b.x), loss_gradient(q, a.y, b.y),
                                                      loss_gradient(q, a.z, b.z), loss_gradient(q, a.w, b.w));
    }
  } else {
    for (int i = lo + t; i < hi; i += kZThreads) g[i] = loss_gradient(q, I[i], F[i]);
  }
}

// Adam on the six pose parameters of each of B poses (rotations and
// translations have separate step sizes, Sec. 3.2 uses separate rates too).  In
// FP64, as the rounding of the quotient alone may move an FP32 pose by its last
// bit, which re-orders some rays' crossings and shows in the next gradient.
// u1, u2: 1 - b1^step, 1 - b2^step.
__global__ void adam_kernel(float* __restrict__ params, const float* __restrict__ grads, float* __restrict__ m,
                            float* __restrict__ v, int n, double u1, double u2, float lr_rot, float lr_trans, float b1,
                            float b2, float eps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double g = grads[i], d1 = b1, d2 = b2;
  const double mi = fma(d1, static_cast<double>(m[i]), (1.0 - d1) * g);
  const double vi = fma(d2, static_cast<double>(v[i]), (1.0 - d2) * g * g);
  m[i] = static_cast<float>(mi);
  v[i] = static_cast<float>(vi);
  const double lr = (i % 6) < 3 ? lr_rot : lr_trans;
  params[i] = static_cast<float>(params[i] - lr * (mi / u1) / (sqrt(vi / u2) + static_cast<double>(eps)));
}

}  // namespace

cudaError_t drr::launch_zncc(const float* moving, const float* fixed, size_t fixed_stride, int B, int npix, float eps,
                             float* loss, float* grad, cudaStream_t stream) {
  const uintptr_t at = reinterpret_cast<uintptr_t>(moving) | reinterpret_cast<uintptr_t>(fixed) |
                       reinterpret_cast<uintptr_t>(grad);
  const bool vec = npix % 4 == 0 && fixed_stride % 4 == 0 && at % 16 == 0;
  constexpr int kMost = 1 << 27;  // pairs per launch (the grid's limit)
  for (int b = 0; b < B; b += kMost) {
    const size_t at0 = static_cast<size_t>(b);
    zncc_kernel<<<kZCluster * std::min(B - b, kMost), kZThreads, 0, stream>>>(
        moving + at0 * npix, fixed + at0 * fixed_stride, fixed_stride, npix, eps, vec, loss ? loss + at0 : nullptr,
        grad ? grad + at0 * npix : nullptr);
  }
  return cudaGetLastError();
}

extern "C" drr_status drr_zncc(const float* moving_dev, const float* fixed_dev, int32_t B, int32_t npix,
                               float eps, float* loss_dev, float* grad_dev, void* cuda_stream) {
  if (B <= 0 || npix <= 0) return drr::set_error(DRR_ERR_INVALID, "B and npix must be positive");
  if (!moving_dev || !fixed_dev || (!loss_dev && !grad_dev)) return drr::set_error(DRR_ERR_INVALID, "NULL pointer");
  if (!(eps >= 0.f)) return drr::set_error(DRR_ERR_INVALID, "eps must be >= 0");
  const int dev = drr::current_device();
  if (drr_status s = drr::device_view(moving_dev, dev, true, "moving", &moving_dev)) return s;
  if (drr_status s = drr::device_view(fixed_dev, dev, true, "fixed", &fixed_dev)) return s;
  if (loss_dev) {
    if (drr_status s = drr::device_view(loss_dev, dev, true, "loss", &loss_dev)) return s;
  }
  if (grad_dev) {
    if (drr_status s = drr::device_view(grad_dev, dev, true, "grad", &grad_dev)) return s;
  }
  cudaError_t e = drr::launch_zncc(moving_dev, fixed_dev, static_cast<size_t>(npix), B, npix, eps, loss_dev, grad_dev,
                                   static_cast<cudaStream_t>(cuda_stream));
  if (e != cudaSuccess) return drr::cuda_error(e, "zncc launch");
  drr::count_launches(1);
  return DRR_OK;
}

extern "C" drr_status drr_adam_step(float* params_dev, const float* grads_dev, float* m_dev, float* v_dev, int32_t B,
                                    int32_t step, float lr_rot, float lr_trans, float beta1, float beta2, float eps,
                                    void* cuda_stream) {
  if (B <= 0 || step <= 0) return drr::set_error(DRR_ERR_INVALID, "B and step must be positive");
  if (!params_dev || !grads_dev || !m_dev || !v_dev) return drr::set_error(DRR_ERR_INVALID, "NULL pointer");
  const int dev = drr::current_device();
  if (drr_status s = drr::device_view(params_dev, dev, true, "params", &params_dev)) return s;
  if (drr_status s = drr::device_view(grads_dev, dev, true, "grads", &grads_dev)) return s;
  if (drr_status s = drr::device_view(m_dev, dev, true, "m", &m_dev)) return s;
  if (drr_status s = drr::device_view(v_dev, dev, true, "v", &v_dev)) return s;
  const int n = 6 * B;
  adam_kernel<<<(n + 255) / 256, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      params_dev, grads_dev, m_dev, v_dev, n, 1.0 - std::pow(static_cast<double>(beta1), step),
      1.0 - std::pow(static_cast<double>(beta2), step), lr_rot, lr_trans, beta1, beta2, eps);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return drr::cuda_error(e, "adam launch");
  drr::count_launches(1);
  return DRR_OK;
}
