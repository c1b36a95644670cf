// The forward warp of a rig whose eyes share their rows (equal orientation, the
// baseline along the image's x axis: the head-mounted rig of Sec. 4.2): every
// sample lands in its own image row, so one CTA owns a row, tests depths in
// shared memory and writes the row's winners once. Any other rig scatters to the
// whole image with 64-bit atomics on a cleared buffer.
#pragma once

#include <math.h>

#include "gs_internal.cuh"

namespace gs {

// Do all samples keep their row? Rrel, trel: dominant camera -> affiliated camera.
// With Y / Z = (d (r_y + e1) + t1) / (d (1 + e2) + t2), Z > kZNear, the projected
// row differs from the source's by at most fy times the bound below, for which a
// quarter of a pixel is allowed. The other quarter is for the float32 evaluation: six
// roundings of y - cy and two of the row, below 2^-21 (H + |cy|) in all (0.006 pixel at
// 8192 rows; past 2^19 rows, or with the principal point as far off, the scatter).
inline bool rows_kept(const double *Rrel, const double *trel, double fx, double fy, double cx, double cy, int W,
                      int H) {
  const double rx = fmax(fabs(cx), fabs(W - 1.0 - cx)) / fx, ry = fmax(fabs(cy), fabs(H - 1.0 - cy)) / fy;
  const double e1 = fabs(Rrel[3]) * rx + fabs(Rrel[4] - 1.0) * ry + fabs(Rrel[5]);
  const double e2 = fabs(Rrel[6]) * rx + fabs(Rrel[7]) * ry + fabs(Rrel[8] - 1.0);
  const double t1 = fabs(trel[1]), t2 = fabs(trel[2]), z = (double)kZNear;
  if (!(e2 < 0.5)) return false;
  const double off = (e1 + ry * e2) * (1.0 + t2 / z) / (1.0 - e2) + (t1 + ry * t2) / z;
  return fy * off < 0.25 && 0x1p-21 * (H + fabs(cy)) < 0.25;
}

// The relative pose X_a = Rrel X_d + trel in FP64 (Eq. 4 followed by Eq. 5), each
// sum in order with fused multiply-adds, as the set-up kernel evaluates it.
inline void relative_pose(const double *Rd, const double *td, const double *Ra, const double *ta, double *Rrel,
                          double *trel) {
  for (int i = 0; i < 3; ++i) {
    double tr = 0.0;
    for (int j = 0; j < 3; ++j) {
      double r = 0.0;
      for (int k = 0; k < 3; ++k) r = fma(Ra[k * 3 + i], Rd[k * 3 + j], r);
      Rrel[i * 3 + j] = r;
      tr = fma(Ra[j * 3 + i], td[j] - ta[j], tr);
    }
    trel[i] = tr;
  }
}

constexpr int kRowThreads = 256;
inline size_t row_warp_smem(int W) { return sizeof(unsigned long long) * (size_t)W; }

// CTA-wide: the winners of a row in zbuf[W] (kNoSample: none). sample(x, T, D, u,
// key) gives source pixel x's destination column and (float depth bits << 32 |
// source index) key from its transmittance and depth proxy, or false. A thread's
// next four pixels are loaded before the first of them is tested (one by one, each
// atomic held the next pixel's loads back).
constexpr int kRowAhead = 4;
template <class Sample>
__device__ __forceinline__ void warp_row(unsigned long long *zbuf, const float *__restrict__ trans,
                                         const float *__restrict__ depth, int W, Sample &&sample) {
  float T[kRowAhead], D[kRowAhead];
  auto load = [&](int x0) {
#pragma unroll
    for (int k = 0; k < kRowAhead; ++k) {
      const int x = x0 + k * kRowThreads;
      T[k] = x < W ? __ldg(trans + x) : 1.f;
      D[k] = x < W ? __ldg(depth + x) : 0.f;
    }
  };
  load(threadIdx.x);
  for (int x = threadIdx.x; x < W; x += kRowThreads) zbuf[x] = kNoSample;
  __syncthreads();
  for (int x0 = threadIdx.x; x0 < W; x0 += kRowAhead * kRowThreads) {
    int u[kRowAhead];
    unsigned long long key[kRowAhead];
    bool on[kRowAhead];
#pragma unroll
    for (int k = 0; k < kRowAhead; ++k) {
      const int x = x0 + k * kRowThreads;
      on[k] = x < W && sample(x, T[k], D[k], u[k], key[k]);
    }
    if (x0 + kRowAhead * kRowThreads < W) load(x0 + kRowAhead * kRowThreads);
#pragma unroll
    for (int k = 0; k < kRowAhead; ++k)
      if (on[k]) atomicMin(zbuf + u[k], key[k]);
  }
  __syncthreads();
}

}  // namespace gs
