// SSIM of an image against a reference on the GPU (the quality metric Table 2
// reports beside PSNR), in the convention of the 2DGS/3DGS evaluation code:
// 11 x 11 Gaussian window (sigma 1.5), same-size filtering with zero padding,
// C1 = 0.01^2, C2 = 0.03^2, the mean of the SSIM map over every pixel of every
// channel.
//
// One CTA per 32 x 32 output tile and channel. Four quantities are filtered, as two
// FP32x2 pairs: a = x + y and d = x - y, and their squares. With A, D their means and
// va, vd their variances, 2 mx my = (A^2 - D^2) / 2, mx^2 + my^2 = (A^2 + D^2) / 2, and
// likewise 2 sxy and sxx + syy from va and vd. So the map's two factors are
//   1 - 2 D^2 / (A^2 + D^2 + 2 C1)  and  1 - 2 vd / (va + vd + 2 C2),
// and half of what their product lacks of 1 is summed. For images that differ little (what
// a quality metric is asked about) that is small and nearly exact, while the rounding of
// va, which is that of squares near 4, is in the denominator alone: flat white with noise
// of 1e-4 is 3e-8 from the 64-bit value, and was 1e-5 from x^2 + y^2 and x y.
// The 42 x 42 window of both images (zero outside)
// goes to shared memory interleaved; a thread filters four columns of a row from
// sixteen pixels in registers, and then eight rows of a column from eighteen
// filtered rows, so an output costs four 16-byte shared-memory loads in place of
// 77 4-byte ones. The map's sum is a double. FP64 runs at a fiftieth of
// the FP32 rate here, so a thread first adds its eight values of a tile as an
// unevaluated float pair (48 bits, exact for values within 2^20 of one another) and
// then the pair to the double. The last CTA adds the partial sums in
// a fixed order, so the result does not depend on scheduling.
// 1919 x 1079 x 3: 56 us a call, bound by instruction issue; 94 for 4-byte loads, five
// quantities, a double addition per value and a kernel to add the sums.
#include "gs_internal.cuh"
#include "gs_launch.cuh"

namespace gs {

namespace {

constexpr int kSsT = 32;                 // output tile edge
constexpr int kSsR = 5;                  // window radius
constexpr int kSsW = kSsT + 2 * kSsR;    // 42: input window edge
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;

constexpr int kSsThreads = 128;
constexpr int kSsCtas = 5;                // resident CTAs per SM
constexpr int kSsUnits = 24;             // 16-byte units (a and d of two pixels) of a window row: 22, padded
constexpr int kSsCols = 4, kSsRows = 8;  // columns and rows a thread filters at a time

struct GaussW {
  float w[2 * kSsR + 1];  // normalised 1-D weights; the 2-D window is their outer product
};

// a + b as an unevaluated sum s + e (Knuth's exact two-term sum).
__device__ __forceinline__ void add_to(float &s, float &e, float b) {
  const float t = s + b, bb = t - s;
  e += (s - (t - bb)) + (b - bb);
  s = t;
}

// The sum of v over the CTA, on warp 0. One warp adds, because an FP64 addition holds the
// unit for 16 cycles whatever its lanes do: 8 in place of 20 when every warp sums its own
// (1919 x 1079 x 3: 57.2 -> 56.1 us).
__device__ __forceinline__ double block_sum(double v, double *s_red) {
  s_red[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = 0.0;
#pragma unroll
    for (int w = 0; w < kSsThreads / 32; ++w) v += s_red[w * 32 + threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return v;
}

// Persistent: a CTA takes tiles blockIdx.x, + gridDim.x, ... and loads the next
// tile's window into registers while it filters the current one (loaded in place,
// the window's latency was a third of the time).
__global__ void __launch_bounds__(kSsThreads, kSsCtas) ssim_kernel(const float *__restrict__ a, const float *__restrict__ b,
                                                             int W, int H, int tiles_x, int tiles_y, uint32_t n,
                                                             GaussW gw, double *part, uint32_t *__restrict__ ticket,
                                                             double count, float *__restrict__ out) {
  griddep_wait();
  constexpr int NW = kSsThreads / 32, RPW = (kSsW + NW - 1) / NW;  // window rows per warp
  // window rows: even units first, then odd ones, so the eight threads of a row
  // read consecutive units
  __shared__ float4 s_in[kSsW][kSsUnits];
  __shared__ float4 s_h[kSsW][kSsT];  // horizontally filtered: a, d, a^2, d^2
  __shared__ double s_red[kSsThreads];
  __shared__ bool s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // a lane's two window columns of a row: lane, and 32 + lane (of 42)
  float va[RPW][2], vb[RPW][2];
  auto load = [&](uint32_t t) {
    const int tx0 = (int)(t % (uint32_t)tiles_x) * kSsT - kSsR;
    const int ty0 = (int)(t / (uint32_t)tiles_x % (uint32_t)tiles_y) * kSsT - kSsR;
    const size_t plane = (size_t)W * H * (t / ((uint32_t)tiles_x * (uint32_t)tiles_y));
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
      const int r = warp + i * NW, y = ty0 + r;
      const bool row = r < kSsW && y >= 0 && y < H;
      const float *pa = a + plane + (size_t)(row ? y : 0) * W, *pb = b + plane + (size_t)(row ? y : 0) * W;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h, x = tx0 + c;
        const bool in = row && c < kSsW && x >= 0 && x < W;
        va[i][h] = in ? pa[x] : 0.f;
        vb[i][h] = in ? pb[x] : 0.f;
      }
    }
  };
  float2 w2[kSsR + 1];  // the weights are symmetric
#pragma unroll
  for (int k = 0; k <= kSsR; ++k) w2[k] = make_float2(gw.w[k], gw.w[k]);
  double total = 0.0;
  if (blockIdx.x < n) load(blockIdx.x);
  for (uint32_t t = blockIdx.x; t < n; t += gridDim.x) {
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = warp + i * NW;
    if (r >= kSsW) continue;  // warp-uniform
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = lane + 32 * h, u = c >> 1;
      if (c < 2 * 22)  // columns 42 and 43 pad the last unit
        reinterpret_cast<float2 *>(&s_in[r][(u & 1) * 12 + (u >> 1)])[c & 1] =
            make_float2(va[i][h] + vb[i][h], va[i][h] - vb[i][h]);
    }
  }
  __syncthreads();
  if (t + gridDim.x < n) load(t + gridDim.x);
  for (int i = tid; i < kSsW * (kSsT / kSsCols); i += kSsThreads) {
    const int r = i >> 3, g = i & 7;  // columns 4 g .. 4 g + 3 from window columns 4 g .. 4 g + 13
    float2 m[kSsCols], v[kSsCols];
#pragma unroll
    for (int o = 0; o < kSsCols; ++o) m[o] = v[o] = make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 7; ++u) {
      const float4 q = s_in[r][(u & 1) * 12 + g + (u >> 1)];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 ad = h ? make_float2(q.z, q.w) : make_float2(q.x, q.y), qq = __fmul2_rn(ad, ad);
#pragma unroll
        for (int o = 0; o < kSsCols; ++o) {
          const int k = 2 * u + h - o;  // tap
          if (k < 0 || k > 2 * kSsR) continue;
          const float2 w = w2[k <= kSsR ? k : 2 * kSsR - k];
          m[o] = __ffma2_rn(w, ad, m[o]);
          v[o] = __ffma2_rn(w, qq, v[o]);
        }
      }
    }
#pragma unroll
    for (int o = 0; o < kSsCols; ++o) s_h[r][kSsCols * g + o] = make_float4(m[o].x, m[o].y, v[o].x, v[o].y);
  }
  __syncthreads();
  const int tx0 = (int)(t % (uint32_t)tiles_x) * kSsT;
  const int ty0 = (int)(t / (uint32_t)tiles_x % (uint32_t)tiles_y) * kSsT;
  {
    static_assert(kSsThreads * kSsRows == kSsT * kSsT, "one block of rows per thread");
    const int c = tid & 31, r0 = (tid >> 5) * kSsRows;
    float2 m[kSsRows], v[kSsRows];
#pragma unroll
    for (int o = 0; o < kSsRows; ++o) m[o] = v[o] = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < kSsRows + 2 * kSsR; ++j) {
      const float4 q = s_h[r0 + j][c];
#pragma unroll
      for (int o = 0; o < kSsRows; ++o) {
        const int k = j - o;
        if (k < 0 || k > 2 * kSsR) continue;
        const float2 w = w2[k <= kSsR ? k : 2 * kSsR - k];
        m[o] = __ffma2_rn(w, make_float2(q.x, q.y), m[o]);
        v[o] = __ffma2_rn(w, make_float2(q.z, q.w), v[o]);
      }
    }
    float sum = 0.f, err = 0.f;
#pragma unroll
    for (int o = 0; o < kSsRows; ++o) {
      if (ty0 + r0 + o >= H || tx0 + c >= W) continue;
      const float2 mm = __fmul2_rn(m[o], m[o]), vv = __ffma2_rn(make_float2(-m[o].x, -m[o].y), m[o], v[o]);
      const float dm = mm.x + mm.y + 2.f * kC1, dv = vv.x + vv.y + 2.f * kC2;
      add_to(sum, err, fmaf(mm.y, dv, vv.y * (mm.x - mm.y + 2.f * kC1)) / (dm * dv));
    }
    total += (double)sum;
    if (isfinite(sum)) total += (double)err;  // of an infinite sum the error term is NaN
  }
  }
  total = block_sum(total, s_red);
  if (tid == 0) {
    part[blockIdx.x] = total;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  // the last CTA: every partial sum is written
  __threadfence();
  double t = 0.0;
#pragma unroll 8
  for (uint32_t i = tid; i < gridDim.x; i += kSsThreads) t += __ldcg(part + i);
  t = block_sum(t, s_red);
  if (tid == 0) {
    *out = (float)(1.0 - 2.0 * t / count);
    *ticket = 0u;  // for the next launch
  }
}

}  // namespace

size_t ssim_partials(int max_w, int max_h) {
  return (size_t)((max_w + kSsT - 1) / kSsT) * (size_t)((max_h + kSsT - 1) / kSsT) * 3;
}

cudaError_t launch_ssim(const float *a, const float *b, int W, int H, int C, double *part, uint32_t *ticket, float *out,
                        cudaStream_t s) {
  GaussW gw;
  double g[2 * kSsR + 1], sum = 0.0;
  for (int k = 0; k <= 2 * kSsR; ++k) {
    const double x = (double)(k - kSsR);
    g[k] = exp(-x * x / (2.0 * 1.5 * 1.5));
    sum += g[k];
  }
  double left = 1.0;
  for (int k = 0; k <= 2 * kSsR; ++k) left -= gw.w[k] = (float)(g[k] / sum);
  // The variances E a^2 - A^2 take mean squares as they are only if the rounded weights
  // sum to 1: the 1.4e-9 they lack made 1.6e-7 of an SSIM of 0.57 (smooth image, noise of
  // 0.05). The outermost weights, whose float spacing is 1e-10, take it.
  gw.w[0] = gw.w[2 * kSsR] = (float)(gw.w[0] + 0.5 * left);
  const int tx = (W + kSsT - 1) / kSsT, ty = (H + kSsT - 1) / kSsT;
  const uint32_t n = (uint32_t)tx * (uint32_t)ty * (uint32_t)C, cap = (uint32_t)sm_grid_cap(kSsCtas);
  GS_LAUNCHED(1);
  return launch_k(ssim_kernel, n < cap ? n : cap, kSsThreads, 0, s, a, b, W, H, tx, ty, n, gw, part, ticket,
                  (double)W * H * C, out);
}

}  // namespace gs
