// Allocation-free forward warp: the depth-tested warp of the dominant eye into
// the affiliated eye, with its per-pixel scratch in a static device array.
//
// Who needs it: code that must not allocate device memory while it renders,
// for instance a compositor or plugin running inside a host framework that
// owns the GPU memory pool and forbids outside allocations, or a frame loop
// with a hard per-frame deadline where a cudaMalloc may stall or fail. Such a
// caller still passes its own input and output buffers; the only scratch, one
// 64-bit key per affiliated pixel, lives in g_warp_keys below, which every
// device that loads this library keeps for the life of the process.
#include <mutex>

#include "gs_internal.cuh"
#include "gs_launch.cuh"
#include "gs_warp.cuh"

namespace gs {
namespace {

// GS_WARP_NOALLOC_MAX_PIXELS = 2^22 pixels (2048 x 2048, or any frame with no
// more pixels): 32 MiB of packed keys.
constexpr int64_t kNoAllocMaxPixels = GS_WARP_NOALLOC_MAX_PIXELS;
constexpr uint32_t kBackgroundBits = 0x7f800000u;

__device__ __align__(256) unsigned long long g_warp_keys[kNoAllocMaxPixels];

struct WarpCams {
  float Rrel[9], trel[3];
  float fx, fy, cx, cy;  // shared by both eyes
};

__global__ void noalloc_clear_kernel(unsigned long long *keys, int64_t n) {
  griddep_wait();
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    keys[p] = kNoSample;
}

// Source pixel -> destination pixel, as the renderer's warp: a surface sample
// (coverage 1 - T >= 0.5) at depth D / (1 - T), else a background sample at
// infinite depth; the packed (float depth bits << 32 | source index) key makes
// one 64-bit atomicMin the depth test.
__device__ __forceinline__ bool noalloc_transfer(const WarpCams &c, int x, int y, float trans, float depth, float &u,
                                                 float &v, uint32_t &zb) {
  const float cov = 1.f - trans;
  const bool surface = cov >= 0.5f;
  const float d = surface ? depth / cov : 0.f;
  const float rx = ((float)x - c.cx) / c.fx, ry = ((float)y - c.cy) / c.fy;
  const float *R = c.Rrel;
  float X, Y, Z;
  if (surface) {
    X = fmaf(R[0], rx * d, fmaf(R[1], ry * d, fmaf(R[2], d, c.trel[0])));
    Y = fmaf(R[3], rx * d, fmaf(R[4], ry * d, fmaf(R[5], d, c.trel[1])));
    Z = fmaf(R[6], rx * d, fmaf(R[7], ry * d, fmaf(R[8], d, c.trel[2])));
    if (!(Z > kZNear)) return false;
  } else {
    X = fmaf(R[0], rx, fmaf(R[1], ry, R[2]));
    Y = fmaf(R[3], rx, fmaf(R[4], ry, R[5]));
    Z = fmaf(R[6], rx, fmaf(R[7], ry, R[8]));
    if (!(Z > 0.f)) return false;
  }
  u = floorf(fmaf(c.fx, X / Z, c.cx) + 0.5f);
  v = floorf(fmaf(c.fy, Y / Z, c.cy) + 0.5f);
  zb = surface ? __float_as_uint(Z) : kBackgroundBits;
  return true;
}

__global__ void noalloc_scatter_kernel(const __grid_constant__ WarpCams c, const float *__restrict__ depth,
                                       const float *__restrict__ trans, unsigned long long *__restrict__ keys, int W,
                                       int H) {
  griddep_wait();
  const int64_t npix = (int64_t)W * H;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npix; p += (int64_t)gridDim.x * blockDim.x) {
    float u, v;
    uint32_t zb;
    if (!noalloc_transfer(c, (int)(p % W), (int)(p / W), trans[p], depth[p], u, v, zb)) continue;
    if (!(u >= 0.f && u <= (float)(W - 1) && v >= 0.f && v <= (float)(H - 1))) continue;
    const int64_t q = (int64_t)v * W + (int64_t)u;
    atomicMin(keys + q, ((unsigned long long)zb << 32) | (unsigned long long)(uint32_t)p);
  }
}

__device__ __forceinline__ void noalloc_resolve(unsigned long long k, int64_t p, int64_t npix,
                                                const float *__restrict__ rgb_dom, float *__restrict__ rgb_out,
                                                float *__restrict__ depth_out, uint8_t *__restrict__ hole_out) {
  const bool hole = k == kNoSample;
  const uint32_t s = (uint32_t)(k & 0xffffffffull);
  for (int ch = 0; ch < 3; ++ch) rgb_out[ch * npix + p] = hole ? 0.f : rgb_dom[ch * npix + s];
  if (depth_out) depth_out[p] = hole ? 0.f : __uint_as_float((uint32_t)(k >> 32));
  if (hole_out) hole_out[p] = hole ? 1 : 0;
}

// A rig that keeps rows: the whole warp in one kernel, one CTA per row, with no
// key array, no clearing and no global atomics (1600 x 1200: 25 us a call, 20 of them
// the kernel; 49 for the pose, clear, scatter and resolve kernels).
__global__ void __launch_bounds__(kRowThreads) noalloc_row_kernel(const __grid_constant__ WarpCams c,
                                                                  const float *__restrict__ rgb_dom,
                                                                  const float *__restrict__ depth,
                                                                  const float *__restrict__ trans, int W, int H,
                                                                  float *__restrict__ rgb_out,
                                                                  float *__restrict__ depth_out,
                                                                  uint8_t *__restrict__ hole_out) {
  griddep_wait();
  extern __shared__ unsigned long long s_zbuf[];
  const int y = blockIdx.x;
  const int64_t row = (int64_t)y * W, npix = (int64_t)W * H;
  warp_row(s_zbuf, trans + row, depth + row, W, [&](int x, float T, float D, int &ux, unsigned long long &key) {
    float u, v;
    uint32_t zb;
    if (!noalloc_transfer(c, x, y, T, D, u, v, zb)) return false;
    if (!(u >= 0.f && u <= (float)(W - 1) && v == (float)y)) return false;  // the row is kept (rows_kept)
    ux = (int)u;
    key = ((unsigned long long)zb << 32) | (unsigned long long)(uint32_t)(row + x);
    return true;
  });
  for (int x = threadIdx.x; x < W; x += kRowThreads)
    noalloc_resolve(s_zbuf[x], row + x, npix, rgb_dom, rgb_out, depth_out, hole_out);
}

// Destination pixel: the winner's colour and depth (+inf for a background
// sample), or a hole (colour 0, depth 0, hole = 1).
__global__ void noalloc_resolve_kernel(const unsigned long long *__restrict__ keys, const float *__restrict__ rgb_dom,
                                       int W, int H, float *__restrict__ rgb_out, float *__restrict__ depth_out,
                                       uint8_t *__restrict__ hole_out) {
  griddep_wait();
  const int64_t npix = (int64_t)W * H;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npix; p += (int64_t)gridDim.x * blockDim.x)
    noalloc_resolve(keys[p], p, npix, rgb_dom, rgb_out, depth_out, hole_out);
}

std::mutex g_mu;
unsigned long long *g_keys_ptr[64];

// Device address of the static scratch on the current device, looked up once
// per device (with that device current).
cudaError_t scratch_on_current_device(unsigned long long **keys) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_keys_ptr[dev]) {
    void *k = nullptr;
    if ((e = cudaGetSymbolAddress(&k, g_warp_keys)) != cudaSuccess) return e;
    g_keys_ptr[dev] = (unsigned long long *)k;
  }
  *keys = g_keys_ptr[dev];
  return cudaSuccess;
}

int grid_for_pixels(int64_t n) {
  const int64_t b = (n + 255) / 256;
  const int64_t cap = sm_grid_cap(16);
  return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace
}  // namespace gs

using namespace gs;

extern "C" gs_status gs_warp_noalloc(const float *rgb_dom, const float *depth_dom, const float *trans_dom,
                                     const gs_pose *pose_dom, const gs_pose *pose_aff, const gs_intrinsics *intr,
                                     float *rgb_warp, float *depth_warp, uint8_t *hole, void *stream) {
  if (!rgb_dom || !depth_dom || !trans_dom || !pose_dom || !pose_aff || !intr || !rgb_warp) return GS_ERR_BAD_ARG;
  if (intr->width <= 0 || intr->height <= 0 || !(intr->fx > 0) || !(intr->fy > 0)) return GS_ERR_BAD_ARG;
  const int64_t npix = (int64_t)intr->width * intr->height;
  if (npix > kNoAllocMaxPixels) return GS_ERR_CAPACITY;  // larger than the static scratch
  cudaStream_t s = (cudaStream_t)stream;
  const int W = intr->width, H = intr->height;
  double Rrel[9], trel[3];
  relative_pose(pose_dom->R, pose_dom->t, pose_aff->R, pose_aff->t, Rrel, trel);
  WarpCams wc;
  for (int k = 0; k < 9; ++k) wc.Rrel[k] = (float)Rrel[k];
  for (int k = 0; k < 3; ++k) wc.trel[k] = (float)trel[k];
  wc.fx = (float)intr->fx; wc.fy = (float)intr->fy; wc.cx = (float)intr->cx; wc.cy = (float)intr->cy;
  cudaError_t e;
  // a row's winners fit the default shared memory up to 6144 columns
  if (row_warp_smem(W) <= 48 * 1024 && rows_kept(Rrel, trel, intr->fx, intr->fy, intr->cx, intr->cy, W, H)) {
    e = launch_k(noalloc_row_kernel, H, kRowThreads, row_warp_smem(W), s, wc, rgb_dom, depth_dom, trans_dom, W, H,
                 rgb_warp, depth_warp, hole);
    GS_LAUNCHED(1);
    return e == cudaSuccess ? GS_OK : record_cuda_failure("gs_noalloc.cu", __LINE__, e);
  }
  unsigned long long *keys = nullptr;
  if ((e = scratch_on_current_device(&keys)) != cudaSuccess) return record_cuda_failure("gs_noalloc.cu", __LINE__, e);
  const int grid = grid_for_pixels(npix);
  e = launch_k(noalloc_clear_kernel, grid, 256, 0, s, keys, npix);
  if (e == cudaSuccess) e = launch_k(noalloc_scatter_kernel, grid, 256, 0, s, wc, depth_dom, trans_dom, keys, W, H);
  if (e == cudaSuccess)
    e = launch_k(noalloc_resolve_kernel, grid, 256, 0, s, (const unsigned long long *)keys, rgb_dom, W, H, rgb_warp,
                 depth_warp, hole);
  GS_LAUNCHED(3);
  return e == cudaSuccess ? GS_OK : record_cuda_failure("gs_noalloc.cu", __LINE__, e);
}
