// Persistent per-tile front-to-back alpha blending with the joint depth proxy.
//
// Paper: Sec. 3.1 Stage 1 - every contributing surfel gets the weight
// w_i = alpha_i T_i, and the same weight accumulates the colour C = sum c_i w_i
// and the depth proxy D = sum d_i w_i in one pass (no separate depth pass).
// Sec. 3.3 (Eq. 2 and the ray-splat intersection) gives alpha.
//
// One launch serves up to kRasterFrames (frame, eye) images - one eye of one
// frame, or one eye of every frame of a batch of scenes with different surfel
// counts and resolutions. The grid fills the SMs once; every CTA takes work
// items, (frame, tile) pairs numbered frame by frame, from a device counter
// until none is left, so the heavy tiles of one frame overlap the light tiles of
// the others and no CTA is launched per tile. A frame either offers every tile
// of its grid or a device list of tiles (the ROI tiles of a masked binning, or
// the masked 16-pixel tiles rendered from the lists of a coarser binning: each
// reads its parent tile's list, every surfel reaching the parent in depth
// order, and the surfels that miss its pixels contribute nothing).
//
// A group of TS^2 / PIX threads blends one TS x TS tile (8 or 16 pixels; a 32-pixel
// tile is four 16-pixel quadrants reading its list). A warp covers a block of
// 8 x (4 PIX) pixels (lane l: column l % 8, rows l / 8 + 4 q for q < PIX). The
// kernel is bound by instruction issue (1600x1200, 500k surfels: 70 (pixel,
// surfel) pairs evaluated per pixel, 57 of them contributing, 178M warp
// instructions, 71 % of the issue slots busy), so three steps cut the
// instructions per contribution:
//   1. the group stages its list in batches and copies only the records whose
//      screen bounds meet the tile; cp.async double-buffers the next batch;
//   2. a warp tests a batch's records one per lane against its own block, with
//      the support itself (support_meets) and not only its bounds: 98 evaluated
//      pairs per pixel with the bounds alone, 70 with the support;
//   3. the survivors are evaluated two records at a time on the packed FP32x2
//      pipe (see the record queue below).
// Measured (dominant eye, 500k surfels at 1600x1200 / 3M at 2448x2448, 32-pixel
// lists): 283 / 1265 us for a 512-thread tile that tested the bounds record by
// record, 214 / 776 us now.
// The homogeneous plane point p of a pixel is affine in the pixel offset (dx, dy)
// from the projected centre, and a pixel's arithmetic depends on its position
// only: not on the tile edge, the block shape or the batch, and a record that a
// test leaves out contributes nothing to the pixels it was tested for. So every
// configuration gives the same image bit for bit. A tile ends as soon as all its
// pixels have terminated.
//
// Ellipsoids (the 3DGS backbone) use the same loop: their record holds a
// Cholesky factor L of the screen conic Sigma2D^-1 = L^T L in place of the
// plane coefficients and a constant third coordinate, so the plane point is
// (L d, 1) and u^2 + v^2 = d^T Sigma2D^-1 d, the EWA exponent; the frame's
// low-pass factor is kNoLowpass (the EWA kernel already carries its 0.3 px^2
// filter) and the depth terms are zero, so every contribution has the centre
// depth.
#include <type_traits>

#include "gs_internal.cuh"
#include "gs_launch.cuh"
#include "gs_scan.cuh"

namespace gs {

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// 1 / (2 ln 2): log2(o Ghat) = (r_c^2 - rho) / (2 ln 2) + log2(1/255)
constexpr float kHalfLog2e = 0.72134752044448170f;
// the row of a pixel that takes no more contributions
#define kNaN __int_as_float(0x7fffffff)

// ---- the warp's record queue ----
// Records that can reach a warp's block are copied, in list order, to a queue of
// the warp's own in shared memory, as pairs: the 16 floats of two consecutive
// records interleaved (f0 of both, f1 of both, ...), then two flags. One
// LDS.128 thus gives the packed FP32x2 pipe two operands, each holding a field
// of both records, so a pixel is evaluated for two records per instruction with
// no operand ever duplicated; the pixel's own column and row are constants of
// the tile. The pair stride of 36 floats spreads the copies over the banks.
constexpr int kPairStride = 36;
constexpr int kQueue = 40;  // records: emptied whenever fewer than 32 slots are free

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// Can the record's support reach a pixel centre of the block |x - xc| <= hx,
// |y - yc| <= hy? `plane` / `disc` are false only when no pixel of the block has
// rho3 <= r_c^2 / rho2 <= r_c^2, in the blend's own float32 arithmetic. The plane point p is affine in the pixel,
// so over the block |p.x| >= U, |p.y| >= V and |p.z| <= Z with the values at the
// centre and the half extents of the affine form; U^2 + V^2 > r_c^2 Z^2 then puts
// every (u, v) outside the support. The low-pass disc needs the block's nearest
// point. Rounding is covered by half extents grown by 0.01 pixel and 1e-6 of the
// centre's distance (the blend's p carries some 2^-22 of its terms) and a
// support radius squared grown by 1e-3. A NaN keeps the record.
__device__ __forceinline__ void support_meets(const float4 a, const float4 b, const float4 c, float xc, float yc,
                                              float hx, float hy, float lowpass, bool &plane, bool &disc) {
  const float dx = xc - a.x, dy = yc - a.y;
  const float gx = fmaf(fabsf(dx), 1e-6f, hx + 0.01f), gy = fmaf(fabsf(dy), 1e-6f, hy + 0.01f);
  const float px = fmaf(dx, b.x, dy * b.z), py = fmaf(dx, b.y, dy * b.w);
  const float pz = fmaf(dx, c.y, fmaf(dy, c.z, c.x));
  const float U = fmaxf(fabsf(px) - fmaf(gx, fabsf(b.x), gy * fabsf(b.z)), 0.f);
  const float V = fmaxf(fabsf(py) - fmaf(gx, fabsf(b.y), gy * fabsf(b.w)), 0.f);
  const float Z = fmaf(gx, fabsf(c.y), fmaf(gy, fabsf(c.z), fmaf(fabsf(c.x), 1e-6f, fabsf(pz))));
  const float k = fmaf(a.z, 1.001f, 1e-6f);
  const float ex = fmaxf(fabsf(dx) - gx, 0.f), ey = fmaxf(fabsf(dy) - gy, 0.f);
  plane = !(fmaf(U, U, V * V) > k * Z * Z);
  disc = !(fmaf(ex, ex, ey * ey) * lowpass > k);
}

// Barriers of a group of NT threads: the CTA's own when it is one group, else
// named barrier 1 + group.
template <int NT, int G>
__device__ __forceinline__ void group_sync(int group) {
  if constexpr (G == 1) __syncthreads();
  else asm volatile("barrier.cta.sync %0, %1;" ::"r"(1 + group), "n"(NT) : "memory");
}
template <int NT, int G>
__device__ __forceinline__ bool group_any(int group, bool v) {
  if constexpr (G == 1) {
    return __syncthreads_or(v) != 0;
  } else {
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 q, %1, 0;\n\tbarrier.cta.red.or.pred p, %2, %3, q;\n\t"
        "selp.s32 %0, 1, 0, p;\n\t}\n"
        : "=r"(r)
        : "r"((int)v), "r"(1 + group), "n"(NT)
        : "memory");
    return r != 0;
  }
}

// Shared memory of one group.
template <int NW, int BATCH>
struct GroupSmem {
  float4 s0[2][BATCH], s1[2][BATCH], s2[2][BATCH], s3[2][BATCH], s4[2][BATCH];  // staged records and bounds
  float q[NW][kQueue / 2 * kPairStride];  // the warps' record queues
  int n[2][BATCH / 32];                   // records kept of every segment
  uint32_t item[2];                       // double-buffered: one barrier per item
};

// The CTA's group `group` of G blends work items until none is left.
template <int TS, int PIX, int BATCH, bool COUNT, int G>
__device__ __forceinline__ void raster_items(const RasterTable &tab, uint32_t *queue, const uint32_t *s_first,
                                             int group, GroupSmem<TS * TS / PIX / 32, BATCH> &sm) {
  constexpr int NT = TS * TS / PIX;  // threads of the group
  constexpr int NW = NT / 32;
  constexpr int RS = 4;              // rows between a thread's pixels
  constexpr int WBX = TS / 8;        // warp blocks per tile row
  constexpr int SEG = BATCH / 32;    // list segments of 32 entries per batch
  static_assert(NT % 32 == 0 && TS % 8 == 0 && TS % (4 * PIX) == 0, "block shape");
  const int tid = threadIdx.x - group * NT;
  const int warp = tid >> 5, lane = tid & 31;
  const int bx0 = (warp % WBX) * 8, by0 = (warp / WBX) * (4 * PIX);  // the warp's block in the tile
  const int lx = bx0 + (lane & 7), ly = by0 + (lane >> 3);

  if (tid == 0) sm.item[0] = atomicAdd(queue, 1u);
  for (int it = 0;; it ^= 1) {
    // orders the item before its reads, and every read of the previous tile's
    // shared records before this tile's staging
    group_sync<NT, G>(group);
    const uint32_t g = sm.item[it];
    if (g >= s_first[tab.n]) break;  // group-uniform
    int f = 0;
    while (f + 1 < tab.n && s_first[f + 1] <= g) ++f;
    const RasterFrame &fr = tab.f[f];
    uint32_t k = g - s_first[f];
    const int quad = fr.split ? (int)(k & 3u) : 0;
    if (fr.split) k >>= 2;
    const int tile = fr.items ? (int)fr.items[k] : (int)k;

    const int W = fr.W, H = fr.H;
    int tcx = tile % fr.tiles_x, tcy = tile / fr.tiles_x;
    // a tile of a finer grid than the binning's reads its parent tile's list
    // (every surfel reaching the parent, a superset of the tile's own)
    const int rt = fr.rshift ? (tcy >> fr.rshift) * fr.rtiles_x + (tcx >> fr.rshift) : tile;
    if (fr.split) {  // the item is a quadrant of the listed tile
      tcx = 2 * tcx + (quad & 1);
      tcy = 2 * tcy + (quad >> 1);
    }
    const int px = tcx * TS + lx;
    const int py = tcy * TS + ly;  // first of rows py, py + RS, ...
    const int rtx = (W + kTile - 1) / kTile;

    const float fx = (float)px;
    const float lowpass = fr.lowpass;
    // the tile and the warp's pixel block (pixel centres), for the record culling
    const float tx0 = (float)(tcx * TS), ty0 = (float)(tcy * TS);
    const float tx1 = tx0 + (float)(TS - 1), ty1 = ty0 + (float)(TS - 1);
    const float wx0 = tx0 + (float)bx0, wy0 = ty0 + (float)by0;
    const float wx1 = wx0 + 7.f, wy1 = wy0 + (float)(4 * PIX - 1);
    constexpr float whx = 3.5f, why = 0.5f * (float)(4 * PIX - 1);
    const float wxc = wx0 + whx, wyc = wy0 + why;
    // the thread's pixel rows; a pixel that is not blending (outside the image
    // or the ROI, or finished) has a NaN row, so every test on it fails
    float fy[PIX];
    float T[PIX], C0[PIX], C1[PIX], C2[PIX], D[PIX];
    unsigned wmask = 0;  // bit k: this thread writes pixel k
#pragma unroll
    for (int q = 0; q < PIX; ++q) {
      T[q] = 1.f; C0[q] = C1[q] = C2[q] = D[q] = 0.f;
      const int y = py + RS * q;
      bool on = px < W && y < H;
      if (on && fr.roi) on = fr.roi[(y / kTile) * rtx + px / kTile] != 0;
      if (on && fr.skip) on = fr.skip[(y / kTile) * rtx + px / kTile] == 0;
      fy[q] = on ? (float)y : kNaN;
      if (on) wmask |= 1u << q;
    }
    unsigned npairs = 0, ncontrib = 0;
    // nothing to blend (a quadrant outside the image or the ROI): no list
    const uint2 rg = group_any<NT, G>(group, wmask != 0u) ? fr.ranges[rt] : make_uint2(0u, 0u);

    // Staging. The list's segments of 32 entries go to the warps in turn; a lane
    // reads its entry's surfel id and screen bounds, and only the records whose
    // bounds meet the tile are copied, packed at the segment's start in list
    // order. A warp's next segment's bounds and the one after's ids are fetched
    // ahead, so neither gather's latency shows.
    auto entry_id = [&](uint32_t seg) -> uint32_t {
      const uint32_t i = rg.x + seg * 32u + (uint32_t)lane;
      return i < rg.y ? fr.ids[i] : 0xffffffffu;
    };
    auto entry_box = [&](uint32_t id) -> float4 {  // ids past the records are never expected: empty bounds
      return id < fr.n_rec ? __ldg(fr.box + id) : make_float4(1.f, 0.f, 1.f, 0.f);
    };
    uint32_t mine = (uint32_t)warp, id1 = 0xffffffffu, id2 = 0xffffffffu;  // the warp's next segment
    float4 bb1 = make_float4(1.f, 0.f, 1.f, 0.f);
    auto stage = [&](int buf, uint32_t batch) {
      while (mine < (batch + 1u) * SEG) {  // warp-uniform
        const bool keep = id1 < fr.n_rec && !(bb1.y < tx0 || bb1.x > tx1 || bb1.w < ty0 || bb1.z > ty1);
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        const int seg = (int)(mine - batch * SEG);
        if (keep) {
          const int slot = seg * 32 + __popc(m & ((1u << lane) - 1u));
          const float4 *r = fr.rec + 4 * (size_t)id1;
          cp_async16(&sm.s0[buf][slot], r + 0);
          cp_async16(&sm.s1[buf][slot], r + 1);
          cp_async16(&sm.s2[buf][slot], r + 2);
          cp_async16(&sm.s3[buf][slot], r + 3);
          sm.s4[buf][slot] = bb1;
        }
        if (lane == 0) sm.n[buf][seg] = __popc(m);
        mine += NW;
        id1 = id2;
        bb1 = entry_box(id1);
        id2 = entry_id(mine + NW);
      }
      cp_async_commit();
    };

    // Two queued records over the thread's pixels, front to back. Without the
    // low-pass term (DISC false: both records' discs miss the warp's block, so
    // rho2 > r_c^2 at all its pixels) a pixel contributes exactly when rho3 <=
    // r_c^2, with rho = rho3 and the plane's depth. Every component of a packed
    // operation is rounded as the scalar operation would be.
    const float2 fx2 = both(fx), minus1 = both(-1.f);
    auto blend_pair = [&](auto disc_tag, const float *qp) {
      constexpr bool DISC = decltype(disc_tag)::value;
      const float4 *q4 = reinterpret_cast<const float4 *>(qp);
      auto lo = [](const float4 &v) { return make_float2(v.x, v.y); };
      auto hi = [](const float4 &v) { return make_float2(v.z, v.w); };
      const float4 v0 = q4[0], v1 = q4[1], v2 = q4[2], v3 = q4[3], v4 = q4[4], v5 = q4[5], v6 = q4[6], v7 = q4[7];
      // homogeneous plane point p = (dx b.x + dy b.z, dx b.y + dy b.w,
      // c.x + dx c.y + dy c.z): the column's dx terms, then dy per pixel
      const float2 dx = ffma2(lo(v0), minus1, fx2);
      const float2 px0 = __fmul2_rn(dx, lo(v2)), py0 = __fmul2_rn(dx, hi(v2)), pz0 = ffma2(dx, hi(v4), lo(v4));
      const float2 az = lo(v1);
#pragma unroll
      for (int q = 0; q < PIX; ++q) {
        const float2 dy = ffma2(hi(v0), minus1, both(fy[q]));
        const float2 qx = ffma2(dy, lo(v3), px0), qy = ffma2(dy, hi(v3), py0), qz = ffma2(dy, lo(v5), pz0);
        const float2 iq = make_float2(rcp_approx(qz.x), rcp_approx(qz.y));
        const float2 u = __fmul2_rn(qx, iq), v = __fmul2_rn(qy, iq);
        const float2 r3 = ffma2(u, u, __fmul2_rn(v, v));
        float2 rho = r3, z = ffma2(hi(v5), u, ffma2(lo(v6), v, hi(v1)));
        if (DISC) {
          const float2 r2 = __fmul2_rn(ffma2(dy, dy, __fmul2_rn(dx, dx)), both(lowpass));
          rho = make_float2(fminf(r3.x, r2.x), fminf(r3.y, r2.y));
          z = make_float2(r3.x <= r2.x ? z.x : v1.z, r3.y <= r2.y ? z.y : v1.w);
        }
        // alpha >= 1/255: rho <= r_c^2 (false for a NaN row)
        const float2 ee = ffma2(ffma2(rho, minus1, az), both(kHalfLog2e), both(kLog2AlphaMin));
        const float al0 = fminf(kAlphaMax, ex2_approx(ee.x)), al1 = fminf(kAlphaMax, ex2_approx(ee.y));
        const bool hit0 = rho.x <= az.x;
        const float Ta = fmaf(-T[q], al0, T[q]), w0 = al0 * T[q];
        const bool on0 = hit0 && Ta >= kTMin, end0 = hit0 && !(Ta >= kTMin);
        if (on0) {
          if (COUNT) ++ncontrib;
          C0[q] = fmaf(w0, hi(v6).x, C0[q]);
          C1[q] = fmaf(w0, lo(v7).x, C1[q]);
          C2[q] = fmaf(w0, hi(v7).x, C2[q]);
          D[q] = fmaf(w0, z.x, D[q]);
          T[q] = Ta;
        }
        const bool hit1 = rho.y <= az.y && !end0;
        const float Tb = fmaf(-T[q], al1, T[q]), w1 = al1 * T[q];
        const bool on1 = hit1 && Tb >= kTMin, end1 = hit1 && !(Tb >= kTMin);
        if (on1) {
          if (COUNT) ++ncontrib;
          C0[q] = fmaf(w1, hi(v6).y, C0[q]);
          C1[q] = fmaf(w1, lo(v7).y, C1[q]);
          C2[q] = fmaf(w1, hi(v7).y, C2[q]);
          D[q] = fmaf(w1, z.y, D[q]);
          T[q] = Tb;
        }
        if (end0 || end1) fy[q] = kNaN;  // the pixel has terminated
      }
    };
    float *wq = sm.q[warp];
    int nq = 0;  // records queued (warp-uniform)
    // empties the queue; a last odd record waits for its partner (moved to the
    // front) unless `all`, when it is paired with a record that reaches nothing
    auto drain = [&](bool all) {
      if (all && (nq & 1)) {
        if (lane < 16) wq[(nq >> 1) * kPairStride + 2 * lane + 1] = lane == 2 ? -1.f : 0.f;  // r_c^2 < 0
        if (lane == 16) wq[(nq >> 1) * kPairStride + 33] = 0.f;
        ++nq;
      }
      __syncwarp();
      const int np = nq >> 1;
      const float *qp = wq;
      for (int i = 0; i < np; ++i, qp += kPairStride) {
        if constexpr (COUNT) {
#pragma unroll
          for (int q = 0; q < PIX; ++q) npairs += fy[q] == fy[q] ? (qp[5] < 0.f ? 1u : 2u) : 0u;
        }
        const float2 fl = *reinterpret_cast<const float2 *>(qp + 32);
        if (fl.x + fl.y != 0.f) blend_pair(std::true_type{}, qp);
        else blend_pair(std::false_type{}, qp);
      }
      __syncwarp();
      if (nq & 1) {
        if (lane < 17) wq[2 * lane] = qp[2 * lane];
        __syncwarp();  // the odd record has left its slot before a lane fills it again
      }
      nq &= 1;
    };
    // a pixel of the thread still blends
    auto alive = [&]() -> bool {
      bool v = false;
#pragma unroll
      for (int q = 0; q < PIX; ++q) v |= fy[q] == fy[q];
      return v;
    };

    int buf = 0;
    if (rg.x < rg.y) {
      id1 = entry_id(mine);
      id2 = entry_id(mine + NW);
      bb1 = entry_box(id1);
      stage(0, 0u);
    }
    uint32_t batch = 0;
    for (uint32_t b0 = rg.x; b0 < rg.y; b0 += BATCH, buf ^= 1, ++batch) {
      cp_async_wait_all();
      // barrier: the batch in `buf` is visible to all, and every thread has
      // finished reading the other buffer, which the prefetch below overwrites
      if (!group_any<NT, G>(group, alive())) break;
      if (b0 + BATCH < rg.y) stage(buf ^ 1, batch + 1u);
#pragma unroll 1
      for (int seg = 0; seg < SEG; ++seg) {
        const int n = sm.n[buf][seg], g0 = seg * 32;
        if (n == 0) continue;
        // a segment's records at once, one per lane: those whose support meets
        // the warp's block join its queue, in list order
        if (!__any_sync(0xffffffffu, alive())) break;  // every pixel of the block has terminated
        const int j = g0 + lane;
        bool plane = false, disc = false;
        if (lane < n) {
          const float4 bb = sm.s4[buf][j];
          if (!(bb.y < wx0 || bb.x > wx1 || bb.w < wy0 || bb.z > wy1))
            support_meets(sm.s0[buf][j], sm.s1[buf][j], sm.s2[buf][j], wxc, wyc, whx, why, lowpass, plane, disc);
        }
        const unsigned m = __ballot_sync(0xffffffffu, plane || disc);
        if (plane || disc) {
          const int pos = nq + __popc(m & ((1u << lane) - 1u));
          float *e = wq + (pos >> 1) * kPairStride + (pos & 1);
          const float4 a = sm.s0[buf][j], b = sm.s1[buf][j], c = sm.s2[buf][j], d = sm.s3[buf][j];
          e[0] = a.x; e[2] = a.y; e[4] = a.z; e[6] = a.w;
          e[8] = b.x; e[10] = b.y; e[12] = b.z; e[14] = b.w;
          e[16] = c.x; e[18] = c.y; e[20] = c.z; e[22] = c.w;
          e[24] = d.x; e[26] = d.y; e[28] = d.z; e[30] = d.w;
          e[32] = disc ? 1.f : 0.f;
        }
        nq += __popc(m);
        if (nq > kQueue - 32) drain(false);
      }
    }
    drain(true);
    cp_async_wait_all();
    // the next item: its round trip overlaps the output stores below
    uint32_t next = 0;
    if (tid == 0) next = atomicAdd(queue, 1u);

    const size_t hw = (size_t)W * H;
    float lo = 3.0e38f, hi = 0.f;
#pragma unroll
    for (int q = 0; q < PIX; ++q) {
      if (!(wmask & (1u << q))) continue;
      const size_t p = (size_t)(py + RS * q) * W + px;
      fr.rgb[p] = fmaf(T[q], fr.bg[0], C0[q]);
      fr.rgb[hw + p] = fmaf(T[q], fr.bg[1], C1[q]);
      fr.rgb[2 * hw + p] = fmaf(T[q], fr.bg[2], C2[q]);
      if (fr.depth) fr.depth[p] = D[q];
      if (fr.trans) fr.trans[p] = T[q];
      if (fr.winit) fr.winit[p] = kNoSample;
      if (fr.cls) fr.cls[p] |= (uint8_t)kClsRender;
      if (1.f - T[q] >= 0.5f) {
        // range of the alpha-normalised depth D / (1 - T) over pixels with coverage >= 0.5
        const float dh = D[q] / (1.f - T[q]);
        lo = fminf(lo, dh);
        hi = fmaxf(hi, dh);
      }
    }
    if (fr.stats) {  // group-uniform
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      }
      if (lane == 0 && hi > 0.f) {
        atomicMin(&fr.ctr->dmin_bits, __float_as_uint(fmaxf(lo, 0.f)));
        atomicMax(&fr.ctr->dmax_bits, __float_as_uint(hi));
      }
    }
    if (tid == 0) sm.item[it ^ 1] = next;  // read after the next barrier
    if (COUNT) {
      unsigned long long v = npairs, cc = ncontrib;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v += __shfl_xor_sync(0xffffffffu, v, o);
        cc += __shfl_xor_sync(0xffffffffu, cc, o);
      }
      if (lane == 0) {
        atomicAdd(&fr.ctr->pairs[fr.eye], v);
        atomicAdd(&fr.ctr->contrib[fr.eye], cc);
      }
    }
  }
}

// First work item of every frame (CTA-wide; s_first[tab.n] is their number).
__device__ __forceinline__ void frame_items(const RasterTable &tab, uint32_t *s_first) {
  if (threadIdx.x < 32) {
    const int f = threadIdx.x;
    uint32_t c = 0;
    if (f < tab.n) {
      const RasterFrame &fr = tab.f[f];
      c = (uint32_t)fr.ntiles;
      if (fr.items) c = min(c, *fr.n_items);
      if (fr.split) c *= 4u;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, c, o);
      if (f >= o) c += y;
    }
    s_first[f + 1] = c;
    if (f == 0) s_first[0] = 0u;
  }
  __syncthreads();
}

// The last CTA out clears the counter and the ticket for the next launch.
__device__ __forceinline__ void leave(uint32_t *queue) {
  __syncthreads();  // every group of the CTA has taken its last item
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(queue + 1, 1u) == gridDim.x - 1) {
      queue[0] = 0u;
      queue[1] = 0u;
    }
  }
}

// 16-pixel tiles (and quadrants of 32-pixel ones). Two groups of 128 threads, two
// pixels per thread, each with its own items (a pixel per thread measured 263
// against 218 us on the 7,600 quadrants of a 1600x1200 frame, four pixels 232); but
// with fewer items than groups in flight the longest item sets the time, and all
// 256 threads share one item at a pixel per thread (192 tiles of a 256x192 frame:
// 48 us against 74; some 350 ROI tiles of a 1080p frame: 29 against 39; 1,230 ROI
// tiles of the 1600x1200 frame: even). 64 registers keep four CTAs resident.
constexpr int kCta16 = 256;
template <int BATCH>
union Smem16 {
  GroupSmem<4, BATCH> two[2];
  GroupSmem<8, BATCH> one;
};
template <int BATCH, bool COUNT>
__global__ void __launch_bounds__(kCta16, 4)
    raster16_kernel(const __grid_constant__ RasterTable tab, uint32_t *__restrict__ queue) {
  griddep_wait();
  __shared__ __align__(16) unsigned char s_raw[sizeof(Smem16<BATCH>)];
  __shared__ uint32_t s_first[kRasterFrames + 1];
  Smem16<BATCH> &sm = *reinterpret_cast<Smem16<BATCH> *>(s_raw);
  frame_items(tab, s_first);
  if (s_first[tab.n] <= 2u * gridDim.x) {
    raster_items<16, 1, BATCH, COUNT, 1>(tab, queue, s_first, 0, sm.one);
  } else {
    const int group = threadIdx.x >> 7;
    raster_items<16, 2, BATCH, COUNT, 2>(tab, queue, s_first, group, sm.two[group]);
  }
  leave(queue);
}

// 8-pixel tiles: one CTA per item.
template <int PIX, int BATCH, bool COUNT>
__global__ void __launch_bounds__(64 / PIX, PIX == 1 ? 16 : 20)
    raster8_kernel(const __grid_constant__ RasterTable tab, uint32_t *__restrict__ queue) {
  griddep_wait();
  __shared__ __align__(16) unsigned char s_raw[sizeof(GroupSmem<2 / PIX, BATCH>)];
  __shared__ uint32_t s_first[kRasterFrames + 1];
  frame_items(tab, s_first);
  raster_items<8, PIX, BATCH, COUNT, 1>(tab, queue, s_first, 0,
                                        *reinterpret_cast<GroupSmem<2 / PIX, BATCH> *>(s_raw));
  leave(queue);
}

// ---------------------------------------------------------------- work order
// Longest tile lists first. The persistent rasterizer takes its work items in
// list order, so a frame whose heaviest tiles come last ends on a few CTAs
// still walking long lists while the other SMs idle. One CTA counting-sorts the
// frame's items by a log-scale bucket of their surfel-list length (eight
// buckets per octave, longest first; the order inside a bucket is arbitrary).
// The order changes no pixel: every item renders its own pixels.
constexpr int kLptThreads = 1024;

__device__ __forceinline__ uint32_t lpt_bucket(uint32_t len) {
  const uint32_t v = len + 1u;
  const uint32_t lg = 31u - (uint32_t)__clz(v);
  const uint32_t frac = lg >= 3u ? (v >> (lg - 3u)) & 7u : (v << (3u - lg)) & 7u;
  return 255u - min(255u, lg * 8u + frac);
}

__global__ void __launch_bounds__(kLptThreads) lpt_order_kernel(const uint32_t *__restrict__ items,
                                                                const uint32_t *n_items, uint32_t n_max,
                                                                const uint2 *__restrict__ ranges, int tiles_x,
                                                                int rshift, int rtiles_x, uint32_t *__restrict__ out) {
  griddep_wait();
  __shared__ uint32_t s_hist[256];
  __shared__ uint32_t s_scan[32];
  const uint32_t n = items ? min(*n_items, n_max) : n_max;
  auto bucket = [&](uint32_t k, uint32_t &tile) {
    tile = items ? items[k] : k;
    const uint32_t rt = rshift ? (tile / (uint32_t)tiles_x >> rshift) * (uint32_t)rtiles_x +
                                     (tile % (uint32_t)tiles_x >> rshift)
                               : tile;
    const uint2 rg = ranges[rt];
    return lpt_bucket(rg.y - rg.x);
  };
  if (threadIdx.x < 256) s_hist[threadIdx.x] = 0u;
  __syncthreads();
  for (uint32_t k = threadIdx.x; k < n; k += kLptThreads) {
    uint32_t t;
    atomicAdd(&s_hist[bucket(k, t)], 1u);
  }
  __syncthreads();
  uint32_t base;
  block_exclusive_scan<kLptThreads>(threadIdx.x < 256 ? s_hist[threadIdx.x] : 0u, &base, s_scan);
  __syncthreads();
  if (threadIdx.x < 256) s_hist[threadIdx.x] = base;
  __syncthreads();
  for (uint32_t k = threadIdx.x; k < n; k += kLptThreads) {
    uint32_t t;
    const uint32_t b = bucket(k, t);
    out[1u + atomicAdd(&s_hist[b], 1u)] = t;
  }
  if (threadIdx.x == 0) out[0] = n;
}

// ---------------------------------------------------------------- host side

namespace {

struct Variant {
  const void *fn;
  int threads;
  int occupancy;  // resident CTAs per SM, 0 until queried
};

// Kernels: 8-pixel tiles with one or two pixels per thread, and the 16-pixel one,
// which also takes 32-pixel tiles as four quadrants reading the tile's list.
constexpr int kShapes = 3;   // (8, 1) (8, 2) 16
constexpr int kBatches = 2;  // 32 64

template <bool C>
void fill_variants(Variant (&v)[kShapes][kBatches]) {
  v[0][0] = Variant{(const void *)raster8_kernel<1, 32, C>, 64, 0};
  v[0][1] = Variant{(const void *)raster8_kernel<1, 64, C>, 64, 0};
  v[1][0] = Variant{(const void *)raster8_kernel<2, 32, C>, 32, 0};
  v[1][1] = Variant{(const void *)raster8_kernel<2, 64, C>, 32, 0};
  v[2][0] = Variant{(const void *)raster16_kernel<32, C>, kCta16, 0};
  v[2][1] = Variant{(const void *)raster16_kernel<64, C>, kCta16, 0};
}

struct VariantTable {
  Variant v[2][kShapes][kBatches];
  VariantTable() {
    fill_variants<false>(v[0]);
    fill_variants<true>(v[1]);
  }
};

VariantTable g_variants;

int shape_index(const RasterConfig &c) {
  switch (c.tile) {
    case 8: return c.pix == 1 ? 0 : c.pix == 2 ? 1 : -1;
    case 16: return c.pix == 2 || c.pix == 4 ? 2 : -1;
    case 32: return c.pix == 2 || c.pix == 4 || c.pix == 8 ? 2 : -1;
  }
  return -1;
}

// Longer stages than 64 entries run as stages of 64: they copy more records past
// the one that ends a tile, and fewer CTAs fit an SM.
int batch_index(int b) { return b == 32 ? 0 : b == 64 || b == 128 || b == 256 ? 1 : -1; }

}  // namespace

int sm_count() {
  static int cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
  if (dev < 64 && cached[dev] > 0) return cached[dev];
  int n = 0;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (dev < 64) cached[dev] = n;
  return n;
}

bool raster_config_ok(const RasterConfig &c) { return shape_index(c) >= 0 && batch_index(c.batch) >= 0; }

int raster_tshift(const RasterConfig &c) { return c.tile == 8 ? 3 : c.tile == 32 ? 5 : 4; }

bool raster_same(const RasterConfig &a, const RasterConfig &b) {
  return a.tile == b.tile && shape_index(a) == shape_index(b) && batch_index(a.batch) == batch_index(b.batch);
}

cudaError_t launch_raster(const RasterTable &t, const RasterConfig &c, bool count_pairs, uint32_t *queue,
                          cudaStream_t s) {
  if (!raster_config_ok(c) || t.n < 0 || t.n > kRasterFrames) return cudaErrorInvalidValue;
  if (t.n == 0) return cudaSuccess;
  Variant &v = g_variants.v[count_pairs ? 1 : 0][shape_index(c)][batch_index(c.batch)];
  if (v.occupancy <= 0) {
    int occ = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, v.fn, v.threads, 0);
    if (e != cudaSuccess) return e;
    v.occupancy = occ > 0 ? occ : 1;
  }
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorNoDevice;
  RasterTable arg = t;
  if (c.tile == 32)
    for (int f = 0; f < arg.n; ++f) arg.f[f].split = arg.f[f].tshift == 5;
  void *args[2] = {(void *)&arg, (void *)&queue};
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((unsigned)(sms * v.occupancy));
  cfg.blockDim = dim3((unsigned)v.threads);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_pdl ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelExC(&cfg, v.fn, args);
  GS_LAUNCHED(1);
  return e;
}

cudaError_t launch_lpt_order(RasterFrame &f, uint32_t *buf, cudaStream_t s) {
  const cudaError_t e = launch_k(lpt_order_kernel, 1, kLptThreads, 0, s, f.items, f.n_items, (uint32_t)f.ntiles,
                                 f.ranges, f.tiles_x, f.rshift, f.rtiles_x, buf);
  GS_LAUNCHED(1);
  f.items = buf + 1;
  f.n_items = buf;
  return e;
}

RasterFrame raster_frame(const Workspace &ws, int eye, int W, int H, int tshift, const uint8_t *mask, float3 bg,
                         float *rgb, float *depth, float *trans, uint8_t *cls, bool stats) {
  RasterFrame f;
  const int ts = 1 << tshift;
  f.ranges = ws.bin[eye].ranges;
  f.ids = ws.bin[eye].ival;
  f.rec = ws.rec[eye];
  f.box = ws.bounds[eye];
  f.roi = (mask && tshift > 4) ? mask : nullptr;  // a 32-pixel tile may hold unmasked 16-pixel tiles
  f.skip = nullptr;
  f.rshift = 0;
  f.rtiles_x = 0;
  f.split = 0;
  f.items = mask ? ws.bin[eye].items : nullptr;
  f.n_items = mask ? &ws.ctr->n_items[eye] : nullptr;
  f.rgb = rgb;
  f.depth = depth;
  f.trans = trans;
  f.cls = cls;
  f.winit = nullptr;
  f.ctr = ws.ctr;
  f.bg[0] = bg.x;
  f.bg[1] = bg.y;
  f.bg[2] = bg.z;
  f.W = W;
  f.H = H;
  f.tiles_x = (W + ts - 1) >> tshift;
  f.ntiles = f.tiles_x * ((H + ts - 1) >> tshift);
  f.tshift = tshift;
  f.eye = eye;
  f.stats = stats ? 1 : 0;
  f.lowpass = ws.prim ? kNoLowpass : 2.f;
  f.n_rec = (uint32_t)ws.max_surfels;
  return f;
}


}  // namespace gs
