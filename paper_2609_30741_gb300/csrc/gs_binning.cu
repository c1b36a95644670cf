// Tile binning: every tile's list of the surfels that can reach it, in the
// order of the packed (tile id | depth) key sort of the 2DGS/3DGS tile
// rasterizer.
//
// Paper: Sec. 3.1 Stage 1 and Sec. 3.5 (16x16 tiles of the 2DGS/3DGS tile
// rasterizer; Sec. 2.2 keeps its depth ordering).
//
// Sorting by (tile, depth) is the same as sorting the surfels by depth first and
// then grouping them by tile without changing their order. So the surfels are
// radix sorted once on their 32 depth bits (ties keep the index order), and
// the grouping by tile is a stable counting sort: the depth-ordered surfels are
// cut into chunks, a first pass counts each chunk's hits per tile into a
// [tile][chunk] table, one scan of that table gives every (tile, chunk) run its
// place, and a second pass writes the surfel ids straight into their slots. The
// per-instance (tile, surfel) pairs are never materialised or radix sorted.
//
// A surfel is binned to a tile only when its support can reach one of the
// tile's pixel centres: the support {o Ghat >= 1/255} is the union of the
// projected disc u^2 + v^2 <= r_c^2 (an ellipse in screen space, because the
// whole disc lies in front of the near plane) and the low-pass disc around the
// projected centre. The test is exact for the continuous tile rectangle (so it
// keeps every contributing pair) with the radius grown by 1e-3 for float32
// safety; the few surfels whose ellipse is too thin and oblique to solve in
// float32 keep their whole bounding rectangle. An ellipsoid's record has the
// same form (its screen conic in place of the plane coefficients) and no
// low-pass disc.
//
// Pipeline per eye (all counts stay on the device):
//   1. tile ranges of every rectangle row (rows_kernel); an ROI binning also
//      selects the surfels whose rectangle holds an ROI tile
//   2. radix sort of the selected surfels over the 32 depth bits, or the dominant
//      eye's order filtered
//   3. per chunk and warp, depth-ordered lists of every tile row's ranges
//   4. per-(tile, chunk) counts (bin_count_kernel)
//   5. tile-major scan of the counts -> run offsets, tile ranges
//   6. placement of every surfel id (bin_place_kernel)
#include <mutex>

#include "gs_conic.cuh"
#include "gs_internal.cuh"
#include "gs_launch.cuh"
#include "gs_scan.cuh"
#include "gs_sort.cuh"

namespace gs {

// Tile columns [t0, t1] (tile edge ts = 1 << tshift) whose pixel centres meet the
// absolute interval [xa, xb].
__device__ __forceinline__ void tile_span(float xa, float xb, int W, int rx0, int rx1, int tshift, int &t0,
                                          int &t1) {
  if (!(xa <= xb) || xa > (float)(W - 1) + kBoundPad || xb < -kBoundPad) {
    t0 = 1;
    t1 = 0;
    return;
  }
  const float ts = (float)(1 << tshift), its = 1.f / ts;  // exact: a power of two
  t0 = max(rx0, (int)ceilf((xa - kBoundPad - (ts - 1.f)) * its));
  t1 = min(rx1, (int)floorf((xb + kBoundPad) * its));
}

// Up to two tile ranges [a0, a1] u [c0, c1] (disjoint, a before c) of tile row ty
// that the surfel's support reaches; empty ranges have lo > hi.
__device__ __forceinline__ void row_ranges(const Conic &q, const float4 r0, int ty, int W, int H, int rx0, int rx1,
                                           int tshift, int &a0, int &a1, int &c0, int &c1) {
  const int ts = 1 << tshift;
  const float y0 = (float)(ty * ts) - kBoundPad;
  const float y1 = (float)min(ty * ts + ts - 1, H - 1) + kBoundPad;
  float elo, ehi, dlo, dhi;
  band_slices(q, y0 - r0.y, y1 - r0.y, elo, ehi, dlo, dhi);
  tile_span(r0.x + elo, r0.x + ehi, W, rx0, rx1, tshift, a0, a1);
  tile_span(r0.x + dlo, r0.x + dhi, W, rx0, rx1, tshift, c0, c1);
  if (a0 > a1) {
    a0 = c0; a1 = c1; c0 = 1; c1 = 0;
  } else if (c0 <= c1) {
    if (c0 <= a1 + 1 && c1 >= a0 - 1) {  // overlapping or adjacent: merge
      a0 = min(a0, c0); a1 = max(a1, c1); c0 = 1; c1 = 0;
    } else if (c1 < a0) {                 // keep the ranges in increasing order
      const int t0 = a0, t1 = a1;
      a0 = c0; a1 = c1; c0 = t0; c1 = t1;
    }
  }
}

// Summed-area table of the ROI tile mask: sat[y][x] = masked tiles with row < y
// and column < x, (tiles_y + 1) x (tiles_x + 1) entries. One block: each warp
// takes whole rows (prefix counts by ballot, 32 columns at a time), then each
// thread adds one column down the rows.
// With roi16 given, the mask is first derived from the ROI mask on the 16-pixel
// grid (rtx x rty tiles): a tile of edge 1 << tshift is masked when it holds a
// masked pixel. clip[0][ty][tx] / clip[1][ty][tx] get the first masked column
// >= tx / the last masked column <= tx of row ty (0xffff: none), by ballots 32
// columns at a time with the carry of the columns already passed. With list16
// given, list16[0] gets the number of masked 16-pixel tiles and list16[1..] the
// tiles (a rasterizer on the 16-pixel grid reading this grid's lists).
__global__ void __launch_bounds__(1024) mask_sat_kernel(uint8_t *mask, int tiles_x, int tiles_y,
                                                        uint32_t *__restrict__ sat, const uint8_t *__restrict__ roi16,
                                                        int rtx, int rty, int tshift, uint16_t *__restrict__ clip,
                                                        uint32_t *__restrict__ list16,
                                                        uint32_t *__restrict__ n_rows,
                                                        uint32_t *__restrict__ n_more) {
  griddep_wait();
  if (threadIdx.x == 0) *n_rows = *n_more = 0u;  // the row spans of this binning follow
  constexpr int kSatSmem = 12000;
  __shared__ uint32_t s_sat[kSatSmem];
  __shared__ uint32_t s_n16;
  if (list16 && roi16) {
    if (threadIdx.x == 0) s_n16 = 0u;
    __syncthreads();
    const int n16 = rtx * rty;
    for (int b0 = (threadIdx.x >> 5) * 32; b0 < n16; b0 += (int)blockDim.x) {  // warp-uniform
      const int t = b0 + (int)(threadIdx.x & 31);
      const bool on = t < n16 && roi16[t] != 0;
      const unsigned bal = __ballot_sync(0xffffffffu, on);
      if (!bal) continue;
      uint32_t base = 0;
      if ((threadIdx.x & 31) == 0) base = atomicAdd(&s_n16, (uint32_t)__popc(bal));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (on) list16[1 + base + (uint32_t)__popc(bal & ((1u << (threadIdx.x & 31)) - 1u))] = (uint32_t)t;
    }
    __syncthreads();
    if (threadIdx.x == 0) list16[0] = s_n16;
  }
  if (roi16) {
    for (int t = threadIdx.x; t < tiles_x * tiles_y; t += blockDim.x) {
      const int x = t % tiles_x, y = t / tiles_x;
      uint8_t v = 0;
      if (tshift <= 4) {
        v = roi16[(y >> (4 - tshift)) * rtx + (x >> (4 - tshift))];
      } else {
        const int sc = 1 << (tshift - 4);
        for (int dy = 0; dy < sc; ++dy)
          for (int dx = 0; dx < sc; ++dx) {
            const int yy = y * sc + dy, xx = x * sc + dx;
            if (yy < rty && xx < rtx) v |= roi16[yy * rtx + xx];
          }
      }
      mask[t] = v ? 1 : 0;
    }
    __syncthreads();
  }
  const int sx = tiles_x + 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int nt = tiles_x * tiles_y;
  for (int y = wid; y < tiles_y; y += nw) {
    const uint8_t *row = mask + (size_t)y * tiles_x;
    uint32_t carry = 0xffffu;  // previous masked column: left to right
    for (int x0 = 0; x0 < tiles_x; x0 += 32) {  // warp-uniform
      const int x = x0 + lane;
      const uint32_t b = __ballot_sync(0xffffffffu, x < tiles_x && row[x] != 0);
      const uint32_t le = b & (0xffffffffu >> (31 - lane));  // columns <= x
      if (x < tiles_x) clip[nt + y * tiles_x + x] = (uint16_t)(le ? (uint32_t)x0 + 31u - __clz(le) : carry);
      if (b) carry = (uint32_t)x0 + 31u - __clz(b);
    }
    carry = 0xffffu;  // next masked column: right to left
    for (int x0 = (tiles_x - 1) & ~31; x0 >= 0; x0 -= 32) {  // warp-uniform
      const int x = x0 + lane;
      const uint32_t b = __ballot_sync(0xffffffffu, x < tiles_x && row[x] != 0);
      const uint32_t ge = b & (0xffffffffu << lane);  // columns >= x
      if (x < tiles_x) clip[y * tiles_x + x] = (uint16_t)(ge ? (uint32_t)x0 + (uint32_t)__ffs(ge) - 1u : carry);
      if (b) carry = (uint32_t)x0 + (uint32_t)__ffs(b) - 1u;
    }
  }
  // the table is built in shared memory when it fits (the column pass is a
  // dependent chain down each column) and then copied out
  const int nsat = (tiles_y + 1) * sx;
  uint32_t *S = nsat <= kSatSmem ? s_sat : sat;
  for (int y = wid; y <= tiles_y; y += nw) {
    uint32_t acc = 0;
    if (lane == 0) S[(size_t)y * sx] = 0u;
    for (int x0 = 0; x0 < tiles_x; x0 += 32) {  // warp-uniform
      const int x = x0 + lane;
      const bool on = y > 0 && x < tiles_x && mask[(size_t)(y - 1) * tiles_x + x] != 0;
      const uint32_t b = __ballot_sync(0xffffffffu, on);
      if (x < tiles_x) S[(size_t)y * sx + x + 1] = acc + (uint32_t)__popc(b & (0xffffffffu >> (31 - lane)));
      acc += (uint32_t)__popc(b);
    }
  }
  __syncthreads();
  for (int x = threadIdx.x; x <= tiles_x; x += blockDim.x) {
    uint32_t acc = 0;
    for (int y = 1; y <= tiles_y; ++y) {
      acc += S[(size_t)y * sx + x];
      S[(size_t)y * sx + x] = acc;
    }
  }
  if (S != sat) {
    __syncthreads();
    for (int i = threadIdx.x; i < nsat; i += blockDim.x) sat[i] = S[i];
  }
}

// Any ROI tile in tile rows [y0, y1] x columns [x0, x1]?
__device__ __forceinline__ bool sat_any(const uint32_t *sat, int tiles_x, int y0, int y1, int x0, int x1) {
  if (y0 > y1 || x0 > x1) return false;
  const int sx = tiles_x + 1;
  const uint32_t v = sat[(size_t)(y1 + 1) * sx + x1 + 1] - sat[(size_t)y0 * sx + x1 + 1] -
                     sat[(size_t)(y1 + 1) * sx + x0] + sat[(size_t)y0 * sx + x0];
  return v != 0u;
}

// The masked tiles of tile row ty between columns [x0, x1]: the span clipped to
// its first and last masked tile (empty, lo > hi, when it has none), from the
// row's next / previous masked-column tables. The tiles in between may still be
// unmasked; the counting sort skips those one by one.
__device__ __forceinline__ void clip_to_mask(const uint16_t *clip, int tiles_x, int tiles_y, int ty, int &x0,
                                             int &x1) {
  if (x0 > x1) return;
  const int first = clip[ty * tiles_x + x0];  // 0xffff when none: beyond any column
  if (first > x1) {
    x0 = 1;
    x1 = 0;
    return;
  }
  x1 = clip[tiles_x * tiles_y + ty * tiles_x + x1];
  x0 = first;
}

// ---------------------------------------------------------------- row spans
constexpr uint32_t kInfoBinned = 1u;  // of a surfel's info: binned by this eye
// A range of tile columns [lo, hi] (empty: [1, 0]) in 18 bits.
constexpr int kColBits = 9;
constexpr uint32_t kColMask = (1u << kColBits) - 1u, kNoRange = 1u << kColBits;
static_assert(kMaxTileCols <= 1 << kColBits, "tile columns of a range");
__device__ __forceinline__ uint32_t pack_range(int lo, int hi) { return (uint32_t)lo << kColBits | (uint32_t)hi; }
__device__ __forceinline__ int range_lo(uint32_t r) { return (int)(r >> kColBits & kColMask); }
__device__ __forceinline__ int range_hi(uint32_t r) { return (int)(r & kColMask); }

// Once per eye and frame, every tile row of every surfel's bounding rectangle
// gets its tile range [a0, a1] (row_ranges; an ill-conditioned ellipse keeps the
// whole row of its rectangle), packed as 2 x 9 bits. The few rows with a second
// range (the low-pass disc apart from the ellipse: at most two a surfel) put it in
// `more`, a surfel's chained from its info. Half the bytes of two ranges a row, and
// the row lists gather them at random. A warp
// takes 32 consecutive surfels (one per lane), reserves slots for all their rows
// with one atomic, and then computes the rows 32 at a time, one per lane, so no
// lane idles while another walks a large surfel. info[i] collects what the row
// lists need of surfel i in one 16-byte record, because they gather it at random
// in depth order: the rectangle, the slot of its first row, and above the flag that
// this eye bins it the place of its first second range in `more`, plus one. An ROI
// binning keeps of each range only the part from its first to its last masked
// tile, skips the surfels whose rectangle holds no ROI tile, and marks the others
// in `bits`, the selection its depth order is taken from: the test then runs once
// per surfel in id order (coalesced), and the order filters a bit mask. The grid
// strides over the surfels, so a small grid can run beside other kernels.
__global__ void __launch_bounds__(256) rows_kernel(uint32_t n, const float4 *__restrict__ rec,
                                                   const ushort4 *__restrict__ rect,
                                                   const uint32_t *__restrict__ vis,
                                                   const CamBlock *__restrict__ cams, int eye, int prim,
                                                   uint4 *__restrict__ info, uint32_t *__restrict__ spans,
                                                   uint32_t cap, uint32_t *__restrict__ n_rows,
                                                   uint2 *__restrict__ more, uint32_t more_cap,
                                                   uint32_t *__restrict__ n_more, uint32_t *__restrict__ status, const uint16_t *__restrict__ clip,
                                                   int clip_tiles_x, int clip_tiles_y,
                                                   const uint32_t *__restrict__ sat, uint32_t *__restrict__ bits) {
  griddep_wait();
  const int lane = threadIdx.x & 31;
  const int W = cams->eye[eye].W, H = cams->eye[eye].H, tshift = cams->eye[eye].tshift;
  const uint32_t stride = gridDim.x * blockDim.x;  // a multiple of 32: j0 stays warp-aligned
  for (uint32_t j0 = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; j0 < n; j0 += stride) {  // warp-uniform
  const uint32_t i = j0 + (uint32_t)lane;
  int nr = 0, ry = 0, rx0 = 0, rx1 = -1;
  Conic q{};
  float cx = 0.f, cy = 0.f;
  bool bin = (vis[j0 >> 5] >> lane) & 1u;
  ushort4 rc = make_ushort4(0, 0, 0, 0);
  if (bin) {
    rc = rect[i];
    if (sat) bin = sat_any(sat, clip_tiles_x, rc.y, rc.w, rc.x, rc.z);  // the binning's ROI test
  }
  if (bits) {
    const uint32_t m = __ballot_sync(0xffffffffu, bin);
    if (lane == 0) bits[j0 >> 5] = m;
    if (!m) continue;  // warp-uniform; the lists hold none of these
  }
  if (bin) {
    nr = (int)rc.w - (int)rc.y + 1;
    ry = rc.y;
    rx0 = rc.x;
    rx1 = rc.z;
    const float4 *r = rec + 4 * (size_t)i;
    const float4 r0 = r[0], r1 = r[1], r2 = r[2];
    q = make_conic(r0, r1, r2);
    if (prim) q.rl2 = -1.f;  // ellipsoids have no low-pass disc
    cx = r0.x;
    cy = r0.y;
  }
  int incl = nr;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  uint32_t base = 0;
  if (lane == 31 && total > 0) base = atomicAdd(n_rows, (uint32_t)total);
  base = __shfl_sync(0xffffffffu, base, 31);
  if (lane == 0 && total > 0 && (uint64_t)base + (uint64_t)total > cap) atomicOr(status, kStCapacity);
  uint32_t head = 0;  // the surfel's second ranges: place in `more` plus one, or none
  for (int q0 = 0; q0 < total; q0 += 32) {
    const int qq = q0 + lane;
    int kl = 0, kh = 31;
#pragma unroll
    for (int it = 0; it < 5; ++it) {
      const int mid = (kl + kh) >> 1;
      if (__shfl_sync(0xffffffffu, incl, mid) > qq) kh = mid; else kl = mid + 1;
    }
    const int k = kl;
    const int excl_k = __shfl_sync(0xffffffffu, incl, k) - __shfl_sync(0xffffffffu, nr, k);
    const int ty = __shfl_sync(0xffffffffu, ry, k) + (qq - excl_k);
    const int sx0 = __shfl_sync(0xffffffffu, rx0, k), sx1 = __shfl_sync(0xffffffffu, rx1, k);
    Conic qk;
    qk.Sxx = __shfl_sync(0xffffffffu, q.Sxx, k);
    qk.Sxy = __shfl_sync(0xffffffffu, q.Sxy, k);
    qk.Syy = __shfl_sync(0xffffffffu, q.Syy, k);
    qk.gx = __shfl_sync(0xffffffffu, q.gx, k);
    qk.gy = __shfl_sync(0xffffffffu, q.gy, k);
    qk.h = __shfl_sync(0xffffffffu, q.h, k);
    qk.dcx = __shfl_sync(0xffffffffu, q.dcx, k);
    qk.dcy = __shfl_sync(0xffffffffu, q.dcy, k);
    qk.ex = __shfl_sync(0xffffffffu, q.ex, k);
    qk.ey = __shfl_sync(0xffffffffu, q.ey, k);
    qk.rl2 = __shfl_sync(0xffffffffu, q.rl2, k);
    qk.inv_sxx = __shfl_sync(0xffffffffu, q.inv_sxx, k);
    qk.slope = __shfl_sync(0xffffffffu, q.slope, k);
    qk.ok = __shfl_sync(0xffffffffu, q.ok ? 1 : 0, k) != 0;
    const float4 ck = make_float4(__shfl_sync(0xffffffffu, cx, k), __shfl_sync(0xffffffffu, cy, k), 0.f, 0.f);
    const uint32_t slot = base + (uint32_t)qq;
    bool two = false;
    uint32_t second = 0;
    if (qq < total && slot < cap) {
      int a0 = sx0, a1 = sx1, c0 = 1, c1 = 0;
      if (qk.ok) row_ranges(qk, ck, ty, W, H, sx0, sx1, tshift, a0, a1, c0, c1);
      if (clip) {  // an ROI binning: only the masked part of each range
        clip_to_mask(clip, clip_tiles_x, clip_tiles_y, ty, a0, a1);
        clip_to_mask(clip, clip_tiles_x, clip_tiles_y, ty, c0, c1);
        if (a0 > a1) { a0 = c0; a1 = c1; c0 = 1; c1 = 0; }
      }
      // empty ranges are stored as [1, 0]
      if (a0 > a1) { a0 = 1; a1 = 0; }
      if (c0 > c1) { c0 = 1; c1 = 0; }
      two = c0 <= c1;
      spans[slot] = pack_range(a0, a1);
      second = pack_range(c0, c1);
    }
    const uint32_t twos = __ballot_sync(0xffffffffu, two);
    if (twos) {  // rare: each joins its surfel's chain
      uint32_t at = 0;
      if (lane == 0) {
        at = atomicAdd(n_more, (uint32_t)__popc(twos));
        if ((uint64_t)at + (uint64_t)__popc(twos) > more_cap) atomicOr(status, kStCapacity);
      }
      at = __shfl_sync(0xffffffffu, at, 0);
      for (uint32_t t = twos; t; t &= t - 1u, ++at) {  // warp-uniform
        const int src = __ffs((int)t) - 1, owner = __shfl_sync(0xffffffffu, k, src);
        const uint32_t next = __shfl_sync(0xffffffffu, head, owner);
        if (at >= more_cap) continue;
        if (lane == src) more[at] = make_uint2(next, (uint32_t)ty << (2 * kColBits) | second);
        if (lane == owner) head = at + 1u;
      }
    }
  }
  if (i < n && (bin || !bits))  // with a selection of its own the lists hold no unbinned surfel
    info[i] = make_uint4((uint32_t)rc.x | ((uint32_t)rc.y << 16), (uint32_t)rc.z | ((uint32_t)rc.w << 16),
                         base + (uint32_t)(incl - nr), (bin ? kInfoBinned : 0u) | head << 1);
  }
}

// ---------------------------------------------------------------- depth order
// A surfel enters the depth sort when its bounding rectangle is not empty and,
// for an ROI binning, when that rectangle holds at least one ROI tile; the union
// variant (dominant eye of a parallel two-eye call) takes every surfel either
// eye bins.
// What the depth order's last CTA sets up for the rest of a binning: the binned
// count, cleared list and tile-list counters, the chunks holding binned surfels
// and the size of the (tile, chunk) table scan over them.
struct BinCounts {
  uint32_t *n_out, *n_band, *n_entries, *n_items, *n_chunks, *n_table;
  uint32_t chunk, ntiles;
  __device__ void operator()(uint32_t total) const {
    *n_out = total;
    *n_band = 0u;
    *n_entries = 0u;
    *n_items = 0u;
    // at least one chunk, so that every tile's range is written
    const uint32_t nc = total > 0u ? (total + chunk - 1) / chunk : 1u;
    *n_chunks = nc;
    *n_table = nc * ntiles;
  }
};

// The affiliated eye's surfels in the dominant eye's depth order: a stable filter
// of that order. For a parallel rig both eyes' keys are identical, so the
// filtered order is exactly the affiliated (depth, index) order.
struct ReuseLoad {
  const uint32_t *order, *n_order;  // the dominant binning's
  uint32_t n_max;
  const uint32_t *bits;             // the selected surfels
  __device__ uint32_t operator()(uint32_t i) const {
    if (i >= load_n(n_order, n_max)) return 0u;
    const uint32_t id = order[i];
    return (bits[id >> 5] >> (id & 31u)) & 1u;
  }
};

struct ReuseApply {
  const uint32_t *order;
  uint32_t *val_out;
  BinCounts bc;
  using Payload = uint32_t;  // surfel id
  __device__ Payload fetch(uint32_t i, uint32_t v) const { return v ? order[i] : 0u; }
  __device__ void operator()(uint32_t, uint32_t prefix, uint32_t v, Payload id) const {
    if (v) val_out[prefix] = id;
  }
  __device__ void end(uint32_t, uint32_t total) const { bc(total); }
};

// ---------------------------------------------------------------- counting sort by tile
//
// The depth-ordered surfels are cut into chunks of kBinWarps sub-chunks of
// `warp_surfels` consecutive surfels (one per warp).
//
//   row lists (one CTA per sub-chunk): per tile row, the tile ranges of the
//     sub-chunk's surfels in that row, in depth order (a row with two ranges gives
//     two entries, one that is empty an empty one), each with its surfel's place in
//     the sub-chunk;
//   mode 0 (CTA per (chunk, kCountRows rows)): each warp counts its lists' hits
//     per tile; the 8 counts of a (tile, chunk) go to table[tile][chunk] as 8 x 16
//     bits;
//   (a tile-major scan of the per-(tile, chunk) sums gives offs[tile][chunk],
//    where chunk c's run of the tile starts; offs[tile][0] starts the tile's list)
//   mode 1 (CTA per (chunk, row)): each warp starts at offs[tile][c] plus the
//     counts of the warps before it and writes every surfel id to its slot.
constexpr int kBinWarps = 8;
constexpr int kBinThreads = kBinWarps * 32;
constexpr int kBandRows = 4;    // rows of a band (gs_usage counts (surfel, band) pairs with a row entry)
static_assert(kBandRows == 4, "row_list_kernel finds a band's rows in a block's nibbles");
constexpr int kCountRows = 4;   // rows a counting CTA takes

// One (surfel, row range) in 32 bits: the surfel's place in its sub-chunk above its
// columns. The sub-chunk's ids (a few KB) stay in L1; with the id itself an entry takes
// 8 bytes, and the pool has to hold as many entries as the eye has spans.
using RowEntry = uint32_t;
static_assert(sizeof(RowEntry) == kRowEntryBytes, "row entry layout");
constexpr uint32_t kMaxWarpSurfels = 1u << (32 - 2 * kColBits);
__device__ __forceinline__ RowEntry row_entry(uint32_t place, uint32_t range) { return place << (2 * kColBits) | range; }
__device__ __forceinline__ uint32_t entry_place(RowEntry e) { return e >> (2 * kColBits); }

struct ListArgs {
  const uint32_t *ids;     // depth-ordered binned surfels
  const uint32_t *n_vis;
  uint32_t n_max;
  const uint4 *info;       // per surfel: rectangle, slot of its first row in spans, flags (rows_kernel)
  const uint32_t *spans;   // tile range of every rectangle row (rows_kernel)
  const uint2 *more;       // the second ranges: next of the surfel plus one, row << 18 | range
  uint32_t span_cap;
  const uint16_t *clip;    // ROI mask: per row and column the next masked column, or null
  int tiles_x, tiles_y;
  uint32_t warp_surfels;
  RowEntry *pool;          // all lists
  uint32_t pool_cap;
  uint32_t *pool_n;        // entries taken (device counter)
  uint32_t *n_band;        // (surfel, band) pairs (device counter)
  uint2 *lists;            // [chunk][row][warp]: (first entry, entries)
  uint32_t *status;
};

// ---- bit matrices over a warp ----
// Bits [lo, hi] of a 32-column block that starts at column `base` (lo = hi + 1:
// none; shl.b32 gives 0 for shifts of 32 and more).
__device__ __forceinline__ uint32_t ones_from(int n) {
  uint32_t v;
  asm("shl.b32 %0, %1, %2;" : "=r"(v) : "r"(0xffffffffu), "r"((uint32_t)max(n, 0)));
  return v;
}
__device__ __forceinline__ uint32_t range_bits(int lo, int hi, int base) {
  return ones_from(lo - base) & ~ones_from(hi + 1 - base);
}

// Transposes the 32 x 32 bit matrix whose row i is lane i's x: lane t gets bit t
// of every lane, lane i's at bit i. Five exchanges of half blocks: a lane keeps
// the half that stays and takes the other lane's rotated by the block's size.
__device__ __forceinline__ uint32_t transpose_bits(uint32_t x, int lane) {
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const uint32_t mk = j == 16 ? 0x0000ffffu : j == 8 ? 0x00ff00ffu : j == 4 ? 0x0f0f0f0fu : j == 2 ? 0x33333333u
                                                                                                   : 0x55555555u;
    const bool up = (lane & j) != 0;
    const uint32_t keep = up ? ~mk : mk;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (x & keep) | (__funnelshift_l(y, y, up ? 32 - j : j) & ~keep);
  }
  return x;
}

// Row lists: one CTA of kBinWarps warps per sub-chunk (the surfels of one
// counting-sort warp). The sub-chunk's 32-surfel groups are split into kBinWarps
// consecutive ranges, one per warp. Pass 0 counts each warp's entries per row; a
// CTA-wide scan turns the counts into the lists' places (rows in order, warps in
// order inside a row, so every list stays in depth order) with one pool
// reservation per sub-chunk; pass 1 walks the same groups again and writes the
// entries. A lane holds one surfel and its rows as a bit mask;
// the transposed masks give every row's surfels, for the counts and the places.
// Bound by the latency of the gathers in depth order (half of them miss L2 at 3M
// surfels at 2448x2448, dominant eye: 113 us; 182 with two ranges in 8 bytes a span and
// 8-byte entries, with which four CTAs per SM instead of six took 199).
__global__ void __launch_bounds__(kBinThreads, 6) row_list_kernel(ListArgs a) {
  griddep_wait();
  // per warp and row (padded to blocks of 32): pass 0 counts, then the warp's write
  // position; the surfels of the group in hand with a range, and with two
  extern __shared__ uint32_t s_dyn[];
  __shared__ uint32_t s_scan[32];
  __shared__ uint32_t s_base, s_bands;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t nv = load_n(a.n_vis, a.n_max);
  const uint32_t sub = blockIdx.x;                  // sub-chunk: chunk sub / kBinWarps, warp sub % kBinWarps
  const uint32_t c = sub / kBinWarps;
  if (c * kBinWarps * a.warp_surfels >= nv) return;  // the counting sort skips the whole chunk
  const int ny = a.tiles_y, nyp = (ny + 31) & ~31;
  uint32_t *s_rows = s_dyn;  // [kBinWarps][ny]
  uint2 *my_lists = a.lists + ((size_t)c * ny) * kBinWarps + (sub % kBinWarps);  // stride kBinWarps per row
  const uint32_t s0 = sub * a.warp_surfels;
  const uint32_t s1 = min(s0 + a.warp_surfels, nv);
  // this warp's groups of 32 surfels: [g0, g1) of the sub-chunk's ng groups
  const uint32_t ng = s1 > s0 ? (s1 - s0 + 31) / 32 : 0u;
  const uint32_t g0 = ng * (uint32_t)w / kBinWarps, g1 = ng * (uint32_t)(w + 1) / kBinWarps;
  uint32_t *cnt = s_rows + w * ny;
  uint32_t *col = s_dyn + kBinWarps * ny + w * 2 * nyp, *colb = col + nyp;
  for (int y = lane; y < ny; y += 32) cnt[y] = 0u;
  if (threadIdx.x == 0) s_bands = 0u;
  __syncthreads();
  uint32_t bands = 0;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    if (pass == 1) {
      // per row: the warps' exclusive offsets inside the row and the row's total;
      // then the rows' places in the sub-chunk's pool range
      __syncthreads();
      uint32_t run = 0;  // entries of the rows before this block of rows
      for (int y0 = 0; y0 < ny; y0 += kBinThreads) {  // CTA-uniform
        const int y = y0 + (int)threadIdx.x;
        uint32_t tot = 0;
        if (y < ny) {
#pragma unroll
          for (int ww = 0; ww < kBinWarps; ++ww) tot += s_rows[ww * ny + y];
        }
        uint32_t off;
        const uint32_t all = block_exclusive_scan<kBinThreads>(tot, &off, s_scan);
        if (y < ny) {
          uint32_t at = run + off;
          my_lists[(size_t)y * kBinWarps] = make_uint2(at, tot);  // relative to the reservation below
#pragma unroll
          for (int ww = 0; ww < kBinWarps; ++ww) {
            const uint32_t v = s_rows[ww * ny + y];
            s_rows[ww * ny + y] = at;
            at += v;
          }
        }
        run += all;
      }
      if (threadIdx.x == 0) {
        uint32_t base = 0;
        if (run > 0) base = atomicAdd(a.pool_n, run);
        if (run > 0 && (uint64_t)base + run > a.pool_cap) atomicOr(a.status, kStCapacity);
        if (s_bands > 0) atomicAdd(a.n_band, s_bands);
        s_base = base;
      }
      __syncthreads();
      const uint32_t base = s_base;
      for (int y = threadIdx.x; y < ny; y += kBinThreads) {
        uint2 l = my_lists[(size_t)y * kBinWarps];  // this thread's own store
        l.x += base;
        l.y = l.x >= a.pool_cap ? 0u : min(l.y, a.pool_cap - l.x);
        my_lists[(size_t)y * kBinWarps] = l;
      }
      for (int y = lane; y < ny; y += 32) cnt[y] += base;
      __syncwarp();
    }
    for (uint32_t g = g0; g < g1; ++g) {  // warp-uniform
      const uint32_t j = s0 + g * 32u + (uint32_t)lane;
      int y0 = 1, y1 = 0;
      uint32_t ro = 0;
      int x0 = 0, x1 = 0;
      uint32_t head = 0;
      uint4 inf = make_uint4(0u, 0u, 0u, 0u);
      if (j < s1) inf = __ldg(a.info + a.ids[j]);
      if (inf.w & kInfoBinned) {
        x0 = (int)(inf.x & 0xffffu); y0 = (int)(inf.x >> 16);
        x1 = (int)(inf.y & 0xffffu); y1 = (int)(inf.y >> 16);
        ro = inf.z;
        head = inf.w >> 1;
      }
      const bool any_split = __any_sync(0xffffffffu, head != 0u);
      const bool has = y0 <= y1;
      const int ymin = __reduce_min_sync(0xffffffffu, has ? y0 : 0x7fffffff);
      const int ymax = __reduce_max_sync(0xffffffffu, has ? y1 : -1);
      const int blk0 = ymin >> 5, blk1 = ymax >> 5;  // blocks of 32 rows
      uint32_t any_rb = 0;  // a row of the group has a second range
      for (int blk = blk0; blk <= blk1; ++blk) {  // warp-uniform
        const int base = blk * 32;
        uint32_t ra = has ? range_bits(y0, y1, base) : 0u;  // the surfel's rows
        if (a.clip) {  // an ROI binning: the rows with a masked tile in the rectangle
          uint32_t t = ra;
          while (t) {
            const int k = __ffs((int)t) - 1;
            t &= t - 1u;
            if ((int)a.clip[(base + k) * a.tiles_x + x0] > x1) ra &= ~(1u << k);
          }
        }
        const uint32_t ca = transpose_bits(ra, lane);  // lane k: the surfels with an entry in row base + k
        uint32_t cb = 0;
        if (any_split) {  // and those with a second one (rare)
          uint32_t rb = 0;
          for (uint32_t h = head; h;) {
            const uint2 m = __ldg(a.more + (h - 1u));
            const uint32_t k = (m.y >> (2 * kColBits)) - (uint32_t)base;
            if (k < 32u) rb |= 1u << k;
            h = m.x;
          }
          any_rb |= __any_sync(0xffffffffu, rb != 0u) ? 1u : 0u;
          cb = transpose_bits(rb, lane);
        }
        if (pass == 0) {
          uint32_t any4 = ra | (ra >> 1);
          any4 |= any4 >> 2;  // bit 4 b: a row of the block's band b
          bands += (uint32_t)__popc(any4 & 0x11111111u);
          if (base + lane < ny) cnt[base + lane] += (uint32_t)(__popc(ca) + __popc(cb));
        } else {
          col[blk * 32 + lane] = ca;
          if (any_split) colb[blk * 32 + lane] = cb;
        }
      }
      if (pass == 1) {
        __syncwarp();
        const uint32_t bit = 1u << lane;
#pragma unroll 4
        for (int y = y0; y <= y1; ++y) {
          const uint32_t m = col[y];
          const uint32_t slot = ro + (uint32_t)(y - y0);
          const uint32_t sp = (m & bit) && slot < a.span_cap ? __ldg(a.spans + slot) : kNoRange;
          uint32_t at = cnt[y] + (uint32_t)__popc(m & lt);
          if (any_rb) at += (uint32_t)__popc(colb[y] & lt);
          if ((m & bit) && at < a.pool_cap) a.pool[at] = row_entry(j - s0, sp);
          if (any_rb && (colb[y] & bit) && at + 1u < a.pool_cap) {
            uint2 m2 = __ldg(a.more + (head - 1u));
            while ((int)(m2.y >> (2 * kColBits)) != y) m2 = __ldg(a.more + (m2.x - 1u));  // the row is in the chain
            a.pool[at + 1u] = row_entry(j - s0, m2.y & ((1u << 2 * kColBits) - 1u));
          }
        }
        __syncwarp();
        for (int blk = blk0; blk <= blk1; ++blk) {
          const int y = blk * 32 + lane;
          if (y < ny) cnt[y] += (uint32_t)(__popc(col[y]) + (any_split ? __popc(colb[y]) : 0));
        }
        __syncwarp();
      }
    }
    if (pass == 0) {
      bands = __reduce_add_sync(0xffffffffu, bands);
      if (lane == 0 && bands) atomicAdd(&s_bands, bands);
    }
  }
}

struct BinArgs {
  const uint32_t *n_vis;   // binned surfels (device)
  uint32_t n_max;
  const uint32_t *ids;     // depth-ordered binned surfels
  const RowEntry *pool;
  const uint2 *lists;      // [chunk][row][warp]
  const uint8_t *mask;     // ROI tile mask, or null
  int tiles_x, tiles_y;
  uint32_t warp_surfels;   // surfels per warp sub-chunk
  uint32_t nch;            // chunks (row length of the tables)
  uint4 *table;            // [tile][chunk] 8 x 16-bit per-warp counts
  const uint32_t *offs;    // [tile][chunk] exclusive offsets (mode 1)
  uint32_t cap;            // instance capacity
  uint32_t *ival;          // surfel id per instance
  uint32_t *ikey;          // tile id per instance, or null
  uint32_t *cnt_bin;       // tiles per surfel, or null (mode 0)
};

__device__ __forceinline__ uint32_t half16(const uint4 &v, int w) {
  const uint32_t x = w < 2 ? v.x : w < 4 ? v.y : w < 6 ? v.z : v.w;
  return (w & 1) ? x >> 16 : x & 0xffffu;
}

// Mode 0. A range adds one at its first column and takes one off after its last:
// two shared-memory atomics an entry however long the range is, and a prefix sum
// along the row then gives the counts (an ROI binning drops the unmasked tiles').
// 1.5M / 3M surfels at 1920x1080 / 2448x2448: 15 / 29 us, against 69 / 163 for one
// atomic per instance.
__global__ void __launch_bounds__(kBinThreads) bin_count_kernel(BinArgs a) {
  griddep_wait();
  extern __shared__ uint32_t s_cnt[];  // [kCountRows][kBinWarps][tiles_x + 1]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t nv = load_n(a.n_vis, a.n_max);
  const uint32_t c = blockIdx.x;
  if (c * kBinWarps * a.warp_surfels >= nv) return;  // the scan reads these counts as 0
  const int tx_n = a.tiles_x, st = tx_n + 1;
  const int y0 = (int)blockIdx.y * kCountRows, ny = min(kCountRows, a.tiles_y - y0);
  uint2 li[kCountRows];
#pragma unroll
  for (int r = 0; r < kCountRows; ++r)
    li[r] = r < ny ? a.lists[((size_t)c * a.tiles_y + y0 + r) * kBinWarps + w] : make_uint2(0u, 0u);
  for (int i = tid; i < kCountRows * kBinWarps * st; i += kBinThreads) s_cnt[i] = 0u;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kCountRows; ++r) {
    if (li[r].y == 0u) continue;  // warp-uniform
    uint32_t *d = s_cnt + (r * kBinWarps + w) * st;
    const RowEntry *q = a.pool + li[r].x;
    for (uint32_t e = (uint32_t)lane; e < li[r].y; e += 32) {
      const RowEntry en = q[e];
      const int c0 = range_lo(en), c1 = range_hi(en);
      atomicAdd(&d[c0], 1u);
      atomicSub(&d[c1 + 1], 1u);
      if (a.cnt_bin) {
        uint32_t n = 0;
        for (int x = c0; x <= c1; ++x) n += !a.mask || a.mask[(size_t)(y0 + r) * tx_n + x] != 0;
        if (n) atomicAdd(&a.cnt_bin[a.ids[(c * kBinWarps + w) * a.warp_surfels + entry_place(en)]], n);
      }
    }
    __syncwarp();
    uint32_t carry = 0;
    for (int base = 0; base < tx_n; base += 32) {  // warp-uniform
      uint32_t v = base + lane < tx_n ? d[base + lane] : 0u;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
      }
      v += carry;
      carry = __shfl_sync(0xffffffffu, v, 31);
      if (base + lane < tx_n) d[base + lane] = v;
    }
  }
  __syncthreads();
  for (int i = tid; i < ny * tx_n; i += kBinThreads) {
    const int r = i / tx_n, x = i - r * tx_n;
    const size_t t = (size_t)(y0 + r) * tx_n + x;
    uint32_t h[kBinWarps];
    const bool on = !a.mask || a.mask[t] != 0;
#pragma unroll
    for (int ww = 0; ww < kBinWarps; ++ww) h[ww] = on ? s_cnt[(r * kBinWarps + ww) * st + x] : 0u;
    a.table[t * a.nch + c] =
        make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
  }
}

// Mode 1. A step takes 32 entries of the row's list, one per lane, and for every
// 32 tile columns they reach: the lane's columns as a bit mask, and the
// transposed matrix, which gives lane t the entries that reach column t. The lane
// walks its bits and writes those entries' ids to its tile's slots in depth
// order: no search for an instance's entry, no atomics and no ranking. One CTA
// per tile row: a whole band of four rows made a warp's chain of steps the time of
// the launch. 1.5M / 3M surfels at 1920x1080 / 2448x2448: 44 / 105 us, against 94 /
// 243 for an instance per lane ranked by shared-memory masks; collecting a CTA's
// instances in shared memory for coalesced copies measured 53 / 112. All with the ids in
// the entries; as gathers they cost 8 us more at 3M, and the row lists 69 less.
// An entry's id is one more gather behind the entry: it goes to shared memory by
// cp.async a step ahead, the first beside the counts' loads (loaded to a register with
// the entry it cost 3 us of the 660 of the 500k-surfel frame).
__device__ __forceinline__ void cp_async4(uint32_t *dst, const uint32_t *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__global__ void __launch_bounds__(kBinThreads, 8) bin_place_kernel(BinArgs a) {
  griddep_wait();
  extern __shared__ uint32_t s_cnt[];  // [kBinWarps][tiles_x]: every warp's next slot per tile
  __shared__ uint32_t s_id[2][kBinWarps][32];
  __shared__ uint32_t s_mask[(kMaxTileCols + 31) / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t nv = load_n(a.n_vis, a.n_max);
  const uint32_t c = blockIdx.x;
  if (c * kBinWarps * a.warp_surfels >= nv) return;
  const int tx_n = a.tiles_x;
  const int ty = (int)blockIdx.y;
  const size_t t0 = (size_t)ty * tx_n;  // first tile of the row
  const uint2 li = a.lists[((size_t)c * a.tiles_y + ty) * kBinWarps + w];
  const RowEntry *q = a.pool + li.x;
  const int qn = (int)li.y;
  const uint32_t *ids = a.ids + (size_t)(c * kBinWarps + w) * a.warp_surfels;
  RowEntry next = lane < qn ? q[lane] : kNoRange;
  if (!__syncthreads_or(qn > 0)) return;  // nothing reaches the row
  if (lane < qn) cp_async4(&s_id[0][w][lane], ids + entry_place(next));
  for (int bt = tid; bt < tx_n; bt += kBinThreads) {
    const size_t e = (t0 + bt) * a.nch + c;
    const uint4 v = a.table[e];
    uint32_t base = a.offs[e];
#pragma unroll
    for (int ww = 0; ww < kBinWarps; ++ww) {
      s_cnt[ww * tx_n + bt] = base;
      base += half16(v, ww);
    }
  }
  if (a.mask) {  // the ROI mask's bits, 32 columns a word
    for (int i = w; i < (tx_n + 31) / 32; i += kBinWarps) {  // warp-uniform
      const int x = i * 32 + lane;
      const uint32_t bits = __ballot_sync(0xffffffffu, x < tx_n && a.mask[t0 + x] != 0);
      if (lane == 0) s_mask[i] = bits;
    }
  }
  __syncthreads();
  uint32_t *my_cnt = s_cnt + w * tx_n;
  for (int qpos = 0, buf = 0; qpos < qn; qpos += 32, buf ^= 1) {  // warp-uniform
    const RowEntry en = next;
    const int e = qpos + 32 + lane;  // the next step's entries are fetched a step ahead
    next = e < qn ? q[e] : kNoRange;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();  // the step's ids are there, and those of the step before have been read
    const int c0 = range_lo(en), c1 = range_hi(en);
    const int lo = __reduce_min_sync(0xffffffffu, c0 <= c1 ? c0 : 0x7fffffff);
    const int hi = __reduce_max_sync(0xffffffffu, c0 <= c1 ? c1 : -1);
    for (int base = lo & ~31; base <= hi; base += 32) {  // warp-uniform
      uint32_t bits = range_bits(c0, c1, base);
      if (a.mask) bits &= s_mask[base >> 5];
      uint32_t m = transpose_bits(bits, lane);  // the entries that reach column base + lane
      if (m) {  // the lane's column is in the row: no other lane touches its counter
        uint32_t pos = my_cnt[base + lane];
        do {
          const uint32_t id = s_id[buf][w][__ffs((int)m) - 1];
          m &= m - 1u;
          if (pos < a.cap) {
            a.ival[pos] = id;
            if (a.ikey) a.ikey[pos] = (uint32_t)(t0 + base + lane);
          }
          ++pos;
        } while (m);
        my_cnt[base + lane] = pos;
      }
    }
    if (e < qn) cp_async4(&s_id[buf ^ 1][w][lane], ids + entry_place(next));
  }
}

// The tile-major scan runs over the (tile, chunk) entries of the chunks that
// hold binned surfels only (one chunk when none does): element i is tile
// i / n_chunks, chunk i % n_chunks (the table rows keep their full length nch).
struct BinTableLoad {
  const uint4 *table;
  const uint32_t *n_chunks, *n_vis;
  uint32_t nch, chunk;
  __device__ uint32_t operator()(uint32_t i) const {
    const uint32_t na = *n_chunks, c = i % na;
    if (c * chunk >= *n_vis) return 0u;  // only with no binned surfel: bin_count_kernel wrote nothing
    const uint4 v = table[(size_t)(i / na) * nch + c];
    const uint32_t lo = (v.x & 0xffffu) + (v.y & 0xffffu) + (v.z & 0xffffu) + (v.w & 0xffffu);
    return lo + (v.x >> 16) + (v.y >> 16) + (v.z >> 16) + (v.w >> 16);
  }
};

// Offsets of every (tile, chunk) run; the first chunk's entry of a tile also
// gives the tile's range (its start, and the end of the tile before it), and a
// masked binning lists its masked tiles for the persistent rasterizer (in any
// order: the rasterizer's tiles are independent).
struct BinOffsetApply {
  uint32_t *offs;
  const uint32_t *n_chunks;
  uint32_t nch;
  uint32_t *n_inst, *n_sort;
  uint32_t cap;
  uint32_t *status;
  uint2 *ranges;
  int ntiles;
  const uint8_t *mask;  // null for a full binning
  uint32_t *items, *n_items;
  using Payload = uint2;  // chunks in use, the tile's mask byte (first chunk only)
  __device__ Payload fetch(uint32_t i, uint32_t) const {
    const uint32_t na = *n_chunks;
    return make_uint2(na, (mask && i % na == 0u) ? (uint32_t)mask[i / na] : 0u);
  }
  __device__ void operator()(uint32_t i, uint32_t prefix, uint32_t, Payload pl) const {
    const uint32_t na = pl.x;
    const uint32_t t = i / na, c = i % na;
    offs[(size_t)t * nch + c] = prefix;
    if (c != 0u) return;
    const uint32_t p = min(prefix, cap);
    ranges[t].x = p;
    if (t > 0u) ranges[t - 1].y = p;
    if (pl.y) items[atomicAdd(n_items, 1u)] = t;
  }
  __device__ void end(uint32_t, uint32_t total) const {
    *n_inst = total;
    *n_sort = total < cap ? total : cap;
    if (total > cap) atomicOr(status, kStCapacity);
    if (ntiles > 0) ranges[ntiles - 1].y = min(total, cap);
  }
};

uint32_t bin_warp_surfels(int max_surfels) {
  const uint32_t per = ((uint32_t)max_surfels + kBinWarps * 256 - 1) / (kBinWarps * 256);
  uint32_t r = (per + 31) / 32 * 32;
  if (r < 64) r = 64;
  if (r > kMaxWarpSurfels) r = kMaxWarpSurfels;  // (and the per-warp counts are 16-bit)
  return r;
}

size_t row_list_words(int max_surfels, int max_tiles_y) {
  return (size_t)bin_chunks(max_surfels) * max_tiles_y * kBinWarps;
}

uint32_t bin_chunks(int max_surfels) {
  const uint32_t chunk = kBinWarps * bin_warp_surfels(max_surfels);
  const uint32_t n = ((uint32_t)max_surfels + chunk - 1) / chunk;
  return n < 1 ? 1 : n;
}

size_t count_smem_bytes(int tiles_x) { return sizeof(uint32_t) * kCountRows * kBinWarps * ((size_t)tiles_x + 1); }
size_t place_smem_bytes(int tiles_x) { return sizeof(uint32_t) * kBinWarps * (size_t)tiles_x; }
size_t list_smem_bytes(int tiles_y) {
  return sizeof(uint32_t) * kBinWarps * ((size_t)tiles_y + 2 * (((size_t)tiles_y + 31) & ~(size_t)31));
}
static_assert(sizeof(uint32_t) * kBinWarps * kMaxTileCols <= 40 * 1024, "bin_place_kernel needs no opt-in");

// The opt-in is a property of the kernel on the device, shared by every
// context: it only ever grows, so a small context created after a large one
// keeps the large one's limit.
cudaError_t prepare_binning(int max_tiles_x, int max_tiles_y) {
  static std::mutex mu;
  static int granted[2][64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  const auto grant = [&](const void *fn, size_t bytes, int *have) {
    const int want = (int)bytes;
    if (e != cudaSuccess || (dev >= 0 && dev < 64 && have[dev] >= want)) return;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, want);
    if (e == cudaSuccess && dev >= 0 && dev < 64) have[dev] = want;
  };
  grant((const void *)bin_count_kernel, count_smem_bytes(max_tiles_x), granted[0]);
  grant((const void *)row_list_kernel, list_smem_bytes(max_tiles_y), granted[1]);
  return e;
}

cudaError_t launch_binning(const Workspace &ws, int eye, int n, int tiles_x, int tiles_y,
                           const uint8_t *tile_mask, cudaStream_t s, int order, const uint8_t *roi16, int W,
                           int H, int tshift, const SideRows *rows) {
  const BinScratch &b = ws.bin[eye];
  cudaError_t err;
  Counters *ctr = ws.ctr;
  const int ntiles = tiles_x * tiles_y;
  const uint32_t cap = (uint32_t)ws.max_inst[eye];
  const RadixScratch rs{b.rs_hist, b.rs_hist + kRsPasses * 256, b.rs_status, b.rs_ctl, &ctr->status};
  if (tile_mask) {  // (the rasterizer-grid mask and) its summed-area table
    launch_k(mask_sat_kernel, 1, 1024, 0, s, const_cast<uint8_t *>(tile_mask), tiles_x, tiles_y, b.mask_sat, roi16,
             (W + kTile - 1) / kTile, (H + kTile - 1) / kTile, roi16 ? tshift : 4, b.mask_clip,
             roi16 ? b.items16 : nullptr, &ctr->n_rows[eye], &ctr->n_more[eye]);
    GS_LAUNCHED(1);
  }
  // 1. the row spans. A full binning's need only the preprocessed records: on a
  // second stream they run beside the depth order. An ROI binning's select its
  // surfels for the depth order and come first.
  const bool side = rows && n > 0 && !tile_mask;
  const bool sort = order != kOrderReuse;
  const uint32_t *bits = tile_mask ? b.bits : ws.vis[eye];
  const auto launch_rows = [&](cudaStream_t st) -> cudaError_t {
    if (n <= 0) return cudaSuccess;
    // beside the sort a small grid leaves its latency-bound passes their SMs; with
    // more surfels the spans are the longer branch, and a third CTA per SM pays. Mono
    // frames with 2 / 3 per SM, us: object scene 425 / 429 at 500k surfels, 495 / 495 at
    // 750k, 567 / 553 at 1M, 646 / 621 at 1.25M; unbounded scene 418 / 424 at 750k,
    // 488 / 483 at 1M, 615 / 605 at 1.5M, 806 / 779 at 2.2M
    const int cap_g = sm_grid_cap(side && sort ? (n > 875000 ? 3 : 2) : 6);
    const int grid = cap_g < (n + 255) / 256 ? cap_g : (n + 255) / 256;
    GS_LAUNCHED(1);
    return launch_k(rows_kernel, grid, 256, 0, st, (uint32_t)n, ws.rec[eye], ws.rect[eye], ws.vis[eye], ws.cams, eye,
                    ws.prim, ws.info[eye], ws.spans[eye], cap, &ctr->n_rows[eye], ws.more[eye], ws.more_cap[eye],
                    &ctr->n_more[eye], &ctr->status, tile_mask ? b.mask_clip : nullptr, tiles_x, tiles_y, tile_mask ? b.mask_sat : nullptr,
                    tile_mask ? b.bits : nullptr);
  };
  if (!side && (err = launch_rows(s)) != cudaSuccess) return err;
  const uint32_t chunk = kBinWarps * ws.bin_warp_surfels;
  const BinCounts bc{&ctr->n_vis[eye], &ctr->n_band[eye], &ctr->n_entries[eye], &ctr->n_items[eye],
                     &ctr->n_chunks[eye], &ctr->n_table[eye], chunk, (uint32_t)ntiles};
  // 2. depth order (the low 32 bits of the packed key; stable, so ties keep id
  // order): the dominant order filtered, or a sort
  const KeySource src{ws.zkey[eye], bits, order == kOrderUnion ? ws.vis[1 - eye] : nullptr};
  if (sort && (err = radix_hist(src, (uint32_t)n, rs, bc, s)) != cudaSuccess) return err;
  if (side) {  // the spans beside the sort's passes: started with the histogram they held the first pass back 20 us
    if ((err = cudaEventRecord(rows->fork, s)) != cudaSuccess) return err;
    if ((err = cudaStreamWaitEvent(rows->stream, rows->fork, 0)) != cudaSuccess) return err;
  }
  err = sort ? radix_passes(src, b.dkey, b.dval, &ctr->n_vis[eye], (uint32_t)n, rs, s)
             : scan_launch(ReuseLoad{ws.bin[0].dval[0], &ctr->n_vis[0], (uint32_t)n, bits},
                           ReuseApply{ws.bin[0].dval[0], b.dval[0], bc}, (const uint32_t *)nullptr, (uint32_t)n,
                           b.scan_tiles, b.scan_ticket, &ctr->status, s);
  if (err != cudaSuccess) return err;
  if (side) {
    if ((err = launch_rows(rows->stream)) != cudaSuccess) return err;
    if ((err = cudaEventRecord(rows->join, rows->stream)) != cudaSuccess) return err;
    if ((err = cudaStreamWaitEvent(s, rows->join, 0)) != cudaSuccess) return err;
  }
  // 3. per sub-chunk: depth-ordered lists of every tile row's ranges
  ListArgs la;
  la.ids = b.dval[0];
  la.n_vis = &ctr->n_vis[eye];
  la.n_max = (uint32_t)n;
  la.info = ws.info[eye];
  la.spans = ws.spans[eye];
  la.more = ws.more[eye];
  la.span_cap = cap;
  la.clip = tile_mask ? b.mask_clip : nullptr;
  la.tiles_x = tiles_x;
  la.tiles_y = tiles_y;
  la.warp_surfels = ws.bin_warp_surfels;
  la.pool = b.row_pool;
  la.pool_cap = ws.row_pool_cap[eye];
  la.pool_n = &ctr->n_entries[eye];
  la.n_band = &ctr->n_band[eye];
  la.lists = b.row_lists;
  la.status = &ctr->status;
  launch_k(row_list_kernel, ws.bin_nch * kBinWarps, kBinThreads, list_smem_bytes(tiles_y), s, la);
  GS_LAUNCHED(1);
  BinArgs a;
  a.n_vis = &ctr->n_vis[eye];
  a.n_max = (uint32_t)n;
  a.ids = b.dval[0];
  a.pool = b.row_pool;
  a.lists = b.row_lists;
  a.mask = tile_mask;
  a.tiles_x = tiles_x;
  a.tiles_y = tiles_y;
  a.warp_surfels = ws.bin_warp_surfels;
  a.nch = ws.bin_nch;
  a.table = b.bin_table;
  a.offs = b.bin_offs;
  a.cap = cap;
  a.ival = b.ival;
  a.ikey = ws.keep_intermediates ? b.ikey : nullptr;
  a.cnt_bin = ws.keep_intermediates ? ws.cnt_bin : nullptr;
  if (a.cnt_bin && n > 0 && (err = cudaMemsetAsync(a.cnt_bin, 0, sizeof(uint32_t) * (size_t)n, s)) != cudaSuccess)
    return err;
  // 4. per-warp counts per (tile, chunk)
  launch_k(bin_count_kernel, dim3(ws.bin_nch, (unsigned)((tiles_y + kCountRows - 1) / kCountRows)), kBinThreads,
           count_smem_bytes(tiles_x), s, a);
  GS_LAUNCHED(1);
  // 5. tile-major scan over the chunks that hold binned surfels: where every
  // (tile, chunk) run starts, every tile's range and, for a mask, the tile list
  err = scan_launch(BinTableLoad{b.bin_table, &ctr->n_chunks[eye], &ctr->n_vis[eye], ws.bin_nch, chunk},
                    BinOffsetApply{b.bin_offs, &ctr->n_chunks[eye], ws.bin_nch, &ctr->n_inst[eye], &ctr->n_sort[eye],
                                   cap, &ctr->status, b.ranges, ntiles, tile_mask, b.items, &ctr->n_items[eye]},
                    &ctr->n_table[eye], (uint32_t)ntiles * ws.bin_nch, b.scan_tiles, b.scan_ticket, &ctr->status, s);
  if (err != cudaSuccess) return err;
  // 6. every surfel id to its slot
  launch_k(bin_place_kernel, dim3(ws.bin_nch, (unsigned)tiles_y), kBinThreads, place_smem_bytes(tiles_x), s, a);
  GS_LAUNCHED(1);
  return cudaGetLastError();
}

}  // namespace gs
