// piko_direct.cuh -- triangles of a few pixels, rasterized by the pass that
// would only have binned them.
//
// The count pass of AssignBin holds a triangle's snapped vertices in
// registers.  For a triangle whose box is a few pixels, binning it (a
// rectangle, a list entry, a second gather of its indices and vertices) costs
// several times the work of rasterizing it, so the pass
// takes its samples right there: a 64-bit atomic minimum per covered sample on
// one key per pixel in global memory (depth << 32 | triangle; the minimum is
// the same in any order).  Larger triangles are binned as before, and the
// Process stage starts each tile from these keys.  A triangle that covers no
// sample, most of a half-pixel micropolygon grid, ends here.
//
// A lane walks its own box: first for coverage only, into a mask of at most 32
// samples, then the covered samples one by one for their depths.  The pass is
// bound by instruction issue, not by the atomics (the same time without them:
// 102 against 108 us for 5.3M micropolygons) nor by its gathers.  Handing the
// covered samples of a warp out to consecutive lanes, as the Process stage
// does for its lists, cost as much in staging as it saved in idle lanes.
#pragma once

#include "piko_tile.cuh"

namespace piko {

constexpr int DIRECT_MAX_PX = 32;  // samples of a box, a bit of the coverage mask each

// Sets n keys to KEY_EMPTY, the whole grid taking part (keys 16-byte aligned).
__device__ __forceinline__ void clear_keys(unsigned long long* keys, size_t n) {
  const size_t step = (size_t)gridDim.x * blockDim.x, first = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  ulonglong2* k2 = reinterpret_cast<ulonglong2*>(keys);
  for (size_t i = first; i < n / 2; i += step) k2[i] = make_ulonglong2(KEY_EMPTY, KEY_EMPTY);
  if ((n & 1) && first == 0) keys[n - 1] = KEY_EMPTY;
}

// Scenes worth it: triangles small on average, at most this many pixels of the
// framebuffer for each.  The lines lie where the route stops paying against binning
// every triangle (us on the direct route / binned, Lambert mesh at 16 x 16 bins):
//   1920x1080   9 pixels a triangle 57 / 81, 10 67 / 84, 11 84 / 87, 12 98 / 90
//   1280x720    9 41 / 46, 10 42 / 47, 11 53 / 49
//   900x600     7 36 / 39, 9 41 / 41, 10 50 / 42
//   640x400     6 25 / 27, 7 25 / 27, 8 35 / 27
//   320x240     4 21 / 23, 5 (sphere) 27 / 24, 7 31 / 23
// as beyond them most tiles hold triangles of both kinds and both routes' launches
// have work; small frames are bound by these launches.  Soups of separate triangles
// share no vertices, and their sizes differ more (power law / equal sizes of three
// times the framebuffer in all, direct / binned):
//   1920x1080   2.5 290 / 311 and 219 / 231, 3 270 / 270 and 215 / 219, 3.5 252 / 229 and 213 / 198
//   560x420     2.5 62 / 67 and 53 / 58, 3 63 / 62 and 55 / 55, 3.5 59 / 56 and 55 / 52
//   320x240     1.5 49 / 50 and 35 / 39, 2 46 / 44 and 39 / 35, 3 47 / 43 and 41 / 35
// (Soups of one-pixel triangles that cover a quarter of the framebuffer would gain up
// to 4 pixels a triangle and beyond, 63 / 89 at 3.9, but counts do not tell them.)
// In a batch the launches are shared and all tiles are one launch's: meshes pay up to
// 10 pixels a triangle (16 heightfields of 600x600: 9 197 / 221, 11 235 / 234) and soups
// to 4 in frames of any size (three of 300x300: 3.9 42 / 49 and 62 / 62; 64 uneven
// scenes 1,663 with the line at 4 and 1,677 at 3).
inline bool direct_scene(long long T, long long V, long long px, bool batch) {
  const bool mesh = V < 2 * T;
  int line;
  if (batch) line = mesh ? 10 : 4;
  else if (px < 1 << 17) line = mesh ? 4 : 2;
  else if (px < 3 << 18) line = mesh ? 7 : 3;
  else line = mesh ? 10 : 3;
  return V > 0 && line * T >= px;
}

// Whether some scene of at most max_t triangles and max_v vertices is one: a
// mesh, which takes fewer triangles than a soup, of as many as there may be.
inline bool direct_scene_within(long long max_t, long long max_v, long long px) {
  return max_v > 0 && max_t > 0 && direct_scene(max_t, 1, px, false);
}

// A triangle of at most 128 pixels a side (its snapped extents below 2^15, so
// that areas and edge functions are exact in 32 bits) whose box, clipped to
// the screen, has at most max_px samples.
__device__ __forceinline__ bool direct_small(int extent_x, int extent_y, int px0, int px1, int py0, int py1, int max_px) {
  return max(extent_x, extent_y) < 32768 && max(px1 - px0, py1 - py0) < 32 &&
         (px1 - px0 + 1) * (py1 - py0 + 1) <= max_px;
}

// Rasterizes one direct_small triangle into keys (the framebuffer's, W wide);
// false for a triangle without area.  t: the triangle of its keys.
//
// Edges 2->0 and 0->1 as seen from vertex 0, negated when the triangle is
// wound the other way (which leaves the vertices, and so the depths, in
// place); the third edge function is A - w1 - w2.
__device__ __forceinline__ bool direct_triangle(int4 p0, int4 p1, int4 p2, unsigned t, int px0, int px1, int py0, int py1,
                                                int W, unsigned long long* __restrict__ keys) {
  int dx1 = p0.x - p2.x, dy1 = p0.y - p2.y, dx2 = p1.x - p0.x, dy2 = p1.y - p0.y;
  int A = dx1 * dy2 - dx2 * dy1;
  if (A == 0) return false;
  if (A < 0) {
    A = -A;
    dx1 = -dx1; dy1 = -dy1; dx2 = -dx2; dy2 = -dy2;
  }
  const int dx0 = -(dx1 + dx2), dy0 = -(dy1 + dy2);
  const int u = 256 * px0 + 128 - p0.x, v = 256 * py0 + 128 - p0.y;
  const int w1 = dx1 * v - dy1 * u, w2 = dx2 * v - dy2 * u;
  const int sx0 = -256 * dy0, sx1 = -256 * dy1, sx2 = -256 * dy2;
  const int sy0 = 256 * dx0, sy1 = 256 * dx1, sy2 = 256 * dx2;
  // less the fill-rule bias: covered iff all three are >= 0
  int r0 = A - w1 - w2 - 1 + top_left(dx0, dy0), r1 = w1 - 1 + top_left(dx1, dy1), r2 = w2 - 1 + top_left(dx2, dy2);
  const int bw = px1 - px0 + 1, n = bw * (py1 - py0 + 1);
  // a sample's sign bit (set: not covered) is shifted in from below, so that
  // sample j of the n ends at bit n - 1 - j
  unsigned out = 0u;
  for (int j = 0; j < n; j += bw) {
    int a0 = r0, a1 = r1, a2 = r2;
    for (int x = 0; x < bw; ++x) {
      out = __funnelshift_l((unsigned)(a0 | a1 | a2), out, 1);
      a0 += sx0; a1 += sx1; a2 += sx2;
    }
    r0 += sy0; r1 += sy1; r2 += sy2;
  }
  unsigned mask = ~out & (0xFFFFFFFFu >> (32 - n));
  if (mask == 0u) return true;
  const int d1 = p1.z - p0.z, d2 = p2.z - p0.z;
  const float rA = approx_rcp((float)A), k1 = rA * (float)d1, k2 = rA * (float)d2;
  // the remainder fits 32 bits (see DepthSetup)
  const bool fast = A < (1 << 27) && abs(d1) + abs(d2) < (1 << 22);
  // 65536 / bw to within 2 ulp, floored, plus one: (j * M) >> 16 = floor(j / bw) for every j < 32
  const unsigned M = __float2uint_rz(__fdividef(65536.0f, (float)bw)) + 1u;
  keys += (size_t)py0 * W + px0;
  do {
    const int bit = 31 - __clz(mask);
    mask ^= 1u << bit;
    const int j = n - 1 - bit;
    const int ry = (int)(((unsigned)j * M) >> 16), rx = j - ry * bw;
    // covered: f1, f2 in [0, A] < 2^30, exact in wrapping 32-bit arithmetic
    const int f1 = w1 + rx * sx1 + ry * sy1, f2 = w2 + rx * sx2 + ry * sy2;
    int q = __float2int_rd(__fmaf_rn((float)f1, k1, (float)f2 * k2));
    if (fast) {
      int r = (int)((unsigned)f1 * (unsigned)d1 + (unsigned)f2 * (unsigned)d2 - (unsigned)q * (unsigned)A);
      if ((unsigned)r >= (unsigned)A) {  // the estimate is a few units off at most
        for (int it = 0; r < 0 && it < DIV_FIX_LIMIT; ++it) { --q; r += A; }
        for (int it = 0; r >= A && it < DIV_FIX_LIMIT; ++it) { ++q; r -= A; }
      }
    } else {
      long long r = (long long)f1 * d1 + (long long)f2 * d2 - (long long)q * A;
      for (int it = 0; r < 0 && it < DIV_FIX_LIMIT; ++it) { --q; r += A; }
      for (int it = 0; r >= A && it < DIV_FIX_LIMIT; ++it) { ++q; r -= A; }
    }
    atomicMin(keys + (ry * W + rx), (unsigned long long)(unsigned)(p0.z + q) << 32 | t);
  } while (mask != 0u);
  return true;
}

// ---------------------------------------------------------------- shading
// Colour and key of pixel (x, y), whose winner (indices id, key k) was
// rasterized directly: its snapped extents are below 2^15, so areas and edge
// functions are exact in 32 bits.
// CLIP: a winner whose vertices the vertex stage rejected was clipped.
template <bool PERSP, bool CLIP>
__device__ __forceinline__ void shade_direct_pixel(const TileScene& p, int3 id, int x, int y, size_t o) {
  const int4 p0 = __ldg(p.vtx + id.x), p1 = __ldg(p.vtx + id.y), p2 = __ldg(p.vtx + id.z);
  if (CLIP && !(p0.w & p1.w & p2.w)) {
    shade_winner<PERSP, true>(p, id, x, y, o);
    return;
  }
  // edges 2->0 and 0->1 and the area, all negative for a triangle wound the
  // other way: the signs cancel in the weights of vertices 1 and 2
  const int dx1 = p0.x - p2.x, dy1 = p0.y - p2.y, dx2 = p1.x - p0.x, dy2 = p1.y - p0.y;
  const int u = 256 * x + 128 - p0.x, v = 256 * y + 128 - p0.y;
  const float rA = __fdividef(1.0f, (float)(dx1 * dy2 - dx2 * dy1));
  float b1 = (float)(dx1 * v - dy1 * u) * rA, b2 = (float)(dx2 * v - dy2 * u) * rA, b0 = 1.0f - b1 - b2;
  if (PERSP) perspective_bary(b0, b1, b2, __ldg(p.invw + id.x), __ldg(p.invw + id.y), __ldg(p.invw + id.z));
  if (p.mode == PIKO_SHADE_LAMBERT)
    shade_lambert(p, id.x, id.y, id.z, b0, b1, b2, o);
  else
    shade_vertices(p, id.x, id.y, id.z, b0, b1, b2, o);
}

// A tile whose winners are all directly rasterized: an 8 x 4 block of pixels
// per warp and step (called by every thread of the CTA; no barrier).
constexpr int SHADE_W = 8, SHADE_H = 4;

// (x, y) may lie outside the framebuffer.
__device__ __forceinline__ unsigned long long direct_key(const TileScene& p, int x, int y) {
  return x < p.g.W && y < p.g.H ? __ldcg(p.dkeys + (size_t)y * p.g.W + x) : KEY_EMPTY;
}

template <bool PERSP, bool CLIP>
__device__ __forceinline__ void shade_direct_block(const TileScene& p, unsigned long long k, int3 id, int x, int y) {
  if (x >= p.g.W || y >= p.g.H) return;
  const size_t o = (size_t)y * p.g.W + x;
  p.key_out[o] = k;
  if (k == KEY_EMPTY)
    write_empty(p, o);
  else
    shade_direct_pixel<PERSP, CLIP>(p, id, x, y, o);
}

template <bool PERSP, bool CLIP>
__device__ __forceinline__ void shade_direct_tile(const TileScene& p, int tile) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int ty = tile / p.g.nbx, tx = tile - ty * p.g.nbx;
  const int per_row = 1 << (p.g.bshift_x - 3), blocks = per_row << (p.g.bshift_y - 2);  // bins are at least 8 x 8
  const int x0 = (tx << p.g.bshift_x) + (lane & (SHADE_W - 1)), y0 = (ty << p.g.bshift_y) + lane / SHADE_W;
  auto at = [&](int b, int& x, int& y) {
    const int by = b >> (p.g.bshift_x - 3), bx = b & (per_row - 1);
    x = x0 + bx * SHADE_W;
    y = b < blocks ? y0 + by * SHADE_H : p.g.H;
  };
  // the key of the block after next and the indices of the next are loaded before a block is shaded
  int x, y, xn, yn, xnn, ynn;
  at(warp, x, y);
  at(warp + nwarps, xn, yn);
  unsigned long long k = direct_key(p, x, y), kn = direct_key(p, xn, yn);
  int3 id = make_int3(0, 0, 0), idn = id;
  if (k != KEY_EMPTY) id = tri_indices(p.tris, (unsigned)k);
  for (int b = warp; b < blocks; b += nwarps) {
    if (kn != KEY_EMPTY) idn = tri_indices(p.tris, (unsigned)kn);
    at(b + 2 * nwarps, xnn, ynn);
    const unsigned long long knn = direct_key(p, xnn, ynn);
    shade_direct_block<PERSP, CLIP>(p, k, id, x, y);
    k = kn; x = xn; y = yn; id = idn;
    kn = knn; xn = xnn; yn = ynn;
  }
}

}  // namespace piko
