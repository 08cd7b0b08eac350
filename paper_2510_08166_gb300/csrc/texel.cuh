// Texel addressing and pixel walks shared by the screen passes and the float chain.
#pragma once

#include <cuda_runtime.h>

#include "jt_internal.cuh"

namespace jt {
namespace {

__device__ __forceinline__ int floor_mod_i(int a, int w) {
  int r = a % w;
  return r < 0 ? r + w : r;
}

// Locates the view of global tile `tile` (views are few and sorted by tile_begin).
__device__ __forceinline__ int view_of_tile(const ViewSet& vs, uint32_t tile) {
  int vi = 0;
#pragma unroll 1
  for (int i = 1; i < vs.n; ++i)
    if (tile >= vs.v[i].tile_begin) vi = i;
  return vi;
}

// Loads up to 4 pixels of row y starting at column x (n = pixels present, 0..4).
__device__ __forceinline__ int load_px4(const View& V, int y, int x, float u[4], float v[4], uint32_t t[4],
                                        uint32_t m[4]) {
  const int n = (y < V.height && x < V.width) ? min(4, V.width - x) : 0;
  const uint32_t p0 = (uint32_t)y * (uint32_t)V.width + (uint32_t)x;
  if (n == 4 && (V.width & 3) == 0) {
    const uint32_t lq = p0 >> 2;
    const float4 a = __ldg(V.uv + 2 * lq), b = __ldg(V.uv + 2 * lq + 1);
    u[0] = a.x; v[0] = a.y; u[1] = a.z; v[1] = a.w;
    u[2] = b.x; v[2] = b.y; u[3] = b.z; v[3] = b.w;
    const uint2 tt = __ldg(reinterpret_cast<const uint2*>(V.tex) + lq);
    t[0] = tt.x & 0xFFFF; t[1] = tt.x >> 16; t[2] = tt.y & 0xFFFF; t[3] = tt.y >> 16;
    const uint32_t mm = __ldg(reinterpret_cast<const uint32_t*>(V.mip) + lq);
    m[0] = mm & 255; m[1] = (mm >> 8) & 255; m[2] = (mm >> 16) & 255; m[3] = mm >> 24;
  } else {
    const float* uvs = reinterpret_cast<const float*>(V.uv);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i < n) {
        u[i] = __ldg(uvs + 2 * (p0 + i));
        v[i] = __ldg(uvs + 2 * (p0 + i) + 1);
        t[i] = __ldg(V.tex + p0 + i);
        m[i] = __ldg(V.mip + p0 + i);
      } else {
        u[i] = v[i] = 0.f;
        t[i] = JT_EMPTY_TEXTURE;
        m[i] = 0;
      }
    }
  }
  return n;
}

// Iterates the (view, row, column) of this thread's quads over the CTA's tiles:
// f(V, y, x) for every row segment a warp owns; warps take rows w, w + nwarps, ...
template <typename F>
__device__ __forceinline__ void for_each_quad(const ViewSet& vs, F&& f) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
#pragma unroll 1
  for (uint32_t tile = blockIdx.x; tile < vs.total_tiles; tile += gridDim.x) {
    const int vi = view_of_tile(vs, tile);
    const View& V = vs.v[vi];
    const uint32_t lt = tile - V.tile_begin;
    const int x = (int)(lt % V.tiles_x) * kTileW + lane * 4;
    const int y0 = (int)(lt / V.tiles_x) * vs.tile_h;
#pragma unroll 1
    for (int r = warp; r < vs.tile_h; r += nwarps) f(V, y0 + r, x);
  }
}

// ---------------------------------------------------------------------------------------
// Texel addressing
// ---------------------------------------------------------------------------------------
// floor(x) for |x| < 2^22 by one round-down add: t = x + 1.5 * 2^23 rounded down is exactly
// floor(x) + 1.5 * 2^23 (the sum lies in [2^23, 2^24), where floats are the integers), so
// t - 1.5 * 2^23 is floor(x) as a float, and the bit pattern of t is that of 1.5 * 2^23
// (a multiple of 2^22) plus floor(x): masked by w - 1 (w a power of two below 2^22) it is
// floor(x) floor-mod w. Pixels outside that range take the general path (conversion
// instructions, which saturate, and a division).
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23

// A pixel's level, from its PixRec (two vector loads; all fields zero for keys outside the
// table, so every address derived from them stays in range).
struct PixL {
  uint32_t gid_base;
  float wf, hf;
  uint32_t masks;  // (w - 1) | (h - 1) << 16
  uint32_t mcus_x;
  uint32_t shift;
  uint32_t info;   // units | kPixJpeg | kPixCoef | kPixPow2
  uint32_t wh;     // w | h << 16
};

__device__ __forceinline__ PixL pix_level(const TexLookup& tl, uint32_t tm) {
  const uint32_t key = min(tm & 0xFFFFu, tl.map_ntex) * kPixLevels + min(tm >> 16, (uint32_t)JT_MAX_LEVELS);
  const uint4 r0 = __ldg(tl.pix + 2 * key), r1 = __ldg(tl.pix + 2 * key + 1);
  PixL P;
  P.gid_base = r0.x;
  P.wf = __uint_as_float(r0.y);
  P.hf = __uint_as_float(r0.z);
  P.masks = r0.w;
  P.mcus_x = r1.x;
  P.shift = r1.y;
  P.info = r1.z;
  P.wh = r1.w;
  return P;
}

// The range test of the fast path is of the round-down sums' exponents: [2^23, 2^24).
__device__ __forceinline__ bool in_range(float tx, float ty) {
  return ((__float_as_uint(tx) ^ 0x4B000000u) | (__float_as_uint(ty) ^ 0x4B000000u)) < 0x00800000u;
}

// Repeat wrap of the fast path: by the record's masks, for levels known to have power-of-two
// sides (kWrapPow2) or with the others left to the general path (kWrapChecked), or by a
// remainder for sides of any size (kWrapAny).
enum Wrap { kWrapChecked, kWrapPow2, kWrapAny };

template <Wrap WRAP>
__device__ __forceinline__ bool wrap_covers(const PixL& P) {
  return WRAP != kWrapChecked || (P.info & kPixPow2) != 0;
}

// floor-mod of the integer in t = n + kMagic by a side (a float), the largest result in m. For
// any side: the quotient (two units in the last place), rounded down, is at most one off for |n| < 2^22, so
// its remainder, exact by the fused step, needs one side added or taken away. Outside that
// range the result is any number, at most m.
template <Wrap WRAP>
__device__ __forceinline__ int wrap_texel(float t, float side, uint32_t m) {
  if (WRAP != kWrapAny) return __float_as_int(t) & (int)m;
  const float n = __fsub_rn(t, kMagic);
  const float q = __fsub_rn(__fadd_rd(__fdividef(n, side), kMagic), kMagic);
  int r = __float_as_int(__fadd_rn(__fmaf_rn(-q, side, n), kMagic)) - 0x4B400000;
  const int w = (int)m + 1;
  r += r < 0 ? w : 0;
  r -= r >= w ? w : 0;
  return (int)min((uint32_t)r, m);
}

template <Wrap WRAP>
__device__ __forceinline__ int next_texel(int x, uint32_t m) {
  return WRAP == kWrapAny ? ((uint32_t)x == m ? 0 : x + 1) : (x + 1) & (int)m;
}

// Bilinear taps on the fast path: |u w|, |v h| < 2^22 and a level that WRAP covers (returns
// false otherwise; every tap is then still inside the level, so loads made from it stay in
// range, but the caller must redo the pixel on the general path). Columns xa, xb = xa + 1,
// rows ya, yb = ya + 1 (repeat wrap), fractions fx, fy.
template <Wrap WRAP = kWrapChecked>
__device__ __forceinline__ bool taps_fast(const PixL& P, float u, float v, int& xa, int& xb, int& ya, int& yb,
                                          float& fx, float& fy) {
  const float xs = __fsub_rn(__fmul_rn(u, P.wf), 0.5f), ys = __fsub_rn(__fmul_rn(v, P.hf), 0.5f);
  const float tx = __fadd_rd(xs, kMagic), ty = __fadd_rd(ys, kMagic);
  fx = __fsub_rn(xs, __fsub_rn(tx, kMagic));
  fy = __fsub_rn(ys, __fsub_rn(ty, kMagic));
  const uint32_t wm = P.masks & 0xFFFFu, hm = P.masks >> 16;
  xa = wrap_texel<WRAP>(tx, P.wf, wm);
  ya = wrap_texel<WRAP>(ty, P.hf, hm);
  xb = next_texel<WRAP>(xa, wm);
  yb = next_texel<WRAP>(ya, hm);
  return wrap_covers<WRAP>(P) && in_range(tx, ty);
}

// Nearest texel on the fast path (same conditions as taps_fast).
template <Wrap WRAP = kWrapChecked>
__device__ __forceinline__ bool nearest_fast(const PixL& P, float u, float v, int& x, int& y) {
  const float tx = __fadd_rd(__fmul_rn(u, P.wf), kMagic), ty = __fadd_rd(__fmul_rn(v, P.hf), kMagic);
  x = wrap_texel<WRAP>(tx, P.wf, P.masks & 0xFFFFu);
  y = wrap_texel<WRAP>(ty, P.hf, P.masks >> 16);
  return wrap_covers<WRAP>(P) && in_range(tx, ty);
}

// The same taps for any level and coordinate (conversion instructions, floor-mod by
// division): the general path.
__device__ __forceinline__ void taps_any(const PixL& P, float u, float v, int& xa, int& xb, int& ya, int& yb,
                                         float& fx, float& fy) {
  const int w = (int)(P.wh & 0xFFFFu), h = (int)(P.wh >> 16);
  const float xs = __fsub_rn(__fmul_rn(u, P.wf), 0.5f), ys = __fsub_rn(__fmul_rn(v, P.hf), 0.5f);
  fx = __fsub_rn(xs, floorf(xs));
  fy = __fsub_rn(ys, floorf(ys));
  xa = floor_mod_i(__float2int_rd(xs), w);  // cvt.rmi saturates out-of-range values
  ya = floor_mod_i(__float2int_rd(ys), h);
  xb = xa + 1 == w ? 0 : xa + 1;
  yb = ya + 1 == h ? 0 : ya + 1;
}

__device__ __forceinline__ void nearest_any(const PixL& P, float u, float v, int& x, int& y) {
  x = floor_mod_i(__float2int_rd(__fmul_rn(u, P.wf)), (int)(P.wh & 0xFFFFu));
  y = floor_mod_i(__float2int_rd(__fmul_rn(v, P.hf)), (int)(P.wh >> 16));
}

}  // namespace
}  // namespace jt
