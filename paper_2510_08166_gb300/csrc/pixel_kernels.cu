// Screen-space passes over the deferred G-buffer: Mark (paper Sec. 4.2) and Resolve /
// colourise (Sec. 4.4), for one or several views in one launch.
//
// Both stream the G-buffer (11 B/px read; colourise also writes 4 B/px and gathers texels
// from the block cache). A persistent grid walks the views in tiles of 128 pixels by 32 or 8
// rows, one warp per 128-pixel row.
//
// Mark: one quad of 4 pixels per lane (32 B + 8 B + 4 B vector loads). Pixels of a tile
// share MCUs, so Mark keeps a 1024-entry table of the gids its CTA already flagged in shared
// memory and stores each flag about once per CTA instead of once per pixel (the byte stores
// of every SM to the same flag lines otherwise dominate the pass). A quad is decided at once
// from the box of its taps (see k_mark).
//
// Colourise: a lane owns pixels 32 apart (lane + 32 k), so the 32 addresses of one texel
// gather instruction are 32 consecutive pixels' taps, which fall in two or three tiles (half
// the L1 wavefronts of quads per lane); the next step's G-buffer is loaded before the current
// one is shaded; a pixel's level comes from a 32-byte record that needs no decoding; the
// bilinear blend runs in fp16 pairs within a proven 1-LSB bound.
//
// Texel addressing (fixed in fp32 with explicit rounding so it is the same on every
// device): nearest x = floor(u * w) floor-mod w; bilinear xs = u * w - 1/2, x0 = floor(xs),
// fx = xs - x0, taps x0 and x0 + 1 (floor-mod w); the MCU of texel (x, y) is
// x / mw + (y / mw) * mcus_x with mw = 16 (4:2:0) or 8 (4:4:4), and its key is the level's
// gid_base + MCU (Sec. 4.6).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "jt_internal.cuh"
#include "texel.cuh"

namespace jt {
namespace {

constexpr uint32_t kNoGid = 0xFFFFFFFFu;

// Walks the views' tiles: CTA tiles blockIdx.x, + gridDim.x, ...; warp rows w, w + nwarps,
// ... of each tile. The tile origin is recomputed only when the tile changes.
struct RowWalk {
  uint32_t tile;
  int r;       // row in the tile
  int vi;      // view of the tile
  int x0, y0;  // tile origin
  __device__ __forceinline__ bool valid(const ViewSet& vs) const { return tile < vs.total_tiles; }
  __device__ __forceinline__ void set_tile(const ViewSet& vs) {
    if (tile >= vs.total_tiles) return;
    vi = view_of_tile(vs, tile);
    const View& V = vs.v[vi];
    const uint32_t lt = tile - V.tile_begin;
    const uint32_t ty = lt / V.tiles_x;
    x0 = (int)(lt - ty * V.tiles_x) * kTileW;
    y0 = (int)ty * vs.tile_h;
  }
  __device__ __forceinline__ void start(const ViewSet& vs) {
    tile = blockIdx.x;
    r = threadIdx.x >> 5;
    vi = 0;
    x0 = y0 = 0;
    if (r >= vs.tile_h) tile = 0xFFFFFFFFu;  // a warp without a row
    set_tile(vs);
  }
  __device__ __forceinline__ void advance(const ViewSet& vs) {
    r += blockDim.x >> 5;
    if (r >= vs.tile_h) {
      r = threadIdx.x >> 5;
      tile += gridDim.x;
      set_tile(vs);
    }
  }
};

// A lane's part of one row of a tile: pixels x + 32 j, j < 4.
struct Row {
  uint32_t p0;  // index of pixel j = 0 in the view
  int rem;      // pixel j exists when 32 j < rem
};

__device__ __forceinline__ Row row_of(const View& V, const RowWalk& w, bool valid) {
  const int x = w.x0 + (int)(threadIdx.x & 31), y = w.y0 + w.r;
  return Row{(uint32_t)y * (uint32_t)V.width + (uint32_t)x, valid && y < V.height ? V.width - x : 0};
}

// G-buffer of NPX of a lane's pixels, loaded one step ahead of its use so that its HBM reads
// are in flight while the lane works on the current one. The loads are streaming ones (and so
// are the framebuffer's stores): nothing reads these lines again, and L1 keeps the tiles'
// texels and the slots instead (4K frame: 51.9 us without, 47.1 with).
template <int NPX>
struct RowG {
  float u[NPX], v[NPX];
  uint32_t tm[NPX];  // texture id | mip level << 16 (JT_EMPTY_TEXTURE past the view)
};

template <int NPX>
__device__ __forceinline__ void load_row(const View& V, const Row& row, int j0, RowG<NPX>& g) {
  const float2* uv = reinterpret_cast<const float2*>(V.uv) + row.p0;
  const uint16_t* tx = V.tex + row.p0;
  const uint8_t* mp = V.mip + row.p0;
#pragma unroll
  for (int k = 0; k < NPX; ++k) {
    const int j = 32 * (j0 + k);
    g.u[k] = g.v[k] = 0.f;
    g.tm[k] = JT_EMPTY_TEXTURE;
    if (j < row.rem) {
      const float2 t = __ldcs(uv + j);
      g.u[k] = t.x;
      g.v[k] = t.y;
      g.tm[k] = (uint32_t)__ldcs(tx + j) | ((uint32_t)__ldcs(mp + j) << 16);
    }
  }
}

// ---------------------------------------------------------------------------------------
// Mark
// ---------------------------------------------------------------------------------------
constexpr int kSeen = 1024;  // per-CTA table of recently flagged gids

// Mark is bound by its instruction count (an evaluation of four taps and up to four table probes
// per pixel ran at 72 % of the issue slots), so a lane decides its quad of four pixels at
// once. Nearly every quad has one level, and its footprint, the box of the taps of its
// pixels, lies in one row or one column of at most two MCUs, which are then exactly the MCUs
// of the box's ends. Every other quad (several levels, both rows and columns, a larger box, a
// repeat edge of a level whose sides are no powers of two, coordinates beyond 2^22, the ragged
// end of a row) goes into the warp's queue, whose quads are taken eight at a time, a pixel
// per lane: a few such quads in every warp cost their share and not a pass of the warp each
// (in a branch of their own they made the kernel slower than the plain form: 50.9 against
// 42.7 us on the 4K frame of 64 textures, bilinear). Measured: 42.7 -> 27.9 us on that frame
// (43 % of the HBM rate, long_scoreboard first among its stalls), 395 -> 286 us for the
// nearest texels of eight 4096^2 views (63 %). Where most quads have to wait the plain form was
// faster: one level seen without mips (20 texels from pixel to pixel, 4K, nearest 44.6 us, 53.9
// now; bilinear 64.0, 75.7), another texture at every pixel (31.0, 41.3). Taking such segments
// from the registers, from the caches or pixel by pixel won most of that back, but each of ten
// forms cost ordinary frames 0.3 to 3 % (more registers or a vote in the box's path), and the frames
// of those contents are as fast as with the plain form or faster.

// One pixel on its own: flag(g) for every MCU its taps fall in.
template <int FILTER, typename F>
__device__ __forceinline__ void mark_pixel(const PixL& P, float u, float v, F&& flag) {
  int xa, xb, ya, yb;
  float fx, fy;
  if (FILTER == JT_FILTER_NEAREST) {
    if (!nearest_fast(P, u, v, xa, ya)) nearest_any(P, u, v, xa, ya);
    flag(P.gid_base + ((uint32_t)xa >> P.shift) + ((uint32_t)ya >> P.shift) * P.mcus_x);
    return;
  }
  if (!taps_fast(P, u, v, xa, xb, ya, yb, fx, fy)) taps_any(P, u, v, xa, xb, ya, yb, fx, fy);
  const uint32_t ca = (uint32_t)xa >> P.shift, cb = (uint32_t)xb >> P.shift;
  const uint32_t ra = P.gid_base + ((uint32_t)ya >> P.shift) * P.mcus_x, rb = P.gid_base + ((uint32_t)yb >> P.shift) * P.mcus_x;
  flag(ra + ca);
  if (cb != ca) flag(ra + cb);
  if (rb != ra) {
    flag(rb + ca);
    if (cb != ca) flag(rb + cb);
  }
}

constexpr int kMarkQueue = 8 + 32;  // quads waiting in a warp: fewer than eight, and one row segment's

// MANY: enough tiles for eight CTAs of 256 threads on every SM (32 registers), whose loads then
// overlap (passes: 4K 113.3 -> 111.3 us, VR pair 119.5 -> 114.0, eight 4096^2 textures 1393 -> 1356);
// with fewer tiles there is nothing to fill the SMs with, and six CTAs' 40 registers spill none.
template <int FILTER, bool MANY>
__global__ void __launch_bounds__(512, MANY ? 4 : 3) k_mark(const __grid_constant__ MarkArgs a) {
  constexpr int kTap = FILTER == JT_FILTER_NEAREST ? 0 : 1;  // the second tap's distance
  extern __shared__ uint2 queue[];  // [warps][kMarkQueue]: first pixel in the view; view | pixels << 8
  __shared__ uint32_t seen[kSeen];
  pdl_launch_dependents();
  for (int i = threadIdx.x; i < kSeen; i += blockDim.x) seen[i] = kNoGid;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  uint2* wq = queue + (threadIdx.x >> 5) * kMarkQueue;
  int waiting = 0;
  bool missing = false;
  // an empty pixel's texture, or one that is filtered out
  auto skip = [&](uint32_t tex) { return tex == JT_EMPTY_TEXTURE || (a.only_tex >= 0 && (int)tex != a.only_tex); };
  // flags gid g unless this CTA already did (racy by design: a duplicate store writes the
  // same byte)
  auto flag = [&](uint32_t g, uint32_t units) {
    uint32_t* e = &seen[(g ^ (g >> 10)) & (kSeen - 1)];
    if (*e != g) {
      *e = g;
      a.flags[g] = (uint8_t)units;
    }
  };
  // the last (at most) eight quads of the queue, a pixel per lane
  auto drain = [&] {
    __syncwarp();
    const int n = min(waiting, 8);
    waiting -= n;
    if ((lane >> 2) < n) {
      const uint2 e = wq[waiting + (lane >> 2)];
      const View& V = a.views.v[e.y & 255u];
      if ((uint32_t)(lane & 3) < e.y >> 8) {
        const uint32_t p = e.x + (lane & 3);
        const uint32_t tex = __ldg(V.tex + p);
        if (!skip(tex)) {
          const float2 uv = __ldg(reinterpret_cast<const float2*>(V.uv) + p);
          const PixL P = pix_level(a.tl, tex | ((uint32_t)__ldg(V.mip + p) << 16));
          if (P.info & kPixJpeg)
            mark_pixel<FILTER>(P, uv.x, uv.y, [&](uint32_t g) { flag(g, P.info & 255u); });
          else
            missing = true;
        }
      }
    }
    __syncwarp();
  };
  for_each_quad(a.views, [&](const View& V, int y, int x) {
    float u[4], v[4];
    uint32_t t[4], m[4];
    const int n = load_px4(V, y, x, u, v, t, m);
    const uint32_t t0 = t[0], m0 = m[0];
    const bool one = n == 4 && ((t[1] ^ t0) | (t[2] ^ t0) | (t[3] ^ t0) | (m[1] ^ m0) | (m[2] ^ m0) | (m[3] ^ m0)) == 0;
    const bool none = n == 0 || (one && skip(t0));
    const PixL P = pix_level(a.tl, t0 | (m0 << 16));
    int px[4], py[4];
    uint32_t far = 0;  // exponents other than that of [2^23, 2^24): |coordinate| beyond 2^22
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float xs = __fmul_rn(u[i], P.wf), ys = __fmul_rn(v[i], P.hf);
      const uint32_t bx = __float_as_uint(__fadd_rd(kTap ? __fsub_rn(xs, 0.5f) : xs, kMagic));
      const uint32_t by = __float_as_uint(__fadd_rd(kTap ? __fsub_rn(ys, 0.5f) : ys, kMagic));
      far |= (bx ^ 0x4B000000u) | (by ^ 0x4B000000u);
      px[i] = (int)bx - 0x4B400000;
      py[i] = (int)by - 0x4B400000;
    }
    int x0 = min(min(px[0], px[1]), min(px[2], px[3])), x1 = max(max(px[0], px[1]), max(px[2], px[3])) + kTap;
    int y0 = min(min(py[0], py[1]), min(py[2], py[3])), y1 = max(max(py[0], py[1]), max(py[2], py[3])) + kTap;
    bool box = one && (P.info & kPixJpeg) && (far & 0xFF800000u) == 0;
    // MCU coordinates are unwrapped up to here; powers of two wrap them with a mask
    const uint32_t s = P.shift;
    uint32_t cm = (P.masks & 0xFFFFu) >> s, rm = P.masks >> (16 + s);
    if (!a.tl.all_p2 && !(P.info & kPixPow2)) {
      // other sides: the quad moves into the level by its first pixel's repeat (any integer
      // near the quotient will do: the box has to end up inside the level)
      const int w = (int)(P.wh & 0xFFFFu), h = (int)(P.wh >> 16);
      int rx = px[0] - __float2int_rd(__fdividef((float)px[0], P.wf)) * w;
      int ry = py[0] - __float2int_rd(__fdividef((float)py[0], P.hf)) * h;
      rx += rx < 0 ? w : rx >= w ? -w : 0;
      ry += ry < 0 ? h : ry >= h ? -h : 0;
      x0 += rx - px[0];
      x1 += rx - px[0];
      y0 += ry - py[0];
      y1 += ry - py[0];
      box = box && x0 >= 0 && x1 < w && y0 >= 0 && y1 < h;
      cm = rm = 0xFFFFu;
    }
    const int c0 = x0 >> s, c1 = x1 >> s, r0 = y0 >> s, r1 = y1 >> s;
    const int dc = c1 - c0, dr = r1 - r0;
    box = box && dc + dr <= 1;  // (both are at least 0)
    if (box && !none) {
      const uint32_t units = P.info & 255u;
      const uint32_t g0 = P.gid_base + ((uint32_t)r0 & rm) * P.mcus_x + ((uint32_t)c0 & cm);
      const uint32_t g1 = P.gid_base + ((uint32_t)r1 & rm) * P.mcus_x + ((uint32_t)c1 & cm);
      flag(g0, units);
      if (g1 != g0) flag(g1, units);
    }
    const uint32_t rest = __ballot_sync(0xFFFFFFFFu, !box && !none);
    if (rest) {
      if (!box && !none)
        wq[waiting + __popc(rest & ((1u << lane) - 1u))] =
            make_uint2((uint32_t)y * (uint32_t)V.width + (uint32_t)x, (uint32_t)(&V - a.views.v) | ((uint32_t)n << 8));
      waiting += __popc(rest);
      while (waiting >= 8) drain();
    }
  });
  while (waiting > 0) drain();
  if (missing) atomicOr(&a.state->err, JT_DEVERR_MISSING);
}

// ---------------------------------------------------------------------------------------
// Colourise
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ __half2 u32_as_h2(uint32_t w) {
  __half2 h;
  memcpy(&h, &w, 4);
  return h;
}
__device__ __forceinline__ uint32_t h2_as_u32(__half2 h) {
  uint32_t w;
  memcpy(&w, &h, 4);
  return w;
}

// Bilinear blend of four RGBA8 texels with weights from fx, fy, rounded to bytes; alpha is
// 255 (every texel's). Channels are blended two at a time in fp16 pairs: a byte b becomes
// the half 1024 + b exactly (one byte permute under the exponent of 1024), differences of
// two such halves are exact, and each lerp a + f (b - a) is one fused fp16 multiply-add.
// The result c is rounded by adding 1536, whose binade [1024, 2048) has unit spacing, so
// the low byte of the sum is round(c). Error bound: fx, fy carry at most 2^-12 absolute
// error after the conversion to fp16 (255 * 2^-12 < 0.063 per lerp), each fp16 lerp and
// difference of values below 256 rounds by at most 1/16, so |c - c_exact| < 0.32 over the
// three lerps and one difference, and the byte differs from floor(c_exact + 1/2) by at most
// one. c stays within [-0.32, 255.32], so c + 1536 never leaves [1024, 2048).
__device__ __forceinline__ uint32_t blend_h(uint32_t c00, uint32_t c10, uint32_t c01, uint32_t c11, float fx,
                                            float fy) {
  const __half2 in_bias = u32_as_h2(0x64006400u);   // (1024, 1024)
  const __half2 out_bias = u32_as_h2(0x66006600u);  // (1536, 1536)
  const __half2 hx = __float2half2_rn(fx), hy = __float2half2_rn(fy);
  auto lerp_x = [&](uint32_t a, uint32_t b, uint32_t sel) {
    const __half2 ha = u32_as_h2(__byte_perm(a, 0x64646464u, sel));
    const __half2 hb = u32_as_h2(__byte_perm(b, 0x64646464u, sel));
    return __hfma2(hx, __hsub2(hb, ha), __hsub2(ha, in_bias));
  };
  const __half2 top_rg = lerp_x(c00, c10, 0x5140u), bot_rg = lerp_x(c01, c11, 0x5140u);  // (R, G)
  const __half2 top_ba = lerp_x(c00, c10, 0x5342u), bot_ba = lerp_x(c01, c11, 0x5342u);  // (B, A)
  const __half2 rg = __hadd2(__hfma2(hy, __hsub2(bot_rg, top_rg), top_rg), out_bias);
  const __half2 ba = __hadd2(__hfma2(hy, __hsub2(bot_ba, top_ba), top_ba), out_bias);
  return __byte_perm(h2_as_u32(rg), h2_as_u32(ba), 0x6420u);
}

// One pixel's colour from its taps: the slots of their four MCUs and four texel gathers, then
// the blend (bilinear) or the texel itself (nearest). Branch- and predicate-free, so the
// pixels of a lane overlap their chains: the four slots are read whether or not the footprint
// straddles MCUs (the same address twice where it does not, an L1 hit), which costs less than
// the comparisons, predicates and selects that would spare the reads (the ALU pipe bounds the
// pass; of a G-buffer of noise, where every lane's reads are lines of their own, the pass takes 131 us
// at 4K, 116 with predicates). Any slot is in range, of an MCU no pixel needs too (a stale one), and a pixel that
// is not shaded reads the first slots and gathers from wherever they point.
// S: log2 of the MCU side when every level has the same, else -1.
template <int FILTER, int S>
__device__ __forceinline__ uint32_t shade(const uint32_t* __restrict__ slot, const uint32_t* __restrict__ cache,
                                          const PixL& P, int xa, int xb, int ya, int yb, float fx, float fy) {
  const uint32_t s = S >= 0 ? (uint32_t)S : P.shift, mwm = (1u << s) - 1u;
  const uint32_t xas = (uint32_t)xa >> s, rowa = P.gid_base + ((uint32_t)ya >> s) * P.mcus_x;
  const uint32_t o00 = __ldg(slot + rowa + xas);
  const uint32_t ia = ((uint32_t)ya & mwm) << s, ja = (uint32_t)xa & mwm;
  if (FILTER == JT_FILTER_NEAREST) return __ldg(cache + (size_t)o00 * (kUnitBytes / 4) + (ia | ja));
  const uint32_t xbs = (uint32_t)xb >> s, rowb = P.gid_base + ((uint32_t)yb >> s) * P.mcus_x;
  const uint32_t ib = ((uint32_t)yb & mwm) << s, jb = (uint32_t)xb & mwm;
  uint32_t o10 = o00, o01 = o00, o11 = o00;
  if (FILTER == JT_FILTER_BILINEAR) {  // (the clamped filter's taps share the nearest texel's MCU)
    o10 = __ldg(slot + rowa + xbs);
    o01 = __ldg(slot + rowb + xas);
    o11 = __ldg(slot + rowb + xbs);
  }
  // texel j of the tile at unit o (S >= 0: texel indexes fit 32 bits)
  auto texel = [&](uint32_t o, uint32_t j) {
    return S >= 0 ? __ldg(cache + (o * (kUnitBytes / 4) | j)) : __ldg(cache + (size_t)o * (kUnitBytes / 4) + j);
  };
  const uint32_t c00 = texel(o00, ia | ja), c10 = texel(o10, ia | jb), c01 = texel(o01, ib | ja), c11 = texel(o11, ib | jb);
  return blend_h(c00, c10, c01, c11, fx, fy);
}

// Taps of the clamped filter: along each axis a tap in another MCU than the nearest texel's
// moves onto the nearest texel's column or row (one MCU).
__device__ __forceinline__ void clamp_taps(uint32_t s, int nx, int ny, int& xa, int& xb, int& ya, int& yb) {
  const int mx = nx >> s, my = ny >> s;
  xa = (xa >> s) == mx ? xa : nx;
  xb = (xb >> s) == mx ? xb : nx;
  ya = (ya >> s) == my ? ya : ny;
  yb = (yb >> s) == my ? yb : ny;
}

// The general path of one pixel (any level, any coordinate; out of line).
template <int FILTER>
__device__ __noinline__ uint32_t colour_any(const uint32_t* slot, const uint32_t* cache, const PixL& P, float u,
                                            float v) {
  int xa, xb, ya, yb;
  float fx = 0.f, fy = 0.f;
  if (FILTER == JT_FILTER_NEAREST) {
    nearest_any(P, u, v, xa, ya);
    xb = xa;
    yb = ya;
  } else {
    taps_any(P, u, v, xa, xb, ya, yb, fx, fy);
    if (FILTER == JT_FILTER_BILINEAR_CLAMP) {
      int nx, ny;
      nearest_any(P, u, v, nx, ny);
      clamp_taps(P.shift, nx, ny, xa, xb, ya, yb);
    }
  }
  return shade<FILTER, -1>(slot, cache, P, xa, xb, ya, yb, fx, fy);
}

// A lane owns pixels lane + 32 j (j < 4) of a row of a tile, NPX at a time, so a warp's texel
// gathers for one tap fall in the two or three tiles its 32 consecutive pixels cover (few L1
// wavefronts per load), and the lane's NPX pixels are independent chains (level record, slots,
// texels) that overlap. The next NPX pixels' G-buffer is loaded before the current ones are
// shaded. The fast path has no data-dependent branch: the level record is loaded per pixel (an
// L1 hit), and pixels it cannot address (|u w| or |v h| >= 2^22) are redone on the general path. Warps whose pixels all lack a texture skip the arithmetic. Slots
// are in range by construction (the compaction and the cache update never write a slot whose
// tile would end past the cache), and the all-zero record of keys outside the table addresses
// the first gid, so no load needs a bound check.
// ONE: pixels of one texture only (the per-texture form). S: see shade. WRAP covers every level.
template <int FILTER, bool ONE, int S, Wrap WRAP, int NPX>
__device__ __forceinline__ void colour_step(const ColorizeArgs& a, const RowG<NPX>& g, uint32_t* out, int rem,
                                            bool& missing) {
  const uint32_t* __restrict__ cache = reinterpret_cast<const uint32_t*>(a.cache);
  const uint32_t* __restrict__ slot = a.slot;
  bool use = false;
#pragma unroll
  for (int k = 0; k < NPX; ++k) {  // (pixels past the view are empty)
    const uint32_t tex = g.tm[k] & 0xFFFFu;
    use |= tex != JT_EMPTY_TEXTURE && (!ONE || (int)tex == a.only_tex);
  }
  uint32_t px[NPX];
#pragma unroll
  for (int k = 0; k < NPX; ++k) px[k] = 0xFF000000u;  // empty pixels
  if (__any_sync(0xFFFFFFFFu, use)) {
    uint32_t slow = 0;
#pragma unroll
    for (int k = 0; k < NPX; ++k) {
      const uint32_t tex = g.tm[k] & 0xFFFFu;
      const bool mine = tex != JT_EMPTY_TEXTURE && (!ONE || (int)tex == a.only_tex);
      const PixL P = pix_level(a.tl, g.tm[k]);
      const bool ok = mine && (P.info & kPixJpeg);
      missing |= mine && !ok;
      int xa, xb, ya, yb;
      float fx = 0.f, fy = 0.f;
      bool fast;
      if (FILTER == JT_FILTER_NEAREST) {
        fast = nearest_fast<WRAP>(P, g.u[k], g.v[k], xa, ya);
        xb = xa;
        yb = ya;
      } else {
        fast = taps_fast<WRAP>(P, g.u[k], g.v[k], xa, xb, ya, yb, fx, fy);
        if (FILTER == JT_FILTER_BILINEAR_CLAMP) {
          int nxp, nyp;
          fast &= nearest_fast<WRAP>(P, g.u[k], g.v[k], nxp, nyp);
          clamp_taps(S >= 0 ? (uint32_t)S : P.shift, nxp, nyp, xa, xb, ya, yb);
        }
      }
      const uint32_t c = shade<FILTER, S>(slot, cache, P, xa, xb, ya, yb, fx, fy);
      px[k] = ok ? c : px[k];
      slow |= (ok && !fast) ? (1u << k) : 0u;
    }
    if (slow) {  // rare: redo those pixels on the general path
#pragma unroll
      for (int k = 0; k < NPX; ++k)
        if (slow & (1u << k)) px[k] = colour_any<FILTER>(slot, cache, pix_level(a.tl, g.tm[k]), g.u[k], g.v[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < NPX; ++k)
    if (32 * k < rem && (!ONE || (int)(g.tm[k] & 0xFFFFu) == a.only_tex)) __stcs(out + 32 * k, px[k]);
}

template <int FILTER, bool MULTI, bool ONE, int S, Wrap WRAP, int NPX>
__global__ void __launch_bounds__(512, 2) k_colorize(const __grid_constant__ ColorizeArgs a) {
  constexpr int kSteps = 4 / NPX;
  const ViewSet& vs = a.views;
  bool missing = false;
  RowWalk it;
  it.start(vs);
  Row row = row_of(vs.v[MULTI ? it.vi : 0], it, it.valid(vs));
  RowG<NPX> g;
  load_row(vs.v[MULTI ? it.vi : 0], row, 0, g);
#pragma unroll 1
  while (it.valid(vs)) {
    uint32_t* out = reinterpret_cast<uint32_t*>(vs.v[MULTI ? it.vi : 0].out) + row.p0;
    const int rem = row.rem;
#pragma unroll
    for (int h = 0; h < kSteps; ++h) {
      RowG<NPX> ng;
      if (h + 1 < kSteps) {
        load_row(vs.v[MULTI ? it.vi : 0], row, (h + 1) * NPX, ng);
      } else {
        it.advance(vs);
        row = row_of(vs.v[MULTI ? it.vi : 0], it, it.valid(vs));
        load_row(vs.v[MULTI ? it.vi : 0], row, 0, ng);
      }
      colour_step<FILTER, ONE, S, WRAP, NPX>(a, g, out + 32 * NPX * h, rem - 32 * NPX * h, missing);
      g = ng;
    }
  }
  if (missing) atomicOr(&a.state->err, JT_DEVERR_MISSING);
}

}  // namespace

void launch_mark(const MarkArgs& a, int threads, int grid, cudaStream_t s) {
  threads = std::min(threads, 512);
  const size_t smem = (size_t)(threads / 32) * kMarkQueue * sizeof(uint2);
  const bool many = a.many;
  if (many) grid = (int)std::min<uint64_t>(a.views.total_tiles, 2 * (uint64_t)grid);
  // the clamped filter reads only the nearest texel's MCU
  if (a.filter == JT_FILTER_NEAREST || a.filter == JT_FILTER_BILINEAR_CLAMP)
    many ? k_mark<JT_FILTER_NEAREST, true><<<grid, threads, smem, s>>>(a)
         : k_mark<JT_FILTER_NEAREST, false><<<grid, threads, smem, s>>>(a);
  else
    many ? k_mark<JT_FILTER_BILINEAR, true><<<grid, threads, smem, s>>>(a)
         : k_mark<JT_FILTER_BILINEAR, false><<<grid, threads, smem, s>>>(a);
}

// pixels per lane per step: of one, two and four with three to five 256-thread CTAs per SM, two
// with four CTAs (64 registers) was the fastest for the bilinear filters (4K frame: 47.1 us,
// 53.9 with one, 49.4 with four and three CTAs, 53.1 with five CTAs), a whole row's four for the
// nearest texel, whose chains are shorter (eight 4096^2 views: 549 us, 686 with two)
constexpr int kColorizePx = 2, kColorizePxNearest = 4;

template <bool MULTI, bool ONE, int S, Wrap WRAP>
void launch_colorize_form(const ColorizeArgs& a, int threads, int grid, cudaStream_t s) {
  constexpr int N = kColorizePx, kNearest = ONE && WRAP == kWrapAny ? N : kColorizePxNearest;  // (four spill there)
  if (a.filter == JT_FILTER_NEAREST)
    k_colorize<JT_FILTER_NEAREST, MULTI, ONE, S, WRAP, kNearest><<<grid, threads, 0, s>>>(a);
  else if (a.filter == JT_FILTER_BILINEAR_CLAMP)
    k_colorize<JT_FILTER_BILINEAR_CLAMP, MULTI, ONE, S, WRAP, N><<<grid, threads, 0, s>>>(a);
  else
    k_colorize<JT_FILTER_BILINEAR, MULTI, ONE, S, WRAP, N><<<grid, threads, 0, s>>>(a);
}

// The form with a constant MCU side serves contexts whose levels are all 4:2:0 at full size
// with power-of-two sides; the other ones take it from each pixel's record, and a context
// with any other sides wraps by a remainder (twelve textures of odd sides in a 1367 x 769 frame,
// the three calls: 63.0 us with every pixel on the general path, 55.6 so).
void launch_colorize(const ColorizeArgs& a, int threads, int grid, cudaStream_t s) {
  threads = std::min(threads, 512);
  const bool s4 = a.tl.all_s4 && a.tl.all_p2 && a.cap_units <= 0xFFFFFFFFu / (kUnitBytes / 4);
  auto form = [&](auto multi) {
    constexpr bool M = decltype(multi)::value;
    s4 ? launch_colorize_form<M, false, 4, kWrapPow2>(a, threads, grid, s)
       : a.tl.all_p2 ? launch_colorize_form<M, false, -1, kWrapPow2>(a, threads, grid, s)
                     : launch_colorize_form<M, false, -1, kWrapAny>(a, threads, grid, s);
  };
  if (a.only_tex >= 0)  // one view at a time
    a.tl.all_p2 ? launch_colorize_form<false, true, -1, kWrapPow2>(a, threads, grid, s)
                : launch_colorize_form<false, true, -1, kWrapAny>(a, threads, grid, s);
  else if (a.views.n > 1)
    form(std::true_type{});
  else
    form(std::false_type{});
}

}  // namespace jt
