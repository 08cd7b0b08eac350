// Scene rasteriser: writes the G-buffer (uv, texture id, mip level) of a procedural scene, a
// perspective ground plane of 2 m texture cells under projective screen-space quads. It
// stands in for the renderer's geometry pass (paper Sec. 4) so that a whole frame, geometry
// included, runs on the GPU.
//
// Every arithmetic step is an explicitly rounded fp32 operation (no contraction) in a fixed
// order, and levels are chosen by exact power-of-two thresholds on the squared footprint, so
// the result is reproducible on any IEEE fp32 implementation of the same steps.
//
// One CTA per tile of up to 256 x 8 pixels: the CTA first lists, in drawing order, the quads whose
// pixel bounds meet the tile (ordered compaction by warp ballots) and copies the edges of the
// last ones (the ones that win) to shared memory, then each warp takes a row, 32 pixels at a
// time: the last listed quad containing it, else the ground, else sky. The kernel is bound by its
// instructions (it reads only the quad list and writes 11 bytes a pixel); what was taken out
// of a pixel: the 64-bit remainder (three 32-bit ones by a precomputed reciprocal), the
// level's loop (the exponent of the footprint), most conversions, where the camera does not roll the ray divisions
// (one per pixel row and its two edges, instead of five per pixel), most of the tiles'
// listing, the hash of a cell the lane's pixel before lay in, and the tests of quads that do not
// reach the 32 pixels. 4K, 200 quads, the whole call: 165 -> 108 us, with the last two 102 us (four
// CTAs per SM at 64 registers; 105 at 74, 118 with five).
#include <cuda_runtime.h>

#include <cmath>

#include "jt_internal.cuh"

namespace jt {
namespace {

constexpr int kThreads = 32 * kRasterTileY;
constexpr int kStagedQuads = 32;

__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }

// SplitMix64 (Steele, Lea, Flood 2014): the ground cells' texture and uv offset come from
// two steps of it keyed by the cell coordinates.
__device__ __forceinline__ uint64_t splitmix_next(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ uint64_t cell_hash(uint64_t seed, uint64_t a, uint64_t b) {
  uint64_t s = seed ^ (a * 0xD1B54A32D192ED03ull) ^ (b * 0x8CB92BA72F3D8DD7ull);
  splitmix_next(s);
  return splitmix_next(s);
}

// hash mod ntex (ntex < 2^16, mod_m = floor(2^32 / ntex), or 2^32 - 1 for 1) in three steps of
// 32 bits: the reciprocal's quotient is at most one short.
__device__ __forceinline__ uint32_t mod32(uint32_t n, uint32_t d, uint32_t m) {
  const uint32_t r = n - __umulhi(n, m) * d;
  return min(r, r - d);
}
__device__ __forceinline__ uint32_t mod_ntex(uint64_t h, const RasterArgs& a) {
  const uint32_t d = (uint32_t)a.ntex, lo = (uint32_t)h;
  uint32_t r = mod32((uint32_t)(h >> 32), d, a.mod_m);
  r = mod32((r << 16) | (lo >> 16), d, a.mod_m);
  return mod32((r << 16) | (lo & 0xFFFFu), d, a.mod_m);
}

// Camera rays: the parts of a pixel column and of a pixel row, and the ground hit where they
// meet; uv = world (x, z) / 2. LEVEL: rot[3] is zero (the camera does not roll), so a row's rays
// have one dy and one ray parameter (the product with zero and its addition change nothing).
struct RayCol {
  float x0, x1, x2;  // rot[0], rot[3], rot[6] times sx
};
struct RayRow {
  float y0, y1, y2;  // rot[1], rot[4], rot[7] times sy
  float t;           // LEVEL: the ray parameter, negative when the row sees no ground
};

__device__ __forceinline__ bool ray_t(const RasterArgs& a, float dy, float& t) {
  if (!(dy < -1e-9f)) return false;
  t = fdiv(-a.cam[1], dy);
  return !(t > a.max_t);
}

__device__ __forceinline__ RayCol ray_col(const RasterArgs& a, float px) {
  const float sx = fmul(fsub(fmul(px, a.ax), 1.0f), a.tan_x);
  return RayCol{fmul(a.rot[0], sx), fmul(a.rot[3], sx), fmul(a.rot[6], sx)};
}

template <bool LEVEL>
__device__ __forceinline__ RayRow ray_row(const RasterArgs& a, float py, bool& hit) {
  const float sy = fmul(fsub(1.0f, fmul(py, a.ay)), a.tan_y);
  RayRow r{fmul(a.rot[1], sy), fmul(a.rot[4], sy), fmul(a.rot[7], sy), 0.f};
  hit = !LEVEL || ray_t(a, fsub(r.y1, a.rot[5]), r.t);
  return r;
}

template <bool LEVEL>
__device__ __forceinline__ bool ground(const RasterArgs& a, const RayCol& c, const RayRow& r, float& u, float& v) {
  const float dx = fsub(fadd(c.x0, r.y0), a.rot[2]), dz = fsub(fadd(c.x2, r.y2), a.rot[8]);
  float t = r.t;
  if (!LEVEL && !ray_t(a, fsub(fadd(c.x1, r.y1), a.rot[5]), t)) return false;
  u = fmul(fadd(a.cam[0], fmul(t, dx)), 0.5f);
  v = fmul(fadd(a.cam[2], fmul(t, dz)), 0.5f);
  return true;
}

// floor(log2(sqrt(r2)) + 1/2) clamped to [0, L-1]: the count of k >= 1 with r2 >= 2^(2k-1), from
// the exponent of r2 (0 for NaN).
__device__ __forceinline__ int level_of(float r2, int L) {
  const int m = ((__float_as_int(r2) >> 23) - 126) >> 1;
  return r2 > 0.0f ? min(max(m, 0), L - 1) : 0;
}

// A texture's level-0 sides as floats and its level count.
struct TexSize {
  float w, h;
  int levels;
};
__device__ __forceinline__ TexSize tex_size(const RasterArgs& a, int t) {
  const float4 r = __ldg(a.sizes + t);
  return TexSize{r.x, r.y, __float_as_int(r.z)};
}

__device__ __forceinline__ float footprint(float u0, float v0, float u1, float v1, const TexSize& z) {
  const float du = fmul(fsub(u1, u0), z.w), dv = fmul(fsub(v1, v0), z.h);
  return fadd(fmul(du, du), fmul(dv, dv));
}

__device__ __forceinline__ void quad_uv(const SceneQuad& q, float x, float y, float& u, float& v) {
  float s = fadd(fadd(fmul(q.h[0], x), fmul(q.h[1], y)), q.h[2]);
  float t = fadd(fadd(fmul(q.h[3], x), fmul(q.h[4], y)), q.h[5]);
  const float w = fadd(fadd(fmul(q.h[6], x), fmul(q.h[7], y)), q.h[8]);
  s = fdiv(s, w);
  t = fdiv(t, w);
  u = fadd(q.ou, fmul(q.rep, fsub(fmul(q.cs, s), fmul(q.sn, t))));
  v = fadd(q.ov, fmul(q.rep, fadd(fmul(q.sn, s), fmul(q.cs, t))));
}

// Conversions without the special-function unit: floor of |x| < 2^22 from the low bits of
// x + 1.5 * 2^23 rounded down, and integers below 2^23 as the low bits of 2^23 + n.
__device__ __forceinline__ uint32_t floor_bits(float x) { return __float_as_uint(__fadd_rd(x, 12582912.0f)); }
__device__ __forceinline__ bool small_floor(uint32_t b) { return (b ^ 0x4B000000u) < 0x00800000u; }
__device__ __forceinline__ int64_t floor_i64(float x, uint32_t b) {
  return small_floor(b) ? (int64_t)((int)b - 0x4B400000) : (int64_t)floorf(x);
}
__device__ __forceinline__ float small_float(uint32_t n) { return fsub(__uint_as_float(0x4B000000u | n), 8388608.0f); }

// A 2 m cell of the ground: its texture and uv offset, and the floors (as floor_bits) it was made
// for, both zero, which no floor_bits are, for a cell too far out to be told by them.
struct Cell {
  uint32_t bu, bv;
  int tex;
  float ou, ov;
  TexSize size;
};
__device__ __forceinline__ Cell cell_of(const RasterArgs& a, float u, float v, uint32_t bu, uint32_t bv) {
  const uint64_t hs = cell_hash(a.cell_seed, (uint64_t)floor_i64(u, bu), (uint64_t)floor_i64(v, bv));
  Cell c;
  const bool known = small_floor(bu) && small_floor(bv);
  c.bu = known ? bu : 0u;
  c.bv = known ? bv : 0u;
  c.tex = (int)mod_ntex(hs, a);
  c.ou = fmul(small_float((uint32_t)(hs >> 16) & 0xFFFFu), 1.0f / 65536.0f);
  c.ov = fmul(small_float((uint32_t)(hs >> 32) & 0xFFFFu), 1.0f / 65536.0f);
  c.size = a.use_mips ? tex_size(a, c.tex) : TexSize{};
  return c;
}

// A quad's containment test: four edges (corner, edge vector) and the pixel bounds.
struct QuadEdges {
  float4 e[4];
  int4 b;
};

__device__ __forceinline__ QuadEdges edges_of(const SceneQuad& q) {
  QuadEdges k;
#pragma unroll
  for (int i = 0; i < 4; ++i) k.e[i] = make_float4(q.cx[i], q.cy[i], q.ex[i], q.ey[i]);
  k.b = make_int4(q.x0, q.y0, q.x1, q.y1);
  return k;
}

__device__ __forceinline__ bool inside(const QuadEdges& k, int x, int y, float qx, float qy) {
  bool in = x >= k.b.x && x <= k.b.z && y >= k.b.y && y <= k.b.w;
#pragma unroll
  for (int i = 0; i < 4; ++i) in &= !(fsub(fmul(k.e[i].z, fsub(qy, k.e[i].y)), fmul(k.e[i].w, fsub(qx, k.e[i].x))) < 0.0f);
  return in;
}

template <bool LEVEL>
__global__ void __launch_bounds__(kThreads, 4) k_raster(const __grid_constant__ RasterArgs a) {
  __shared__ uint16_t list[kMaxSceneQuads];
  __shared__ __align__(16) QuadEdges staged[kStagedQuads];
  __shared__ uint32_t warp_count[kThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx0 = blockIdx.x * a.tile_x, ty0 = blockIdx.y * kRasterTileY;
  const int tx1 = min(tx0 + a.tile_x, a.width) - 1, ty1 = min(ty0 + kRasterTileY, a.height) - 1;

  // the quads that may cover the tile, in drawing order
  uint32_t count = 0;
#pragma unroll 1
  for (int base = 0; base < a.nquads; base += kThreads) {
    const int n = base + tid;
    bool meets = false;
    if (n < a.nquads) {
      const SceneQuad& q = a.quads[n];
      meets = q.x0 <= tx1 && q.x1 >= tx0 && q.y0 <= ty1 && q.y1 >= ty0;
    }
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, meets);
    if (lane == 0) warp_count[warp] = __popc(b);
    __syncthreads();
    uint32_t before = count, total = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
      before += w < warp ? warp_count[w] : 0u;
      total += warp_count[w];
    }
    if (meets) list[before + __popc(b & ((1u << lane) - 1u))] = (uint16_t)n;
    count += total;
    __syncthreads();
  }
  // edges of the last ones: entry i of the list at staged[count - 1 - i]
  if (tid < min((int)count, kStagedQuads)) staged[tid] = edges_of(a.quads[list[count - 1 - tid]]);
  __syncthreads();

  const int y = ty0 + warp;
  if (y >= a.height) return;
  const float fy = fadd((float)y, 0.5f), qy = fmul(fy, a.ky);
  bool hr, h0, h1;  // the rays of the row, of its upper and of its lower edge
  const RayRow r = ray_row<LEVEL>(a, fy, hr), r0 = ray_row<LEVEL>(a, (float)y, h0),
               r1 = ray_row<LEVEL>(a, fadd((float)y, 1.0f), h1);
  // lane i's staged quad: the columns it may cover in this row (none past the list)
  const int4 mine = lane < (int)count ? staged[lane].b : make_int4(1, 1, 0, 0);
  const bool in_row = y >= mine.y && y <= mine.w;
  Cell cell{};
#pragma unroll 1
  for (int xc = tx0; xc <= tx1; xc += 32) {
    uint32_t near = __ballot_sync(0xFFFFFFFFu, in_row && mine.x <= xc + 31 && mine.z >= xc);
    const int x = xc + lane;
    if (x > tx1) break;
    const float xf = a.width < (1 << 23) ? small_float((uint32_t)x) : (float)x;
    const float fx = fadd(xf, 0.5f), qx = fsub(fmul(fx, a.kx), a.shift);
    int hit = -1;
    while (near) {  // the last quad drawn wins
      const int i = __ffs(near) - 1;
      near &= near - 1;
      if (inside(staged[i], x, y, qx, qy)) {
        hit = list[count - 1 - i];
        break;
      }
    }
    if (hit < 0 && count > kStagedQuads) {
#pragma unroll 1
      for (int i = kStagedQuads; i < (int)count; ++i) {
        const int n = list[count - 1 - i];
        if (inside(edges_of(a.quads[n]), x, y, qx, qy)) {
          hit = n;
          break;
        }
      }
    }
    float u = 0.f, v = 0.f;
    int t = JT_EMPTY_TEXTURE, lvl = 0;
    if (hit >= 0) {
      const SceneQuad& q = a.quads[hit];
      t = q.tex;
      quad_uv(q, qx, qy, u, v);
      if (a.use_mips) {
        const TexSize z = tex_size(a, t);
        const float hx = fmul(a.kx, 0.5f), hy = fmul(a.ky, 0.5f);
        float u0, v0, u1, v1, u2, v2, u3, v3;
        quad_uv(q, fsub(qx, hx), qy, u0, v0);
        quad_uv(q, fadd(qx, hx), qy, u1, v1);
        quad_uv(q, qx, fsub(qy, hy), u2, v2);
        quad_uv(q, qx, fadd(qy, hy), u3, v3);
        const float rx = footprint(u0, v0, u1, v1, z);
        const float ry = footprint(u2, v2, u3, v3, z);
        lvl = level_of(fmaxf(rx, ry), z.levels);
      }
    } else {
      const RayCol c = ray_col(a, fx);
      if (hr && ground<LEVEL>(a, c, r, u, v)) {
        const uint32_t bu = floor_bits(u), bv = floor_bits(v);
        if (bu != cell.bu || bv != cell.bv) cell = cell_of(a, u, v, bu, bv);
        t = cell.tex;
        u = fadd(u, cell.ou);
        v = fadd(v, cell.ov);
        if (a.use_mips) {
          const TexSize z = cell.size;
          float u0, v0, u1, v1, u2, v2, u3, v3;
          const bool ok = ground<LEVEL>(a, ray_col(a, xf), r, u0, v0) &&
                          ground<LEVEL>(a, ray_col(a, fadd(xf, 1.0f)), r, u1, v1) &&
                          h0 && ground<LEVEL>(a, c, r0, u2, v2) && h1 && ground<LEVEL>(a, c, r1, u3, v3);
          if (!ok) {
            lvl = z.levels - 1;
          } else {
            const float rx = footprint(u0, v0, u1, v1, z);
            const float ry = footprint(u2, v2, u3, v3, z);
            lvl = level_of(fmaxf(rx, ry), z.levels);
          }
        }
      }
    }
    const size_t o = (size_t)y * a.width + x;
    a.uv[o] = make_float2(u, v);
    a.tex[o] = (uint16_t)t;
    a.mip[o] = (uint8_t)lvl;
  }
}

}  // namespace

void launch_raster(const RasterArgs& a, cudaStream_t s) {
  const dim3 grid((a.width + a.tile_x - 1) / a.tile_x, (a.height + kRasterTileY - 1) / kRasterTileY);
  // a finite column factor times zero adds nothing to dy: the camera does not roll
  if (a.rot[3] == 0.0f && std::isfinite(a.ax * (a.width + 1.0f)) && std::isfinite(a.tan_x) &&
      std::isfinite((a.ax * (a.width + 1.0f) - 1.0f) * a.tan_x))
    k_raster<true><<<grid, kThreads, 0, s>>>(a);
  else
    k_raster<false><<<grid, kThreads, 0, s>>>(a);
}

}  // namespace jt
