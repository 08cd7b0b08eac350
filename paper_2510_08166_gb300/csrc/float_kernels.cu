// Float chain (differentiable colourise, not in the paper): bilinear taps over the texels of
// coefficient textures, F = sum_k w_k colour(texel_k), each data unit's texels f = A c A^T (A the
// orthonormal DCT-III basis, a row per position), and its adjoint: dL/dc = A^T g A with g the
// texels' gradients, the w dL/dF of the pixels whose taps fall on them.
//
// The pixel -> MCU map is inverted first, in the same way for both passes:
//   k_float_count    per pixel, +1 to the count of each distinct MCU its taps touch (an entry);
//   k_float_sums, k_float_offsets   one scan over the counts: each MCU's entry offset, the
//                    needed MCUs' work list and slots (an MCU is needed when its count is not
//                    0), and the counts turned into fill cursors;
//   k_float_fill     the same visits again, each writing its 16-byte entry: the pixel, the
//                    first texel, which taps of each axis are in the MCU, fx, fy;
//   k_float_forward  a warp takes pairs of MCUs one after the other: transforms the pair in shared
//                    memory, then a lane per entry adds its taps' sums into the pixel's value
//                    (a pixel with one entry stores it);
//   k_float_backward the same pairs (every MCU is written once): the entries' weighted terms added
//                    into the pair's gradients in shared memory, then the adjoint transforms.
// The order of the sums (atomics, the entries' places) is the only non-determinism.
//
// A lane transforms whole rows and columns in registers (even and odd halves: 32 fused
// multiply-adds per eight values), three of each per pair; with an output per lane and scalar
// shared reads a transform took 480 warp instructions and 82 % of the shared-memory pipe.
// What then bounds the gathers is the round trips of each pair (ranges, coefficients, entries,
// pixels): 1.5 KB per MCU at 5 K cycles of latency. So a pair's ranges come for the whole share of
// the warp at once, and the next pair's coefficients (asynchronous copies, which leave the
// first-level cache out), entries and gradients are under way while this one is worked on.
// Measured on sixteen 2048^2 textures under a 1920x1080 plane (244 K MCUs needed, 2.3 M entries,
// 375 MB of coefficients each way: 55 us): k_float_forward 170 -> 104 us, k_float_backward
// 198 -> 131 us, the inversion of both passes 275 -> 104 us; both passes 626 -> 370 us. Tried and slower:
// each entry straight from the coefficients (341 us backward: 48 16-byte shared reads per entry),
// pairs on a persistent grid (248 us forward), loads through the first-level cache.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "jt_internal.cuh"
#include "texel.cuh"

namespace jt {
namespace {

// A pixel's taps.
struct Taps {
  uint32_t gid;    // gid of MCU (0, 0) of its texture, relative to the first coefficient MCU
  uint32_t mcus_x;
  int xa, xb, ya, yb;
  float fx, fy;
  bool ok;
};

// MCU (relative to the first coefficient MCU) of column tap x, row tap y.
__device__ __forceinline__ uint32_t mcu_of(const Taps& T, int x, int y) {
  return T.gid + (uint32_t)(x >> 4) + (uint32_t)(y >> 4) * T.mcus_x;
}

// Taps of the quad's pixel i: ok is false when it is empty or names no coefficient texture.
__device__ __forceinline__ Taps taps_of(const FloatArgs& a, float u, float v, uint32_t tex, uint32_t mip,
                                        bool& missing) {
  Taps T{};
  const PixL P = pix_level(a.tl, tex | (mip << 16));
  T.ok = (P.info & kPixCoef) != 0;
  missing |= !T.ok && tex != JT_EMPTY_TEXTURE;
  T.gid = P.gid_base - a.coef_gid_base;
  T.mcus_x = P.mcus_x;
  if (T.ok && !taps_fast(P, u, v, T.xa, T.xb, T.ya, T.yb, T.fx, T.fy))
    taps_any(P, u, v, T.xa, T.xb, T.ya, T.yb, T.fx, T.fy);
  return T;
}

// Whether every tap's MCU is among the first tile_cap of the work list, the ones the pass serves
// (asked only when there are more; slots past the cache point at unit 0).
__device__ __forceinline__ bool served(const FloatArgs& a, const Taps& T) {
  auto in = [&](int x, int y) {
    const uint32_t g = a.coef_gid_base + mcu_of(T, x, y), s = __ldg(a.slot + g);
    return s < a.tile_cap && __ldg(a.work + s) == g;
  };
  return in(T.xa, T.ya) && in(T.xb, T.ya) && in(T.xa, T.yb) && in(T.xb, T.yb);
}

__global__ void k_float_count(const __grid_constant__ FloatArgs a) {
  bool missing = false;
  for_each_quad(a.views, [&](const View& V, int y, int x) {
    float u[4], v[4];
    uint32_t t[4], m[4];
    load_px4(V, y, x, u, v, t, m);
    uint32_t mcu = 0, n = 0;  // entries not yet counted: n of MCU mcu (neighbouring pixels mostly share theirs)
    auto add = [&](uint32_t g) {
      if (n && g != mcu) {
        atomicAdd(a.cursor + mcu, n);
        n = 0;
      }
      mcu = g;
      ++n;
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const Taps T = taps_of(a, u[i], v[i], t[i], m[i], missing);
      if (!T.ok) continue;
      const bool cx = T.xa >> 4 != T.xb >> 4, cy = T.ya >> 4 != T.yb >> 4;
      if (cx && cy) add(mcu_of(T, T.xb, T.yb));
      if (cy) add(mcu_of(T, T.xa, T.yb));
      if (cx) add(mcu_of(T, T.xb, T.ya));
      add(mcu_of(T, T.xa, T.ya));
    }
    if (n) atomicAdd(a.cursor + mcu, n);
  });
  if (missing) atomicOr(&a.state->err, JT_DEVERR_MISSING);
}

// Block-wide sum of one value per thread (256 threads).
__device__ __forceinline__ uint64_t block_sum256(uint64_t v, uint64_t* s_part) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
  __syncthreads();
  uint64_t t = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) t += s_part[i];
  __syncthreads();
  return t;
}

// Counts of MCUs first .. first + 3 (0 past the last), four per thread.
__device__ __forceinline__ uint4 counts_at(const FloatArgs& a, uint32_t first) {
  if (first + 4 <= a.coef_mcus) return *reinterpret_cast<const uint4*>(a.cursor + first);
  uint32_t c[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) c[k] = first + k < a.coef_mcus ? a.cursor[first + k] : 0u;
  return make_uint4(c[0], c[1], c[2], c[3]);
}

// Needed MCUs << 32 | entries of four counts.
__device__ __forceinline__ uint64_t needed_entries(const uint4& c) {
  const uint32_t needed = (c.x != 0) + (c.y != 0) + (c.z != 0) + (c.w != 0);
  return ((uint64_t)needed << 32) + c.x + c.y + c.z + c.w;
}

__global__ void __launch_bounds__(256) k_float_sums(const __grid_constant__ FloatArgs a) {
  __shared__ uint64_t s_part[8];
  const uint64_t t = block_sum256(needed_entries(counts_at(a, blockIdx.x * kFloatScan + threadIdx.x * 4)), s_part);
  if (threadIdx.x == 0) a.block_sum[blockIdx.x] = t;
}

__global__ void __launch_bounds__(256) k_float_offsets(const __grid_constant__ FloatArgs a) {
  __shared__ uint64_t s_part[8], s_warp[8];
  const uint32_t first = blockIdx.x * kFloatScan + threadIdx.x * 4;
  uint64_t pre = 0;  // sums of the blocks before this one
  for (uint32_t j = threadIdx.x; j < blockIdx.x; j += 256) pre += a.block_sum[j];
  pre = block_sum256(pre, s_part);
  const uint4 c4 = counts_at(a, first);
  const uint64_t mine = needed_entries(c4);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t inc = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t o = __shfl_up_sync(0xFFFFFFFFu, inc, d);
    if (lane >= d) inc += o;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) pre += i < warp ? s_warp[i] : 0u;
  uint64_t at = pre + inc - mine;
  const uint32_t c[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t i = first + k;
    if (i >= a.coef_mcus) break;
    const uint32_t pos = (uint32_t)(at >> 32), off = (uint32_t)at;
    a.offset[i] = off;  // the MCU's entries are [offset, cursor) once the fill has run
    a.cursor[i] = off;
    if (c[k]) {
      // as the compaction does: a position past the cache points at unit 0
      a.slot[a.coef_gid_base + i] = pos < a.cap_units ? pos : 0u;
      if (pos < a.work_cap) a.work[pos] = a.coef_gid_base + i;
    }
    at += ((uint64_t)(c[k] != 0) << 32) + c[k];
    if (i == a.coef_mcus - 1) {  // the totals
      const uint32_t total = (uint32_t)(at >> 32);
      a.state->count = total;
      a.state->units = total;
      a.state->decode_next = 0;
      if (total > a.tile_cap || total > a.cap_units || total > a.work_cap) atomicOr(&a.state->err, JT_DEVERR_CAPACITY);
    }
  }
}

// An entry: x the pixel's index; y the first texel of its taps in the MCU (y << 4 | x), then for
// each axis whether the second tap is there too and whether the first one is the pixel's second
// tap, then the last texel (which a wrap may have put before the first); z, w: fx, fy.
constexpr uint32_t kBothX = 1u << 8, kLastX = 1u << 9, kBothY = 1u << 10, kLastY = 1u << 11;

__global__ void k_float_fill(const __grid_constant__ FloatArgs a) {
  const bool check = *reinterpret_cast<const volatile uint32_t*>(&a.state->count) > a.tile_cap;
  bool missing = false;
  for_each_quad(a.views, [&](const View& V, int y, int x) {
    float u[4], v[4];
    uint32_t t[4], m[4];
    load_px4(V, y, x, u, v, t, m);
    const uint32_t p0 = (uint32_t)y * (uint32_t)V.width + (uint32_t)x;
    Taps T[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      T[i] = taps_of(a, u[i], v[i], t[i], m[i], missing);
      if (check && T[i].ok) T[i].ok = served(a, T[i]);
    }
    // places of the four kinds of entries (by the pixel's first or second tap of each axis), all
    // asked for before the first entry is written: the pass is bound by the atomics' round trips
    uint32_t pos[4][4];
    auto take = [&](auto second_x, auto second_y) {
      constexpr bool SX = decltype(second_x)::value, SY = decltype(second_y)::value;
      uint32_t(&at)[4] = pos[2 * SY + SX];
      uint32_t mcu[4], run[4];
      bool on[4], with_last[4];  // neighbours with one MCU take their places by one atomic
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        on[i] = T[i].ok && (!SX || T[i].xa >> 4 != T[i].xb >> 4) && (!SY || T[i].ya >> 4 != T[i].yb >> 4);
        mcu[i] = mcu_of(T[i], SX ? T[i].xb : T[i].xa, SY ? T[i].yb : T[i].ya);
        with_last[i] = i > 0 && on[i] && on[i - 1] && mcu[i] == mcu[i - 1];
      }
#pragma unroll
      for (int i = 3; i >= 0; --i) {
        run[i] = 1 + (i < 3 && with_last[i + 1] ? run[i + 1] : 0u);
        at[i] = a.bucket_cap;
        if (on[i] && !with_last[i]) at[i] = atomicAdd(a.cursor + mcu[i], run[i]);
      }
    };
    auto write = [&](auto second_x, auto second_y) {
      constexpr bool SX = decltype(second_x)::value, SY = decltype(second_y)::value;
      uint32_t(&at)[4] = pos[2 * SY + SX];
      uint32_t last = 0;  // the MCU of the pixel before, and whether it has an entry of the kind
      bool last_on = false;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int tx = SX ? T[i].xb : T[i].xa, ty = SY ? T[i].yb : T[i].ya;
        const bool on = T[i].ok && (!SX || T[i].xa >> 4 != T[i].xb >> 4) && (!SY || T[i].ya >> 4 != T[i].yb >> 4);
        const uint32_t mcu = mcu_of(T[i], tx, ty);
        if (i > 0) at[i] = on && last_on && mcu == last ? at[i - 1] + 1 : at[i];
        last = mcu;
        last_on = on;
        if (at[i] >= a.bucket_cap) continue;
        const bool bx = !SX && T[i].xa >> 4 == T[i].xb >> 4, by = !SY && T[i].ya >> 4 == T[i].yb >> 4;
        const int lx = bx ? T[i].xb : tx, ly = by ? T[i].yb : ty;
        const uint32_t info = (uint32_t)((ty & 15) << 4 | (tx & 15)) | (SX ? kLastX : bx ? kBothX : 0u) |
                              (SY ? kLastY : by ? kBothY : 0u) | (uint32_t)((ly & 15) << 16 | (lx & 15) << 12);
        a.bucket[at[i]] = make_uint4(p0 + (uint32_t)i, info, __float_as_uint(T[i].fx), __float_as_uint(T[i].fy));
      }
    };
    auto each = [](auto&& f) {
      f(std::false_type{}, std::false_type{});
      f(std::true_type{}, std::false_type{});
      f(std::false_type{}, std::true_type{});
      f(std::true_type{}, std::true_type{});
    };
    each(take);
    each(write);
  });
}

// Weights of an entry's first and second texel along an axis.
__device__ __forceinline__ float2 axis_weights(uint32_t info, uint32_t both, uint32_t last, float f) {
  return make_float2((info & last) ? f : 1.f - f, (info & both) ? f : 0.f);
}

// 1-D transforms of eight values by even and odd halves (A[7-x][u] = (-1)^u A[x][u]):
// o[x] = sum_u A[x][u] i[u], and the adjoint o[u] = sum_x A[x][u] i[x].
__device__ __forceinline__ void transform8(const float* A, const float (&i)[8], float (&o)[8]) {
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    float e = A[x * 8] * i[0], d = A[x * 8 + 1] * i[1];
#pragma unroll
    for (int u = 2; u < 8; u += 2) {
      e = fmaf(A[x * 8 + u], i[u], e);
      d = fmaf(A[x * 8 + u + 1], i[u + 1], d);
    }
    o[x] = e + d;
    o[7 - x] = e - d;
  }
}
__device__ __forceinline__ void adjoint8(const float* A, const float (&i)[8], float (&o)[8]) {
  float s[4], d[4];
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    s[x] = i[x] + i[7 - x];
    d[x] = i[x] - i[7 - x];
  }
#pragma unroll
  for (int u = 0; u < 8; u += 2) {
    o[u] = A[u] * s[0];
    o[u + 1] = A[u + 1] * d[0];
#pragma unroll
    for (int x = 1; x < 4; ++x) {
      o[u] = fmaf(A[x * 8 + u], s[x], o[u]);
      o[u + 1] = fmaf(A[x * 8 + u + 1], d[x], o[u + 1]);
    }
  }
}

// Shared memory of a pair of MCUs: a data unit's 64 values row by row, padded to 72, so that 32 lanes at
// one row of the columns of four data units hit different banks. A row's two halves are
// stored and read by lanes in an order that depends on the row, for the same reason.
constexpr int kDu = 72, kMcu = 6 * kDu;

__device__ __forceinline__ void put_row(float* row, int v, const float (&r)[8]) {
  const bool up = v >= 4;
  float4* p = reinterpret_cast<float4*>(row);
  p[up] = up ? make_float4(r[4], r[5], r[6], r[7]) : make_float4(r[0], r[1], r[2], r[3]);
  p[!up] = up ? make_float4(r[0], r[1], r[2], r[3]) : make_float4(r[4], r[5], r[6], r[7]);
}
__device__ __forceinline__ void get_row(const float* row, int v, float (&r)[8]) {
  const bool up = v >= 4;
  const float4* p = reinterpret_cast<const float4*>(row);
  const float4 a = p[up], b = p[!up];
  const float4 lo = up ? b : a, hi = up ? a : b;
  r[0] = lo.x; r[1] = lo.y; r[2] = lo.z; r[3] = lo.w;
  r[4] = hi.x; r[5] = hi.y; r[6] = hi.z; r[7] = hi.w;
}

// A warp takes a.pairs pairs of neighbouring MCUs, one pair at a time; the grid covers all pairs
// (a persistent grid waited for its slowest warps: 560 K cycles against 330 K on average).
// First MCU of this warp.
__device__ __forceinline__ uint32_t first_mcu(const FloatArgs& a) {
  return (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (2u * (uint32_t)a.pairs);
}

// Entry range of lane k < 2 a.pairs's MCU m0 + k, whose cursor is zeroed for the next pass's
// count: x its first entry, y how many.
__device__ __forceinline__ uint2 load_ranges(const FloatArgs& a, uint32_t m0) {
  const uint32_t lane = threadIdx.x & 31, m = m0 + lane;
  uint2 r = make_uint2(0, 0);
  if (lane < 2u * (uint32_t)a.pairs && m < a.coef_mcus) {
    r = make_uint2(a.offset[m], min(a.cursor[m], a.bucket_cap));
    a.cursor[m] = 0;
  }
  r.y = r.y > r.x ? r.y - r.x : 0u;
  return r;
}

// Pair p's entries: the first MCU's n0 from b0, the second's n1 from b1.
struct Pair {
  uint32_t b0, n0, b1, n1;
  __device__ __forceinline__ uint32_t total() const { return n0 + n1; }
  __device__ __forceinline__ uint4 entry(const FloatArgs& a, uint32_t j) const {
    return j < total() ? __ldcs(a.bucket + (j < n0 ? b0 + j : b1 + (j - n0))) : make_uint4(0, 0, 0, 0);
  }
};

// The backward's walk of a lane over n entries: from first on by step up to end. Neighbouring entries are
// mostly neighbouring pixels, so where many pixels fall on a texel (kDense entries in a pair), 32
// of them at a time would add into one or two addresses: there each lane takes a run of its own
// (backward, sixteen pixels a texel each way in 40 MCUs: 63.8 ms by 32 neighbours, 5.6 by runs;
// one pixel a texel, 580 entries in a pair: 91 us, and 123 by runs).
constexpr uint32_t kDense = 1024;
struct Walk {
  uint32_t first, step, end;
};
__device__ __forceinline__ Walk walk_of(uint32_t n) {
  const uint32_t lane = threadIdx.x & 31, run = (n + 31) / 32;
  return n < kDense ? Walk{lane, 32u, n} : Walk{lane * run, 1u, min(n, lane * run + run)};
}
__device__ __forceinline__ Pair pair_of(uint2 r, int p) {
  return Pair{__shfl_sync(0xFFFFFFFFu, r.x, 2 * p), __shfl_sync(0xFFFFFFFFu, r.y, 2 * p), __shfl_sync(0xFFFFFFFFu, r.x, 2 * p + 1), __shfl_sync(0xFFFFFFFFu, r.y, 2 * p + 1)};
}

// Offsets in an MCU of an entry's two luma columns and rows and chroma columns and rows.
struct EntryPlaces {
  int x[2], y[2], cx[2], cy[2];
};
__device__ __forceinline__ EntryPlaces places_of(uint32_t info) {
  EntryPlaces q;
#pragma unroll
  for (int k = 0; k < 2; ++k) {  // (without a second tap the first one's place, with weight 0)
    const int tx = (int)(info >> 12 * k & 15u), ty = (int)(info >> (4 + 12 * k) & 15u);
    q.x[k] = (tx >> 3) * kDu + (tx & 7);
    q.y[k] = (ty >> 3) * (2 * kDu) + (ty & 7) * 8;
    q.cx[k] = 4 * kDu + (tx >> 1);
    q.cy[k] = (ty >> 1) * 8;
  }
  return q;
}

// Values that are not finite spread by the taps of weight zero (0 * inf), which the sums below add as they
// are: where one is met, the sum is taken tap by tap.
__device__ __forceinline__ bool finite3(float a, float b, float c) {
  return fabsf(a) + fabsf(b) + fabsf(c) < __int_as_float(0x7F800000);
}

__device__ __forceinline__ void copy16_async(float* to, const float* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}

__global__ void __launch_bounds__(kFloatWarps * 32, kForwardCtas) k_float_forward(const __grid_constant__ FloatArgs a) {
  extern __shared__ __align__(16) float pair_mem[];  // [warps][2][kMcu] texels, [warps][768] coefficients
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* f = pair_mem + warp * (2 * kMcu);
  float* raw = pair_mem + (blockDim.x >> 5) * (2 * kMcu) + warp * 768;
  const uint32_t m0 = first_mcu(a);
  const uint2 ranges = load_ranges(a, m0);
  // the next pair's coefficients and first entries are fetched while this one is worked on
  auto fetch = [&](const Pair& r, int p) {
    const float* src = a.coef + (size_t)(m0 + 2u * (uint32_t)p) * 384 + lane * 4;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      if (k < 3 ? r.n0 : r.n1) copy16_async(raw + (k * 32 + lane) * 4, src + k * 128);
    }
  };
  Pair next = pair_of(ranges, 0);
  fetch(next, 0);
  uint4 first = next.entry(a, (uint32_t)lane);
#pragma unroll 1
  for (int p = 0; p < a.pairs; ++p) {
    const Pair r = next;
    uint4 ent = first;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();  // every lane's copies
    if (r.total()) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {  // the pair's 96 rows (an MCU that was not fetched is not read below)
        const int q = lane + 32 * k;
        float in[8], out[8];
        get_row(raw + q * 8, q & 7, in);
        transform8(a.basis, in, out);
        put_row(f + (q >> 3) * kDu + (q & 7) * 8, q & 7, out);
      }
      __syncwarp();
    }
    if (p + 1 < a.pairs) {
      next = pair_of(ranges, p + 1);
      fetch(next, p + 1);
      first = next.entry(a, (uint32_t)lane);
    }
    if (r.total() == 0) continue;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int q = lane + 32 * k;
      float* col = f + (q >> 3) * kDu + (q & 7);
      float in[8], out[8];
#pragma unroll
      for (int v = 0; v < 8; ++v) in[v] = col[8 * v];
      transform8(a.basis, in, out);
#pragma unroll
      for (int v = 0; v < 8; ++v) col[8 * v] = out[v];
    }
    __syncwarp();
#pragma unroll 1
    for (uint32_t j = (uint32_t)lane; j < r.total(); j += 32) {
      const uint4 after = r.entry(a, j + 32);
      const float2 wx = axis_weights(ent.y, kBothX, kLastX, __uint_as_float(ent.z));
      const float2 wy = axis_weights(ent.y, kBothY, kLastY, __uint_as_float(ent.w));
      const EntryPlaces q = places_of(ent.y);
      const float* t = f + (j < r.n0 ? 0 : kMcu);
      auto sum = [&](const float* g, const int (&x)[2], const int (&y)[2]) {
        return fmaf(wy.y, fmaf(wx.y, g[y[1] + x[1]], wx.x * g[y[1] + x[0]]), wy.x * fmaf(wx.y, g[y[0] + x[1]], wx.x * g[y[0] + x[0]]));
      };
      const float Y = fmaf(128.f, (wx.x + wx.y) * (wy.x + wy.y), sum(t, q.x, q.y));
      const float cb = sum(t, q.cx, q.cy), cr = sum(t + kDu, q.cx, q.cy);
      float red = fmaf(kCr2R, cr, Y), grn = fmaf(-kCr2G, cr, fmaf(-kCb2G, cb, Y)), blu = fmaf(kCb2B, cb, Y);
      if (!finite3(red, grn, blu)) {  // tap by tap, without those of weight zero
        red = grn = blu = 0.f;
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
          const float w = (k & 1 ? wx.y : wx.x) * (k & 2 ? wy.y : wy.x);
          if (w == 0.f) continue;
          const float* c = t + (k & 1 ? q.cx[1] : q.cx[0]) + (k & 2 ? q.cy[1] : q.cy[0]);
          const float y = t[(k & 1 ? q.x[1] : q.x[0]) + (k & 2 ? q.y[1] : q.y[0])] + 128.f;
          red = fmaf(w, fmaf(kCr2R, c[kDu], y), red);
          grn = fmaf(w, fmaf(-kCr2G, c[kDu], fmaf(-kCb2G, c[0], y)), grn);
          blu = fmaf(w, fmaf(kCb2B, c[0], y), blu);
        }
      }
      float* out = a.frame + 3 * (size_t)ent.x;
      if ((ent.y & (kBothX | kBothY)) == (kBothX | kBothY)) {  // the pixel's only entry
        out[0] = red;
        out[1] = grn;
        out[2] = blu;
      } else {
        atomicAdd(out, red);
        atomicAdd(out + 1, grn);
        atomicAdd(out + 2, blu);
      }
      ent = after;
    }
    __syncwarp();  // the pair's memory is written again
  }
}

__global__ void __launch_bounds__(kFloatWarps * 32, kBackwardCtas) k_float_backward(const __grid_constant__ FloatArgs a) {
  extern __shared__ __align__(16) float pair_mem[];  // [warps][2][kMcu]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* f = pair_mem + warp * (2 * kMcu);
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  const uint32_t m0 = first_mcu(a);
  const uint2 ranges = load_ranges(a, m0);
  // the next pair's first entries and their pixels' gradients are fetched ahead
  Pair next = pair_of(ranges, 0);
  uint4 first = next.entry(a, walk_of(next.total()).first);
  float3 grad;
  auto fetch = [&](uint32_t px) {
    const float* gf = a.frame + 3 * (size_t)px;
    grad = make_float3(__ldg(gf), __ldg(gf + 1), __ldg(gf + 2));
  };
  fetch(first.x);
#pragma unroll 1
  for (int p = 0; p < a.pairs; ++p) {
    const uint32_t m = m0 + 2u * (uint32_t)p;
    if (m >= a.coef_mcus) break;
    const Pair r = next;
    const Walk w = walk_of(r.total());
    uint4 ent = first, after = r.entry(a, w.first + w.step);
    if (p + 1 < a.pairs) {
      next = pair_of(ranges, p + 1);
      first = next.entry(a, walk_of(next.total()).first);
    }
    if (r.total()) {
#pragma unroll
      for (int k = 0; k < 7; ++k) {
        if (k < 6 || lane < 2 * kMcu / 4 - 192) reinterpret_cast<float4*>(f)[k * 32 + lane] = z;
      }
      __syncwarp();
#pragma unroll 1
      for (uint32_t j = w.first; j < w.end; j += w.step) {
        const float gy = grad.x + grad.y + grad.z, gcb = kCb2B * grad.z - kCb2G * grad.y, gcr = kCr2R * grad.x - kCr2G * grad.y;
        float2 wx = axis_weights(ent.y, kBothX, kLastX, __uint_as_float(ent.z));
        float2 wy = axis_weights(ent.y, kBothY, kLastY, __uint_as_float(ent.w));
        const EntryPlaces q = places_of(ent.y);
        float* g = f + (j < r.n0 ? 0 : kMcu);
        const bool bx = (ent.y & kBothX) != 0, by = (ent.y & kBothY) != 0;
        // the next entry's gradient and the entry after it are under way during this one's sums (one
        // after the other at the head of the loop they took longer than the sums)
        ent = after;
        fetch(ent.x);
        after = r.entry(a, j + 2 * w.step);
        if (!finite3(gy, gcb, gcr)) {
#pragma unroll 1
          for (int k = 0; k < 4; ++k) {
            const float v = (k & 1 ? wx.y : wx.x) * (k & 2 ? wy.y : wy.x);
            if (v == 0.f) continue;
            float* c = g + (k & 1 ? q.cx[1] : q.cx[0]) + (k & 2 ? q.cy[1] : q.cy[0]);
            atomicAdd(g + (k & 1 ? q.x[1] : q.x[0]) + (k & 2 ? q.y[1] : q.y[0]), v * gy);
            atomicAdd(c, v * gcb);
            atomicAdd(c + kDu, v * gcr);
          }
          continue;
        }
        atomicAdd(g + q.y[0] + q.x[0], wx.x * wy.x * gy);
        if (bx) atomicAdd(g + q.y[0] + q.x[1], wx.y * wy.x * gy);
        if (by) atomicAdd(g + q.y[1] + q.x[0], wx.x * wy.y * gy);
        if (bx && by) atomicAdd(g + q.y[1] + q.x[1], wx.y * wy.y * gy);
        // chroma (upsample^T): two taps of one sample are one term
        const bool sx = q.cx[1] != q.cx[0], sy = q.cy[1] != q.cy[0];
        if (!sx) wx.x += wx.y;
        if (!sy) wy.x += wy.y;
        auto chroma = [&](int at, float w) {
          atomicAdd(g + at, w * gcb);
          atomicAdd(g + kDu + at, w * gcr);
        };
        chroma(q.cy[0] + q.cx[0], wx.x * wy.x);
        if (sx) chroma(q.cy[0] + q.cx[1], wx.y * wy.x);
        if (sy) chroma(q.cy[1] + q.cx[0], wx.x * wy.y);
        if (sx && sy) chroma(q.cy[1] + q.cx[1], wx.y * wy.y);
      }
      __syncwarp();
    }
    fetch(first.x);
    float4* dst = reinterpret_cast<float4*>(a.grad_coef + (size_t)m * 384) + lane;
    if (r.total()) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {  // the pair's 96 columns, then its rows
        const int q = lane + 32 * k;
        float* col = f + (q >> 3) * kDu + (q & 7);
        float in[8], out[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) in[v] = col[8 * v];
        adjoint8(a.basis, in, out);
#pragma unroll
        for (int v = 0; v < 8; ++v) col[8 * v] = out[v];
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int q = lane + 32 * k;
        float* row = f + (q >> 3) * kDu + (q & 7) * 8;
        float in[8], out[8];
        get_row(row, q & 7, in);
        adjoint8(a.basis, in, out);
        put_row(row, q & 7, out);
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 6; ++k) {  // (an MCU without entries: the transforms of its zeros)
        const int q = lane + 32 * k;
        if (k < 3 || m + 1 < a.coef_mcus) __stcs(dst + 32 * k, *reinterpret_cast<const float4*>(f + (q >> 4) * kDu + (q & 15) * 4));
      }
      __syncwarp();  // the pair's memory is written again
    } else {
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        if (k < 3 || m + 1 < a.coef_mcus) __stcs(dst + 32 * k, z);
      }
    }
  }
}

constexpr size_t kBackwardSmem = 2 * kMcu * sizeof(float), kForwardSmem = kBackwardSmem + 768 * sizeof(float);  // a warp

void launch_inversion(const FloatArgs& a, int threads, int pixel_grid, cudaStream_t s) {
  const int blocks = (int)((a.coef_mcus + kFloatScan - 1) / kFloatScan);
  k_float_count<<<pixel_grid, threads, 0, s>>>(a);
  k_float_sums<<<blocks, 256, 0, s>>>(a);
  k_float_offsets<<<blocks, 256, 0, s>>>(a);
  k_float_fill<<<pixel_grid, std::min(threads, 512), 0, s>>>(a);  // (its registers allow no more)
}

// Launches a gather of `ctas` resident CTAs per SM with up to `most` pairs for each warp: fewer where
// there are not enough to fill the chip, then smaller CTAs, so that few MCUs (which then hold many
// entries) spread over its SMs. One 1080p frame, forward / backward: one 128^2 texture (64 MCUs)
// 7.9 / 29.1 ms with the most pairs and whole CTAs, 1.7 / 3.9 so; one of 512^2 723 / 1430 us, 246 / 402;
// two of 1024^2 184 / 262 us, 108 / 143.
void launch_gather(void (*gather)(FloatArgs), FloatArgs a, int most, int ctas, size_t warp_smem, cudaStream_t s) {
  const uint64_t pairs = ((uint64_t)a.coef_mcus + 1) / 2, sms = (uint64_t)a.sms;
  for (a.pairs = most; a.pairs > 1 && pairs < sms * ctas * kFloatWarps * a.pairs; a.pairs /= 2) {
  }
  const uint64_t tasks = (pairs + a.pairs - 1) / a.pairs;
  int warps = kFloatWarps;
  while (warps > 1 && tasks < sms * warps) warps /= 2;
  gather<<<(int)((tasks + warps - 1) / warps), warps * 32, warps * warp_smem, s>>>(a);
}

}  // namespace

// Sets the gather kernels' shared-memory attributes on the current device.
bool float_configure() {
  return cudaFuncSetAttribute(k_float_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kFloatWarps * kForwardSmem)) == cudaSuccess &&
         cudaFuncSetAttribute(k_float_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kFloatWarps * kBackwardSmem)) == cudaSuccess;
}

// The cursors must be zero on entry (the gathers leave them so; after a failed launch the caller
// clears them), and the forward's frame.
void launch_float_forward(const FloatArgs& a, int threads, int pixel_grid, cudaStream_t s) {
  launch_inversion(a, threads, pixel_grid, s);
  launch_gather(k_float_forward, a, kForwardPairs, kForwardCtas, kForwardSmem, s);
}

void launch_float_backward(const FloatArgs& a, int threads, int pixel_grid, cudaStream_t s) {
  launch_inversion(a, threads, pixel_grid, s);
  launch_gather(k_float_backward, a, kBackwardPairs, kBackwardCtas, kBackwardSmem, s);
}

}  // namespace jt
