// Decode (paper Sec. 4.3): every MCU of the work list is Huffman-decoded from its index
// entry (bit offset + DC predictors, Sec. 5.1 / Sec. 5.3), dequantised, inverse-DCT'd,
// chroma-upsampled, colour-converted and written as an RGBA8 tile into the block cache.
//
// GB300 design (the paper's one 64-thread block per MCU with a 32-lane code compare,
// Sec. 5.2, is prior art here):
//  * persistent grid; each warp takes batches of m_eff <= M work items (M = 4, 8, 16 or 32, the
//    buffer width), chosen from the list's length on the device, so the count never goes to
//    the host. The first batch of each warp is fixed, later ones come from a device counter,
//    so uneven MCU sizes balance dynamically;
//  * entropy phase: lane m < m_eff runs MCU m's serial chain over all its data units from a
//    byte-swapped copy of its words staged in shared memory (a per-warp pool shared out by a
//    prefix sum). The chain bounds the pass (it ends with the heaviest MCU), so a symbol's
//    dependent path is kept to one table read and a few ALU operations (entropy_fast);
//  * pixel phase: the warp takes its MCUs one by one. Both IDCT passes of an 8x8 data unit
//    are one mma.sync each (an 8x8 by 8x8 product, exact in fp32: see idct_pass), the
//    fragment layouts make the first product's output the second one's input without a
//    shuffle, and a lane ends up with two pixels of every data unit of the MCU in registers,
//    which it colour-converts in packed 16-bit pairs and stores as 32-byte rows of texels.
//    Nothing goes through memory between the coefficients and the tile.
//
// Decode spec (identical in the oracle): dequantised d = clamp16(q * Q); column pass
// t = clamp16(floor((sum_v K[y][v] d[v][u] + 2^8) / 2^9)); row pass
// p = clamp(floor((sum_u K[x][u] t[y][u] + 2^18) / 2^19) + 128, 0, 255) with
// K[x][u] = round(2^14 c_u cos((2x+1) u pi / 16)); JFIF colour in 16-bit fixed point;
// 4:2:0 chroma replicated within the MCU; DC values wrap modulo 2^16. A reduced level
// (1/2^r) uses K_N[x][u] = round(2^14 c_u cos((2x+1) u pi / (2N))) on the N x N lowest
// frequencies, N = 8 >> r, with the same rounding.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>

#include "jt_internal.cuh"

namespace jt {
namespace {

extern __shared__ __align__(16) uint8_t smem[];

// ---- integer IDCT constants: round(8192 cos(k pi / 16)), k = 1..7 ----
constexpr int C1 = 8035, C2 = 7568, C3 = 6811, C4 = 5793, C5 = 4551, C6 = 3135, C7 = 1598;

// Position in zig-zag order of natural index r*8+c (closed form: cells before the
// anti-diagonal s = r+c, plus the offset along it; odd diagonals run downwards).
__host__ __device__ constexpr int zz_pos(int r, int c) {
  const int s = r + c;
  const int before = s <= 7 ? s * (s + 1) / 2 : 64 - (15 - s) * (16 - s) / 2;
  const int along = (s & 1) ? r - (s > 7 ? s - 7 : 0) : (s < 7 ? s : 7) - r;
  return before + along;
}
static_assert(zz_pos(0, 0) == 0 && zz_pos(0, 1) == 1 && zz_pos(1, 0) == 2 && zz_pos(2, 0) == 3 &&
                  zz_pos(0, 2) == 5 && zz_pos(7, 6) == 62 && zz_pos(7, 7) == 63 && zz_pos(3, 4) == 31 && zz_pos(4, 3) == 32,
              "zig-zag positions");

// K_N[x][u] for N = 8 >> r (zero outside N x N): the N-point cosines are the 8-point ones at
// multiples of 8 / N.
__device__ __forceinline__ int idct_k(int x, int u, int r) {
  const int n = 8 >> r;
  if (x >= n || u >= n) return 0;
  int i = ((2 * x + 1) * u << r) & 31;  // angle in units of pi / 16
  i = i > 16 ? 32 - i : i;
  const int j = i > 8 ? 16 - i : i;  // 1..7 unless u = 0
  const int c = j == 1 ? C1 : j == 2 ? C2 : j == 3 ? C3 : j == 4 ? C4 : j == 5 ? C5 : j == 6 ? C6 : C7;
  return u == 0 ? C4 : (i > 8 ? -c : c);
}

// Words of the MCUs' entropy-coded data copied to shared memory before their serial decode
// (random loads from HBM take thousands of cycles and would otherwise sit on the serial
// chain once per word). A warp has kStageWords words per MCU as one pool, shared out by a
// prefix sum over its lanes, so a long MCU can use what short ones leave (the mean MCU of a
// scene needs about a quarter). When the batch's MCUs do not fit, each is staged in parts: its
// chain stops short of the staged words' end and goes on when the next part is there. Words
// are stored big-endian-swapped.
constexpr int kStageWords = 32;

// Shared memory of one warp: per MCU six data units of 64 int16 coefficients in zig-zag order,
// then the staged words [M * kStageWords]. An MCU's 772 bytes are an odd number of words,
// so that lanes storing the same coefficient of their MCUs hit different banks; a data unit
// is 32 words, so the pixel phase's reads of one data unit never conflict.
// A batch of 4:4:4 MCUs alone packs them in 388 bytes, two for one of the others.
constexpr int kMcuBytes = 6 * 128 + 4, kMcuBytes444 = 3 * 128 + 4;
static_assert(kMcuBytes444 / 4 % 2 == 1 && 4 * kMcuBytes444 % 16 == 0 && 2 * kMcuBytes444 < kMcuBytes + 4 * kStageWords, "as below");
static_assert(kMcuBytes / 4 % 2 == 1 && 4 * kMcuBytes % 16 == 0, "bank spread, and 16-byte whole for M >= 4");
__host__ __device__ constexpr size_t warp_smem(int M) { return (size_t)M * (kMcuBytes + kStageWords * 4); }

__device__ __forceinline__ uint32_t bswap(uint32_t w) { return __byte_perm(w, 0, 0x0123); }

__device__ __forceinline__ uint32_t sm_u32(uint32_t off) { return *reinterpret_cast<const uint32_t*>(smem + off); }
__device__ __forceinline__ int16_t& sm_i16(uint32_t off) { return *reinterpret_cast<int16_t*>(smem + off); }

// Signed value of a symbol with entry e whose code starts at the top of w (T.81 EXTEND; 0
// without value bits).
__device__ __forceinline__ int symbol_value(uint32_t w, uint32_t e) {
  const int m = (int)(0xFFFFFFFFu << ((e >> 5) & 15u));      // -2^s
  const int raw = (int)(__funnelshift_l(w, 0u, e) & ~m);     // (shifts by the low five bits of e)
  return raw + (2 * raw + m < 0 ? m + 1 : 0);
}

// Stores a coefficient when c holds: a predicated store, never a branch.
__device__ __forceinline__ void store_if(bool c, uint32_t off, int v) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.shared.u16 [%0], %1;\n\t}" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(smem) + off),
               "h"((int16_t)v), "r"((uint32_t)c)
               : "memory");
}

// Reads a table record when c holds: predicated loads, which nothing waits for where they are
// not made.
template <bool CAP>
__device__ __forceinline__ void load_if(bool p, uint32_t off, uint4& t, uint4& c) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(smem) + off;
  if (CAP)
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %9, 0;\n\t@q ld.shared.v4.u32 {%0, %1, %2, %3}, [%8];\n\t"
                 "@q ld.shared.v4.u32 {%4, %5, %6, %7}, [%8+16];\n\t}"
                 : "+r"(t.x), "+r"(t.y), "+r"(t.z), "+r"(t.w), "+r"(c.x), "+r"(c.y), "+r"(c.z), "+r"(c.w)
                 : "r"(a), "r"((uint32_t)p));
  else
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %6, 0;\n\t@q ld.shared.v4.u32 {%0, %1, %2, %3}, [%5];\n\t"
                 "@q ld.shared.u32 %4, [%5+16];\n\t}"
                 : "+r"(t.x), "+r"(t.y), "+r"(t.z), "+r"(t.w), "+r"(c.x)
                 : "r"(a), "r"((uint32_t)p));
}
__device__ __forceinline__ void load_if(bool p, const char* a, uint4& t, uint4& c) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %9, 0;\n\t@q ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%8];\n\t"
               "@q ld.global.nc.v4.u32 {%4, %5, %6, %7}, [%8+16];\n\t}"
               : "+r"(t.x), "+r"(t.y), "+r"(t.z), "+r"(t.w), "+r"(c.x), "+r"(c.y), "+r"(c.z), "+r"(c.w)
               : "l"(a), "r"((uint32_t)p));
}

constexpr uint32_t kNoSet = 0xFFFFFFFFu;
constexpr uint32_t kBusyWarps = 12;         // three per SM sub-partition
constexpr uint32_t kLongRun = 10;           // full batches per warp from which a list is long
constexpr uint32_t kInvalid = 0x80000000u;  // an invalid coding (bit positions stay far below)
constexpr uint32_t kSizeMask = 15u << 5;
constexpr uint32_t kPast = (64u << kRunShift) - (1u << (kRunShift - 1));  // k + entry past slot 63, or kNoEntry at any k
static_assert((63u << kRunShift) + kSizeMask + 31u < kPast && kNoEntry >= kPast, "the last valid place, and no entry");
constexpr uint32_t kSlackBytes = 1344;      // shared memory a chain may read past its staged words

// Entropy-decodes the `ndu` data units of one MCU (or one data unit) from words staged whole at
// shared offset st (nst of them) into coef (shared offset; [du][k] int16 in zig-zag order,
// zero on entry), with the tables of record seq of the set (SH: the staged set 0, else
// `set`). DC slots receive the DC *difference*.
//
// The serial chain per symbol bounds the pass: it ends with the heaviest MCU, decoded by a
// warp with few other lanes left, which issues in order, so what counts is the number of
// instructions per symbol and that none of them is a branch (a branch costs a lone warp 20
// to 30 cycles; the loop's back edge is taken once per kSymbols symbols). One table read
// serves codes of any length (see HuffSet). The bits behind the 32-bit window are cut from
// the staged words again for every symbol, which is cheaper than refilling a buffer. Data-unit
// bookkeeping is a record pointer: the tables come from the record, and a chain past its
// last data unit reads a table of zeros (a symbol without value or length). Measured on the
// heaviest 4:2:0 MCU of a 1080p frame (193 symbols): 360 cycles a symbol with the same work in
// branches, 208 with a buffer refilled by selects and a two-level table, 133 with both
// successors' entries read and one selected.
//
// Runs from ch.pos to the end of the chain or to the first group of kSymbols symbols that starts
// at bit `limit` (of shared memory) or later; returns false for a symbol without a table entry
// or past the data unit's end. Bits past the staged words are whatever lies there (at most 384
// symbols of 27 bits on, inside the allocation with its slack): the caller redoes the MCU with
// entropy_any when it consumed any, or for false.
constexpr int kSymbols = 4;
constexpr uint32_t kGroupBits = kSymbols * 27 + 64;  // a group consumes and looks ahead at most this far

struct Chain {
  uint32_t pos;      // bit position in the stream (of the symbol of e)
  uint32_t e;        // its entry (kFresh: not read yet)
  uint32_t k;        // k << kRunShift
  uint32_t q, qend;  // table record of the data unit, the record past the last
  uint32_t coef;     // shared offset of the data unit's coefficients
};
constexpr uint32_t kFresh = 0xFFFFFFFFu;

// SH: the tables staged in shared memory; CAP: a set that needs its tables' caps.
template <bool SH, bool CAP>
__device__ __forceinline__ bool entropy_fast(Chain& ch, uint32_t st, uint32_t w0, uint32_t limit, const HuffSet* set) {
  const char* gt = reinterpret_cast<const char*>(set);
  auto entry = [&](uint32_t o) {
    return SH ? (uint32_t)*reinterpret_cast<const uint16_t*>(smem + o)
              : (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(gt + o));
  };
  auto rec = [&](uint32_t o) {
    return SH ? *reinterpret_cast<const uint4*>(smem + o) : __ldg(reinterpret_cast<const uint4*>(gt + o));
  };
  uint32_t q = ch.q, coef = ch.coef, k = ch.k, e = ch.e;
  const uint32_t qend = ch.qend;
  // AC table, next first table; next first k << kRunShift, their caps
  uint4 t = rec(q), c = rec(q + 16);
  uint32_t p = 8 * st + (ch.pos - 32 * w0);  // in bits of shared memory (stages are 16-byte aligned)
  uint32_t o = (p >> 3) & ~3u;
  const uint32_t x0 = sm_u32(o), x1 = sm_u32(o + 4), x2 = sm_u32(o + 8);
  uint32_t b0 = __funnelshift_l(x1, x0, p), b1 = __funnelshift_l(x2, x1, p);
  if (e == kFresh) {
    const uint4 t0 = rec(q + 32);
    k = t0.z;
    e = entry(t0.x + 2u * table_index<CAP>(b0, (int)t0.y, (int)t0.w));
  }
  uint32_t bad = 0;
#pragma unroll 1
  do {
#pragma unroll
    for (int i = 0; i < kSymbols; ++i) {
      // the next symbol's read
      const uint32_t kr = k + e;
      const bool done = kr >= (63u << kRunShift);  // the run reaches slot 63
      const uint32_t w = b0;
      b0 = __funnelshift_l(b1, b0, e);
      const uint32_t en = entry((done ? t.z : t.x) +
                                2u * table_index<CAP>(b0, (int)(done ? t.w : t.y), (int)(done ? c.z : c.y)));
      p += e & 31u;
      o = (p >> 3) & ~3u;
      b1 = __funnelshift_l(sm_u32(o + 8), sm_u32(o + 4), p);
      // the current one's value and place
      const bool past = kr >= kPast, val = (e & kSizeMask) != 0;
      store_if(val & !past, coef + (kr >> (kRunShift - 1)), symbol_value(w, e));
      bad = val & past ? 1u : bad;
      k = done ? c.x : (kr | ((1u << kRunShift) - 1u)) + 1u;
      coef += done ? 128u : 0u;
      q += done ? (uint32_t)sizeof(HuffSeq) : 0u;
      if (SH)
        load_if<CAP>(done, q, t, c);
      else
        load_if(done, gt + q, t, c);
      e = en;
    }
  } while ((q != qend) & (bad == 0) & (p < limit));
  ch.pos = p - 8 * st + 32 * w0;
  ch.e = e;
  ch.k = k;
  ch.q = q;
  ch.coef = coef;
  return bad == 0;
}

// The general form of entropy_fast from global memory, and the last word on invalid codings:
// `gw` are the stream's words from the MCU's first one on (ngw readable, zeros past them),
// bit0 its first bit there. Returns the bit position after the last symbol, or kInvalid plus the
// number of data units whose DC was reached (the coefficients decoded before the invalid
// symbol stay). nl: luma data units (0 for a chroma unit of its own); cpt: the compact form.
// Out of line: a rare path.
__device__ __noinline__ uint32_t entropy_any(const uint32_t* gw, uint32_t ngw, uint32_t bit0, const HuffSet* set,
                                             int ndu, int nl, bool cpt, uint32_t coef) {
  for (int i = 0; i < 32 * ndu; ++i) *reinterpret_cast<uint32_t*>(smem + coef + 4 * i) = 0;
  auto word = [&](uint32_t i) { return i < ngw ? bswap(__ldg(gw + i)) : 0u; };
  uint32_t pos = bit0;
  int du = 0, k = cpt ? 1 : 0;
#pragma unroll 1
  for (int it = 0; it < 64 * 6; ++it) {  // at most 64 symbols per data unit: each advances k
    const HuffTable* t = set->table + (k == 0 ? 0 : 1) + (du < nl ? 0 : 2);
    const uint32_t w = __funnelshift_l(word((pos >> 5) + 1), word(pos >> 5), pos & 31u);
    const uint32_t x = table_index<true>(w, __ldg(&t->d), __ldg(&t->cap));
    const uint32_t e = __ldg(reinterpret_cast<const uint16_t*>(reinterpret_cast<const char*>(set) + __ldg(&t->base)) + x);
    if (e == kNoEntry) return kInvalid + (uint32_t)(du + (k > 0 ? 1 : 0));
    const bool val = (e & kSizeMask) != 0;
    const int kst = k + (int)(e >> kRunShift);
    if (val) sm_i16(coef + (uint32_t)(du * 128 + 2 * min(kst, 63))) = (int16_t)symbol_value(w, e);
    if (val && kst > 63) return kInvalid + (uint32_t)(du + 1);
    pos += e & 31u;
    k = kst + 1;
    if (kst >= 63) {
      ++du;
      if (du == ndu) return pos;
      k = cpt && du >= nl ? 1 : 0;
    }
  }
  return kInvalid + (uint32_t)ndu;  // (not reached)
}

// ---- pixel phase ----

// An 8x8 transform pass of a data unit is one tensor-core product with exact results.
//
// D = K X with K the 14-bit integer matrix and X 16-bit integers. K is split as Kh 2^7 + Kl
// (|Kh| <= 63, -64 <= Kl < 64), X as Xh 2^8 + Xl (Xh a signed, Xl an unsigned byte); every
// part is exact in fp16, the products are exact, and the sums are exact in fp32. The 16 x 16
// operand A holds Kh 2^7 in rows 0-7 and Kl in rows 8-15, columns 0-7 meeting Xh and columns
// 8-15 (scaled by 2^-8) meeting Xl in the 16 x 8 operand B, so D's rows 0-7 are
// (Kh 2^7) X 2^-8, multiples of 2^-1 below 2^23 in magnitude, and rows 8-15 are Kl X 2^-8,
// multiples of 2^-8 below 2^16. A lane (g = lane / 4, t = lane % 4) gets both parts of the
// elements (g, 2t) and (g, 2t + 1); the accumulators of the high parts start at the pass's
// rounding constant. The parts' sum rounded down, scaled and rounded down again onto
// 1.5 * 2^23 is the pass's floor (every threshold is representable), in the low mantissa bits.
// The first product's output elements are the second one's B elements of the same lane, so
// the row pass computes the transposed product K T^T and nothing moves between lanes.
struct Frag {
  uint32_t h0, l0, h1, l1;  // A: Kh 2^7, Kl, Kh 2^-1, Kl 2^-8, each the columns 2t, 2t + 1 of row g
};

__device__ __forceinline__ uint32_t h2_bits(__half2 h) { return *reinterpret_cast<uint32_t*>(&h); }
__device__ __forceinline__ __half2 bits_h2(uint32_t w) { return *reinterpret_cast<__half2*>(&w); }

__device__ __forceinline__ Frag idct_frag(int r, int lane) {
  const int g = lane >> 2, t = lane & 3;
  const int ka = idct_k(g, 2 * t, r), kb = idct_k(g, 2 * t + 1, r);
  const int ha = (ka + 64) >> 7, hb = (kb + 64) >> 7;
  const float la = (float)(ka - ha * 128), lb = (float)(kb - hb * 128);
  Frag f;
  f.h0 = h2_bits(__floats2half2_rn(ha * 128.f, hb * 128.f));
  f.l0 = h2_bits(__floats2half2_rn(la, lb));
  f.h1 = h2_bits(__floats2half2_rn(ha * 0.5f, hb * 0.5f));
  f.l1 = h2_bits(__floats2half2_rn(la * (1.f / 256), lb * (1.f / 256)));
  return f;
}

constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23

// K X of the lane's B elements (rows 2t, 2t + 1 of column g) given as packed int16 plus 2^15,
// plus bias, times 2^-8: the two parts of elements (g, 2t), (g, 2t + 1).
__device__ __forceinline__ float4 idct_product(const Frag& f, uint32_t x, float bias) {
  const uint32_t xl = h2_bits(__hsub2(bits_h2(__byte_perm(x, 0x64646464u, 0x4240)), bits_h2(0x64006400u)));
  const uint32_t xh = h2_bits(__hsub2(bits_h2(__byte_perm(x, 0x64646464u, 0x4341)), bits_h2(0x64806480u)));
  float4 c = make_float4(bias, bias, 0.f, 0.f);
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c.x), "+f"(c.y), "+f"(c.z), "+f"(c.w)
      : "r"(f.h0), "r"(f.l0), "r"(f.h1), "r"(f.l1), "r"(xh), "r"(xl));
  return c;
}

// Row pass from the lane's column-pass results (row g, columns 2t, 2t + 1, packed int16 plus
// 2^15): clamp(floor((sum + 2^18) / 2^19) + 128, 0, 255) of its pixels (rows 2t, 2t + 1,
// column g) in the halves of a word. The saturating multiply clamps to [0, 256], the packed
// minimum to 255.
__device__ __forceinline__ uint32_t row_pass(const Frag& f, uint32_t t) {
  const float4 c = idct_product(f, t, 1024.0f + 262144.0f);
  const float a = __saturatef(__fadd_rd(c.x, c.z) * (1.0f / 524288)), b = __saturatef(__fadd_rd(c.y, c.w) * (1.0f / 524288));
  const uint32_t p = __byte_perm(__float_as_uint(__fmaf_rd(a, 256.0f, kMagic)),
                                 __float_as_uint(__fmaf_rd(b, 256.0f, kMagic)), 0x5410);
  return __viaddmin_s16x2(p, 0u, 0x00FF00FFu);
}

__device__ __forceinline__ int sat16(int v) { return min(32767, max(-32768, v)); }

// Column pass of any coefficients: t = clamp16(floor((sum + 2^8) / 2^9)) of d = clamp16(q Q);
// q, Q: the lane's two coefficients and their steps.
__device__ __forceinline__ uint32_t column_pass_any(const Frag& f, int qa, int qb, int Qa, int Qb) {
  const uint32_t x = __byte_perm((uint32_t)(sat16(qa * Qa) + 32768), (uint32_t)(sat16(qb * Qb) + 32768), 0x5410);
  const float4 c = idct_product(f, x, 1.0f);
  const float a = fminf(fmaxf(__fadd_rd(c.x, c.z), -65536.0f), 65535.99609375f);
  const float b = fminf(fmaxf(__fadd_rd(c.y, c.w), -65536.0f), 65535.99609375f);
  return __byte_perm(__float_as_uint(__fmaf_rd(a, 0.5f, kMagic + 32768.0f)),
                     __float_as_uint(__fmaf_rd(b, 0.5f, kMagic + 32768.0f)), 0x5410);
}

// Column pass of small dequantised coefficients, exact in fp16 as they are (one product of
// depth 8, no split of X): |DC| <= kSmallDc, |AC| <= kSmallAc, so that |t| <=
// (5793 * 1200 + 37491 * 256) / 2^9 < 2^15 needs no clamp and every sum stays below 2^24.
constexpr float kSmallDc = 1200.0f, kSmallAc = 256.0f;
__device__ __forceinline__ uint32_t column_pass_small(const Frag& f, __half2 x) {
  float4 c = make_float4(256.0f, 256.0f, 0.f, 0.f);
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
      : "+f"(c.x), "+f"(c.y), "+f"(c.z), "+f"(c.w)
      : "r"(f.h0), "r"(f.l0), "r"(h2_bits(x)));
  return __byte_perm(__float_as_uint(__fmaf_rd(c.x + c.z, 1.0f / 512, kMagic + 32768.0f)),
                     __float_as_uint(__fmaf_rd(c.y + c.w, 1.0f / 512, kMagic + 32768.0f)), 0x5410);
}

// What a lane needs of an MCU's quantisation tables: the steps of its two coefficients (luma,
// chroma), as integers and as fp16 pairs.
struct Steps {
  int la, lb, ca, cb;
  __half2 l, c;
};

// Pixels (rows 2t, 2t + 1, column g) of an MCU's NDU data units, coefficients at shared offset
// coef. Data units go through the small form when all of the MCU's do: quantised values in
// [-512, 511] (so that 1536 + q is exact in fp16 and its exponent field says so) and the
// bounds of column_pass_small (a step above 2048 is infinite or inexact in fp16, and any
// product with it then fails the bound; with q = 0 a finite step gives 0).
template <int NDU>
__device__ __forceinline__ void mcu_idct(const Frag& f, uint32_t coef, uint32_t oa, uint32_t ob, const Steps& Q,
                                         __half2 bound, uint32_t (&p)[NDU]) {
  __half2 x[NDU], worst = __float2half2_rn(0.f);
  uint32_t odd = 0;
#pragma unroll
  for (int d = 0; d < NDU; ++d) {
    const uint32_t q = __byte_perm((uint32_t)(uint16_t)sm_i16(coef + 128 * d + oa), (uint32_t)(uint16_t)sm_i16(coef + 128 * d + ob), 0x5410);
    const uint32_t h = __viaddmax_s16x2(q, 0x66006600u, 0x80008000u);  // 1536 + q
    odd |= h ^ 0x64006400u;
    x[d] = __hmul2(__hsub2(bits_h2(h), bits_h2(0x66006600u)), d < NDU - 2 ? Q.l : Q.c);
    worst = __hmax2_nan(worst, __habs2(x[d]));
  }
  const bool small = (odd & 0xFC00FC00u) == 0 && __hble2(worst, bound);
  if (__all_sync(0xFFFFFFFFu, small)) {
#pragma unroll
    for (int d = 0; d < NDU; ++d) p[d] = row_pass(f, column_pass_small(f, x[d]));
  } else {
#pragma unroll
    for (int d = 0; d < NDU; ++d)
      p[d] = row_pass(f, column_pass_any(f, sm_i16(coef + 128 * d + oa), sm_i16(coef + 128 * d + ob),
                                         d < NDU - 2 ? Q.la : Q.ca, d < NDU - 2 ? Q.lb : Q.cb));
  }
}

// RGBA8 of two texels: luma and offsets in the halves of y, ro, go, bo.
__device__ __forceinline__ uint2 texel_pair(uint32_t y, uint32_t ro, uint32_t go, uint32_t bo) {
  const uint32_t m = 0x00FF00FFu;
  const uint32_t r = __viaddmin_s16x2_relu(y, ro, m), g = __viaddmin_s16x2_relu(y, go, m),
                 b = __viaddmin_s16x2_relu(y, bo, m);
  const uint32_t rg = __byte_perm(r, g, 0x6240), ba = __byte_perm(b, 0xFFFFFFFFu, 0x4240);
  return make_uint2(__byte_perm(rg, ba, 0x5410), __byte_perm(rg, ba, 0x7632));
}

// (R, G, B) offsets of one chroma pair times 2^16 (JFIF in 16-bit fixed point; the upper half
// of each word is the offset).
__device__ __forceinline__ void chroma_offsets(int cb, int cr, uint32_t& r, uint32_t& g, uint32_t& b) {
  r = (uint32_t)(91881 * cr + (32768 - 91881 * 128));
  g = (uint32_t)(-22554 * cb - 46802 * cr + (32768 + (22554 + 46802) * 128));
  b = (uint32_t)(116130 * cb + (32768 - 116130 * 128));
}

// IDCT, colour and tile of one MCU by the whole warp. coef: shared offset of its
// coefficients; tile: its cache block, (mw >> r)^2 texels. RED: a reduced level, only pixels
// below N = 8 >> r of each data unit exist.
template <bool S420, bool RED>
__device__ __forceinline__ void mcu_pixels(const Frag& f, uint32_t coef, uint32_t oa, uint32_t ob, const Steps& Q,
                                           __half2 bound, int r, uint32_t* tile, int lane) {
  const int g = lane >> 2, t = lane & 3;
  const int n = RED ? 8 >> r : 8;
  const bool in0 = !RED || (g < n && 2 * t < n), in1 = !RED || (g < n && 2 * t + 1 < n);
  if (S420) {
    uint32_t p[6];
    mcu_idct<6>(f, coef, oa, ob, Q, bound, p);
    const uint32_t cc = __byte_perm(p[4], p[5], 0x6420);  // Cb of rows 2t and 2t + 1, then Cr
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      // texels (di n + 2t + e, dj n + g) use chroma sample (row, col) = half of that
      const int di = d >> 1, dj = d & 1;
      const int row = (di * n >> 1) + t, col = (dj * n >> 1) + (g >> 1);
      const uint32_t w = __shfl_sync(0xFFFFFFFFu, cc, (col * 4 + (row >> 1)) & 31);
      const uint32_t sel = 0x4440u + (uint32_t)(row & 1);
      uint32_t ro, go, bo;
      chroma_offsets((int)__byte_perm(w, 0, sel), (int)__byte_perm(w, 0, sel + 2), ro, go, bo);
      const uint2 px = texel_pair(p[d], __byte_perm(ro, 0, 0x3232), __byte_perm(go, 0, 0x3232), __byte_perm(bo, 0, 0x3232));
      uint32_t* o = tile + (di * n + 2 * t) * (2 * n) + dj * n + g;
      if (in0) o[0] = px.x;
      if (in1) o[2 * n] = px.y;
    }
  } else {
    uint32_t p[3];
    mcu_idct<3>(f, coef, oa, ob, Q, bound, p);
    uint32_t r0, g0, b0, r1, g1, b1;
    chroma_offsets((int)(p[1] & 255u), (int)(p[2] & 255u), r0, g0, b0);
    chroma_offsets((int)(p[1] >> 16), (int)(p[2] >> 16), r1, g1, b1);
    const uint2 px = texel_pair(p[0], __byte_perm(r0, r1, 0x7632), __byte_perm(g0, g1, 0x7632), __byte_perm(b0, b1, 0x7632));
    uint32_t* o = tile + 2 * t * n + g;
    if (in0) o[0] = px.x;
    if (in1) o[n] = px.y;
  }
}

// UNITS: the variant for contexts with data-unit starts. Each MCU of a batch then takes six
// lanes, lane 6m + d decoding data unit d of MCU m from its own start (levels without
// starts are decoded whole by lane 6m); MCUs per batch are at most 4.
// LONG: the variant that takes long lists in batches of twice the width.
template <bool UNITS, bool LONG>
__global__ void __launch_bounds__(512, 1) k_decode(const __grid_constant__ DecodeArgs a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int M = a.mcus_per_warp;
  const uint32_t coef0 = kStagedTables + (uint32_t)warp * (uint32_t)warp_smem(M);
  // this lane's MCU slot and data unit (the whole MCU outside the unit variant)
  const int lm = UNITS ? lane / 6 : lane, ld = UNITS ? lane % 6 : 0;
  const int max_batch = UNITS ? min(M, 4) : M;

  // stages set i of the Huffman tables when it fits; kNoSet when it does not
  auto stage_set = [&](uint32_t i) {
    const uint32_t used = __ldg(&a.huff[i].used);
    if (used > kStagedTables) return kNoSet;
    for (uint32_t j = threadIdx.x; j < (used + 15) / 16; j += blockDim.x)
      reinterpret_cast<uint4*>(smem)[j] = __ldg(reinterpret_cast<const uint4*>(a.huff + i) + j);
    return i;
  };
  // a context's only set is staged before the wait for the kernel before (it was written at
  // upload)
  uint32_t staged = a.nsets == 1 ? stage_set(0) : kNoSet;
  // the lane's two coefficients of a data unit and its transform fragments
  const int fg = lane >> 2, ft = lane & 3;
  const uint32_t oa = 2 * (uint32_t)zz_pos(2 * ft, fg), ob = 2 * (uint32_t)zz_pos(2 * ft + 1, fg);
  const Frag f8 = idct_frag(0, lane);
  const __half2 bound = __floats2half2_rn(lane == 0 ? kSmallDc : kSmallAc, kSmallAc);
  __syncthreads();
  pdl_wait();  // the work list, slots and counts come from the compaction or the cache update

  const uint32_t count = min(*(volatile uint32_t*)&a.state->count, a.work_cap);
  bool any_bad = false;
  // MCUs per batch: the smallest power of two <= M that covers the list in one batch for each
  // of kBusyWarps warps of a CTA: short lists spread one MCU per warp (latency), long ones fill
  // the lanes, and between them few warps with more lanes beat more warps (their chains share
  // the issue slots): 27 MCUs per SM took 59.5 us a frame with 7 warps of 4 against 61.2 with 14 of 2.
  // The first batches are fixed: dealt warp by warp over the CTAs, so that neighbours (alike in
  // length) fall on different SMs, or, with several sets of Huffman tables, in runs of
  // neighbours, so that a CTA's MCUs mostly share a texture and with it the staged set. What
  // they leave of a long list is handed out by a counter.
  const uint32_t warps = blockDim.x >> 5, run = (count + gridDim.x - 1) / gridDim.x;
  const uint32_t busy = min(warps, kBusyWarps), per_warp = (run + busy - 1) / busy;
  int meff = 1;
  while ((uint32_t)meff < per_warp && meff < max_batch) meff *= 2;
  if (LONG && 2 * M <= 32 && run >= kLongRun * warps * (uint32_t)M) meff = 2 * M;
  const bool runs = a.nsets > 1;
  const uint32_t span = runs ? min(run, warps * (uint32_t)meff) : warps * (uint32_t)meff;
  const uint32_t first = blockIdx.x * span;
  if (runs) {  // stage the set of the CTA's first MCU
    uint32_t i = kNoSet;
    if (first < count) {
      const uint32_t d = __ldg(a.desc_of_gid + __ldg(a.work + first));
      if (d < a.ndesc) i = a.descs[d].hset;
    }
    if (i != kNoSet) staged = stage_set(i);
    __syncthreads();
  }
  const bool staged_cap = staged != kNoSet && __ldg(&a.huff[staged].capped) != 0;

#pragma unroll 1
  for (uint32_t it = 0;; ++it) {
    uint32_t base = runs ? first + (uint32_t)(warp * meff) : ((uint32_t)warp * gridDim.x + blockIdx.x) * (uint32_t)meff;
    uint32_t limit = runs ? min(first + span, count) : count;
    if (it != 0) {
      if (run <= span) break;  // the first batches covered the list
      uint32_t b = 0;
      if (lane == 0) b = atomicAdd(&a.state->decode_next, (uint32_t)meff);
      base = __shfl_sync(0xFFFFFFFFu, b, 0) + gridDim.x * span;
      limit = count;
    }
    if (base >= limit) break;

    auto clear = [&](int bytes) {
      uint4* z = reinterpret_cast<uint4*>(smem + coef0);
      const int nz = (bytes + 15) / 16;
#pragma unroll 4
      for (int i = lane; i < nz; i += 32) z[i] = make_uint4(0, 0, 0, 0);
    };
    clear(LONG && meff > M ? 2 * M * kMcuBytes444 : meff * kMcuBytes);  // the first part's coefficients

    // ---- set-up: lanes of MCU slot m < m_eff take item base + m ----
    const uint32_t item = base + lm;
    bool act = lm < meff && item < limit;
    bool unit = false;  // this lane decodes data unit ld only
    const uint32_t gid = act ? __ldg(a.work + item) : 0u;
    const uint32_t di = act ? __ldg(a.desc_of_gid + gid) : 0u;
    int ndu = 0;
    bool s420 = true, store = false;
    uint32_t off = 0, nbits = 0, bitpos = 0, endbit = 0, nwords = 0;
    bool cpt = false;
    int red = 0;  // reduced-resolution level: 1/2^red
    const uint32_t* words = nullptr;
    uint32_t qs = 0;  // the MCU's quantisation table set
    int16_t pr0 = 0, pr1 = 0, pr2 = 0;
    const HuffSet* hs = a.huff;
    bool staged_set = false;  // its Huffman tables are the staged ones
    if (act && di < a.ndesc) {
      const DevDesc d = a.descs[di];
      const uint32_t mcu = gid - d.gid_base;
      if (d.sampling == kSamplingCoef || mcu >= d.nmcu) {
        act = false;  // not a JPEG level: nothing to decode
      } else {
        s420 = d.sampling == kSampling420;
        ndu = s420 ? 6 : 3;
        off = __ldg(a.slot + gid);
        store = off + d.units <= a.cap_units;
        cpt = d.compact != 0;
        red = d.reduce;
        if (cpt) {
          // compact form (Sec. 5.1, 5.3): byte offsets from the two-level table, the three
          // stored DCs from the MCU's 36-bit record (at a multiple of 4 bits, so two words)
          const uint32_t ng = (d.nmcu + 8) / 9;
          const uint32_t* ab = reinterpret_cast<const uint32_t*>(d.index);
          const uint16_t* rl = d.index + 2 * (size_t)ng;
          const uint32_t* rec = ab + 5 * (size_t)ng;
          auto start = [&](uint32_t m) {
            const uint32_t j = m / 9, i = m - 9 * j;
            return 8u * (__ldg(ab + j) + (i ? (uint32_t)__ldg(rl + 8 * j + i - 1) : 0u));
          };
          bitpos = start(mcu);
          endbit = mcu + 1 < d.nmcu ? start(mcu + 1) : d.nbits;
          const uint64_t at = 36ull * mcu;
          const uint64_t r = ((uint64_t)__ldg(rec + (at >> 5)) | ((uint64_t)__ldg(rec + (at >> 5) + 1) << 32)) >>
                             (at & 31);
          pr0 = (int16_t)((int32_t)((uint32_t)r << 20) >> 20);  // 12-bit two's complement
          pr1 = (int16_t)((int32_t)((uint32_t)(r >> 12) << 20) >> 20);
          pr2 = (int16_t)((int32_t)((uint32_t)(r >> 24) << 20) >> 20);
        } else {
          const uint16_t* ix = d.index + (size_t)mcu * 5;
          bitpos = (uint32_t)__ldg(ix) | ((uint32_t)__ldg(ix + 1) << 16);
          pr0 = (int16_t)__ldg(ix + 2);
          pr1 = (int16_t)__ldg(ix + 3);
          pr2 = (int16_t)__ldg(ix + 4);
          endbit = mcu + 1 < d.nmcu ? ((uint32_t)__ldg(ix + 5) | ((uint32_t)__ldg(ix + 6) << 16)) : d.nbits;
          if (UNITS && d.du_index != nullptr) {  // this lane's data unit and its bit range
            unit = true;
            const uint16_t* du = d.du_index + (size_t)mcu * (ndu - 1);
            const uint32_t mcu0 = bitpos;
            if (ld >= ndu) act = false;
            if (ld > 0 && ld < ndu) bitpos = mcu0 + __ldg(du + ld - 1);
            if (ld + 1 < ndu) endbit = mcu0 + __ldg(du + ld);
          }
        }
        if (UNITS && !unit && ld != 0) act = false;  // decoded whole by the MCU's first lane
        words = d.stream;
        nwords = d.nwords;
        nbits = d.nbits;
        hs = a.huff + d.hset;
        staged_set = d.hset == staged;
        qs = d.qset;
      }
    } else {
      act = false;
    }
    // A batch of more than M (of a long list) goes as one part when all of its MCUs are 4:4:4
    // (packed), and in parts of M otherwise.
    const bool packed = LONG && meff > M && !__any_sync(0xFFFFFFFFu, act && s420);
    const int part_mcus = packed || !LONG ? meff : min(meff, M);
    const uint32_t stride = packed ? kMcuBytes444 : kMcuBytes;
    const uint32_t stage0 = coef0 + (packed ? 2u * kMcuBytes444 : (uint32_t)kMcuBytes) * (uint32_t)M;
    const uint32_t pool = (coef0 + (uint32_t)warp_smem(M) - stage0) / 4;
#pragma unroll 1
    for (int part = 0; part < (LONG ? meff : 1); part += part_mcus) {
      const bool in_part = lm >= part && lm < part + part_mcus, on = act && (!LONG || in_part);
      const uint32_t mine = coef0 + (in_part ? (uint32_t)(lm - part) * stride : 0u);
      if (part != 0) clear(M * kMcuBytes);
      if (LONG) __syncwarp();  // (the packed clear ends inside the other form's stage)
      // ---- entropy phase: each active lane decodes all data units of its MCU (or, with
      // data-unit starts, one data unit), in rounds of staging and decoding (one round unless
      // the batch's words exceed the pool) ----
      int nd = ndu, nl = ndu - 2, seq = s420 ? (cpt ? kSeqCompact420 : kSeq420) : (cpt ? kSeqCompact444 : kSeq444);
      uint32_t dst = mine;
      if (UNITS && unit) {
        nl = ld < nl ? 1 : 0;
        nd = 1;
        seq = nl ? kSeqLuma : kSeqChroma;
        dst += 128 * (uint32_t)ld;
      }
      Chain ch{bitpos, kFresh, 0u, (uint32_t)(seq * sizeof(HuffSeq)), (uint32_t)((seq + nd) * sizeof(HuffSeq)), dst};
      int reached = ndu;  // data units whose DC difference was decoded
      bool more = on;
#pragma unroll 1
      do {
        // the chain's words: from its next one (16 B aligned) to the next MCU's start plus the
        // window's look-ahead (3 words)
        const uint32_t w0 = (ch.pos >> 5) & ~3u;
        uint32_t all = (max(endbit, ch.pos) >> 5) + 3 - w0;
        all = (all + 3) & ~3u;
        if (w0 + all > nwords) all = nwords > w0 ? (nwords - w0) & ~3u : 0u;
        if (!more) all = 0;
        // share the warp's stage pool out by a prefix sum of the lanes' word counts, in equal
        // shares when they exceed it (at least 12 words: a group of symbols from any bit of the
        // first four ends inside them, so the first unfinished chain always advances)
        uint32_t want = all;
        if (__reduce_add_sync(0xFFFFFFFFu, all) > pool)
          want = min(all, max(pool / (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, all != 0)) & ~3u, 12u));
        uint32_t sbeg = want;
#pragma unroll
        for (int dlt = 1; dlt < 32; dlt <<= 1) {
          const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, sbeg, dlt);
          if (lane >= dlt) sbeg += o;
        }
        sbeg -= want;  // exclusive
        const uint32_t nst = sbeg >= pool ? 0u : min(want, pool - sbeg);
        if (more) {
          const uint4* src4 = reinterpret_cast<const uint4*>(words + w0);
          uint4* dst4 = reinterpret_cast<uint4*>(smem + stage0 + 4 * sbeg);
#pragma unroll 1
          for (uint32_t j = 0; j < nst / 4; j += 4) {
            uint4 r[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) r[t] = j + t < nst / 4 ? __ldg(src4 + j + t) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int t = 0; t < 4; ++t)
              if (j + t < nst / 4) dst4[j + t] = make_uint4(bswap(r[t].x), bswap(r[t].y), bswap(r[t].z), bswap(r[t].w));
          }
        }
        __syncwarp();
        const bool whole = nst >= all;  // staged to its end
        if (more && (whole || nst >= 12)) {
          const uint32_t st = stage0 + 4 * sbeg, limit = whole ? 0xFFFFFFFFu : 8 * st + 32 * nst - kGroupBits;
          bool ok = all != 0;
          if (ok)
            ok = !staged_set  ? entropy_fast<false, true>(ch, st, w0, limit, hs)
                 : staged_cap ? entropy_fast<true, true>(ch, st, w0, limit, hs)
                              : entropy_fast<true, false>(ch, st, w0, limit, hs);
          more = ok && ch.q != ch.qend;
          if (!more) {
            uint64_t end = 32ull * w0 + (ch.pos - 32 * w0);  // after the last symbol
            // an invalid symbol, or bits past the stage: from the start again, word by word
            if (!ok || ch.pos - 32 * w0 + 32 > 32 * nst) {
              const uint32_t f = (bitpos >> 5) & ~3u;
              const uint32_t r = entropy_any(words + f, nwords > f ? nwords - f : 0u, bitpos - 32 * f, hs, nd, nl, cpt, dst);
              ok = r < kInvalid;
              end = 32ull * f + r;
              if (!ok && !unit) reached = (int)(r - kInvalid);
            }
            // the coding must be valid and end inside the stream; a compact MCU inside its own
            // bytes, a data unit at or before the next one's start
            if (!ok || end > ((cpt || unit) ? endbit : nbits)) any_bad = true;
          }
        }
        __syncwarp();
      } while (__any_sync(0xFFFFFFFFu, more));
      __syncwarp();
      if (on && ld == 0) {  // chain the DC differences (modulo 2^16)
        uint32_t o = mine;
        int c0 = pr0;
#pragma unroll 1
        for (int d = 0; d < min(ndu - 2, reached); ++d, o += 128) {
          c0 = (int16_t)(uint16_t)(c0 + (int)sm_i16(o));
          sm_i16(o) = (int16_t)c0;
        }
        if (reached > ndu - 2) sm_i16(o) = (int16_t)(uint16_t)((int)pr1 + (int)sm_i16(o));
        if (reached > ndu - 1) sm_i16(o + 128) = (int16_t)(uint16_t)((int)pr2 + (int)sm_i16(o + 128));
      }
      // ---- pixel phase: the warp takes the batch's MCUs one by one ----
      const uint32_t minfo = (on && store ? 1u : 0u) | (s420 ? 2u : 0u) | ((uint32_t)red << 2) | (qs << 8);
      __syncwarp();  // every lane's coefficients are visible to the warp
      Steps Q{};
      Frag fr = f8;  // fragments of the last reduced level
      int rcur = 0;
      uint32_t qcur = 0xFFFFFFFFu;
#pragma unroll 1
      for (int m = 0; m < part_mcus; ++m) {
        const uint32_t im = __shfl_sync(0xFFFFFFFFu, minfo, UNITS ? 6 * m : part + m);
        const uint32_t om = __shfl_sync(0xFFFFFFFFu, off, UNITS ? 6 * m : part + m);
        if (!(im & 1u)) continue;
        if (im >> 8 != qcur) {
          qcur = im >> 8;
          const uint16_t* q = a.quant + (size_t)qcur * 128;
          Q.la = __ldg(q + oa / 2);
          Q.lb = __ldg(q + ob / 2);
          Q.ca = __ldg(q + 64 + oa / 2);
          Q.cb = __ldg(q + 64 + ob / 2);
          Q.l = __floats2half2_rn(fminf((float)Q.la, 32768.f), fminf((float)Q.lb, 32768.f));
          Q.c = __floats2half2_rn(fminf((float)Q.ca, 32768.f), fminf((float)Q.cb, 32768.f));
        }
        const uint32_t cm = coef0 + (uint32_t)m * stride;
        uint32_t* tile = reinterpret_cast<uint32_t*>(a.cache + (size_t)om * kUnitBytes);
        const int rm = (int)((im >> 2) & 3u);
        if (rm == 0) {
          if (im & 2u)
            mcu_pixels<true, false>(f8, cm, oa, ob, Q, bound, 0, tile, lane);
          else
            mcu_pixels<false, false>(f8, cm, oa, ob, Q, bound, 0, tile, lane);
        } else {
          if (rm != rcur) {
            rcur = rm;
            fr = idct_frag(rm, lane);
          }
          if (im & 2u)
            mcu_pixels<true, true>(fr, cm, oa, ob, Q, bound, rm, tile, lane);
          else
            mcu_pixels<false, true>(fr, cm, oa, ob, Q, bound, rm, tile, lane);
        }
      }
      __syncwarp();  // the buffers are cleared for the next items
    }
  }
  if (any_bad) atomicOr(&a.state->err, JT_DEVERR_CORRUPT);
}

size_t smem_bytes(int warps, int M) { return kStagedTables + (size_t)warps * warp_smem(M) + kSlackBytes; }

template <bool UNITS, bool LONG>
int occupancy_of(int warps, int M) {
  const size_t smem_b = smem_bytes(warps, M);
  if (smem_b > 227 * 1024) return 0;
  if (cudaFuncSetAttribute(k_decode<UNITS, LONG>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_decode<UNITS, LONG>, warps * 32, smem_b) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

}  // namespace

size_t decode_smem_bytes(int warps, int mcus_per_warp) { return smem_bytes(warps, mcus_per_warp); }

// The dynamic shared-memory attribute of the variants is set by decode_max_ctas_per_sm(),
// which the context calls for every (warps, M) on its device before the first launch.
//
// The variant for long lists serves contexts whose lists can be long: as many MCUs and cache units
// as kLongRun full batches for every warp. It takes 32 MCUs a batch, so that the set-up's dependent
// loads serve twice as many, and packs 4:4:4 ones, so that all lanes decode: 1440 -> 1376 us for
// eight 4096^2 textures to pixels, half of them 4:4:4 (1.3 M MCUs). It is a kernel of its own
// because the parts cost a short list time (1080p frame 54.4 -> 54.9 us in one kernel), which a
// short list of a context that can have long ones still pays: the host does not know a list's length.
// Hence the line at ten full batches a warp, well above where the two forms meet (textures to pixels
// with every list taken as the one kind or the other, default shape: 1.2 batches 78.2 us, 84.9 as long;
// 2.4 111.1, 112.6; 4.8 221.2, 213.5; 9.6 391.1, 381.1; 19 733, 705; 38 1425, 1361).
void launch_decode(const DecodeArgs& a, int warps, int grid, cudaStream_t s) {
  const size_t smem_b = smem_bytes(warps, a.mcus_per_warp);
  const uint64_t most = std::min<uint64_t>(a.ngid, a.cap_units), batch = (uint64_t)grid * (uint32_t)(warps * a.mcus_per_warp);
  if (a.unit_mode)
    launch_pdl(k_decode<true, false>, grid, warps * 32, smem_b, s, a);
  else if (most >= kLongRun * batch)
    launch_pdl(k_decode<false, true>, grid, warps * 32, smem_b, s, a);
  else
    launch_pdl(k_decode<false, false>, grid, warps * 32, smem_b, s, a);
}

// Resident CTAs per SM that every variant reaches (the launch picks one per frame).
int decode_max_ctas_per_sm(int warps, int mcus_per_warp) {
  return std::min({occupancy_of<false, false>(warps, mcus_per_warp), occupancy_of<false, true>(warps, mcus_per_warp),
                   occupancy_of<true, false>(warps, mcus_per_warp)});
}

void idct_constants(int out[8]) {
  const int c[8] = {0, C1, C2, C3, C4, C5, C6, C7};
  for (int i = 0; i < 8; ++i) out[i] = c[i];
}

}  // namespace jt
