// Internal device-side data model of the texture path (shared by the kernels and the
// host implementation of the C ABI in jt_api.cu).
//
// HBM layout
//   descs      DevDesc[ndesc]        one per uploaded (texture, level), sorted by gid_base
//   pix        PixRec[(ntex + 1) * 17]  (tex_id, level) -> the screen passes' record
//   streams    per level: uint32 words of the unstuffed entropy stream + >= 64 zero bytes
//   index      per level: packed 10-byte {bit_offset, dc_pred[3]} entries
//   huff       HuffSet[nh]           decode tables, deduplicated by content
//   quant      uint16[nq][2][64]     quantisation tables in zig-zag order
//   flags      uint8[ngid]           per-frame marks: cache units of the MCU (4, 1) or 0
//   slot       uint32[ngid]          cache-unit offset of each needed gid
//   work       uint32[ngid]          work list (needed gids, ascending)
//   cache      uint8[cap_units*256]  RGBA8 tiles; a 4:2:0 MCU = 4 units, 4:4:4 = 1 unit
//   state      FrameState            counts, work counter, error word
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "jt.h"

namespace jt {

// ---- programmatic dependent launch ----
// The frame's compaction (or cache update) and decode are launched with programmatic stream
// serialisation (colourise is not: its CTAs, launched early, would wait on the SMs the decode
// is using, and the 4K frame measured 0.181 ms with it against 0.176 ms without):
// a kernel may start while the one before it in the stream is still running, and waits on
// the device (pdl_wait) before it reads or writes anything an earlier kernel of the stream
// produces or consumes. Each kernel lets its dependents launch as soon as it starts
// (pdl_launch_dependents); a dependent's CTAs are only scheduled once every CTA of the
// running grid has started, so they never hold resources that grid still needs. Without
// the attribute (or after a non-kernel operation) both instructions are no-ops.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

constexpr int kLutBits = 10;                 // first-level Huffman LUT: next 10 bits
constexpr int kLutSize = 1 << kLutBits;
constexpr int kLut2Size = 256 * 32 + 8;      // entries for longer codes: 256 codes of up to 32 prefixes, one empty
constexpr int kStreamPadBytes = 64;          // zero padding after each entropy stream
constexpr uint32_t kUnitBytes = 256;         // cache unit
constexpr int kSampling420 = 0, kSampling444 = 1, kSamplingCoef = 2;

// Decode tables of one set of four Huffman specs (T.81 Annex C canonical codes; DC luma, AC
// luma, DC chroma, AC chroma). A symbol entry is 16 bits:
//   bits 0..4    code length plus value bits s (at most 27)
//   bits 5..8    s
//   bits 10..15  run r: AC value (r, s) -> store at k + r, advance k by r + 1; ZRL (15, 0) ->
//                advance 16; EOB (63, 0); DC (0, s). The top field, so that an entry added to
//                k << 10 gives the coefficient's place there.
// The s value bits follow the code in the stream; the decoder cuts them from its window
// itself (T.81 EXTEND), so an entry depends on the code alone. kNoEntry marks the rest: value
// bits and a run that is past slot 63 from any k.
//
// A table's entries are one array over two granularities. Codes of at most kLutBits bits are
// indexed by the next kLutBits bits w >> 22. In canonical order the longer codes are the
// numerically largest: they start at the 16-bit left-aligned prefix `first` (a multiple of
// 64), and their entries, one per 16-bit prefix, start where the short ones end, at
// first >> 6. The index of any code is then max(w >> 22, (w >> 16) + d) with
// d = (first >> 6) - first: the second term grows 64 times as fast and passes the first one
// exactly at `first`. So a symbol is one read, without a branch or a select. Every code has its
// entry, kNoEntry in the place of invalid codes and of symbols invalid for the table's class (DC
// category > 11, AC size > 10, AC size 0 with a run other than 0 or 15). With room for 4096 entries
// of longer codes, MCUs that met one of a table with more went through the general chain: 154
// codes of 11 bits, decode of 576 MCUs 53.4 us (now 17.4), of 23,040 90.5 us (33.6).
__host__ __device__ constexpr uint16_t huff_entry(uint32_t l, uint32_t s, uint32_t r) {
  return (uint16_t)((l + s) | (s << 5) | (r << 10));
}
constexpr uint32_t kRunEob = 63;
constexpr int kRunShift = 10;
constexpr uint16_t kNoEntry = 0xFFE0;

// Index in a table of the entry for window w. CAP: a table that needs its cap (see below). The cap
// comes after the maximum: capping both terms side by side shortens the chain of such tables (small
// frames 0.7 % faster), but in the kernel that all tables share it cost the others 0.3 %.
template <bool CAP>
__host__ __device__ __forceinline__ uint32_t table_index(uint32_t w, int d, int cap) {
  const int t = (int)(w >> 16), i = (int)(w >> (32 - kLutBits));
#ifdef __CUDA_ARCH__
  const int x = __viaddmax_s32(t, d, i);
#else
  const int x = t + d > i ? t + d : i;
#endif
  return (uint32_t)(CAP && x > cap ? cap : x);
}

// A code that leaves prefixes unused above its last one (`end`, 65536 for a complete code) has
// entries up to there only, and the index is also capped, at the table's last entry
// (kNoEntry): the index as a whole, because past `end` a table of few long codes is
// shorter than 1 << kLutBits, and there w >> 22 lies beyond it too.
//
// Where one spec's entries are: the byte offset of the first one in the set, d and the last one's index.
struct HuffTable {
  uint32_t base;
  int32_t d, cap;
  uint32_t pad;
};

// The tables a chain of data units uses, one record per data unit and one past the last: those
// of its AC symbols and of the next data unit's first symbol (byte offset in the set, d, cap),
// and the next data unit's first k << kRunShift (k = 1 where the DC is stored apart).
// The last data unit's next table and both of the record past it are the table of zeros.
// start_*: of the data unit's own first symbol.
struct HuffSeq {
  uint32_t ac_base;
  int32_t ac_d;
  uint32_t next_base;
  int32_t next_d;
  uint32_t next_k;
  int32_t ac_cap, next_cap;
  uint32_t pad;
  uint32_t start_base;
  int32_t start_d;
  uint32_t start_k;
  int32_t start_cap;
};
static_assert(sizeof(HuffSeq) == 48, "read as 16-byte words");
// records: 4:2:0 and 4:4:4 MCUs, the same in the compact form, one luma, one chroma data unit
constexpr int kSeq420 = 0, kSeq444 = 7, kSeqCompact420 = 11, kSeqCompact444 = 18, kSeqLuma = 22, kSeqChroma = 24;
constexpr int kSeqRecords = 26;
constexpr int kMaxTableEntries = kLutSize + kLut2Size;

struct HuffSet {
  HuffSeq seq[kSeqRecords];
  uint32_t used;    // bytes from the start of the set to the end of its entries
  uint32_t capped;  // some table needs its cap
  uint32_t pad[2];
  uint16_t none[kLutSize];               // zeros: a symbol without value, run or length
  uint16_t lut[4 * kMaxTableEntries];  // the four tables' entries, back to back
  HuffTable table[4];
};
static_assert(sizeof(HuffSet) % 16 == 0 && offsetof(HuffSet, lut) % 16 == 0, "copied in 16-byte words");
// A decode CTA stages one set in shared memory when it is at most this long (the typical tables
// of the standard take 12,828 bytes).
constexpr uint32_t kStagedTables = 18432;

struct DevDesc {
  const uint32_t* stream;      // big-endian words (word i = bytes 4i..4i+3)
  // standard form: packed 10-byte entries, read as 5 halfwords. Compact form: the side
  // table [abs uint32 x G][rel uint16 x 8G][DC records uint32 x (ceil(36 n / 32) + 1)],
  // G = ceil(n / 9)
  const uint16_t* index;
  uint32_t gid_base;
  uint32_t nmcu;
  uint32_t nwords;             // readable words including padding
  uint32_t nbits;              // coded bits
  uint16_t width, height;
  uint16_t mcus_x, mcus_y;
  uint8_t sampling;            // kSampling420 / kSampling444 / kSamplingCoef
  uint8_t units;               // cache units per MCU: 4 or 1
  uint8_t hset, qset;
  uint8_t compact;             // 1: the compact form (byte-aligned MCUs, stored DCs)
  uint8_t reduce;              // r > 0: tiles at 1/2^r from the lowest N x N frequencies, N = 8 >> r
  uint8_t pad0[2];
  const uint16_t* du_index;    // optional data-unit starts [mcu][ndu - 1] (bits from the MCU start)
  uint64_t pad1;
};
static_assert(sizeof(DevDesc) == 64, "descriptor layout");

struct FrameState {
  uint32_t count;        // needed MCUs after the last compaction
  uint32_t units;        // cache units they occupy
  uint32_t decode_next;  // next work item for the persistent decoder
  uint32_t err;          // JT_DEVERR_* bits
  uint32_t spare;        // unused
  uint32_t pad[3];
};

// Screen passes walk each view in tiles of kTileW x tile_h pixels (one CTA per tile at a
// time, one warp per 128-pixel row segment), so a CTA's pixels share MCUs. High tiles share
// more of them; low ones spread a small frame over the SMs, whose 510 tiles of 1080p leave a
// quarter of the warps idle (frame with 32 rows, 16 and 8: 1080p 55.9, 53.9 and 52.3 us, 4K
// 110.6, 115.1 and 117.5; 1440p with 32 and 8: 68.5 and 72.1). So views of fewer high tiles than
// kFewTilesPerSm CTAs for each SM get low ones.
constexpr int kTileW = 128, kTileHigh = 32, kTileLow = 8;
constexpr uint64_t kFewTilesPerSm = 4, kManyTilesPerSm = 8;

// One view of a (possibly batched) frame, passed by value in the kernel parameters.
struct View {
  const float4* uv;      // two pixels per float4
  const uint16_t* tex;
  const uint8_t* mip;
  uint4* out;            // four RGBA8 pixels per uint4
  uint32_t npx;
  uint32_t quad_begin;   // prefix sum of ceil(npx/4) over earlier views
  int32_t width, height;
  uint32_t tiles_x;      // ceil(width / kTileW)
  uint32_t tile_begin;   // prefix sum of tile counts over earlier views
};

struct ViewSet {
  View v[JT_MAX_VIEWS];
  int n;
  uint32_t total_quads;
  uint32_t total_tiles;
  int tile_h;  // rows of a tile
};

// The screen passes' record of one (texture, level): 32 bytes (two vector loads that hit
// L1, since a warp's pixels mostly share a level), every field in the form the texel
// addressing uses, so no per-pixel branch or decoding is needed. Indexed by
// min(tex, map_ntex) * kPixLevels + min(level, JT_MAX_LEVELS): every texture has one record
// more than it can have levels, and there is one texture more than the table holds, all of
// them zero, as are the records of levels that do not exist (empty pixels, unknown textures
// or levels).
struct PixRec {
  uint32_t gid_base;
  float wf, hf;     // sides as floats
  uint32_t masks;   // (w - 1) | (h - 1) << 16: floor-mod masks of power-of-two sides
  uint32_t mcus_x;
  uint32_t shift;   // log2 of the MCU side in texels
  uint32_t info;    // units | kPixJpeg | kPixCoef | kPixPow2
  uint32_t wh;      // w | h << 16
};
static_assert(sizeof(PixRec) == 32, "screen-pass record layout");
constexpr uint32_t kPixLevels = JT_MAX_LEVELS + 1;
constexpr uint32_t kPixJpeg = 1u << 16;  // an uploaded JPEG level (colourise, mark)
constexpr uint32_t kPixCoef = 1u << 17;  // a coefficient level (the float chain)
constexpr uint32_t kPixPow2 = 1u << 18;  // both sides are powers of two

struct TexLookup {
  const uint4* pix;     // PixRec per (tex, level) as two uint4, indexed as PixRec says
  uint32_t map_ntex;
  uint32_t all_p2;      // every level has power-of-two sides
  uint32_t all_s4;      // every JPEG level has 16-texel MCUs (4:2:0 at full size)
};

// ---- launchers (defined in the kernel translation units) ----
struct MarkArgs {
  ViewSet views;
  TexLookup tl;
  uint8_t* flags;
  FrameState* state;
  int filter;
  int only_tex;   // -1: all textures; otherwise only pixels with this texture id
  bool many;      // high tiles, at least kManyTilesPerSm for each SM
};
void launch_mark(const MarkArgs& a, int threads, int grid, cudaStream_t s);

struct ScanArgs {
  uint8_t* flags;        // flags of gids [gid_lo, gid_lo + n)
  uint32_t gid_lo;
  uint32_t n;
  uint32_t* slot;        // indexed by gid
  uint32_t* work;
  uint32_t work_cap;
  uint64_t* tile_status; // one word per tile: its (count << 32 | units)
  FrameState* state;
  uint32_t cap_units;
};
constexpr int kScanThreads = 256;
constexpr int kScanPerThread = 16;  // one 16-byte load
constexpr int kScanTile = kScanThreads * kScanPerThread;  // 4096 flags
void launch_scan(const ScanArgs& a, cudaStream_t s);  // two launches; tile_status: one word per tile

// Cross-frame block cache (Sec. 4.1, Sec. 4.5): a residency bitmap over the gids; a resident
// gid's slot (4 x its block) is the one the previous frame gave it; free blocks in a ring,
// positions [head, head + free_count) modulo nblocks. A block is 4 cache units. Every counter
// but head, free_count, visible and evicted is zero between frames.
struct CacheState {
  uint32_t head;         // ring position of the first free block
  uint32_t free_count;   // free blocks
  uint32_t taken;        // misses of the current update (blocks asked for)
  uint32_t spare;        // (unused)
  uint32_t evict_n;      // blocks evicted by the current update
  uint32_t visible_acc;  // MCUs the current update has seen needed
  uint32_t done;         // CTAs of the current update that have finished
  uint32_t visible;      // MCUs the last frame needed
  uint32_t evicted;      // blocks evicted since the counter was last cleared
};
struct CacheArgs {
  uint8_t* flags;  // flags[gid], cleared by the update
  uint32_t n;      // gids
  uint16_t* resbits;    // residency bitmap, 16 gids per word ...
  uint32_t* resbits32;  // ... the same memory as 32-bit words (a whole number of them)
  uint32_t* ring;       // [nblocks] free blocks
  uint32_t* deferred;   // [nblocks] misses waiting for a block evicted by the same update
  uint32_t nblocks;
  uint32_t* slot;
  uint32_t* work;
  uint32_t work_cap;
  FrameState* state;
  CacheState* cs;
};
constexpr int kCacheThreads = 256;
void launch_cache_update(const CacheArgs& a, int max_grid, cudaStream_t s);  // one launch

// Scene rasteriser (geometry-pass stand-in): one quad, laid out as jt_scene_quad.
struct SceneQuad {
  float cx[4], cy[4], ex[4], ey[4], h[9], rep, cs, sn, ou, ov;
  int32_t tex, x0, y0, x1, y1;
};
static_assert(sizeof(SceneQuad) == 140, "scene quad layout");
constexpr int kMaxSceneQuads = 4096;
struct RasterArgs {
  int32_t width, height;
  float cam[3], rot[9];
  float ax, ay, tan_x, tan_y, max_t, kx, ky, shift;
  uint64_t cell_seed;
  int32_t ntex, use_mips, nquads;
  int32_t tile_x;             // columns of a CTA's tile
  uint32_t mod_m;             // floor(2^32 / ntex), or 2^32 - 1 for one texture
  const float4* sizes;        // device copies: per texture its level-0 sides and (bits of) its level count,
  const SceneQuad* quads;     // then the quads
  float2* uv;
  uint16_t* tex;
  uint8_t* mip;
};
constexpr int kRasterTileY = 8;  // rows of a CTA's tile
void launch_raster(const RasterArgs& a, cudaStream_t s);

struct DecodeArgs {
  const DevDesc* descs;
  uint32_t ndesc;
  const uint32_t* desc_of_gid;  // descriptor index of each gid
  int mcus_per_warp;      // M, the buffer width: 4, 8, 16 or 32 (batches may be smaller)
  int unit_mode;          // some level has data-unit starts: the kernel that decodes them in parallel
  const HuffSet* huff;    // a CTA stages one of them in shared memory
  uint32_t nsets;
  const uint16_t* quant;  // [nq][2][64] zig-zag order
  const uint32_t* work;
  uint32_t work_cap;
  uint32_t ngid;          // MCUs of the context: no list is longer
  const uint32_t* slot;
  uint8_t* cache;
  uint32_t cap_units;
  FrameState* state;
};
size_t decode_smem_bytes(int warps, int mcus_per_warp);
void launch_decode(const DecodeArgs& a, int warps, int grid, cudaStream_t s);
int decode_max_ctas_per_sm(int warps, int mcus_per_warp);

struct ColorizeArgs {
  ViewSet views;
  TexLookup tl;
  const uint32_t* slot;
  const uint8_t* cache;
  uint32_t cap_units;
  FrameState* state;
  int filter;
  int only_tex;
};
void launch_colorize(const ColorizeArgs& a, int threads, int grid, cudaStream_t s);

// Float chain (differentiable colourise; not in the paper; float_kernels.cu). Coefficient
// textures are 4:2:0 level-0 textures; an MCU is needed when a pixel's taps touch it, and slot[gid]
// is then its position in the work list.
struct FloatArgs {
  ViewSet views;          // one view
  TexLookup tl;
  uint32_t* slot;
  uint32_t* work;
  uint32_t work_cap;
  uint32_t cap_units;     // slots stay below it
  const float* coef;      // [T][my][mx][6][64], natural order k = v*8+u
  uint32_t coef_gid_base; // gid of coefficient texture 0, MCU 0
  uint32_t coef_mcus;     // MCUs of all coefficient textures
  uint32_t tile_cap;      // needed coefficient MCUs a pass serves (more: JT_DEVERR_CAPACITY)
  float* frame;           // [npx][3]: forward output (zero on entry), or the backward's dL/dF
  float* grad_coef;       // [T][my][mx][6][64]: backward output
  FrameState* state;
  // the view's pixels bucketed under the coefficient MCUs their taps touch
  uint32_t* cursor;       // [coef_mcus] counts, then fill cursors; zero between passes
  uint32_t* offset;       // [coef_mcus] first entry of each MCU
  uint64_t* block_sum;    // [ceil(coef_mcus / kFloatScan)] needed MCUs << 32 | entries
  uint4* bucket;          // [bucket_cap] entries
  uint32_t bucket_cap;    // >= 4 pixels of the view (a pixel's taps touch at most 4 MCUs)
  int sms;                // SMs of the device
  int pairs;              // pairs of MCUs per warp of a gather (chosen by its launcher)
  float basis[64];        // A[x][u] = C(u)/2 cos((2x+1)u pi/16), C(0) = 1/sqrt(2); x*8+u
};
// JFIF colour of the float chain: R = Y + kCr2R Cr, G = Y - kCb2G Cb - kCr2G Cr, B = Y + kCb2B Cb
constexpr float kCr2R = 1.402f, kCb2G = 0.344136f, kCr2G = 0.714136f, kCb2B = 1.772f;
constexpr int kFloatWarps = 8;     // warps per CTA of the gathers
constexpr int kForwardCtas = 4, kBackwardCtas = 5;    // CTAs per SM there
constexpr int kForwardPairs = 8, kBackwardPairs = 4;  // pairs of MCUs per warp there, at most (2: 152/152 us, 4: 115/131, 8: 104/140, 16: 107/169)
constexpr int kFloatScan = 1024;   // counts per CTA of the scan (256 threads x 4)
bool float_configure();
void launch_float_forward(const FloatArgs& a, int threads, int pixel_grid, cudaStream_t s);
void launch_float_backward(const FloatArgs& a, int threads, int pixel_grid, cudaStream_t s);

// The integer IDCT constants the decode kernel is compiled with, for the host-side check
// against round(8192 cos(k pi / 16)), k = 1..7.
void idct_constants(int out[8]);

}  // namespace jt
