// jt_api.cu on a CUDA runtime of host memory, for tests of the library's host logic without a GPU:
// built by test_host_runtime.py with the host compiler. "Device" memory is host memory; work on a
// stream waits in a queue until the next synchronising call, so that a copy reads its source
// as late as a real one may; memory given back by delete is overwritten (and kept), so that a
// late read of it shows. The launch functions stand for the kernels: each leaves behind what the
// tests look at.
#include <malloc.h>

#include <functional>
#include <memory>

#include "jt_api.cu"

namespace {

using Queue = std::vector<std::function<void()>>;
struct FakeGraph {
  Queue ops;
  std::vector<std::function<void()>> owned;  // destructors of the user objects it holds
};
struct FakeObject {
  void* p;
  cudaHostFn_t destroy;
};

Queue pending;
FakeGraph* capture = nullptr;
cudaError_t last_error = cudaSuccess;
int sm_count = 152, fast_mcus = 0, fast_warps = 0, run_mcus = 0, run_warps = 0;
bool fail_gather = false, cursors_dirty = false;
std::vector<uint8_t> scene_tables;
int tile_x = 0, tile_h = 0, many = 0;
size_t last_malloc = 0, fail_malloc = 0;
int tables_on_device = 0;

void put(std::function<void()> f) { (capture ? capture->ops : pending).push_back(std::move(f)); }
cudaError_t wait() {
  Queue q;
  q.swap(pending);
  for (auto& f : q) f();
  return cudaSuccess;
}

// a float pass: counts, then (unless its gather fails to launch) zeroed counts
void float_pass(const FloatArgs& a) {
  const bool gather = !fail_gather;
  if (!gather) last_error = cudaErrorInvalidConfiguration;
  put([=] {
    for (uint32_t i = 0; i < a.coef_mcus; ++i) {
      if (a.cursor[i]) cursors_dirty = true;
      a.cursor[i] = gather ? 0 : 1;
    }
  });
}

}  // namespace

void operator delete(void* p) noexcept {
  if (p) memset(p, 0xDD, malloc_usable_size(p));
}
void operator delete(void* p, std::size_t) noexcept { operator delete(p); }

extern "C" {

// ---- the runtime ----
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  *p = cudaDeviceProp{};
  p->multiProcessorCount = sm_count;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  if (fail_malloc && n >= fail_malloc) return fail_malloc = 0, last_error = cudaErrorMemoryAllocation;
  return *p = calloc(last_malloc = n, 1), cudaSuccess;
}
cudaError_t cudaFree(void* p) { return wait(), free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return wait(), memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { return wait(), memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  return put([=] { memcpy(d, s, n); }), cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return put([=] { memset(d, v, n); }), cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return wait(); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return wait(); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)1, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)1, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t)1, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return wait(); }
// a frame takes a millisecond in the fast decode shape and two in the others
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  return *ms = run_mcus == fast_mcus && run_warps == fast_warps ? 1.f : 2.f, cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  return *s = capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus* st, unsigned long long* id, cudaGraph_t* g,
                                     const cudaGraphNode_t**, const cudaGraphEdgeData**, size_t*) {
  if (id) *id = 1;
  if (g) *g = (cudaGraph_t)capture;
  return cudaStreamIsCapturing(s, st);
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return capture = new FakeGraph, cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = (cudaGraph_t)capture;
  capture = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) { return *e = (cudaGraphExec_t)g, cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  for (auto& f : ((FakeGraph*)e)->ops) pending.push_back(f);
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  for (auto& f : ((FakeGraph*)g)->owned) f();
  ((FakeGraph*)g)->owned.clear();
  return cudaSuccess;
}
cudaError_t cudaUserObjectCreate(cudaUserObject_t* o, void* p, cudaHostFn_t destroy, unsigned, unsigned) {
  return *o = (cudaUserObject_t) new FakeObject{p, destroy}, cudaSuccess;
}
cudaError_t cudaUserObjectRelease(cudaUserObject_t, unsigned) { return cudaSuccess; }
cudaError_t cudaGraphRetainUserObject(cudaGraph_t g, cudaUserObject_t o, unsigned, unsigned) {
  const FakeObject f = *(FakeObject*)o;
  ((FakeGraph*)g)->owned.push_back([=] { f.destroy(f.p); });
  return cudaSuccess;
}

// ---- what the tests set and read ----
void fake_sm_count(int n) { sm_count = n; }
void fake_fast_shape(int mcus, int warps) { fast_mcus = mcus, fast_warps = warps; }
void fake_fail_gather(int on) { fail_gather = on != 0; }
int fake_cursors_dirty() { return cursors_dirty; }
int fake_tile_h() { return tile_h; }
int fake_tile_x() { return tile_x; }
int fake_many() { return many; }
size_t fake_last_malloc() { return last_malloc; }
void fake_fail_malloc(size_t n) { fail_malloc = n; }  // the next allocation of n bytes or more
size_t fake_set_bytes() { return sizeof(HuffSet); }
int fake_tables_on_device() { return wait(), tables_on_device; }
size_t fake_scene_tables(uint8_t* out) {  // the tables the last rasteriser pass that ran has read
  wait();
  if (out) memcpy(out, scene_tables.data(), scene_tables.size());
  return scene_tables.size();
}
void* fake_begin_capture() { return capture = new FakeGraph; }
void fake_end_capture() { capture = nullptr; }
void fake_launch_graph(void* g) { cudaGraphLaunch((cudaGraphExec_t)g, nullptr); }
int fake_owned(void* g) { return (int)((FakeGraph*)g)->owned.size(); }
void fake_destroy_graph(void* g) { cudaGraphDestroy((cudaGraph_t)g); }

// The decoder's entry for every 16-bit prefix in each of a context's tables, or -1 where the index
// leaves the table: out[set][table][65536].
void fake_table_entries(jt_ctx* c, int32_t* out) {
  for (auto& v : c->hsets) {
    const HuffSet& hs = v[0];
    for (int t = 0; t < 4; ++t) {
      const HuffTable& w = hs.table[t];
      const uint32_t first = (w.base - (uint32_t)offsetof(HuffSet, lut)) / 2;
      for (uint32_t p = 0; p < 65536; ++p) {
        const uint32_t x = hs.capped ? table_index<true>(p << 16, w.d, w.cap) : table_index<false>(p << 16, w.d, w.cap);
        *out++ = x <= (uint32_t)w.cap ? hs.lut[first + x] : -1;
      }
    }
  }
}

}  // extern "C"

// ---- the kernels ----
namespace jt {
void launch_mark(const MarkArgs& a, int, int, cudaStream_t) {
  tile_h = a.views.tile_h;
  many = a.many;
}
void launch_scan(const ScanArgs&, cudaStream_t) {}
void launch_cache_update(const CacheArgs&, int, cudaStream_t) {}
void launch_decode(const DecodeArgs& a, int warps, int, cudaStream_t) {
  put([a, m = a.mcus_per_warp, warps] {
    run_mcus = m, run_warps = warps;
    tables_on_device = 0;  // of the levels' sets, those that the decoder finds
    for (uint32_t d = 0, seen = 0; a.huff && a.quant && d < a.ndesc; ++d)
      if (!(seen >> a.descs[d].hset & 1) && a.huff[a.descs[d].hset].used != 0) ++tables_on_device, seen |= 1u << a.descs[d].hset;
  });
}
void launch_colorize(const ColorizeArgs&, int, int, cudaStream_t) {}
void launch_raster(const RasterArgs& a, cudaStream_t) {
  tile_x = a.tile_x;
  put([a] {
    const uint8_t* p = reinterpret_cast<const uint8_t*>(a.sizes);
    scene_tables.assign(p, p + (size_t)a.ntex * 16 + (size_t)a.nquads * sizeof(SceneQuad));
  });
}
size_t decode_smem_bytes(int warps, int m) { return (size_t)warps * m; }
int decode_max_ctas_per_sm(int warps, int m) { return warps * m <= 236 ? 1 : 0; }
bool float_configure() { return true; }
void launch_float_forward(const FloatArgs& a, int, int, cudaStream_t) { float_pass(a); }
void launch_float_backward(const FloatArgs& a, int, int, cudaStream_t) { float_pass(a); }
void idct_constants(int out[8]) {
  for (int k = 0; k < 8; ++k) out[k] = (int)std::lround(8192.0 * std::cos(k * M_PI / 16.0));
}
}  // namespace jt
