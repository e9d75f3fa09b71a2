// The host side of libslpic (csrc/api.cu, compiled as C++) on a CUDA runtime
// made for tests: streams are queues whose work runs only when something that
// is ordered after it is waited for, so a missing wait shows every time.
// Device memory is host memory, and the kernels are models: a step adds 1 to
// v_x of the markers in the tiles that were planned.
//
//   host_runtime SCENARIO     prints what differs; exit code 0: nothing does
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <memory>
#include <string>
#include <utility>
#include <vector>

#include "slpic.h"
#include "slpic_internal.h"

// ---- streams, events, graphs -------------------------------------------------
using Work = std::function<void()>;
struct CUgraph_st {
  std::vector<Work> work;
};
struct CUgraphExec_st : CUgraph_st {};
struct CUstream_st {
  struct Op {
    Work run;
    std::vector<std::pair<CUstream_st*, size_t>> after;
  };
  bool blocking = true;  // ordered with the NULL stream
  std::vector<Op> ops;
  size_t done = 0;
  CUgraph_st* capture = nullptr;
  bool invalid = false, destroyed = false;
};
struct CUevent_st {
  CUstream_st* stream = nullptr;
  size_t upto = 0;
};

static CUstream_st g_null;
static std::vector<CUstream_st*> g_streams;
static std::map<char*, size_t> g_device, g_pinned;
static int g_fail_copy = -1;  // asynchronous copies until one fails

static CUstream_st* of(cudaStream_t s) {
  CUstream_st* p = s == nullptr || s == cudaStreamLegacy ? &g_null : s;
  if (p->destroyed) {
    std::printf("a destroyed stream was used\n");
    std::exit(1);
  }
  return p;
}
static void add(CUstream_st* s, Work w, CUevent_st* wait = nullptr) {
  if (s->capture) {
    s->capture->work.push_back(std::move(w));
    return;
  }
  if (s == &g_null)
    for (CUstream_st* b : g_streams)
      if (b->blocking && b->capture) b->invalid = true;
  CUstream_st::Op op{std::move(w), {}};
  if (wait && wait->stream) op.after.push_back({wait->stream, wait->upto});
  if (s == &g_null) {
    for (CUstream_st* b : g_streams)
      if (b->blocking) op.after.push_back({b, b->ops.size()});
  } else if (s->blocking) {
    op.after.push_back({&g_null, g_null.ops.size()});
  }
  s->ops.push_back(std::move(op));
}
static void run(CUstream_st* s, size_t upto) {
  while (s->done < upto) {
    CUstream_st::Op op = s->ops[s->done];
    for (auto& a : op.after) run(a.first, a.second);
    op.run();
    ++s->done;
  }
}
static void run_all() {
  run(&g_null, g_null.ops.size());
  for (CUstream_st* s : g_streams) run(s, s->ops.size());
}
static bool inside(const std::map<char*, size_t>& m, const void* p, char** base = nullptr,
                   size_t* size = nullptr) {
  auto it = m.upper_bound((char*)p);
  if (it == m.begin()) return false;
  --it;
  if ((char*)p >= it->first + it->second) return false;
  if (base) *base = it->first;
  if (size) *size = it->second;
  return true;
}

static CUresult fake_ctx(CUcontext* c) {
  *c = (CUcontext)&g_null;
  return CUDA_SUCCESS;
}
static CUresult fake_range(CUdeviceptr* base, size_t* size, CUdeviceptr p) {
  char* b = nullptr;
  if (!inside(g_device, (void*)p, &b, size)) return CUDA_ERROR_INVALID_VALUE;
  *base = (CUdeviceptr)b;
  return CUDA_SUCCESS;
}

extern "C" {
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "an error"; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 4, cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  return *p = (void*)s, cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned int,
                                             unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = std::strcmp(name, "cuMemGetAddressRange") == 0 ? (void*)fake_range : (void*)fake_ctx;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = std::malloc(n);
  std::memset(*p, 0x7B, n);
  g_device[(char*)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  run_all();
  g_device.erase((char*)p);
  return std::free(p), cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned int) {
  *p = std::malloc(n);
  g_pinned[(char*)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  run_all();
  g_pinned.erase((char*)p);
  return std::free(p), cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::memset(a, 0, sizeof *a);
  a->type = inside(g_device, p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
// what the copy's source or target outside pinned memory means for the caller:
// the source may change at once, the target is filled on return
static cudaError_t copy(void* d, const void* s, size_t n, cudaMemcpyKind kind, CUstream_st* st) {
  if (kind == cudaMemcpyHostToDevice && !inside(g_pinned, s)) {
    auto b = std::make_shared<std::vector<char>>((const char*)s, (const char*)s + n);
    add(st, [=] { std::memcpy(d, b->data(), n); });
  } else {
    add(st, [=] { std::memcpy(d, s, n); });
    if (kind == cudaMemcpyDeviceToHost && !inside(g_pinned, d)) run(st, st->ops.size());
  }
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind kind) {
  run(&g_null, g_null.ops.size());  // (and may return before its own copy has arrived)
  return copy(d, s, n, kind, &g_null);
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind,
                            cudaStream_t st) {
  if (g_fail_copy >= 0 && g_fail_copy-- == 0) return cudaErrorInvalidValue;
  return copy(d, s, n, kind, of(st));
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  return add(&g_null, [=] { std::memset(d, v, n); }), cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t s) {
  return add(of(s), [=] { std::memset(d, v, n); }), cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned int flags) {
  *s = new CUstream_st;
  (*s)->blocking = !(flags & cudaStreamNonBlocking);
  g_streams.push_back(*s);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return of(s)->destroyed = true, cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  CUstream_st* p = of(s);
  if (p->capture) return p->invalid = true, cudaErrorStreamCaptureUnsupported;
  return run(p, p->ops.size()), cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
  *st = of(s)->capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamGetFlags(cudaStream_t s, unsigned int* flags) {
  return *flags = of(s)->blocking ? cudaStreamDefault : cudaStreamNonBlocking, cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) {
  static cudaStreamCaptureMode mode = cudaStreamCaptureModeGlobal;
  std::swap(*m, mode);
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  of(s)->capture = new CUgraph_st;
  of(s)->invalid = false;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  *g = of(s)->capture;
  of(s)->capture = nullptr;
  return of(s)->invalid ? cudaErrorStreamCaptureInvalidated : cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  *e = new CUgraphExec_st;
  (*e)->work = g->work;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) {
  for (auto& w : e->work) add(of(s), w);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return delete g, cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return delete e, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = new CUevent_st, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned int) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete e, cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  return *ms = 1.0f, cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  CUstream_st* p = of(s);
  if (p->capture) return p->invalid = true, cudaErrorStreamCaptureUnsupported;
  add(p, [] {});
  e->stream = p;
  e->upto = p->ops.size();
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  if (e->stream) run(e->stream, e->upto);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned int) {
  CUstream_st* p = of(s);
  if (p->capture) return p->invalid = true, cudaErrorStreamCaptureIsolation;
  return add(p, [] {}, e), cudaSuccess;
}
}  // extern "C"

// ---- the kernels, as models ----------------------------------------------------
namespace slpic {
static Markers<float> store(const DeviceRefs& r, int seg, uint32_t cur) {
  return Markers<float>{r.inst[seg >> 1].sp[seg & 1].buf[cur]};
}
static uint32_t* fills(const DeviceRefs& r, int seg, uint32_t cur) {
  return r.inst[seg >> 1].sp[seg & 1].fill[cur];
}
void launch_push(const DeviceRefs& r, int, cudaStream_t s) {
  add(of(s), [r] {
    for (int g = 0; g < 2 * r.n_inst; ++g) {
      const uint32_t cur = r.sstate[g].cur;
      for (uint32_t k = 0; k < r.seg_start[g + 1] - r.seg_start[g]; ++k)
        for (uint32_t i = 0; i < fills(r, g, cur)[k]; ++i) store(r, g, cur).at(k, i).vx() += 1;
    }
  });
}
void launch_finish(const DeviceRefs& r, int mode, cudaStream_t s) {
  add(of(s), [r, mode] {
    if (mode == 0)
      for (int i = 0; i < r.n_inst; ++i) ++r.istate[i].step, ++r.istate[i].n_steps_done;
    r.seg_start[0] = 0;
    for (int g = 0; g < 2 * r.n_inst; ++g) r.seg_start[g + 1] = r.seg_start[g] + r.sstate[g].n_tiles;
  });
}
void launch_collide(const DeviceRefs&, int, cudaStream_t) {}
void launch_move(const DeviceRefs&, int, cudaStream_t) {}
void launch_phi(const DeviceRefs& r, int inst, int, cudaStream_t s) {
  add(of(s), [=] { r.inst[inst].phi[1] = (double)r.istate[inst].step; });
}
void launch_vacuum(const InstDev& P, double E, float E32, cudaStream_t s) {
  add(of(s), [=] {
    for (int k = 0; k <= P.n_cells; ++k) P.phi[k] = P.V * k / P.n_cells, P.E64[k] = E, P.E32[k] = E32;
  });
}
void launch_fills(uint32_t* f, uint32_t first, uint32_t end, cudaStream_t s) {
  add(of(s), [=] {
    for (uint32_t k = first; k * kTile < end; ++k) f[k] = std::min(end - k * kTile, (uint32_t)kTile);
  });
}
void launch_prefix(const uint32_t* f, uint32_t n, uint32_t* pre, uint32_t* total, cudaStream_t s) {
  add(of(s), [=] {
    *total = 0;
    for (uint32_t k = 0; k < n; ++k) pre[k] = *total, *total += f[k];
  });
}
void launch_deposit(const DeviceRefs& r, int inst, int, int, int, cudaStream_t s) {
  add(of(s), [=] {
    for (int sp = 0; sp < 2; ++sp)
      for (uint32_t k = 0; k < r.sstate[2 * inst + sp].n_tiles; ++k)
        r.inst[inst].rho_last[sp][0] += fills(r, 2 * inst + sp, r.sstate[2 * inst + sp].cur)[k];
  });
}
void launch_seed(const DeviceRefs& r, int inst, int sp, uint32_t base, uint32_t id, uint32_t n, int,
                 double, double, double, double wj, cudaStream_t s) {
  add(of(s), [=] {
    const int g = 2 * inst + sp;
    for (uint32_t i = 0; i < n; ++i) {
      const Slot<float> m = store(r, g, r.sstate[g].cur)[base + i];
      m.cell() = 0, m.off() = m.vx() = m.vy() = m.vz() = 0, m.wj() = (float)wj, m.id() = id + i;
    }
  });
}
void launch_place(int, const void* const src[7], unsigned char* buf, uint32_t n, int, int shift,
                  unsigned int*, unsigned long long* wsum, cudaStream_t s) {
  const std::vector<const void*> f(src, src + 7);
  add(of(s), [=] {
    for (uint32_t i = 0; i < n; ++i) {
      const Slot<float> m = Markers<float>{buf}[i];
      m.cell() = ((const int*)f[0])[i], m.id() = ((const uint32_t*)f[6])[i];
      m.off() = ((const float*)f[1])[i], m.vx() = ((const float*)f[2])[i];
      m.vy() = ((const float*)f[3])[i], m.vz() = ((const float*)f[4])[i];
      m.wj() = ((const float*)f[5])[i];
      *wsum += (unsigned long long)(m.wj() * (double)(1ull << shift));
    }
  });
}
void launch_gather(int, const unsigned char* buf, const uint32_t* fill, const uint32_t* pre,
                   uint32_t n, void* const dst[7], cudaStream_t s) {
  const std::vector<void*> f(dst, dst + 7);
  add(of(s), [=] {
    for (uint32_t k = 0; k < n; ++k)
      for (uint32_t i = 0; i < fill[k]; ++i) {
        const Slot<float> m = Markers<float>{(unsigned char*)buf}.at(k, i);
        const uint32_t o = pre[k] + i;
        ((int*)f[0])[o] = m.cell(), ((uint32_t*)f[6])[o] = m.id();
        ((float*)f[1])[o] = m.off(), ((float*)f[2])[o] = m.vx(), ((float*)f[3])[o] = m.vy();
        ((float*)f[4])[o] = m.vz(), ((float*)f[5])[o] = m.wj();
      }
  });
}
int push_config(int, int, int* warps, int* bps) { return *warps = 20, *bps = 1, 0; }
int push_blocks_per_sm(int, int, int, int* bps) { return *bps = 1, 0; }
int collide_config(int, int, int* resident, int* nodes) { return *resident = 1, *nodes = 0, 0; }
int deposit_config(int) { return 0; }
int small_config(int, int, size_t* bytes, int* bps) { return *bytes = 0, *bps = 0, 0; }
int launch_small(const DeviceRefs&, long long, int, size_t, cudaStream_t) { return 0; }
int philox_preload() { return 0; }
void launch_philox(uint32_t, uint32_t, const uint32_t*, uint32_t*, long long, cudaStream_t) {}
void launch_philox2(uint32_t, const uint32_t*, uint32_t*, long long, cudaStream_t) {}
}  // namespace slpic

// ---- scenarios ------------------------------------------------------------------
static int g_bad = 0;
static void expect(bool ok, const char* what) {
  if (!ok) std::printf("%s\n", what), ++g_bad;
}
static void ok(int rc) { expect(rc == SLPIC_OK, "a call failed"); }

struct Host {
  std::vector<int> cell;
  std::vector<unsigned> id;
  std::vector<float> r[5];
  slpic_soa_f32 soa;
  explicit Host(int n, float vx = 0) : cell(n, 1), id(n) {
    for (int k = 0; k < 5; ++k) r[k].assign(n, k == 1 ? vx : k == 4 ? 1.0f : 0.25f);
    for (int i = 0; i < n; ++i) id[i] = i;
    soa = {cell.data(), r[0].data(), r[1].data(), r[2].data(), r[3].data(), r[4].data(), id.data()};
  }
};
struct Sim {
  slpic_ctx* c = nullptr;
  explicit Sim(cudaStream_t s = nullptr, int field_mode = SLPIC_FIELD_FROZEN,
               int64_t capacity = 1 << 15) {
    const float xs[2] = {1e-20f, 1e-20f};
    ok(slpic_create(&c, 0, 1));
    ok(slpic_set_stream(c, s));
    ok(slpic_set_gap(c, 0, 1e-3, 8, 100.0, field_mode, 1.0));
    ok(slpic_set_gas(c, 0, 100.0, 300.0));
    ok(slpic_set_cross_sections(c, 0, 0, 0, 1, xs, xs, 11.5, xs, 15.8));
    ok(slpic_set_species(c, 0, 0, 9.1e-31, -1.6e-19, 1e5, capacity));
    ok(slpic_set_species(c, 0, 1, 6.6e-26, 1.6e-19, 0.0, capacity));
    ok(slpic_set_dt(c, 0, 1e-12));
  }
  ~Sim() { slpic_destroy(c); }
  void load(int n, float vx = 0) const {
    Host h(n, vx);
    ok(slpic_load_particles(c, 0, 0, &h.soa, n, n));
  }
  std::vector<float> vx() const {
    int64_t n = 0;
    ok(slpic_count(c, 0, 0, &n));
    Host h((int)n);
    ok(slpic_read_particles(c, 0, 0, &h.soa, n, &n));
    return h.r[1];
  }
};
static cudaStream_t stream(bool blocking = false) {
  cudaStream_t s;
  cudaStreamCreateWithFlags(&s, blocking ? cudaStreamDefault : cudaStreamNonBlocking);
  return s;
}
static cudaGraphExec_t captured(const Sim& sim, cudaStream_t s, int steps) {
  cudaGraph_t g;
  cudaGraphExec_t e;
  cudaStreamBeginCapture(s, cudaStreamCaptureModeRelaxed);
  ok(slpic_step(sim.c, steps));
  expect(cudaStreamEndCapture(s, &g) == cudaSuccess, "the capture is invalid");
  cudaGraphInstantiate(&e, g, 0);
  return e;
}

// Steps captured when the plan of the next step was made, replayed after the
// stores have changed.
static void replay_after_changes() {
  cudaStream_t s = stream(), other = stream();
  Sim sim(s), plain;
  for (const Sim* p : {&sim, &plain}) p->load(300), ok(slpic_step(p->c, 1));
  cudaGraphExec_t g = captured(sim, s, 1);
  auto both = [&](const std::function<void(slpic_ctx*)>& f, const char* what) {
    f(sim.c);
    f(plain.c);
    cudaGraphLaunch(g, other);
    cudaStreamSynchronize(other);
    ok(slpic_step(plain.c, 1));
    expect(sim.vx() == plain.vx(), what);
  };
  for (int n : {3000, 200})
    both([&](slpic_ctx* c) {
      Host h(n);
      ok(slpic_load_particles(c, 0, 0, &h.soa, n, n));
    }, "load");
  both([](slpic_ctx* c) { ok(slpic_seed(c, 0, 0, 1000, SLPIC_SEED_REST, 0, 0, 0, 1)); }, "seed");
  size_t size = 0;
  ok(slpic_save(plain.c, nullptr, 0, &size));
  std::vector<char> snap(size);
  ok(slpic_save(plain.c, snap.data(), size, &size));
  both([](slpic_ctx* c) { ok(slpic_seed(c, 0, 0, 5000, SLPIC_SEED_REST, 0, 0, 0, 1)); }, "seed");
  both([&](slpic_ctx* c) { ok(slpic_load(c, snap.data(), size)); }, "snapshot");
  both([](slpic_ctx* c) { ok(slpic_clear_error(c)); }, "clear_error");
  both([](slpic_ctx* c) { ok(slpic_set_launch_shape(c, 8, 2)); }, "launch shape");
}

// A change of stream right after steps: what follows on the new stream finds
// them finished, also through a stream that did nothing, into a capture, or
// when the old stream is gone.
static void stream_changed_after_steps() {
  enum { kRead, kLoad, kSeed, kCapture, kTwice, kDestroyed, kRefused, kEnd };
  for (int from = 0; from < 5; ++from)
    for (int what = kRead; what < kEnd; ++what) {
      cudaStream_t a = from % 3 ? stream(from == 2) : nullptr, b = stream(from > 2);
      Sim sim(a), plain;
      sim.load(300), plain.load(300);
      ok(slpic_step(sim.c, 40)), ok(slpic_step(plain.c, 40));
      if (what == kRefused)  // (its first act is the deposit of the markers that are there)
        for (const Sim* p : {&sim, &plain})
          expect(slpic_seed(p->c, 0, 0, 1 << 20, SLPIC_SEED_REST, 0, 0, 0, 1) == SLPIC_ERR_CAPACITY,
                 "too many markers");
      if (what == kDestroyed && a) cudaStreamDestroy(a);
      if (what == kTwice) ok(slpic_set_stream(sim.c, stream()));
      cudaGraph_t g = nullptr;
      if (what == kCapture) cudaStreamBeginCapture(b, cudaStreamCaptureModeRelaxed);
      ok(slpic_set_stream(sim.c, b));
      if (what == kCapture) {
        cudaGraphExec_t e;
        ok(slpic_step(sim.c, 1));
        expect(cudaStreamEndCapture(b, &g) == cudaSuccess, "the capture is invalid");
        ok(slpic_step(plain.c, 1));
        cudaGraphInstantiate(&e, g, 0);
        cudaGraphLaunch(e, b);
      }
      for (const Sim* p : {&sim, &plain}) {
        if (what == kLoad) p->load(200);
        if (what == kSeed) ok(slpic_seed(p->c, 0, 0, 70, SLPIC_SEED_REST, 0, 0, 0, 1));
        if (what == kLoad || what == kSeed) ok(slpic_step(p->c, 2));
      }
      int64_t q[2][9];
      if (what == kRefused) {
        ok(slpic_read_charge(sim.c, 0, 0, q[0], 9));
        ok(slpic_read_charge(plain.c, 0, 0, q[1], 9));
        expect(std::equal(q[0], q[0] + 9, q[1]), "charge after a change of stream");
      }
      expect(sim.vx() == plain.vx(), "markers after a change of stream");
      slpic_tallies t[2];
      int64_t n[2] = {0, 0};
      ok(slpic_read_history(sim.c, 0, &t[0], 1, &n[0]));
      ok(slpic_read_history(plain.c, 0, &t[1], 1, &n[1]));
      expect(n[0] == n[1], "steps after a change of stream");
    }
}

// Steps that a caller replays on the NULL stream, or on one that it waits for,
// come before the calls that follow on a stream that does not wait for it.
static void replays_on_the_null_stream() {
  for (int mode : {SLPIC_FIELD_FROZEN, SLPIC_FIELD_POISSON})
    for (cudaStream_t on : {(cudaStream_t) nullptr, stream(true)})
      for (int what = 0; what < 6; ++what) {
        cudaStream_t s = stream();
        Sim sim(s, mode), plain(nullptr, mode);
        sim.load(300), plain.load(300);
        cudaGraphExec_t g = captured(sim, s, 1);
        cudaStreamSynchronize(nullptr);
        cudaGraphLaunch(g, on), cudaGraphLaunch(g, on);
        ok(slpic_step(plain.c, 2));
        double f[2][2][9];
        int64_t q[2][9], n[2];
        slpic_tallies t;
        const slpic_ctx* c = sim.c;
        for (const Sim* p : {&sim, &plain}) {
          const int k = p->c != c;
          if (what == 0) ok(slpic_read_field(p->c, 0, f[k][0], f[k][1], 9));
          if (what == 1) ok(slpic_read_charge(p->c, 0, 0, q[k], 9));
          if (what == 2) ok(slpic_read_history(p->c, 0, &t, 1, &n[k]));
          if (what == 3) ok(slpic_seed(p->c, 0, 0, 70, SLPIC_SEED_REST, 0, 0, 0, 1));
          if (what == 4) ok(slpic_clear_error(p->c));
          if (what == 5) ok(slpic_read_tallies(p->c, 0, &t));
          if (!k) expect(!on || on->done == on->ops.size(), "replays after a call");
        }
        if (what == 0) expect(!std::memcmp(f[0], f[1], sizeof f[0]), "field after replays");
        if (what == 1) expect(!std::memcmp(q[0], q[1], sizeof q[0]), "charge after replays");
        if (what == 2) expect(n[0] == n[1], "steps after replays");
        const std::vector<float> a = sim.vx(), b = plain.vx();
        expect(a == b, "markers after replays");
      }
}

// Device arrays, and pinned ones, that work on the NULL stream fills, loaded on
// a stream that does not wait for it.
static void device_arrays() {
  Sim sim(stream()), plain;
  Host h(500, 3.0f);
  const void* src[7] = {h.soa.cell, h.soa.off, h.soa.vx, h.soa.vy, h.soa.vz, h.soa.wj, h.soa.id};
  void* d[7];
  for (int k = 0; k < 7; ++k) cudaMalloc(&d[k], 2000);
  sim.load(10), plain.load(500, 3.0f);
  for (int k = 0; k < 7; ++k) cudaMemcpyAsync(d[k], src[k], 2000, cudaMemcpyHostToDevice, nullptr);
  slpic_soa_f32 soa = {(int32_t*)d[0], (float*)d[1], (float*)d[2],   (float*)d[3],
                       (float*)d[4],   (float*)d[5], (uint32_t*)d[6]};
  ok(slpic_load_particles_device(sim.c, 0, 0, &soa, 500, 500));
  expect(sim.vx() == plain.vx(), "markers from device arrays");
  void* p[7];
  for (int k = 0; k < 7; ++k) {
    cudaHostAlloc(&p[k], 2000, 0);
    std::memset(p[k], 0, 2000);
    cudaMemcpyAsync(p[k], d[k], 2000, cudaMemcpyDeviceToHost, nullptr);
  }
  slpic_soa_f32 pinned = {(int32_t*)p[0], (float*)p[1], (float*)p[2],   (float*)p[3],
                          (float*)p[4],   (float*)p[5], (uint32_t*)p[6]};
  sim.load(10);
  ok(slpic_load_particles(sim.c, 0, 0, &pinned, 500, 500));
  expect(sim.vx() == plain.vx(), "markers from pinned arrays");
}

// A snapshot restored, and a context set up, on a stream that does not wait for
// the NULL stream.
static void copies_on_the_null_stream() {
  Sim plain(nullptr, SLPIC_FIELD_FROZEN);
  plain.load(300);
  ok(slpic_step(plain.c, 1));
  int64_t q[2][9];
  size_t size = 0;
  ok(slpic_seed(plain.c, 0, 1, 50, SLPIC_SEED_REST, 0, 0, 0, 1));
  ok(slpic_step(plain.c, 1));
  ok(slpic_save(plain.c, nullptr, 0, &size));
  std::vector<char> snap(size);
  ok(slpic_save(plain.c, snap.data(), size, &size));
  ok(slpic_read_charge(plain.c, 0, 1, q[1], 9));
  cudaStreamSynchronize(nullptr);
  Sim sim(stream());
  int64_t n = 0;
  ok(slpic_count(sim.c, 0, 0, &n));
  expect(g_null.done == g_null.ops.size(), "copies of the set-up");
  ok(slpic_set_spin_limit(sim.c, 1000));
  expect(g_null.done == g_null.ops.size(), "copy of the spin limit");
  ok(slpic_test_skip_barrier(sim.c, 0, 3));
  expect(g_null.done == g_null.ops.size(), "copies of the skipped barrier");
  int64_t waits = 0, longest = 0;
  ok(slpic_read_wait_stats(sim.c, &waits, &longest));
  expect(g_null.done == g_null.ops.size(), "copies of the wait statistics");
  ok(slpic_load(sim.c, snap.data(), size));
  expect(g_null.done == g_null.ops.size(), "copies of the snapshot");
  ok(slpic_read_charge(sim.c, 0, 1, q[0], 9));
  expect(std::equal(q[0], q[0] + 9, q[1]), "charge of a snapshot");
  expect(sim.vx() == plain.vx(), "markers of a snapshot");
}

// A read of markers that fails on the way leaves nothing behind that would
// write to the caller's arrays later.
static void failed_read() {
  const int n = 200000;  // the cells go through pinned memory, the reals do not
  Sim sim(nullptr, SLPIC_FIELD_FROZEN, n);
  ok(slpic_set_precision(sim.c, 64));
  ok(slpic_seed(sim.c, 0, 0, n, SLPIC_SEED_REST, 0, 0, 0, 1));
  int64_t got = 0;
  ok(slpic_count(sim.c, 0, 0, &got));
  std::vector<int32_t> cell(n, -7);
  std::vector<uint32_t> id(n);
  std::vector<double> r(5 * n);
  slpic_soa_f64 soa = {cell.data(), r.data(), r.data() + n, r.data() + 2 * n, r.data() + 3 * n,
                       r.data() + 4 * n, id.data()};
  g_fail_copy = 1;
  expect(slpic_read_particles_f64(sim.c, 0, 0, &soa, n, &got) == SLPIC_ERR_CUDA, "a failing copy");
  slpic_tallies t;
  ok(slpic_read_tallies(sim.c, 0, &t));
  expect(std::count(cell.begin(), cell.end(), -7) == n, "an array written after its call");
}

int main(int argc, char** argv) {
  const std::map<std::string, std::function<void()>> all = {
      {"replay_after_changes", replay_after_changes},
      {"stream_changed_after_steps", stream_changed_after_steps},
      {"replays_on_the_null_stream", replays_on_the_null_stream},
      {"device_arrays", device_arrays},
      {"failed_read", failed_read},
      {"copies_on_the_null_stream", copies_on_the_null_stream},
  };
  if (argc != 2 || !all.count(argv[1])) return 2;
  all.at(argv[1])();
  return g_bad ? 1 : 0;
}
