// A device that only keeps the order of things.  Linked with the library's host code in place of the
// CUDA runtime and of the kernels' launchers: every launch and copy is an operation on a stream with
// the memory that it reads and writes, streams and events carry vector clocks, and two operations that
// touch the same memory (one of them writing) without an order between them are a race.
#include <stdint.h>
#include <stdio.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "xkv_internal.cuh"

namespace {

typedef std::map<const void*, uint64_t> Clock;      // stream -> its operations that have happened before
void join(Clock& into, const Clock& from) {
  for (auto& e : from) into[e.first] = std::max(into[e.first], e.second);
}

struct Access { uintptr_t lo, hi; bool write; std::string what; };
struct Op { const void* stream; uint64_t seq; std::string name; std::vector<Access> mem; };
struct Event { Clock clock; int epoch; };

std::recursive_mutex g_mutex;
std::map<const void*, Clock> g_streams;
Clock g_host;
std::map<const void*, Event> g_events;
std::vector<Op> g_ops;
std::string g_report;
std::string g_fail_name;       // the next operation of this name fails
std::map<const void*, int> g_means_of;     // head-mean array -> frame of the cache that it was computed for
std::string g_hook_name;       // before the g_hook_after-th operation of this name, g_hook is called
int g_hook_after = 0;
void (*g_hook)() = nullptr;
int g_epoch = 0;
uintptr_t g_handles = 0x1000;

void note(const std::string& line) { if (g_report.size() < 4000) g_report += line + "\n"; }

struct Builder {
  Op op;
  Builder(const char* name, const void* stream) { op.name = name; op.stream = stream; }
  void add(const void* p, size_t bytes, bool write, const char* what) {
    if (p && bytes) op.mem.push_back({(uintptr_t)p, (uintptr_t)p + bytes, write, what});
  }
  void reads(const void* p, size_t bytes, const char* what) { add(p, bytes, false, what); }
  void writes(const void* p, size_t bytes, const char* what) { add(p, bytes, true, what); }
  cudaError_t run() {
    if (g_hook && g_hook_name == op.name && --g_hook_after == 0) {
      void (*hook)() = g_hook;
      g_hook = nullptr;
      hook();
    }
    std::lock_guard<std::recursive_mutex> lock(g_mutex);
    if (g_fail_name == op.name) { g_fail_name.clear(); return cudaErrorLaunchFailure; }
    Clock& now = g_streams[op.stream];
    join(now, g_host);
    for (const Op& old : g_ops) {
      auto seen = now.find(old.stream);
      if (old.stream == op.stream || (seen != now.end() && old.seq <= seen->second)) continue;
      for (const Access& x : old.mem)
        for (const Access& y : op.mem)
          if ((x.write || y.write) && x.lo < y.hi && y.lo < x.hi)
            note("race: " + op.name + " (" + y.what + ") is not ordered after " + old.name + " (" + x.what + ")");
    }
    op.seq = ++now[op.stream];
    g_ops.push_back(op);
    return cudaSuccess;
  }
};

void tensor(Builder& b, const void* p, int H, int n, int64_t ts, int64_t hs, bool write, const char* what) {
  b.add(p, (size_t)((H - 1) * hs + (n - 1) * ts + xkv::kHeadDim) * 2, write, what);
}

// The arrays of a buffer set, whole.
void key_arrays(Builder& b, const xkv_cache* c, const xkv::BufSet& s, bool write) {
  const size_t H = c->p.n_heads, cap = c->cap;
  b.add(s.k, H * cap * c->row_bytes, write, "key codes");
  if (c->p.key_mode == XKV_KEYS_ONCE) b.add(s.kslot, cap * 4, write, "group references");
  else b.add(s.kpar, H * (cap / 64) * 64 * 8, write, "key parameters");
}
void buffers(Builder& b, const xkv_cache* c, const xkv::BufSet& s, bool write) {
  const size_t H = c->p.n_heads, cap = c->cap;
  key_arrays(b, c, s, write);
  b.add(s.v, H * cap * c->row_bytes, write, "value codes");
  b.add(s.vpar, H * cap * 8, write, "value parameters");
  b.add(s.origin, cap * 4, write, "origins");
}
void head_means(Builder& b, const xkv_cache* c, const xkv::BufSet& s, bool write) {
  b.add(s.kbar, (size_t)c->cap * 64 * 4, write, "head means");
}

}  // namespace

extern "C" {
// ---- for the test --------------------------------------------------------------
XKV_API const char* fake_report() { return g_report.c_str(); }
XKV_API int fake_ops(const char* name) {
  int n = 0;
  for (const Op& o : g_ops) n += o.name == name;
  return n;
}
XKV_API void fake_fail_next(const char* name) { g_fail_name = name; }
XKV_API void fake_hook(const char* name, int nth, void (*fn)()) { g_hook_name = name; g_hook_after = nth; g_hook = fn; }
XKV_API void fake_clear() { g_report.clear(); g_ops.clear(); g_fail_name.clear(); }   // (the clocks go on)
// From here on a wait on an event that was recorded before is an error, as inside a stream capture.
XKV_API void fake_begin_capture() { ++g_epoch; }

// ---- the runtime calls of the host code ------------------------------------------
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)(g_handles += 16); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)(g_handles += 16); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { g_events.erase(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  join(g_streams[s], g_host);
  g_events[e] = {g_streams[s], g_epoch};
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  auto it = g_events.find(e);
  if (it == g_events.end()) return cudaSuccess;
  if (it->second.epoch != g_epoch) note("capture: a wait on an event from before");
  join(g_streams[s], it->second.clock);
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  if (g_events.count(e)) join(g_host, g_events[e].clock);
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  std::lock_guard<std::recursive_mutex> lock(g_mutex);
  join(g_host, g_streams[s]);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t s) {
  Builder b("copy", s);
  b.reads(src, n, "source of a copy");
  b.writes(dst, n, "destination of a copy");
  return b.run();
}
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int, size_t n, cudaStream_t s) {
  Builder b("clear", s);
  b.writes(p, n, "workspace");
  return b.run();
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
// what nvcc's host code registers at load time
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
}

// ---- the launchers ----------------------------------------------------------------
namespace xkv {

cudaError_t launch_maint(xkv_cache* const* cs, MaintArgs* as, int count, int cat, cudaStream_t st) {
  Builder b(cat == XKV_PROF_KBAR ? "head means" : "maintenance", st);
  for (int i = 0; i < count; ++i) {
    const xkv_cache* c = cs[i];
    const MaintArgs& a = as[i];
    const bool once = c->p.key_mode == XKV_KEYS_ONCE, regroup = c->p.kv_bits == 4 && !once;
    const size_t table = once ? (size_t)c->n_slots * a.H * 64 * 8 : 0;
    if (a.phases & kPhAppend) {
      tensor(b, a.k, a.H, a.n, a.ts_kv, a.hs_kv, false, "keys");
      tensor(b, a.v, a.H, a.n, a.ts_kv, a.hs_kv, false, "values");
      if (regroup) b.writes(a.kstage, (size_t)a.H * a.max_n * 128, "staged keys");
      buffers(b, c, a.oth, true);
      if (a.first) buffers(b, c, a.cur, true);
      b.writes(a.ktab32, table, "key table");
    }
    if (a.phases & kPhPool) {
      tensor(b, a.q, a.H, a.n_q, a.ts_q, a.hs_q, false, "queries");
      b.writes(a.qbar, 256, "pooled query");
    }
    if (a.phases & kPhKbar) {
      key_arrays(b, c, a.cur, false);
      head_means(b, c, a.cur, true);
    }
    if (a.phases & kPhKbarNew) {
      key_arrays(b, c, a.oth, false);
      b.reads(a.ktab32, table, "key table");
      head_means(b, c, a.oth, true);
    }
    if (a.phases & kPhScore) {
      if (!once && !(a.phases & kPhKbar) && g_means_of[a.cur.kbar] != c->frames) note("scores from head means of another frame");
      head_means(b, c, a.cur, false);
      b.writes(a.scores, 4, "scores");
    }
    if (a.phases & kPhSel) b.writes(a.kept, 4, "kept positions");
    if (a.phases & kPhPack) {
      buffers(b, c, a.cur, false);
      buffers(b, c, a.oth, true);
      if (once) { head_means(b, c, a.cur, false); head_means(b, c, a.oth, true); }
    }
  }
  const cudaError_t e = b.run();
  for (int i = 0; i < count && e == cudaSuccess; ++i)
    if (as[i].phases & kPhKbar) g_means_of[as[i].cur.kbar] = cs[i]->frames;
  return e;
}
cudaError_t launch_regroup(xkv_cache* const* cs, const MaintArgs* as, int count, cudaStream_t st) {
  Builder b("regroup", st);
  for (int i = 0; i < count; ++i) {
    const MaintArgs& a = as[i];
    buffers(b, cs[i], a.cur, a.first != 0);
    buffers(b, cs[i], a.oth, true);
    b.reads(a.kstage, (size_t)a.H * a.max_n * 128, "staged keys");
    b.reads(a.kept, 4, "kept positions");
  }
  return b.run();
}
cudaError_t launch_attn_tc(const AttnCall* calls, int count, int64_t ts, int64_t hs, float, cudaStream_t st) {
  if (calls[0].k_tail && calls[0].cache->p.kv_bits == 8) return cudaErrorNotSupported;
  Builder b("attention", st);
  for (int i = 0; i < count; ++i) {
    const AttnCall& k = calls[i];
    const xkv_cache* c = k.cache;
    const int H = c->p.n_heads;
    const size_t first = b.op.mem.size();
    buffers(b, c, c->buf[c->cur], false);
    if (c->p.key_mode == XKV_KEYS_ONCE) b.reads(c->ktab32, (size_t)c->n_slots * H * 64 * 8, "key table");
    tensor(b, k.q, H, k.n, ts, hs, false, "queries");
    if (k.k_tail) {
      tensor(b, k.k_tail, H, k.n, ts, hs, false, "tail keys");
      tensor(b, k.v_tail, H, k.n, ts, hs, false, "tail values");
    }
    tensor(b, k.out, H, k.n, ts, hs, true, "output");
    // calls of one launch run in no order
    for (size_t x = 0; x < first; ++x)
      for (size_t y = first; y < b.op.mem.size(); ++y) {
        const Access &p = b.op.mem[x], &q = b.op.mem[y];
        if ((p.write || q.write) && p.lo < q.hi && q.lo < p.hi) note("race inside one attention launch: " + p.what + ", " + q.what);
      }
  }
  b.writes(calls[0].cache->attn_part, 4, "partial results");
  return b.run();
}
cudaError_t launch_attn_tc_static(const AttnCall& call, int64_t ts, int64_t hs, float scale, cudaStream_t st) {
  return launch_attn_tc(&call, 1, ts, hs, scale, st);
}
cudaError_t launch_attn_simple(xkv_cache*, const void*, void*, int, int64_t, int64_t, float, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_once_init(xkv_cache*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_timeout_probe(xkv_cache*, cudaStream_t) { return cudaSuccess; }
size_t attn_tc_scratch_bytes(const xkv_params*) { return 4096; }

}  // namespace xkv
