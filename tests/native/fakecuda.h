// fakecuda.h -- test helper: a CUDA runtime in host memory, enough to run the
// library's host side (csrc/capi.cpp, csrc/mechanism.cpp) without a GPU.
//
// "Device" memory is host memory.  A non-blocking stream runs its work at once.
// The legacy default stream runs its work as late as it may, when something
// waits for it, as it does behind a long queue: cudaMemset, and the last part of
// a cudaMemcpy from pageable host memory, return before they are done.  Work on
// another stream that touches memory with such a write pending is a missing wait
// and is counted in `races`.
#pragma once

#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <vector>

namespace fake {

struct Alloc {
  size_t bytes;
};
inline std::map<char *, Alloc> memory;          // live allocations
inline size_t live = 0, n_malloc = 0;           // bytes, calls
inline long fail_malloc = -1;                   // that many more calls succeed (-1: all)
inline int device = 0;

struct Pending {
  char *p;
  size_t n;
  std::function<void()> run;
};
inline std::vector<Pending> legacy;
inline long races = 0;

struct Stream {
  bool capturing = false;
  std::vector<std::function<void()>> captured;
};

inline void drain_legacy() {
  std::vector<Pending> q;
  q.swap(legacy);
  for (auto &x : q) x.run();
}

// work on a stream touches these bytes
inline void touch(const void *p, size_t n) {
  const char *a = (const char *)p;
  for (const Pending &x : legacy)
    if (a < x.p + x.n && x.p < a + n) {
      ++races;
      return;
    }
}

inline void enqueue(cudaStream_t s, char *p, size_t n, std::function<void()> f) {
  if (!s) {
    legacy.push_back({p, n, f});
    return;
  }
  Stream *st = (Stream *)s;
  if (st->capturing) st->captured.push_back(f);
  else f();
}

}  // namespace fake

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = fake::device; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "fake error"; }
cudaError_t cudaMalloc(void **p, size_t n) {
  if (fake::fail_malloc == 0) return cudaErrorMemoryAllocation;
  if (fake::fail_malloc > 0) --fake::fail_malloc;
  char *q = (char *)std::malloc(n ? n : 1);
  std::memset(q, 0xa5, n);
  fake::memory[q] = {n};
  fake::live += n;
  ++fake::n_malloc;
  *p = q;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  if (!p) return cudaSuccess;
  auto it = fake::memory.find((char *)p);
  if (it == fake::memory.end()) { std::printf("free of memory that was not allocated\n"); std::exit(9); }
  fake::drain_legacy();
  fake::live -= it->second.bytes;
  fake::memory.erase(it);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) {
  fake::enqueue(s, (char *)p, n, [=] { if (s) fake::touch(p, n); std::memset(p, v, n); });
  return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { return cudaMemsetAsync(p, v, n, nullptr); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  fake::enqueue(st, (char *)d, n, [=] { if (st) { fake::touch(s, n); fake::touch(d, n); } std::memcpy(d, s, n); });
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t st) {
  fake::enqueue(st, (char *)d, (h - 1) * dp + w, [=] {
    for (size_t i = 0; i < h; ++i) {
      if (st) { fake::touch((const char *)s + i * sp, w); fake::touch((char *)d + i * dp, w); }
      std::memcpy((char *)d + i * dp, (const char *)s + i * sp, w);
    }
  });
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) {
  fake::drain_legacy();
  if (k == cudaMemcpyHostToDevice) {            // staged; the last part may still be under way on return
    std::vector<char> stage((const char *)s, (const char *)s + n);
    fake::enqueue(nullptr, (char *)d, n, [=] { std::memcpy(d, stage.data(), n); });
  } else {
    std::memcpy(d, s, n);
  }
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t) new fake::Stream(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { delete (fake::Stream *)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { if (!s) fake::drain_legacy(); return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { ((fake::Stream *)s)->capturing = true; return cudaSuccess; }
typedef std::vector<std::function<void()>> FakeGraph;
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) {
  fake::Stream *st = (fake::Stream *)s;
  st->capturing = false;
  *g = (cudaGraph_t) new FakeGraph(st->captured);
  st->captured.clear();
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long) { *x = (cudaGraphExec_t) new FakeGraph(*(FakeGraph *)g); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (FakeGraph *)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete (FakeGraph *)x; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) {
  if (!s) fake::drain_legacy();
  for (auto &f : *(FakeGraph *)x) f();
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) {
  a->type = cudaMemoryTypeDevice;
  a->device = fake::device;
  return cudaSuccess;
}
}
