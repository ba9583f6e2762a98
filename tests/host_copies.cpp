// Runs calls of the library against a stand-in for the CUDA runtime, on the
// host, and reports every block of host memory that is given back while a copy
// from or to it is still pending. The stand-in holds all stream work back until
// the stream is waited for (device memory is host memory, kernels do nothing),
// which a real runtime may do with any asynchronous copy. Linked with the
// library's own object files; prints one line per fault and exits with 1.
#include <cuda_runtime_api.h>
#include <malloc.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "../include/dbbc.h"

// ------------------------------------------------------------------ stand-in
namespace {
struct Op {
  enum { COPY, FILL, FREE } kind;
  char* dst;
  const char* src;
  size_t n;
  int value;
};
struct Work {  // everything enqueued and not yet run (all streams in order); its memory never goes through delete
  Op ops[4096];
  size_t n = 0;
  const char* call = "";
  int faults = 0;
};
Work& work() {
  static Work* w = new (std::calloc(1, sizeof(Work))) Work;
  return *w;
}
void enqueue(Op op) {
  Work& w = work();
  if (w.n == sizeof(w.ops) / sizeof(w.ops[0])) std::abort();
  w.ops[w.n++] = op;
}
void run_all() {
  Work& w = work();
  for (size_t i = 0; i < w.n; i++) {
    const Op& o = w.ops[i];
    if (o.kind == Op::COPY) std::memcpy(o.dst, o.src, o.n);
    if (o.kind == Op::FILL) std::memset(o.dst, o.value, o.n);
    if (o.kind == Op::FREE) std::free(o.dst);
  }
  w.n = 0;
}
void given_back(void* p) {
  if (!p) return;
  Work& w = work();
  const char* a = static_cast<char*>(p);
  const char* b = a + malloc_usable_size(p);
  for (size_t i = 0; i < w.n; i++) {
    const Op& o = w.ops[i];
    if (o.kind == Op::COPY && ((o.src < b && o.src + o.n > a) || (o.dst < b && o.dst + o.n > a))) {
      std::printf("%s: %zu bytes freed before their copy ran\n", w.call, o.n);
      w.faults++;
      w.ops[i].n = 0;  // not run
    }
  }
}
}  // namespace

void* operator new(size_t n) {
  void* p = std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept {
  given_back(p);
  std::free(p);
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }

extern "C" {
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 4;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidSymbol; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t*, const cudaMemPoolProps*) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  *p = std::calloc(n, 1);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t s) {
  return cudaMallocAsync(p, n, s);
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  enqueue(Op{Op::FREE, static_cast<char*>(p), nullptr, 0, 0});
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t) {
  enqueue(Op{Op::COPY, static_cast<char*>(dst), static_cast<const char*>(src), n, 0});
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* dst, int value, size_t n, cudaStream_t) {
  enqueue(Op{Op::FILL, static_cast<char*>(dst), nullptr, n, value});
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  run_all();
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = nullptr;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = nullptr;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0;
  return cudaSuccess;
}
}

// ------------------------------------------------------------------ calls
namespace {
int g_calls = 0, g_fail_at = -1;  // the allocation that fails

void* hook_alloc(size_t n, void*, void*) { return g_calls++ == g_fail_at ? nullptr : std::calloc(n, 1); }
void hook_free(void* p, void*, void*) { cudaFreeAsync(p, nullptr); }

struct Edges {  // three small graphs, edge lists in host memory
  std::vector<int32_t> u{0, 0, 1, 1, 0, 1, 2, 0}, v{0, 1, 0, 1, 0, 0, 1, 0}, n_u{2, 3, 1}, n_v{2, 2, 1};
  std::vector<int8_t> s{1, -1, 1, 1, 1, -1, 1, 1};
  std::vector<int64_t> off{0, 4, 7, 8};
};

dbbc_graph* build(bool of_union, uint32_t flags = 0) {
  const Edges e;  // the caller's arrays are gone when the call has returned
  dbbc_graph* g = nullptr;
  const dbbc_status st =
      of_union ? dbbc_graph_from_coo_multi(e.u.data(), e.v.data(), e.s.data(), e.off.data(), e.n_u.data(),
                                           e.n_v.data(), 3, flags, nullptr, &g)
               : dbbc_graph_from_coo(e.u.data(), e.v.data(), e.s.data(), 4, 2, 2, flags, nullptr, &g);
  return st == DBBC_OK ? g : nullptr;
}

// Runs `call` with every allocation succeeding, then with each one failing.
template <typename F>
void sweep(const char* name, F&& call) {
  Work& w = work();
  static char label[128];
  w.call = label;
  std::snprintf(label, sizeof(label), "%s", name);
  g_fail_at = -1;
  g_calls = 0;
  const bool ok = call();
  const int n = g_calls;
  if (!ok || n == 0) {
    std::printf("%s: the call failed\n", name);
    w.faults++;
  }
  run_all();
  for (int k = 0; k < n; k++) {
    std::snprintf(label, sizeof(label), "%s, allocation %d fails", name, k);
    g_calls = 0;
    g_fail_at = k;
    if (call()) {
      std::printf("%s: the call succeeded\n", label);
      w.faults++;
    }
    run_all();
  }
  g_fail_at = -1;
}
}  // namespace

int main() {
  dbbc_set_allocator(hook_alloc, hook_free, nullptr);
  for (bool of_union : {false, true})
    sweep(of_union ? "dbbc_graph_from_coo_multi" : "dbbc_graph_from_coo", [&] {
      dbbc_graph* g = build(of_union);
      dbbc_graph_free(g);
      return g != nullptr;
    });
  dbbc_graph* g = build(false);
  dbbc_graph* un = build(true);
  if (!g || !un) return 2;
  uint64_t a[3], b[3];
  sweep("dbbc_count_components", [&] { return dbbc_count_components(un, nullptr, a, b) == DBBC_OK; });
  sweep("dbbc_count_partition", [&] { return dbbc_count_partition(g, nullptr, 0, 2, a, b) == DBBC_OK; });
  const dbbc_graph* gs[2] = {g, g};
  sweep("dbbc_count_batch", [&] { return dbbc_count_batch(gs, 2, nullptr, a, b) == DBBC_OK; });
  sweep("dbbc_count_batch_async", [&] {
    std::vector<uint64_t> out(4);  // stands for device memory
    const bool ok = dbbc_count_batch_async(gs, 2, nullptr, out.data()) == DBBC_OK;
    run_all();
    return ok;
  });
  sweep("dbbc_batch_create", [&] {
    dbbc_batch* p = nullptr;
    const bool ok = dbbc_batch_create(gs, 2, nullptr, &p) == DBBC_OK;
    dbbc_batch_free(p);
    return ok;
  });
  dbbc_graph_free(g);
  dbbc_graph_free(un);
  run_all();
  if (work().faults == 0) std::printf("no host memory freed before its copy\n");
  return work().faults ? 1 : 0;
}
