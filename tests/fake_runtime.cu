// A CUDA runtime without a device, for host tests: linked with the library's
// objects in the place of the real one.  Device memory is host memory, copies are
// done at once, kernels do nothing (k_setup marks its records valid, a persistent
// sampler ends its runs at once), and what the host code did in an order that
// the device would not keep is noted, one line each (fake_report).
//
// Ordering rules (CUDA programming guide, API synchronisation behaviour): a copy
// of pageable memory or a memset on the default stream may return before it is
// done, and a non-blocking stream does not wait for it; work on two streams has
// no order until the host has waited for one of them; an asynchronous copy may read
// its host array until then.
#include <cuda_runtime.h>
#include <sys/uio.h>
#include <unistd.h>

#include <cerrno>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <vector>

#include "../paper_2607_28265_gb300/csrc/chain.h"

using namespace swig;

namespace {

struct Source {  // of an asynchronous copy to the device
  cudaStream_t stream;
  const void* p;
  std::vector<char> bytes;
};

struct Fake {
  std::mutex lock;
  std::map<const char*, size_t> blocks;           // device allocations
  std::map<const void*, std::string> names;       // kernels by their host stub
  std::map<const void*, int> smem_limit;          // dynamic shared memory allowed
  std::map<const void*, size_t> vars;
  std::set<const void*> hosts;                    // page-locked host allocations
  std::set<cudaStream_t> busy;                    // streams with work the host has not waited for
  std::vector<Source> sources;
  std::map<std::string, long long> calls;
  std::string report;
  int sms = 152;
  bool capturing = false;
  dim3 grid, block;
  size_t shared = 0;
  cudaStream_t stream = nullptr;
  void note(const std::string& s) { report += s + "\n"; }
};
Fake& F() {
  static Fake* f = new Fake;
  return *f;
}

// The bytes from p to the end of its allocation (0: not device memory).
size_t room(const void* p) {
  auto it = F().blocks.upper_bound(static_cast<const char*>(p));
  if (it == F().blocks.begin()) return 0;
  --it;
  const size_t off = static_cast<const char*>(p) - it->first;
  return off < it->second ? it->second - off : 0;
}

void on_write(const char* what, const void* dst, size_t n) {
  if (n > room(dst)) F().note(std::string(what) + ": past the end of its allocation");
}

// The host has waited for st: the arrays that its copies read still have to be
// what they were.
void waited(cudaStream_t st) {
  F().busy.erase(st);
  std::vector<Source> left;
  for (Source& s : F().sources) {
    if (s.stream != st) {
      left.push_back(std::move(s));
      continue;
    }
    std::vector<char> now(s.bytes.size());
    iovec to{now.data(), now.size()}, from{const_cast<void*>(s.p), now.size()};  // (fails where nothing is mapped)
    const ssize_t got = process_vm_readv(getpid(), &to, 1, &from, 1, 0);
    if (got < 0 && errno != EFAULT) continue;  // not allowed here
    if (got != (ssize_t)now.size() || now != s.bytes)
      F().note("cudaMemcpyAsync: host array gone before the copy was waited for");
  }
  F().sources.swap(left);
}

cudaError_t launch(const void* f, dim3 grid, dim3 block, void** args, size_t shared, cudaStream_t st) {
  const std::string& name = F().names[f];
  F().calls["launch"] += 1;
  F().calls["launch " + name] += 1;
  if (F().capturing) return cudaSuccess;
  if (st && F().busy.count(nullptr)) F().note(name + ": launched while a default-stream copy may be under way");
  for (cudaStream_t s : F().busy)
    if (s && s != st && F().calls["check streams"]) F().note(name + ": launched while another stream has work");
  const int limit = F().smem_limit.count(f) ? F().smem_limit[f] : 48 * 1024;
  if ((long long)shared > limit) {
    F().note(name + ": more dynamic shared memory than allowed");
    return cudaErrorInvalidValue;
  }
  F().busy.insert(st);
  if (name.find("k_setup") != std::string::npos) {
    const int n = *static_cast<int*>(args[2]);
    EvalRecord* r = *static_cast<EvalRecord**>(args[3]);
    on_write("k_setup", r, sizeof(EvalRecord) * n);
    for (int i = 0; i < n; ++i) {
      r[i].valid = 1;
      for (int d = 0; d < SWIG_MAX_DET; ++d) r[i].cre[d] = 1.0;
    }
  }
  if (name.find("6k_foldI") != std::string::npos) {
    const LikeConst& L = *static_cast<LikeConst*>(args[0]);
    const int n = *static_cast<int*>(args[3]);
    const FoldStrays& S = *static_cast<FoldStrays*>(args[7]);
    if (room(*static_cast<void**>(args[2])) < sizeof(EvalRecord) * n) F().note("k_fold's records: past the end");
    if (room(S.ctl) < 16 || room(S.list) < 4 * (size_t)n || room(S.done) < 4 * (size_t)n ||
        room(S.part) < sizeof(float) * kPartialStride * L.n_slices * n)
      F().note("k_fold's strays: past the end");
    if ((const char*)S.ctl < *static_cast<char**>(args[2]) + sizeof(EvalRecord) * n &&
        (const char*)S.ctl >= *static_cast<char**>(args[2]))
      F().note("k_fold's strays: over the records");
    if ((size_t)S.part % 16) F().note("k_fold's strays: alignment");
  }
  if (name.find("k_ns_chain") != std::string::npos) {
    const ChainEvent* ev = *static_cast<ChainEvent**>(args[0]);
    const int n_ev = *static_cast<int*>(args[1]);
    for (int e = 0; e < n_ev; ++e) {
      ev[e].P.g->status = ST_TERMINATED;
      ev[e].P.g->iter = 1;
    }
    // every CTA adds its counters to the first event's rows
    if (ev[0].P.cta_prof) on_write("k_ns_chain's CTA counters", ev[0].P.cta_prof, 32 * (size_t)grid.x);
  }
  if (name.find("k_ns_flow") != std::string::npos) {
    const SamplerPtrs* P = static_cast<SamplerPtrs*>(args[3]);
    P->g->status = ST_TERMINATED;
    P->g->iter = 1;
    if (P->cta_prof) on_write("k_ns_flow's CTA counters", P->cta_prof, 32 * (size_t)grid.x);
  }
  return cudaSuccess;
}

cudaError_t copy(const char* what, void* dst, const void* src, size_t n, cudaMemcpyKind kind) {
  F().calls[what] += 1;
  if (kind == cudaMemcpyHostToDevice) on_write(what, dst, n);
  if (kind == cudaMemcpyDeviceToHost && n > room(src)) F().note(std::string(what) + ": reads past its allocation");
  std::memmove(dst, src, n);
  return cudaSuccess;
}

using Guard = std::lock_guard<std::mutex>;

}  // namespace

extern "C" {

int fake_report(char* out, int n) {
  Guard g(F().lock);
  std::strncpy(out, F().report.c_str(), n - 1);
  out[n - 1] = 0;
  return (int)F().report.size();
}
// Clears what was noted and counted; what: "sms" (of the device), "capturing",
// "check streams" are settings, "forget hosts" frees page-locked memory as a device
// reset does, anything else is a count to read.
void fake_reset() {
  Guard g(F().lock);
  F().report.clear();
  F().calls.clear();
}
long long fake_get(const char* what) {
  Guard g(F().lock);
  if (std::string(what) == "bytes") {
    long long n = 0;
    for (const auto& b : F().blocks) n += (long long)b.second;
    return n;
  }
  if (std::string(what) == "hosts") return (long long)F().hosts.size();
  if (std::string(what) == "blocks") return (long long)F().blocks.size();
  return F().calls[what];
}
void fake_set(const char* what, int v) {
  Guard g(F().lock);
  if (std::string(what) == "sms")
    F().sms = v;
  else if (std::string(what) == "forget hosts")
    F().hosts.clear();
  else if (std::string(what) == "capturing")
    F().capturing = v != 0;
  else
    F().calls[what] = v;
}

void** __cudaRegisterFatBinary(void* p) { return (void**)p; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  F().names[host] = name;
}
void __cudaRegisterVar(void**, char* host, char*, const char*, int, size_t size, int, int) { F().vars[host] = size; }
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, cudaStream_t st) {
  F().grid = grid, F().block = block, F().shared = shared, F().stream = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shared, void* st) {
  *grid = F().grid, *block = F().block, *shared = F().shared, *(cudaStream_t*)st = F().stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void** args, size_t shared, cudaStream_t st) {
  Guard g(F().lock);
  return launch((const void*)k, grid, block, args, shared, st);
}

// (the toolkit's headers define some of these for device code: other names here,
// the runtime's in the object file)
#define RT(type, name, args)          \
  type fake_##name args __asm__(#name); \
  type fake_##name args

RT(cudaError_t, cudaLaunchKernelExC, (const cudaLaunchConfig_t* c, const void* f, void** args)) {
  Guard g(F().lock);
  return launch(f, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, c->stream);
}
RT(cudaError_t, cudaLaunchCooperativeKernel, (const void* f, dim3 grid, dim3 block, void** args, size_t shared,
                                        cudaStream_t st)) {
  Guard g(F().lock);
  return launch(f, grid, block, args, shared, st);
}

RT(cudaError_t, cudaMalloc, (void** p, size_t n)) {
  Guard g(F().lock);
  F().calls["cudaMalloc"] += 1;
  if (F().capturing) return cudaErrorStreamCaptureUnsupported;
  *p = std::calloc(1, n ? n : 1);
  F().blocks[(const char*)*p] = n;
  return cudaSuccess;
}
RT(cudaError_t, cudaFree, (void* p)) {
  Guard g(F().lock);
  if (!p) return cudaSuccess;
  F().calls["cudaFree"] += 1;
  if (F().capturing) return cudaErrorStreamCaptureUnsupported;
  if (!F().blocks.erase((const char*)p)) F().note("cudaFree: not an allocation");
  std::free(p);
  return cudaSuccess;
}
RT(cudaError_t, cudaHostAlloc, (void** p, size_t n, unsigned)) {
  Guard g(F().lock);
  F().calls["cudaHostAlloc"] += 1;
  *p = std::calloc(1, n);
  F().hosts.insert(*p);
  return cudaSuccess;
}
RT(cudaError_t, cudaFreeHost, (void* p)) {
  Guard g(F().lock);
  F().calls["cudaFreeHost"] += 1;
  if (!F().hosts.erase(p)) F().note("cudaFreeHost: not an allocation");
  std::free(p);
  return cudaSuccess;
}
RT(cudaError_t, cudaMemcpy, (void* dst, const void* src, size_t n, cudaMemcpyKind kind)) {
  Guard g(F().lock);
  if (kind == cudaMemcpyHostToDevice)
    F().busy.insert(nullptr);
  else
    F().busy.erase(nullptr);  // it waits for its own stream
  return copy("cudaMemcpy", dst, src, n, kind);
}
RT(cudaError_t, cudaMemcpyAsync, (void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t st)) {
  Guard g(F().lock);
  F().busy.insert(st);
  const char* p = static_cast<const char*>(src);
  if (kind == cudaMemcpyHostToDevice) F().sources.push_back({st, src, std::vector<char>(p, p + n)});
  return copy("cudaMemcpyAsync", dst, src, n, kind);
}
RT(cudaError_t, cudaMemset, (void* p, int v, size_t n)) {
  Guard g(F().lock);
  F().busy.insert(nullptr);
  on_write("cudaMemset", p, n);
  std::memset(p, v, n);
  return cudaSuccess;
}
RT(cudaError_t, cudaMemsetAsync, (void* p, int v, size_t n, cudaStream_t st)) {
  Guard g(F().lock);
  F().busy.insert(st);
  on_write("cudaMemsetAsync", p, n);
  std::memset(p, v, n);
  return cudaSuccess;
}

RT(cudaError_t, cudaStreamCreateWithFlags, (cudaStream_t* s, unsigned)) {
  *s = (cudaStream_t)std::malloc(8);
  return cudaSuccess;
}
RT(cudaError_t, cudaStreamDestroy, (cudaStream_t s)) {
  Guard g(F().lock);
  waited(s);
  std::free(s);
  return cudaSuccess;
}
RT(cudaError_t, cudaStreamSynchronize, (cudaStream_t s)) {
  Guard g(F().lock);
  waited(s);
  return cudaSuccess;
}
RT(cudaError_t, cudaStreamIsCapturing, (cudaStream_t, cudaStreamCaptureStatus* s)) {
  *s = F().capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
RT(cudaError_t, cudaEventCreate, (cudaEvent_t* e)) {
  *e = (cudaEvent_t)std::calloc(1, sizeof(cudaStream_t));
  return cudaSuccess;
}
RT(cudaError_t, cudaEventDestroy, (cudaEvent_t e)) {
  std::free(e);
  return cudaSuccess;
}
RT(cudaError_t, cudaEventRecord, (cudaEvent_t e, cudaStream_t s)) {
  *(cudaStream_t*)e = s;
  return cudaSuccess;
}
RT(cudaError_t, cudaEventSynchronize, (cudaEvent_t e)) {  // (recorded behind all of its stream's work)
  Guard g(F().lock);
  waited(*(cudaStream_t*)e);
  return cudaSuccess;
}
RT(cudaError_t, cudaEventElapsedTime_v2, (float* ms, cudaEvent_t, cudaEvent_t)) {
  *ms = 1.0f;
  return cudaSuccess;
}
RT(cudaError_t, cudaEventElapsedTime, (float* ms, cudaEvent_t, cudaEvent_t)) {
  *ms = 1.0f;
  return cudaSuccess;
}

RT(cudaError_t, cudaGetDeviceCount, (int* n)) {
  *n = 1;
  return cudaSuccess;
}
RT(cudaError_t, cudaGetDevice, (int* d)) {
  *d = 0;
  return cudaSuccess;
}
RT(cudaError_t, cudaSetDevice, (int)) { return cudaSuccess; }
RT(cudaError_t, cudaDeviceGetAttribute, (int* v, cudaDeviceAttr a, int)) {
  *v = a == cudaDevAttrMultiProcessorCount ? F().sms : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024 : 0;
  return cudaSuccess;
}
RT(cudaError_t, cudaFuncGetAttributes, (cudaFuncAttributes* a, const void*)) {
  std::memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
RT(cudaError_t, cudaFuncSetAttribute, (const void* f, cudaFuncAttribute, int v)) {
  Guard g(F().lock);
  F().calls["cudaFuncSetAttribute"] += 1;
  if (F().smem_limit.count(f) && v < F().smem_limit[f]) F().note(F().names[f] + ": shared-memory limit lowered");
  F().smem_limit[f] = v;
  return cudaSuccess;
}
RT(cudaError_t, cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags, (int* n, const void*, int, size_t, unsigned)) {
  *n = 1;
  return cudaSuccess;
}
RT(cudaError_t, cudaPointerGetAttributes, (cudaPointerAttributes* a, const void* p)) {
  Guard g(F().lock);
  std::memset(a, 0, sizeof(*a));
  a->type = F().hosts.count(p) ? cudaMemoryTypeHost : room(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
RT(cudaError_t, cudaGetSymbolAddress, (void** p, const void* var)) {
  Guard g(F().lock);
  *p = const_cast<void*>(var);
  F().blocks[(const char*)var] = F().vars[var];
  return cudaSuccess;
}
RT(const char*, cudaGetErrorString, (cudaError_t e)) { return e == cudaSuccess ? "no error" : "fake error"; }
RT(cudaError_t, cudaGetLastError, ()) { return cudaSuccess; }

}  // extern "C"
