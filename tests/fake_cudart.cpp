// A stand-in for the CUDA runtime, linked into a copy of the library so that its host code runs without a GPU.
//
// "Device" memory is host memory.  Every asynchronous call is queued, on one stream, and executed as late as the
// documentation allows: when the stream or an event behind it is waited for, or by a synchronous call.  A copy from
// ordinary host memory is no exception ("might be synchronous" promises nothing), so a source that was changed before the
// copy ran is seen: the copy keeps the bytes that it was given and compares.  Kernels do nothing; their names are kept.
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <map>
#include <set>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "ss_internal.h"

namespace {
struct Op {
  enum Kind { kCopy, kCopy2D, kSet, kKernel, kEvent } kind;
  std::string name;                       // kernel
  void* dst = nullptr;
  const void* src = nullptr;
  size_t n = 0, dpitch = 0, spitch = 0, rows = 1;
  int value = 0;
  std::vector<uint8_t> given;             // host source at the time of the call
};
struct Event {
  uint64_t at = 0;                        // operations that precede it
};
std::deque<Op> queue;
uint64_t enqueued = 0, executed = 0;
int64_t changed_sources = 0;
std::string bad_kernel;                   // the kernel (part of its name) whose execution fails, once, and how
cudaError_t bad_kernel_error = cudaSuccess, pending_error = cudaSuccess;
std::map<const void*, std::string>& kernel_names() {      // filled while other objects are still being constructed
  static std::map<const void*, std::string> names;
  return names;
}

void execute(const Op& op) {
  switch (op.kind) {
    case Op::kCopy:
      if (!op.given.empty() && std::memcmp(op.given.data(), op.src, op.n) != 0) ++changed_sources;
      std::memcpy(op.dst, op.src, op.n);
      break;
    case Op::kCopy2D:
      for (size_t r = 0; r < op.rows; ++r)
        std::memcpy((char*)op.dst + r * op.dpitch, (const char*)op.src + r * op.spitch, op.n);
      break;
    case Op::kSet: std::memset(op.dst, op.value, op.n); break;
    case Op::kKernel:
      if (!bad_kernel.empty() && op.name.find(bad_kernel) != std::string::npos) {
        pending_error = bad_kernel_error;
        bad_kernel.clear();
      }
      break;
    default: break;
  }
}
void run_until(uint64_t at) {
  while (executed < at && !queue.empty()) {
    execute(queue.front());
    queue.pop_front();
    ++executed;
  }
}
cudaError_t waited() {                    // the next wait reports an error, once
  const cudaError_t e = pending_error;
  pending_error = cudaSuccess;
  return e;
}
void add(Op op) { queue.push_back(std::move(op)); ++enqueued; }
std::set<std::string> loaded_kernels;                   // kernels that an attribute was set for (a real one is loaded by that)
std::map<std::string, long long> wait_limits;            // what the prompt-pass kernels were last told, by name
void add_kernel(const void* fn, void** args) {
  Op op{Op::kKernel};
  op.name = kernel_names()[fn];
  if (op.name.find("gemm_wx") != std::string::npos) wait_limits[op.name] = ((const ss::GemmArgs*)args[2])->wait_limit;
  if (op.name.find("attn_prefill") != std::string::npos) wait_limits[op.name] = *(const long long*)args[5];
  add(op);
}
int encode_tiled(...) { return 0; }
}  // namespace

extern "C" {
// ---- what a test asks
int64_t fake_changed_sources() { return changed_sources; }
void fake_fail_wait_behind(const char* part, int error) { bad_kernel = part; bad_kernel_error = (cudaError_t)error; }
// The limit (SM cycles) that the last launch of the kernel was given, -1 if there was none.
int64_t fake_wait_limit(const char* part) {
  for (const auto& w : wait_limits)
    if (w.first.find(part) != std::string::npos) return w.second;
  return -1;
}
// Kernels loaded since the last call whose (mangled) name contains `part`.
int64_t fake_loaded(const char* part) {
  int64_t n = 0;
  for (const std::string& k : loaded_kernels) n += k.find(part) != std::string::npos;
  loaded_kernels.clear();
  return n;
}
// Launches of kernels whose (mangled) name contains `part` that have not been executed.
int64_t fake_pending(const char* part) {
  int64_t n = 0;
  for (const Op& op : queue) n += op.kind == Op::kKernel && op.name.find(part) != std::string::npos;
  return n;
}

// ---- the runtime
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  kernel_names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }

cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 148 : a == cudaDevAttrClockRate ? 1965000 : 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidSymbol; }
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult*) {
  *fn = (void*)&encode_tiled;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute, int) { loaded_kernels.insert(kernel_names()[fn]); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(n, 1); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }

cudaError_t cudaLaunchKernel(const void* fn, dim3, dim3, void** args, size_t, cudaStream_t) { add_kernel(fn, args); return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* fn, void** args) { add_kernel(fn, args); return cudaSuccess; }
cudaError_t cudaLaunchCooperativeKernel(const void* fn, dim3, dim3, void** args, size_t, cudaStream_t) { add_kernel(fn, args); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }

cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  Op op{Op::kCopy};
  op.dst = dst; op.src = src; op.n = n;
  if (kind == cudaMemcpyHostToDevice) op.given.assign((const uint8_t*)src, (const uint8_t*)src + n);
  add(op);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* dst, size_t dpitch, const void* src, size_t spitch, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
  Op op{Op::kCopy2D};
  op.dst = dst; op.src = src; op.n = w; op.dpitch = dpitch; op.spitch = spitch; op.rows = h;
  add(op);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* dst, int value, size_t n, cudaStream_t) {
  Op op{Op::kSet};
  op.dst = dst; op.value = value; op.n = n;
  add(op);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind) {
  run_until(enqueued);
  std::memcpy(dst, src, n);
  return waited();
}
cudaError_t cudaMemset(void* dst, int value, size_t n) {
  run_until(enqueued);
  std::memset(dst, value, n);
  return waited();
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { run_until(enqueued); return waited(); }

cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t) new Event; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete (Event*)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
  add(Op{Op::kEvent});
  ((Event*)e)->at = enqueued;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { run_until(((Event*)e)->at); return waited(); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}
