#include "fake_cuda.h"

#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <unordered_map>

namespace fake {

State& state() {
  static State s;
  return s;
}

static std::unordered_map<void*, size_t> g_sizes;
static cudaError_t g_last = cudaSuccess;
static uintptr_t g_next = 0x1000;

static cudaError_t work(Op op, cudaStream_t st, uintptr_t ev = 0) {
  State& s = state();
  if (s.work++ == s.fail_at) {
    g_last = cudaErrorUnknown;
    return g_last;
  }
  s.log.push_back({op, (uintptr_t)st, ev});
  return cudaSuccess;
}
static cudaError_t note(Op op, cudaStream_t st, uintptr_t ev = 0) {
  state().log.push_back({op, (uintptr_t)st, ev});
  return cudaSuccess;
}
static cudaError_t take(void** p, size_t bytes) {
  State& s = state();
  const long nr = s.allocations++;
  const bool refuse = s.refuse_at >= 0 && (nr == s.refuse_at || nr == s.refuse_at + 1);
  if (refuse || s.live + s.kept + s.foreign + bytes > s.total) {
    ++s.refused;
    g_last = cudaErrorMemoryAllocation;
    return g_last;
  }
  *p = calloc(1, bytes);
  g_sizes[*p] = bytes;
  s.live += bytes;
  s.high = std::max(s.high, s.live);
  return cudaSuccess;
}
template <typename T>
static cudaError_t handle(T* h) {
  *h = (T)(g_next += 0x10);
  return cudaSuccess;
}

}  // namespace fake

using namespace fake;
typedef cudaError_t E;

extern "C" {

void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
static dim3 g_grid, g_block;
static size_t g_smem;
static cudaStream_t g_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, CUstream_st* st) {
  g_grid = g;
  g_block = b;
  g_smem = sm;
  g_stream = st;
  return 0;
}
E __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* st) {
  *g = g_grid;
  *b = g_block;
  *sm = g_smem;
  *(cudaStream_t*)st = g_stream;
  return cudaSuccess;
}
E __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
E __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t st) { return work(LAUNCH, st); }
E cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) { return work(LAUNCH, c->stream); }
E cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t st) {
  const E e = work(COPY, st);
  if (e != cudaSuccess || kind == cudaMemcpyDeviceToDevice) return e;
  memcpy(dst, src, n);
  // results of reductions: up to four inner products, or a table of norms
  if (kind == cudaMemcpyDeviceToHost && state().ones && (n > 256 || n == 16 || n == 32))
    std::fill_n((double*)dst, n / sizeof(double), 1.0);
  return e;
}
E cudaMemsetAsync(void*, int, size_t, cudaStream_t st) { return work(MEMSET, st); }
E cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return take(p, n); }
E cudaMallocAsync(void** p, size_t n, cudaStream_t) { return take(p, n); }
E cudaFreeAsync(void* p, cudaStream_t st) {
  state().live -= g_sizes[p];
  state().kept += g_sizes[p];
  g_sizes.erase(p);
  free(p);
  return note(FREE, st);
}
E cudaMallocHost(void** p, size_t n) {
  *p = calloc(1, n);
  ++state().host_blocks;
  return cudaSuccess;
}
E cudaFreeHost(void* p) {
  --state().host_blocks;
  free(p);
  return cudaSuccess;
}
E cudaMemGetInfo(size_t* f, size_t* t) {
  *t = state().total;
  *f = state().total - state().live - state().kept - state().foreign;
  return cudaSuccess;
}
E cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { return handle(p); }
E cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
E cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void* v) {
  *(uint64_t*)v = state().live + (a == cudaMemPoolAttrReservedMemCurrent ? state().kept : 0);
  return cudaSuccess;
}
E cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void* v) {
  if (a == cudaMemPoolAttrReleaseThreshold) state().threshold = *(uint64_t*)v;
  return cudaSuccess;
}
E cudaMemPoolTrimTo(cudaMemPool_t, size_t) {
  if (state().kept) ++state().trims;
  state().kept = 0;
  return cudaSuccess;
}
E cudaEventCreate(cudaEvent_t* e) { return handle(e); }
E cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
E cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
E cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}
E cudaEventRecord(cudaEvent_t e, cudaStream_t st) { return work(RECORD, st, (uintptr_t)e); }
E cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t st, unsigned) { return work(RECORD, st, (uintptr_t)e); }
E cudaEventSynchronize(cudaEvent_t e) { return note(EVENT_SYNC, nullptr, (uintptr_t)e); }
E cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
E cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
E cudaStreamSynchronize(cudaStream_t st) {
  State& s = state();
  s.kept = std::min(s.kept, s.threshold > s.live ? s.threshold - s.live : 0);
  return note(STREAM_SYNC, st);
}
E cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) { return note(STREAM_WAIT, st, (uintptr_t)e); }
E cudaDeviceSynchronize() { return cudaSuccess; }
E cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
// no capture: the solver launches its steps directly, on the same stream
E cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
E cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
E cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
E cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
E cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
E cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
E cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
E cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
  return cudaSuccess;
}
E cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
E cudaGetSymbolAddress(void** p, const void*) {
  *p = nullptr;
  return cudaSuccess;
}
E cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
E cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 1;
  return cudaSuccess;
}
E cudaGetLastError() {
  const E e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(E) { return "error made by the test"; }

}  // extern "C"
