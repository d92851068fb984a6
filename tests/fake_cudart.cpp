// A CUDA runtime without a device, for tests of the host driver: device memory
// is host memory, launches do nothing, and the calls a test names fail.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>

#include "feti.h"
#include "feti_internal.h"

namespace {
std::mutex mu;
cudaError_t last = cudaSuccess;
std::map<void*, size_t> live;   // device allocations
size_t live_bytes = 0, peak_bytes = 0, capacity = (size_t)-1;
int refuse = 0;                 // 1: launches of the fixed-point apply are refused while a stream is captured
int capturing = 0, graphs = 0, graph_launches = 0, fixed_launches = 0;
float cost[3] = {};             // of the fixed-point, row and block products' launches
float now = 0.0f;               // the costs of what was launched
cudaError_t fail(cudaError_t e) { return last = e; }
}  // namespace

extern "C" {
void fake_reset() {
  last = cudaSuccess;
  capacity = (size_t)-1;
  peak_bytes = live_bytes;
  refuse = capturing = graphs = graph_launches = fixed_launches = 0;
  cost[0] = cost[1] = cost[2] = 0.0f;
}
void fake_capacity(size_t bytes) { capacity = bytes; }
void fake_cost(float fixed, float rows, float block) { cost[0] = fixed, cost[1] = rows, cost[2] = block; }
void fake_refuse_in_capture(int on) { refuse = on; }
size_t fake_live_bytes() { return live_bytes; }
size_t fake_peak_bytes() { return peak_bytes; }
int fake_count(int what) { return what == 0 ? graphs : what == 1 ? graph_launches : what == 2 ? fixed_launches : capturing; }


feti_status feti_dual_apply_noalloc(feti_ctx*, const double*, double*, double*) { return FETI_ERR_STATE; }

long fake_rows_launch() { return now += cost[1], 0; }
long fake_block_launch() { return now += cost[2], 0; }
long fake_fixed_launch() {
  ++fixed_launches;
  now += cost[0];
  return refuse && capturing ? fail(cudaErrorInvalidValue) : cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t n) {
  std::lock_guard<std::mutex> lk(mu);
  if (n > capacity || live_bytes > capacity - n) return fail(cudaErrorMemoryAllocation);
  *p = std::calloc(n ? n : 1, 1);
  live[*p] = n;
  live_bytes += n;
  if (live_bytes > peak_bytes) peak_bytes = live_bytes;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  std::lock_guard<std::mutex> lk(mu);
  if (!p) return cudaSuccess;
  auto it = live.find(p);
  if (it == live.end()) return fail(cudaErrorInvalidValue);
  live_bytes -= it->second;
  live.erase(it);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
  for (size_t i = 0; i < h; ++i) std::memcpy((char*)d + i * dp, (const char*)s + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError() { return last; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "fake error"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 2000000; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return capturing ? fail(cudaErrorStreamCaptureUnsupported) : cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  if (capturing) return fail(cudaErrorIllegalState);
  capturing = 1;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { capturing = 0; *g = (cudaGraph_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  ++graphs;
  *e = (cudaGraphExec_t)std::malloc(1);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { std::free(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { ++graph_launches; return capturing ? fail(cudaErrorIllegalState) : cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)std::calloc(1, sizeof(float)); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { *(float*)e = now; return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { *ms = 1.0f + *(float*)b - *(float*)a; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult*) {
  *f = nullptr;
  return fail(cudaErrorInvalidValue);
}
}

namespace feti {
int64_t fix_entries(int m) { return (int64_t)m * (m + 16) / 2; }
int64_t chol_scratch_bytes(int n, int) { return 1024 * (int64_t)n; }
bool symv_fixed_fits(int) { return true; }
int scatter_partials() { return 304; }
cudaError_t noalloc_scratch_lookup(double** p, size_t* n) { *p = nullptr; *n = 0; return cudaSuccess; }
}  // namespace feti
