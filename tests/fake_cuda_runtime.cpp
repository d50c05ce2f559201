// Stands in for the CUDA runtime and for the kernels' launchers when csrc/asl_api.cu is compiled for the CPU: every
// launch, event record and wait is written to a log from which a test works out what is ordered behind what.  A stream is
// a number whose hundreds digit names its device.  fake_fail makes the n-th call of one name (from now on) fail.
#include <map>
#include <string>

#include "asl_internal.cuh"

namespace {
struct Event { int id, device; };
std::string g_log, g_fail;
int g_device = 0, g_events = 0, g_alive = 0, g_in = 0;

bool fails(const char* name) { return g_fail == name && --g_in == 0; }
int number(const void* p) { return (int)reinterpret_cast<uintptr_t>(p); }
void note(const char* what, int a, int b) { g_log += std::string(what) + " " + std::to_string(a) + " " + std::to_string(b) + "\n"; }
asl_status launch(const char* name, cudaStream_t st) {
  if (fails(name)) return ASL_ERR_CUDA;
  g_log += std::string("run ") + name + " " + std::to_string(number(st)) + "\n";
  return ASL_OK;
}
cudaError_t on_device(cudaEvent_t e, cudaStream_t st) {
  return reinterpret_cast<Event*>(e)->device == number(st) / 100 ? cudaSuccess : cudaErrorInvalidResourceHandle;
}
}  // namespace

extern "C" {
const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
void fake_fail(const char* name, int nth) { g_fail = name; g_in = nth; }
int fake_alive() { return g_alive; }                       // events and allocations not yet given back
int fake_device() { return g_device; }

cudaError_t cudaGetDeviceCount(int* n) { *n = 2; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) { *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : 148; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  if (fails("malloc")) return cudaErrorMemoryAllocation;
  *p = malloc(n);
  ++g_alive;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { free(p); --g_alive; return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { if (fails("memset")) return cudaErrorInvalidValue; memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  if (fails("event")) return cudaErrorMemoryAllocation;
  *e = reinterpret_cast<cudaEvent_t>(new Event{g_events++, g_device});
  ++g_alive;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete reinterpret_cast<Event*>(e); --g_alive; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
  if (!e || on_device(e, st) != cudaSuccess) return cudaErrorInvalidResourceHandle;
  note("record", reinterpret_cast<Event*>(e)->id, number(st));
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) {
  if (!e) return cudaErrorInvalidResourceHandle;
  note("wait", reinterpret_cast<Event*>(e)->id, number(st));
  return cudaSuccess;
}
}  // extern "C"

asl_status asl_launch_window_lse(asl_ctx*, const char*, float*, cudaStream_t st) { return launch("lse", st); }
bool asl_tc_plan(asl_ctx* c) { c->tc.nchunk = c->tc.nseg = 1; c->tc.NC = 128; return true; }
void asl_tc_free(asl_ctx*) {}
size_t asl_tc_partial_bytes(const asl_ctx*) { return 256; }
asl_status asl_tc_reset_sync(asl_ctx*, cudaStream_t) { return ASL_OK; }
asl_status asl_launch_wait_selftest(asl_ctx*, int, unsigned long long, cudaStream_t st) { return launch("selftest", st); }
asl_status asl_launch_score_tc(asl_ctx*, const void*, const void*, const float*, float*, char*, bool, cudaStream_t st) { return launch("score", st); }
asl_status asl_launch_pool(asl_ctx*, const float*, float*, float*, cudaStream_t st) { return launch("pool", st); }
asl_status asl_launch_live_phases(asl_ctx*, bool, bool, cudaStream_t st) { return launch("live", st); }
asl_status asl_launch_rank(asl_ctx*, const float*, int32_t, int32_t, int32_t*, asl_stat*, char*, cudaStream_t st) { return launch("rank", st); }
asl_status asl_rank_ready() { return ASL_OK; }
asl_status asl_launch_topk(asl_ctx*, const float*, int32_t, int32_t*, const asl_stat*, int32_t, char*, cudaStream_t st) { return launch("topk", st); }
bool asl_topk_plan(asl_ctx*) { return true; }
size_t asl_topk_scratch_bytes(int64_t, int64_t) { return 256; }
asl_status asl_launch_compact(asl_ctx*, const void*, const void*, const int32_t*, void*, void*, cudaStream_t st) { return launch("compact", st); }
asl_status asl_launch_compact_rows(asl_ctx*, const void*, const int32_t*, void*, int64_t, cudaStream_t st) { return launch("rows", st); }
