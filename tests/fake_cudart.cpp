// A CUDA runtime without a GPU for tests of the library's host code: streams
// and events are numbers, copies and launches are lines of a log, and the test
// says which call fails and whether a stream is being captured.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <map>
#include <string>

namespace {
std::string log_;
std::map<const void*, std::string> kernels;
size_t next_handle = 0x100;
int copies_until_failure = -1, launches_until_failure = -1;
cudaError_t last = cudaSuccess;
bool capturing = false;

void* handle() { return reinterpret_cast<void*>(next_handle++); }
void line(const char* what, const void* stream, const char* detail = "") {
  char b[64];
  std::snprintf(b, sizeof b, " %zx ", reinterpret_cast<size_t>(stream));
  log_ += what + std::string(b) + detail + "\n";
}
cudaError_t launch(const void* f, cudaStream_t st) {
  if (launches_until_failure == 0) {
    launches_until_failure = -1;
    return last = cudaErrorLaunchFailure;
  }
  if (launches_until_failure > 0) --launches_until_failure;
  line("launch", st, kernels[f].c_str());
  return cudaSuccess;
}
int zero_map(void* map) {
  for (int i = 0; i < 128; ++i) static_cast<char*>(map)[i] = 0;
  return 0;
}
}  // namespace

extern "C" {
const char* fake_log() { return log_.c_str(); }
void fake_clear() { log_.clear(); }
void fake_fail_copy(int n) {
  copies_until_failure = n;
  last = cudaSuccess;
}
void fake_fail_launch(int n) {
  launches_until_failure = n;
  last = cudaSuccess;
}
void fake_capture(int on) { capturing = on; }

cudaError_t cudaMalloc(void** p, size_t n) { return *p = std::calloc(1, n), cudaSuccess; }
cudaError_t cudaFree(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return *p = std::calloc(1, n), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t st) { return line("set", st), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t st) {
  if (copies_until_failure == 0) {
    copies_until_failure = -1;
    return last = cudaErrorInvalidValue;
  }
  if (copies_until_failure > 0) --copies_until_failure;
  return line("copy", st), cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)handle(), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return line("sync", s), cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) { return line("wait", s), cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
  *st = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = (cudaGraph_t)handle(), cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  return *e = (cudaGraphExec_t)handle(), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { return line("graph", s), cudaSuccess; }

cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)handle(), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return *e = (cudaEvent_t)handle(), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t s) { return line("record", s), cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }

cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { return *n = 2, cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 2, cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) { return *a = {}, cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return *p = nullptr, cudaErrorInvalidSymbol; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *f = reinterpret_cast<void*>(zero_map);
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "made by the test"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  return last = cudaSuccess, e;
}

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->stream); }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t st) { return launch(k, st); }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  return *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f)), cudaSuccess;
}
static struct { size_t smem; void* stream; } config;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t smem, cudaStream_t st) {
  config = {smem, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  *g = *b = dim3{1, 1, 1};
  *smem = config.smem;
  *static_cast<void**>(st) = config.stream;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { return static_cast<void**>(handle()); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, void*, void*, void*, void*, int*) {
  kernels[f] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
