// A CUDA runtime that runs nothing: it logs the launches, stream waits, event records
// and stream synchronisations that the library issues, so that its schedules are
// tested without a GPU.  Device memory is never touched (device addresses may be
// invented); copies to the host deliver zeros, which the library reads as a clean run.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <map>
#include <string>

static std::string g_log;
static std::map<const void*, std::string> g_names;
static size_t g_next = 1;
static int g_capturing = 0;
struct Config { dim3 grid, block; size_t smem; void* stream; };
static Config g_config;

static void line(const char* what, const char* name, size_t a, size_t b, dim3 g = dim3(0, 0, 0)) {
  char buf[512];
  snprintf(buf, sizeof buf, "%s %s %zu %zu %u %u %u\n", what, name, a, b, g.x, g.y, g.z);
  g_log += buf;
}
static size_t id(const void* p) { return (size_t)p; }
template <class T> static cudaError_t make(T* out) {
  *out = (T)(g_next++);
  return cudaSuccess;
}

extern "C" {
const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* s) {
  g_config = Config{grid, block, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  *grid = g_config.grid;
  *block = g_config.block;
  *smem = g_config.smem;
  *(void**)s = g_config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void**, size_t, cudaStream_t s) {
  line("launch", g_names[(const void*)k].c_str(), id(s), g_capturing, grid);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  line("launch", g_names[f].c_str(), id(c->stream), g_capturing, c->gridDim);
  return cudaSuccess;
}

cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrL2CacheSize ? 132644864 : (a == cudaDevAttrMultiProcessorCount ? 152 : 0);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return make(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return make(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  line("record", "-", id(s), id(e));
  return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) {
  return cudaEventRecord(e, s);
}
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
static int fake_encode(void* map, ...) {
  memset(map, 0, 128);
  return 0;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             enum cudaDriverEntryPointQueryResult* q) {
  *f = (void*)fake_encode;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = (void*)(size_t)0x700000000000;
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  return make(x);
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) {
  line("graph", "-", id(s), id(x));
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t) {
  *p = (void*)((size_t)0x600000000000 + (g_next++ << 40));
  return cudaSuccess;
}
static cudaError_t copy(void* dst, size_t n, enum cudaMemcpyKind k) {
  if (k == cudaMemcpyDeviceToHost) memset(dst, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void*, size_t n, enum cudaMemcpyKind k) {
  return copy(dst, n, k);
}
cudaError_t cudaMemcpyAsync(void* dst, const void*, size_t n, enum cudaMemcpyKind k, cudaStream_t s) {
  line(k == cudaMemcpyDeviceToHost ? "d2h" : "h2d", "-", id(s), n);
  return copy(dst, n, k);
}
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t n, size_t, enum cudaMemcpyKind) {
  line("symbol", "-", 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, enum cudaStreamCaptureMode) {
  g_capturing = 1;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  g_capturing = 0;
  return make(g);
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return make(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  line("sync", "-", id(s), 0);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  line("wait", "-", id(s), id(e));
  return cudaSuccess;
}
}
