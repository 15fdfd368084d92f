// A CUDA runtime without a GPU, for tests of the host code: the library's
// objects are linked with it in place of the real one.  Device memory is host
// memory, copies and fills are made at once, kernels do nothing, and every call
// that puts work on a stream leaves a line in a log, in program order:
//   launch NAME STREAM GX GY GZ ARG2 ARG3   (pointer arguments 2, 3 of the copy kernels, else 0)
//   copy KIND DST SRC BYTES STREAM          (STREAM "sync": cudaMemcpy)
//   fill DST BYTES STREAM
//   record EVENT STREAM / wait STREAM EVENT / sync STREAM
// A launch outside the grid limits fails, as the real one does.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <string>

static std::string g_log;
static std::map<const void*, std::string> g_names;
static cudaError_t g_last = cudaSuccess;
static const char *g_far_lo = nullptr, *g_far_hi = nullptr;
static size_t g_handles = 0x100;

static void note(const char* fmt, ...) {
  char line[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(line, sizeof line, fmt, ap);
  va_end(ap);
  g_log += line;
  g_log += '\n';
}
static void move(void* d, const void* s, size_t n) {
  if (n <= 1 << 20) memcpy(d, s, n);
}
template <typename T>
static T fresh() { return (T)(g_handles += 0x10); }

extern "C" {
const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
// memory of another device from here on
void fake_foreign(const void* p, size_t n) { g_far_lo = (const char*)p; g_far_hi = g_far_lo + n; }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

static struct { dim3 g, b; size_t smem; void* st; } g_cfg;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* st) {
  g_cfg = {g, b, smem, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  *g = g_cfg.g;
  *b = g_cfg.b;
  *smem = g_cfg.smem;
  *(void**)st = g_cfg.st;
  return cudaSuccess;
}
static cudaError_t launch(const void* f, dim3 g, void** args, void* st) {
  const std::string& name = g_names[f];
  if (g.x < 1 || g.y < 1 || g.z < 1 || g.x > 0x7fffffffu || g.y > 65535 || g.z > 65535) {
    note("refused %s", name.c_str());
    return g_last = cudaErrorInvalidConfiguration;
  }
  const bool copies = name.find("pack_kernel") != std::string::npos;
  note("launch %s %p %u %u %u %p %p", name.c_str(), st, g.x, g.y, g.z, copies ? *(void**)args[2] : nullptr,
       copies ? *(void**)args[3] : nullptr);
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void** args, size_t, cudaStream_t st) {
  return launch((const void*)k, g, args, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  return launch(f, c->gridDim, args, c->stream);
}

cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) { *lo = 0; *hi = -5; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeDevice;
  a->device = (const char*)p >= g_far_lo && (const char*)p < g_far_hi ? 1 : 0;
  a->devicePointer = (void*)p;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
static CUresult encode_map(void) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *f = (void*)encode_map;
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaErrorInvalidSymbol; }

cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
  note("copy %d %p %p %zu sync", (int)k, d, s, n);
  move(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  note("copy %d %p %p %zu %p", (int)k, d, s, n, (void*)st);
  move(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind k,
                              cudaStream_t st) {
  note("copy %d %p %p %zu %p", (int)k, d, s, w * h, (void*)st);
  for (size_t r = 0; r < h; ++r) move((char*)d + r * dp, (const char*)s + r * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  note("fill %p %zu %p", d, n, (void*)st);
  if (n <= 1 << 20) memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { *s = fresh<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { note("sync %p", (void*)st); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) {
  note("wait %p %p", (void*)st, (void*)e);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = fresh<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = fresh<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
  note("record %p %p", (void*)e, (void*)st);
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
}
