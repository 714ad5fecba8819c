// A CUDA runtime without a GPU for the library's host code: device memory is
// host memory, copies and memsets run at once, kernels do nothing, and every call
// that matters for ordering is written to a log.  Two devices.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <map>
#include <string>

namespace {

struct Poke {
  size_t size, offset;
  uint32_t value;
};

std::string g_log;
std::map<char*, std::pair<size_t, int>> g_mem;  // device memory: bytes, device
std::deque<Poke> g_pokes;
std::map<const void*, std::string> g_kernels;
int g_device = 0;
cudaError_t g_error = cudaSuccess;  // of a launch
void* g_capturing = nullptr;  // stream under capture
uintptr_t g_next = 0x1000;    // streams, events, pools

void note(const char* what, const void* p = nullptr) {
  char line[160];
  snprintf(line, sizeof(line), "%s dev=%d ptr=%p\n", what, g_device, p);
  g_log += line;
}

void* device_alloc(size_t bytes) {
  char* p = (char*)aligned_alloc(256, (bytes + 511) / 256 * 256);
  memset(p, 0xA5, bytes);
  g_mem[p] = {bytes, g_device};
  return p;
}

void device_free(void* p) {
  g_mem.erase((char*)p);
  free(p);
}

const std::pair<size_t, int>* device_of(const void* p) {
  auto it = g_mem.upper_bound((char*)p);
  if (it == g_mem.begin()) return nullptr;
  --it;
  return (char*)p < it->first + it->second.first ? &it->second : nullptr;
}

template <typename T>
T handle() {
  return (T)(g_next += 16);
}

cudaError_t copy(void* dst, const void* src, size_t n, cudaMemcpyKind kind) {
  memcpy(dst, src, n);
  if (kind == cudaMemcpyDeviceToHost)
    for (auto it = g_pokes.begin(); it != g_pokes.end(); ++it)
      if (it->size == n) {
        memcpy((char*)dst + it->offset, &it->value, 4);
        g_pokes.erase(it);
        break;
      }
  return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- the test's side
const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
void fake_set_capturing(void* stream) { g_capturing = stream; }
// The next device-to-host copy of `size` bytes gets `value` at `offset`.
void fake_poke(size_t size, size_t offset, uint32_t value) { g_pokes.push_back({size, offset, value}); }
void* fake_alloc(size_t bytes) { return device_alloc(bytes); }
void fake_free(void* p) { device_free(p); }
size_t fake_allocations() { return g_mem.size(); }

// ---- devices
cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_device = d; note("set"); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { note("sync"); return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 1;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_error;
  g_error = cudaSuccess;
  return e;
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) { *p = device_alloc(n); note("malloc", *p); return cudaSuccess; }
cudaError_t cudaFree(void* p) { note("free", p); if (p) device_free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { note("free_async", p); device_free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { *p = handle<cudaMemPool_t>(); return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t) { note("trim", p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return copy(d, s, n, k); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  if (k == cudaMemcpyHostToDevice) note(g_capturing && st == g_capturing ? "captured_upload" : "upload", d);
  return copy(d, s, n, k);
}
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyToSymbolAsync(const void*, const void*, size_t, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = device_alloc(8 << 20); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof(*a));
  const auto* m = device_of(p);
  a->type = m ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  a->device = m ? m->second : 0;
  return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = handle<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { note("sync_stream", s); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
  *st = g_capturing && s == g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = handle<cudaGraph_t>(); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = handle<cudaGraphExec_t>(); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }

// ---- kernels
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 1; return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3, void**, size_t, cudaStream_t) {
  char line[64];
  snprintf(line, sizeof(line), "grid=%ux%ux%u ", grid.x, grid.y, grid.z);
  const auto it = g_kernels.find(f);
  note((std::string("launch ") + line + (it == g_kernels.end() ? "?" : it->second)).c_str());
  if (grid.x < 1 || grid.y < 1 || grid.z < 1 || grid.y > 65535 || grid.z > 65535)
    g_error = cudaErrorInvalidConfiguration;
  return g_error;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** a, size_t sm, cudaStream_t s) {
  return cudaLaunchKernel((const void*)k, g, b, a, sm, s);
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
static struct { dim3 g, b; size_t sm; cudaStream_t s; } g_call;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, cudaStream_t s) {
  g_call.g = g; g_call.b = b; g_call.sm = sm; g_call.s = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* s) {
  *g = g_call.g; *b = g_call.b; *sm = g_call.sm; *(cudaStream_t*)s = g_call.s;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, void*, void*, void*, void*, int*) {
  g_kernels[f] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

}  // extern "C"
