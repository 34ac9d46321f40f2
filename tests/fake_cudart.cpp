// A CUDA runtime without a GPU, for tests of the library's host code: "device"
// memory is host memory (reserved, not committed), launches and copies are
// recorded in order and kernels do nothing.  Linked with the library's objects
// in place of the runtime (tests/fake_cuda.py).
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstdio>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
std::map<const void*, std::string> g_name;  // kernels by host stub
std::map<void*, size_t> g_mem;
std::vector<float> g_elapsed;
struct Pending { const char* src; std::vector<char> was; cudaStream_t s; };
std::vector<Pending> g_pending;  // uploads that nothing has waited for
size_t g_used, g_limit, g_elapsed_at;
std::string g_log;
struct { dim3 grid, block; size_t smem; cudaStream_t s; } g_call;
int g_host_mapped, g_capturing, g_recording;  // the last: between begin and end of a capture

template <typename... A>
void note(const char* fmt, A... a) {
  char line[512];
  snprintf(line, sizeof line, fmt, a...);
  g_log += line;
  g_log += '\n';
}
cudaError_t launch(const void* f, dim3 g, dim3 b, size_t sm, cudaStream_t s) {
  note("launch %s %u %u %u %u %zu %p", g_name[f].c_str(), g.x, g.y, g.z, b.x * b.y * b.z, sm, (void*)s);
  return g.x > 0 && g.y > 0 && g.y <= 65535 && g.z > 0 && g.z <= 65535 ? cudaSuccess : cudaErrorInvalidConfiguration;
}
}  // namespace

extern "C" {
void fake_reset(size_t limit) {  // bytes that cudaMalloc may hand out at once (0: no limit)
  g_log.clear();
  g_limit = limit;
  g_elapsed.clear();
  g_elapsed_at = 0;
  g_host_mapped = 0;
}
const char* fake_log() { return g_log.c_str(); }
// Uploads under way whose source is no longer what it was at the call (the copy may read it until the stream is waited for).
int fake_lost_uploads() {
  int n = 0;
  for (const Pending& p : g_pending) n += memcmp(p.src, p.was.data(), p.was.size()) != 0;
  return n;
}
void fake_forget_uploads() { g_pending.clear(); }
int fake_uploads() { return (int)g_pending.size(); }
size_t fake_used() { return g_used; }
void fake_elapsed(const float* ms, int n) { g_elapsed.assign(ms, ms + n); g_elapsed_at = 0; }
void fake_capturing(int on) { g_capturing = on; }
void fake_host_mapped(int on) { g_host_mapped = on; }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_name[f] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, cudaStream_t s) {
  g_call = {g, b, sm, s};
  return cudaSuccess;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* s) {
  *g = g_call.grid, *b = g_call.block, *sm = g_call.smem, *(cudaStream_t*)s = g_call.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t sm, cudaStream_t s) {
  return launch((const void*)k, g, b, sm, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream);
}

cudaError_t cudaMalloc(void** p, size_t n) {
  note("malloc %zu", n);
  if (g_limit && g_used + n > g_limit) return cudaErrorMemoryAllocation;
  *p = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (*p == MAP_FAILED) return cudaErrorMemoryAllocation;
  g_mem[*p] = n;
  g_used += n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  note("free %zu", g_mem[p]);
  g_used -= g_mem[p];
  munmap(p, g_mem[p]);
  g_mem.erase(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { note("copy %zu", n); memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  note("copy_async %zu %p", n, (void*)st);
  if (k == cudaMemcpyHostToDevice && !g_recording) g_pending.push_back({(const char*)s, {(const char*)s, (const char*)s + n}, st});
  if (!g_recording) memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t n) { note("memset %zu", n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t n, cudaStream_t s) { note("memset_async %zu %p", n, (void*)s); return cudaSuccess; }
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t n, size_t, cudaMemcpyKind) { note("copy_symbol %zu", n); return cudaSuccess; }
cudaError_t cudaMemcpyFromSymbolAsync(void*, const void*, size_t, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaSuccess; }

cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  note("attribute %s %d %d", g_name[f].c_str(), (int)a, v);
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  a->sharedSizeBytes = 1024;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof *a);
  if (g_host_mapped) a->type = cudaMemoryTypeHost, a->devicePointer = const_cast<void*>(p), a->hostPointer = a->devicePointer;
  return cudaSuccess;
}

cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  note("synchronize %p", (void*)s);
  for (size_t i = g_pending.size(); i-- > 0;)
    if (g_pending[i].s == s) g_pending.erase(g_pending.begin() + i);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)0x51; return cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { *s = (cudaStream_t)0x52; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* a, int* b) { *a = 0, *b = -5; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)0x61; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)0x61; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { g_pending.clear(); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = g_elapsed_at < g_elapsed.size() ? g_elapsed[g_elapsed_at++] : 1.f;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
  *c = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { note("%s", "capture"); g_recording = 1; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)0x71; g_recording = 0; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  note("%s", "instantiate");
  *e = (cudaGraphExec_t)0x72;
  return cudaSuccess;
}
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t, cudaGraph_t, cudaGraphExecUpdateResultInfo* r) {
  note("%s", "update");
  r->result = cudaGraphExecUpdateSuccess;
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { note("graph_launch %p", (void*)s); return cudaSuccess; }
}
