// A stand-in for the CUDA runtime, loaded before it (LD_PRELOAD) where there is no GPU.  Device memory
// is host memory and kernels do nothing: what it keeps is the order of the library's calls, and it
// reports the orders that CUDA does not promise:
//   - work enqueued on a non-blocking stream while an upload (cudaMemcpy from pageable memory,
//     cudaMemcpyToSymbol) or a cudaMemset on the default stream may not have landed: both can return
//     before the device is done, and a non-blocking stream does not wait for the default one;
//   - a copy or cudaMemset on the default stream, over device memory, while work on a non-blocking stream
//     may still be running.
// A device or stream synchronisation, a copy back to the host on the same stream and a wait for an event
// recorded behind the work end what is pending.  cudaFree is not counted on.  It also lists the launches.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

namespace {
std::string report, uploads;              // violations; what is pending on the default stream
std::string launches;                      // kernels in the order of their launches: name, grid, block
std::map<cudaStream_t, std::string> busy;  // pending work of the other streams
std::map<cudaEvent_t, cudaStream_t> recorded;
std::set<cudaStream_t> capturing;
std::map<const void*, std::string> names;  // host entry -> kernel name
struct Call { dim3 g, b; size_t sm; cudaStream_t s; };
std::vector<Call> calls;
long serial = 0;

void violation(const std::string& m) { report += m + "\n"; }
cudaError_t enqueue(cudaStream_t s, const std::string& what) {
  if (capturing.count(s)) return cudaSuccess;
  if (!uploads.empty()) violation(what + " enqueued while pending on the default stream: " + uploads);
  busy[s] = what;
  return cudaSuccess;
}
cudaError_t launch(cudaStream_t s, const std::string& name, dim3 g, dim3 b) {
  launches += name + " " + std::to_string(g.x) + " " + std::to_string(b.x) + "\n";
  return enqueue(s, name);
}
void on_default(const std::string& what, bool pending) {
  for (auto& b : busy)
    if (!b.second.empty()) violation(what + " on the default stream while pending elsewhere: " + b.second);
  if (pending) uploads += (uploads.empty() ? "" : ", ") + what;
  else uploads.clear();
}
size_t free_bytes() {  // free device memory, as long as the test says so
  const char* e = getenv("ORDER_FREE");
  return e ? strtoull(e, nullptr, 10) : (size_t)200 << 30;
}
std::string sized(const char* op, size_t n) { return std::string(op) + " of " + std::to_string(n) + " bytes"; }
}  // namespace

extern "C" {
const char* order_report() { return report.c_str(); }
const char* order_launches() { return launches.c_str(); }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, CUstream_st* s) {
  calls.push_back({g, b, sm, s});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* s) {
  const Call c = calls.back();
  calls.pop_back();
  *g = c.g;
  *b = c.b;
  *sm = c.sm;
  *static_cast<cudaStream_t*>(s) = c.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
  *k = (cudaKernel_t)host;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t, cudaStream_t s) {
  return launch(s, names[(const void*)k], g, b);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(c->stream, names[f], c->gridDim, c->blockDim);
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { return enqueue(s, "a graph"); }

cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
  on_default(sized("cudaMemcpy", n), k != cudaMemcpyDeviceToHost);
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t n, size_t, cudaMemcpyKind) {
  uploads += sized(uploads.empty() ? "cudaMemcpyToSymbol" : ", cudaMemcpyToSymbol", n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  on_default(sized("cudaMemset", n), true);
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  memcpy(d, s, n);
  return enqueue(st, sized("cudaMemcpyAsync", n));
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  memset(d, v, n);
  return enqueue(st, sized("cudaMemsetAsync", n));
}
cudaError_t cudaDeviceSynchronize() {
  uploads.clear();
  busy.clear();
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  busy[s].clear();
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  recorded[e] = s;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return cudaStreamSynchronize(recorded[e]); }

cudaError_t cudaMalloc(void** p, size_t n) {
  *p = n > free_bytes() ? nullptr : aligned_alloc(256, (n + 255) / 256 * 256);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
  *f = free_bytes();
  *t = (size_t)280 << 30;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)(0x1000 + 16 * ++serial); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { capturing.insert(s); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  capturing.erase(s);
  *g = (cudaGraph_t)(0x1000 + 16 * ++serial);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = (cudaGraphExec_t)(0x1000 + 16 * ++serial);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)(0x1000 + 16 * ++serial); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrComputeCapabilityMajor ? 10
       : a == cudaDevAttrComputeCapabilityMinor ? 3
       : a == cudaDevAttrMultiProcessorCount ? 152
       : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 1;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  a->maxThreadsPerBlock = 512;
  a->sharedSizeBytes = 1024;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = 1; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error of the stand-in runtime"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
}
