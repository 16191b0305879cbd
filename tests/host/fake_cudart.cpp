// The part of the CUDA runtime that the library's host code calls, without a GPU: kernel launches and
// shared-memory grants are recorded per device and everything else succeeds without doing anything.
// A launch that asks for more than 48 KB of dynamic shared memory without a grant on the current
// device fails, as it does on a GPU.  Linked with the library's object files by
// tests/test_host_launches.py.
#include <cuda_runtime_api.h>

#include <map>
#include <string>
#include <utility>
#include <vector>

namespace {
struct Launch { std::string name; unsigned grid[3], block[3]; size_t smem; int device; };
std::map<const void*, std::string>& names() { static std::map<const void*, std::string> m; return m; }
std::vector<Launch> launches;
std::map<std::pair<int, const void*>, size_t> granted;   // (device, kernel) -> bytes
int device = 0, occupancy_queries = 0;
cudaError_t last = cudaSuccess;
struct Config { dim3 grid, block; size_t smem; cudaStream_t st; } config;
}  // namespace

extern "C" {

void fake_set_device(int d) { device = d; }
void fake_clear() { launches.clear(); occupancy_queries = 0; }
int fake_count() { return (int)launches.size(); }
int fake_occupancy_queries() { return occupancy_queries; }
const char* fake_name(int i) { return launches[i].name.c_str(); }
void fake_dims(int i, unsigned long long* out) {
  for (int k = 0; k < 3; ++k) { out[k] = launches[i].grid[k]; out[3 + k] = launches[i].block[k]; }
  out[6] = launches[i].smem;
}

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t st) {
  config = Config{grid, block, smem, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st) {
  *grid = config.grid;
  *block = config.block;
  *smem = config.smem;
  *(cudaStream_t*)st = config.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t) {
  const auto it = granted.find({device, (const void*)k});
  if (smem > 48 * 1024 && (it == granted.end() || it->second < smem)) return last = cudaErrorInvalidValue;
  launches.push_back(Launch{names()[(const void*)k], {g.x, g.y, g.z}, {b.x, b.y, b.z}, smem, device});
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int bytes) {
  granted[{device, f}] = (size_t)bytes;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  ++occupancy_queries;
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = (void*)((size_t)1 << 40); return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t) { *p = (void*)((size_t)1 << 40); return cudaSuccess; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)1; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* g, cudaGraph_t, unsigned long long) { *g = (cudaGraphExec_t)1; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

}  // extern "C"
