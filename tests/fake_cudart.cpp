// A CUDA runtime without a GPU, preloaded by tests of the host code: "device"
// memory is host memory, copies are memcpy, kernels are recorded and not run.
// Only the calls that libqt.so makes are here.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Config { dim3 grid, block; size_t smem; void* stream; };
thread_local Config pushed;
std::map<const void*, std::string> kernel_names;
std::string launches;                       // "name grid block smem" lines
std::string fail_kernel, set_kernel;
int* flag = nullptr;                        // the last int cleared on the device
cudaError_t last_error = cudaSuccess;
size_t fail_bytes = 0;                      // the next fail_count allocations of that many bytes or more fail
int fail_count = 0;

cudaError_t launch(const void* kernel, dim3 grid, dim3 block, size_t smem) {
  const std::string& name = kernel_names[kernel];
  launches += name + " " + std::to_string(grid.x) + " " + std::to_string(block.x) + " " + std::to_string(smem) + "\n";
  if (!fail_kernel.empty() && name.find(fail_kernel) != std::string::npos) return last_error = cudaErrorLaunchOutOfResources;
  if (flag && !set_kernel.empty() && name.find(set_kernel) != std::string::npos) *flag = 1;
  return cudaSuccess;
}

cudaError_t allocate(void** p, size_t n) {
  if (fail_count > 0 && n >= fail_bytes) {
    --fail_count;
    return last_error = cudaErrorMemoryAllocation;
  }
  *p = std::aligned_alloc(256, (n + 511) & ~static_cast<size_t>(255));
  if (*p && n < (size_t{1} << 24)) std::memset(*p, 0, n);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}

char token[8];
template <typename T> cudaError_t handle(T* h) { *h = reinterpret_cast<T>(token); return cudaSuccess; }

}  // namespace

extern "C" {

// control, for the test
const char* fake_launches() { return launches.c_str(); }
void fake_clear() { launches.clear(); }
void fake_fail(const char* kernel) { fail_kernel = kernel; }
void fake_fail_alloc(size_t bytes, int count) { fail_bytes = bytes; fail_count = count; }
// launches of `kernel` set the error flag, the last int that was cleared
void fake_set(const char* kernel) { set_kernel = kernel; }

void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(token); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  kernel_names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
  pushed = {grid, block, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = pushed.grid;
  *block = pushed.block;
  *smem = pushed.smem;
  *static_cast<void**>(stream) = pushed.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
  *k = static_cast<cudaKernel_t>(const_cast<void*>(host));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t) {
  return launch(k, grid, block, smem);
}
cudaError_t cudaLaunchKernel(const void* k, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t) {
  return launch(k, grid, block, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* k, void**) {
  return launch(k, c->gridDim, c->blockDim, c->dynamicSmemBytes);
}

cudaError_t cudaGetLastError() { const cudaError_t e = last_error; last_error = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { *a = {}; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { static char sym[1 << 20]; *p = sym; return cudaSuccess; }

cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return allocate(p, n); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return allocate(p, n); }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  if (n == sizeof(int)) flag = static_cast<int*>(d);
  std::memset(d, v, n);
  return cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return handle(g); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { return handle(e); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }

}  // extern "C"
