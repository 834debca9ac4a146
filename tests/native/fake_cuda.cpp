// A stand-in for the CUDA runtime with several devices, for host code that
// launches kernels: kernels do not run; a launch fails, as on a GPU, when it asks
// for more dynamic shared memory than its kernel may use on the current device, and
// occupancy belongs to the device too.
#include <cuda_runtime_api.h>

#include <map>
#include <utility>

int fake_device = 0;

namespace {
constexpr size_t kDefaultShared = 48 * 1024, kMostShared = 227 * 1024;
cudaError_t error = cudaSuccess;
dim3 config_grid, config_block;
size_t config_shared;
cudaStream_t config_stream;
std::map<std::pair<int, const void*>, size_t> opted_in;
size_t allowed(const void* f) {
  const auto it = opted_in.find({fake_device, f});
  return it == opted_in.end() ? kDefaultShared : it->second;
}
}  // namespace

extern "C" {
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, struct CUstream_st* stream) {
  config_grid = grid;
  config_block = block;
  config_shared = shared;
  config_stream = stream;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shared, void* stream) {
  *grid = config_grid;
  *block = config_block;
  *shared = config_shared;
  *(cudaStream_t*)stream = config_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* kernel, const void* f) {
  *kernel = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3 grid, dim3 block, void**, size_t shared, cudaStream_t) {
  const bool ok = grid.x > 0 && block.x > 0 && block.x <= 1024 && shared <= allowed((const void*)kernel);
  if (!ok) error = cudaErrorInvalidValue;
  return ok ? cudaSuccess : cudaErrorInvalidValue;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute attr, int value) {
  if (attr != cudaFuncAttributeMaxDynamicSharedMemorySize || (size_t)value > kMostShared) return cudaErrorInvalidValue;
  opted_in[{fake_device, f}] = (size_t)value;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* blocks, const void* f, int, size_t shared,
                                                                   unsigned) {
  if (shared > allowed(f)) return cudaErrorInvalidValue;
  *blocks = 2;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* device) {
  *device = fake_device;
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = error;
  error = cudaSuccess;
  return e;
}
}
