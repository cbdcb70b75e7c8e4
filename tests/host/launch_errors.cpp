// The part of the CUDA runtime that launch_errors.cu calls: a launch of more
// threads than a block takes is refused, and the error stays until it is read.
#include <driver_types.h>

cudaError_t last_error = cudaSuccess;
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void*, void**) {
  return last_error = cfg->blockDim.x > 1024 ? cudaErrorInvalidConfiguration : cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}
// what the compiler's start-up code calls: there is no device code to register
extern "C" void** __cudaRegisterFatBinary(void*) { return nullptr; }
extern "C" void __cudaRegisterFatBinaryEnd(void**) {}
extern "C" void __cudaUnregisterFatBinary(void**) {}
extern "C" char __cudaInitModule(void**) { return 0; }
