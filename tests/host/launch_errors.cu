// A refused launch is reported by the call that made it and leaves no error
// behind in the runtime for the next call to find. launch_errors.cpp stands in
// for the runtime, so no driver or device is needed and nothing runs.
#include <cstdio>

#include "launch.h"

extern cudaError_t last_error;
static void kernel(float*) {}

int main() {
  float* p = nullptr;
  if (fst::launch_pdl(kernel, dim3(1), dim3(32), 0, nullptr, p) != cudaSuccess) return std::puts("refused"), 1;
  if (fst::launch_pdl(kernel, dim3(1), dim3(4096), 0, nullptr, p) != cudaErrorInvalidConfiguration)
    return std::puts("not refused"), 1;
  if (last_error != cudaSuccess) return std::puts("an error was left behind"), 1;
  return std::puts("ok"), 0;
}
