// cudaLaunchCooperativeKernel that refuses every call after the first `allowed`
// ones, as the runtime does where the grid does not fit; linked into a copy of
// the library with --wrap.
#include <cuda_runtime.h>

extern "C" {
int refused_allowed = 0;
int refused_calls = 0;

cudaError_t __real_cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t);
cudaError_t __wrap_cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void** a, size_t s, cudaStream_t st) {
  if (refused_allowed > 0) {
    --refused_allowed;
    return __real_cudaLaunchCooperativeKernel(f, g, b, a, s, st);
  }
  ++refused_calls;
  return cudaErrorCooperativeLaunchTooLarge;
}
}
