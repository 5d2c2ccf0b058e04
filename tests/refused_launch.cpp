// A device that takes no cooperative launch, for test_gpu_refused_launch.py: the
// solvers built against this function in the place of cudaLaunchCooperativeKernel.
#include <cuda_runtime.h>

extern "C" {
int helm_refused_launches = 0;
cudaError_t helm_refused_launch(const void*, dim3, dim3, void**, size_t, cudaStream_t) {
  ++helm_refused_launches;
  return cudaErrorCooperativeLaunchTooLarge;
}
}
