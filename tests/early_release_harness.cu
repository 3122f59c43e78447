// A kernel of "another library" for the stream-order tests: it lets its
// successor on the stream start at once, waits about `microseconds`, and only
// then copies src to dst. The wait is bounded by its step count.
#include <cuda_runtime.h>

__global__ void late_copy(const float* src, float* dst, int n, int microseconds) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = 0; i < microseconds; ++i) __nanosleep(1000);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i];
}

extern "C" int late_copy_launch(const float* src, float* dst, int n, int microseconds, void* stream) {
  late_copy<<<4, 256, 0, static_cast<cudaStream_t>(stream)>>>(src, dst, n, microseconds);
  return static_cast<int>(cudaGetLastError());
}
