// A caller's kernel that lets the next kernel of its stream in at once
// (griddepcontrol.launch_dependents), runs on for `ns` nanoseconds and then
// writes dst: whatever was let in early has to wait for it. Compiled by
// tests/test_gpu_early_release.py; it ends by itself.
#include <cstdint>
#include <cuda_runtime.h>

__global__ void early_release_kernel(const int *src, int *dst, long long n, unsigned long long ns) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  do {
    __nanosleep(2000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  } while (t - t0 < ns);
  for (long long i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

extern "C" int early_release(const int *src, int *dst, long long n, unsigned long long ns, cudaStream_t stream) {
  early_release_kernel<<<1, 256, 0, stream>>>(src, dst, n, ns);
  return static_cast<int>(cudaGetLastError());
}
