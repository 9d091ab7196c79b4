// A kernel that lets its successor start at once (programmatic dependent launch) and then stays for `ms` milliseconds:
// what a caller's own kernel may do in front of a call of the library.  It ends by the clock, or after a bounded number
// of sleeps.
#include <cuda_runtime.h>

__global__ void early_trigger_kernel(unsigned long long ns, int max_sleeps) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (int i = 0; i < max_sleeps; ++i) {
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > ns) break;
    __nanosleep(100000);
  }
}

extern "C" int early_trigger(int ms, void* stream) {
  if (ms < 1 || ms > 5000) return -1;
  early_trigger_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(1000000ull * (unsigned long long)ms, 100 * ms);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
