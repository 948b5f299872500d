// Kernels for test_gpu_bounded_waits.py.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tc05.cuh"

using namespace radar::tc05;

__device__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// A wait of each kind for an arrival that never comes, one thread each: ns[i] it took, seen[i] its outcome; then, in ns[2] and
// seen[2], 1000 waits behind the first one that ran out.
__global__ void waits_that_run_out_kernel(unsigned long long* ns, int* seen) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
    }
    __syncthreads();
    if ((threadIdx.x & 31) != 0) return;
    const int i = threadIdx.x >> 5;
    const unsigned long long t0 = now_ns();
    bool ok = i == 0 ? mbar_wait_while(true, &bar, 0) : mbar_wait_lazy(true, &bar, 0);
    const unsigned long long t1 = now_ns();
    ns[i] = t1 - t0;
    seen[i] = ok;
    if (i == 0) {
        for (int n = 0; n < 1000; ++n) ok = mbar_wait_while(ok, &bar, 0);
        ns[2] = now_ns() - t1;
        seen[2] = ok;
    }
}
extern "C" int waits_that_run_out(unsigned long long* ns, int* seen) {
    waits_that_run_out_kernel<<<1, 64>>>(ns, seen);
    return (int)cudaDeviceSynchronize();
}

// A predecessor that lets its dependents start at once and then takes `ns` nanoseconds (bounded by its naps as well).
__global__ void slow_predecessor_kernel(unsigned long long ns, int naps) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned long long end = now_ns() + ns;
    for (int i = 0; i < naps && now_ns() < end; ++i) __nanosleep(500000);
}
extern "C" int launch_slow_predecessor(void* stream, unsigned long long ns) {
    slow_predecessor_kernel<<<1, 1, 0, reinterpret_cast<cudaStream_t>(stream)>>>(ns, (int)(ns / 100000));
    return (int)cudaGetLastError();
}
