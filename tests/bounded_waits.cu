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

// Waits for an arrival that never comes, one thread each: ns[i] it took, seen[i] its outcome.  0: a wait that polls, 1: one that
// naps, 2: 1000 waits behind the first, 3: a block's wait for what it has in flight.
__global__ void waits_that_run_out_kernel(unsigned long long* ns, int* seen) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_barrier_init();
    }
    __syncthreads();
    if ((threadIdx.x & 31) != 0) return;
    auto timed = [&](int i, auto wait) {
        const unsigned long long t0 = now_ns();
        seen[i] = wait();
        ns[i] = now_ns() - t0;
    };
    switch (threadIdx.x >> 5) {
        case 0:
            timed(0, [&] { return mbar_wait_while(true, &bar, 0); });
            timed(2, [&] {
                bool ok = false;
                for (int n = 0; n < 1000; ++n) ok |= mbar_wait_while(false, &bar, 0);
                return ok;
            });
            break;
        case 1: timed(1, [&] { return mbar_wait_lazy(true, &bar, 0); }); break;
        case 2: timed(3, [&] { return mbar_drain(&bar, 0); }); break;
    }
}
extern "C" int waits_that_run_out(unsigned long long* ns, int* seen) {
    waits_that_run_out_kernel<<<1, 96>>>(ns, seen);
    return (int)cudaDeviceSynchronize();
}
extern "C" unsigned ring_parity(unsigned slot, unsigned next, unsigned par) { return last_armed_parity(slot, next, par); }

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
