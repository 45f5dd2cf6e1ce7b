// A simulated camera on a caller's stream: lets its dependents launch at once, waits some
// microseconds (by the global timer, and at most `polls` readings of it), then copies a frame.
#include <cstdint>
#include <cuda_runtime.h>

__global__ void producer_kernel(uint16_t* dst, const uint16_t* src, long long n, unsigned long long wait_ns, unsigned polls) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (unsigned k = 0; k < polls; ++k) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 >= wait_ns) break;
    }
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = src[i];
}

extern "C" int produce(uint16_t* dst, const uint16_t* src, long long n, unsigned long long wait_ns, void* stream) {
    producer_kernel<<<4, 256, 0, static_cast<cudaStream_t>(stream)>>>(dst, src, n, wait_ns, 100000u);
    return static_cast<int>(cudaPeekAtLastError());
}
