// Holds 'bytes' of shared memory on every SM for about 'ms' milliseconds of the
// global timer (checked at most 2^24 times).
#include <cuda_runtime.h>

__global__ void k_hold(unsigned long long ns) {
    extern __shared__ int s[];
    if (threadIdx.x == 0) s[0] = 1;
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (int i = 0; i < (1 << 24); i++) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 >= ns) break;
        __nanosleep(1000);
    }
}

extern "C" int hold_shared(int bytes, int ms, void *stream) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaFuncSetAttribute(k_hold, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    // the SMs set up for all of their shared memory, not for what this kernel takes
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_hold, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return (int)e;
    k_hold<<<sms, 32, bytes, (cudaStream_t)stream>>>(1000000ull * ms);
    return (int)cudaGetLastError();
}
