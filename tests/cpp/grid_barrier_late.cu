// The grid barrier when a CTA is late: three CTAs give up after 20 ms, the last one
// arrives at 100 ms. Every CTA has to return false, the late one at once and not after
// a limit of its own, and status word 1 has to be set; in time, all return true.
// Prints "ok".
#include <cstdio>
#include <cuda_runtime.h>

#include "common.cuh"

__device__ uint64_t now() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void barrier_kernel(uint64_t *bar, int *status, uint64_t late_ns, int *left, uint64_t *waited) {
    uint64_t target = 0;
    for (int k = 0; k < 3; ++k) {
        if (k == 1 && blockIdx.x == gridDim.x - 1) {   // bounded: ends by the clock
            const uint64_t t0 = now();
            while (now() - t0 < late_ns) {}
        }
        const uint64_t t0 = now();
        const bool ok = lne::grid_barrier(bar, target, status, 20000000ull);
        if (threadIdx.x == 0) {
            left[blockIdx.x] = ok ? k + 1 : -(k + 1);
            waited[blockIdx.x] = now() - t0;
        }
        if (!ok) return;
    }
}

int main() {
    const int ctas = 4;
    uint64_t *bar, *waited;
    int *status, *left;
    cudaMalloc(&bar, 8);
    cudaMalloc(&waited, 8 * ctas);
    cudaMalloc(&status, 16);
    cudaMalloc(&left, 4 * ctas);
    for (int late = 0; late < 2; ++late) {
        cudaMemset(bar, 0, 8);
        cudaMemset(status, 0, 16);
        uint64_t ns = late ? 100000000ull : 0ull;
        void *args[] = {&bar, &status, &ns, &left, &waited};
        cudaLaunchCooperativeKernel((const void *)barrier_kernel, dim3(ctas), dim3(64), args, 0, nullptr);
        int h[ctas], hs[4];
        uint64_t hw[ctas];
        cudaMemcpy(h, left, sizeof(h), cudaMemcpyDeviceToHost);
        cudaMemcpy(hs, status, sizeof(hs), cudaMemcpyDeviceToHost);
        cudaMemcpy(hw, waited, sizeof(hw), cudaMemcpyDeviceToHost);
        const cudaError_t e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return std::printf("%s\n", cudaGetErrorString(e)), 1;
        for (int b = 0; b < ctas; ++b)
            if (h[b] != (late ? -2 : 3)) return std::printf("late %d: CTA %d left with %d\n", late, b, h[b]), 1;
        if (hs[1] != late) return std::printf("late %d: status %d\n", late, hs[1]), 1;
        if (late && hw[ctas - 1] > 10000000ull) return std::printf("the late CTA waited\n"), 1;
    }
    std::printf("ok\n");
    return 0;
}
