// Barrier over the blocks of a cooperative launch, and such a launch with as many blocks as are wanted and
// fit the device at once.
#pragma once
#include <algorithm>
#include <cuda_runtime.h>

namespace imf {

// Barrier over the grid: false once it, or another block's, gave up (five seconds). `bar`: two words, the
// arrivals and the error, zeroed before the launch. Data that other blocks wrote is read past L1 (__ldcg).
struct GridBarrier {
    unsigned *bar;
    unsigned target = 0;
    __device__ __forceinline__ static unsigned long long now_ns()
    {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        return t;
    }
    __device__ __forceinline__ bool wait()
    {
        __shared__ unsigned bad;
        target += gridDim.x;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(bar, 1u);
            unsigned v, b = 0;
            unsigned long long t0 = 0;
            for (unsigned n = 0;; ++n) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
                if ((int)(v - target) >= 0) break;
                if ((n & 255u) == 255u) {
                    if (!t0) t0 = now_ns();
                    if (now_ns() - t0 > 5000000000ull || *(volatile unsigned *)(bar + 1)) {
                        b = 1;
                        atomicExch(bar + 1, 1u);
                        break;
                    }
                }
            }
            __threadfence();
            bad = b;
        }
        __syncthreads();
        return bad == 0;
    }
};

// Calls launch(blocks) with `want` blocks, or half as many, and so on down to one, until they fit. What fits is not known
// beforehand: a stream may own only some of the device's SMs (a green context).
template <typename F> cudaError_t launch_fitting(long want, F &&launch)
{
    for (long n = std::max(1L, want);; n = (n + 1) / 2) {
        const cudaError_t e = launch(n);
        if (e != cudaErrorCooperativeLaunchTooLarge || n == 1) return e;
        cudaGetLastError();              // the refused launch left it behind
    }
}

// Launches kernel(args) cooperatively with `threads` threads a block and `want` blocks, or as many as the
// device holds at once, or fewer (launch_fitting; the kernel's loops stride over the grid).
template <typename A> cudaError_t launch_cooperative(void (*kernel)(A), const A &args, int threads, long want, cudaStream_t s)
{
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0);
    if (e != cudaSuccess) return e;
    const long most = (long)std::max(per, 1) * sms;
    void *p[1] = {const_cast<A *>(&args)};
    return launch_fitting(std::min(most, want), [&](long n) {
        return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(kernel), dim3((unsigned)n), dim3(threads), p, 0, s);
    });
}

} // namespace imf
