// The first error that a call's kernel launches left. The runtime's own record does not last until the call ends: a
// later successful cudaFuncSetAttribute clears it, and results of launches that never ran were returned as good.
#pragma once
#include <cuda_runtime.h>

namespace imf {

struct LaunchErrors {
    cudaError_t first = cudaSuccess;

    void note(cudaError_t e)
    {
        if (first == cudaSuccess) first = e;
    }
    // what the call reports: its first launch error, else `now`; clears the record for the next call
    cudaError_t take(cudaError_t now)
    {
        const cudaError_t e = first != cudaSuccess ? first : now;
        first = cudaSuccess;
        return e;
    }
};

} // namespace imf
