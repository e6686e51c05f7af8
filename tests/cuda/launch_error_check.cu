// launch_dependent over stand-ins for the runtime's launch and error calls: a failed launch's error is
// returned and none is left pending.
#include <cuda_runtime.h>

#include <cstdio>

static cudaError_t pending = cudaSuccess, outcome = cudaSuccess;

template <typename C, typename K>
static cudaError_t launch_stand_in(C, K)
{
    return pending = outcome;
}

static cudaError_t last_error_stand_in()
{
    const cudaError_t e = pending;
    pending = cudaSuccess;
    return e;
}

#define cudaLaunchKernelEx launch_stand_in
#define cudaGetLastError last_error_stand_in
#include "ga_internal.h"

__global__ void nothing() {}

int main()
{
    for (cudaError_t e : {cudaSuccess, cudaErrorInvalidConfiguration, cudaErrorStreamCaptureInvalidated}) {
        outcome = e;
        const cudaError_t got = ga::launch_dependent(nothing, 1, 32, nullptr);
        std::printf("%d %d\n", got == e, static_cast<int>(pending));
    }
    return 0;
}
