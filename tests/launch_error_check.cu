// launch_error_check.cu -- launch_pass (passes.cuh) over a launch call that
// refuses, on a stand-in for the runtime's launch and last-error calls (without
// a device the real ones fail before they look at the launch).  Built and run
// by tests/test_launch_error_host.py.  Prints the status that launch_pass
// returns and the error that it leaves to the caller's next check.
#include <cuda_runtime.h>
#include <stdio.h>

static cudaError_t g_last = cudaSuccess;
template <typename... A>
static cudaError_t refused_launch(const cudaLaunchConfig_t *, A...)
{
    return g_last = cudaErrorInvalidConfiguration;
}
static cudaError_t take_last_error()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
#define cudaLaunchKernelEx refused_launch
#define cudaGetLastError take_last_error
#include "passes.cuh"

namespace isofft {
void count_launch() {}
}  // namespace isofft

static __global__ void k_nothing(int *) {}

int main()
{
    const cudaError_t e = isofft::launch_pass(k_nothing, dim3(1), 4096, 0, (cudaStream_t)0, (int *)nullptr);
    printf("%d %d\n", (int)e, (int)g_last);
    return 0;
}
