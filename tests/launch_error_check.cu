// launch_error_check.cu -- a launch that the runtime refuses (more threads in a
// block than any device takes; without a device, any launch) through
// launch_pass (passes.cuh).  Built and run by tests/test_launch_error_host.py.
// Prints the status that launch_pass returns and the error that it leaves to
// the caller's next check.
#include <stdio.h>

#include "passes.cuh"

namespace isofft {
void count_launch() {}
}  // namespace isofft

static __global__ void k_nothing(int *) {}

int main()
{
    cudaGetLastError();
    const cudaError_t e = isofft::launch_pass(k_nothing, dim3(1), 4096, 0, (cudaStream_t)0, (int *)nullptr);
    const cudaError_t left = cudaPeekAtLastError();
    printf("%d %d\n", (int)e, (int)left);
    return 0;
}
