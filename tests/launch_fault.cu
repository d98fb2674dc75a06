// A stand-in for the runtime's kernel launches that refuses one of them: linked
// with the library's objects (--wrap on the three symbols below), it counts the
// launches and answers the n-th with an error without making it.  Nothing fails
// on the GPU: the error is made on the host.
#include <cuda_runtime.h>

extern "C" {

cudaError_t __real_cudaLaunchKernelExC(const cudaLaunchConfig_t *config, const void *func, void **args);
cudaError_t __real___cudaLaunchKernel(cudaKernel_t kernel, dim3 grid, dim3 block, void **args, size_t shared,
                                      cudaStream_t stream);
cudaError_t __real_cudaGetLastError(void);

static int left = 0;  // launches up to and with the one that is refused; 0: none
static cudaError_t pending = cudaSuccess;

void launch_fault_in(int n) { left = n; }
int launch_fault_left(void) { return left; }

static bool refused(void) { return left > 0 && --left == 0; }

cudaError_t __wrap_cudaLaunchKernelExC(const cudaLaunchConfig_t *config, const void *func, void **args)
{
    return refused() ? cudaErrorLaunchOutOfResources : __real_cudaLaunchKernelExC(config, func, args);
}

cudaError_t __wrap___cudaLaunchKernel(cudaKernel_t kernel, dim3 grid, dim3 block, void **args, size_t shared,
                                      cudaStream_t stream)
{
    if (!refused()) return __real___cudaLaunchKernel(kernel, grid, block, args, shared, stream);
    return pending = cudaErrorLaunchOutOfResources;  // also what cudaGetLastError answers next
}

cudaError_t __wrap_cudaGetLastError(void)
{
    const cudaError_t e = pending;
    pending = cudaSuccess;
    return e != cudaSuccess ? e : __real_cudaGetLastError();
}

}  // extern "C"
