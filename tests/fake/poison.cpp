// Linked into a copy of the library with --wrap=cudaMalloc: device memory comes filled with 0x7f bytes, large numbers as
// any integer type, where the driver may hand out cleared memory.
#include <cuda_runtime_api.h>

extern "C" {

cudaError_t __real_cudaMalloc(void **p, size_t n);

cudaError_t __wrap_cudaMalloc(void **p, size_t n)
{
    const cudaError_t e = __real_cudaMalloc(p, n);
    return e == cudaSuccess ? cudaMemset(*p, 0x7f, n) : e;
}

}
