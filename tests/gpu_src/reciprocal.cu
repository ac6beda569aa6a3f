// Test-only: the kernels' reciprocal on [1, 2] against the division, for every binary32
// value there.  Built by the test that uses it.
#include <cuda_runtime.h>

#include "laps_device.cuh"

__global__ void compare_kernel(unsigned* bad) {
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > (1u << 23)) return;
    const float x = __uint_as_float(0x3f800000u + i);
    if (__float_as_uint(laps::rcp_1_2(x)) != __float_as_uint(1.0f / x)) atomicAdd(bad, 1u);
}

// *bad (device, zeroed by the caller): values of [1, 2] on which the two differ
extern "C" int compare_reciprocal(unsigned* bad, void* stream) {
    compare_kernel<<<(1 << 23) / 256 + 1, 256, 0, (cudaStream_t)stream>>>(bad);
    return (int)cudaGetLastError();
}
