// Compares reciprocal() with the IEEE reciprocal over every float it meets.
#include <cuda_runtime.h>
#include <stdint.h>

#include "snap_device.cuh"

namespace {

// mismatches[0]: [1, 2^126), bit for bit; [1]: [2^126, infinity], the
// coefficients of the forces and of U^r; [2]: NaN stays NaN.
__global__ void compare(unsigned long long *mismatches) {
    const uint32_t one = 0x3F800000u, big = 0x7E800000u, inf = 0x7F800000u, end = 0x7FFFFFFFu;
    unsigned long long bad[3] = {0, 0, 0};
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = one + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= end; b += stride) {
        const float d = __uint_as_float((uint32_t)b);
        const float q = snap::reciprocal_of<true>(d), w = snap::reciprocal_of<false>(d);
        if (b < big) {
            bad[0] += __float_as_uint(q) != __float_as_uint(w);
        } else if (b <= inf) {
            bad[1] += fmaf(snap::kBeta, q, 1.0f) != fmaf(snap::kBeta, w, 1.0f) || q * q != w * w;
        } else {
            bad[2] += q == q;
        }
    }
    for (int m = 0; m < 3; ++m)
        if (bad[m]) atomicAdd(mismatches + m, bad[m]);
}

}  // namespace

extern "C" int compare_reciprocals(unsigned long long *out) {
    unsigned long long *d = nullptr;
    cudaError_t err = cudaMalloc(&d, 3 * sizeof(*d));
    if (err == cudaSuccess) err = cudaMemset(d, 0, 3 * sizeof(*d));
    if (err == cudaSuccess) {
        compare<<<1216, 256>>>(d);
        err = cudaGetLastError();
    }
    if (err == cudaSuccess) err = cudaMemcpy(out, d, 3 * sizeof(*d), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)err;
}
