// recip_exact (csrc/d3q19.cuh), the reciprocal of the density in node pairs,
// against the division of the one-node kernels: every FP32 bit pattern, in
// either lane beside an unrelated value. Built and called by
// test_gpu_recip_exact.py.
#include "d3q19.cuh"

namespace {

// counts[lane]: patterns whose result is not the quotient's bits (NaN counts as any NaN).
__global__ void k_compare(unsigned long long *counts) {
    unsigned long long bad[2] = {0, 0};
    const unsigned step = gridDim.x * blockDim.x;  // a power of two: divides 2^32
    unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    for (unsigned long long k = 0; k < (1ull << 32) / step; ++k, i += step) {
        const float x = __uint_as_float(i), other = __uint_as_float(~i * 2654435761u);
        const float want = 1.0f / x;
        const float got[2] = {clbm::recip_exact(clbm::f2{make_float2(x, other)}).v.x,
                              clbm::recip_exact(clbm::f2{make_float2(other, x)}).v.y};
        for (int lane = 0; lane < 2; ++lane) {
            const bool same = want != want ? got[lane] != got[lane]
                                           : __float_as_uint(got[lane]) == __float_as_uint(want);
            bad[lane] += !same;
        }
    }
    for (int lane = 0; lane < 2; ++lane)
        if (bad[lane]) atomicAdd(counts + lane, bad[lane]);
}

}  // namespace

extern "C" int recip_exact_mismatches(unsigned long long *out) {
    unsigned long long *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 16);
    if (e == cudaSuccess) e = cudaMemset(d, 0, 16);
    if (e == cudaSuccess) {
        k_compare<<<1024, 256>>>(d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d, 16, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
