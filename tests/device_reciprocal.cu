// Test library: the reciprocals and the sign test of the kernels on arrays in device memory.
#include "hb_cells.cuh"

namespace {

__global__ void evaluate(const double* x, int n, double* normal, double* any, unsigned char* positive)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    normal[k] = hb::rcp64_normal(x[k]);
    any[k] = hb::rcp64(x[k]);
    positive[k] = hb::pos64(x[k]);
}

}  // namespace

extern "C" int device_reciprocal(const double* x, int n, double* normal, double* any, unsigned char* positive)
{
    evaluate<<<(n + 255) / 256, 256>>>(x, n, normal, any, positive);
    return (int)cudaDeviceSynchronize();
}
