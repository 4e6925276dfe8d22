// Test library: the reciprocals, the sign test and the temperature power of the kernels on arrays in device memory.
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

// here: x^-w as the kernels form it; power: pow of the rounded quotient
__global__ void evaluate_power(const double* x, const double* w, int n, double* here, double* power)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    here[k] = hb::temperature_power(x[k], hb::rcp64(x[k]), w[k]);
    power[k] = pow(1.0 / x[k], w[k]);
}

}  // namespace

extern "C" int device_power(const double* x, const double* w, int n, double* here, double* power)
{
    evaluate_power<<<(n + 255) / 256, 256>>>(x, w, n, here, power);
    return (int)cudaDeviceSynchronize();
}

extern "C" int device_reciprocal(const double* x, int n, double* normal, double* any, unsigned char* positive)
{
    evaluate<<<(n + 255) / 256, 256>>>(x, n, normal, any, positive);
    return (int)cudaDeviceSynchronize();
}
