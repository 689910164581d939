// Element-wise wrappers of device helpers of the library, for
// test_gpu_device_math.py: one thread per element, device pointers in and out.
#include "lbt_synth.cu"

namespace {

template <class T>
__global__ void k_inverse(const T* x, T* y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = lbt::fast_inverse(x[i]);
}
template <class T>
__global__ void k_ratio(const T* j, const T* rho, T* y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = lbt::ratio(j[i], rho[i], lbt::fast_inverse(rho[i]));
}
__global__ void k_sqrt(const double* x, double* y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = lbt::quick_sqrt(x[i]);
}
__global__ void k_widen(const float* x, double* y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = lbt::widen(x[i]);
}

}  // namespace

extern "C" {

int t_inverse_f64(const double* x, double* y, int n)
{
    k_inverse<double><<<(n + 255) / 256, 256>>>(x, y, n);
    return cudaDeviceSynchronize();
}
int t_inverse_f32(const float* x, float* y, int n)
{
    k_inverse<float><<<(n + 255) / 256, 256>>>(x, y, n);
    return cudaDeviceSynchronize();
}
int t_ratio_f64(const double* j, const double* rho, double* y, int n)
{
    k_ratio<double><<<(n + 255) / 256, 256>>>(j, rho, y, n);
    return cudaDeviceSynchronize();
}
int t_ratio_f32(const float* j, const float* rho, float* y, int n)
{
    k_ratio<float><<<(n + 255) / 256, 256>>>(j, rho, y, n);
    return cudaDeviceSynchronize();
}
int t_sqrt(const double* x, double* y, int n)
{
    k_sqrt<<<(n + 255) / 256, 256>>>(x, y, n);
    return cudaDeviceSynchronize();
}
int t_widen(const float* x, double* y, int n)
{
    k_widen<<<(n + 255) / 256, 256>>>(x, y, n);
    return cudaDeviceSynchronize();
}

}  // extern "C"
