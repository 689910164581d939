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

// pairs a, b (n x 3): listed within the radius rl of a?
__global__ void k_listed(const double* a, const double* b, const double* rl2, float* y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 x = lbt::list_copy(a[3 * i], a[3 * i + 1], a[3 * i + 2]);
    const float4 q = lbt::list_copy(b[3 * i], b[3 * i + 1], b[3 * i + 2]);
    y[i] = lbt::list_near(x, q, lbt::list_reach2(sqrtf((float)rl2[i]), x.w)) ? 1.f : 0.f;
}

}  // namespace

extern "C" {

int t_listed(const double* a, const double* b, const double* rl2, float* y, int n)
{
    k_listed<<<(n + 255) / 256, 256>>>(a, b, rl2, y, n);
    return cudaDeviceSynchronize();
}

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
