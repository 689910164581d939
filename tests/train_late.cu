// The reduction with Adam of the training step on gradient partials given by
// the test (test_gpu_train_late.py): some marked late, as the training kernel
// does when its bounded wait for the tensor cores has run out.
#include "lbt_mlp_train.cu"

extern "C" int t_reduce(const float* partial, const double* loss_part, const int* late, int nparts, int K, float* grad,
                        double* loss, float* master, float* m, float* v, unsigned char* params)
{
    const lbt::MlpLayout L = lbt::mlp_layout(K);
    const lbt::AdamArgs A{master, m, v, params, 1e-3f, 0.9f, 0.999f, 1e-8f, 0.1f, 0.001f};
    lbt::k_mlp_reduce<true><<<(unsigned)((L.nmaster + 31) / 32), 32 * lbt::kRdSlices>>>(partial, loss_part, late, nparts, L,
                                                                                      grad, nullptr, loss, nullptr, A);
    return cudaDeviceSynchronize();
}
