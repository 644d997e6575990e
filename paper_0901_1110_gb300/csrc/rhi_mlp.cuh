// Declarations of the learned-guess MLP kernels (rhi_mlp.cu).
#pragma once

#include <cuda_bf16.h>

#include <cstring>

#include "rhi_internal.cuh"

namespace rhi {

constexpr int MLP_IN = RHI_MLP_IN, MLP_HID = RHI_MLP_HID, MLP_OUT = RHI_MLP_OUT;
// Row strides (bf16) of the packed weights: 8 words more than a multiple of 32 (or 8), so that the
// eight-byte fragment loads of a half-warp (4 rows x 4 pieces) fall into different banks
constexpr int RS1 = 16;
constexpr int RS2 = 80;
// place of input k in a packed row: within each 16, a thread's four values of an m16n8k16 B
// fragment (k = 2t, 2t + 1, 2t + 8, 2t + 9) side by side
__host__ __device__ constexpr int packed_k(int k) {
    return (k & ~15) + 4 * ((k & 7) >> 1) + 2 * ((k >> 3) & 1) + (k & 1);
}

// inference weights: BF16 rows in fragment order, padded for conflict-free loads, FP32 biases and
// the input normalisation (mean, 1 / scale)
struct MlpPacked {
    __nv_bfloat16 W1[MLP_HID * RS1];
    __nv_bfloat16 W2[MLP_HID * RS2];
    __nv_bfloat16 W3[MLP_HID * RS2];
    __nv_bfloat16 W4[8 * RS2];
    float b1[MLP_HID], b2[MLP_HID], b3[MLP_HID], b4[8];
    float mean[MLP_IN], iscale[MLP_IN];
};

struct MlpArgs {
    long long N;
    int ns;
    double y_he, iu_E, iu_e, iu_n, dt, gam_per_E;
    const double* E;
    const double* e;
    const double* n;
    const double* nH;
    const double* src;
    // the state before the last accepted step (null: none yet) and log10(dt / dt^{n-1})
    const double* E_p;
    const double* e_p;
    const double* n_p;
    float ldt_ratio;
    float gate;
    float ood;                                // |normalised feature| above this keeps U^n
    int isothermal;                           // guess keeps e_c = 0
    double* U0;                               // guess (e_c | n | E), MODE 1
};

cudaError_t launch_mlp_pack(const float* w, MlpPacked* out, cudaStream_t st);
cudaError_t launch_mlp_features(const MlpArgs& A, float* X, cudaStream_t st);
cudaError_t launch_mlp_targets(const MlpArgs& A, const double* E0, const double* e0,
                               const double* n0, float* Y, cudaStream_t st);
cudaError_t launch_mlp_infer(const MlpArgs& A, const MlpPacked* pk, const float* X, float* Y,
                             long long n_rows, int guess, cudaStream_t st);
// Forward and backward of m samples: the gradients (mlp_ntrain() floats) of mlp_train_blocks(m)
// blocks into gpart, their squared errors into partials; then their sum (grad) or the Adam update
int mlp_train_blocks(long long m);
int mlp_ntrain();
cudaError_t launch_mlp_train(const float* w, const float* X, const float* Y, long long m, float* gpart,
                             double* partials, cudaStream_t st);
cudaError_t launch_mlp_grad(const float* gpart, int nb, float* grad, cudaStream_t st);
cudaError_t launch_mlp_adam(const float* gpart, int nb, float* w, float* m1, float* m2, float lr,
                            float b1t, float b2t, cudaStream_t st);

}  // namespace rhi
