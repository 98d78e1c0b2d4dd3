// Shared declarations of the warm-start network's kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace dm {

// Partial gradients of layer l's share z: its weights (256 x 64, 256 x 256,
// 256 x 256 [out][in]; the output layer's transposed, 256 x 64 [in][out]),
// then the hidden layers' 256 bias sums; the shares of layer 0 (s_small),
// 1, 2 (s_big each) and 3 (s_small) one after another.
__host__ __device__ inline size_t mlp_part_size(int l) {
  return (size_t)256 * (l == 0 || l == 3 ? 64 : 256) + (l < 3 ? 256 : 0);
}
__host__ __device__ inline size_t mlp_part_offset(int l, int s_small, int s_big) {
  size_t o = 0;
  for (int k = 0; k < l; ++k) o += mlp_part_size(k) * (size_t)(k == 0 || k == 3 ? s_small : s_big);
  return o;
}

struct MlpTrainShape {
  int ctas, s_small, s_big;
};
MlpTrainShape mlp_train_shape(int M);
cudaError_t launch_mlp_fused(int M, const void *X, const void *const W[4], const float *const b[4],
                             float *Y, int *err, cudaStream_t st);
cudaError_t launch_mlp_train(int M, const void *X, const float *target, int n_valid, const void *const W[4],
                             const void *const Wt[4], const float *const b[4], void *const act[3],
                             void *const dz[3], void *dy, double *loss, float *part, float *gb4, int *err,
                             cudaStream_t st);
cudaError_t launch_gemm_bf16(int M, int N, int K, const void *A, const void *B, const float *bias,
                             void *C, int relu, int out_f32, int *err, cudaStream_t st);

}  // namespace dm
