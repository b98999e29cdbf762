// Warm-start MLP: launch descriptions shared by mlp.cu and mlp_api.cpp.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace treeot {

enum MlpMode : int32_t {
  MLP_PLAIN = 0,
  MLP_GELU = 1,      // C = z, H = bf16(gelu(z))
  MLP_GELU_BWD = 2,  // C = product * gelu'(z), H = bf16(C)
};

// one product of a step (operand layout: see mlp.cu)
struct MlpGemm {
  const void *A, *B;  // BF16
  float* C;
  const float* bias;  // per column, or null
  const float* z;     // MLP_GELU_BWD: pre-activations, layout of C
  void* H;            // BF16 result, row stride ldh
  int32_t lda, ta, ldb, tb, ldc, ldh, M, N, K, mode, tiles_n, tiles;
};
// column sums out[n] = sum_m x[m * N + n]
struct MlpColsum {
  const float* x;
  float* out;
  int32_t M, N;
};
// independent work of one launch
struct MlpStep {
  MlpGemm gemm[2];
  MlpColsum sum;  // x = null: none
  int32_t ngemm;
};
// where the three weight tensors of the flat parameter vector keep their BF16 copies
struct MlpW16 {
  int64_t off[3], len[3];
  int32_t cols[3], ld[3];
  void* dst[3];
};

MlpGemm mlp_gemm(const void* A, int lda, int ta, const void* B, int ldb, int tb, float* C, int ldc, int M, int N, int K);
cudaError_t mlp_step(const MlpStep& st, cudaStream_t s);
cudaError_t mlp_input(const float* x, void* y, int64_t rows, int cols, int ld, int nlog, float floor_, float scale,
                      double* loss, cudaStream_t s);
cudaError_t mlp_to_bf16(const float* x, const MlpW16& w, int64_t n, cudaStream_t s);
cudaError_t mlp_mse(const float* y, const float* t, float* dy32, void* dy16, int rows, int cols, int ld, double* loss,
                    cudaStream_t s);
cudaError_t mlp_adam(float* w, const float* g, float* m1, float* m2, const MlpW16& w16, int64_t n, float lr, float b1,
                     float b2, float eps, float c1, float c2, cudaStream_t s);

}  // namespace treeot
