// Warm-start predictor: a 3-layer MLP (in -> hidden -> hidden -> out, GELU
// after the first two layers) with BF16 weights and activations feeding
// tensor-core MMAs (mma.sync m16n8k16, FP32 accumulation), FP32 master
// weights and Adam.  Forward, backward and the optimiser step are all kernels
// of this file; the host side lives in api.cpp (tree_ot_mlp_*).
//
// GEMM convention: C[M,N] = sum_k A(m,k) B(k,n), with A(m,k) read from a
// row-major array either as A[m*lda + k] (plain) or A[k*lda + m] (transposed),
// and the same for B(k,n) = B[k*ldb + n] or B[n*ldb + k].  Every BF16 operand is
// one of the network's own buffers, its rows padded with zeros to a multiple of
// eight, so all loads are 16-byte ones.
//
// At these sizes (256 x 512 x 1025 and the like, under 0.3 GFLOP) a product is
// bound by the latency of its K loop, not by a rate: 32 x 32 tiles give every
// product 128 to 528 CTAs, and a four-stage cp.async ring keeps three K steps of
// 64 in flight.  (64 x 64 tiles with scalar loads and no overlap: 54 us per
// product; now 4-5 us.)  Bias, GELU and its derivative are applied to the
// accumulators, and independent products and column sums of one step share a
// launch.  K is not split: the sums keep their order.
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>

#include "internal.h"
#include "mlp.h"

namespace treeot {
namespace {

constexpr int kT = 32;            // CTA tile (4 warps, each 16 x 16)
constexpr int kTK = 64;           // K step
constexpr int kStages = 4;
constexpr int kLdK = kTK + 8;     // row stride of a tile stored [m or n][k]: ldmatrix rows in distinct banks
constexpr int kLdM = kT + 8;      // row stride of a tile stored [k][m or n]
constexpr int kTileElems = kTK * kLdM > kT * kLdK ? kTK * kLdM : kT * kLdK;

// D = A (16x16, bf16, row) * B (16x8, bf16, col) + C, FP32
__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t* r, uint32_t addr) {
  if (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// 16 bytes from global to shared memory, zeros where !on
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0) : "memory");
}

// one K step of an operand tile: rows r0.. of the M (or N) index, columns k0.. of K.  trans: stored [k][r].
__device__ __forceinline__ void load_tile(uint32_t dst, const __nv_bfloat16* P, int ld, int trans, int r0, int k0, int R,
                                          int K) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int v = threadIdx.x + 128 * i;  // 256 vectors of 8
    if (trans) {
      const int kk = v >> 2, rr = (v & 3) * 8;
      const bool on = k0 + kk < K && r0 + rr < R;
      cp_async16(dst + 2 * (kk * kLdM + rr), on ? P + (int64_t)(k0 + kk) * ld + r0 + rr : P, on);
    } else {
      const int rr = v >> 3, kk = (v & 7) * 8;
      const bool on = r0 + rr < R && k0 + kk < K;
      cp_async16(dst + 2 * (rr * kLdK + kk), on ? P + (int64_t)(r0 + rr) * ld + k0 + kk : P, on);
    }
  }
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  const float cdf = 0.5f * (1.f + erff(z * 0.70710678118654752f));
  const float pdf = 0.39894228040143268f * expf(-0.5f * z * z);
  return cdf + z * pdf;
}


__device__ void gemm_tile(const MlpGemm& J, int tile, __nv_bfloat16* sm) {
  const __nv_bfloat16 *A = static_cast<const __nv_bfloat16*>(J.A), *B = static_cast<const __nv_bfloat16*>(J.B);
  const int m0 = tile / J.tiles_n * kT, n0 = tile % J.tiles_n * kT;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
  const int mat = lane >> 3, r = lane & 7;
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
  // byte offsets of this lane's ldmatrix rows at K offset 0 (A: matrices (m, k) = (0,0) (8,0) (0,8) (8,8);
  // B: (n, k) = (0,0) (0,8) (8,0) (8,8))
  const uint32_t oa = 2 * (J.ta ? ((mat >> 1) * 8 + r) * kLdM + wm + (mat & 1) * 8
                                : (wm + (mat & 1) * 8 + r) * kLdK + (mat >> 1) * 8);
  const uint32_t ob = 2 * (J.tb ? (wn + (mat >> 1) * 8 + r) * kLdK + (mat & 1) * 8
                                : ((mat & 1) * 8 + r) * kLdM + wn + (mat >> 1) * 8);
  const uint32_t ka = 2 * (J.ta ? kLdM : 1), kb = 2 * (J.tb ? 1 : kLdM);  // bytes per K
  float acc[2][4] = {};
  const int steps = (J.K + kTK - 1) / kTK;
  auto issue = [&](int st) {
    if (st < steps) {
      const uint32_t d = base + 2 * (st % kStages) * (2 * kTileElems);
      load_tile(d, A, J.lda, J.ta, m0, st * kTK, J.M, J.K);
      load_tile(d + 2 * kTileElems, B, J.ldb, !J.tb, n0, st * kTK, J.N, J.K);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int st = 0; st < kStages - 1; ++st) issue(st);
  for (int st = 0; st < steps; ++st) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // step st has landed for every thread; its ring slot's predecessor is read
    issue(st + kStages - 1);
    const uint32_t d = base + 2 * (st % kStages) * (2 * kTileElems);
#pragma unroll
    for (int ks = 0; ks < kTK; ks += 16) {
      uint32_t a[4], b[4];
      if (J.ta)
        ldmatrix4<true>(a, d + oa + ks * ka);
      else
        ldmatrix4<false>(a, d + oa + ks * ka);
      if (J.tb)
        ldmatrix4<false>(b, d + 2 * kTileElems + ob + ks * kb);
      else
        ldmatrix4<true>(b, d + 2 * kTileElems + ob + ks * kb);
      mma16816(acc[0], a, b);
      mma16816(acc[1], a, b + 2);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  const int gid = lane >> 2, tig = lane & 3;
  __nv_bfloat16* H = static_cast<__nv_bfloat16*>(J.H);
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int m = m0 + wm + gid + (q >= 2 ? 8 : 0);
      const int n = n0 + wn + 8 * j + 2 * tig + (q & 1);
      if (m >= J.M || n >= J.N) continue;
      float v = acc[j][q];
      if (J.bias) v += J.bias[n];
      if (J.mode == MLP_GELU_BWD) v *= gelu_grad(J.z[(int64_t)m * J.ldc + n]);
      J.C[(int64_t)m * J.ldc + n] = v;
      if (J.mode == MLP_GELU)
        H[(int64_t)m * J.ldh + n] = __float2bfloat16(gelu(v));
      else if (J.mode == MLP_GELU_BWD)
        H[(int64_t)m * J.ldh + n] = __float2bfloat16(v);
    }
}

// out[n] = sum_m x[m, n] of 32 columns: four row slices, added in order
__device__ void colsum_tile(const MlpColsum& J, int tile, float* sm) {
  const int c = threadIdx.x & 31, sl = threadIdx.x >> 5;  // four slices
  const int n = tile * 32 + c;
  float s = 0.f;
  if (n < J.N)
#pragma unroll 8
    for (int m = sl; m < J.M; m += 4) s += J.x[(int64_t)m * J.N + n];
  sm[sl * 32 + c] = s;
  __syncthreads();
  if (sl == 0 && n < J.N) J.out[n] = (sm[c] + sm[32 + c]) + (sm[64 + c] + sm[96 + c]);
}

__global__ void __launch_bounds__(128) mlp_step_kernel(MlpStep S) {
  __shared__ __align__(16) __nv_bfloat16 sm[kStages * 2 * kTileElems];
  int b = blockIdx.x;
  for (int i = 0; i < S.ngemm; ++i) {  // block-uniform
    if (b < S.gemm[i].tiles) {
      gemm_tile(S.gemm[i], b, sm);
      return;
    }
    b -= S.gemm[i].tiles;
  }
  colsum_tile(S.sum, b, reinterpret_cast<float*>(sm));
}

// first-layer input: the first `nlog` features of every row become
// log(max(x, floor)) * scale (the marginal enters as log-probabilities), the rest pass through;
// clears the loss of the coming backward pass
__global__ void input_kernel(const float* x, __nv_bfloat16* y, int64_t rows, int cols, int ld, int nlog, float floor_,
                             float scale, double* loss) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *loss = 0.0;
  const int64_t n = rows * cols;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / cols;
    const int c = (int)(i - r * cols);
    float v = x[i];
    if (c < nlog) v = logf(fmaxf(v, floor_)) * scale;
    y[r * ld + c] = __float2bfloat16(v);
  }
}

// the BF16 copy of parameter i (weights only, rows padded; its row by a 64-bit division: Adam on 9.4 M parameters
// takes 73 us, 44 with an unpadded copy, in a training step of 310 us that took 1573 with unpadded operands)
__device__ __forceinline__ void put_w16(const MlpW16& W, int64_t i, float v) {
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    const int64_t k = i - W.off[t];
    if (k >= 0 && k < W.len[t]) {
      const int64_t r = k / W.cols[t];
      static_cast<__nv_bfloat16*>(W.dst[t])[r * W.ld[t] + (k - r * W.cols[t])] = __float2bfloat16(v);
    }
  }
}

__global__ void to_bf16_kernel(const float* x, MlpW16 W, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    put_w16(W, i, x[i]);
}

// loss = mean((y - t)^2); dy = 2 (y - t) / count (FP32 and BF16 copies); loss summed into *loss (FP64)
__global__ void mse_kernel(const float* y, const float* t, float* dy32, __nv_bfloat16* dy16, int rows, int cols, int ld,
                           double* loss) {
  __shared__ double red[8];
  double local = 0.0;
  const int64_t n = (int64_t)rows * cols;
  const float scale = 2.f / (float)n;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / cols;
    const float d = y[i] - t[i];
    local += (double)d * d;
    const float g = scale * d;
    dy32[i] = g;
    dy16[r * ld + (i - r * cols)] = __float2bfloat16(g);
  }
  for (int o = 16; o; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = local;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    atomicAdd(loss, s / (double)n);
  }
}

// Adam on FP32 master weights, refresh of the BF16 working copy (bias-corrected moments)
__global__ void adam_kernel(float* w, const float* g, float* m1, float* m2, MlpW16 W, int64_t n, float lr, float b1,
                            float b2, float eps, float c1, float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.f - b1) * gi;
    const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    const float wi = w[i] - lr * (a / c1) / (sqrtf(b / c2) + eps);
    w[i] = wi;
    put_w16(W, i, wi);
  }
}

int blocks_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)(b > 2048 ? 2048 : (b < 1 ? 1 : b));
}

}  // namespace

MlpGemm mlp_gemm(const void* A, int lda, int ta, const void* B, int ldb, int tb, float* C, int ldc, int M, int N, int K) {
  MlpGemm J{};
  J.A = A, J.lda = lda, J.ta = ta;
  J.B = B, J.ldb = ldb, J.tb = tb;
  J.C = C, J.ldc = ldc;
  J.M = M, J.N = N, J.K = K;
  J.tiles_n = (N + kT - 1) / kT;
  J.tiles = J.tiles_n * ((M + kT - 1) / kT);
  return J;
}

cudaError_t mlp_step(const MlpStep& st, cudaStream_t s) {
  int grid = st.sum.x ? (st.sum.N + 31) / 32 : 0;
  for (int i = 0; i < st.ngemm; ++i) grid += st.gemm[i].tiles;
  mlp_step_kernel<<<grid, 128, 0, s>>>(st);
  return cudaGetLastError();
}

cudaError_t mlp_input(const float* x, void* y, int64_t rows, int cols, int ld, int nlog, float floor_, float scale,
                      double* loss, cudaStream_t s) {
  input_kernel<<<blocks_for(rows * cols), 256, 0, s>>>(x, static_cast<__nv_bfloat16*>(y), rows, cols, ld, nlog, floor_,
                                                       scale, loss);
  return cudaGetLastError();
}

cudaError_t mlp_to_bf16(const float* x, const MlpW16& w, int64_t n, cudaStream_t s) {
  to_bf16_kernel<<<blocks_for(n), 256, 0, s>>>(x, w, n);
  return cudaGetLastError();
}

cudaError_t mlp_mse(const float* y, const float* t, float* dy32, void* dy16, int rows, int cols, int ld, double* loss,
                    cudaStream_t s) {
  const int b = blocks_for((int64_t)rows * cols);
  mse_kernel<<<b > 304 ? 304 : b, 256, 0, s>>>(y, t, dy32, static_cast<__nv_bfloat16*>(dy16), rows, cols, ld, loss);
  return cudaGetLastError();
}

cudaError_t mlp_adam(float* w, const float* g, float* m1, float* m2, const MlpW16& w16, int64_t n, float lr, float b1,
                     float b2, float eps, float c1, float c2, cudaStream_t s) {
  adam_kernel<<<blocks_for(n), 256, 0, s>>>(w, g, m1, m2, w16, n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace treeot
