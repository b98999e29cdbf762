// Compact groups of support points for the factored recomputed-cost apply
// (fact_task.cuh): every node's points are sorted into groups of 64, 32 or 16
// close-by points, at create.
//
// Sort-tile-recursive order: the points of a chunk (at most 4096, in their
// given order) are sorted along the first coordinate into slabs, each slab along
// the second into tiles (and along the third), a tile holding one group.  One
// CTA per chunk, a bitonic sort of 64-bit keys (segment, coordinate, index) in
// shared memory; a support of more than 4096 points is grouped chunk by chunk,
// its groups as compact as those of 4096 points spread over the same region.
//
// Which size.  The factored form's error grows with kappa = s r^2 (s = scale
// log2(e) / eps, r^2 the mean over the groups of the squared half of a group's
// longer side), the difference form's with the squared transport distance.
// Measured on the GPU against FP64 iterates (rms error of the potentials in
// units of eps after 2 and 6 half-steps, random trees of 64..900 points, D = 1..3,
// eps 0.004..0.05, geometric mean over 27 shapes): difference form 1.35e-7;
// factored within kappa limits 2, 2, 2: 1.21e-7; 4, 3, 3: 1.33e-7, but single
// shapes then lose up to 1.8x (2-D, 900 points, eps 0.004), all of them through
// groups of 32 and 16 above 2.  The iterates' floor (largest marginal error after
// 1600-3000 half-steps): 2.4e-7 -> 1.4e-7 on 16 x 16 stars, 1.2e-7 -> 0.7e-7 on 2-D
// clouds at eps 0.02, 1.0e-7 -> 0.6e-7 on 1-D barycenters.  A node takes the
// largest group size within its limit (larger groups share a staged value among
// more outputs), and the difference form if none is.
#include <cmath>

#include "internal.h"
#include "ptx.cuh"

namespace treeot {
namespace {

constexpr int kGroupThreads = 512;

__device__ __forceinline__ uint32_t float_key(float v) {  // order-preserving bits
  const uint32_t b = __float_as_uint(v);
  return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}

__device__ void bitonic_sort(uint64_t* k, int m) {
  for (int size = 2; size <= m; size <<= 1)
    for (int stride = size >> 1; stride; stride >>= 1) {
      __syncthreads();
      for (int i = threadIdx.x; i < m / 2; i += kGroupThreads) {
        const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
        const uint64_t a = k[lo], b = k[hi];
        const bool up = (lo & size) == 0;
        if ((a > b) == up) {
          k[lo] = b;
          k[hi] = a;
        }
      }
    }
  __syncthreads();
}

// the smallest q with q^p >= v (small integers)
__device__ __forceinline__ int iroot(int v, int p) {
  int q = 1;
  while ((p == 2 ? q * q : q * q * q) < v) ++q;
  return q;
}

// key order of the chunk's points for groups of gs; on return the low 16 bits
// of keys[i] are the chunk-relative index of the i-th point
__device__ void str_order(const float* x, int D, int cnt, int m, int gs, uint64_t* keys) {
  for (int i = threadIdx.x; i < m; i += kGroupThreads)
    keys[i] = i < cnt ? ((uint64_t)float_key(x[(int64_t)i * D]) << 16) | (uint32_t)i : ~0ull;
  bitonic_sort(keys, m);
  if (D == 1) return;
  const int ng = (cnt + gs - 1) / gs;
  const int S = iroot(ng, D);
  const int per = (ng + S - 1) / S * gs;  // points per slab
  for (int i = threadIdx.x; i < cnt; i += kGroupThreads) {
    const uint32_t idx = (uint32_t)keys[i] & 0xffffu;
    keys[i] = ((uint64_t)(i / per) << 48) | ((uint64_t)float_key(x[(int64_t)idx * D + 1]) << 16) | idx;
  }
  bitonic_sort(keys, m);
  if (D == 2) return;
  for (int i = threadIdx.x; i < cnt; i += kGroupThreads) {
    const uint32_t idx = (uint32_t)keys[i] & 0xffffu;
    const int slab = i / per, in = i - slab * per;
    const int ng2 = (min(per, cnt - slab * per) + gs - 1) / gs;
    const int S2 = iroot(ng2, 2);
    const int p2 = (ng2 + S2 - 1) / S2 * gs;
    const uint64_t seg = (uint64_t)slab * 64 + in / p2;
    keys[i] = (seg << 48) | ((uint64_t)float_key(x[(int64_t)idx * D + 2]) << 16) | idx;
  }
  bitonic_sort(keys, m);
}

__device__ __forceinline__ int pow2_at_least(int n) {
  int m = 2;
  while (m < n) m <<= 1;
  return m;
}

// sum over the chunk's groups of (half the longer side)^2, for every group size
__global__ void __launch_bounds__(kGroupThreads) group_measure_kernel(const GroupWork* work, const NodeD* nodes,
                                                                      const ProbD* probs, const float* coords,
                                                                      float* out) {
  __shared__ uint64_t keys[kGroupChunk];
  __shared__ float part[kGroupThreads];
  const GroupWork w = work[blockIdx.x];
  const NodeD nd = nodes[w.node];
  const int D = probs[nd.prob].dim;
  const float* x = coords + nd.coord_off + (int64_t)w.x0 * D;
  const int m = pow2_at_least(w.cnt);
  for (int v = 0; v < kGroupSizes; ++v) {
    const int gs = 64 >> v;
    str_order(x, D, w.cnt, m, gs, keys);
    const int ng = (w.cnt + gs - 1) / gs;
    float r2 = 0.f;
    for (int g = threadIdx.x; g < ng; g += kGroupThreads) {
      float side = 0.f;
      for (int k = 0; k < D; ++k) {
        float lo = INFINITY, hi = -INFINITY;
        for (int i = g * gs; i < min((g + 1) * gs, w.cnt); ++i) {
          const float c = x[(int64_t)((uint32_t)keys[i] & 0xffffu) * D + k];
          lo = fminf(lo, c);
          hi = fmaxf(hi, c);
        }
        side = fmaxf(side, hi - lo);
      }
      r2 += 0.25f * side * side;
    }
    part[threadIdx.x] = r2;
    __syncthreads();
    if (threadIdx.x == 0) {
      float s = 0.f;
      for (int i = 0; i < kGroupThreads; ++i) s += part[i];
      out[kGroupSizes * blockIdx.x + v] = s;
    }
    __syncthreads();
  }
}

// slots and group records of a chunk whose node takes groups of nd.gs
__global__ void __launch_bounds__(kGroupThreads) group_build_kernel(const GroupWork* work, const NodeD* nodes,
                                                                    const ProbD* probs, const float* coords,
                                                                    const uint32_t* cmax, float4* slot_x,
                                                                    float2* slot_q, float4* grp) {
  __shared__ uint64_t keys[kGroupChunk];
  const GroupWork w = work[blockIdx.x];
  const NodeD nd = nodes[w.node];
  const int gs = nd.gs;
  if (gs == 0) return;
  const int D = probs[nd.prob].dim;
  const double s = probs[nd.prob].cost_scale * kLog2e * probs[nd.prob].inv_eps;
  const float* x = coords + nd.coord_off + (int64_t)w.x0 * D;
  str_order(x, D, w.cnt, pow2_at_least(w.cnt), gs, keys);
  const float cm = __uint_as_float(cmax[nd.prob]);
  int e = 0;
  if (cm > 0.f) (void)frexpf(cm, &e);
  const float unit = ldexpf(1.f, e - 10);  // the grid of split_coords_kernel
  // a chunk but the last holds a multiple of 64 points; pads run to the end of the last block of 64
  const int slots = (w.cnt + 63) / 64 * 64;
  for (int g = threadIdx.x; g < slots / gs; g += kGroupThreads) {
    const int i0 = g * gs, i1 = min(i0 + gs, w.cnt);
    float c[3] = {0.f, 0.f, 0.f};
    float M[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // second moments 00 01 02 11 12 22
    for (int k = 0; k < D; ++k) {
      float sum = 0.f;
      for (int i = i0; i < i1; ++i) sum += x[(int64_t)((uint32_t)keys[i] & 0xffffu) * D + k];
      if (i1 > i0) c[k] = rintf(sum / (float)(i1 - i0) / unit) * unit;
    }
    for (int i = i0; i < i0 + gs; ++i) {
      const uint32_t idx = (uint32_t)keys[min(i, w.cnt - 1)] & 0xffffu;  // pads repeat the last point
      float d[3] = {0.f, 0.f, 0.f};
      double q = 0.0;
      if (i < i1)
        for (int k = 0; k < D; ++k) {
          const float v = x[(int64_t)idx * D + k];
          d[k] = v - c[k];
          const double dd = (double)v - (double)c[k];
          q += dd * dd;
        }
      M[0] += d[0] * d[0], M[1] += d[0] * d[1], M[2] += d[0] * d[2];
      M[3] += d[1] * d[1], M[4] += d[1] * d[2], M[5] += d[2] * d[2];
      // s |x'|^2 as a two-float, its high part on the 2^-10 grid
      q *= s;
      const float qh = (float)(rint(q * kGrid) / kGrid);
      const int64_t at = nd.slot_off + w.x0 + i;
      slot_x[at] = make_float4(d[0], d[1], d[2], __int_as_float(w.x0 + (int)idx));
      slot_q[at] = make_float2(qh, (float)(q - (double)qh));
    }
    // inverse of the second moments (with a small ridge; zero for a single place)
    const float ridge = 1e-3f * (M[0] + M[3] + M[5]) / D + 1e-30f;
    float I[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float a = M[0] + ridge, d1 = M[3] + ridge, f = M[5] + ridge;
    if (D == 1) {
      I[0] = 1.f / a;
    } else if (D == 2) {
      const float det = a * d1 - M[1] * M[1];
      I[0] = d1 / det, I[1] = -M[1] / det, I[2] = a / det;
    } else {
      const float A00 = d1 * f - M[4] * M[4], A01 = M[2] * M[4] - M[1] * f, A02 = M[1] * M[4] - M[2] * d1;
      const float det = a * A00 + M[1] * A01 + M[2] * A02;
      I[0] = A00 / det, I[1] = A01 / det, I[2] = A02 / det;
      I[3] = (a * f - M[2] * M[2]) / det, I[4] = (M[1] * M[2] - a * M[4]) / det, I[5] = (a * d1 - M[1] * M[1]) / det;
    }
    for (int k = 0; k < 6; ++k)
      if (!isfinite(I[k]) || ridge < 1e-25f) I[k] = 0.f;
    float4* r = grp + 3 * ((nd.slot_off + w.x0 + i0) / 8);
    r[0] = make_float4(c[0], c[1], c[2], unit);
    r[1] = make_float4(I[0], I[1], I[2], I[3]);
    r[2] = make_float4(I[4], I[5], 0.f, 0.f);
  }
}

}  // namespace

cudaError_t launch_group_measure(const GroupWork* work, int32_t nwork, const NodeD* nodes, const ProbD* probs,
                                 const float* coords, float* out, cudaStream_t s) {
  if (nwork <= 0) return cudaSuccess;
  group_measure_kernel<<<nwork, kGroupThreads, 0, s>>>(work, nodes, probs, coords, out);
  return cudaGetLastError();
}

cudaError_t launch_group_build(const GroupWork* work, int32_t nwork, const NodeD* nodes, const ProbD* probs,
                               const float* coords, const uint32_t* cmax, float4* slot_x, float2* slot_q, float4* grp,
                               cudaStream_t s) {
  if (nwork <= 0) return cudaSuccess;
  group_build_kernel<<<nwork, kGroupThreads, 0, s>>>(work, nodes, probs, coords, cmax, slot_x, slot_q, grp);
  return cudaGetLastError();
}

}  // namespace treeot
