// Compact groups of support points for the factored recomputed-cost apply
// (fact_task.cuh): every node's points are sorted into groups of 64, 32 or 16
// close-by points, at create.
//
// Sort-tile-recursive order: the points of a chunk (at most 4096, in their
// given order) are sorted along the first coordinate into slabs, each slab along
// the second into tiles (and along the third), a tile holding one group.  Slabs
// and tiles hold whole groups, as even in number as they divide: with the
// remainder in a last narrow slab its few groups spanned the slab's whole
// length (2048 uniform points in the square: one group in 16 had 6 times the
// mean's squared extent, now the widest has twice).  One
// CTA per chunk, a bitonic sort of 64-bit keys (segment, coordinate, index) in
// shared memory; a support of more than 4096 points is grouped chunk by chunk,
// its groups as compact as those of 4096 points spread over the same region.
//
// Which groups.  The factored form's error grows with kappa = s r^2 of the
// output's own group (s = scale log2(e) / eps, r the largest coordinate
// difference to the group's centre), the difference form's with the squared
// transport distance.  Measured on the GPU against FP64 messages of the same
// potentials (uniform, radially concentrated and outlier-ridden supports of 400 to 4096
// points, D = 1..3, eps 0.002..0.03; rms and largest error of the message in
// nats, by the kappa of the output's group, factored against difference form):
//   kappa    <= 1             1..2            2..4            5..6            8..10           > 20
//   rms      0.7e-7 / 1.2e-7  0.8e-7 / 1.2e-7 0.9e-7 / 1.2e-7 0.9e-7 / 1.2e-7 1.1e-7 / 1.2e-7 5.9e-7 / 1.5e-7
//   largest  4.0e-7 / 5.9e-7  3.9e-7 / 5.6e-7 5.3e-7 / 5.3e-7 1.3e-6 / 0.6e-6 1.2e-6 / 0.9e-6 8.5e-6 / 1.5e-6
// A group takes the factored form up to kappa = 4 (groups of 16 in three
// dimensions up to 2: 1.3e-7 against 1.1e-7 between 2 and 4), where neither error
// is larger than the difference form's; a wider one is summed by the difference
// form (the fallback in fact_task.cuh, about four times a group's time).  A node
// takes the largest group size (larger groups share a staged value among more
// outputs) that leaves few enough of its points in wide groups, and the
// difference form throughout if none does: an eighth of them on a large handle,
// whose per-warp queue takes the costlier blocks first (128 trees of 128-2048
// points, 16 half-steps, shares of 1/32, 1/16, 1/8: 11.23, 11.05, 10.91 ms), a 32nd on
// a small one, where a CTA waits for its slowest warp (64 trees of 64-512 points,
// 32 half-steps, 1/32 and 1/8: 1.71, 1.82 ms).  (With the limit on the node's mean
// kappa instead, single groups of clustered supports ran factored at kappa 40
// and beyond.)
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

// the p-th root of v to the nearest integer (p = 2 or 3, small v >= 1)
__device__ __forceinline__ int iroot(int v, int p) {
  int q = 1;
  while ((p == 2 ? (2 * q + 1) * (2 * q + 1) / 4 : (2 * q + 1) * (2 * q + 1) * (2 * q + 1) / 8) < v) ++q;
  return q;
}

// part k of n groups in S parts begins at group k n / S; the part that holds group g
__device__ __forceinline__ int part_of(int g, int n, int S) { return ((g + 1) * S - 1) / n; }

// the chunk's points in order of their first coordinate; on return the low 16 bits
// of keys[i] are the chunk-relative index of the i-th point
__device__ void first_order(const float* x, int D, int cnt, int m, uint64_t* keys) {
  for (int i = threadIdx.x; i < m; i += kGroupThreads)
    keys[i] = i < cnt ? ((uint64_t)float_key(x[(int64_t)i * D]) << 16) | (uint32_t)i : ~0ull;
  bitonic_sort(keys, m);
}

// from there the order for groups of gs (D > 1; in one dimension the first order is it)
__device__ void str_order(const float* x, int D, int cnt, int m, int gs, uint64_t* keys) {
  const int ng = (cnt + gs - 1) / gs;
  const int S = iroot(ng, D);
  for (int i = threadIdx.x; i < cnt; i += kGroupThreads) {
    const uint32_t idx = (uint32_t)keys[i] & 0xffffu;
    const int slab = part_of(i / gs, ng, S);
    keys[i] = ((uint64_t)slab << 48) | ((uint64_t)float_key(x[(int64_t)idx * D + 1]) << 16) | idx;
  }
  bitonic_sort(keys, m);
  if (D == 2) return;
  for (int i = threadIdx.x; i < cnt; i += kGroupThreads) {
    const uint32_t idx = (uint32_t)keys[i] & 0xffffu;
    const int slab = part_of(i / gs, ng, S);
    const int g0 = slab * ng / S, ng2 = (slab + 1) * ng / S - g0;
    const uint64_t seg = (uint64_t)slab * 64 + part_of(i / gs - g0, ng2, iroot(ng2, 2));
    keys[i] = (seg << 48) | ((uint64_t)float_key(x[(int64_t)idx * D + 2]) << 16) | idx;
  }
  bitonic_sort(keys, m);
}

__device__ __forceinline__ int pow2_at_least(int n) {
  int m = 2;
  while (m < n) m <<= 1;
  return m;
}

// the grid of split_coords_kernel
__device__ __forceinline__ float grid_unit(float cm) {
  int e = 0;
  if (cm > 0.f) (void)frexpf(cm, &e);
  return ldexpf(1.f, e - 10);
}

// the centre of the points keys[i0 .. i1): their mean, on the grid
__device__ __forceinline__ void group_centre(const float* x, int D, const uint64_t* keys, int i0, int i1, float unit,
                                             float* c) {
  for (int k = 0; k < D; ++k) {
    float sum = 0.f;
    for (int i = i0; i < i1; ++i) sum += x[(int64_t)((uint32_t)keys[i] & 0xffffu) * D + k];
    if (i1 > i0) c[k] = rintf(sum / (float)(i1 - i0) / unit) * unit;
  }
}

// too wide for the factored form: kappa = s r^2 above the limit (false for no points)
__device__ __forceinline__ bool group_wide(int gs, int D, float s, float r) {
  return !(s * r * r <= (gs == 16 && D == 3 ? kGroupKappa16 : kGroupKappa));
}

// slots and group records of a chunk in groups of gs, its points in the order of keys
__device__ void build_groups(const GroupWork& w, const ProbD& P, const float* x, const uint64_t* keys, int gs,
                             float unit, const GroupTables& T) {
  const int D = P.dim;
  const double s = P.cost_scale * kLog2e * P.inv_eps;
  // a chunk but the last holds a multiple of 64 points; pads run to the end of the last block of 64
  const int slots = (w.cnt + 63) / 64 * 64;
  for (int g = threadIdx.x; g < slots / gs; g += kGroupThreads) {
    const int i0 = g * gs, i1 = min(i0 + gs, w.cnt);
    float c[3] = {0.f, 0.f, 0.f};
    float M[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // second moments 00 01 02 11 12 22
    float far = 0.f;  // the largest coordinate difference to the centre
    group_centre(x, D, keys, i0, i1, unit, c);
    for (int i = i0; i < i0 + gs; ++i) {
      const uint32_t idx = (uint32_t)keys[min(i, w.cnt - 1)] & 0xffffu;  // pads repeat the last point
      float d[3] = {0.f, 0.f, 0.f};
      double q = 0.0;
      if (i < i1)
        for (int k = 0; k < D; ++k) {
          const float v = x[(int64_t)idx * D + k];
          d[k] = v - c[k];
          far = fmaxf(far, fabsf(d[k]));
          const double dd = (double)v - (double)c[k];
          q += dd * dd;
        }
      // in units of the grid: the coordinates' own unit may put squares, and a determinant of them, out of range
      const float e0 = d[0] / unit, e1 = d[1] / unit, e2 = d[2] / unit;
      M[0] += e0 * e0, M[1] += e0 * e1, M[2] += e0 * e2;
      M[3] += e1 * e1, M[4] += e1 * e2, M[5] += e2 * e2;
      // s |x'|^2 as a two-float, its high part on the 2^-10 grid
      q *= s;
      const float qh = (float)(rint(q * kGrid) / kGrid);
      const int64_t at = w.slot + i;
      T.slot_x[at] = make_float4(d[0], d[1], d[2], __int_as_float(w.x0 + (int)idx));
      T.slot_q[at] = make_float2(qh, (float)(q - (double)qh));
    }
    // inverse of the second moments (with a small ridge; zero for a single place)
    const float ridge = 1e-3f * (M[0] + M[3] + M[5]) / D;
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
    for (int k = 0; k < 6; ++k) {
      I[k] = I[k] / unit / unit;
      if (!isfinite(I[k])) I[k] = 0.f;
    }
    float4* r = T.grp + 3 * ((w.slot + i0) / 8);
    r[0] = make_float4(c[0], c[1], c[2], unit);
    r[1] = make_float4(I[0], I[1], I[2], I[3]);
    const bool wide = i1 > i0 && group_wide(gs, D, P.s2_scaled, far);
    r[2] = make_float4(I[4], I[5], wide ? 1.f : 0.f, 0.f);
    if (wide) atomicAdd(&T.block_wide[(w.slot + i0) / 64], i1 - i0);
  }
}

// the chunks of nodes with several, once the host has chosen the node's size (nd.gs; 0: none)
__global__ void __launch_bounds__(kGroupThreads) group_build_kernel(const GroupWork* work, const NodeD* nodes,
                                                                    const ProbD* probs, const float* coords,
                                                                    const uint32_t* cmax, GroupTables T) {
  __shared__ uint64_t keys[kGroupChunk];
  const GroupWork w = work[blockIdx.x];
  const NodeD nd = nodes[w.node];
  if (nd.gs == 0 || w.cnt == nd.n) return;  // block-uniform
  const ProbD P = probs[nd.prob];
  const float* x = coords + nd.coord_off + (int64_t)w.x0 * P.dim;
  first_order(x, P.dim, w.cnt, pow2_at_least(w.cnt), keys);
  if (P.dim > 1) str_order(x, P.dim, w.cnt, pow2_at_least(w.cnt), nd.gs, keys);
  build_groups(w, P, x, keys, nd.gs, grid_unit(__uint_as_float(cmax[nd.prob])), T);
}

// The points of the chunk that lie in wide groups, for every group size.  A node of a single chunk stops at the
// first size that leaves few enough of them (a 1 / share; the sizes after it count as wide throughout) and builds
// its groups there and then: a second launch, and the host's choice before it, would add some 60 us to every create.
__global__ void __launch_bounds__(kGroupThreads) group_plan_kernel(const GroupWork* work, const NodeD* nodes,
                                                                   const ProbD* probs, const float* coords,
                                                                   const uint32_t* cmax, int32_t share, int32_t* out,
                                                                   GroupTables T) {
  __shared__ uint64_t keys[kGroupChunk];
  __shared__ uint16_t first[kGroupChunk];
  __shared__ int s_wide;
  const GroupWork w = work[blockIdx.x];
  const NodeD nd = nodes[w.node];
  const int D = probs[nd.prob].dim;
  const float s = probs[nd.prob].s2_scaled;
  const float* x = coords + nd.coord_off + (int64_t)w.x0 * D;
  const float unit = grid_unit(__uint_as_float(cmax[nd.prob]));
  const int m = pow2_at_least(w.cnt);
  bool found = false;
  first_order(x, D, w.cnt, m, keys);
  if (D > 1)
    for (int i = threadIdx.x; i < w.cnt; i += kGroupThreads) first[i] = (uint16_t)keys[i];
  for (int v = 0; v < kGroupSizes; ++v) {
    const int gs = 64 >> v;
    if (found) {  // block-uniform
      if (threadIdx.x == 0) out[kGroupSizes * blockIdx.x + v] = w.cnt;
      continue;
    }
    if (D > 1) {
      __syncthreads();
      if (v > 0)
        for (int i = threadIdx.x; i < m; i += kGroupThreads) keys[i] = i < w.cnt ? first[i] : ~0ull;
      __syncthreads();
      str_order(x, D, w.cnt, m, gs, keys);
    }
    if (threadIdx.x == 0) s_wide = 0;
    __syncthreads();
    for (int g = threadIdx.x; g < (w.cnt + gs - 1) / gs; g += kGroupThreads) {
      const int i0 = g * gs, i1 = min(i0 + gs, w.cnt);
      float c[3] = {0.f, 0.f, 0.f}, r = 0.f;
      group_centre(x, D, keys, i0, i1, unit, c);
      for (int i = i0; i < i1; ++i)
        for (int k = 0; k < D; ++k)
          r = fmaxf(r, fabsf(x[(int64_t)((uint32_t)keys[i] & 0xffffu) * D + k] - c[k]));
      if (group_wide(gs, D, s, r)) atomicAdd(&s_wide, i1 - i0);
    }
    __syncthreads();
    if (threadIdx.x == 0) out[kGroupSizes * blockIdx.x + v] = s_wide;
    found = w.cnt == nd.n && s_wide * share <= w.cnt;
    __syncthreads();
    if (found) build_groups(w, probs[nd.prob], x, keys, gs, unit, T);  // block-uniform; only reads keys
  }
}

}  // namespace

cudaError_t launch_group_plan(const GroupWork* work, int32_t nwork, const NodeD* nodes, const ProbD* probs,
                              const float* coords, const uint32_t* cmax, int32_t share, int32_t* out,
                              const GroupTables& t, cudaStream_t s) {
  if (nwork <= 0) return cudaSuccess;
  group_plan_kernel<<<nwork, kGroupThreads, 0, s>>>(work, nodes, probs, coords, cmax, share, out, t);
  return cudaGetLastError();
}

cudaError_t launch_group_build(const GroupWork* work, int32_t nwork, const NodeD* nodes, const ProbD* probs,
                               const float* coords, const uint32_t* cmax, const GroupTables& t, cudaStream_t s) {
  if (nwork <= 0) return cudaSuccess;
  group_build_kernel<<<nwork, kGroupThreads, 0, s>>>(work, nodes, probs, coords, cmax, t);
  return cudaGetLastError();
}

}  // namespace treeot
