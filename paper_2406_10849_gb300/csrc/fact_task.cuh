// Recomputed-cost edge apply over compact groups of output points (factored
// form), shared by the per-half-step apply kernel and the persistent forest
// kernel.  The planner (group.cu) sorts every node's points into compact groups
// of 64, 32 or 16; a warp takes 64 of them at a time, two outputs per lane.
//
// The argument.  With a group's centre c and a second centre cy near the
// group's transport targets, x' = x - c, y' = y - cy,
//   -s |x - y|^2 = -s |y - c|^2 + 2s x'.y'  +  [2s x'.(cy - c) - s |x'|^2],
// so per (group, y) one staged value A(y) = h(y) - F - s |y - c|^2 and the
// vector Y(y) = 2s y' serve every output of the group, the bracket off(x) is
// added to the output's frame once, and a term costs D FMAs, one ex2 and one
// FMA into the sum:  t = A + sum_k x'_k Y_k,  sum += 2^t w(y).
// (The difference form of recomp_task.cuh needs 3D + 2 FP32 operations before
// the exponential.)  The MUFU is the floor (32 ex2 per clock and SM, against 3 of
// 4 issue and FP32 slots used per term for D = 2).  Measured on 64 trees of 128 ..
// 2048 points: 262 us per launch, MUFU 49 % and issue slots 61 % busy while an SM
// has work, and a fifth of the launch in its tail.
//
// Accuracy.  Differences are taken on the 2^-10 sigma coordinate grid of
// split_coords_kernel: |y - c|^2 is exact up to its small low part, A lives on
// the 2^-10 grid of the operands, and what is left of it, with the operand's low
// part (|e| <= 2^-10 together), is the term's weight w = 2^e.  The remaining roundings are those of the products
// x'_k Y_k, of size s r |y'|; cy comes from a least-squares slope of the
// previous messages' frames over the group, which makes y' of the significant
// terms small (the spread of the targets, not the transport distance).  The
// planner marks groups where s r^2 (r: the largest coordinate of x') is too large
// for the result to be at least as accurate as the difference form's; those are
// summed by that form (see group.cu).
//
// Range.  One frame F per group: an output's sum is about 2^(b(x) - F), b the
// previous message's frame less off(x).  F lies kFactRoom binades above the
// largest b, so that every argument is below -2: there ex2.approx has one mean
// relative error for all (-5.05e-8, against -0.1e-8 on [-1, 1) and +3.4e-8 from
// 2 on, measured over each unit interval), which the final scaling takes out;
// what is left of it is 3e-8 rms and independent between terms.  With F at the
// middle of b both signs met within a node.  A group whose frames
// spread over more than kFactSpread binades, or one of whose sums leaves
// [2^-84, 2^100] (frames that moved far since the last half-step), is summed again
// by the difference form with each output's own maximum.
#pragma once
#include "recomp_task.cuh"

namespace treeot {
namespace {

// shared memory per warp (floats): 32 staged records of 10; for each of 64 outputs x' and index, a (frame, sum)
// pair and a two-float sum; the constants of up to 8 groups
constexpr int kFactWarp = 32 * 10 + 64 * 8 + 8 * 8;
constexpr int kFactSmemFloats = 8 * kFactWarp;
constexpr float kFactRoom = 4.f;
constexpr float kEx2Bias = 5.05e-8f;       // minus the mean relative error of ex2.approx below -2
constexpr float kFactSpread = 76.f;
constexpr float kFactLo = 5.1698788e-26f;  // 2^-84: a term below 2^-126 (flushed) weighs less than 2^-42
constexpr float kFactHi = 1.2676506e30f;   // 2^100

// a packed pair (v, v)
__device__ __forceinline__ uint64_t pair_of(float v) {
  uint64_t p;
  asm volatile("mov.b64 %0, {%1, %1};" : "=l"(p) : "f"(v));
  return p;
}
// x * b + c per lane, x a packed pair
__device__ __forceinline__ float2 fma2p(uint64_t x, float2 b, float2 c) {
  uint64_t r;
  asm("{\n\t.reg .b64 b, c;\n\tmov.b64 b, {%2, %3};\n\tmov.b64 c, {%4, %5};\n\tfma.rn.f32x2 %0, %1, b, c;\n\t}"
      : "=l"(r)
      : "l"(x), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
  return v;
}

// a + b = s + e exactly
__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

// (s, l) += v with the sum's rounding error kept in l
__device__ __forceinline__ void add_to(float& s, float& l, float v) {
  const float2 t = two_sum(s, v);
  s = t.x;
  l += t.y;
}

// A lane's four outputs summed by the difference form over the points [y0, y1) of its slice (every
// kSlices-th), each relative to its own maximum: the fallback of a group whose frames do not fit.  Two passes
// (maximum, sum) over points staged in the warp's shared memory, 64 at a time.  A stage's terms are summed in
// FP32 (32 at most) and the stages as a two-float.  out: frames in, (frame, sum) out.
template <int D>
__device__ __noinline__ void fact_slow(const ApplyArgs& A, const float4* rows, int64_t coord_own, int64_t coord_nbr,
                                       int64_t h_off, int y0, int y1, int slice, int slices, float shi, float slo,
                                       float4* stage, float2* out) {
  float* wts = reinterpret_cast<float*>(stage + 64);
  const int lane = threadIdx.x & 31;
  float px[4][D], cm[4], R[4], S[4], Sl[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = __float_as_int(rows[r].w);
#pragma unroll
    for (int k = 0; k < D; ++k) px[r][k] = A.coords[coord_own + (int64_t)row * D + k];
    cm[r] = -kInf;
    S[r] = Sl[r] = 0.f;
    R[r] = out[r].x;
  }
  for (int pass = 0; pass < 2; ++pass) {
    for (int b = y0; b < y1; b += 64) {
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int y = min(b + lane + 32 * h, y1 - 1);
        const float* q = A.coords + coord_nbr + (int64_t)y * D;
        const float hh = b + lane + 32 * h < y1 ? A.hh[h_off + y] : -kInf;
        const float u = A.hl[h_off + y] * 0.69314718f;
        wts[lane + 32 * h] = fmaf(u, fmaf(u, fmaf(u, 1.f / 6.f, 0.5f), 1.f), 1.f);
        stage[lane + 32 * h] = make_float4(q[0], D > 1 ? q[D > 1 ? 1 : 0] : 0.f, D > 2 ? q[D > 2 ? 2 : 0] : 0.f, hh);
      }
      __syncwarp();
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
      for (int i = slice; i < 64; i += slices) {
        const float4 q = stage[i];
        const float w = wts[i];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          float dx = px[r][0] - q.x;
          float c = dx * dx;
          if (D > 1) {
            dx = px[r][D > 1 ? 1 : 0] - q.y;
            c = fmaf(dx, dx, c);
          }
          if (D > 2) {
            dx = px[r][D > 2 ? 2 : 0] - q.z;
            c = fmaf(dx, dx, c);
          }
          const float t = fmaf(-c, slo, fmaf(-c, shi, q.w - R[r]));
          if (pass == 0)
            cm[r] = fmaxf(cm[r], t);
          else
            acc[r] = fmaf(ex2(t), w, acc[r]);
        }
      }
      if (pass == 1)
#pragma unroll
        for (int r = 0; r < 4; ++r) add_to(S[r], Sl[r], acc[r]);
    }
    if (pass == 0)
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (cm[r] > -kInf) R[r] += quant(cm[r]);
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) out[r] = make_float2(R[r], S[r] + Sl[r]);
  __syncwarp();
}

// raw data of a pair of reduction points: 8- or 16-byte loads (even points: the operand starts at a
// multiple of 32, a node's coordinates at a multiple of 4 floats).  The second point of an odd
// support's last pair is padding (finite; the staging masks it).
template <int D>
struct FactRaw {
  float2 hh, hl;
  float2 h[D], l[D];  // the pair's 2 D coordinates, hi and lo, in memory order
};

// loads that stay where they are written (a stage ahead of their use)
__device__ __forceinline__ float2 ld_ahead2(const float* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_ahead4(const float* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

template <int D>
__device__ __forceinline__ void fact_load(const ApplyArgs& A, int64_t coord_off, int64_t h_off, int y, FactRaw<D>& v) {
  v.hh = ld_ahead2(A.hh + h_off + y);
  v.hl = ld_ahead2(A.hl + h_off + y);
  const float* ph = A.coords_hi + coord_off + (int64_t)y * D;
  const float* pl = A.coords_lo + coord_off + (int64_t)y * D;
  if (D == 2) {
    const float4 a = ld_ahead4(ph), b = ld_ahead4(pl);
    v.h[0] = make_float2(a.x, a.y), v.h[D > 1 ? 1 : 0] = make_float2(a.z, a.w);
    v.l[0] = make_float2(b.x, b.y), v.l[D > 1 ? 1 : 0] = make_float2(b.z, b.w);
  } else {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      v.h[k] = ld_ahead2(ph + 2 * k);
      v.l[k] = ld_ahead2(pl + 2 * k);
    }
  }
}

// coordinate k of the two points of a pair stored in memory order
template <int D>
__device__ __forceinline__ float2 fact_pick(const float2* m, int k) {
  const float a = k % 2 ? m[k / 2].y : m[k / 2].x;
  const float b = (D + k) % 2 ? m[(D + k) / 2].y : m[(D + k) / 2].x;
  return make_float2(a, b);
}

// v on the 2^-10 grid by the magic addition (|v| < 2^12; beyond that a coarser grid, with terms far
// below anything that counts)
__device__ __forceinline__ float2 quant2(float2 v) {
  const float2 m = make_float2(12288.f, 12288.f), n = make_float2(-12288.f, -12288.f);
  return add2(add2(v, m), n);
}

// merge two (frame, sum) pieces, either empty
__device__ __forceinline__ float2 merge2(float2 a, float2 b) {
  if (!(b.y > 0.f)) return a;
  if (!(a.y > 0.f)) return b;
  const float R = fmaxf(a.x, b.x);
  return make_float2(R, a.y * ex2(a.x - R) + b.y * ex2(b.x - R));
}

// A block of 64 of the owner's output slots (64 / GS groups) against points of the neighbour, by one warp.
// The set-up runs for all 64 outputs at once, two per lane; then each group in turn: GS / 4 lanes hold its
// outputs, four each, and the 128 / GS lane sets ("slices") take turns on the staged point pairs, so a staged
// record is read from shared memory once per four outputs (with two per lane the shared-memory reads were the
// limit: 64 % of their peak rate against 41 % of the MUFU's).  SHARED: 2^lw warps of the CTA take equal shares
// of the points and meet in shared memory (every warp of the CTA calls; nrow = 0: no block).
template <int D, int GS, bool SHARED>
__device__ __forceinline__ void fact_block(const ApplyArgs& A, const FactItem& it, float* sm, int warp, int lw) {
  constexpr int NG = 64 / GS;          // groups
  constexpr int kLanes = GS / 4;       // lanes per slice
  constexpr int kSlices = 32 / kLanes;
  constexpr int kSteps = 32 / kSlices; // staged pairs per slice and stage
  constexpr int kChunk = kSteps < 4 ? kSteps : 4;
  constexpr int kFlush = 32;           // stages (2048 points) per running sum
  const float shi = it.shi, slo = it.slo;
  const int lane = threadIdx.x & 31;
  const int wpb = SHARED ? 1 << lw : 1;
  const int share = SHARED ? warp & (wpb - 1) : 0;
  // per warp: 32 records (A, A, w, w), (Y0, Y0, Y1, Y1), then for D = 3 (Y2, Y2); 64 outputs' x' and index;
  // their frames; their sums; the groups' (F, c, cy)
  float* base = sm + warp * kFactWarp;
  float4* s0 = reinterpret_cast<float4*>(base);
  float4* s1 = s0 + 32;
  float2* s2 = reinterpret_cast<float2*>(s1 + 32);
  float4* sx = reinterpret_cast<float4*>(s2 + 32);
  float2* comb = reinterpret_cast<float2*>(sx + 64);  // (frame, sum) per output
  float2* sums = comb + 64;                           // two-float sum per output
  float* gc = reinterpret_cast<float*>(sums + 64);    // 8 floats per group
  const int nst = (it.n_nbr + 63) / 64;
  const int st0 = SHARED ? (int)((int64_t)nst * share >> lw) : 0;
  const int st1 = SHARED ? (int)((int64_t)nst * (share + 1) >> lw) : nst;
  const float2 nshi = make_float2(-shi, -shi), nslo = make_float2(-slo, -slo);
  const bool live = !SHARED || it.nrow > 0;
  const int nrow = it.nrow;
  const int last = (it.n_nbr - 1) & ~1;  // the last pair: loads past it repeat it
  int y = st0 * 64 + 2 * lane;
  FactRaw<D> raw;  // the first stage, in flight during the set-up
  fact_load<D>(A, it.coord_nbr, it.rev_off, min(y, last), raw);
  bool good[2];  // the lane's two outputs: r = 0, 1 -> lane + 32 r
  bool wide[2] = {false, false};  // of a group too wide for the factored form
  {
    float xp[2][D], frm[2], v[2];
    float2 off[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float4 x = A.slot_x[it.slot0 + lane + 32 * r];  // pads repeat a valid output
      sx[lane + 32 * r] = x;
      xp[r][0] = x.x;
      if (D > 1) xp[r][D > 1 ? 1 : 0] = x.y;
      if (D > 2) xp[r][D > 2 ? 2 : 0] = x.z;
      frm[r] = A.fr[it.off + __float_as_int(x.w)];
      const float2 rq = A.slot_q[it.slot0 + lane + 32 * r];
      off[r] = make_float2(-rq.x, -rq.y);
      v[r] = frm[r] + rq.x;
    }
    const float inv2s = 0.5f / shi;
    constexpr int kSpan = GS < 32 ? GS : 32;  // lanes that hold a group's outputs
    float c[D], cy[D];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int g = (lane + 32 * r) / GS;
      if (NG > 1 || r == 0) {  // one group over both outputs of every lane: worked out once
        const float4* gr = A.grp + 3 * ((it.slot0 + g * GS) / 8);
        const float4 g0 = gr[0], g1 = gr[1], g2 = gr[2];
        wide[r] = g2.z != 0.f;
        if (NG == 1) wide[1] = wide[0];
        // slope of the frames over the group: 2s (cy - c)
        const float vref = __shfl_sync(0xffffffffu, NG == 1 ? v[0] : v[r], lane & ~(kSpan - 1));
        float gs[D], e[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
          gs[k] = 0.f;
          if (NG == 1) {
            if (lane < nrow) gs[k] = (v[0] - vref) * xp[0][k];
            if (lane + 32 < nrow) gs[k] = fmaf(v[1] - vref, xp[1][k], gs[k]);
          } else if (lane + 32 * r < nrow) {
            gs[k] = (v[r] - vref) * xp[r][k];
          }
#pragma unroll
          for (int o = kSpan / 2; o; o >>= 1) gs[k] += __shfl_xor_sync(0xffffffffu, gs[k], o);
        }
        if (D == 1) e[0] = g1.x * gs[0];
        if (D == 2) {
          e[0] = fmaf(g1.x, gs[0], g1.y * gs[D > 1 ? 1 : 0]);
          e[D > 1 ? 1 : 0] = fmaf(g1.y, gs[0], g1.z * gs[D > 1 ? 1 : 0]);
        }
        if (D == 3) {
          const float p = gs[0], q = gs[D > 1 ? 1 : 0], w = gs[D > 2 ? 2 : 0];
          e[0] = fmaf(g1.x, p, fmaf(g1.y, q, g1.z * w));
          e[D > 1 ? 1 : 0] = fmaf(g1.y, p, fmaf(g1.w, q, g2.x * w));
          e[D > 2 ? 2 : 0] = fmaf(g1.z, p, fmaf(g2.x, q, g2.y * w));
        }
        const float unit = g0.w, inv_unit = 1.f / unit;
#pragma unroll
        for (int k = 0; k < D; ++k) {
          c[k] = k == 0 ? g0.x : k == 1 ? g0.y : g0.z;
          // a target outside the coordinates' range [-1024, 1024] units says nothing: stay inside it
          cy[k] = fminf(fmaxf(rintf((c[k] + e[k] * inv2s) * inv_unit), -1024.f), 1024.f) * unit;
        }
      }
#pragma unroll
      for (int k = 0; k < D; ++k) {
        // off(x) = 2s x'.(cy - c) - s |x'|^2 as a two-float; cy - c is exact (both on the grid)
        const float dc = cy[k] - c[k];
        const float eh = 2.f * shi * dc, el = fmaf(2.f * shi, dc, -eh) + 2.f * slo * dc;
        const float p = xp[r][k] * eh, pe = fmaf(xp[r][k], eh, -p) + xp[r][k] * el;
        const float2 ts = two_sum(off[r].x, p);
        off[r] = make_float2(ts.x, off[r].y + (ts.y + pe));
      }
      if ((lane & (kSpan - 1)) == 0) {
#pragma unroll
        for (int k = 0; k < D; ++k) {
          gc[8 * g + 1 + k] = c[k];
          gc[8 * g + 4 + k] = cy[k];
        }
      }
    }
    float hi[2], lo[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const bool on = lane + 32 * r < nrow;
      hi[r] = on ? frm[r] - off[r].x : -kInf;
      lo[r] = on ? off[r].x - frm[r] : -kInf;
    }
    if (NG == 1) {
      hi[0] = hi[1] = fmaxf(hi[0], hi[1]);
      lo[0] = lo[1] = fmaxf(lo[0], lo[1]);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (NG == 1 && r == 1) {
        hi[1] = hi[0];
        lo[1] = lo[0];
      } else
#pragma unroll
      for (int o = kSpan / 2; o; o >>= 1) {
        hi[r] = fmaxf(hi[r], __shfl_xor_sync(0xffffffffu, hi[r], o));
        lo[r] = fmaxf(lo[r], __shfl_xor_sync(0xffffffffu, lo[r], o));
      }
      const float F = hi[r] > -kInf ? quant(hi[r]) + kFactRoom : 0.f;
      good[r] = !(hi[r] + lo[r] > kFactSpread) && !wide[r];
      if ((lane & (kSpan - 1)) == 0) {
        gc[8 * ((lane + 32 * r) / GS)] = F;
        gc[8 * ((lane + 32 * r) / GS) + 7] = wide[r] ? 1.f : 0.f;
      }
      // frame F + off back on the grid, and what it leaves over, for the end
      const float2 fs = two_sum(F, off[r].x);
      const float q = quant(fs.x);
      comb[lane + 32 * r] = make_float2(q, (fs.x - q) + (fs.y + off[r].y));
    }
  }
  __syncwarp();
  const int ll = lane & (kLanes - 1), slice = lane / kLanes;
#pragma unroll 1
  for (int g = 0; g < NG; ++g) {
    if (g * GS >= nrow) break;  // warp-uniform
    if (gc[8 * g + 7] != 0.f) {  // warp-uniform: a wide group's sums come from the fallback below
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (slice == 0) sums[g * GS + ll + kLanes * r] = make_float2(0.f, 0.f);
      continue;
    }
    // (x, x) pairs, opaque so that they stay in registers instead of being rebuilt before every use
    uint64_t X[4][D];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 x = sx[g * GS + ll + kLanes * r];
      X[r][0] = pair_of(x.x);
      if (D > 1) X[r][D > 1 ? 1 : 0] = pair_of(x.y);
      if (D > 2) X[r][D > 2 ? 2 : 0] = pair_of(x.z);
    }
    const float F = gc[8 * g];
    float cst[D], cyst[D];
#pragma unroll
    for (int k = 0; k < D; ++k) cst[k] = gc[8 * g + 1 + k], cyst[k] = gc[8 * g + 4 + k];
    // the output's sum outside the loop as a two-float: every addition exact but the last rounding
    float S[4] = {0.f, 0.f, 0.f, 0.f}, Sl[4] = {0.f, 0.f, 0.f, 0.f};
    float2 acc[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r] = make_float2(0.f, 0.f);
    for (int st = st0; st < st1; ++st) {
      {
        // A and w: |y - c|^2 = P + Pe, P exact on the grid (see recomp_task_exact)
        float2 P = make_float2(0.f, 0.f), Pe = make_float2(0.f, 0.f);
        float2 Y[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
          const float2 ch = fact_pick<D>(raw.h, k), dl = fact_pick<D>(raw.l, k);
          const float2 dh = add2(ch, make_float2(-cst[k], -cst[k]));
          P = fma2(dh, dh, P);
          Pe = fma2(dl, fma2(make_float2(2.f, 2.f), dh, dl), Pe);
          const float2 dy = add2(add2(ch, make_float2(-cyst[k], -cyst[k])), dl);
          Y[k] = fma2(dy, make_float2(2.f * slo, 2.f * slo), mul2(dy, make_float2(2.f * shi, 2.f * shi)));
        }
        const float2 H = add2(raw.hh, make_float2(-F, -F));  // exact: both on the 2^-10 grid
        const float2 a = fma2(Pe, nshi, fma2(P, nshi, H));
        float2 ah = quant2(a);
        float2 ee = fma2(P, nshi, add2(H, make_float2(-ah.x, -ah.y)));
        ee = fma2(P, nslo, ee);
        ee = fma2(Pe, nshi, ee);
        ee = add2(ee, raw.hl);
        // no term (past the support, or h = -inf): A = -inf with an ordinary weight
        if (y >= it.n_nbr || raw.hh.x == -kInf) ah.x = -kInf, ee.x = 0.f;
        if (y + 1 >= it.n_nbr || raw.hh.y == -kInf) ah.y = -kInf, ee.y = 0.f;
        // w = 2^e by its Taylor series (|e| <= 2^-10: truncation below 2^-33)
        const float2 u = mul2(ee, make_float2(0.69314718f, 0.69314718f));
        const float2 w = fma2(u, fma2(u, make_float2(0.5f, 0.5f), make_float2(1.f, 1.f)), make_float2(1.f, 1.f));
        s0[lane] = make_float4(ah.x, ah.y, w.x, w.y);
        if (D == 1) s1[lane] = make_float4(Y[0].x, Y[0].y, 0.f, 0.f);
        if (D > 1) s1[lane] = make_float4(Y[0].x, Y[0].y, Y[D > 1 ? 1 : 0].x, Y[D > 1 ? 1 : 0].y);
        if (D > 2) s2[lane] = Y[D > 2 ? 2 : 0];
      }
      __syncwarp();
      y = st + 1 < st1 ? y + 64 : st0 * 64 + 2 * lane;  // the next stage, or the next group's first
      fact_load<D>(A, it.coord_nbr, it.rev_off, min(y, last), raw);
#pragma unroll 1
      for (int i0 = 0; i0 < kSteps; i0 += kChunk) {
        float2 s[4];
#pragma unroll
        for (int i = 0; i < kChunk; ++i) {
          const int j = (i0 + i) * kSlices + slice;
          const float4 q0 = s0[j], q1 = s1[j];
          const float2 q2 = D > 2 ? s2[j] : make_float2(0.f, 0.f);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            float2 tt = fma2p(X[r][0], make_float2(q1.x, q1.y), make_float2(q0.x, q0.y));
            if (D > 1) tt = fma2p(X[r][D > 1 ? 1 : 0], make_float2(q1.z, q1.w), tt);
            if (D > 2) tt = fma2p(X[r][D > 2 ? 2 : 0], q2, tt);
            const float2 ex = make_float2(ex2(tt.x), ex2(tt.y));
            const float2 w = make_float2(q0.z, q0.w);
            s[r] = i == 0 ? mul2(ex, w) : fma2(ex, w, s[r]);
          }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = add2(acc[r], s[r]);
      }
      if (((st - st0) & (kFlush - 1)) == kFlush - 1)  // bounds the length of a running sum
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          add_to(S[r], Sl[r], acc[r].x);
          add_to(S[r], Sl[r], acc[r].y);
          acc[r] = make_float2(0.f, 0.f);
        }
      __syncwarp();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      add_to(S[r], Sl[r], acc[r].x);
      add_to(S[r], Sl[r], acc[r].y);
#pragma unroll
      for (int o = kLanes; o < 32; o <<= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, S[r], o), ol = __shfl_xor_sync(0xffffffffu, Sl[r], o);
        const float2 ts = two_sum(S[r], oh);
        S[r] = ts.x;
        Sl[r] = (Sl[r] + ol) + ts.y;
      }
      if (slice == 0) sums[g * GS + ll + kLanes * r] = make_float2(S[r], Sl[r]);
    }
  }
  if (SHARED && wpb > 1)
    __syncthreads();
  else
    __syncwarp();
  float2 out[2];
  unsigned bad[2];  // ballots over the block's outputs
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int x = lane + 32 * r;
    float S = 0.f, Sl = 0.f;
    if (SHARED && wpb > 1) {  // the shares of a block, added in the order of its warps
      for (int w = 0; w < wpb; ++w) {
        const float2 q = sums[(w - share) * (kFactWarp / 2) + x];
        add_to(S, Sl, q.x);
        Sl += q.y;
      }
    } else {
      S = sums[x].x;
      Sl = sums[x].y;
    }
    if (x < nrow) good[r] = good[r] && S > kFactLo && S < kFactHi;
    bad[r] = __ballot_sync(0xffffffffu, x < nrow && !good[r]);
    const float2 fq = comb[x];
    const float u = fmaf(fq.y, 0.69314718f, kEx2Bias);
    out[r] = make_float2(fq.x, S + fmaf(S, fmaf(0.5f * u, u, u), Sl));  // one rounding
  }
  const bool slow = (bad[0] | bad[1]) != 0u;  // the same for every warp of a block
  if (slow) {
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 2; ++r) comb[lane + 32 * r] = out[r];
    __syncwarp();
    const int64_t coord_own = A.nodes[A.dedges[it.dedge].owner].coord_off;
#pragma unroll 1
    for (int g = 0; g < NG; ++g) {
      const unsigned m = GS == 64 ? bad[0] | bad[1]
                                  : (g * GS < 32 ? bad[0] : bad[1]) & (((GS < 32 ? 1u << (GS & 31) : 0u) - 1u) << ((g * GS) & 31));
      if (!m) continue;  // warp-uniform
      if (lane == 0 && share == 0 && gc[8 * g + 7] == 0.f) atomicAdd(A.fallbacks, 1ull);
      float4 rw[4];
      float2 so[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        rw[r] = sx[g * GS + ll + kLanes * r];
        so[r] = make_float2(A.fr[it.off + __float_as_int(rw[r].w)], 0.f);
      }
      fact_slow<D>(A, rw, coord_own, it.coord_nbr, it.rev_off, st0 * 64, min(st1 * 64, it.n_nbr), slice, kSlices, shi,
                   slo, s0, so);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int o = kLanes; o < 32; o <<= 1)
          so[r] = merge2(so[r], make_float2(__shfl_xor_sync(0xffffffffu, so[r].x, o),
                                            __shfl_xor_sync(0xffffffffu, so[r].y, o)));
        if (slice == 0) comb[g * GS + ll + kLanes * r] = so[r];
      }
    }
    __syncwarp();
  }
  if (SHARED && wpb > 1) {
    // the slow groups' shares merge through shared memory
    __syncthreads();
    if (slow && share == 0) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int x = lane + 32 * r, g = x / GS;
        const unsigned m = GS == 64 ? bad[0] | bad[1]
                                    : bad[r] & (((GS < 32 ? 1u << (GS & 31) : 0u) - 1u) << ((g * GS) & 31));
        out[r] = comb[x];
        if (m)
          for (int w = 1; w < wpb; ++w) out[r] = merge2(out[r], comb[w * (kFactWarp / 2) + x]);
      }
    }
  } else if (slow) {
#pragma unroll
    for (int r = 0; r < 2; ++r) out[r] = comb[lane + 32 * r];
  }
  if (live && share == 0)
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (lane + 32 * r < nrow) A.part32[it.part_off + __float_as_int(sx[lane + 32 * r].w)] = out[r];
  __syncwarp();
}

// A task of the CTA: the outputs in slots [o0, o0 + ocount) of the owner, 2^(kind - TASK_FACT) warps per block
// of 64
template <int D, int GS>
__device__ void fact_task(const ApplyArgs& A, const Task& t, float* sm) {
  const DEdgeD d = A.dedges[t.dedge];
  const NodeD own = A.nodes[d.owner];
  const NodeD nbn = A.nodes[d.nbr];
  const int lw = t.kind - TASK_FACT;
  const int warp = threadIdx.x >> 5, b = warp >> lw;
  FactItem it;
  it.slot0 = own.slot_off + t.o0;
  it.nrow = 0;
  if (b * 64 < t.ocount) {
    it.slot0 += b * 64;
    it.nrow = min(64, t.ocount - b * 64);
  }
  it.part_off = d.part_off + (int64_t)t.split * own.n;
  it.off = d.off;
  it.rev_off = d.rev_off + t.r0;
  it.coord_nbr = nbn.coord_off + (int64_t)t.r0 * D;
  it.n_nbr = t.rcount;
  it.dedge = t.dedge;
  it.shi = A.probs[d.prob].s2_scaled;
  it.slo = A.probs[d.prob].s2_scaled_lo;
  fact_block<D, GS, true>(A, it, sm, warp, lw);
}

template <int D>
__device__ __forceinline__ void fact_dispatch(const ApplyArgs& A, const Task& t, float* sm) {
  const int gs = A.nodes[A.dedges[t.dedge].owner].gs;
  if (gs == 64)
    fact_task<D, 64>(A, t, sm);
  else if (gs == 32)
    fact_task<D, 32>(A, t, sm);
  else
    fact_task<D, 16>(A, t, sm);
}

}  // namespace
}  // namespace treeot
