// A lane's running sums of the weighted posterior moments of every degree, kept
// in registers as f32x2 pairs around a reference that the lanes of a warp
// share: S = sum w, S2 = sum w^2, A = sum w d, B = sum w d^2, with w = exp(lw -
// m_ref) and d = c - ref.  A trace is added to all four degrees with its
// weight masked (40 paired operations: no shuffle and no branch on the
// degree); when the reference moves, the sums move with it exactly.
//
// Squares are formed as (w d) d and never as w (d d): d^2 leaves FP32's range at
// |d| = 1.8e19, and its product with another degree's zero weight would be a NaN
// in that degree's sums.  (With d^2 shared by the degrees 31 operations: 2^24
// records summarised and resampled 435 us against 438 so, 1024 sets x 2^16 traces
// under their proposals 1987 against 2003.)
#pragma once

#include "posterior.cuh"
#include "trace.cuh"

namespace ppl {

// A reference moves to a better trace once that lies this far above it: the
// weights stay in range and the reference within a few standard deviations
// of the traces that carry weight.
constexpr float kRebaseNats = 8.0f;

struct LaneSums {
  unsigned long long s12, A[kMaxCoef / 2], B[kMaxCoef / 2];
};

__device__ __forceinline__ void lane_zero(LaneSums& a) {
  a.s12 = 0ull;
#pragma unroll
  for (int j = 0; j < kMaxCoef / 2; ++j) a.A[j] = a.B[j] = 0ull;
}

// Add a trace of degree index d (none when it matches no degree) and weight w:
// coefficients c, its degree's reference in f0 (ref 0-3) and f1.xy (ref 4, 5).
__device__ __forceinline__ void lane_add(LaneSums (&a)[kMaxDegrees], int d, float w,
                                         const float (&c)[kMaxCoef], const float4& f0,
                                         const float4& f1) {
  const unsigned long long d2[kMaxCoef / 2] = {
      f2_sub(f2_pack(c[0], c[1]), f2_pack(f0.x, f0.y)),
      f2_sub(f2_pack(c[2], c[3]), f2_pack(f0.z, f0.w)),
      f2_sub(f2_pack(c[4], c[5]), f2_pack(f1.x, f1.y))};
  const unsigned long long one_w = f2_pack(1.0f, w);
#pragma unroll
  for (int k = 0; k < kMaxDegrees; ++k) {
    const float wk = d == k ? w : 0.0f;
    const unsigned long long ww = f2_pack(wk, wk);
    a[k].s12 = f2_fma(ww, one_w, a[k].s12);
#pragma unroll
    for (int j = 0; j < kMaxCoef / 2; ++j) {
      a[k].A[j] = f2_fma(ww, d2[j], a[k].A[j]);
      a[k].B[j] = f2_fma(f2_mul(ww, d2[j]), d2[j], a[k].B[j]);
    }
  }
}

// Move a lane's sums to a reference g below the old one (g = old - new per
// coefficient), rescaling the weights by ex (first: a reference far away that
// carried a negligible weight moves without leaving FP32's range).
__device__ __forceinline__ void lane_move(LaneSums& a, const float (&g)[kMaxCoef], float ex) {
  const float2 s = f2_unpack(a.s12);
  const float es = s.x * ex;
  const unsigned long long ee = f2_pack(ex, ex), ss = f2_pack(es, es);
#pragma unroll
  for (int j = 0; j < kMaxCoef / 2; ++j) {
    const unsigned long long gg = f2_pack(g[2 * j], g[2 * j + 1]), A0 = f2_mul(ee, a.A[j]);
    const unsigned long long A1 = f2_fma(ss, gg, A0);  // A + S g
    a.B[j] = f2_fma(gg, f2_add(A0, A1), f2_mul(ee, a.B[j]));
    a.A[j] = A1;
  }
  a.s12 = f2_pack(es, s.y * ex * ex);
}

// The warp's partial of one degree in every lane: its lanes' sums around ref
// (c[6], m_ref), rescaled to the log-weight m of trace arg (-inf: none).
__device__ __forceinline__ DegPartial lane_partial(const LaneSums& a, const float* ref, float m,
                                                   int arg) {
  const float2 s = f2_unpack(a.s12);
  const float S = warp_sum(s.x), S2 = warp_sum(s.y);
  float A[kMaxCoef], B[kMaxCoef];
#pragma unroll
  for (int j = 0; j < kMaxCoef / 2; ++j) {
    const float2 av = f2_unpack(a.A[j]), bv = f2_unpack(a.B[j]);
    A[2 * j] = warp_sum(av.x);
    A[2 * j + 1] = warp_sum(av.y);
    B[2 * j] = warp_sum(bv.x);
    B[2 * j + 1] = warp_sum(bv.y);
  }
  DegPartial r;
  deg_empty(r);
  r.m = m;
  r.arg = arg;
  if (m > -INFINITY && S > 0.0f) {
    const float ex = expf(ref[6] - m), inv = 1.0f / S;
    r.S = S * ex;
    r.S2 = S2 * ex * ex;
#pragma unroll
    for (int j = 0; j < kMaxCoef; ++j) {
      const float sh = A[j] * inv;
      r.mean[j] = ref[j] + sh;
      r.M2[j] = fmaxf(fmaf(-sh, A[j], B[j]), 0.0f) * ex;
    }
  }
  return r;
}

}  // namespace ppl
