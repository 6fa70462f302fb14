// Draw policy of a learned proposal: the trace's random choices come from
// q(n, c | data) computed by the network (mlp.cu); the log-weight gains
// log p(n, c) - log q(n, c), so importance weighting (§3.6.2) still targets the
// posterior of the model of Fig. 1.  The draw reuses the prior trace's words
// (purpose POLY_TRACE): the degree by the inverse CDF of q at u = u01(w6), and
// c_j = mu + s z_j with the prior's Box-Muller normals.  A proposal equal to the
// prior therefore gives the prior trace bit for bit (correction exactly 0).
#pragma once

#include "trace.cuh"

namespace ppl {

constexpr int kMaxSlots = 22;  // coefficient slots the 48 network outputs can describe

struct ProposalSmem {
  float cum[kMaxDegrees];
  float logq[kMaxDegrees];
  int base[kMaxDegrees];
  float4 slot[kMaxSlots];  // mu, s, 1 / s, log s: one load per coefficient
  float log_p, log_sigma, sigma, inv_sigma;
};

// Proposal of one data set from its 48 network outputs, by the 32 lanes of one
// warp: lane i takes slot i, every lane the degrees.
__device__ __forceinline__ void load_proposal(const PolyParams& p, const float* o,
                                              ProposalSmem& ps) {
  const int lane = threadIdx.x & 31;
  float mx = -INFINITY;
  for (int k = 0; k < p.n_deg; ++k) mx = fmaxf(mx, o[k]);
  float se = 0.0f;
  for (int k = 0; k < p.n_deg; ++k) se += expf(o[k] - mx);
  const float lse = logf(se);
  float cum = 0.0f;
  int base = 0;
  for (int k = 0; k < kMaxDegrees; ++k) {
    float ck = 2.0f, lq = 0.0f;
    int bk = 0;
    if (k < p.n_deg) {
      cum += expf(o[k] - mx) / se;
      ck = cum;
      lq = (o[k] - mx) - lse;
      bk = base;
      base += p.min_deg + k + p.coef_offset;
    }
    if (lane == 0) {
      ps.cum[k] = ck;
      ps.logq[k] = lq;
      ps.base[k] = bk;
    }
  }
  const float log_sigma = logf(p.prior_sigma);
  if (lane == 0) {
    ps.sigma = p.prior_sigma;
    ps.inv_sigma = 1.0f / p.prior_sigma;
    ps.log_sigma = log_sigma;
    ps.log_p = -logf((float)p.n_deg);
  }
  if (lane < kMaxSlots && lane < base) {
    const float t = fminf(fmaxf(o[5 + 2 * lane], -9.0f), 1.0f);
    const float s = p.prior_sigma * expf(t);
    const float mu = p.prior_sigma * o[4 + 2 * lane];
    // (1 / s is the prior's reciprocal when s equals sigma).  Where the mean is NaN
    // or infinite, the density is NaN and the draws are made around 0: every such
    // trace has a NaN log-weight as before, but no coefficient that 0 x NaN would
    // carry into other degrees' sums.
    const bool ok = fabsf(mu) < INFINITY;
    ps.slot[lane] = make_float4(ok ? mu : 0.0f, s, 1.0f / s, ok ? log_sigma + t : NAN);
  }
}

// log N(x; mu, s^2) with 1/s given (one multiply instead of a division, in
// the same form for the prior and the proposal, so a proposal equal to the
// prior cancels exactly)
__device__ __forceinline__ float log_normal32(float x, float mu, float inv_s, float logs) {
  const float z = (x - mu) * inv_s;
  return -0.918938533f - logs - 0.5f * z * z;
}

struct LearnedDraw {
  PolyParams p;
  uint64_t seed;
  uint32_t instance;
  const ProposalSmem* ps;
  __device__ __forceinline__ int operator()(uint32_t i, float (&c)[kMaxCoef], float& corr) const {
    const uint4 a = philox_block(seed, i, instance, 0, kPolyTrace, 0);
    const uint4 b = philox_block(seed, i, instance, 0, kPolyTrace, 1);
    float z[kMaxCoef];
    box_muller(a.x, a.y, z[0], z[1]);
    box_muller(a.z, a.w, z[2], z[3]);
    box_muller(b.x, b.y, z[4], z[5]);
    // the inverse CDF of q at u: the first degree whose cumulative mass
    // exceeds u (the last one when rounding leaves u above every mass)
    const float u = u01(b.z);
    int k = 0;
#pragma unroll
    for (int kk = 0; kk < kMaxDegrees - 1; ++kk) k += (kk < p.n_deg - 1 && u >= ps->cum[kk]);
    const int n = p.min_deg + k, ncoef = n + p.coef_offset, base = ps->base[k];
    float cr = ps->log_p - ps->logq[k];
#pragma unroll
    for (int j = 0; j < kMaxCoef; ++j) {
      if (j < ncoef) {
        const float4 q = ps->slot[base + j];
        c[j] = fmaf(q.y, z[j], q.x);
        cr += log_normal32(c[j], 0.0f, ps->inv_sigma, ps->log_sigma) -
              log_normal32(c[j], q.x, q.z, q.w);
      } else {
        c[j] = 0.0f;
      }
    }
    corr = cr;
    return n;
  }
};

}  // namespace ppl
