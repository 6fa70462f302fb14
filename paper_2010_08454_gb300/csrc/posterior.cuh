// One-pass posterior reduction of weighted line-fitting traces (§3.6.2 the
// normalisation of the log-weights; Fig. 1 the returned coefficients).
//
// A group of traces (one warp's or block's of one instance) is reduced to a
// per-degree partial: the best log-weight m and its index, S = sum exp(lw - m),
// S2 = sum exp(2 (lw - m)), and the weighted mean and second central moment
// M2 = sum w (c - mean)^2 of every coefficient.  Within a group the moments are
// formed around the group's best trace of that degree (a shift that keeps the
// FP32 sums well conditioned), and partials merge exactly in real arithmetic:
// rescale by exp(m_a - m), then combine means and M2 by the parallel-variance
// rule (Chan, Golub and LeVeque 1979).  The LSE, ESS, degree masses and pooled
// moments all follow from the per-degree partials.
#pragma once

#include "common.cuh"
#include "dfloat.cuh"
#include "poly.cuh"

namespace ppl {

struct __align__(16) DegPartial {
  float m;
  int arg;
  float S, S2;
  float mean[kMaxCoef];
  float M2[kMaxCoef];
};

__device__ __forceinline__ void deg_empty(DegPartial& p) {
  p.m = -INFINITY;
  p.arg = 0x7fffffff;
  p.S = 0.0f;
  p.S2 = 0.0f;
#pragma unroll
  for (int k = 0; k < kMaxCoef; ++k) {
    p.mean[k] = 0.0f;
    p.M2[k] = 0.0f;
  }
}

// a <- merge(a, b)
__device__ __forceinline__ void deg_merge(DegPartial& a, const DegPartial& b) {
  if (b.m == -INFINITY) return;
  if (a.m == -INFINITY) {
    a = b;
    return;
  }
  const float M = fmaxf(a.m, b.m);
  const float ea = expf(a.m - M), eb = expf(b.m - M);
  const float wa = a.S * ea, wb = b.S * eb, w = wa + wb;
  const float fb = wb / w, cross = wa * fb;
#pragma unroll
  for (int k = 0; k < kMaxCoef; ++k) {
    const float d = b.mean[k] - a.mean[k];
    a.mean[k] = fmaf(d, fb, a.mean[k]);
    a.M2[k] = fmaf(d * d, cross, fmaf(a.M2[k], ea, b.M2[k] * eb));
  }
  a.S2 = fmaf(a.S2, ea * ea, b.S2 * eb * eb);
  a.S = w;
  if (b.m > a.m || (b.m == a.m && b.arg < a.arg)) a.arg = b.arg;
  a.m = M;
}

__device__ __forceinline__ DegPartial deg_shfl_xor(const DegPartial& p, int mask) {
  DegPartial o;
  o.m = __shfl_xor_sync(0xffffffffu, p.m, mask);
  o.arg = __shfl_xor_sync(0xffffffffu, p.arg, mask);
  o.S = __shfl_xor_sync(0xffffffffu, p.S, mask);
  o.S2 = __shfl_xor_sync(0xffffffffu, p.S2, mask);
#pragma unroll
  for (int k = 0; k < kMaxCoef; ++k) {
    o.mean[k] = __shfl_xor_sync(0xffffffffu, p.mean[k], mask);
    o.M2[k] = __shfl_xor_sync(0xffffffffu, p.M2[k], mask);
  }
  return o;
}

// Load a partial written by another block of the running kernel, from L2.
__device__ __forceinline__ DegPartial ld_partial_cg(const DegPartial* src) {
  static_assert(sizeof(DegPartial) == 64, "DegPartial is four 16-byte words");
  DegPartial o;
  const float4* s = reinterpret_cast<const float4*>(src);
  float4* d = reinterpret_cast<float4*>(&o);
#pragma unroll
  for (int i = 0; i < 4; ++i) d[i] = __ldcg(s + i);
  return o;
}

// Summary of a population from its four per-degree partials (in shared
// memory), by the 32 lanes of one warp (every lane calls it).  S and S2 are
// the per-degree sums around each degree's maximum as double-floats.  No FP64
// arithmetic but single conversions and power-of-two scalings (GB300's FP64
// pipe is narrow: a chain of FP64 exp, log and divisions took about 7 us): the
// degree weights e^(m_k - M) = 2^n_k w_k (exp_split, so a degree's mass keeps
// its relative precision far below FP32's range), the masses w_k S_k and their
// total s in double-float, log s by df_log, p(n) and the ESS as corrected FP32
// quotients scaled back by 2^n_k in FP64.  Lane k < 4 works out degree k, lanes
// 0 and 1 the two logarithms, lanes 0-23 one (degree, coefficient) variance
// each, lanes 0-5 one pooled mean each: the code runs once per launch, cold
// in the instruction caches, so what bounds it is its length (one copy of
// each function spread over lanes instead of four unrolled ones).
__device__ __forceinline__ void write_summary_warp(const DegPartial* p, const float2* S,
                                                   const float2* S2, int n_deg,
                                                   int min_deg, int64_t N, int32_t status,
                                                   ppl_is_result* res) {
  const int lane = threadIdx.x & 31;
  const int k = lane & (kMaxDegrees - 1);  // (lanes 4.. repeat lanes 0-3 up to the shuffles)
  const bool has = k < n_deg && p[k].m != -INFINITY;
  const float mk = has ? p[k].m : -INFINITY;
  const float2 Sk = S[k], S2k = S2[k];
  float M = mk;
  int32_t arg = has ? p[k].arg : 0x7fffffff;
#pragma unroll
  for (int o = 1; o < kMaxDegrees; o <<= 1) {
    const float om = __shfl_xor_sync(0xffffffffu, M, o);
    const int32_t oa = __shfl_xor_sync(0xffffffffu, arg, o);
    if (om > M || (om == M && oa < arg)) {
      M = om;
      arg = oa;
    }
  }
  if (M == -INFINITY) arg = -1;
  // degree k's mass 2^n mw and e^(2 (m_k - M)) S2_k; s, s2 their totals
  // (terms below 2^-120 of the best degree's, which is at least 1, vanish
  // at double-float precision)
  int n = 0;
  float2 mw = make_float2(0.0f, 0.0f), s = mw, s2 = mw;
  if (has && Sk.x > 0.0f) {
    // m_k - M = dh + dl exactly (TwoSum of two floats); e^dl = 1 + dl
    const float dh = __fsub_rn(mk, M);
    const float bb = __fsub_rn(dh, mk);
    const float dl = __fsub_rn(__fsub_rn(mk, __fsub_rn(dh, bb)), __fadd_rn(M, bb));
    const ExpSplit e = exp_split(dh);
    const float2 w = df_add(make_float2(e.m, 0.0f), make_float2(__fmul_rn(e.m, dl), 0.0f));
    n = e.n;
    mw = df_mul(Sk, w);
    if (e.n >= -120) s = df_mul(mw, exp2i(e.n));
    if (e.n >= -60) s2 = df_mul(df_mul(df_mul(S2k, w), w), exp2i(2 * e.n));
  }
#pragma unroll
  for (int o = 1; o < kMaxDegrees; o <<= 1) {
    s = df_add(s, df_shfl_xor(s, o));
    s2 = df_add(s2, df_shfl_xor(s2, o));
  }
  // p(n): the FP32 quotient mw / s scaled by 2^n (FP32 value for the pooled
  // means, FP64 for the output)
  const float pq = (s.x > 0.0f && mw.x > 0.0f) ? df_div(mw, s) : 0.0f;
  const float pf = n >= -120 ? __fmul_rn(pq, exp2i(n)) : 0.0f;
  // lanes 0-23: (degree kk, coefficient j) mean and variance
  if (lane < kMaxDegrees * kMaxCoef) {
    const int kk = lane / kMaxCoef, j = lane % kMaxCoef;
    const bool ok = kk < n_deg && p[kk].m != -INFINITY && S[kk].x > 0.0f && p[kk].S > 0.0f;
    res->deg_mean[kk][j] = ok ? (double)p[kk].mean[j] : 0.0;
    res->deg_var[kk][j] = ok ? (double)__fdiv_rn(p[kk].M2[j], p[kk].S) : 0.0;
  }
  // pooled coefficient means (written by lanes 0-5) and the heaviest degree
  {
    const int j = lane < kMaxCoef ? lane : 0;
    float2 mc = make_float2(0.0f, 0.0f);
    float best_p = 0.0f;
    int best = 0;
#pragma unroll 1
    for (int kk = 0; kk < kMaxDegrees; ++kk) {
      const float pk = __shfl_sync(0xffffffffu, pf, kk);
      if (pk > best_p) {
        best_p = pk;
        best = kk;
      }
      if (kk < n_deg && p[kk].m != -INFINITY && S[kk].x > 0.0f && p[kk].S > 0.0f)
        mc = df_add(mc, df_prod(pk, p[kk].mean[j]));
    }
    if (lane < kMaxCoef) res->mean_c[lane] = df_to_double(mc);
    if (lane == 0) res->map_deg = min_deg + best;
  }
  if (lane < kMaxDegrees) {
    // 2^n as an FP64 value (n >= -1022; smaller masses underflow to 0)
    const double scale = n >= -1022 ? __hiloint2double((n + 1023) << 20, 0) : 0.0;
    res->p_n[k] = (double)pq * scale;
    res->deg_max_lw[k] = has ? (double)mk : -INFINITY;
    res->deg_argmax[k] = has ? p[k].arg : -1;
  }
  // lane 0: log s, lane 1: log N
  const float2 lg = df_log(lane == 1 || !(s.x > 0.0f) ? df_from_i64(N) : s);
  const float2 log_n = make_float2(__shfl_sync(0xffffffffu, lg.x, 1), __shfl_sync(0xffffffffu, lg.y, 1));
  if (lane == 0) {
    if (s.x > 0.0f) {
      res->lse = (double)M + df_to_double(lg);
      res->log_z = (double)M + df_to_double(df_add(lg, df_neg(log_n)));
      res->ess = (double)df_div(df_mul(s, s), s2);
    } else {  // no finite weight
      res->lse = -INFINITY;
      res->log_z = -INFINITY;
      res->ess = nan("");
    }
    res->max_lw = (double)M;
    res->argmax = arg;
    res->n_particles = N;
    res->n_deg = n_deg;
    res->status = status;
    res->pad = 0;  // every field is written: callers need not clear the result
  }
}

// A degree's sums S, S2 over partials q rescaled to the merged maximum M
// (FP32 exp of the difference, double-float products and sums), added by the
// lanes of a warp; every lane gets the totals.
struct DegSums {
  float2 S, S2;
  __device__ __forceinline__ void zero() {
    S = make_float2(0.0f, 0.0f);
    S2 = make_float2(0.0f, 0.0f);
  }
  __device__ __forceinline__ void add(float qm, float2 qS, float2 qS2, float M) {
    if (qm == -INFINITY) return;
    const float e = expf(qm - M);
    S = df_add(S, df_mul(qS, e));
    S2 = df_add(S2, df_mul(df_mul(qS2, e), e));
  }
  __device__ __forceinline__ void warp_total() {
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
      S = df_add(S, df_shfl_xor(S, o));
      S2 = df_add(S2, df_shfl_xor(S2, o));
    }
  }
};

// ---------------------------------------------------------------------------
// Final merge of the per-block partials, by the last block: warp k merges
// degree k's partials (merge_degree), warp 0 writes the summary.
// ---------------------------------------------------------------------------
// Warp `warp` (< kMaxDegrees) merges degree `warp` of G block partials in two
// passes over them: the maximum and its index first, then every partial's
// sums rescaled to that maximum once and added (S, S2 and sum w (mean - ref)
// in double-float, ref the mean of the partial that holds the maximum; second
// moments in FP32), so the additions of a pass are independent and nothing
// waits on a chain of pairwise merges, each with two exponentials and a
// division.  (With sum w (mean - ref) in FP32 the mean of 2^22 unit normals
// lost to the pairwise chain: 1.0e-6 against 6.4e-7 of its norm.)
__device__ __forceinline__ void merge_degree(const DegPartial* parts, int G, int warp, int lane,
                                             DegPartial& a, DegSums& ds) {
  // This code runs once per launch, by one block, after the kernel's data
  // have streamed through L2: its instructions are fetched cold, so the loops
  // stay rolled (fewer instruction fetches), and the next partial is loaded
  // while the current one is merged.
  deg_empty(a);
  ds.zero();
  const DegPartial* mine = parts + warp;
  float M = -INFINITY;
  int arg = 0x7fffffff, at = 0;
#pragma unroll 4
  for (int b = lane; b < G; b += 32) {
    const float2 h = __ldcg(reinterpret_cast<const float2*>(mine + b * kMaxDegrees));
    const int ha = __float_as_int(h.y);
    if (h.x > M || (h.x == M && ha < arg)) {
      M = h.x;
      arg = ha;
      at = b;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float om = __shfl_xor_sync(0xffffffffu, M, o);
    const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
    const int ob = __shfl_xor_sync(0xffffffffu, at, o);
    if (om > M || (om == M && oa < arg)) {
      M = om;
      arg = oa;
      at = ob;
    }
  }
  if (M == -INFINITY) return;  // the same for the whole warp
  const DegPartial ref = ld_partial_cg(mine + at * kMaxDegrees);
  float2 A[kMaxCoef];
  float B[kMaxCoef];
#pragma unroll
  for (int k = 0; k < kMaxCoef; ++k) {
    A[k] = make_float2(0.0f, 0.0f);
    B[k] = 0.0f;
  }
  DegPartial nxt;
  if (lane < G) nxt = ld_partial_cg(mine + lane * kMaxDegrees);
#pragma unroll 1
  for (int b = lane; b < G; b += 32) {
    const DegPartial cur = nxt;
    if (b + 32 < G) nxt = ld_partial_cg(mine + (b + 32) * kMaxDegrees);
    if (cur.m == -INFINITY) continue;
    const float e = expf(cur.m - M), w = cur.S * e;
    ds.S = df_add(ds.S, df_prod(cur.S, e));
    ds.S2 = df_add(ds.S2, df_mul(df_prod(cur.S2, e), e));
#pragma unroll
    for (int k = 0; k < kMaxCoef; ++k) {
      const float d = cur.mean[k] - ref.mean[k];
      A[k] = df_add(A[k], df_prod(w, d));
      B[k] = fmaf(cur.M2[k], e, fmaf(w * d, d, B[k]));
    }
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    ds.S = df_add(ds.S, df_shfl_xor(ds.S, o));
    ds.S2 = df_add(ds.S2, df_shfl_xor(ds.S2, o));
#pragma unroll
    for (int k = 0; k < kMaxCoef; ++k) {
      A[k] = df_add(A[k], df_shfl_xor(A[k], o));
      B[k] += __shfl_xor_sync(0xffffffffu, B[k], o);
    }
  }
  a.m = M;
  a.arg = arg;
  a.S = ds.S.x;
  a.S2 = ds.S2.x;
  if (a.S > 0.0f) {
    const float inv = __frcp_rn(a.S);
#pragma unroll
    for (int k = 0; k < kMaxCoef; ++k) {
      // ref + A / S with the quotient's and the sum's remainders (they may cancel)
      const float q = __fmul_rn(A[k].x, inv);
      const float r = __fadd_rn(__fmaf_rn(-q, ds.S.x, A[k].x), __fmaf_rn(-q, ds.S.y, A[k].y));
      const float2 mean = df_add(make_float2(ref.mean[k], 0.0f), make_float2(q, __fmul_rn(r, inv)));
      a.mean[k] = mean.x;
      a.M2[k] = fmaxf(fmaf(-q, A[k].x, B[k]), 0.0f);
    }
  }
}

__device__ __forceinline__ void finalize_partials(const DegPartial* parts, int G, int n_deg,
                                                  int min_deg, int64_t N, WsHeader* hdr,
                                                  ppl_is_result* res) {
  __shared__ DegPartial fin[kMaxDegrees];
  __shared__ float2 fS[kMaxDegrees], fS2[kMaxDegrees];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < kMaxDegrees) {
    DegPartial a;
    DegSums ds;
    merge_degree(parts, G, warp, lane, a, ds);
    if (lane == 0) {
      fin[warp] = a;
      fS[warp] = ds.S;
      fS2[warp] = ds.S2;
    }
  }
  __syncthreads();
  if (warp == 0) {
    int32_t st = 0;
    if (lane == 0) {
      bool any = false;
      for (int k = 0; k < n_deg; ++k) any |= fin[k].m != -INFINITY;
      if (!any) record_status(&hdr->status, PPL_EEMPTY);
      st = ld_volatile_i32(&hdr->status);
    }
    if (res) write_summary_warp(fin, fS, fS2, n_deg, min_deg, N, st, res);
  }
}



// ---------------------------------------------------------------------------
// One shard's share of a likelihood-weighting pass whose particles are split
// over several devices: its per-degree partials merged (FP32 means and
// second moments, double-float sums around each degree's maximum), its particle
// count and device status.  Shards merge exactly like blocks (§3.6.2: the
// normalisation runs over all samples, wherever they were drawn).
// ---------------------------------------------------------------------------
struct __align__(16) IsPartial {
  DegPartial deg[kMaxDegrees];
  float2 S[kMaxDegrees], S2[kMaxDegrees];  // double-float sums around each degree's maximum
  int64_t n;
  int32_t status, n_deg, min_deg, pad0;
  unsigned char pad[32];
};
static_assert(sizeof(IsPartial) == 384, "the public ppl_is_partial is 384 bytes");

// The last block's merge of the block partials into a shard partial (the
// first part of finalize_partials, without the summary).
__device__ __forceinline__ void finalize_to_partial(const DegPartial* parts, int G, int n_deg,
                                                    int min_deg, int64_t N, WsHeader* hdr,
                                                    IsPartial* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < kMaxDegrees) {
    DegPartial a;
    DegSums ds;
    merge_degree(parts, G, warp, lane, a, ds);
    if (lane == 0) {
      out->deg[warp] = a;
      out->S[warp] = ds.S;
      out->S2[warp] = ds.S2;
    }
  }
  if (threadIdx.x == 0) {
    out->n = N;
    out->n_deg = n_deg;
    out->min_deg = min_deg;
    out->status = ld_volatile_i32(&hdr->status);
  }
}

// Merge of P shard partials into the summary of the whole population, by one
// block: warp k merges degree k (the maxima exactly, means and second
// moments by the parallel rule in FP32, the sums rescaled to the merged
// maximum in double-float).  N is the total particle count.
__device__ __forceinline__ void merge_shard_partials(const IsPartial* parts, int P, int64_t N,
                                                     int32_t status, ppl_is_result* res) {
  __shared__ DegPartial fin[kMaxDegrees];
  __shared__ float2 fS[kMaxDegrees], fS2[kMaxDegrees];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_deg = parts[0].n_deg, min_deg = parts[0].min_deg;
  if (warp < kMaxDegrees) {
    DegPartial a;
    deg_empty(a);
    for (int g = lane; g < P; g += 32) deg_merge(a, parts[g].deg[warp]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const DegPartial other = deg_shfl_xor(a, o);
      deg_merge(a, other);
    }
    DegSums ds;
    ds.zero();
    if (a.m != -INFINITY)
      for (int g = lane; g < P; g += 32)
        ds.add(parts[g].deg[warp].m, parts[g].S[warp], parts[g].S2[warp], a.m);
    ds.warp_total();
    if (lane == 0) {
      fin[warp] = a;
      fS[warp] = ds.S;
      fS2[warp] = ds.S2;
    }
  }
  __syncthreads();
  if (warp == 0) {
    int32_t st = status;
    for (int g = 0; g < P && st == 0; ++g) st = parts[g].status;
    bool any = false;
    for (int k = 0; k < n_deg; ++k) any |= fin[k].m != -INFINITY;
    if (st == 0 && !any) st = PPL_EEMPTY;
    write_summary_warp(fin, fS, fS2, n_deg, min_deg, N, st, res);
  }
}

}  // namespace ppl
