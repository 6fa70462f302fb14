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

// a <- merge(a, b).  kFar: for partials of small groups, one of which may hold
// nothing but a trace far away with next to no weight: the mean moves from the
// heavier side's, and squares are weighted before they are formed (d^2 leaves
// FP32's range at 1.8e19).  The trace kernels' folds, whose coefficients come
// from the prior, do without (their last bits, and 1 % of their time).
template <bool kFar = false>
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
  const bool from_b = kFar && wb > wa;
  const float f = from_b ? -(wa / w) : fb;
#pragma unroll
  for (int k = 0; k < kMaxCoef; ++k) {
    const float d = b.mean[k] - a.mean[k];
    a.mean[k] = fmaf(d, f, from_b ? b.mean[k] : a.mean[k]);
    const float m2 = fmaf(a.M2[k], ea, b.M2[k] * eb);
    a.M2[k] = kFar ? fmaf(d * cross, d, m2) : fmaf(d * d, cross, m2);
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
    res->deg_var[kk][j] = ok ? (double)df_div(make_float2(p[kk].M2[j], 0.0f), S[kk]) : 0.0;
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
// Warp `warp` (< kMaxDegrees) merges degree `warp` of G block partials into *out,
// with its sums S and S2 in double-float (written by several lanes: a barrier
// before they are read).  Two passes over the partials: the maximum and its
// index first, then every partial's sums rescaled to that maximum once and
// added, so the additions of a pass are independent and nothing waits on a
// chain of pairwise merges, each with two exponentials and a division.  The sums
// are S, S2, W = sum w (w = S e^(m - M) in FP32: the moments' weight) and, per
// coefficient, A = sum w d and B = sum (w d^2 + M2), d = mean - ref, ref the mean
// of the partial that holds the maximum.  The differences d, A, B and B - A^2 / W
// carry two FP32 words: ref may lie far from the rest of the population (a best
// trace alone in its block), where B is (distance / deviation)^2 times what is
// left of it.  In one word that lost 1.6e-3 of the variance at 100 deviations
// (pairwise merges: 1e-7), and sum w d the mean of 2^22 unit normals by half
// as much again.
//
// This code runs once per launch, by one block, after the kernel's data have
// streamed through L2: its instructions are fetched cold, so their number is
// what bounds it.  The loops stay rolled, two coefficients go through one f32x2
// instruction, and the eight pairs of sums leave the lanes by recursive halving
// (a lane sends half of what it holds and adds the other half).  The next
// partial is loaded while the current one is merged; up to 32 are read once,
// their reference coming from the lane that holds it.  10^5 traces x 32 points,
// whole call: 34.8 us with B in one word, 34.9 so (36.1 without the pairs); the
// 4096 uneven sets 10.6 and 9.6 ms (fewer live registers beside their hot loop).
struct PairSum {  // two sums, each in two words
  unsigned long long hi, lo;
};

// a + b; words normalised when a's and b's are
__device__ __forceinline__ PairSum pair_add(const PairSum& a, const PairSum& b) {
  const unsigned long long s = f2_add(a.hi, b.hi), bb = f2_sub(s, a.hi);
  const unsigned long long e = f2_add(f2_sub(a.hi, f2_sub(s, bb)), f2_sub(b.hi, bb));
  const unsigned long long t = f2_add(e, f2_add(a.lo, b.lo));
  PairSum r;
  r.hi = f2_add(s, t);
  r.lo = f2_sub(t, f2_sub(r.hi, s));
  return r;
}
__device__ __forceinline__ PairSum pair_shfl_xor(const PairSum& a, int o) {
  return PairSum{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
template <int H>
__device__ __forceinline__ void halve_sums(PairSum (&v)[8], int lane, int o) {
  const bool up = lane & o;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const PairSum give = up ? v[i] : v[i + H], keep = up ? v[i + H] : v[i];
    v[i] = pair_add(keep, pair_shfl_xor(give, o));
  }
}

__device__ __forceinline__ void merge_degree(const DegPartial* parts, int G, int warp, int lane,
                                             DegPartial* out, float2* S_out, float2* S2_out) {
  constexpr int kP = kMaxCoef / 2;
  static_assert(kMaxCoef == 6, "the sums make eight pairs");
  const DegPartial* mine = parts + warp;
  DegPartial nxt;
  deg_empty(nxt);
  if (lane < G) nxt = ld_partial_cg(mine + lane * kMaxDegrees);
  float M = nxt.m;
  int arg = nxt.arg, at = lane;
#pragma unroll 4
  for (int b = lane + 32; b < G; b += 32) {
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
  if (M == -INFINITY) {  // the same for the whole warp
    if (lane == 0) {
      deg_empty(*out);
      *S_out = *S2_out = make_float2(0.0f, 0.0f);
    }
    return;
  }
  DegPartial far = nxt;
  if (G > 32) far = ld_partial_cg(mine + at * kMaxDegrees);
  const int from = G > 32 ? lane : at;
  unsigned long long ref[kP];
#pragma unroll
  for (int k = 0; k < kP; ++k)
    ref[k] = __shfl_sync(0xffffffffu, f2_pack(far.mean[2 * k], far.mean[2 * k + 1]), from);
  PairSum v[8];  // (S, S2), (W, 0), A, B
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i].hi = v[i].lo = 0ull;
#pragma unroll 1
  for (int b = lane; b < G; b += 32) {
    const DegPartial cur = nxt;
    if (b + 32 < G) nxt = ld_partial_cg(mine + (b + 32) * kMaxDegrees);
    if (cur.m == -INFINITY) continue;
    const float e = expf(cur.m - M);
    // add x = (hi, lo) to a running sum: the high words' sum exactly, what it
    // rounds off and the low word in one word
    auto acc = [](PairSum& a, unsigned long long hi, unsigned long long lo) {
      const unsigned long long s = f2_add(a.hi, hi), bb = f2_sub(s, a.hi);
      const unsigned long long r = f2_add(f2_sub(a.hi, f2_sub(s, bb)), f2_sub(hi, bb));
      a.hi = s;
      a.lo = f2_add(a.lo, f2_add(r, lo));
    };
    const float2 w = df_prod(cur.S, e), s2 = df_mul(df_prod(cur.S2, e), e);
    acc(v[0], f2_pack(w.x, s2.x), f2_pack(w.y, s2.y));
    acc(v[1], f2_pack(w.x, 0.0f), 0ull);
    const unsigned long long ww = f2_pack(w.x, w.x), nw = f2_pack(-w.x, -w.x), ee = f2_pack(e, e);
#pragma unroll
    for (int k = 0; k < kP; ++k) {
      // d = mean - ref, t = w d, q = t d in two words (the negated products
      // give the FMAs their remainders)
      const unsigned long long mk = f2_pack(cur.mean[2 * k], cur.mean[2 * k + 1]);
      const unsigned long long d = f2_sub(mk, ref[k]), bb = f2_sub(d, mk);
      const unsigned long long dl = f2_sub(f2_sub(mk, f2_sub(d, bb)), f2_add(ref[k], bb));
      const unsigned long long t = f2_mul_rn(ww, d), nt = f2_mul(nw, d);
      const unsigned long long tl = f2_fma(ww, dl, f2_fma(ww, d, nt));
      acc(v[2 + k], t, tl);
      const unsigned long long q = f2_mul_rn(t, d), nq = f2_mul(nt, d);
      unsigned long long ql = f2_fma(t, dl, f2_fma(tl, d, f2_fma(t, d, nq)));
      // (second moments are not negative: nothing cancels in their sum)
      ql = f2_fma(f2_pack(cur.M2[2 * k], cur.M2[2 * k + 1]), ee, ql);
      acc(v[2 + kP + k], q, ql);
    }
  }
  halve_sums<4>(v, lane, 16);
  halve_sums<2>(v, lane, 8);
  halve_sums<1>(v, lane, 4);
#pragma unroll
  for (int o = 2; o > 0; o >>= 1) v[0] = pair_add(v[0], pair_shfl_xor(v[0], o));
  // lanes 4 i .. 4 i + 3 hold pair i; lane k < 6 forms coefficient k
  const float2 th = f2_unpack(v[0].hi), tl = f2_unpack(v[0].lo);
  const float2 t0 = make_float2(th.x, tl.x), t1 = make_float2(th.y, tl.y);
  const int k = lane < kMaxCoef ? lane : 0;
  const float2 S = df_shfl(t0, 0), S2 = df_shfl(t1, 0), W = df_shfl(t0, 4);
  const int at_a = 8 + 4 * (k / 2), at_b = at_a + 4 * kP;
  float2 A = df_shfl(t0, at_a), B = df_shfl(t0, at_b);
  const float2 A1 = df_shfl(t1, at_a), B1 = df_shfl(t1, at_b);
  if (k & 1) {
    A = A1;
    B = B1;
  }
  if (lane < kMaxCoef) {
    float mean = 0.0f, M2 = 0.0f;
    if (S.x > 0.0f) {
      const float rk = __ldcg((mine + at * kMaxDegrees)->mean + k);
      // A / W as the quotient and its remainder; the sum with ref may cancel
      const float inv = __frcp_rn(W.x), q = __fmul_rn(A.x, inv);
      const float r = __fadd_rn(__fmaf_rn(-q, W.x, A.x), __fmaf_rn(-q, W.y, A.y));
      const float2 sh = df_sum(q, __fmul_rn(r, inv));
      mean = df_add(make_float2(rk, 0.0f), sh).x;
      M2 = df_add(B, df_neg(df_mul(A, sh))).x;
      if (M2 < 0.0f) M2 = 0.0f;
      if (M2 != M2) {
        // a moment that is not finite, which the low words turn into NaN: its
        // sum in one word, infinite or NaN as its terms are
        M2 = 0.0f;
#pragma unroll 1
        for (int b = 0; b < G; ++b) {
          const DegPartial* cur = mine + b * kMaxDegrees;
          const float e = expf(__ldcg(&cur->m) - M), d = __ldcg(cur->mean + k) - rk;
          if (e > 0.0f) M2 += fmaf(__ldcg(&cur->S) * e * d, d, __ldcg(cur->M2 + k) * e);
        }
      }
    }
    out->mean[k] = mean;
    out->M2[k] = M2;
  }
  if (lane == 0) {
    out->m = M;
    out->arg = arg;
    out->S = S.x;
    out->S2 = S2.x;
    *S_out = S;
    *S2_out = S2;
  }
}

__device__ __forceinline__ void finalize_partials(const DegPartial* parts, int G, int n_deg,
                                                  int min_deg, int64_t N, WsHeader* hdr,
                                                  ppl_is_result* res) {
  __shared__ DegPartial fin[kMaxDegrees];
  __shared__ float2 fS[kMaxDegrees], fS2[kMaxDegrees];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < kMaxDegrees)
    merge_degree(parts, G, warp, lane, fin + warp, fS + warp, fS2 + warp);
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
  if (warp < kMaxDegrees)
    merge_degree(parts, G, warp, lane, out->deg + warp, out->S + warp, out->S2 + warp);
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
