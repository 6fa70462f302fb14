// The whole bootstrap particle filter on the linear-Gaussian state-space model
// in one persistent kernel (particle methods: the paper's stated future work,
// §6; observe as in §3.4, Fig. 2): a cooperative grid, described here, or for
// small populations one thread-block cluster (smc_cluster_kernel).  One block of 1024 threads per
// SM; each thread keeps its R particles' state and log-weights in registers
// for all T steps; the steps are separated by grid barriers instead of kernel
// launches.  The arithmetic of a step is exactly that of ppl_smc_step (same
// draws, same FP32 operations, same fixed-point systematic resampling), so
// both give the same particles.
//
// A step is: propagate and weight (registers) -> block partial -> barrier 1,
// after which every block merges all the partials itself, in one fixed order,
// so that all take the same resampling decision; when resampling: fixed-point
// weights and block totals -> barrier 2, after which every block scans all
// the totals itself and finds which output slots its particles are the
// ancestors of -> each block writes its particles' states into those slots
// -> barrier 3 -> every thread reads its slots.  The three barriers are plain
// arrival counts: a merge or scan done once by the last arriving block and
// published to the others would add its own latency and that of the release
// to every step, for a few kilobytes that every block reads from L2 in one
// round trip.
//
// Every barrier wait is bounded; a block whose wait runs out records
// PPL_ETIMEOUT and every block leaves at its next wait, so the kernel always
// ends.  The launch is cooperative, which guarantees that all blocks are
// resident at once (or fails to launch).
#include <algorithm>

#include "dfloat.cuh"
#include "gridsync.cuh"
#include "kernels.h"
#include "rng.cuh"

namespace ppl {

constexpr int kSmcTpb = 1024;          // threads of a block: one block per SM
constexpr int kSmcWarps = kSmcTpb / 32;
constexpr int kSmcMaxGrid = kSmcTpb;   // the merging block holds one partial per thread
constexpr int kSmcOut = 24576;         // output slots of a block's mark table
constexpr int kSmcShort = 6;           // rows a thread marks alone
constexpr int kSmcRuns = 128;          // longer runs of a block (its threads mark any beyond)

// A block's normalisation partial: m = max lw, s = sum exp(lw - m),
// s2 = sum exp(2 (lw - m)), nan = some lw is NaN.  One 16-byte load.
struct __align__(16) SmcPart {
  float m, s, s2;
  int nan;
};

// What one step leaves for the evidence and ESS outputs, which are formed in
// FP64 once after the last step: M the maximum log-weight, S and S2 the sums of
// exp(lw - M) and exp(2 (lw - M)) as unevaluated FP32 pairs.
struct __align__(16) SmcStep {
  float M, s_hi, s_lo, s2_hi, s2_lo;
  int32_t flag, pad[2];
};

// Control block at offset 0 of the workspace: the status word (first, where
// ppl_workspace_status reads it) on its own line, then the barrier words.
struct __align__(128) SmcCtl {
  int32_t status;
  int32_t pad[31];
  GridCtl g;
};

struct SmcArgs {
  LgssmParams p;
  const float* y;  // [T]
  int32_t T;
  uint64_t seed;
  int64_t N;
  float* x_out;
  float* lw_out;
  double* logz;        // [1]
  int32_t* resampled;  // [T]
  double* ess;         // [T]
  SmcCtl* ctl;
  SmcPart* parts;      // [2][grid] block partials of even and odd steps
  uint64_t* bsum;      // [grid] block totals of the fixed-point weights
  SmcStep* stash;      // [T]
  float* xbuf;         // [N] the resampled states, by output slot
};

// One particle's step: the FP32 operations of ppl_smc_step, in its order, one
// rounding each.
__device__ __forceinline__ void smc_propagate(const SmcArgs& a, uint32_t i, uint32_t t, float yt,
                                              float& x, float& lw) {
  const uint4 w = philox_block(a.seed, i, 0, t, kLgssmPropagate, 0);
  const float z0 = normal32(w.x, w.y);
  const float xi = __fadd_rn(__fmul_rn(a.p.phi, x), __fmul_rn(a.p.q_sigma, z0));
  const float d = __fsub_rn(yt, xi);
  lw = __fadd_rn(lw, __fadd_rn(a.p.obs_const, __fmul_rn(__fmul_rn(a.p.neg_half_inv_r2, d), d)));
  x = xi;
}

// evidence and ESS of every step, in FP64, by block 0 after the last step:
// log Z = sum over resampling steps of (lse_t - log N), plus lse_T - log N
// when the last step did not resample (its weights are carried unnormalised)
__device__ __forceinline__ void smc_outputs(const SmcArgs& a, double* sh_z) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double log_n = log((double)a.N);
  double z = 0.0;
  for (int t = tid; t < a.T; t += kSmcTpb) {
    const float4 h0 = __ldcg(reinterpret_cast<const float4*>(a.stash + t));
    const float4 h1 = __ldcg(reinterpret_cast<const float4*>(a.stash + t) + 1);
    const double S1 = (double)h0.y + (double)h0.z;
    const double S2 = (double)h0.w + (double)h1.x;
    const int flag = __float_as_int(h1.y);
    const double lse = (double)h0.x + log(S1);
    a.ess[t] = S1 * S1 / S2;
    a.resampled[t] = flag;
    if (flag || t == a.T - 1) z += lse - log_n;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  if (lane == 0) sh_z[warp] = z;
  __syncthreads();
  if (warp == 0) {
    z = sh_z[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    if (lane == 0) a.logz[0] = z;
  }
}

// Inclusive warp scan.  The filter's weights are quantised log-weights, whose
// sums cannot pass 2^61 (N weights of at most 2^(61 - ceil(log2 N))): plain sums.
__device__ __forceinline__ uint64_t warp_scan_plain(uint64_t v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// Thread `tid` of block b holds particles i0 .. i0 + R - 1, i0 = (b kSmcTpb + tid) R,
// so a thread's fixed-point weights are consecutive terms of the prefix sum.
template <int R>
__global__ void __launch_bounds__(kSmcTpb, 1) smc_persistent_kernel(SmcArgs a) {
  constexpr int64_t P = (int64_t)kSmcTpb * R;  // particles of one block
  extern __shared__ __align__(16) unsigned char smc_dyn[];
  uint64_t* sA = reinterpret_cast<uint64_t*>(smc_dyn);  // [P] local prefix sums (merge path)
  float* sX = reinterpret_cast<float*>(sA + P);           // [P] states
  int32_t* marks = reinterpret_cast<int32_t*>(sX + P);    // [kSmcOut] marks, zero between steps
  __shared__ int3 runs[kSmcRuns];  // long runs: first and last row, mark
  __shared__ int n_runs;
  __shared__ float sh_max[kSmcWarps];
  __shared__ int sh_nan[kSmcWarps];
  __shared__ float2 sh_s[kSmcWarps];
  __shared__ float j_max[kSmcWarps];
  __shared__ int j_nan[kSmcWarps];
  __shared__ float2 j_s[kSmcWarps], j_s2[kSmcWarps];
  __shared__ uint64_t sh_tot[kSmcWarps], j_tot[kSmcWarps];
  __shared__ double sh_z[kSmcWarps];
  __shared__ unsigned long long rel;
  __shared__ uint64_t view[6];  // T, stride, u, C at the block start, K_b, K_b+1
  __shared__ unsigned long long decision;  // bad << 33 | resample << 32 | bits of M
  __shared__ uint32_t resample_word;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned G = gridDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * P + (int64_t)tid * R;
  const int64_t N = a.N;
  SmcCtl* ctl = a.ctl;
  float x[R], lw[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    x[r] = 0.0f;
    lw[r] = 0.0f;
  }
  for (int j = tid; j < kSmcOut; j += kSmcTpb) marks[j] = 0;  // (a barrier follows before their use)
  int S = 0;
  while (((int64_t)1 << S) < N) ++S;
  const float scale = __int_as_float((127 + 61 - S) << 23);  // 2^(61 - ceil(log2 N))
  const float half_n = 0.5f * (float)N;                      // exact: N < 2^24
  const DivInv by_n = div_inv((uint64_t)N);
  unsigned long long e = 0;                                  // barriers passed
  float y_next = a.y[0];

  for (int t = 1; t <= a.T; ++t) {
    if (tid == 0) resample_word = philox_block(a.seed, 0, 0, (uint32_t)t, kResample, 0).x;
    const float yt = y_next;
    if (t < a.T) y_next = __ldg(a.y + t);  // in flight during this step
    // this step's half of the partials: a block may write step t + 1's
    // partial while slower blocks still read step t's, but not step t + 2's
    // (it has to pass barrier 1 of step t + 1 first, which they reach only
    // after reading)
    SmcPart* const parts_t = a.parts + (size_t)(t & 1) * G;
    int nan = 0;
    float tm = -INFINITY;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t i = i0 + r;
      if (i < N) {
        smc_propagate(a, (uint32_t)i, (uint32_t)t, yt, x[r], lw[r]);
        const float li = lw[r];
        nan |= (li != li);
        tm = fmaxf(tm, li);
      }
    }
    // block partial: the maximum (every warp reduces the 32 warp maxima), then
    // the sums around it (warp 0 adds the 32 warp sums)
    tm = warp_max(tm);
    nan = __any_sync(0xffffffffu, nan);
    if (lane == 0) {
      sh_max[warp] = tm;
      sh_nan[warp] = nan;
    }
    __syncthreads();
    const float bm = warp_max(sh_max[lane]);
    float ts = 0.0f, ts2 = 0.0f;
    if (bm > -INFINITY) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (i0 + r < N && lw[r] > -INFINITY) {
          const float ex = expf(lw[r] - bm);
          ts += ex;
          ts2 = fmaf(ex, ex, ts2);
        }
    }
    ts = warp_sum(ts);
    ts2 = warp_sum(ts2);
    if (lane == 0) sh_s[warp] = make_float2(ts, ts2);
    __syncthreads();
    if (warp == 0) {
      const float bs = warp_sum(sh_s[lane].x), bs2 = warp_sum(sh_s[lane].y);
      const int bn = __any_sync(0xffffffffu, sh_nan[lane]);
      if (lane == 0) {
        SmcPart q;
        q.m = bm;
        q.s = bs;
        q.s2 = bs2;
        q.nan = bn;
        *reinterpret_cast<float4*>(parts_t + blockIdx.x) = *reinterpret_cast<const float4*>(&q);
      }
    }
    // barrier 1, then every block merges all partials in the same fixed order
    // (thread b reads block b's): the maximum M, the sums around it as
    // double-float pairs, the NaN and empty checks and the decision
    if (!grid_sync<false>(&ctl->g, &ctl->status, G, ++e, &rel, [] { return 0ull; }, [] {})) return;
    {
      // (only the warps that hold partials: the others would take their issue
      // slots with sums of zeros)
      const bool holds = warp * 32 < (int)G;
      SmcPart q;
      q.m = -INFINITY;
      q.s = q.s2 = 0.0f;
      q.nan = 0;
      if ((unsigned)tid < G) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(parts_t + tid));
        q = *reinterpret_cast<const SmcPart*>(&v);
      }
      if (holds) {
        const float gm = warp_max(q.m);
        const int gn = __any_sync(0xffffffffu, q.nan);
        if (lane == 0) {
          j_max[warp] = gm;
          j_nan[warp] = gn;
        }
      }
      __syncthreads();
      const int n_hold = ((int)G + 31) / 32;
      const float M = warp_max(lane < n_hold ? j_max[lane] : -INFINITY);
      const int any_nan = __any_sync(0xffffffffu, lane < n_hold ? j_nan[lane] : 0);
      float2 Ss = make_float2(0.0f, 0.0f), Ss2 = make_float2(0.0f, 0.0f);
      if (holds) {
        if (M > -INFINITY && q.m > -INFINITY) {
          const float ex = expf(q.m - M);
          Ss = df_prod(q.s, ex);
          Ss2 = df_prod(q.s2, ex * ex);
        }
        Ss = df_warp_sum(Ss);
        Ss2 = df_warp_sum(Ss2);
        if (lane == 0) {
          j_s[warp] = Ss;
          j_s2[warp] = Ss2;
        }
      }
      __syncthreads();
      if (warp == 0) {
        const float2 zero = make_float2(0.0f, 0.0f);
        Ss = df_warp_sum(lane < n_hold ? j_s[lane] : zero);
        Ss2 = df_warp_sum(lane < n_hold ? j_s2[lane] : zero);
        if (lane == 0) {
          // ESS = S^2 / S2 < N / 2  <=>  S^2 - (N / 2) S2 < 0, in double-float
          const float2 lhs = df_mul(Ss, Ss), rhs = df_mul(make_float2(half_n, 0.0f), Ss2);
          const bool bad = any_nan || !(M > -INFINITY);
          const bool res =
              !bad && __fadd_rn(__fsub_rn(lhs.x, rhs.x), __fsub_rn(lhs.y, rhs.y)) < 0.0f;
          if (blockIdx.x == 0) {  // one block records the step
            if (any_nan) record_status(&ctl->status, PPL_ENAN);
            else if (bad) record_status(&ctl->status, PPL_EEMPTY);
            SmcStep st;
            st.M = M;
            st.s_hi = Ss.x;
            st.s_lo = Ss.y;
            st.s2_hi = Ss2.x;
            st.s2_lo = Ss2.y;
            st.flag = res ? 1 : 0;
            st.pad[0] = st.pad[1] = 0;
            a.stash[t - 1] = st;
          }
          decision = ((unsigned long long)bad << 33) | ((unsigned long long)res << 32) |
                     (unsigned long long)__float_as_uint(M);
        }
      }
      __syncthreads();
    }
    const unsigned long long r1 = decision;
    if ((r1 >> 33) & 1) return;  // a NaN or no finite weight: every block leaves
    if (!((r1 >> 32) & 1)) continue;
    const float M = __uint_as_float((uint32_t)r1);

    // 1. this thread's fixed-point weights and their sum, the states into shared
    // memory in particle order, then the block's exclusive scan
    uint64_t q[R], own = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      q[r] = i0 + r < N ? quantize(lw[r], M, scale) : 0ull;
      sX[tid * R + r] = x[r];
      own += q[r];
    }
    if (tid == 0) n_runs = 0;
    const uint64_t inc = warp_scan_plain(own, lane);
    if (lane == 31) sh_tot[warp] = inc;
    __syncthreads();
    uint64_t texcl, btot;
    {
      const uint64_t v = sh_tot[lane], wi = warp_scan_plain(v, lane);
      texcl = __shfl_sync(0xffffffffu, wi - v, warp) + (inc - own);
      btot = __shfl_sync(0xffffffffu, wi, 31);
    }
    if (tid == 0) a.bsum[blockIdx.x] = btot;
    // barrier 2, then every block scans the G block totals itself (the same
    // integer sums in every block): T, the stride floor(T / N), the systematic
    // offset u, and the first outputs whose ancestors this block and the next
    // hold, K_b = cnt(C at the block's start), where cnt(c) = #{k >= 0 : u + k
    // stride < c} (K_G = N)
    if (!grid_sync<false>(&ctl->g, &ctl->status, G, ++e, &rel, [] { return 0ull; }, [] {})) return;
    {
      const unsigned b = blockIdx.x;
      const int n_hold = ((int)G + 31) / 32;
      uint64_t v = 0, wi = 0;
      if (warp < n_hold) {
        v = (unsigned)tid < G ? __ldcg(a.bsum + tid) : 0ull;
        wi = warp_scan_plain(v, lane);
        if (lane == 31) j_tot[warp] = wi;
      }
      __syncthreads();
      if (warp == (int)(b >> 5) || warp == (int)((b + 1) >> 5)) {  // b + 1 <= G <= kSmcTpb
        const uint64_t jv = lane < n_hold ? j_tot[lane] : 0ull, ji = warp_scan_plain(jv, lane);
        const uint64_t ex = __shfl_sync(0xffffffffu, ji - jv, warp) + (wi - v);  // C at block tid's start
        const uint64_t T = __shfl_sync(0xffffffffu, ji, 31);
        const bool valid = T >= (uint64_t)N && T <= (1ull << 61);
        if ((unsigned)tid == b || (unsigned)tid == b + 1) {
          uint64_t stride = 0, u = 0;
          if (valid) {
            const uint64_t w0 = resample_word;
            stride = div_by(T, by_n);
            u = (__umul64hi(w0, stride) << 32) | ((w0 * stride) >> 32);
          }
          const uint64_t k = valid ? (uint64_t)positions_below(ex, u, stride, N) : 0ull;
          if ((unsigned)tid == b) {
            view[0] = T;
            view[1] = stride;
            view[2] = u;
            view[3] = ex;
            view[4] = k;
            if (b + 1 == G) view[5] = (uint64_t)N;
            if (b == 0 && !valid) record_status(&ctl->status, T == 0 ? PPL_EEMPTY : PPL_EINVAL);
          } else if (b + 1 < G) {
            view[5] = k;
          }
        }
      }
      __syncthreads();
    }
    const uint64_t T = view[0];
    if (T < (uint64_t)N || T > (1ull << 61)) return;  // every block sees the same T and leaves
    // 2. systematic resampling of this block's outputs k in [K_b, K_b+1), whose
    // ancestors a_k = min{j : C_j > u + k stride} are all in this block.
    // Particle j's offspring are the k with C_{j-1} <= u + k stride < C_j (one
    // small division per particle): it marks the first of them and, when they
    // run on, the first slot of every later row of 32 they reach, so that a
    // slot's ancestor is the last mark at or before it in its own row: one
    // ballot and one shuffle a row, and the states leave for global memory
    // coalesced.  (A merge path over the prefix sums and the positions took
    // 10K of a step's 45K cycles in dependent shared-memory loads; a loop over
    // each particle's offspring took twice that in divergent branches.)
    // A block with more outputs than its table takes the merge path below.
    const uint64_t stride = view[1], offset = view[2], cstart = view[3];
    const int64_t Kb = (int64_t)view[4], nB = (int64_t)view[5] - Kb;
    if (nB <= kSmcOut) {
      const int n = (int)nB;
      const StepDiv dv(offset + (uint64_t)Kb * stride, stride);
      {
        uint64_t c = cstart + texcl;
        int k0 = (int)min(dv.below(c), (uint32_t)n);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          c += q[r];
          const int k1 = (int)min(dv.below(c), (uint32_t)n);
          if (k1 > k0) {
            marks[k0] = tid * R + r + 1;
            const int first_row = k0 / 32 + 1, last_row = (k1 - 1) / 32;
            if (last_row - first_row < kSmcShort) {
              for (int row = first_row; row <= last_row; ++row) marks[row * 32] = tid * R + r + 1;
            } else {  // a long run: left to the block
              const int at = atomicAdd(&n_runs, 1);
              if (at < kSmcRuns) runs[at] = make_int3(first_row, last_row, tid * R + r + 1);
              else
                for (int row = first_row; row <= last_row; ++row) marks[row * 32] = tid * R + r + 1;
            }
          }
          k0 = k1;
        }
      }
      __syncthreads();
      if (n_runs > 0) {  // the same for the whole block
        const int nr = min(n_runs, kSmcRuns);
        for (int e = warp; e < nr; e += kSmcWarps) {
          const int3 w = runs[e];
          for (int row = w.x + lane; row <= w.y; row += 32) marks[row * 32] = w.z;
        }
        __syncthreads();
      }
      const int n_rows = (n + 31) / 32;
      for (int row = warp; row < n_rows; row += kSmcWarps) {
        const int j = row * 32 + lane;
        const int mk = marks[j];
        marks[j] = 0;
        const unsigned at = __ballot_sync(0xffffffffu, mk != 0);
        const int an = __shfl_sync(0xffffffffu, mk, 31 - __clz(at & (0xffffffffu >> (31 - lane))));
        if (j < n) a.xbuf[Kb + j] = sX[an - 1];
      }
    } else {
      // with A_i the block-local inclusive prefix sums and B_j = u + (K_b + j)
      // stride - C_start, a_k is the number of A's not above B_j, i.e. B_j's
      // place in the merge of the two sorted lists (ties: A first).  The merge
      // is cut into equal slices, one per thread (merge path: Green, McColl,
      // Bader, "GPU merge path", ICS 2012).
      uint64_t run = texcl;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        run += q[r];
        sA[tid * R + r] = run;
      }
      __syncthreads();
      const int nA = (int)P, nBi = (int)nB;
      const int64_t L = (int64_t)nA + nB;
      const int d0 = (int)(L * tid / kSmcTpb), d1 = (int)(L * (tid + 1) / kSmcTpb);
      // B_j relative to the block start (>= 0: the outputs from K_b on lie at or past it)
      const uint64_t b0 = offset + (uint64_t)Kb * stride - cstart;
      int lo = d0 > nBi ? d0 - nBi : 0, hi = d0 < nA ? d0 : nA;
      while (lo < hi) {  // the A's among the first d0 merged items
        const int mid = (lo + hi) >> 1;
        if (sA[mid] <= b0 + (uint64_t)(d0 - 1 - mid) * stride) lo = mid + 1;
        else hi = mid;
      }
      int i = lo, j = d0 - lo;
      uint64_t bj = b0 + (uint64_t)j * stride;
      uint64_t ai = i < nA ? sA[i] : ~0ull;
      for (int s = d0; s < d1; ++s) {
        if (j >= nBi || ai <= bj) {
          ++i;
          ai = i < nA ? sA[i] : ~0ull;
        } else {  // output K_b + j: ancestor i (A_i > B_j, so i < nA)
          a.xbuf[Kb + j] = sX[i < nA ? i : nA - 1];
          ++j;
          bj += stride;
        }
      }
    }
    if (!grid_sync<false>(&ctl->g, &ctl->status, G, ++e, &rel, [] { return 0ull; }, [] {})) return;
    // 3. the new population: this thread's outputs are i0 .. i0 + R - 1
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (i0 + r < N) x[r] = __ldcg(a.xbuf + i0 + r);
      lw[r] = 0.0f;
    }
  }
  if (blockIdx.x == 0) smc_outputs(a, sh_z);
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (i0 + r < N) {
      a.x_out[i0 + r] = x[r];
      a.lw_out[i0 + r] = lw[r];
    }
}

// ---------------------------------------------------------------------------
// The same filter for populations that one thread-block cluster holds.  A step
// of a small filter is all latency: the grid barriers go through L2 (about
// 2.3 us each, two or three a step), and so do the partials, totals and states
// between them.  In a cluster the barrier is the hardware's, and blocks push
// their partials, totals and resampled states straight into the shared memory
// of the blocks that read them (distributed shared memory), so every read
// after a barrier is local, and every warp merges the partials by itself
// without a block barrier.  10^4 particles x 100 steps: 939 us on grid
// barriers, 410 us in a cluster of 10.
//
// Block b of the cluster stands for the V blocks b V .. b V + V - 1 of 1024
// particles that smc_persistent_kernel<1> would run, thread tid holding
// particle tid of each: the partials of each are formed and merged in that
// kernel's order, so that both give the same bits (its R is 1 up to 1024
// particles per SM, more than a cluster holds).
// ---------------------------------------------------------------------------
constexpr int kClMaxBlocks = 16;  // blocks of a cluster (8 where 16 do not fit)
// Largest population run in one cluster, two virtual blocks per block: 32768
// particles x 100 steps take 627 us so and 755 us on grid barriers (16384: 442
// and 750); with four per block (65536) the cluster was the slower one, 1217
// against 870 us, its 16 SMs then bound by the propagation.
constexpr int64_t kClMaxParticles = 32768;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// The address of this block's shared variable in block `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(r)
      : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}

template <int V>
__global__ void __launch_bounds__(kSmcTpb, 1) smc_cluster_kernel(SmcArgs a) {
  constexpr int kParts = kClMaxBlocks * V;
  __shared__ __align__(16) SmcPart parts[2][kParts];  // by step parity, as in the grid version
  __shared__ uint64_t tots[kClMaxBlocks];             // blocks' sums of fixed-point weights
  // this block's resampled states, and whether the slot was written (0 between steps)
  __shared__ __align__(8) int2 slots[V * kSmcTpb];
  __shared__ float sh_max[V][kSmcWarps];
  __shared__ int sh_nan[V][kSmcWarps];
  __shared__ float2 sh_s[V][kSmcWarps];
  __shared__ uint64_t wtot[V][kSmcWarps];
  __shared__ double sh_z[kSmcWarps];
  __shared__ uint32_t resample_word;
  __shared__ unsigned long long decision;  // bad << 33 | resample << 32 | bits of M
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int CS = (int)gridDim.x, rank = (int)blockIdx.x;  // the grid is one cluster
  const int N = (int)a.N;
  const int Gv = (N + kSmcTpb - 1) / kSmcTpb;  // virtual blocks that hold particles
  const int i0 = rank * V * kSmcTpb + tid;     // particle of register r: i0 + 1024 r
  int32_t* status = &a.ctl->status;
  int S = 0;
  while (((int64_t)1 << S) < a.N) ++S;
  const float scale = __int_as_float((127 + 61 - S) << 23);  // 2^(61 - ceil(log2 N))
  const float half_n = 0.5f * (float)N;
  const DivInv by_n = div_inv((uint64_t)N);
  float x[V], lw[V];
#pragma unroll
  for (int r = 0; r < V; ++r) {
    x[r] = lw[r] = 0.0f;
    slots[r * kSmcTpb + tid].y = 0;
  }
  float y_next = a.y[0];
  cluster_sync();  // every block of the cluster runs before any remote store

  for (int t = 1; t <= a.T; ++t) {
    if (tid == kSmcTpb - 1) resample_word = philox_block(a.seed, 0, 0, (uint32_t)t, kResample, 0).x;
    const float yt = y_next;
    if (t < a.T) y_next = __ldg(a.y + t);
    SmcPart* const parts_t = parts[t & 1];
    // every virtual block's partial, in smc_persistent_kernel's order
#pragma unroll
    for (int r = 0; r < V; ++r) {
      const int i = i0 + r * kSmcTpb;
      int nan = 0;
      float tm = -INFINITY;
      if (i < N) {
        smc_propagate(a, (uint32_t)i, (uint32_t)t, yt, x[r], lw[r]);
        nan = lw[r] != lw[r];
        tm = fmaxf(tm, lw[r]);
      }
      tm = warp_max(tm);
      nan = __any_sync(0xffffffffu, nan);
      if (lane == 0) {
        sh_max[r][warp] = tm;
        sh_nan[r][warp] = nan;
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < V; ++r) {
      const float bm = warp_max(sh_max[r][lane]);
      float ts = 0.0f, ts2 = 0.0f;
      if (bm > -INFINITY && i0 + r * kSmcTpb < N && lw[r] > -INFINITY) {
        const float ex = expf(lw[r] - bm);
        ts += ex;
        ts2 = fmaf(ex, ex, ts2);
      }
      ts = warp_sum(ts);
      ts2 = warp_sum(ts2);
      if (lane == 0) sh_s[r][warp] = make_float2(ts, ts2);
    }
    __syncthreads();
    if (warp < V && rank * V + warp < Gv) {
      const float bm = warp_max(sh_max[warp][lane]);
      const float bs = warp_sum(sh_s[warp][lane].x), bs2 = warp_sum(sh_s[warp][lane].y);
      const int bn = __any_sync(0xffffffffu, sh_nan[warp][lane]);
      if (lane < CS)
        asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                         cluster_addr(parts_t + rank * V + warp, lane)),
                     "r"(__float_as_int(bm)), "r"(__float_as_int(bs)), "r"(__float_as_int(bs2)),
                     "r"(bn)
                     : "memory");
    }
    // barrier 1, then warp 0 merges all partials in the grid version's order (32
    // at a time across lanes, then those sums).  (All 32 warps doing it saves a
    // block barrier, but fills the issue slots with 32 copies of it.)
    cluster_sync();
    if (warp == 0) {
      constexpr int kG = (kParts + 31) / 32;
      static_assert(kG <= 2, "two groups of 32 partials at most");
      float M = -INFINITY;
      int any_nan = 0;
      SmcPart q[kG];
#pragma unroll
      for (int g = 0; g < kG; ++g) {
        q[g].m = -INFINITY;
        q[g].s = q[g].s2 = 0.0f;
        q[g].nan = 0;
        if (g * 32 + lane < Gv) q[g] = parts_t[g * 32 + lane];
        M = fmaxf(M, q[g].m);
        any_nan |= q[g].nan;
      }
      M = warp_max(M);
      any_nan = __any_sync(0xffffffffu, any_nan);
      float2 Ss = make_float2(0.0f, 0.0f), Ss2 = Ss;
#pragma unroll
      for (int g = 0; g < kG; ++g) {
        float2 gs = make_float2(0.0f, 0.0f), gs2 = gs;
        if (M > -INFINITY && q[g].m > -INFINITY) {
          const float ex = expf(q[g].m - M);
          gs = df_prod(q[g].s, ex);
          gs2 = df_prod(q[g].s2, ex * ex);
        }
        Ss = df_add(Ss, df_warp_sum(gs));
        Ss2 = df_add(Ss2, df_warp_sum(gs2));
      }
      if (lane == 0) {
        // ESS = S^2 / S2 < N / 2  <=>  S^2 - (N / 2) S2 < 0, in double-float
        const float2 lhs = df_mul(Ss, Ss), rhs = df_mul(make_float2(half_n, 0.0f), Ss2);
        const bool bad = any_nan || !(M > -INFINITY);
        const bool res = !bad && __fadd_rn(__fsub_rn(lhs.x, rhs.x), __fsub_rn(lhs.y, rhs.y)) < 0.0f;
        if (rank == 0) {  // one block records the step
          if (any_nan) record_status(status, PPL_ENAN);
          else if (bad) record_status(status, PPL_EEMPTY);
          a.stash[t - 1] = SmcStep{M, Ss.x, Ss.y, Ss2.x, Ss2.y, res ? 1 : 0, {0, 0}};
        }
        decision = ((unsigned long long)bad << 33) | ((unsigned long long)res << 32) |
                   (unsigned long long)__float_as_uint(M);
      }
    }
    __syncthreads();
    const unsigned long long r1 = decision;
    if ((r1 >> 33) & 1) return;  // the same in every thread of the cluster; no remote access is under way
    if (!((r1 >> 32) & 1)) continue;
    const float M = __uint_as_float((uint32_t)r1);

    // fixed-point weights and the block's sums in particle order (register by
    // register, warp by warp)
    uint64_t inc[V];
#pragma unroll
    for (int r = 0; r < V; ++r) {
      inc[r] = warp_scan_plain(i0 + r * kSmcTpb < N ? quantize(lw[r], M, scale) : 0ull, lane);
      if (lane == 31) wtot[r][warp] = inc[r];
    }
    __syncthreads();
    uint64_t btot = 0, wbase[V];  // the block's sum; the sum before each of the warp's rows
#pragma unroll
    for (int r = 0; r < V; ++r) {
      const uint64_t v = wtot[r][lane], wi = warp_scan_plain(v, lane);
      wbase[r] = btot + __shfl_sync(0xffffffffu, wi - v, warp);
      inc[r] += wbase[r];
      btot += __shfl_sync(0xffffffffu, wi, 31);
    }
    if (warp == 0 && lane < CS)
      asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(cluster_addr(tots + rank, lane)),
                   "l"(btot)
                   : "memory");
    // barrier 2, then every warp scans the blocks' totals
    cluster_sync();
    const uint64_t tv = lane < CS ? tots[lane] : 0ull;
    const uint64_t ti = warp_scan_plain(tv, lane);
    const uint64_t cstart = __shfl_sync(0xffffffffu, ti - tv, rank);
    const uint64_t T = __shfl_sync(0xffffffffu, ti, 31);
    if (T < (uint64_t)N || T > (1ull << 61)) {
      if (rank == 0 && tid == 0) record_status(status, T == 0 ? PPL_EEMPTY : PPL_EINVAL);
      return;  // the same in every thread of the cluster
    }
    const uint64_t stride = div_by(T, by_n), w0 = resample_word;
    const uint64_t u = (__umul64hi(w0, stride) << 32) | ((w0 * stride) >> 32);
    const StepDiv dv(u, stride);
    // particle j's offspring are the outputs k with C_{j-1} <= u + k stride <
    // C_j: its state goes to the first of their slots, in the shared memory of
    // the block that holds it, and to the first slot of every later row of 32
    // that they reach, so that a row's other slots are filled from within it
#pragma unroll
    for (int r = 0; r < V; ++r) {
      const uint64_t c1 = cstart + inc[r];
      const int ke = (int)min(dv.below(c1), (uint32_t)N);
      int ks = __shfl_up_sync(0xffffffffu, ke, 1);
      if (lane == 0) ks = (int)min(dv.below(cstart + wbase[r]), (uint32_t)N);
      auto put = [&](int k, float v) {
        const int to = k / (V * kSmcTpb);
        asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(
                         cluster_addr(slots + (k - to * V * kSmcTpb), to)),
                     "r"(__float_as_int(v)), "r"(1)
                     : "memory");
      };
      const int row0 = ks / 32 + 1, row1 = ke > ks ? (ke - 1) / 32 : -1;
      if (ke > ks) put(ks, x[r]);
      const bool longr = row1 - row0 >= kSmcShort;
      if (!longr)
        for (int row = row0; row <= row1; ++row) put(row * 32, x[r]);
      unsigned lm = __ballot_sync(0xffffffffu, longr);
      while (lm) {
        const int src = __ffs(lm) - 1;
        lm &= lm - 1;
        const int s0 = __shfl_sync(0xffffffffu, row0, src), s1 = __shfl_sync(0xffffffffu, row1, src);
        const float v = __shfl_sync(0xffffffffu, x[r], src);
        for (int row = s0 + lane; row <= s1; row += 32) put(row * 32, v);
      }
    }
    // barrier 3, then the new population
    cluster_sync();
#pragma unroll
    for (int r = 0; r < V; ++r) {
      const int2 sl = slots[r * kSmcTpb + tid];
      slots[r * kSmcTpb + tid].y = 0;
      const unsigned at = __ballot_sync(0xffffffffu, sl.y != 0) & (0xffffffffu >> (31 - lane));
      x[r] = __int_as_float(__shfl_sync(0xffffffffu, sl.x, at ? 31 - __clz(at) : lane));
      lw[r] = 0.0f;
    }
  }
  __syncthreads();  // the last step's record
  if (rank == 0) smc_outputs(a, sh_z);
#pragma unroll
  for (int r = 0; r < V; ++r)
    if (i0 + r * kSmcTpb < N) {
      a.x_out[i0 + r * kSmcTpb] = x[r];
      a.lw_out[i0 + r * kSmcTpb] = lw[r];
    }
}

// The filter's grid barriers with nothing between them: what the step
// separators alone cost at the filter's launch shape.
__global__ void __launch_bounds__(kSmcTpb) grid_barrier_probe_kernel(SmcCtl* ctl, int n) {
  __shared__ unsigned long long rel;
  for (int e = 1; e <= n; ++e)
    if (!grid_sync<false>(&ctl->g, &ctl->status, gridDim.x, (unsigned long long)e, &rel,
                          [] { return 0ull; }, [] {}))
      return;
}

cudaError_t launch_grid_barrier_probe(int blocks, int n_barriers, void* ws, cudaStream_t s) {
  SmcCtl* ctl = static_cast<SmcCtl*>(ws);
  cudaError_t e = cudaMemsetAsync(ctl, 0, sizeof(SmcCtl), s);
  if (e != cudaSuccess) return e;
  void* args[] = {&ctl, &n_barriers};
  return cudaLaunchCooperativeKernel((const void*)grid_barrier_probe_kernel, dim3((unsigned)blocks),
                                     dim3(kSmcTpb), args, 0, s);
}

size_t smc_run_workspace(int64_t N, int64_t T) {
  return 8 * 256 + (size_t)kSmcMaxGrid * (2 * sizeof(SmcPart) + 8) +
         (size_t)std::max<int64_t>(T, 0) * sizeof(SmcStep) + (size_t)N * 4;
}

template <int R>
static cudaError_t launch_r(SmcArgs& a, cudaStream_t s, bool* fits) {
  const int64_t grid = (a.N + (int64_t)kSmcTpb * R - 1) / ((int64_t)kSmcTpb * R);
  constexpr size_t dyn = (size_t)R * kSmcTpb * (8 + 4) + (size_t)kSmcOut * 4;
  cudaError_t e = cudaFuncSetAttribute(smc_persistent_kernel<R>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, smc_persistent_kernel<R>, kSmcTpb,
                                                    dyn);
  if (e != cudaSuccess) return e;
  *fits = grid <= std::min<int64_t>((int64_t)num_sms() * per_sm, kSmcMaxGrid);
  if (!*fits) return cudaSuccess;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)smc_persistent_kernel<R>, dim3((unsigned)grid),
                                     dim3(kSmcTpb), args, dyn, s);
}

// One cluster that holds the population, if a cluster of that size can run
// here (asked once per device); *fits false otherwise.
template <int V>
static cudaError_t launch_cluster(SmcArgs& a, cudaStream_t s, bool* fits) {
  const int64_t need = (a.N + (int64_t)kSmcTpb * V - 1) / ((int64_t)kSmcTpb * V);
  *fits = false;
  const void* fn = (const void*)smc_cluster_kernel<V>;
  auto config = [&](int blocks, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)blocks);
    c.blockDim = dim3(kSmcTpb);
    c.stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)blocks;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    c.attrs = at;
    c.numAttrs = 1;
    return c;
  };
  int most = 0;  // blocks of the largest cluster
  const cudaError_t e = device_once(fn, &most, [&](int* v) {
    cudaError_t r = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (r != cudaSuccess) return r;
    for (int b = kClMaxBlocks; b >= 8 && *v == 0; b /= 2) {
      cudaLaunchAttribute at;
      cudaLaunchConfig_t c = config(b, &at);
      int n = 0;
      r = cudaOccupancyMaxActiveClusters(&n, fn, &c);
      if (r != cudaSuccess) {
        (void)cudaGetLastError();  // this size is not offered: ask for the next
        continue;
      }
      if (n > 0) *v = b;
    }
    return cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  if (need > most) return cudaSuccess;
  *fits = true;
  cudaLaunchAttribute at;
  cudaLaunchConfig_t c = config((int)need, &at);
  void* args[] = {&a};
  return cudaLaunchKernelExC(&c, fn, args);
}

cudaError_t launch_smc_persistent(const LgssmParams& p, const float* y, int32_t T, uint64_t seed,
                                  int64_t N, float* x_out, float* lw_out, double* logz,
                                  int32_t* resampled, double* ess, char* ws, size_t ws_bytes,
                                  int32_t** status_out, cudaStream_t s) {
  if (T < 1 || T > (1 << 27)) return cudaErrorInvalidValue;  // barrier numbers fit 30 bits
  SmcArgs a;
  a.p = p;
  a.y = y;
  a.T = T;
  a.seed = seed;
  a.N = N;
  a.x_out = x_out;
  a.lw_out = lw_out;
  a.logz = logz;
  a.resampled = resampled;
  a.ess = ess;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* q = ws + off;
    off += (bytes + 255) / 256 * 256;
    return q;
  };
  a.ctl = reinterpret_cast<SmcCtl*>(take(sizeof(SmcCtl)));
  a.parts = reinterpret_cast<SmcPart*>(take(2 * (size_t)kSmcMaxGrid * sizeof(SmcPart)));
  a.bsum = reinterpret_cast<uint64_t*>(take((size_t)kSmcMaxGrid * 8));
  a.stash = reinterpret_cast<SmcStep*>(take((size_t)T * sizeof(SmcStep)));
  a.xbuf = reinterpret_cast<float*>(take((size_t)N * 4));
  if (off > ws_bytes) return cudaErrorInvalidValue;
  *status_out = &a.ctl->status;
  cudaError_t e = cudaMemsetAsync(a.ctl, 0, sizeof(SmcCtl), s);
  if (e != cudaSuccess) return e;
  bool fits = false;
  if (N <= kClMaxParticles) {
    if ((e = launch_cluster<1>(a, s, &fits)) != cudaSuccess || fits) return e;
    if ((e = launch_cluster<2>(a, s, &fits)) != cudaSuccess || fits) return e;
  }
  // fewest particles per thread whose grid is resident at once
  if ((e = launch_r<1>(a, s, &fits)) != cudaSuccess || fits) return e;
  if ((e = launch_r<2>(a, s, &fits)) != cudaSuccess || fits) return e;
  if ((e = launch_r<3>(a, s, &fits)) != cudaSuccess || fits) return e;
  if ((e = launch_r<4>(a, s, &fits)) != cudaSuccess || fits) return e;
  if ((e = launch_r<5>(a, s, &fits)) != cudaSuccess || fits) return e;
  if ((e = launch_r<6>(a, s, &fits)) != cudaSuccess || fits) return e;
  if ((e = launch_r<7>(a, s, &fits)) != cudaSuccess || fits) return e;
  if ((e = launch_r<8>(a, s, &fits)) != cudaSuccess || fits) return e;
  return cudaErrorInvalidValue;  // more particles than resident threads can hold
}

}  // namespace ppl
