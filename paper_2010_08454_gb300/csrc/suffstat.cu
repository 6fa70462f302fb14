// Likelihood weighting with the factor from the data's sufficient statistics
// (suffstat.cuh): the statistics of a data set (power sums in FP64 over the
// points, one read of the data, then the Cholesky factor of the 6 x 6 Gram
// matrix, the forward substitution and the per-degree distances), and the
// pass over the traces.
#include "kernels.h"
#include "suffstat.cuh"
#include "trace.cuh"

namespace ppl {

constexpr int kSsPow = 2 * kMaxCoef - 1;  // x^0 .. x^10
constexpr int kSsGroups = 14;             // partial sums of a total (18 totals x 14 threads)

__global__ void __launch_bounds__(kTpb) suffstat_kernel(const float* __restrict__ xs,
                                                        const float* __restrict__ ys, int64_t L,
                                                        int d_max, SuffStat* out) {
  constexpr int V = kSsPow + kMaxCoef + 1;  // sum x^k, sum x^k y, sum y^2
  __shared__ double part[V][kTpb], red[V][kSsGroups];
  double acc[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc[v] = 0.0;
  for (int64_t l = threadIdx.x; l < L; l += kTpb) {
    const double x = xs[l], y = ys[l];
    double pw = 1.0;
#pragma unroll
    for (int k = 0; k < kSsPow; ++k) {
      acc[k] += pw;
      if (k < kMaxCoef) acc[kSsPow + k] += pw * y;
      pw *= x;
    }
    acc[V - 1] += y * y;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the block's sums through shared memory, each addition once (butterflies
  // over the lanes do every addition 32 times over, on an FP64 pipe of two
  // lanes a clock: 6 us of them)
#pragma unroll
  for (int v = 0; v < V; ++v) part[v][threadIdx.x] = acc[v];
  __syncthreads();
  if (threadIdx.x < V * kSsGroups) {
    const int v = threadIdx.x / kSsGroups, g = threadIdx.x % kSsGroups;
    double a = 0.0;
    for (int t = g; t < kTpb; t += kSsGroups) a += part[v][t];
    red[v][g] = a;
  }
  __syncthreads();
  if (warp != 0) return;
  double tot = 0.0;  // lane v's sum
  if (lane < V)
    for (int g = 0; g < kSsGroups; ++g) tot += red[lane][g];
  // Cholesky G = R^T R of the leading d_max x d_max block (G_ij = sum
  // x^(i+j)) by rows, lane j the column j and lane 6 the right-hand side Phi^T
  // y, whose column becomes w = R^-T Phi^T y: a row is one reciprocal square
  // root and one broadcast.  (One thread's divisions and square roots in
  // turn took 33 us; 12 us so, with the sums above.)
  double col[kMaxCoef];  // R[i][j], i <= j; w[i] in lane 6
  const int j = lane;
  int ok = 1;
#pragma unroll
  for (int i = 0; i < kMaxCoef; ++i) {
    const double gij = __shfl_sync(0xffffffffu, tot, j < kMaxCoef ? i + j : (j == kMaxCoef ? kSsPow + i : 0));
    const double gii = __shfl_sync(0xffffffffu, tot, 2 * i);
    double v = gij;
#pragma unroll
    for (int k = 0; k < i; ++k) v -= __shfl_sync(0xffffffffu, col[k], i) * col[k];
    const double pivot = __shfl_sync(0xffffffffu, v, i);
    // a pivot that lost all but ~8 digits of the diagonal marks G singular for FP32 use
    if (i < d_max && !(pivot > 1e-8 * gii)) ok = 0;
    const bool use = ok && i < d_max && (j == kMaxCoef || (j >= i && j < d_max));
    col[i] = use ? v * rsqrt(pivot) : 0.0;
  }
  // a failed factorisation leaves the statistics unused (ok = 0)
  double base = __shfl_sync(0xffffffffu, tot, V - 1);
  if (lane < kMaxCoef)
#pragma unroll
    for (int i = 0; i < kMaxCoef; ++i) out->R[i][lane] = (float)col[i];
  if (lane == kMaxCoef) {
    out->base[0] = (float)base;
#pragma unroll
    for (int i = 0; i < kMaxCoef; ++i) {
      out->w[i] = (float)col[i];
      base -= col[i] * col[i];
      out->base[i + 1] = (float)(base > 0.0 ? base : 0.0);
    }
    out->ok = ok;
    out->pad[0] = out->pad[1] = 0;
  }
}

// ---------------------------------------------------------------------------
// The pass over the traces.  The factor is a few dozen multiply-adds, so the
// pass is bound by the issue of the draws (two Philox blocks, three Box-Muller
// pairs: about 300 of its instructions a trace).  Nothing in it depends on
// the degree but a mask, so the degree sort, shared-memory round trip and
// block barriers of the point-by-point kernel are left out: every thread
// draws, evaluates and writes its own traces, two at a time (their chains
// overlap), and the warps fold on their own.  R and w stay in registers.
// 2^24 traces: 364 us in the point-by-point kernel's frame (528 instructions a
// trace), 231 us so (375 instructions); three blocks per SM spill (270 us), four
// traces at a time or one are slower (255, 244).
// ---------------------------------------------------------------------------
constexpr int kSsU = 2;  // traces of a thread at a time
constexpr int kSsBlocksPerSm = 2;

__global__ void __launch_bounds__(kTpb, kSsBlocksPerSm) suffstat_trace_kernel(
    PolyParams p, const SuffStat* __restrict__ stat, int64_t N, uint64_t seed, uint32_t instance,
    float* __restrict__ lw_out, ppl_poly_particle* __restrict__ rec_out, WsHeader* hdr,
    DegPartial* parts, ppl_is_result* res) {
  if (!stat->ok) return;  // the point-by-point kernel runs instead
  __shared__ DegPartial wrun[(kTpb / 32) * kMaxDegrees];
  __shared__ float sbase[kMaxCoef + 1];
  __shared__ int any_nan;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < (kTpb / 32) * kMaxDegrees) deg_empty(wrun[tid]);
  if (tid <= kMaxCoef) sbase[tid] = stat->base[tid];
  if (tid == 0) any_nan = 0;
  SuffStat st;
#pragma unroll
  for (int i = 0; i < kMaxCoef; ++i) {
    st.w[i] = stat->w[i];
#pragma unroll
    for (int j = 0; j < kMaxCoef; ++j) st.R[i][j] = j >= i ? stat->R[i][j] : 0.0f;
  }
  __syncthreads();
  DegPartial* wr = wrun + warp * kMaxDegrees;
  const bool rec_v8 = (reinterpret_cast<uintptr_t>(rec_out) & 31) == 0;
  int nan = 0;
  const int64_t step = (int64_t)gridDim.x * kTpb * kSsU;
  // a warp takes 32 kSsU consecutive traces
  for (int64_t i0 = ((int64_t)blockIdx.x * kTpb + warp * 32) * kSsU; i0 < N; i0 += step) {
    float c[kSsU][kMaxCoef], lw[kSsU];
    int d[kSsU];
    bool cand = false;
#pragma unroll
    for (int u = 0; u < kSsU; ++u) {
      const int64_t i = i0 + u * 32 + lane;
      const bool in = i < N;
      const int n = poly_draw(p, seed, instance, (uint32_t)i, c[u]);
      if (in && rec_out) {
        if (rec_v8) {
          st_global_v8(rec_out + i, c[u][0], c[u][1], c[u][2], c[u][3], c[u][4], c[u][5],
                       __int_as_float(n), __uint_as_float((uint32_t)i));
        } else {
          float4* dst = reinterpret_cast<float4*>(rec_out + i);
          dst[0] = make_float4(c[u][0], c[u][1], c[u][2], c[u][3]);
          dst[1] = make_float4(c[u][4], c[u][5], __int_as_float(n), __uint_as_float((uint32_t)i));
        }
      }
      lw[u] = suff_residual(st, sbase, c[u], n + p.coef_offset) * p.neg_half_inv_var;
      if (in && lw_out) lw_out[i] = lw[u];
      d[u] = in ? n - p.min_deg : -1;
      cand |= in && !(lw[u] <= wr[in ? d[u] : 0].m - kSkipNats);  // a NaN too
    }
    if (__any_sync(0xffffffffu, cand)) {
#pragma unroll
      for (int u = 0; u < kSsU; ++u)
        fold_warp(wr, lw[u], d[u], (int)(i0 + u * 32 + lane), c[u], lane, nan);
    }
  }
  if (__any_sync(0xffffffffu, nan) && lane == 0) any_nan = 1;
  __syncthreads();
  // merge the warps' partials: warp d merges degree d over the block's 8 warps
  if (warp < kMaxDegrees) {
    DegPartial q;
    deg_empty(q);
    if (lane < kTpb / 32) q = wrun[lane * kMaxDegrees + warp];
#pragma unroll 1
    for (int o = 1; o < kTpb / 32; o <<= 1) {
      const DegPartial other = deg_shfl_xor(q, o);
      deg_merge(q, other);
    }
    if (lane == 0) parts[blockIdx.x * kMaxDegrees + warp] = q;
  }
  if (tid == 0 && any_nan) record_status(&hdr->status, PPL_ENAN);
  if (elect_last_block(&hdr->ticket[0]))
    finalize_partials(parts, gridDim.x, p.n_deg, p.min_deg, N, hdr, res);
}

size_t suffstat_bytes() { return sizeof(SuffStat); }

cudaError_t launch_suffstat(const float* x, const float* y, int64_t L, int d_max, void* out,
                            cudaStream_t s) {
  if (d_max < 1 || d_max > kMaxCoef) return cudaErrorInvalidValue;
  suffstat_kernel<<<1, kTpb, 0, s>>>(x, y, L, d_max, reinterpret_cast<SuffStat*>(out));
  return cudaGetLastError();
}

cudaError_t launch_suffstat_trace(const PolyParams& p, const void* stat, int64_t N, uint64_t seed,
                                  uint32_t instance, float* lw_out, ppl_poly_particle* rec_out,
                                  WsHeader* hdr, void* parts, ppl_is_result* res, cudaStream_t s) {
  const int64_t blocks = (N + (int64_t)kTpb * kSsU - 1) / ((int64_t)kTpb * kSsU);
  const int grid = (int)std::max<int64_t>(
      1, std::min<int64_t>(blocks, (int64_t)num_sms() * kSsBlocksPerSm));
  suffstat_trace_kernel<<<grid, kTpb, 0, s>>>(p, (const SuffStat*)stat, N, seed, instance, lw_out,
                                              rec_out, hdr, (DegPartial*)parts, res);
  return cudaGetLastError();
}

}  // namespace ppl
