// Likelihood weighting (§3.6.2) on many independent line-fitting data sets of
// uneven size in one persistent launch.
//
// Work items are (instance, particle tile) pairs.  The host plan orders them
// heaviest first (by data length, the per-trace cost) so the persistent blocks,
// which take items from an atomic queue, end together (longest-processing-time
// order).  Each item reduces its traces to per-degree partials; the last item of
// an instance to finish merges that instance's partials into its summary.  The
// launch itself only clears counters and starts one kernel, so it can be
// captured in a CUDA graph and replayed.  The autotuner picks the traces per
// thread and the resident blocks per SM by timing the candidates, and caches
// the choice in a JSON file.  Large batches of short data sets run in a kernel
// of their own (lanes_kernel).
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <numeric>
#include <string>
#include <vector>

#include "kernels.h"
#include "lanesums.cuh"
#include "learned.cuh"
#include "posterior.cuh"
#include "trace.cuh"

namespace ppl {

struct BatchItem {
  int32_t inst;
  int32_t tile;
};

// Workspace layout of a prepared plan (offsets from the workspace base).
struct BatchLayout {
  size_t header, items, first, count_tmpl, count, inst_max, parts, total;
};

static size_t align256(size_t v) { return (v + 255) / 256 * 256; }

constexpr int kWarpParts = (kTpb / 32) * kMaxDegrees;  // partials one tile leaves

static BatchLayout batch_layout(int64_t n_items, int32_t n_inst) {
  BatchLayout l;
  size_t off = 0;
  l.header = off;
  off += 512;
  l.items = off;
  off += align256((size_t)n_items * sizeof(BatchItem));
  l.first = off;
  off += align256((size_t)n_inst * sizeof(int32_t));
  l.count_tmpl = off;
  off += align256((size_t)n_inst * sizeof(int32_t));
  l.count = off;
  off += align256((size_t)n_inst * sizeof(int32_t));
  l.inst_max = off;
  off += align256((size_t)n_inst * kMaxDegrees * sizeof(int32_t));
  l.parts = off;
  off += align256((size_t)n_items * kWarpParts * sizeof(DegPartial));
  l.total = off;
  return l;
}

// The summary of an instance from its `tiles` tiles' partials, by one block.
__device__ __forceinline__ void finish_instance(const PolyParams& p, const DegPartial* parts,
                                                int64_t tiles, int64_t N, WsHeader* hdr,
                                                ppl_is_result* out) {
  __shared__ DegPartial fin[kMaxDegrees];
  __shared__ float2 fS[kMaxDegrees], fS2[kMaxDegrees];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < kMaxDegrees)  // (tile, warp) partials of degree `warp`
    merge_degree(parts, (int)(tiles * (kTpb / 32)), warp, lane, fin + warp, fS + warp, fS2 + warp);
  __syncthreads();
  if (warp == 0)
    write_summary_warp(fin, fS, fS2, p.n_deg, p.min_deg, N,
                       lane == 0 ? ld_volatile_i32(&hdr->status) : 0, out);
  __syncthreads();
}

constexpr int kBatchChunk = 4096;  // data points staged in shared memory at a time

template <int PPT, bool LEARNED>
__global__ void __launch_bounds__(kTpb, PPT >= 8 ? 2 : (LEARNED ? 3 : 4)) batched_kernel(
    PolyParams p, const float* __restrict__ xs, const float* __restrict__ ys,
    const int64_t* __restrict__ data_off, const int64_t* __restrict__ part_off,
    const BatchItem* __restrict__ items, int64_t n_items, const int32_t* __restrict__ first,
    int32_t* count, uint64_t seed, const float* __restrict__ proposal, unsigned* inst_max,
    WsHeader* hdr, DegPartial* parts, ppl_is_result* out) {
  extern __shared__ __align__(16) unsigned char smem[];
  TraceSmem<PPT>& ts = *reinterpret_cast<TraceSmem<PPT>*>(smem);
  float2* sdata = reinterpret_cast<float2*>(smem + trace_smem_bytes<PPT>());
  __shared__ int64_t item_sh;
  __shared__ bool last_sh;
  __shared__ ProposalSmem prop;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  reset_warp_partials(ts);
  int cur = -1;      // instance whose data is staged
  int cur_prop = -1;  // instance whose proposal is loaded
  while (true) {
    if (tid == 0) item_sh = (int64_t)atomicAdd(&hdr->tile_counter[1], 1u);
    __syncthreads();
    const int64_t it = item_sh;
    if (it >= n_items) break;
    const int b = items[it].inst;
    const int64_t d0 = data_off[b], L = data_off[b + 1] - d0;
    const int64_t N = part_off[b + 1] - part_off[b];
    const bool resident = L <= kBatchChunk;
    if (resident && b != cur) {
      for (int l = tid; l < L; l += kTpb) sdata[l] = make_float2(xs[d0 + l], ys[d0 + l]);
      __syncthreads();
      cur = b;
    } else if (!resident) {
      cur = -1;  // the chunks overwrite the staged data
    }
    const int64_t tbase = (int64_t)items[it].tile * kTpb * PPT;
    // maxima already reached by this instance's finished items bound the final
    // maxima from below: traces far beneath them are skipped (trace_group)
    if (tid < kMaxDegrees) {
      const unsigned k = (unsigned)ld_volatile_i32(reinterpret_cast<const int32_t*>(inst_max) +
                                                   (int64_t)b * kMaxDegrees + tid);
      ts.ext_max[tid] = (k == 0) ? -INFINITY : key_float(k);
    }
    __syncthreads();
    if (LEARNED) {
      if (b != cur_prop) {
        __syncthreads();
        if (warp == 0) load_proposal(p, proposal + (int64_t)b * 48, prop);
        __syncthreads();
        cur_prop = b;
      }
      trace_group<PPT>(LearnedDraw{p, seed, (uint32_t)b, &prop}, p, xs + d0, ys + d0, L,
                       kBatchChunk, resident, sdata, N, tbase, nullptr, nullptr, ts);
    } else {
      trace_group<PPT>(PriorDraw{p, seed, (uint32_t)b}, p, xs + d0, ys + d0, L, kBatchChunk,
                       resident, sdata, N, tbase, nullptr, nullptr, ts);
    }
    // each warp leaves its per-degree partials of this tile in the tile's slot
    // and raises the instance's running maxima; no block-level merge per tile
    {
      const int64_t slot0 = ((int64_t)first[b] + items[it].tile) * kWarpParts + warp * kMaxDegrees;
      __syncwarp();
      if (lane < kMaxDegrees * 4) {
        const float4* src = reinterpret_cast<const float4*>(&ts.wrun[warp * kMaxDegrees]);
        reinterpret_cast<float4*>(parts + slot0)[lane] = src[lane];
      }
      if (lane < kMaxDegrees) {
        const float m = ts.wrun[warp * kMaxDegrees + lane].m;
        if (m > -INFINITY) atomicMax(inst_max + (int64_t)b * kMaxDegrees + lane, float_key(m));
      }
      __syncwarp();
      if (lane < kMaxDegrees) deg_empty(ts.wrun[warp * kMaxDegrees + lane]);
      if (tid < kMaxDegrees) ts.ext_max[tid] = -INFINITY;
    }
    if (tid == 0 && ts.nan) record_status(&hdr->status, PPL_ENAN);
    // the last item of the instance merges the instance's partials; the
    // barrier and thread 0's fence order every warp's partial writes before
    // the count (fences are cumulative)
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      last_sh = atomicSub(&count[b], 1) == 1;
    }
    __syncthreads();
    if (last_sh) {
      __threadfence();
      const int64_t ni = (N + (int64_t)kTpb * PPT - 1) / ((int64_t)kTpb * PPT);
      finish_instance(p, parts + (int64_t)first[b] * kWarpParts, ni, N, hdr, out + b);
    }
  }
}

// ---------------------------------------------------------------------------
// Short data sets.  With a few dozen points the factor is no longer what a
// trace costs: the degree sort is (about 150 instructions a trace with its
// shared-memory round trip and barriers), and under a learned proposal, whose
// weights are nearly even, the fold of nearly every trace by warp reductions
// (70 shuffles per degree present in a warp's 256 traces).  Here a thread keeps
// its traces to itself: two at a time, Horner chains padded to six
// coefficients as f32x2 pairs (the same log-weights, bit for bit: padding adds
// exact zeros), and lane sums of all four degrees in registers
// (lanesums.cuh), reduced once per run of tiles.
//
// A block takes runs of consecutive tiles of one instance from the queue, in
// instance order, and leaves one partial per warp in the run's first slot
// (empty ones in the others).  A warp's reference is the best of its first
// traces and moves when a trace lies kRebaseNats above it; nothing a run
// computes depends on the other runs, so the result does not depend on timing.
//
// Sorted kernel and this one, us, 32 points, near-posterior proposals | prior draws:
//   256 sets x 2^14 (2^22 traces)   200  173 | 137  141
//   256 x 2^15 (2^23)               385  329 | 237  267
//   256 x 2^16 (2^24)               773  547 | 435  446
//   1024 x 2^14 (2^24)              790  546 | 474  454
//   1024 x 2^15 (2^25)             1583 1052 | 865  873
//   1024 x 2^16 (2^26)             3180 2005 | 1654 1657
// and 1720 and 1380 us for prior draws on 16 points (2^26).  A run costs about 13
// us of a block besides its traces (the first traces' references, the
// reduction); smaller batches than these are 2 to 4 times slower here.  Under
// proposals this kernel wins from 2^22 traces on; prior draws, which skip most
// traces in either kernel, lose 3 to 13 % up to 2^24 and are even from 2^25 on:
// the line lies where neither draw loses.  Above 32 points the padded chains
// outweigh the sort (prior draws, 64 points: 1055 and 1160 us).
// Both draws take the same kernel, so that a proposal equal to the prior gives
// the prior's run bit for bit.
// ---------------------------------------------------------------------------
constexpr int kLanesMaxLen = 32;  // a multiple of 16
constexpr int64_t kRunTraces = 16384, kLanesMinMean = kRunTraces, kLanesMinTotal = (int64_t)1 << 25;

struct __align__(16) LaneRef {
  float v[kMaxDegrees][8];  // ref c[6], m_ref, the best log-weight so far
  int arg[kMaxDegrees];     // and its trace
};

template <bool LEARNED>
__global__ void __launch_bounds__(kTpb, 2) lanes_kernel(
    PolyParams p, const float* __restrict__ xs, const float* __restrict__ ys,
    const int64_t* __restrict__ data_off, const int64_t* __restrict__ part_off, int n_inst,
    int64_t n_tiles, int tile_traces, int run_tiles, const int32_t* __restrict__ first,
    int32_t* count, uint64_t seed, const float* __restrict__ proposal, WsHeader* hdr,
    DegPartial* parts, ppl_is_result* out) {
  __shared__ __align__(16) ulonglong2 sdata[kLanesMaxLen];  // (x, x), (y, y)
  __shared__ LaneRef refs[kTpb / 32];
  __shared__ ProposalSmem prop;
  __shared__ int64_t run_sh;
  __shared__ int last_sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  LaneRef& rf = refs[warp];
  int cur = -1;  // instance whose data and proposal are staged
  while (true) {
    if (tid == 0) run_sh = (int64_t)atomicAdd(&hdr->tile_counter[1], 1u);
    __syncthreads();
    int64_t s = run_sh * run_tiles;
    const int64_t s_end = s + run_tiles < n_tiles ? s + run_tiles : n_tiles;
    if (s >= n_tiles) break;
    while (s < s_end) {  // the same for the whole block
      // the instance of slot s: the last with first <= s (32 probes a round)
      int lo = 0, hi = n_inst;  // first[lo] <= s < first[hi]
      while (hi - lo > 1) {
        const int w = (hi - lo + 31) / 32, q = lo + lane * w;
        const unsigned m = __ballot_sync(0xffffffffu, q < hi && __ldg(first + q) <= s);
        const int f = 31 - __clz(m);  // lane 0 probes lo: m != 0
        hi = min(hi, lo + (f + 1) * w);
        lo += f * w;
      }
      const int b = lo;
      const int64_t d0 = data_off[b], L = data_off[b + 1] - d0;
      const int64_t N = part_off[b + 1] - part_off[b];
      const int64_t tiles = (b + 1 < n_inst ? (int64_t)first[b + 1] : n_tiles) - first[b];
      const int64_t t0 = s - first[b], t1 = min(tiles, s_end - first[b]);
      __syncthreads();  // the previous run's data and refs have been read
      if (b != cur) {
        for (int l = tid; l < kLanesMaxLen && l < L; l += kTpb)
          sdata[l] = make_ulonglong2(f2_pack(xs[d0 + l], xs[d0 + l]), f2_pack(ys[d0 + l], ys[d0 + l]));
        if (LEARNED && warp == 0) load_proposal(p, proposal + (int64_t)b * 48, prop);
        cur = b;
      }
      if (lane < kMaxDegrees) {
        rf.arg[lane] = 0x7fffffff;
#pragma unroll
        for (int j = 0; j < kMaxCoef; ++j) rf.v[lane][j] = 0.0f;
        rf.v[lane][6] = rf.v[lane][7] = -INFINITY;
      }
      __syncthreads();
      LaneSums a[kMaxDegrees];
#pragma unroll
      for (int k = 0; k < kMaxDegrees; ++k) lane_zero(a[k]);
      int nan = 0;
      const int64_t i_end = min(N, t1 * tile_traces);
      // a warp takes 64 consecutive traces, two per lane
      for (int64_t i0 = t0 * tile_traces + warp * 64; i0 < i_end; i0 += (kTpb / 32) * 64) {
        float c[2][kMaxCoef], corr[2], lw[2];
        int d[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int64_t i = i0 + u * 32 + lane;
          const uint32_t gi = (uint32_t)(i < i_end ? i : 0);
          const int n = LEARNED ? LearnedDraw{p, seed, (uint32_t)b, &prop}(gi, c[u], corr[u])
                                : PriorDraw{p, seed, (uint32_t)b}(gi, c[u], corr[u]);
          d[u] = i < i_end ? n - p.min_deg : -1;
        }
        {
          unsigned long long cc[kMaxCoef];
#pragma unroll
          for (int k = 0; k < kMaxCoef; ++k) cc[k] = f2_pack(c[0][k], c[1][k]);
          float ss[2] = {0.0f, 0.0f}, comp[2] = {0.0f, 0.0f};
          unsigned long long part = 0ull;
          auto point = [&](const ulonglong2 pt) {
            unsigned long long f = cc[kMaxCoef - 1];
#pragma unroll
            for (int k = kMaxCoef - 2; k >= 0; --k) f = f2_fma(f, pt.x, cc[k]);
            const unsigned long long r = f2_sub(pt.y, f);
            part = f2_fma(r, r, part);
          };
          for (int64_t l = 0; l < L; l += 16) {  // blocks of 16 points, compensated between
            const int nb = L - l < 16 ? (int)(L - l) : 16;
            part = 0ull;
            if (l >= kLanesMaxLen) {  // past what the plan announced
              for (int j = 0; j < nb; ++j) {
                const float xv = xs[d0 + l + j], yv = ys[d0 + l + j];
                point(make_ulonglong2(f2_pack(xv, xv), f2_pack(yv, yv)));
              }
            } else if (nb == 16) {
#pragma unroll 4
              for (int j = 0; j < 16; ++j) point(sdata[l + j]);
            } else {
              for (int j = 0; j < nb; ++j) point(sdata[l + j]);
            }
            const float2 v = f2_unpack(part);
            kahan_add(ss[0], comp[0], v.x);
            kahan_add(ss[1], comp[1], v.y);
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) lw[u] = ss[u] * p.neg_half_inv_var + corr[u];
        }
        float4 f0[2], f1[2];
        bool rare = false;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float4* rp = reinterpret_cast<const float4*>(rf.v[d[u] >= 0 ? d[u] : 0]);
          f0[u] = rp[0];
          f1[u] = rp[1];
          rare |= d[u] >= 0 && !(lw[u] <= f1[u].w);  // a NaN too
        }
        if (__any_sync(0xffffffffu, rare)) {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            nan |= d[u] >= 0 && lw[u] != lw[u];
#pragma unroll
            for (int k = 0; k < kMaxDegrees; ++k) {
              const bool mine = d[u] == k && lw[u] > rf.v[k][7];
              if (!__any_sync(0xffffffffu, mine)) continue;
              const float mx = warp_max(mine ? lw[u] : -INFINITY);
              // lanes hold increasing indices: the first lane at the maximum is the lowest
              const int src = __ffs(__ballot_sync(0xffffffffu, mine && lw[u] == mx)) - 1;
              const float m0 = rf.v[k][6];
              if (!(mx <= m0 + kRebaseNats)) {
                float g[kMaxCoef], nc[kMaxCoef];
#pragma unroll
                for (int j = 0; j < kMaxCoef; ++j) {
                  nc[j] = __shfl_sync(0xffffffffu, c[u][j], src);
                  g[j] = rf.v[k][j] - nc[j];
                }
                lane_move(a[k], g, m0 > -INFINITY ? expf(m0 - mx) : 0.0f);
                __syncwarp();
                if (lane == 0) {
#pragma unroll
                  for (int j = 0; j < kMaxCoef; ++j) rf.v[k][j] = nc[j];
                  rf.v[k][6] = mx;
                }
              }
              if (lane == src) {
                rf.v[k][7] = mx;
                rf.arg[k] = (int)(i0 + u * 32 + lane);
              }
              __syncwarp();
            }
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const float4* rp = reinterpret_cast<const float4*>(rf.v[d[u] >= 0 ? d[u] : 0]);
            f0[u] = rp[0];
            f1[u] = rp[1];
          }
        }
        // under the prior few traces carry weight (FP32's exponential is 0 below -104)
        if (!LEARNED) {
          const bool some = !(lw[0] - f1[0].z < -104.0f) || !(lw[1] - f1[1].z < -104.0f);
          if (!__any_sync(0xffffffffu, some)) continue;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          // -inf and NaN log-weights carry nothing
          const float w = d[u] >= 0 && lw[u] > -INFINITY ? expf(lw[u] - f1[u].z) : 0.0f;
          lane_add(a, d[u], w, c[u], f0[u], f1[u]);
        }
      }
      // the warp's partials into the run's first slot, empty ones into the rest
      DegPartial* slot0 = parts + (s * (kTpb / 32) + warp) * kMaxDegrees;
#pragma unroll
      for (int k = 0; k < kMaxDegrees; ++k) {
        const DegPartial r = lane_partial(a[k], rf.v[k], rf.v[k][7], rf.arg[k]);
        if (lane == 0) slot0[k] = r;
      }
      for (int64_t t = t0 + 1; t < t1; ++t)
        if (lane < kMaxDegrees) deg_empty(slot0[(t - t0) * kWarpParts + lane]);
      if (__any_sync(0xffffffffu, nan) && lane == 0) record_status(&hdr->status, PPL_ENAN);
      // the last run of the instance merges its partials; the barrier and
      // thread 0's fence order every warp's partial writes before the count
      __syncthreads();
      if (tid == 0) {
        __threadfence();
        last_sh = atomicSub(&count[b], (int)(t1 - t0)) == (int)(t1 - t0);
      }
      __syncthreads();
      if (last_sh) {
        __threadfence();
        finish_instance(p, parts + (int64_t)first[b] * kWarpParts, tiles, N, hdr, out + b);
      }
      s += t1 - t0;
    }
    __syncthreads();  // run_sh is rewritten
  }
}

// Whether a batch runs in lanes_kernel (which takes two blocks per SM, whatever
// the plan says).
static bool in_lanes(int64_t max_len, int64_t total, int32_t n_inst) {
  return max_len <= kLanesMaxLen && total >= kLanesMinTotal && total / n_inst >= kLanesMinMean;
}

template <int PPT, bool LEARNED>
static cudaError_t launch_batched_t(const PolyParams& p, const float* x, const float* y,
                                    const int64_t* data_off, const int64_t* part_off,
                                    int32_t n_inst, int64_t n_items, int64_t max_len, int64_t total,
                                    int blocks_per_sm, uint64_t seed, const float* proposal,
                                    char* ws, ppl_is_result* out, cudaStream_t s) {
  const BatchLayout l = batch_layout(n_items, n_inst);
  WsHeader* hdr = reinterpret_cast<WsHeader*>(ws + l.header);
  cudaError_t e = cudaMemsetAsync(ws + l.header, 0, 512, s);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(ws + l.count, ws + l.count_tmpl, (size_t)n_inst * sizeof(int32_t),
                      cudaMemcpyDeviceToDevice, s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(ws + l.inst_max, 0, (size_t)n_inst * kMaxDegrees * sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  if (in_lanes(max_len, total, n_inst)) {
    const int64_t blocks = (int64_t)num_sms() * 2;
    const int run = (int)std::max<int64_t>(1, kRunTraces / (kTpb * PPT));
    const int64_t runs = (n_items + run - 1) / run;
    lanes_kernel<LEARNED><<<(unsigned)std::min(runs, blocks), kTpb, 0, s>>>(
        p, x, y, data_off, part_off, n_inst, n_items, kTpb * PPT, run,
        reinterpret_cast<const int32_t*>(ws + l.first), reinterpret_cast<int32_t*>(ws + l.count),
        seed, proposal, hdr, reinterpret_cast<DegPartial*>(ws + l.parts), out);
    return cudaGetLastError();
  }
  const size_t smem = trace_smem_bytes<PPT>() + kBatchChunk * sizeof(float2);
  int unused = 0;
  e = device_once((const void*)batched_kernel<PPT, LEARNED>, &unused, [smem](int*) {
    return cudaFuncSetAttribute(batched_kernel<PPT, LEARNED>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batched_kernel<PPT, LEARNED>, kTpb,
                                                    smem);
  if (e != cudaSuccess) return e;
  const int bps = std::max(1, std::min(blocks_per_sm, std::max(1, per_sm)));
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(n_items, (int64_t)num_sms() * bps));
  batched_kernel<PPT, LEARNED><<<(unsigned)grid, kTpb, smem, s>>>(
      p, x, y, data_off, part_off, reinterpret_cast<const BatchItem*>(ws + l.items), n_items,
      reinterpret_cast<const int32_t*>(ws + l.first), reinterpret_cast<int32_t*>(ws + l.count),
      seed, proposal, reinterpret_cast<unsigned*>(ws + l.inst_max), hdr,
      reinterpret_cast<DegPartial*>(ws + l.parts), out);
  return cudaGetLastError();
}

cudaError_t launch_batched(const PolyParams& p, const float* x, const float* y,
                           const int64_t* data_off, const int64_t* part_off, int32_t n_inst,
                           int64_t n_items, int64_t max_len, int64_t total, int ppt,
                           int blocks_per_sm, uint64_t seed, const float* proposal, char* ws,
                           ppl_is_result* out, cudaStream_t s) {
#define PPL_BATCHED_CASE(P)                                                                   \
  case P:                                                                                     \
    return proposal ? launch_batched_t<P, true>(p, x, y, data_off, part_off, n_inst, n_items, \
                                                max_len, total, blocks_per_sm, seed, proposal, \
                                                ws, out, s)                                   \
                    : launch_batched_t<P, false>(p, x, y, data_off, part_off, n_inst, n_items, \
                                                 max_len, total, blocks_per_sm, seed, nullptr, \
                                                 ws, out, s);
  switch (ppt) {
    PPL_BATCHED_CASE(1)
    PPL_BATCHED_CASE(2)
    PPL_BATCHED_CASE(4)
    PPL_BATCHED_CASE(8)
    default: return cudaErrorInvalidValue;
  }
#undef PPL_BATCHED_CASE
}

// Host plan.  Items are issued in rounds: round r holds tile r of every
// instance with more than r tiles, heaviest (longest data) first.  An
// instance's first tile thus finishes early and its maxima let the later
// tiles skip negligible traces; within a round the heaviest-first order keeps
// the blocks finishing together.  first[b] is instance b's base among the
// per-tile partial slots (contiguous per instance); count[b] its tile count.
static int64_t build_plan(const int64_t* data_off, const int64_t* part_off, int32_t n_inst,
                          int ppt, std::vector<BatchItem>* items, std::vector<int32_t>* first,
                          std::vector<int32_t>* count, int64_t* max_len, double* work) {
  const int64_t tile = (int64_t)kTpb * ppt;
  std::vector<int32_t> order(n_inst);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
    return (data_off[a + 1] - data_off[a]) > (data_off[b + 1] - data_off[b]);
  });
  items->clear();
  first->assign(n_inst, 0);
  count->assign(n_inst, 0);
  *max_len = 0;
  *work = 0.0;
  int64_t slots = 0, max_tiles = 0;
  for (int32_t b = 0; b < n_inst; ++b) {
    const int64_t L = data_off[b + 1] - data_off[b];
    const int64_t N = part_off[b + 1] - part_off[b];
    const int64_t tiles = (N + tile - 1) / tile;
    (*first)[b] = (int32_t)slots;
    (*count)[b] = (int32_t)tiles;
    slots += tiles;
    max_tiles = std::max(max_tiles, tiles);
    *max_len = std::max(*max_len, L);
    *work += (double)N * (double)L;
  }
  for (int64_t r = 0; r < max_tiles; ++r)
    for (int32_t b : order)
      if (r < (*count)[b]) items->push_back(BatchItem{b, (int32_t)r});
  return (int64_t)items->size();
}

static bool valid_offsets(const int64_t* data_off, const int64_t* part_off, int32_t n_inst) {
  if (!data_off || !part_off || n_inst < 1) return false;
  if (data_off[0] != 0 || part_off[0] != 0) return false;
  for (int32_t b = 0; b < n_inst; ++b) {
    const int64_t L = data_off[b + 1] - data_off[b], N = part_off[b + 1] - part_off[b];
    if (L < 0 || N < 1 || N > 0x7fffffffll) return false;
  }
  return true;
}

}  // namespace ppl

using namespace ppl;

namespace {

ppl_status poly_params_b(const ppl_model* m, PolyParams* p) {
  if (!m || m->id != PPL_MODEL_POLY) return PPL_EINVAL;
  const int n_deg = m->max_deg - m->min_deg + 1;
  if (m->min_deg < 0 || n_deg < 1 || n_deg > kMaxDegrees || m->coef_offset < 0 ||
      m->max_deg + m->coef_offset > kMaxCoef || !(m->obs_sigma > 0.0f))
    return PPL_EINVAL;
  p->min_deg = m->min_deg;
  p->n_deg = n_deg;
  p->coef_offset = m->coef_offset;
  p->prior_sigma = m->prior_sigma;
  p->neg_half_inv_var = (float)(-1.0 / (2.0 * (double)m->obs_sigma * (double)m->obs_sigma));
  return PPL_OK;
}

bool valid_ppt(int ppt) { return ppt == 1 || ppt == 2 || ppt == 4 || ppt == 8; }

}  // namespace

extern "C" {

size_t ppl_batched_workspace_size(const int64_t* data_off_host, const int64_t* part_off_host,
                                  int32_t n_inst, int32_t ppt) {
  if (!valid_offsets(data_off_host, part_off_host, n_inst) || !valid_ppt(ppt)) return 0;
  std::vector<BatchItem> items;
  std::vector<int32_t> first, count;
  int64_t max_len;
  double work;
  const int64_t n_items =
      build_plan(data_off_host, part_off_host, n_inst, ppt, &items, &first, &count, &max_len,
                 &work);
  // the largest plan of any candidate configuration (ppt = 1 has the most items)
  std::vector<BatchItem> i1;
  const int64_t n1 = build_plan(data_off_host, part_off_host, n_inst, 1, &i1, &first, &count,
                                &max_len, &work);
  return batch_layout(std::max(n_items, n1), n_inst).total;
}

ppl_status ppl_batched_prepare(const ppl_model* model, const int64_t* data_off_host,
                               const int64_t* part_off_host, int32_t n_inst, int32_t ppt,
                               int32_t blocks_per_sm, ppl_batch_plan* plan, void* ws,
                               size_t ws_bytes, ppl_stream stream) {
  PolyParams p;
  if (poly_params_b(model, &p) != PPL_OK) return PPL_EINVAL;
  if (!plan || !ws || !valid_ppt(ppt) || blocks_per_sm < 1 || blocks_per_sm > 32)
    return PPL_EINVAL;
  if (!valid_offsets(data_off_host, part_off_host, n_inst)) return PPL_EINVAL;
  if (reinterpret_cast<uintptr_t>(ws) % 256) return PPL_EINVAL;
  std::vector<BatchItem> items;
  std::vector<int32_t> first, count;
  int64_t max_len;
  double work;
  const int64_t n_items =
      build_plan(data_off_host, part_off_host, n_inst, ppt, &items, &first, &count, &max_len,
                 &work);
  const BatchLayout l = batch_layout(n_items, n_inst);
  if (ws_bytes < l.total) return PPL_EINVAL;
  char* base = static_cast<char*>(ws);
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemcpyAsync(base + l.items, items.data(), items.size() * sizeof(BatchItem),
                      cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(base + l.first, first.data(), first.size() * sizeof(int32_t),
                      cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(base + l.count_tmpl, count.data(), count.size() * sizeof(int32_t),
                      cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return PPL_ECUDA;
  plan->ppt = ppt;
  plan->blocks_per_sm = blocks_per_sm;
  plan->n_inst = n_inst;
  plan->n_items = n_items;
  plan->max_len = max_len;
  plan->total_particles = part_off_host[n_inst];
  plan->work = work;
  return PPL_OK;
}

ppl_status ppl_infer_is_batched(const ppl_model* model, const float* x, const float* y,
                                const int64_t* data_off, const int64_t* part_off,
                                int32_t n_inst, uint64_t seed, const ppl_batch_plan* plan,
                                ppl_is_result* out_dev, void* ws, size_t ws_bytes,
                                ppl_stream stream) {
  PolyParams p;
  if (poly_params_b(model, &p) != PPL_OK) return PPL_EINVAL;
  if (!plan || !x || !y || !data_off || !part_off || !out_dev || !ws) return PPL_EINVAL;
  if (plan->n_inst != n_inst || !valid_ppt(plan->ppt)) return PPL_EINVAL;
  if (ws_bytes < batch_layout(plan->n_items, n_inst).total) return PPL_EINVAL;
  const cudaError_t e =
      launch_batched(p, x, y, data_off, part_off, n_inst, plan->n_items, plan->max_len,
                     plan->total_particles, plan->ppt,
                     plan->blocks_per_sm, seed, nullptr, static_cast<char*>(ws), out_dev,
                     (cudaStream_t)stream);
  return e == cudaSuccess ? PPL_OK : PPL_ECUDA;
}

ppl_status ppl_infer_is_learned(const ppl_model* model, const float* x, const float* y,
                                const int64_t* data_off, const int64_t* part_off,
                                int32_t n_inst, uint64_t seed, const ppl_batch_plan* plan,
                                const float* proposal, ppl_is_result* out_dev, void* ws,
                                size_t ws_bytes, ppl_stream stream) {
  PolyParams p;
  if (poly_params_b(model, &p) != PPL_OK || !(model->prior_sigma > 0.0f)) return PPL_EINVAL;
  int slots = 0;
  for (int k = 0; k < p.n_deg; ++k) slots += p.min_deg + k + p.coef_offset;
  if (slots > kMaxSlots) return PPL_EINVAL;
  if (!plan || !x || !y || !data_off || !part_off || !out_dev || !ws || !proposal)
    return PPL_EINVAL;
  if (plan->n_inst != n_inst || !valid_ppt(plan->ppt)) return PPL_EINVAL;
  if (ws_bytes < batch_layout(plan->n_items, n_inst).total) return PPL_EINVAL;
  const cudaError_t e =
      launch_batched(p, x, y, data_off, part_off, n_inst, plan->n_items, plan->max_len,
                     plan->total_particles, plan->ppt,
                     plan->blocks_per_sm, seed, proposal, static_cast<char*>(ws), out_dev,
                     (cudaStream_t)stream);
  return e == cudaSuccess ? PPL_OK : PPL_ECUDA;
}

ppl_status ppl_batched_status(const void* ws, ppl_stream stream) {
  return ppl_workspace_status(ws, stream);
}

// Autotuner: times every (ppt, blocks_per_sm) candidate on the caller's data
// (every ppt where the kernel has its own number of blocks)
// (two warm-up launches, then the median of three), keeps the fastest, and
// records it in `cache_path` (a one-line JSON object keyed by the batch's
// shape).  A cached entry with the same key is reused without timing.
ppl_status ppl_batched_autotune(const ppl_model* model, const float* x, const float* y,
                                const int64_t* data_off_dev, const int64_t* part_off_dev,
                                const int64_t* data_off_host, const int64_t* part_off_host,
                                int32_t n_inst, uint64_t seed, ppl_is_result* out_dev, void* ws,
                                size_t ws_bytes, const char* cache_path, ppl_batch_plan* best,
                                ppl_stream stream) {
  if (!best || !valid_offsets(data_off_host, part_off_host, n_inst)) return PPL_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  double work = 0.0;
  int64_t max_len = 0;
  for (int32_t b = 0; b < n_inst; ++b) {
    const int64_t L = data_off_host[b + 1] - data_off_host[b];
    work += (double)(part_off_host[b + 1] - part_off_host[b]) * (double)L;
    max_len = std::max(max_len, L);
  }
  char key[160];
  snprintf(key, sizeof key, "n%d_p%lld_w%.6e_L%lld_sm%d", n_inst,
           (long long)part_off_host[n_inst], work, (long long)max_len, num_sms());
  if (cache_path) {
    FILE* f = fopen(cache_path, "r");
    if (f) {
      char line[512] = {0};
      const size_t got = fread(line, 1, sizeof line - 1, f);
      fclose(f);
      line[got] = 0;
      char k[160] = {0};
      int ppt = 0, bps = 0;
      const char* kp = strstr(line, "\"key\": \"");
      const char* pp = strstr(line, "\"ppt\": ");
      const char* bp = strstr(line, "\"blocks_per_sm\": ");
      if (kp && pp && bp && sscanf(kp + 8, "%159[^\"]", k) == 1 && sscanf(pp + 7, "%d", &ppt) == 1 &&
          sscanf(bp + 17, "%d", &bps) == 1 && strcmp(k, key) == 0 && valid_ppt(ppt)) {
        return ppl_batched_prepare(model, data_off_host, part_off_host, n_inst, ppt, bps, best,
                                   ws, ws_bytes, stream);
      }
    }
  }
  const int ppts[] = {1, 2, 4, 8};
  const int bpss[] = {1, 2, 3, 4};
  float best_ms = 1e30f;
  int best_ppt = 4, best_bps = 2;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
    return PPL_ECUDA;
  const bool lanes = in_lanes(max_len, part_off_host[n_inst], n_inst);
  for (int ppt : ppts) {
    for (int bps : bpss) {
      if (lanes && bps != 2) continue;  // the same launch
      ppl_batch_plan plan;
      ppl_status st = ppl_batched_prepare(model, data_off_host, part_off_host, n_inst, ppt, bps,
                                          &plan, ws, ws_bytes, stream);
      if (st != PPL_OK) {
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        return st;
      }
      float t[3];
      for (int r = 0; r < 5; ++r) {
        cudaEventRecord(e0, s);
        st = ppl_infer_is_batched(model, x, y, data_off_dev, part_off_dev, n_inst, seed, &plan,
                                  out_dev, ws, ws_bytes, stream);
        cudaEventRecord(e1, s);
        if (st != PPL_OK || cudaEventSynchronize(e1) != cudaSuccess) {
          cudaEventDestroy(e0);
          cudaEventDestroy(e1);
          return st != PPL_OK ? st : PPL_ECUDA;
        }
        if (r >= 2) cudaEventElapsedTime(&t[r - 2], e0, e1);
      }
      std::sort(t, t + 3);
      if (t[1] < best_ms) {
        best_ms = t[1];
        best_ppt = ppt;
        best_bps = bps;
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (cache_path) {
    FILE* f = fopen(cache_path, "w");
    if (f) {
      fprintf(f, "{\"key\": \"%s\", \"ppt\": %d, \"blocks_per_sm\": %d, \"ms\": %.4f}\n", key,
              best_ppt, best_bps, best_ms);
      fclose(f);
    }
  }
  return ppl_batched_prepare(model, data_off_host, part_off_host, n_inst, best_ppt, best_bps,
                             best, ws, ws_bytes, stream);
}

}  // extern "C"
