// The proposal network's passes (mlp.cu defines network, loss and training):
// two kernels in place of nine products with their reductions.
//
// net_kernel: forward, loss gradient and the gradients with respect to the
// activations for 128 pairs per CTA.  Everything between the features and
// those gradients stays on the SM: activations in shared memory as the next
// product's A operand, accumulators in tensor memory, weights streamed from
// L2 in 64-column chunks (cp.async, double-buffered).  A step's batch is a
// few tiles, so what bounds it is the chain of 17 dependent products, not
// their FLOPs: as separate launches each cost 15 to 31 us, mostly launch,
// operand staging and strided stores, and the whole chain 143 us; here
// 39 us (1024 pairs; half of it the issue of its 172 products, 117 cycles
// each, half the epilogues' strided stores).
//
// dw_kernel: the weight gradients (contractions over the batch) of all three
// layers in one launch, split along the batch into slices whose raw tiles,
// and the bias gradients' column sums, go to `partial`; the consumer (Adam or
// grad_kernel) adds the slices in order, so results are the same on every
// run.  The operands are read as they lie ([pair][unit], the contraction
// along the rows) through MN-major descriptors.  Before: three products and
// three reductions, 73 us, and three one-block column sums of 55 to 66 us
// each; 12 us.
//
// Operands sit in shared memory in the canonical layout without swizzle: 8 x 8
// core matrices of 128 contiguous bytes (8 rows of 16 bytes, along K for a
// K-major operand, along M or N for an MN-major one), contraction-adjacent
// cores 128 B apart (leading byte offset), the others (K / 8) 128 B (stride
// byte offset).  Every mbarrier wait is bounded; one that runs out records
// PPL_ETIMEOUT, and tensor memory is freed on every path.
#include <cuda_bf16.h>

#include "kernels.h"
#include "mlp.cuh"

namespace ppl {
namespace {

constexpr int kNetRows = 128;      // pairs per CTA (MMA M, tensor-memory lanes)
constexpr int kNetThreads = 256;   // two warpgroups, 32 columns of a chunk each
constexpr int kNetN = 64;          // columns of a chunk (MMA N)
constexpr uint32_t kNetCols = 256; // tensor-memory columns: up to four K slices of a chunk
constexpr int kNetSpin = 1 << 22;  // bound of one mbarrier wait (polls)
// shared memory (bytes)
constexpr int kOffH1 = 0, kOffH2 = 65536, kOffFd = 131072, kOffWb = 147456, kWbBytes = 32768,
              kOffBias = kOffWb + 2 * kWbBytes, kNetSmem = kOffBias + (2 * kHid + kOut) * 4;
constexpr int kRowStride = kOut + 1;  // FP32 rows of the outputs in a free weight buffer
static_assert(kNetRows * kRowStride * 4 <= kWbBytes, "the output rows fit a weight buffer");

// Instruction descriptor, kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A
// and B (bits 7-9, 10-12 = 1), A and B MN-major (bits 15, 16), N >> 3 at bit
// 17, M >> 4 at bit 24.
__device__ __forceinline__ constexpr uint32_t idesc(int m, int n, bool a_mn, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t mma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3fffu) | ((uint64_t)((lbo >> 4) & 0x3fffu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3fffu) << 32) | (1ull << 46);
}

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t id,
                                        uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   mbar)
               : "memory");
}

__device__ __forceinline__ bool mma_wait(uint32_t mbar, uint32_t phase) {
  for (int i = 0; i < kNetSpin; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(mbar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols)
               : "memory");
}

// 32 consecutive FP32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void cp16(void* dst, const void* src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(in ? 16 : 0)
               : "memory");
}

// rows x kt elements of a row-major matrix as a K-major operand; rows from
// `valid` on are zero.  Eight lanes take a core's rows, four of these its
// neighbours along K, so that a warp reads 64-byte runs and its 16-byte
// stores are free of bank conflicts.
template <int kt>
__device__ __forceinline__ void stage_k(unsigned char* dst, const __nv_bfloat16* src, int ld,
                                        int rows, int valid, int tid) {
  constexpr int kg = kt / 8, kq = kg / 4;
#pragma unroll 4
  for (int u = tid; u < rows * kg; u += kNetThreads) {
    const int rl = u & 7, v = u >> 5, g = (v % kq) * 4 + ((u >> 3) & 3), rg = v / kq;
    const int row = rg * 8 + rl;
    const bool in = row < valid;
    cp16(dst + (rg * kg + g) * 128 + rl * 16, in ? src + (int64_t)row * ld + g * 8 : src, in);
  }
}

// kt x 64 elements of a row-major matrix, the contraction along its rows, as
// an MN-major operand of 64 columns.
template <int kt>
__device__ __forceinline__ void stage_mn(unsigned char* dst, const __nv_bfloat16* src, int ld,
                                         int tid) {
  constexpr int kg = kt / 8;
#pragma unroll 4
  for (int u = tid; u < kt * 8; u += kNetThreads) {
    const int kl = u & 7, v = u >> 5, g = (v & 1) * 4 + ((u >> 3) & 3), og = v >> 1;
    cp16(dst + (g * kg + og) * 128 + kl * 16, src + (int64_t)(og * 8 + kl) * ld + g * 8, true);
  }
}

__device__ __forceinline__ uint4 pack8(const float* v) {
  uint4 o;
  __nv_bfloat162 p;
  p = __floats2bfloat162_rn(v[0], v[1]); o.x = *reinterpret_cast<uint32_t*>(&p);
  p = __floats2bfloat162_rn(v[2], v[3]); o.y = *reinterpret_cast<uint32_t*>(&p);
  p = __floats2bfloat162_rn(v[4], v[5]); o.z = *reinterpret_cast<uint32_t*>(&p);
  p = __floats2bfloat162_rn(v[6], v[7]); o.w = *reinterpret_cast<uint32_t*>(&p);
  return o;
}
// v[e] = 0 where the e-th BF16 of m is not positive
__device__ __forceinline__ void mask8(float* v, const uint4& m) {
  const uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (!(__uint_as_float(w[e] << 16) > 0.0f)) v[2 * e] = 0.0f;
    if (!(__uint_as_float(w[e] & 0xffff0000u) > 0.0f)) v[2 * e + 1] = 0.0f;
  }
}

}  // namespace

// The weights' chunks in the order of the chain: layer 1 (4 chunks), layer 2
// (4), outputs (1), then dh2 = dout W3 (4) and dh1 = dh2 W2 (4).
constexpr int kChunkL2 = 4, kChunkOut = 8, kChunkD2 = 9, kChunkD1 = 13, kChunks = 17;

__global__ void __launch_bounds__(kNetThreads, 1) net_kernel(NetArgs a) {
  extern __shared__ __align__(1024) unsigned char nsm[];
  unsigned char *h1 = nsm + kOffH1, *h2 = nsm + kOffH2, *fd = nsm + kOffFd;
  float* bias = reinterpret_cast<float*>(nsm + kOffBias);
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base;
  __shared__ int failed;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int half = warp >> 2;                 // the warpgroup's 32 columns of a chunk
  const int r = (warp & 3) * 32 + lane;       // this thread's pair within the tile
  const int row0 = blockIdx.x * kNetRows, row = row0 + r;
  const int valid = min(kNetRows, a.B - row0);
  const bool in = r < valid;
  const int n_chunks = a.backward ? kChunks : kChunkD2;
  const uint32_t mb = smem_u32(&mbar);

  auto stage = [&](int c) {
    unsigned char* wb = nsm + kOffWb + (c & 1) * kWbBytes;
    if (c < kChunkL2) stage_k<kIn>(wb, a.pb + kOffW1 + c * kNetN * kIn, kIn, kNetN, kNetN, tid);
    else if (c < kChunkOut)
      stage_k<kHid>(wb, a.pb + kOffW2 + (c - kChunkL2) * kNetN * kHid, kHid, kNetN, kNetN, tid);
    else if (c == kChunkOut) stage_k<kHid>(wb, a.pb + kOffW3, kHid, kOut, kOut, tid);
    else if (c < kChunkD1) stage_mn<kOut>(wb, a.pb + kOffW3 + (c - kChunkD2) * kNetN, kHid, tid);
    else stage_mn<kHid>(wb, a.pb + kOffW2 + (c - kChunkD1) * kNetN, kHid, tid);
  };
  stage_k<kIn>(fd, a.feat + (int64_t)row0 * kIn, kIn, kNetRows, valid, tid);
  stage(0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int i = tid; i < 2 * kHid + kOut; i += kNetThreads)
    bias[i] = i < kHid ? a.params[kOffB1 + i]
                       : (i < 2 * kHid ? a.params[kOffB2 + i - kHid] : a.params[kOffB3 + i - 2 * kHid]);
  if (warp == 0) tmem_alloc(&tmem_base, kNetCols);
  if (tid == 0) {
    failed = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base, t_lane = (uint32_t)((warp & 3) * 32) << 16;

  for (int c = 0; c < n_chunks; ++c) {
    // the chunk's weights have arrived, the A operand is written and the
    // accumulator's last readers are done
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // K slices: the sums of a long contraction are formed over S slices, added
    // in order in the epilogue
    const int K = c < kChunkL2 ? kIn : (c >= kChunkD2 && c < kChunkD1 ? kOut : kHid);
    const int S = K != kHid ? 1 : (c == kChunkOut ? a.slices_out : a.slices_hid);
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const unsigned char* A = c < kChunkL2 || K == kOut ? fd : (c < kChunkOut ? h1 : h2);
      const uint32_t sa = smem_u32(A), sb = smem_u32(nsm + kOffWb + (c & 1) * kWbBytes);
      const uint32_t sbo = (uint32_t)(K / 8) * 128;
      const uint32_t id = idesc(kNetRows, c == kChunkOut ? kOut : kNetN, false, c >= kChunkD2);
      // (each K step of 16 lies 256 bytes on: the descriptors' address field
      // advances by 16, and one thread's issue is the chain's longest part)
      const int steps = K / 16 / S;
      uint64_t da = mma_desc(sa, 128, sbo), db = mma_desc(sb, 128, sbo);
      for (int z = 0; z < S; ++z) {
        const uint32_t d = tmem + z * kNetN;
        mma_f16(d, da, db, id, 0u);
        da += 16;
        db += 16;
#pragma unroll 3
        for (int k = 1; k < steps; ++k) {
          mma_f16(d, da, db, id, 1u);
          da += 16;
          db += 16;
        }
      }
      mma_commit(mb);
    }
    if (c + 1 < n_chunks) stage(c + 1);  // into the buffer of the chunk before, whose products are done
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (!mma_wait(mb, (uint32_t)(c & 1))) {
      atomicExch(&failed, 1);
      record_status(a.status, PPL_ETIMEOUT);
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    float x[32];
    tmem_ld32(tmem + t_lane + half * 32, x);
#pragma unroll 1
    for (int z = 1; z < S; ++z) {
      float v[32];
      tmem_ld32(tmem + t_lane + z * kNetN + half * 32, v);
#pragma unroll
      for (int j = 0; j < 32; ++j) x[j] += v[j];
    }
    if (c == kChunkOut) {
      // the output rows, FP32, in this chunk's (read) weight buffer
      float* orow = reinterpret_cast<float*>(nsm + kOffWb + (c & 1) * kWbBytes) + r * kRowStride;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (half * 32 + j < kOut) orow[half * 32 + j] = x[j] + bias[2 * kHid + half * 32 + j];
      __syncthreads();
      if (a.out) {
        const float* o0 = reinterpret_cast<const float*>(nsm + kOffWb + (c & 1) * kWbBytes);
        for (int e = tid; e < valid * kOut; e += kNetThreads)
          a.out[(int64_t)row0 * kOut + e] = o0[(e / kOut) * kRowStride + e % kOut];
      }
      if (a.backward && half == 0) {
        // loss -log q of the pair and its gradient with respect to the outputs
        float loss = 0.0f;
        const ProposalShape& q = a.shape;
        if (in) {
          const int n = a.n_t[row], k = n - q.min_deg;
          float lg[kMaxDegrees], mx = -INFINITY;
#pragma unroll
          for (int i = 0; i < kMaxDegrees; ++i) {
            lg[i] = i < q.n_deg ? orow[i] : -INFINITY;
            if (i < q.n_deg) mx = fmaxf(mx, lg[i]);
          }
          float se = 0.0f, ok = 0.0f;
#pragma unroll
          for (int i = 0; i < kMaxDegrees; ++i) {
            if (i < q.n_deg) se += expf(lg[i] - mx);
            if (i == k) ok = lg[i];
          }
          loss = -(ok - mx - logf(se));
#pragma unroll
          for (int i = 0; i < kMaxDegrees; ++i)
            lg[i] = i < q.n_deg ? expf(lg[i] - mx) / se - (i == k ? 1.0f : 0.0f) : 0.0f;
          const int ncoef = n + q.coef_offset, base = slot_base(q, k);
          float gm[kMaxCoef], gs[kMaxCoef];
#pragma unroll
          for (int j = 0; j < kMaxCoef; ++j) {
            gm[j] = gs[j] = 0.0f;
            if (j < ncoef) {
              const float om = orow[4 + 2 * (base + j)], os = orow[5 + 2 * (base + j)];
              const float t = fminf(fmaxf(os, -9.0f), 1.0f);
              const float mu = q.prior_sigma * om, sd = q.prior_sigma * expf(t);
              const float z = (a.c_t[(int64_t)row * kMaxCoef + j] - mu) / sd;
              loss += 0.91893853320467274f + q.log_prior_sigma + t + 0.5f * z * z;
              gm[j] = -z / sd * q.prior_sigma;
              gs[j] = (os > -9.0f && os < 1.0f) ? (1.0f - z * z) : 0.0f;
            }
          }
          for (int i = 0; i < kOut; ++i) orow[i] = 0.0f;
#pragma unroll
          for (int i = 0; i < kMaxDegrees; ++i) orow[i] = lg[i];
#pragma unroll
          for (int j = 0; j < kMaxCoef; ++j)
            if (j < ncoef) {
              orow[4 + 2 * (base + j)] = gm[j];
              orow[5 + 2 * (base + j)] = gs[j];
            }
        } else {
          for (int i = 0; i < kOut; ++i) orow[i] = 0.0f;
        }
        loss = warp_sum(loss);
        if (lane == 0) a.warp_loss[row0 / 32 + warp] = loss;
        // dout, divided by the batch size: FP32 and BF16 to memory, and the
        // BF16 operand of the next products over the features
        const float inv = 1.0f / (float)a.B;
#pragma unroll
        for (int g = 0; g < kOut / 8; ++g) {
          float v[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) v[e] = orow[g * 8 + e] * inv;
          const uint4 p = pack8(v);
          *reinterpret_cast<uint4*>(fd + ((r >> 3) * (kOut / 8) + g) * 128 + (r & 7) * 16) = p;
          if (in) {
            float4* df = reinterpret_cast<float4*>(a.dout + (int64_t)row * kOut + g * 8);
            df[0] = make_float4(v[0], v[1], v[2], v[3]);
            df[1] = make_float4(v[4], v[5], v[6], v[7]);
            *reinterpret_cast<uint4*>(a.dout_b + (int64_t)row * kOut + g * 8) = p;
          }
        }
      }
    } else {
      const int l = c < kChunkL2 ? c : (c < kChunkOut ? c - kChunkL2 : (c < kChunkD1 ? c - kChunkD2 : c - kChunkD1));
      const int n0 = l * kNetN + half * 32;  // first unit of this thread's columns
      unsigned char* dst = c < kChunkL2 ? h1 : h2;
      __nv_bfloat16* gdst = c < kChunkL2 ? a.h1 : (c < kChunkOut ? a.h2 : (c < kChunkD1 ? a.dh2 : a.dh1));
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int so = ((r >> 3) * (kHid / 8) + n0 / 8 + g) * 128 + (r & 7) * 16;
        if (c < kChunkOut) {
          const float4* bv = reinterpret_cast<const float4*>(bias + (c < kChunkL2 ? 0 : kHid) + n0 + g * 8);
          const float4 b0 = bv[0], b1 = bv[1];
          const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
          for (int e = 0; e < 8; ++e) x[g * 8 + e] = fmaxf(x[g * 8 + e] + b[e], 0.0f);
        } else {  // the ReLU's gradient: where the activation is positive
          mask8(x + g * 8, *reinterpret_cast<const uint4*>((c < kChunkD1 ? h2 : h1) + so));
        }
        const uint4 p = pack8(x + g * 8);
        if (c < kChunkD1) *reinterpret_cast<uint4*>(dst + so) = p;  // dh2 takes h2's place
        if (in && gdst) *reinterpret_cast<uint4*>(gdst + (int64_t)row * kHid + n0 + g * 8) = p;
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (__syncthreads_or(failed)) break;  // the same for every thread
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) tmem_free(tmem, kNetCols);
}

// ---------------------------------------------------------------------------
// Weight gradients.  blockIdx.x: 4 tiles of dW3, 8 of dW2, 2 of dW1 (128 x 64
// each, dW3 48 x 64), then the column sums of dh2, dh1 and dout; blockIdx.y:
// the slice of the batch.
// ---------------------------------------------------------------------------
constexpr int kDwTiles = 14, kDwBlocks = kDwTiles + 3, kDwThreads = 128, kDwK = 64;

// 64 pairs x `cols` units (a multiple of 8) as an MN-major operand of `width`.
template <int width>
__device__ __forceinline__ void stage_pairs(unsigned char* dst, const __nv_bfloat16* src, int ld,
                                            int cols, int b0, int b1, int tid) {
  constexpr int gq = width / 32;  // runs of four 8-unit groups
#pragma unroll 4
  for (int u = tid; u < kDwK * width / 8; u += kDwThreads) {
    const int bl = u & 7, v = u >> 5, g = (v % gq) * 4 + ((u >> 3) & 3), bg = v / gq;
    const int b = b0 + bg * 8 + bl;
    const bool in = b < b1 && g * 8 < cols;
    cp16(dst + (g * (kDwK / 8) + bg) * 128 + bl * 16, in ? src + (int64_t)b * ld + g * 8 : src, in);
  }
}

__global__ void __launch_bounds__(kDwThreads) dw_kernel(NetArgs a, int rows_per_slice) {
  __shared__ __align__(1024) unsigned char sm[2 * (128 + 64) * kDwK * 2];  // two steps of A and B
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_base;
  __shared__ int failed;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = blockIdx.x, z = blockIdx.y;
  const int b_begin = z * rows_per_slice, b_end = min(a.B, b_begin + rows_per_slice);
  float* part = a.partial + (size_t)z * kNumParams;

  if (t >= kDwTiles) {
    if (t == kDwTiles + 2) {  // dout, FP32: 48 columns, two groups of rows
      const int col = tid % 64, grp = tid / 64;
      float s = 0.0f;
      if (col < kOut) {
#pragma unroll 8
        for (int b = b_begin + grp; b < b_end; b += 2) s += a.dout[(int64_t)b * kOut + col];
      }
      float* red = reinterpret_cast<float*>(sm);
      red[tid] = s;
      __syncthreads();
      if (tid < kOut) part[kOffB3 + tid] = red[tid] + red[64 + tid];
      // the step's loss, from the warps' sums in the order of blocks of 256
      // pairs: FP32 within a block, FP64 over the blocks
      if (z == 0 && warp == 3 && a.loss) {
        double d = 0.0;
        const int nw = (a.B + kNetRows - 1) / kNetRows * (kNetRows / 32);
        for (int g = lane; g * 8 < nw; g += 32) {
          float f = 0.0f;
#pragma unroll
          for (int w = 0; w < 8; ++w)
            if (g * 8 + w < nw) f += a.warp_loss[g * 8 + w];
          d += (double)f;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0) {
          if (a.step) {  // a training run: the counter advances, the loss goes to its slot
            const int32_t s1 = *a.step + 1;
            *a.step = s1;
            if (a.loss_out) a.loss_out[s1 - 1] = d;
          }
          *a.loss = d;
        }
      }
      return;
    }
    // dh2 or dh1: lane l takes columns 8 l .. 8 l + 7, the warps every fourth row
    const __nv_bfloat16* d = t == kDwTiles ? a.dh2 : a.dh1;
    float s[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) s[e] = 0.0f;
#pragma unroll 8
    for (int b = b_begin + warp; b < b_end; b += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(d + (int64_t)b * kHid + lane * 8);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        s[2 * e] += __uint_as_float(w[e] << 16);
        s[2 * e + 1] += __uint_as_float(w[e] & 0xffff0000u);
      }
    }
    float* red = reinterpret_cast<float*>(sm);  // [4][256]
#pragma unroll
    for (int e = 0; e < 8; ++e) red[warp * kHid + lane * 8 + e] = s[e];
    __syncthreads();
    float* db = part + (t == kDwTiles ? kOffB2 : kOffB1);
    for (int i = tid; i < kHid; i += kDwThreads)
      db[i] = (red[i] + red[kHid + i]) + (red[2 * kHid + i] + red[3 * kHid + i]);
    return;
  }

  // this tile's operands: A the output-side gradients, B the inputs
  const __nv_bfloat16 *A, *Bm;
  int lda, ldb, m0, n0, M, ldw;
  size_t off;
  if (t < 4) {
    A = a.dout_b; lda = kOut; m0 = 0; M = kOut; Bm = a.h2; ldb = kHid; n0 = t * 64; off = kOffW3; ldw = kHid;
  } else if (t < 12) {
    A = a.dh2; lda = kHid; m0 = ((t - 4) >> 2) * 128; M = 128; Bm = a.h1; ldb = kHid;
    n0 = ((t - 4) & 3) * 64; off = kOffW2; ldw = kHid;
  } else {
    A = a.dh1; lda = kHid; m0 = (t - 12) * 128; M = 128; Bm = a.feat; ldb = kIn; n0 = 0; off = kOffW1; ldw = kIn;
  }
  const uint32_t mb = smem_u32(&mbar);
  auto stage = [&](int k, int buf) {
    unsigned char* p = sm + buf * (128 + 64) * kDwK * 2;
    const int b0 = b_begin + k * kDwK;
    stage_pairs<128>(p, A + m0, lda, M, b0, b_end, tid);
    stage_pairs<64>(p + 128 * kDwK * 2, Bm + n0, ldb, 64, b0, b_end, tid);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int steps = (b_end - b_begin + kDwK - 1) / kDwK;
  stage(0, 0);
  if (warp == 0) tmem_alloc(&tmem_base, 64);
  if (tid == 0) {
    failed = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  for (int k = 0; k < steps; ++k) {
    // step k's products are issued once its operands are in; the wait for
    // step k - 1's frees the buffer that step k + 1 is staged into
    if (k > 0 && !mma_wait(mb, (uint32_t)((k - 1) & 1))) {
      atomicExch(&failed, 1);
      record_status(a.status, PPL_ETIMEOUT);
    }
    if (k + 1 < steps) {
      stage(k + 1, (k + 1) & 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (__syncthreads_or(failed)) break;  // the same for every thread
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = smem_u32(sm + (k & 1) * (128 + 64) * kDwK * 2), sb = sa + 128 * kDwK * 2;
#pragma unroll
      for (int kk = 0; kk < kDwK / 16; ++kk)
        mma_f16(tmem, mma_desc(sa + kk * 256, 128, 1024), mma_desc(sb + kk * 256, 128, 1024),
                idesc(128, 64, true, true), (k > 0 || kk > 0) ? 1u : 0u);
      mma_commit(mb);
    }
  }
  if (!failed && !mma_wait(mb, (uint32_t)((steps - 1) & 1))) {
    atomicExch(&failed, 1);
    record_status(a.status, PPL_ETIMEOUT);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!__syncthreads_or(failed)) {
    const int m = warp * 32 + lane;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float v[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + h * 32, v);
      if (m < M) {
        float4* dst = reinterpret_cast<float4*>(part + off + (size_t)(m0 + m) * ldw + n0 + h * 32);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          dst[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) tmem_free(tmem, 64);
}

// K slices of the 256-wide contractions with N outputs: as many as kept the
// SMs busy and their FP32 tiles within 2^20 words when each slice was a CTA's
// work.  The fused chain has no use for them, but they fix the order of the
// FP32 sums, and with it the last bits of the BF16 activations: a trained
// network goes on giving the outputs it was trained with.
static int k_slices(int64_t B, int N) {
  const int64_t tiles = ((B + kNetRows - 1) / kNetRows) * ((N + kNetN - 1) / kNetN);
  int s = 1;
  while (tiles * s * 2 <= (int64_t)num_sms() * 2 && kHid / (s * 2) >= 64 &&
         s * 2 * B * N <= (int64_t)1 << 20)
    s *= 2;
  return s;
}

cudaError_t launch_net(NetArgs a, cudaStream_t s) {
  int unused = 0;
  const cudaError_t e = device_once((const void*)net_kernel, &unused, [](int*) {
    return cudaFuncSetAttribute(net_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kNetSmem);
  });
  if (e != cudaSuccess) return e;
  const int64_t m_tiles = ((int64_t)a.B + kNetRows - 1) / kNetRows;
  a.slices_hid = k_slices(a.B, kHid);
  a.slices_out = k_slices(a.B, kOut);
  net_kernel<<<(unsigned)m_tiles, kNetThreads, kNetSmem, s>>>(a);
  return cudaGetLastError();
}

int dw_slices(int64_t B) {
  const int64_t want = std::min<int64_t>(kDwSlices, (B + kDwK - 1) / kDwK);
  const int64_t rows = ((B + want - 1) / want + kDwK - 1) / kDwK * kDwK;
  return (int)((B + rows - 1) / rows);
}

cudaError_t launch_dw(const NetArgs& a, cudaStream_t s) {
  const int64_t want = std::min<int64_t>(kDwSlices, ((int64_t)a.B + kDwK - 1) / kDwK);
  const int rows = (int)((((int64_t)a.B + want - 1) / want + kDwK - 1) / kDwK * kDwK);
  dw_kernel<<<dim3(kDwBlocks, (unsigned)dw_slices(a.B)), kDwThreads, 0, s>>>(a, rows);
  return cudaGetLastError();
}

}  // namespace ppl
