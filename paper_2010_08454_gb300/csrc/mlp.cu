// The learned proposal's network: forward simulation of training pairs from
// the line-fitting model (Fig. 1), the features of a data set, the BF16
// tensor-core MLP (FP32 accumulation), the loss -log q(n, c | data) and its
// gradient, backpropagation and Adam (FP32 master weights).  The proposal is
// the inference-compilation construction (Le, Baydin and Wood, AISTATS 2017);
// importance weights correct it to the posterior (§3.6.2).
//
// Network and proposal (identical to the definitions the oracle restates):
//   in[64]  = the 32 points sorted by x (ties by position): (x, y / 10), BF16
//   h1 = relu(W1 in + b1), h2 = relu(W2 h1 + b2) (BF16), out = W3 h2 + b3 (FP32)
//   q(k) = softmax(out[0..n_deg))_k; for coefficient j of degree slot k:
//   mu = prior_sigma out[4 + 2 (base_k + j)], s = prior_sigma exp(t),
//   t = clamp(out[5 + 2 (base_k + j)], -9, 1).
#include <cuda_bf16.h>

#include "kernels.h"
#include "mlp.cuh"
#include "poly.cuh"
#include "rng.cuh"

namespace ppl {

// ---------------------------------------------------------------------------
// Features: one warp per data set; lane l holds point l; bitonic sort by
// (x, original position) with shuffles; lane l writes features 2l, 2l + 1.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void warp_features(float x, float y, int lane, __nv_bfloat16* feat) {
  int idx = lane;
#pragma unroll
  for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const float ox = __shfl_xor_sync(0xffffffffu, x, j);
      const float oy = __shfl_xor_sync(0xffffffffu, y, j);
      const int oi = __shfl_xor_sync(0xffffffffu, idx, j);
      const bool other_smaller = (ox < x) || (ox == x && oi < idx);
      const bool ascending = (lane & k) == 0;
      const bool lower = (lane & j) == 0;
      const bool take = (lower == ascending) ? other_smaller : !other_smaller;
      if (take) {
        x = ox;
        y = oy;
        idx = oi;
      }
    }
  }
  feat[2 * lane] = __float2bfloat16_rn(x);
  feat[2 * lane + 1] = __float2bfloat16_rn(__fdiv_rn(y, 10.0f));
}

__global__ void __launch_bounds__(kTpb) features_kernel(const float* __restrict__ x,
                                                        const float* __restrict__ y,
                                                        int32_t n_sets,
                                                        __nv_bfloat16* __restrict__ feat) {
  const int warp = (blockIdx.x * kTpb + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= n_sets) return;
  warp_features(x[(int64_t)warp * kPts + lane], y[(int64_t)warp * kPts + lane], lane,
                feat + (int64_t)warp * kIn);
}

// Training pair p (purpose FORWARD_SIM, instance 0): blocks 0, 1 draw the trace
// as a prior trace; block 2 + l draws point l: x = 2 u01(w0) - 1 and
// y = f(x) + obs_sigma BoxMuller(w1, w2).z0.
// With `step` (a training run's device step counter, steps done so far) the
// batch is pairs [(step mod steps_per_epoch) B, + B) instead of [pair0, + B),
// so a run of training steps needs no value from the host.
__global__ void __launch_bounds__(kTpb) forward_sim_kernel(PolyParams p, float obs_sigma,
                                                           uint64_t seed, int64_t pair0,
                                                           int32_t B,
                                                           __nv_bfloat16* __restrict__ feat,
                                                           int32_t* __restrict__ n_out,
                                                           float* __restrict__ c_out,
                                                           const int32_t* step = nullptr,
                                                           int64_t steps_per_epoch = 1) {
  const int warp = (blockIdx.x * kTpb + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= B) return;
  if (step) pair0 = ((int64_t)*step % steps_per_epoch) * B;
  const uint32_t pair = (uint32_t)(pair0 + warp);
  const uint4 a = philox_block(seed, pair, 0, 0, kForwardSim, 0);
  const uint4 b = philox_block(seed, pair, 0, 0, kForwardSim, 1);
  float z[kMaxCoef], c[kMaxCoef];
  box_muller(a.x, a.y, z[0], z[1]);
  box_muller(a.z, a.w, z[2], z[3]);
  box_muller(b.x, b.y, z[4], z[5]);
  const int n = uniform_discrete(b.z, p.min_deg, p.min_deg + p.n_deg - 1);
  const int ncoef = n + p.coef_offset;
#pragma unroll
  for (int k = 0; k < kMaxCoef; ++k) c[k] = (k < ncoef) ? p.prior_sigma * z[k] : 0.0f;
  const uint4 v = philox_block(seed, pair, 0, 0, kForwardSim, 2 + (uint32_t)lane);
  const float xl = __fsub_rn(__fmul_rn(2.0f, u01(v.x)), 1.0f);
  float e0, e1;
  box_muller(v.y, v.z, e0, e1);
  float f = c[5];
#pragma unroll
  for (int k = 4; k >= 0; --k) f = fmaf(f, xl, c[k]);
  const float yl = fmaf(obs_sigma, e0, f);
  warp_features(xl, yl, lane, feat + (int64_t)warp * kIn);
  if (lane == 0) n_out[warp] = n;
  if (lane < kMaxCoef) c_out[(int64_t)warp * kMaxCoef + lane] = c[lane];
}

// A parameter's gradient: the sum of its batch slices, in order.
__device__ __forceinline__ float slice_sum(const float* __restrict__ partial, int S, int64_t i) {
  float g = 0.0f;
#pragma unroll 4
  for (int z = 0; z < S; ++z) g += partial[(size_t)z * kNumParams + i];
  return g;
}

__global__ void __launch_bounds__(kTpb) grad_kernel(const float* __restrict__ partial, int S,
                                                    float* __restrict__ grad) {
  const int64_t i = (int64_t)blockIdx.x * kTpb + threadIdx.x;
  if (i < (int64_t)kNumParams) grad[i] = slice_sum(partial, S, i);
}

// Adam (Kingma and Ba 2015) on the FP32 master parameters; refreshes the BF16
// copy of the weights.  step = 1, 2, ... for the bias corrections.
__global__ void __launch_bounds__(kTpb) adam_kernel(float* __restrict__ p,
                                                    const float* __restrict__ partial, int S,
                                                    float* __restrict__ m, float* __restrict__ v,
                                                    __nv_bfloat16* __restrict__ pb, int64_t n,
                                                    float lr, float b1, float b2, float eps,
                                                    const int32_t* step) {
  const int64_t i = (int64_t)blockIdx.x * kTpb + threadIdx.x;
  if (i >= n) return;
  const float t = (float)(*step);
  const float gi = slice_sum(partial, S, i);
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float mh = mi / (1.0f - powf(b1, t)), vh = vi / (1.0f - powf(b2, t));
  const float pi = p[i] - lr * mh / (sqrtf(vh) + eps);
  p[i] = pi;
  pb[i] = __float2bfloat16_rn(pi);
}

__global__ void to_bf16_kernel(const float* __restrict__ p, __nv_bfloat16* __restrict__ pb,
                               int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * kTpb + threadIdx.x;
  if (i < n) pb[i] = __float2bfloat16_rn(p[i]);
}

// ---------------------------------------------------------------------------
// Workspace of the network for a batch of B rows.
// ---------------------------------------------------------------------------
struct MlpWs {
  int32_t* status;  // first word: a tensor-core wait that ran out (ppl_workspace_status)
  __nv_bfloat16 *pb, *feat, *h1, *h2, *dout_b, *dh2, *dh1;
  float *dout, *partial, *warp_loss;
  int32_t* n_t;
  float* c_t;
  double* loss;
  int32_t* step;
  size_t total;
};

static size_t a256(size_t v) { return (v + 255) / 256 * 256; }

// The status word is the workspace's first; the step counter and the loss
// follow it, and the arrays start at the next 256-byte address, so that the
// kernels' 16-byte accesses are aligned wherever the caller's workspace lies.
static MlpWs mlp_ws(char* base, int64_t B) {
  constexpr size_t kHead = 768;  // the head and the arrays' alignment
  const size_t start = base ? a256(reinterpret_cast<uintptr_t>(base) + 64) -
                                  reinterpret_cast<uintptr_t>(base) : 0;
  MlpWs w;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base ? base + start + off : nullptr;
    off += a256(bytes);
    return p;
  };
  // 8-byte aligned, past the status word
  char* head = base ? reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(base) + 4 + 7) / 8 * 8)
                    : nullptr;
  w.status = reinterpret_cast<int32_t*>(base);
  w.loss = reinterpret_cast<double*>(head);
  w.step = reinterpret_cast<int32_t*>(head ? head + 8 : nullptr);
  w.pb = (__nv_bfloat16*)take(kNumParams * 2);
  w.feat = (__nv_bfloat16*)take(B * kIn * 2);
  w.h1 = (__nv_bfloat16*)take(B * kHid * 2);
  w.h2 = (__nv_bfloat16*)take(B * kHid * 2);
  w.dout = (float*)take(B * kOut * 4);
  w.dout_b = (__nv_bfloat16*)take(B * kOut * 2);
  w.dh2 = (__nv_bfloat16*)take(B * kHid * 2);
  w.dh1 = (__nv_bfloat16*)take(B * kHid * 2);
  w.n_t = (int32_t*)take(B * 4);
  w.c_t = (float*)take(B * kMaxCoef * 4);
  w.warp_loss = (float*)take((size_t)((B + 127) / 128) * 4 * 4);
  w.partial = (float*)take((size_t)kDwSlices * kNumParams * 4);
  w.total = off + kHead;
  return w;
}

static NetArgs net_args(const float* params, const MlpWs& w, int B) {
  NetArgs a{};
  a.params = params;
  a.pb = w.pb;
  a.feat = w.feat;
  a.B = B;
  a.status = w.status;
  return a;
}

// Forward, loss and gradients of B pairs (w.feat, w.n_t, w.c_t): the weight
// gradients' slices into w.partial, the summed loss into *w.loss.
static cudaError_t mlp_backward(const float* params, const ProposalShape& q, const MlpWs& w, int B,
                                int32_t* step, double* loss_out, cudaStream_t s) {
  NetArgs a = net_args(params, w, B);
  a.backward = 1;
  a.shape = q;
  a.n_t = w.n_t;
  a.c_t = w.c_t;
  a.h1 = w.h1;
  a.h2 = w.h2;
  a.dh2 = w.dh2;
  a.dh1 = w.dh1;
  a.dout = w.dout;
  a.dout_b = w.dout_b;
  a.warp_loss = w.warp_loss;
  a.partial = w.partial;
  a.loss = w.loss;
  a.step = step;
  a.loss_out = loss_out;
  const cudaError_t e = launch_net(a, s);
  return e != cudaSuccess ? e : launch_dw(a, s);
}

static ProposalShape shape_of(const PolyParams& p, float prior_sigma) {
  ProposalShape q;
  q.min_deg = p.min_deg;
  q.n_deg = p.n_deg;
  q.coef_offset = p.coef_offset;
  q.prior_sigma = prior_sigma;
  q.log_prior_sigma = logf(prior_sigma);
  return q;
}

}  // namespace ppl

using namespace ppl;

namespace {

ppl_status mlp_model(const ppl_model* m, PolyParams* p) {
  if (!m || m->id != PPL_MODEL_POLY) return PPL_EINVAL;
  const int n_deg = m->max_deg - m->min_deg + 1;
  if (m->min_deg < 0 || n_deg < 1 || n_deg > kMaxDegrees || m->coef_offset < 0 ||
      m->max_deg + m->coef_offset > kMaxCoef || !(m->obs_sigma > 0.0f) ||
      !(m->prior_sigma > 0.0f))
    return PPL_EINVAL;
  // the 48 outputs hold 4 logits and (mu, log s) for at most 22 coefficient slots
  int slots = 0;
  for (int k = 0; k < n_deg; ++k) slots += m->min_deg + k + m->coef_offset;
  if (4 + 2 * slots > kOut) return PPL_EINVAL;
  p->min_deg = m->min_deg;
  p->n_deg = n_deg;
  p->coef_offset = m->coef_offset;
  p->prior_sigma = m->prior_sigma;
  p->neg_half_inv_var = (float)(-1.0 / (2.0 * (double)m->obs_sigma * (double)m->obs_sigma));
  return PPL_OK;
}

inline ppl_status st(cudaError_t e) { return e == cudaSuccess ? PPL_OK : PPL_ECUDA; }

}  // namespace

extern "C" {

int64_t ppl_proposal_num_params(void) { return (int64_t)kNumParams; }

size_t ppl_proposal_workspace_size(int32_t batch) {
  if (batch < 1) return 0;
  return mlp_ws(nullptr, batch).total;
}

ppl_status ppl_proposal_forward(const ppl_model* model, const float* params, const float* x,
                                const float* y, int32_t n_sets, float* out_dev, void* ws,
                                size_t ws_bytes, ppl_stream stream) {
  PolyParams p;
  if (mlp_model(model, &p) != PPL_OK || !params || !x || !y || !out_dev || n_sets < 1 || !ws)
    return PPL_EINVAL;
  MlpWs w = mlp_ws(static_cast<char*>(ws), n_sets);
  if (ws_bytes < w.total) return PPL_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(w.status, 0, sizeof(int32_t), s) != cudaSuccess) return PPL_ECUDA;
  to_bf16_kernel<<<(unsigned)((kNumParams + kTpb - 1) / kTpb), kTpb, 0, s>>>(params, w.pb,
                                                                            kNumParams);
  features_kernel<<<(unsigned)(((int64_t)n_sets * 32 + kTpb - 1) / kTpb), kTpb, 0, s>>>(
      x, y, n_sets, w.feat);
  NetArgs a = net_args(params, w, n_sets);
  a.out = out_dev;
  return st(launch_net(a, s));
}

ppl_status ppl_proposal_features(const float* x, const float* y, int32_t n_sets, void* feat_dev,
                                 ppl_stream stream) {
  if (!x || !y || !feat_dev || n_sets < 1) return PPL_EINVAL;
  features_kernel<<<(unsigned)(((int64_t)n_sets * 32 + kTpb - 1) / kTpb), kTpb, 0,
                    (cudaStream_t)stream>>>(x, y, n_sets,
                                            static_cast<__nv_bfloat16*>(feat_dev));
  return st(cudaGetLastError());
}

ppl_status ppl_proposal_grad(const ppl_model* model, const float* params, int64_t pair0,
                             int32_t batch, uint64_t seed, float* grad_out, double* loss_out,
                             void* ws, size_t ws_bytes, ppl_stream stream) {
  PolyParams p;
  if (mlp_model(model, &p) != PPL_OK || !params || !grad_out || !loss_out || batch < 1 || !ws ||
      pair0 < 0 || pair0 + batch > 0xffffffffll)
    return PPL_EINVAL;
  MlpWs w = mlp_ws(static_cast<char*>(ws), batch);
  if (ws_bytes < w.total) return PPL_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(w.status, 0, sizeof(int32_t), s) != cudaSuccess) return PPL_ECUDA;
  to_bf16_kernel<<<(unsigned)((kNumParams + kTpb - 1) / kTpb), kTpb, 0, s>>>(params, w.pb,
                                                                            kNumParams);
  forward_sim_kernel<<<(unsigned)(((int64_t)batch * 32 + kTpb - 1) / kTpb), kTpb, 0, s>>>(
      p, model->obs_sigma, seed, pair0, batch, w.feat, w.n_t, w.c_t);
  w.loss = loss_out;
  const ppl_status r = st(mlp_backward(params, shape_of(p, model->prior_sigma), w, batch, nullptr,
                                       nullptr, s));
  if (r != PPL_OK) return r;
  grad_kernel<<<(unsigned)((kNumParams + kTpb - 1) / kTpb), kTpb, 0, s>>>(
      w.partial, dw_slices(batch), grad_out);
  return st(cudaGetLastError());
}

ppl_status ppl_proposal_train_init(const float* params, int32_t batch, void* ws,
                                   size_t ws_bytes, ppl_stream stream) {
  if (!params || batch < 1 || !ws) return PPL_EINVAL;
  MlpWs w = mlp_ws(static_cast<char*>(ws), batch);
  if (ws_bytes < w.total) return PPL_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(w.status, 0, sizeof(int32_t), s) != cudaSuccess ||
      cudaMemsetAsync(w.step, 0, sizeof(int32_t), s) != cudaSuccess)
    return PPL_ECUDA;
  to_bf16_kernel<<<(unsigned)((kNumParams + kTpb - 1) / kTpb), kTpb, 0, s>>>(params, w.pb,
                                                                            kNumParams);
  return st(cudaGetLastError());
}

ppl_status ppl_proposal_train_steps(const ppl_model* model, float* params, float* adam_m,
                                    float* adam_v, int64_t n_pairs, int32_t batch,
                                    int32_t n_steps, uint64_t seed, float lr,
                                    double* loss_per_step, void* ws, size_t ws_bytes,
                                    ppl_stream stream) {
  PolyParams p;
  if (mlp_model(model, &p) != PPL_OK || !params || !adam_m || !adam_v || batch < 1 ||
      n_pairs < batch || n_steps < 0 || !ws || !(lr > 0.0f) || n_pairs > 0xffffffffll)
    return PPL_EINVAL;
  MlpWs w = mlp_ws(static_cast<char*>(ws), batch);
  if (ws_bytes < w.total) return PPL_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  const ProposalShape q = shape_of(p, model->prior_sigma);
  const int64_t steps_per_epoch = n_pairs / batch;
  for (int32_t it = 0; it < n_steps; ++it) {
    forward_sim_kernel<<<(unsigned)(((int64_t)batch * 32 + kTpb - 1) / kTpb), kTpb, 0, s>>>(
        p, model->obs_sigma, seed, 0, batch, w.feat, w.n_t, w.c_t, w.step, steps_per_epoch);
    const ppl_status r = st(mlp_backward(params, q, w, batch, w.step, loss_per_step, s));
    if (r != PPL_OK) return r;
    adam_kernel<<<(unsigned)((kNumParams + kTpb - 1) / kTpb), kTpb, 0, s>>>(
        params, w.partial, dw_slices(batch), adam_m, adam_v, w.pb, kNumParams, lr, 0.9f, 0.999f,
        1e-8f, w.step);
  }
  return st(cudaGetLastError());
}

ppl_status ppl_proposal_train(const ppl_model* model, float* params, float* adam_m,
                              float* adam_v, int64_t n_pairs, int32_t batch, int32_t epochs,
                              uint64_t seed, float lr, double* loss_per_step, void* ws,
                              size_t ws_bytes, ppl_stream stream) {
  if (epochs < 1 || batch < 1 || n_pairs < batch) return PPL_EINVAL;
  const int64_t steps = (int64_t)epochs * (n_pairs / batch);
  if (steps > 0x7fffffffll) return PPL_EINVAL;
  ppl_status r = ppl_proposal_train_init(params, batch, ws, ws_bytes, stream);
  if (r != PPL_OK) return r;
  return ppl_proposal_train_steps(model, params, adam_m, adam_v, n_pairs, batch, (int32_t)steps,
                                  seed, lr, loss_per_step, ws, ws_bytes, stream);
}

}  // extern "C"
