// Learned codec selector: batched inference and full-batch training of the per-block
// MLP (8 -> 32 -> 32 -> 3, ReLU) that predicts log2 bits per element of each codec.
// Training rows come from the method itself (csz_selector_rows: features and exact
// encoded sizes of every block).  The loss is the mean over rows and outputs of the
// squared error; the optimiser is Adam.
//
// Kernel layout: one warp per pair of rows at a time, lane i owning hidden unit i of both
// layers, so the activations go to every lane through shared memory and the backward
// pass accumulates each lane's rows of dW1 and dW2 in registers.  Partial
// sums per CTA go to the workspace and are added in a fixed order by the update
// kernel, so a training run is reproducible bit for bit on one GPU model.
#include <cmath>
#include <cstring>

#include "cszp.h"
#include "kernels.h"

namespace cszp {
namespace {

constexpr int kTrainThreads = 384;
constexpr int kTrainWarps = kTrainThreads / 32;
constexpr int kPart = kMlpParams + 2;  // gradient sums, loss sum, row count
constexpr float kAdamB1 = 0.9f, kAdamB2 = 0.999f, kAdamEps = 1e-8f;

__global__ __launch_bounds__(256) void mlp_predict_kernel(const float* __restrict__ w,
                                                          const float* __restrict__ feat, uint64_t n,
                                                          float* __restrict__ out) {
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const int lane = threadIdx.x & 31;
  for (uint64_t r = warp; r < n; r += nwarps) {
    float f[kMlpIn];
#pragma unroll
    for (int j = 0; j < kMlpIn; j++) f[j] = __ldg(&feat[r * kMlpIn + j]);
    float y[kMlpOut];
    mlp_forward_warp(w, f, y);
    const float mine = lane == 0 ? y[0] : (lane == 1 ? y[1] : y[2]);
    if (lane < kMlpOut) out[r * kMlpOut + lane] = mine;
  }
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(~0u, v, o);
  return v;
}

// Forward and backward over rows gw, gw + nw, ... of every warp; per-CTA sums of the
// unscaled gradient (d(e^2)/dy = 2e), of e^2 and of the row count go to part[cta].
//
// Bound by instruction issue (about 200 warp instructions a row) and, with few warps an SM
// for the registers the weights take, by the chains in between.  A row's activations reach
// the 32 lanes as 16-byte shared-memory words (a shuffle each, 64 a row, kept the one
// shuffle result a cycle and SM busy for half the time) and are read again for dW2 instead
// of held, which leaves registers for 12 warps an SM where 198 a thread left 8; and a warp
// works on two rows at once.  Rows that take no part are skipped by a ballot over 32 of
// them.  A training step on 28,672 rows, with the update below: 35 -> 21 us.
//
// Lane i owns row i of W2 and dW2, whose packed layout puts the 32 lanes' words in 32 cache
// lines (and one bank): the parameters are staged in shared memory with W2's rows padded to
// 33 words, and dW2 is handed over transposed with the same padding, so that neither the
// loads nor the reduction serialise.
constexpr int kPitch = kMlpHid + 1;
constexpr int kStage = kMlpHid * (kPitch - kMlpHid);  // words the padding adds
// a parameter's word in the padded layout: W2's entries at pitch 33
__device__ __forceinline__ int padded(int p) {
  return p < kMlpW2 ? p : (p < kMlpB2 ? p + (p - kMlpW2) / kMlpHid : p + kStage);
}
// the same for the sums, which hold dW2 transposed
__device__ __forceinline__ int padded_t(int p) {
  if (p < kMlpW2 || p >= kMlpB2) return padded(p);
  const int k = p - kMlpW2;
  return kMlpW2 + (k % kMlpHid) * kPitch + k / kMlpHid;
}
// One row's sums over the lanes' hidden units, four independent chains
__device__ __forceinline__ float dot32(const float (&w)[kMlpHid], const float* s, float first) {
  float acc[4] = {first, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int j = 0; j < kMlpHid; j += 4) {
    const float4 v = *reinterpret_cast<const float4*>(s + j);
    acc[0] = fmaf(w[j], v.x, acc[0]);
    acc[1] = fmaf(w[j + 1], v.y, acc[1]);
    acc[2] = fmaf(w[j + 2], v.z, acc[2]);
    acc[3] = fmaf(w[j + 3], v.w, acc[3]);
  }
  return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

// x becomes the rounded sum of x and y; returns what rounding took from it (Knuth's TwoSum;
// after an infinity a NaN that says nothing).
__device__ __forceinline__ float two_sum(float& x, float y) {
  const float s = __fadd_rn(x, y), b = __fsub_rn(s, x);
  const float e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, b)), __fsub_rn(y, b));
  x = s;
  return e;
}

constexpr int kRedWarps = kTrainWarps / 2;  // the warps' sums meet in two turns
__global__ __launch_bounds__(kTrainThreads) void mlp_grad_kernel(const float* w, const float* feat, const float* tgt,
                                                                 const uint8_t* valid, uint64_t n, float* part) {
  chained_begin();
  __shared__ float s_red[kRedWarps][kPart + kStage];
  __shared__ __align__(16) float s_act[kTrainWarps][4][kMlpHid];  // per warp: h1 and da2 of two rows
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float* sw = s_red[0];  // the staged parameters, until the sums need the words
  for (int p = threadIdx.x; p < kMlpParams; p += kTrainThreads) sw[padded(p)] = w[p];
  __syncthreads();
  float w1[kMlpIn], w2r[kMlpHid], w2c[kMlpHid], w3[kMlpOut], b3[kMlpOut];
  const float b1 = sw[kMlpB1 + lane], b2 = sw[kMlpB2 + kStage + lane];
#pragma unroll
  for (int j = 0; j < kMlpIn; j++) w1[j] = sw[kMlpW1 + lane * kMlpIn + j];
#pragma unroll
  for (int j = 0; j < kMlpHid; j++) {
    w2r[j] = sw[kMlpW2 + lane * kPitch + j];
    w2c[j] = sw[kMlpW2 + j * kPitch + lane];
  }
#pragma unroll
  for (int c = 0; c < kMlpOut; c++) {
    w3[c] = sw[kMlpW3 + kStage + c * kMlpHid + lane];
    b3[c] = sw[kMlpB3 + kStage + c];
  }
  __syncthreads();
  float g1[kMlpIn], g2[kMlpHid], g3[kMlpOut], gb3[kMlpOut];
  float gb1 = 0.0f, gb2 = 0.0f, loss = 0.0f, cnt = 0.0f;
#pragma unroll
  for (int j = 0; j < kMlpIn; j++) g1[j] = 0.0f;
#pragma unroll
  for (int j = 0; j < kMlpHid; j++) g2[j] = 0.0f;
#pragma unroll
  for (int c = 0; c < kMlpOut; c++) g3[c] = gb3[c] = 0.0f;

  float(*act)[kMlpHid] = s_act[wid];
  const uint64_t nw = (uint64_t)gridDim.x * kTrainWarps;
  for (uint64_t r0 = (uint64_t)blockIdx.x * kTrainWarps + wid; r0 < n; r0 += 32 * nw) {
    const uint64_t mine = r0 + lane * nw;
    uint32_t todo = __ballot_sync(~0u, mine < n && (!valid || valid[mine]));
    while (todo) {
      // two of the rows, or one: then the second's place holds zeros from its inputs to its
      // errors, so that it adds nothing whatever the weights and the first row's values are
      // (a repeated row times an error of 0 would be a NaN where its activations overflow)
      uint64_t row[2];
      row[0] = r0 + (__ffs(todo) - 1) * nw;
      todo &= todo - 1;
      const bool both = todo != 0;
      row[1] = both ? r0 + (__ffs(todo) - 1) * nw : row[0];
      todo &= todo - 1;
      float x[2][kMlpIn], a1[2], a2[2], h2[2], dy[2][kMlpOut], da2[2], da1[2];
      const bool live[2] = {true, both};
      // forward
#pragma unroll
      for (int k = 0; k < 2; k++) {
        a1[k] = b1;
#pragma unroll
        for (int j = 0; j < kMlpIn; j++) x[k][j] = live[k] ? feat[row[k] * kMlpIn + j] : 0.0f;
#pragma unroll
        for (int j = 0; j < kMlpIn; j++) a1[k] = fmaf(w1[j], x[k][j], a1[k]);
        act[k][lane] = live[k] && a1[k] > 0.0f ? a1[k] : 0.0f;
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 2; k++) {
        a2[k] = dot32(w2r, act[k], b2);
        h2[k] = live[k] && a2[k] > 0.0f ? a2[k] : 0.0f;
      }
#pragma unroll
      for (int k = 0; k < 2; k++) {
#pragma unroll
        for (int c = 0; c < kMlpOut; c++) {
          const float y = b3[c] + warp_sum_f(w3[c] * h2[k]);
          const float e = live[k] ? y - tgt[row[k] * kMlpOut + c] : 0.0f;
          loss = fmaf(e, e, loss);
          dy[k][c] = 2.0f * e;
        }
      }
      cnt += both ? 2.0f : 1.0f;
      // backward
#pragma unroll
      for (int k = 0; k < 2; k++) {
        float dh2 = 0.0f;
#pragma unroll
        for (int c = 0; c < kMlpOut; c++) {
          g3[c] = fmaf(dy[k][c], h2[k], g3[c]);
          gb3[c] += dy[k][c];
          dh2 = fmaf(dy[k][c], w3[c], dh2);
        }
        da2[k] = live[k] && a2[k] > 0.0f ? dh2 : 0.0f;
        act[2 + k][lane] = da2[k];
        gb2 += da2[k];
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 2; k++) {
#pragma unroll
        for (int j = 0; j < kMlpHid; j += 4) {
          const float4 h = *reinterpret_cast<const float4*>(&act[k][j]);
          g2[j] = fmaf(da2[k], h.x, g2[j]);
          g2[j + 1] = fmaf(da2[k], h.y, g2[j + 1]);
          g2[j + 2] = fmaf(da2[k], h.z, g2[j + 2]);
          g2[j + 3] = fmaf(da2[k], h.w, g2[j + 3]);
        }
        const float dh1 = dot32(w2c, act[2 + k], 0.0f);
        da1[k] = live[k] && a1[k] > 0.0f ? dh1 : 0.0f;
#pragma unroll
        for (int j = 0; j < kMlpIn; j++) g1[j] = fmaf(da1[k], x[k][j], g1[j]);
        gb1 += da1[k];
      }
      __syncwarp();  // act is free again
    }
  }

  // the sums of warps kRedWarps and up, then those of the others added to them
  for (int turn = 1; turn >= 0; turn--) {
    if (wid / kRedWarps == turn) {
      float* my = s_red[wid % kRedWarps];
      auto put = [&](int at, float v) { my[at] = turn ? v : my[at] + v; };
#pragma unroll
      for (int j = 0; j < kMlpIn; j++) put(kMlpW1 + lane * kMlpIn + j, g1[j]);
      put(kMlpB1 + lane, gb1);
#pragma unroll
      for (int j = 0; j < kMlpHid; j++) put(kMlpW2 + j * kPitch + lane, g2[j]);
      put(kMlpB2 + kStage + lane, gb2);
#pragma unroll
      for (int c = 0; c < kMlpOut; c++) put(kMlpW3 + kStage + c * kMlpHid + lane, g3[c]);
      if (lane == 0) {
#pragma unroll
        for (int c = 0; c < kMlpOut; c++) put(kMlpB3 + kStage + c, gb3[c]);
        put(kStage + kMlpParams, loss);
        put(kStage + kMlpParams + 1, cnt);
      }
    }
    __syncthreads();
  }
  // (rounded once: the CTA's sum has one rounding for every two warps and a last one)
  for (int p = threadIdx.x; p < kPart; p += kTrainThreads) {
    const int q = padded_t(p);
    float acc = s_red[0][q], low = 0.0f;
#pragma unroll
    for (int wv = 1; wv < kRedWarps; wv++) low = __fadd_rn(low, two_sum(acc, s_red[wv][q]));
    part[(uint64_t)blockIdx.x * kPart + p] = isfinite(low) ? __fadd_rn(acc, low) : acc;
  }
}

// A sum in three floats, each holding what rounding took from the one before: 72 bits, more
// than a double's 53.
struct Sum3 {
  float h, m, l;
  __device__ __forceinline__ void add(float x) { l = __fadd_rn(l, two_sum(m, two_sum(h, x))); }
  __device__ __forceinline__ void add(const Sum3& o) {
    add(o.h);
    l = __fadd_rn(l, __fadd_rn(two_sum(m, o.m), o.l));
  }
  __device__ __forceinline__ Sum3 shfl_xor(int o) const {
    return Sum3{__shfl_xor_sync(~0u, h, o), __shfl_xor_sync(~0u, m, o), __shfl_xor_sync(~0u, l, o)};
  }
};

// Sum of the CTA partials, scaled to the mean over rows and outputs; optionally one Adam
// step on the weights.  Parameter kMlpParams is the loss.
//
// Bound by latency, then by issue: the CTAs start as the gradient launch ends, many of them on
// the first SMs that become free.  So a CTA takes 8 parameters: a warp reads 8 of four partials
// at a time (32 bytes each, all in flight) and adds every 32nd, and the sums meet by shuffles
// and through shared memory, always in the same order, so runs stay reproducible.  The sums run
// in three floats: in doubles the FP64 pipe, 2 results a cycle and SM, takes most of the launch
// for converting and adding (50 steps on 28,672 rows: 1186 us in doubles where pairs of floats,
// which hold 48 bits, take 915; in turn with pairs, 849 and 855 us so, and 915 and 936 with 32
// parameters a CTA).  Doubles are left for the last combination and the one scale, and for sums
// that are not finite or overflow a float, which start again in them.  c1, c2: Adam's bias
// corrections of this step.
constexpr int kUpdThreads = 256, kUpdWarps = kUpdThreads / 32, kUpdParams = 8, kMaxParts = 512;
__global__ __launch_bounds__(kUpdThreads) void mlp_update_kernel(const float* part, int nparts, float* w,
                                                                 float* grad_out, double* loss_out, float* m,
                                                                 float* v, uint32_t step, float lr, float c1, float c2) {
  chained_begin();
  __shared__ Sum3 s_sum[kUpdWarps][kUpdParams];
  __shared__ unsigned long long s_c[kUpdWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int p = blockIdx.x * kUpdParams + (lane & 7);
  Sum3 acc{0.0f, 0.0f, 0.0f};
  {
    const int q = min(p, kMlpParams);
#pragma unroll 5
    for (int g = 4 * wid + (lane >> 3); g < nparts; g += 4 * kUpdWarps) acc.add(part[(uint64_t)g * kPart + q]);
  }
  // row counts: whole numbers
  unsigned long long cnt = 0;
  for (int g = threadIdx.x; g < nparts; g += kUpdThreads)
    cnt += (unsigned long long)part[(uint64_t)g * kPart + kMlpParams + 1];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(~0u, cnt, o);
  acc.add(acc.shfl_xor(8));
  acc.add(acc.shfl_xor(16));
  if (lane < kUpdParams) s_sum[wid][lane] = acc;
  if (lane == 0) s_c[wid] = cnt;
  __syncthreads();
  if (wid) return;
  acc = s_sum[lane >> 3][lane & 7];
  acc.add(s_sum[4 + (lane >> 3)][lane & 7]);
  acc.add(acc.shfl_xor(8));
  acc.add(acc.shfl_xor(16));
  cnt = 0;
#pragma unroll
  for (int k = 0; k < kUpdWarps; k++) cnt += s_c[k];
  if (lane >= kUpdParams || p > kMlpParams) return;
  double sum = (double)acc.h + ((double)acc.m + (double)acc.l);
  if (!isfinite(sum)) {
    sum = 0.0;
    for (int g = 0; g < nparts; g++) sum += (double)part[(uint64_t)g * kPart + p];
  }
  const double scale = cnt ? 1.0 / (3.0 * (double)cnt) : 0.0;
  if (p == kMlpParams) {
    if (loss_out) *loss_out = sum * scale;
    return;
  }
  const float gr = (float)(sum * scale);
  if (grad_out) grad_out[p] = gr;
  if (step) {
    const float mt = kAdamB1 * m[p] + (1.0f - kAdamB1) * gr;
    const float vt = kAdamB2 * v[p] + (1.0f - kAdamB2) * gr * gr;
    m[p] = mt;
    v[p] = vt;
    w[p] -= lr * (mt / c1) / (sqrtf(vt / c2) + kAdamEps);
  }
}

int train_grid(uint64_t nrows) {
  const int sms = sm_count();
  // a CTA an SM, or two in turn where a warp would add more than 32 rows into one FP32 sum
  // (its rounding grows with them)
  const uint64_t want = (nrows + 4 * kTrainWarps - 1) / (4 * kTrainWarps);
  const int ctas = nrows > 32ull * kTrainWarps * (uint64_t)sms ? 2 * sms : sms;
  const uint64_t cap = (uint64_t)(ctas < kMaxParts ? ctas : kMaxParts);
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

uint64_t a256(uint64_t v) { return (v + 255) & ~255ull; }

// workspace: partials [grid][kPart] f32 | Adam m, v [params] f32 | loss f64
struct TrainLayout {
  uint64_t part, m, v, loss, total;
};

TrainLayout train_layout(int grid) {
  TrainLayout L;
  L.part = 0;
  L.m = a256((uint64_t)grid * kPart * 4);
  L.v = L.m + a256(kMlpParams * 4);
  L.loss = L.v + a256(kMlpParams * 4);
  L.total = L.loss + 256;
  return L;
}

template <typename T>
T* at(void* base, uint64_t off) {
  return reinterpret_cast<T*>(static_cast<unsigned char*>(base) + off);
}

}  // namespace

cudaError_t launch_mlp_grad(const float* w, const float* feat, const float* tgt, const uint8_t* valid,
                            uint64_t n, float* part, int grid, cudaStream_t s) {
  trace_begin(K_MLP_GRAD, s);
  launch_chained(mlp_grad_kernel, grid, kTrainThreads, 0, s, w, feat, tgt, valid, n, part);
  trace_end(K_MLP_GRAD, s);
  return cudaGetLastError();
}

cudaError_t launch_mlp_update(const float* part, int nparts, float* w, float* grad, double* loss, float* m,
                              float* v, uint32_t step, float lr, cudaStream_t s) {
  trace_begin(K_MLP_UPDATE, s);
  const float c1 = (float)(1.0 - std::pow((double)kAdamB1, (double)step));
  const float c2 = (float)(1.0 - std::pow((double)kAdamB2, (double)step));
  launch_chained(mlp_update_kernel, (kMlpParams + kUpdParams) / kUpdParams, kUpdThreads, 0, s, part, nparts, w, grad, loss, m, v,
                                                                                  step, lr, c1, c2);
  trace_end(K_MLP_UPDATE, s);
  return cudaGetLastError();
}

}  // namespace cszp

using namespace cszp;

extern "C" {

size_t csz_selector_workspace_bytes(uint64_t nrows) { return (size_t)train_layout(train_grid(nrows)).total; }

csz_status csz_selector_predict(const float* d_w, const float* d_feat, uint64_t nrows, float* d_out, void* stream) {
  if (!d_w || (nrows && (!d_feat || !d_out))) return CSZ_E_ARG;
  if (nrows == 0) return CSZ_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint64_t blocks = (nrows + 7) / 8;
  const unsigned grid = (unsigned)(blocks < 4096 ? blocks : 4096);
  trace_begin(K_MLP_PREDICT, s);
  mlp_predict_kernel<<<grid, 256, 0, s>>>(d_w, d_feat, nrows, d_out);
  trace_end(K_MLP_PREDICT, s);
  if (cudaGetLastError() != cudaSuccess) return CSZ_E_CUDA;
  return cudaStreamSynchronize(s) == cudaSuccess ? CSZ_OK : CSZ_E_CUDA;
}

csz_status csz_selector_grad(const float* d_w, const float* d_feat, const float* d_target, const uint8_t* d_valid,
                             uint64_t nrows, float* d_grad, double* h_loss, void* d_ws, size_t ws_bytes,
                             void* stream) {
  if (!d_w || !d_grad || !d_ws || (nrows && (!d_feat || !d_target))) return CSZ_E_ARG;
  const int grid = train_grid(nrows);
  const TrainLayout L = train_layout(grid);
  if (ws_bytes < L.total) return CSZ_E_CAPACITY;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* part = at<float>(d_ws, L.part);
  double* loss = at<double>(d_ws, L.loss);
  if (launch_mlp_grad(d_w, d_feat, d_target, d_valid, nrows, part, grid, s) != cudaSuccess) return CSZ_E_CUDA;
  if (launch_mlp_update(part, grid, nullptr, d_grad, loss, nullptr, nullptr, 0, 0.0f, s) != cudaSuccess)
    return CSZ_E_CUDA;
  double hl = 0.0;
  if (cudaMemcpyAsync(&hl, loss, sizeof(hl), cudaMemcpyDeviceToHost, s) != cudaSuccess) return CSZ_E_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return CSZ_E_CUDA;
  if (h_loss) *h_loss = hl;
  return CSZ_OK;
}

csz_status csz_selector_train(float* d_w, const float* d_feat, const float* d_target, const uint8_t* d_valid,
                              uint64_t nrows, uint32_t steps, float lr, void* d_ws, size_t ws_bytes,
                              double* h_loss, void* stream) {
  if (!d_w || !d_ws || (nrows && (!d_feat || !d_target))) return CSZ_E_ARG;
  if (!(lr > 0.0f) || !std::isfinite(lr)) return CSZ_E_ARG;
  const int grid = train_grid(nrows);
  const TrainLayout L = train_layout(grid);
  if (ws_bytes < L.total) return CSZ_E_CAPACITY;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* part = at<float>(d_ws, L.part);
  float* m = at<float>(d_ws, L.m);
  float* v = at<float>(d_ws, L.v);
  double* loss = at<double>(d_ws, L.loss);
  if (cudaMemsetAsync(m, 0, L.loss - L.m, s) != cudaSuccess) return CSZ_E_CUDA;
  for (uint32_t t = 1; t <= steps; t++) {
    // learning rate decays linearly to a tenth of lr over the run
    const float lr_t = lr * (1.0f - 0.9f * (float)(t - 1) / (float)steps);
    if (launch_mlp_grad(d_w, d_feat, d_target, d_valid, nrows, part, grid, s) != cudaSuccess) return CSZ_E_CUDA;
    if (launch_mlp_update(part, grid, d_w, nullptr, loss, m, v, t, lr_t, s) != cudaSuccess) return CSZ_E_CUDA;
  }
  double hl = 0.0;
  if (steps && cudaMemcpyAsync(&hl, loss, sizeof(hl), cudaMemcpyDeviceToHost, s) != cudaSuccess) return CSZ_E_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return CSZ_E_CUDA;
  if (h_loss) *h_loss = hl;
  return CSZ_OK;
}

}  // extern "C"
