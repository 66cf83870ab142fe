// The attention-recall diagnostic (appendix on attention recall).
#pragma once

#include "pkv_common.cuh"

namespace pkv {

struct RecallParams {
  const float* scores;      // [batch][H_kv][ld]
  int64_t ld_scores;
  const int32_t* indices;   // packed rows
  float* recall;            // [batch][H_kv]
  SeqTable seq;
  int32_t num_kv_heads;
};

// grid (H_kv, batch), block 256.  Share of the window's attention that falls on kept keys:
//   recall = 1 - (sum of the scores of the evicted prefix keys) / alpha,
// because every window row's attention sums to one over the prefix and window keys, and window keys are kept.
__global__ void __launch_bounds__(256) attention_recall_kernel(const RecallParams p) {
  __shared__ float part[2][8];
  pdl_trigger();
  pdl_wait();
  const int h = blockIdx.x, b = blockIdx.y;
  const int alpha = p.seq.alpha, P = p.seq.n[b] - alpha, count = p.seq.count[b], k = count - alpha;
  const float* s = p.scores + (static_cast<int64_t>(b) * p.num_kv_heads + h) * p.ld_scores;
  const int32_t* idx = p.indices + p.seq.row_off[b] + static_cast<int64_t>(h) * count;
  float all = 0.f, kept = 0.f;
  for (int i = threadIdx.x; i < P; i += 256) all += s[i];
  for (int j = threadIdx.x; j < k; j += 256) {
    const int i = idx[j];
    if (i >= 0 && i < P) kept += s[i];                      // an entry that is no prefix position counts as not kept
  }
  for (int o = 16; o > 0; o >>= 1) {
    all += __shfl_xor_sync(0xffffffffu, all, o);
    kept += __shfl_xor_sync(0xffffffffu, kept, o);
  }
  if ((threadIdx.x & 31) == 0) { part[0][threadIdx.x >> 5] = all; part[1][threadIdx.x >> 5] = kept; }
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.f, kk = 0.f;
    for (int w = 0; w < 8; ++w) { a += part[0][w]; kk += part[1][w]; }
    p.recall[b * p.num_kv_heads + h] = 1.0f - (a - kk) / static_cast<float>(alpha);
  }
}

}  // namespace pkv
