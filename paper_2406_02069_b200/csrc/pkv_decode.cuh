// Decode attention over the compact cache of one layer (Section 4.1: after compression only K_s, V_s are used for
// inference): out[b][g] = softmax(q[b][g] . K_s^T / sqrt(d)) V_s for one new token per sequence, packed or paged rows.
//
// What bounds it: the cache is read once, so the floor is its bytes over the memory bandwidth (a few microseconds);
// below that it is a chain of latencies (launch, loads, merges).  The work is therefore split for loads in flight:
//   * one cluster of 1..16 CTAs per (sequence, KV head, block of at most 8 query heads): every K and V row is read once
//     for all query heads of its group, and few long rows lists still spread over the chip.  No scratch memory is
//     needed, the CTAs of a cluster merge through distributed shared memory (this call has no workspace);
//   * inside a CTA a team of D / 8 lanes takes kDecRows rows at a time, 8 elements of a row per lane (16 bytes of a
//     16-bit row), K and V loads of a step issued together;
//   * the row x head dot products of a step are summed over the team's lanes by halving: every exchange also halves the
//     number of values a lane holds, so that reducing n values over L lanes costs about n exchanges instead of
//     n log2 L, and each softmax weight is evaluated once instead of once per lane.
// Everything stays in fp32.  Measured on one B200, one token through 32 layers, 8 KV heads x 4 query heads, d = 128,
// bf16: 2048 rows a head on average, one sequence (269 MB): 8.8 ms with one CTA per query head (32 CTAs, each K and V
// row read four times, a dependent exponential and four exchanges per row), 0.37 ms now (0.46 with clusters of at most
// 8); 512 rows on average, eight sequences, pages of 16 rows (543 MB): 3.3 ms -> 0.40 ms.
#pragma once

#include <cooperative_groups.h>

#include "pkv_common.cuh"
#include "pkv_paged.cuh"

namespace pkv {

constexpr int kDecThreads = 256;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecMaxCluster = 16;
constexpr int kDecMinRows = 64;            // rows a CTA should have before a cluster grows: one step of its teams

struct DecodeParams {
  const void* q;            // [batch][H_q][d], config dtype, contiguous
  const void* k_cache;      // packed rows [sum_b H_kv * c_b][d]; with PAGED the pool [num_pages][page_size][d]
  const void* v_cache;
  PageTable pt;             // PAGED only
  uint32_t* status;         // PAGED only: where a bad table entry is recorded
  float* out;               // [batch][H_q][d] fp32
  SeqTable seq;
  int32_t num_kv_heads, group;
  int32_t head_blocks;      // ceil(group / GT)
  float scale_log2;         // log2(e) / sqrt(d)
};

// Eight consecutive elements of a row, as loaded and as four packed pairs of floats.
template <typename T>
struct Dec8 {
  uint4 u;
  __device__ __forceinline__ void load(const T* p) { u = *reinterpret_cast<const uint4*>(p); }
  __device__ __forceinline__ void zero() { u = make_uint4(0, 0, 0, 0); }
  __device__ __forceinline__ unsigned long long pair(int i) const {
    const uint32_t w = i == 0 ? u.x : (i == 1 ? u.y : (i == 2 ? u.z : u.w));
    if (sizeof(T) == 2 && __is_same(T, __half)) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w));
      return pack2(f.x, f.y);
    }
    return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));      // bfloat16: the upper half of a float
  }
};
template <>
struct Dec8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = reinterpret_cast<const float4*>(p)[0];
    b = reinterpret_cast<const float4*>(p)[1];
  }
  __device__ __forceinline__ void zero() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ unsigned long long pair(int i) const {
    return i == 0 ? pack2(a.x, a.y) : (i == 1 ? pack2(a.z, a.w) : (i == 2 ? pack2(b.x, b.y) : pack2(b.z, b.w)));
  }
};

// grid (cluster * H_kv * head_blocks, batch), cluster (cluster, 1, 1), block kDecThreads.  GT: query heads per CTA (a
// power of two; heads beyond the group are computed on zeros and not written).
template <typename T, int D, int GT, bool PAGED>
__global__ void __launch_bounds__(kDecThreads) decode_attention_kernel(const DecodeParams p) {
  constexpr int L = D / 8;                       // lanes per row
  constexpr int RPW = 32 / L;                    // teams per warp
  constexpr int TEAMS = kDecWarps * RPW;
  constexpr int U = GT == 1 ? 8 : 4;             // rows per team and step
  constexpr int NV = U * GT;                     // dot products of a step
  constexpr int PER = NV > L ? NV / L : 1;       // ... of which a lane ends up with this many (consecutive ones)
  constexpr int SHARE = NV < L ? L / NV : 1;     // ... or this many lanes hold the same one
  static_assert(PER <= U, "a lane's values belong to one head");
  namespace cg = cooperative_groups;
  __shared__ float s_acc[kDecWarps][GT * D];
  __shared__ float s_m[kDecWarps][GT], s_z[kDecWarps][GT];
  __shared__ float s_cm[GT], s_cz[GT];
  pdl_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = cluster.dim_blocks().x, rank = cluster.block_rank();
  const int unit = blockIdx.x / C, b = blockIdx.y;
  const int h = unit / p.head_blocks, g0 = (unit % p.head_blocks) * GT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sub = lane & (L - 1), team = warp * RPW + lane / L;
  const int count = p.seq.count[b];
  const int64_t row0 = p.seq.row_off[b] + static_cast<int64_t>(h) * count;
  const int lo = static_cast<int>(static_cast<int64_t>(count) * rank / C);
  const int hi = static_cast<int>(static_cast<int64_t>(count) * (rank + 1) / C);
  const int64_t hq0 = static_cast<int64_t>(b) * p.num_kv_heads * p.group + static_cast<int64_t>(h) * p.group + g0;
  pdl_wait();

  unsigned long long q2[GT][4], acc[GT][4];
#pragma unroll
  for (int g = 0; g < GT; ++g) {
    Dec8<T> raw;
    if (g0 + g < p.group) raw.load(static_cast<const T*>(p.q) + (hq0 + g) * D + sub * 8);
    else raw.zero();
#pragma unroll
    for (int c = 0; c < 4; ++c) { q2[g][c] = raw.pair(c); acc[g][c] = 0ull; }
  }
  const int my_head = sub * PER / SHARE / U;     // head of the dot products this lane ends up with (see the halving below)
  const int my_row = (sub * PER / SHARE) % U;    // ... and the row of the first of them
  float m = -INFINITY, z = 0.f;                  // of head my_head: m over the team's rows, z over this lane's

  for (int r0 = lo; r0 < hi; r0 += U * TEAMS) {
    Dec8<T> kr[U], vr[U];
    uint32_t live = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = r0 + u * TEAMS + team;
      int64_t at = r < hi ? row0 + r : -1;
      if (PAGED && r < hi) {
        at = paged_row(p.pt, b, h, r);
        if (at < 0 && sub == 0) atomicOr(p.status, kStatusBadPage);
      }
      if (at >= 0) {
        kr[u].load(static_cast<const T*>(p.k_cache) + at * D + sub * 8);
        vr[u].load(static_cast<const T*>(p.v_cache) + at * D + sub * 8);
        live |= 1u << u;
      } else {
        kr[u].zero();
        vr[u].zero();
      }
    }
    float val[NV];                               // index g * U + u
#pragma unroll
    for (int u = 0; u < U; ++u) {
      unsigned long long k2[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) k2[c] = kr[u].pair(c);
#pragma unroll
      for (int g = 0; g < GT; ++g) {
        unsigned long long d = mul2(q2[g][0], k2[0]);
#pragma unroll
        for (int c = 1; c < 4; ++c) d = fma2(q2[g][c], k2[c], d);
        float x, y;
        unpack2(d, x, y);
        val[g * U + u] = x + y;
      }
    }
    // sum over the team's lanes: the lane bit s picks the half of the values a lane keeps, highest bit first
    {
      int cnt = NV;
#pragma unroll
      for (int s = L / 2; s >= 1; s >>= 1) {
        if (cnt > 1) {
          const int half = cnt / 2;
          const bool upper = (sub & s) != 0;
#pragma unroll
          for (int i = 0; i < NV / 2; ++i)
            if (i < half) {
              const float send = upper ? val[i] : val[i + half];
              const float keep = upper ? val[i + half] : val[i];
              val[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
            }
          cnt = half;
        } else {
          val[0] += __shfl_xor_sync(0xffffffffu, val[0], s);
        }
      }
    }
    // softmax weights of this lane's values; the reference exponent of a head is the team's running maximum
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      val[i] = ((live >> (my_row + i)) & 1u) ? val[i] * p.scale_log2 : -INFINITY;
      mx = fmaxf(mx, val[i]);
    }
#pragma unroll
    for (int s = SHARE; s < SHARE * (U / PER); s <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    const float mn = fmaxf(m, mx);
    const float ref = mn == -INFINITY ? 0.f : mn;
    const float corr = exp2f(m - ref);
    const bool grew = mn > m;
    z *= corr;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      val[i] = exp2f(val[i] - ref);
      z += val[i];
    }
    m = mn;
    if (__any_sync(0xffffffffu, grew)) {
#pragma unroll
      for (int g = 0; g < GT; ++g) {
        const float f = __shfl_sync(0xffffffffu, corr, g * U / PER * SHARE, L);
        const unsigned long long f2 = pack2(f, f);
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[g][c] = mul2(acc[g][c], f2);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      unsigned long long v2[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) v2[c] = vr[u].pair(c);
#pragma unroll
      for (int g = 0; g < GT; ++g) {
        const int i = g * U + u;
        const float w = __shfl_sync(0xffffffffu, val[i % PER], i / PER * SHARE, L);
        const unsigned long long w2 = pack2(w, w);
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[g][c] = fma2(w2, v2[c], acc[g][c]);
      }
    }
  }

  // ---- the teams of a warp, then the warps, then the CTAs of the cluster
#pragma unroll
  for (int s = SHARE; s < SHARE * (U / PER); s <<= 1) z += __shfl_xor_sync(0xffffffffu, z, s);
  float mw = m;
#pragma unroll
  for (int s = L; s < 32; s <<= 1) mw = fmaxf(mw, __shfl_xor_sync(0xffffffffu, mw, s));
  const float scale = m == -INFINITY ? 0.f : exp2f(m - mw);
  z *= scale;
#pragma unroll
  for (int s = L; s < 32; s <<= 1) z += __shfl_xor_sync(0xffffffffu, z, s);
#pragma unroll
  for (int g = 0; g < GT; ++g) {
    const float f = __shfl_sync(0xffffffffu, scale, g * U / PER * SHARE, L);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float x, y;
      unpack2(acc[g][c], x, y);
      x *= f;
      y *= f;
#pragma unroll
      for (int s = L; s < 32; s <<= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, s);
        y += __shfl_xor_sync(0xffffffffu, y, s);
      }
      if (lane < L) *reinterpret_cast<float2*>(&s_acc[warp][g * D + sub * 8 + 2 * c]) = make_float2(x, y);
    }
  }
  if (lane < L && sub % (L / GT) == 0) {         // one lane per head
    s_m[warp][my_head] = mw;
    s_z[warp][my_head] = z;
  }
  __syncthreads();
  for (int o = tid; o < GT * D; o += kDecThreads) {
    const int g = o / D;
    float mm = -INFINITY;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) mm = fmaxf(mm, s_m[w][g]);
    float zz = 0.f, a = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) {
      if (s_m[w][g] == -INFINITY) continue;      // the warp saw no row
      const float f = exp2f(s_m[w][g] - mm);
      zz += s_z[w][g] * f;
      a += s_acc[w][o] * f;
    }
    if (C == 1) {
      if (g0 + g < p.group) p.out[hq0 * D + o] = a / zz;
    } else {
      s_acc[0][o] = a;                           // only this thread reads these entries
      if (o % D == 0) { s_cm[g] = mm; s_cz[g] = zz; }
    }
  }
  if (C == 1) return;
  cluster.sync();
  for (int o = rank * kDecThreads + tid; o < GT * D; o += C * kDecThreads) {
    const int g = o / D;
    if (g0 + g >= p.group) continue;
    float mm = -INFINITY, zz = 0.f, a = 0.f;
    for (int c = 0; c < C; ++c) mm = fmaxf(mm, *cluster.map_shared_rank(&s_cm[g], c));
    for (int c = 0; c < C; ++c) {
      const float mc = *cluster.map_shared_rank(&s_cm[g], c);
      if (mc == -INFINITY) continue;
      const float f = exp2f(mc - mm);
      zz += *cluster.map_shared_rank(&s_cz[g], c) * f;
      a += *cluster.map_shared_rank(&s_acc[0][o], c) * f;
    }
    p.out[hq0 * D + o] = a / zz;
  }
  cluster.sync();                                // nobody reads this CTA's shared memory any more
}

}  // namespace pkv
