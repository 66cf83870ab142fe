// Decode attention over the compact cache of one layer (Section 4.1: after compression only K_s, V_s are used for
// inference): out[b][g] = softmax(q[b][g] . K_s^T / sqrt(d)) V_s for one new token per sequence, packed or paged rows.
//
// What bounds it: the cache is read once, so the floor is its bytes over the memory bandwidth (a few microseconds);
// below that it is a chain of latencies (launch, loads, merges) and, on the fp32 pipe, the instructions per row: with one
// warp instruction per 2 rows x 8 channels a step of 8 rows took a warp 400 of them.
//   * One cluster of 1..8 CTAs per (sequence, KV head, block of query heads): every K and V row is read once for all
//     query heads of its block, and few long row lists still spread over the chip.  No scratch memory is needed (this
//     call has no workspace): the CTAs hand their sums to one another through distributed shared memory, each channel
//     to the CTA that finishes it, with one cluster barrier.
//   * 16-bit rows go through mma.sync (decode_mma_kernel): M = query heads, fp32 accumulation.  The softmax weights stay
//     fp32 in effect: each is split into three 16-bit parts (hi + mid + lo carry 24 bits and more), which stand in
//     different rows of the same M = 16 operand (4 heads x 3 parts), so that the split costs no extra products.
//     Rows come by asynchronous copies into a ring in shared memory, three tiles of 16 rows per warp: a tile in registers
//     at a time left the warp waiting some 1.1 us for every tile, and took the registers that a second CTA on the SM needs.
//   * fp32 rows stay on the fp32 pipe (decode_attention_kernel).
// Measured on one B200, one token through 32 layers, 8 KV heads x 4 query heads, d = 128, bf16: 2048 rows a head on
// average, one sequence (269 MB): 8.8 ms with one CTA per query head (32 CTAs, each K and V row read four times), 365 us
// with clusters on the fp32 pipe, 258 on mma.sync with rows in registers, 197 with the ring; 512 rows, eight sequences, pages
// of 16 rows (543 MB): 3.3 ms, 397, 319, 247 us.  A call of few rows takes 5 us from one wait for the kernels ahead to the
// next: rows out of the L2 1.2, products and merges of the warps 0.7, the cluster's exchange 1.2, end of the grid 1.7.
#pragma once

#include <cooperative_groups.h>

#include "pkv_common.cuh"
#include "pkv_paged.cuh"

namespace pkv {

constexpr int kDecThreads = 256;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecMaxCluster = 8;         // 16 CTAs need a GPC to themselves: their launches cannot overlap (+4.5 us each)
constexpr int kDecStages = 3;             // tiles of a warp in shared memory or on their way
constexpr int kDecPrefetchRows = 512;     // rows a CTA brings into the L2 while it waits
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

// Eight consecutive floats of a row as four packed pairs.
struct Dec8 {
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

// Shared memory in which the warps of a CTA, then the CTAs of a cluster meet.
template <int D, int GT, int WARPS>
struct DecMerge {
  static constexpr int kHead = D + 4;            // floats from a head's sums to the next one's: other banks
  float acc[WARPS][GT * kHead];
  float m[WARPS][GT], z[WARPS][GT];
  float in[GT * D];                                                              // this CTA's channels, from every CTA
  float2 mz[kDecMaxCluster][GT];                                                 // every CTA's (maximum, sum) per head
};

// Sums relative to 2^m are added up with the factors 2^(m - largest m); a warp or CTA without a row has NaN for m, which fmaxf and
// fminf pass over.  The factors are those of exp2f: ex2 gives its bits, but makes zeros of subnormal numbers, and those
// count where the values are large or infinite, so where one may be subnormal the sums are formed again.  (exp2f throughout:
// 32 layers of 2048 rows 201 us instead of 197, paged 250 either way; no second look, 196 and 247.)
constexpr float kDecLeast = 126.f;
__device__ __forceinline__ float dec_none(float m) { return m == -INFINITY ? __int_as_float(0x7fffffff) : m; }
template <bool SUBNORMAL>
__device__ __forceinline__ float dec_factor(float m, float largest) {
  return m != m ? 0.f : SUBNORMAL ? exp2f(m - largest) : ex2(m - largest);
}

// Sums of the warps (in shared memory behind a barrier) -> output.  hq0: first query head of the block.  The cluster's
// barrier has been arrived at once at the start of the kernel.  C is a power of two, so every CTA finishes GT * D / C channels.
template <int D, int GT, int WARPS>
__device__ __forceinline__ void dec_finish(DecMerge<D, GT, WARPS>& s, const DecodeParams& p, int C, int rank, int64_t hq0, int heads) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  if (C > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");        // every CTA of the cluster has started
  const int share = GT * D / C;                  // channels each CTA finishes
  for (int o = threadIdx.x * 2; o < GT * D; o += WARPS * 64) {                   // two channels of a head
    const int g = o / D;
    float mm = -INFINITY;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) mm = fmaxf(mm, s.m[w][g]);
    float zz = 0.f;
    float2 a = make_float2(0.f, 0.f);
    auto add = [&](int w, float f) {
      const float2 v = *reinterpret_cast<const float2*>(&s.acc[w][g * DecMerge<D, GT, WARPS>::kHead + o % D]);
      zz += s.z[w][g] * f;
      a.x += v.x * f;
      a.y += v.y * f;
    };
    float least = mm;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
      least = fminf(least, s.m[w][g]);
      add(w, dec_factor<false>(s.m[w][g], mm));
    }
    if (mm - least > kDecLeast) {
      zz = a.x = a.y = 0.f;
#pragma unroll 1
      for (int w = 0; w < WARPS; ++w) add(w, dec_factor<true>(s.m[w][g], mm));
    }
    if (C == 1) {
      if (g < heads) {                           // (the output is as aligned as a float)
        p.out[hq0 * D + o] = a.x / zz;
        p.out[hq0 * D + o + 1] = a.y / zz;
      }
    } else {
      const int to = o / share;
      *reinterpret_cast<float2*>(cluster.map_shared_rank(s.in, to) + rank * share + o - to * share) = a;
      if (o == to * share || o % D == 0) cluster.map_shared_rank(&s.mz[0][0], to)[rank * GT + g] = make_float2(dec_none(mm), zz);
    }
  }
  if (C == 1) return;
  cluster.sync();
  for (int i = threadIdx.x; i < share; i += WARPS * 32) {
    const int o = rank * share + i, g = o / D;
    if (g >= heads) continue;
    float2 mz[kDecMaxCluster];
    float in[kDecMaxCluster];
    float mm = -INFINITY, zz = 0.f, a = 0.f;
#pragma unroll
    for (int c = 0; c < kDecMaxCluster; ++c) {
      mz[c] = c < C ? s.mz[c][g] : make_float2(dec_none(-INFINITY), 0.f);
      in[c] = c < C ? s.in[c * share + i] : 0.f;
      mm = fmaxf(mm, mz[c].x);
    }
    float least = mm;
#pragma unroll
    for (int c = 0; c < kDecMaxCluster; ++c) {
      const float f = dec_factor<false>(mz[c].x, mm);
      least = fminf(least, mz[c].x);
      zz += mz[c].y * f;
      a += in[c] * f;
    }
    if (mm - least > kDecLeast) {
      zz = a = 0.f;
#pragma unroll 1
      for (int c = 0; c < C; ++c) {
        const float f = dec_factor<true>(s.mz[c][g].x, mm);
        zz += s.mz[c][g].y * f;
        a += s.in[c * share + i] * f;
      }
    }
    p.out[hq0 * D + o] = a / zz;
  }
}

// fp32 rows.  grid (cluster * H_kv * head_blocks, batch), cluster (cluster, 1, 1), block kDecThreads.  GT: query heads per
// CTA (a power of two; heads beyond the group are computed on zeros and not written).  A team of D / 8 lanes takes four
// (eight) rows at a time, 8 channels of a row per lane.  The row x head dot products of a step are summed over the team's
// lanes by halving: every exchange also halves the number of values a lane holds, so that reducing n values over L lanes
// costs about n exchanges instead of n log2 L, and each softmax weight is evaluated once instead of once per lane.
template <int D, int GT, bool PAGED>
__global__ void __launch_bounds__(kDecThreads) decode_attention_kernel(const DecodeParams p) {
  constexpr int L = D / 8;                       // lanes per row
  constexpr int RPW = 32 / L;                    // teams per warp
  constexpr int TEAMS = kDecWarps * RPW;
  constexpr int U = GT == 1 ? 8 : 4;             // rows per team and step
  constexpr int NV = U * GT;                     // dot products of a step
  constexpr int PER = NV > L ? NV / L : 1;       // ... of which a lane ends up with this many (consecutive ones)
  constexpr int SHARE = NV < L ? L / NV : 1;     // ... or this many lanes hold the same one
  static_assert(PER <= U, "a lane's values belong to one head");
  using T = float;
  namespace cg = cooperative_groups;
  __shared__ DecMerge<D, GT, kDecWarps> s_mrg;
  pdl_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = cluster.dim_blocks().x, rank = cluster.block_rank();
  if (C > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");      // this CTA's shared memory may be written
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
    Dec8 raw;
    if (g0 + g < p.group) raw.load(static_cast<const T*>(p.q) + (hq0 + g) * D + sub * 8);
    else raw.zero();
#pragma unroll
    for (int c = 0; c < 4; ++c) { q2[g][c] = raw.pair(c); acc[g][c] = 0ull; }
  }
  const int my_head = sub * PER / SHARE / U;     // head of the dot products this lane ends up with (see the halving below)
  const int my_row = (sub * PER / SHARE) % U;    // ... and the row of the first of them
  float m = -INFINITY, z = 0.f;                  // of head my_head: m over the team's rows, z over this lane's

  for (int r0 = lo; r0 < hi; r0 += U * TEAMS) {
    Dec8 kr[U], vr[U];
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
      if (lane < L) *reinterpret_cast<float2*>(&s_mrg.acc[warp][g * (D + 4) + sub * 8 + 2 * c]) = make_float2(x, y);
    }
  }
  if (lane < L && sub % (L / GT) == 0) {         // one lane per head
    s_mrg.m[warp][my_head] = dec_none(mw);
    s_mrg.z[warp][my_head] = z;
  }
  __syncthreads();
  dec_finish<D, GT, kDecWarps>(s_mrg, p, C, rank, hq0, p.group - g0);
}

// ------------------------------------------------------------------ 16-bit rows
constexpr int kDecMmaHeads = 4;           // query heads per CTA: 4 heads x 3 parts of the weights in the 16 rows of an MMA

template <typename T>
struct Dec16;
template <>
struct Dec16<__nv_bfloat16> {
  static constexpr float kShift = 0.f;    // bfloat16 has the range of fp32
  __device__ __forceinline__ static uint32_t pack(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  __device__ __forceinline__ static float2 unpack(uint32_t u) {
    return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
  }
  __device__ __forceinline__ static void mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  }
};
template <>
struct Dec16<__half> {
  static constexpr float kShift = 13.f;   // weights carry 2^13, so that the third part of small ones is not subnormal
  __device__ __forceinline__ static uint32_t pack(float lo, float hi) {
    const __half2 v = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  __device__ __forceinline__ static float2 unpack(uint32_t u) { return __half22float2(*reinterpret_cast<const __half2*>(&u)); }
  __device__ __forceinline__ static void mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  }
};

// One head's sums over a warp's rows on the fp32 pipe, D / 32 channels per lane: for rows that hold infinities or NaN.  In the
// matrix product every part of a weight meets every value, and a part that is zero or negative makes NaN of an infinity;
// one weight, one product gives what the sum says (an infinity of the value's sign, NaN where both signs or NaN are
// summed).  ref: the exponent that the warp's weights are relative to.
template <typename T, int D, bool PAGED, int WARPS>
__device__ __forceinline__ void dec_sum_special(const DecodeParams& p, int b, int h, const T* q, int64_t row0, int first, int hi,
                                                float ref, float* acc) {
  constexpr int PER = D / 32;
  const int lane = threadIdx.x & 31;
  float qv[PER], a[PER];
#pragma unroll
  for (int c = 0; c < PER; ++c) {
    qv[c] = to_float(q[lane * PER + c]);
    a[c] = 0.f;
  }
#pragma unroll 1
  for (int t0 = first; t0 < hi; t0 += WARPS * 16)
#pragma unroll 1
    for (int r = t0; r < min(t0 + 16, hi); ++r) {
      const int64_t at = PAGED ? paged_row(p.pt, b, h, r) : row0 + r;
      if (at < 0) continue;
      const T* k = static_cast<const T*>(p.k_cache) + at * D + lane * PER;
      const T* v = static_cast<const T*>(p.v_cache) + at * D + lane * PER;
      float dot = 0.f;
#pragma unroll
      for (int c = 0; c < PER; ++c) dot = fmaf(qv[c], to_float(k[c]), dot);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
      const float w = exp2f(dot * p.scale_log2 - ref);
#pragma unroll
      for (int c = 0; c < PER; ++c) a[c] = fmaf(w, to_float(v[c]), a[c]);
    }
#pragma unroll
  for (int c = 0; c < PER; ++c) acc[lane * PER + c] = a[c];
}

// Bytes from global to shared memory past the registers, zeros where `there` is false.
__device__ __forceinline__ void dec_copy16(uint32_t to, const void* from, bool there) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(there ? 16u : 0u) : "memory");
}
__device__ __forceinline__ uint4 dec_lds16(uint32_t at) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
  return v;
}

// grid, cluster as above, WARPS warps, kDecMmaHeads query heads per CTA.  A warp takes tiles of 16 rows, STAGES of them in
// shared memory or on their way there (dynamic, WARPS * STAGES * 64 * D bytes).  With g = lane / 4 and c = lane % 4 the
// fragments of m16n8k16 are
//   S  = Q K^T   A: row i = head i % 4 (every head four times), B: n = row g of 8, channels dealt so that a lane's B words are
//                its own 16-byte pieces of K (the order of the contraction is free as long as Q has the same one);
//                result: head g % 4, rows 2c, 2c + 1
//   O += P V     A: rows 0-3 the high parts of the weights, 4-7 the middle ones, 8-11 the low ones, 12-15 zero: in the very
//                lanes and positions where S came out; B: rows 2c, 2c + 1 (+ 8, 9) of channel 64 j + 8 g + i, from 16-byte
//                pieces of V with the halves of two rows interleaved.
// A lane holds sums of one head only, so rescaling needs no exchange; O is the sum over the three parts.
// In shared memory the 16-byte pieces of a row are exchanged (K: by the row's lowest bit, V: by the next two), so that eight
// lanes that read together touch every bank once.
template <typename T, int D, bool PAGED, int WARPS, int STAGES>
__global__ void __launch_bounds__(WARPS * 32, WARPS == 8 ? 1 : 2) decode_mma_kernel(const DecodeParams p) {
  constexpr int GT = kDecMmaHeads, KC = D / 32, VC = D / 64, THREADS = WARPS * 32;
  constexpr int PIECES = D / 8, ROWS_AT_ONCE = 32 / PIECES;    // 16-byte pieces of a row; rows that a warp copies per step
  constexpr uint32_t ROW = D * 2, TILE = 16 * ROW;
  using X = Dec16<T>;
  namespace cg = cooperative_groups;
  extern __shared__ __align__(128) uint8_t dec_smem[];
  __shared__ __align__(16) DecMerge<D, GT, WARPS> s_mrg;
  pdl_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = cluster.dim_blocks().x, rank = cluster.block_rank();
  if (C > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");      // this CTA's shared memory may be written
  const int unit = blockIdx.x / C, b = blockIdx.y;
  const int h = unit / p.head_blocks, g0 = (unit % p.head_blocks) * GT;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, c = lane & 3;
  const int count = p.seq.count[b];
  const int64_t row0 = p.seq.row_off[b] + static_cast<int64_t>(h) * count;
  const int lo = static_cast<int>(static_cast<int64_t>(count) * rank / C);
  const int hi = static_cast<int>(static_cast<int64_t>(count) * (rank + 1) / C);
  const int64_t hq0 = static_cast<int64_t>(b) * p.num_kv_heads * p.group + static_cast<int64_t>(h) * p.group + g0;
  const T* kc = static_cast<const T*>(p.k_cache);
  const T* vc = static_cast<const T*>(p.v_cache);
  const T* q_head = static_cast<const T*>(p.q) + (hq0 + min(g % GT, p.group - g0 - 1)) * D;
  // While the kernels ahead in the stream finish, this CTA's rows come into the L2 (a prefetch hands no data to anybody, so
  // it does not matter whether they are still being written; a page table read here is only used for it).
  if (warp == 0 && c < KC / 2) asm volatile("prefetch.global.L2 [%0];" ::"l"(q_head + c * 64));
  for (int i = threadIdx.x; i < min(hi - lo, kDecPrefetchRows) * 2; i += THREADS) {         // K and V rows in turn
    int64_t at = row0 + lo + i / 2;
    if (PAGED) {
      const int r = lo + i / 2;
      const int page = __ldcg(p.pt.table + p.pt.tab_off[b] + static_cast<int64_t>(h) * p.pt.pages[b] + r / p.pt.page_size);
      if (page < 0 || page >= p.pt.num_pages) continue;
      at = static_cast<int64_t>(page) * p.pt.page_size + r % p.pt.page_size;
    }
    const T* row = (i & 1 ? vc : kc) + at * D;
#pragma unroll
    for (int e = 0; e < D; e += 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + e));
  }
  pdl_wait();

  // Rows of a tile: lane l (and l + 16) looks up where row l lies (-1: not there).
  auto look_up = [&](int t0) -> int64_t {
    const int r = t0 + (lane & 15);
    if (r >= hi) return -1;
    if (!PAGED) return row0 + r;
    const int64_t at = paged_row(p.pt, b, h, r);
    if (at < 0 && lane < 16) atomicOr(p.status, kStatusBadPage);
    return at;
  };
  const uint32_t ring = static_cast<uint32_t>(__cvta_generic_to_shared(dec_smem)) + warp * (STAGES * 2 * TILE);
  // One group of copies per tile, empty behind the last one.
  auto copy_tile = [&](int t0, int slot, int64_t mine) {
    if (t0 < hi) {
#pragma unroll
      for (int s = 0; s < 16 / ROWS_AT_ONCE; ++s) {
        const int r = s * ROWS_AT_ONCE + lane / PIECES, piece = lane % PIECES;
        const int64_t at = __shfl_sync(0xffffffffu, mine, r);
        const int64_t from = (at >= 0 ? at : 0) * D + piece * 8;
        const uint32_t to = ring + slot * (2 * TILE) + r * ROW;
        dec_copy16(to + ((piece ^ ((r & 1) << 2)) << 4), kc + from, at >= 0);
        dec_copy16(to + TILE + ((piece ^ (((r >> 1) & 3) << 1)) << 4), vc + from, at >= 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int first = lo + warp * 16;
  constexpr int STEP = WARPS * 16;
  uint32_t there[STAGES];                        // rows of the tiles in the ring
  {
    int64_t mine[STAGES];
#pragma unroll
    for (int s = 0; s < STAGES; ++s) mine[s] = look_up(first + s * STEP);
#pragma unroll
    for (int s = 0; s < STAGES; ++s) {
      copy_tile(first + s * STEP, s, mine[s]);
      there[s] = __ballot_sync(0xffffffffu, mine[s] >= 0);
    }
  }
  int64_t mine = look_up(first + STAGES * STEP);                // of the tile that is copied next
  uint4 q[KC];
#pragma unroll
  for (int j = 0; j < KC; ++j)
    q[j] = g0 + g % GT < p.group ? *reinterpret_cast<const uint4*>(q_head + j * 32 + c * 8) : make_uint4(0, 0, 0, 0);
  float o[VC * 8][4];
#pragma unroll
  for (int i = 0; i < VC * 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m = -INFINITY, z = 0.f;                  // of head g % 4: m over the warp's rows, z over this lane's
  for (int t0 = first; t0 < hi;) {
#pragma unroll
    for (int slot = 0; slot < STAGES; ++slot) {
      if (t0 >= hi) break;                       // (uniform over the warp)
      asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 1) : "memory");
      __syncwarp();
      const uint32_t k_at = ring + slot * (2 * TILE), v_at = k_at + TILE;
      float x[2][2];
      float mx = -INFINITY;
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < KC; ++j) {
          const uint4 k = dec_lds16(k_at + (t * 8 + g) * ROW + (((j * 4 + c) ^ ((g & 1) << 2)) << 4));
          X::mma(s0, q[j].x, q[j].x, q[j].y, q[j].y, k.x, k.y);
          X::mma(s1, q[j].z, q[j].z, q[j].w, q[j].w, k.z, k.w);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          x[t][i] = (there[slot] >> (t * 8 + 2 * c + i)) & 1u ? (s0[i] + s1[i]) * p.scale_log2 : -INFINITY;
          mx = fmaxf(mx, x[t][i]);
        }
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float mn = fmaxf(m, mx);
      const float ref = mn == -INFINITY ? 0.f : mn - X::kShift;
      if (__any_sync(0xffffffffu, mn > m)) {
        const float corr = m == -INFINITY ? 0.f : ex2(m - mn);
        z *= corr;
#pragma unroll
        for (int i = 0; i < VC * 8; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) o[i][e] *= corr;
      }
      m = mn;
      uint32_t a[2][2];                          // [rows 2c.. / 2c + 8..][fragment row g / g + 8]
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const float w0 = ex2(x[t][0] - ref), w1 = ex2(x[t][1] - ref);
        z += w0 + w1;
        const uint32_t high = X::pack(w0, w1);
        const float2 hf = X::unpack(high);
        const uint32_t mid = X::pack(w0 - hf.x, w1 - hf.y);
        const float2 mf = X::unpack(mid);
        const uint32_t low = X::pack(w0 - hf.x - mf.x, w1 - hf.y - mf.y);
        a[t][0] = g < 4 ? high : mid;
        a[t][1] = g < 4 ? low : 0u;
      }
#pragma unroll
      for (int j = 0; j < VC; ++j) {
        uint4 v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t)              // row (t / 2) * 8 + 2c + t % 2
          v[t] = dec_lds16(v_at + ((t >> 1) * 8 + 2 * c + (t & 1)) * ROW + (((j * 8 + g) ^ (c << 1)) << 4));
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const uint32_t v0 = reinterpret_cast<const uint32_t*>(&v[0])[w], v1 = reinterpret_cast<const uint32_t*>(&v[1])[w];
          const uint32_t v2 = reinterpret_cast<const uint32_t*>(&v[2])[w], v3 = reinterpret_cast<const uint32_t*>(&v[3])[w];
          X::mma(o[j * 8 + 2 * w], a[0][0], a[0][1], a[1][0], a[1][1], __byte_perm(v0, v1, 0x5410), __byte_perm(v2, v3, 0x5410));
          X::mma(o[j * 8 + 2 * w + 1], a[0][0], a[0][1], a[1][0], a[1][1], __byte_perm(v0, v1, 0x7632), __byte_perm(v2, v3, 0x7632));
        }
      }
      __syncwarp();                              // the tile has been read
      copy_tile(t0 + STAGES * STEP, slot, mine);
      there[slot] = __ballot_sync(0xffffffffu, mine >= 0);
      t0 += STEP;
      mine = look_up(t0 + STAGES * STEP);
    }
  }
  // ---- the parts, then the warps, then the CTAs of the cluster
  z += __shfl_xor_sync(0xffffffffu, z, 1);
  z += __shfl_xor_sync(0xffffffffu, z, 2);
  float special[4] = {0.f, 0.f, 0.f, 0.f};       // NaN once a sum is not finite
  // Lanes g and g + 4 hold parts of the same sums: each keeps one of the two channel octets 64 j + 8 (2c + e) + 0 .. 7 of head
  // g % 4, the lower one e = 0.  (Sixteen-byte stores; scalar ones met in two banks, eight lanes each, 0.7 us.)
  const bool upper = g >= 4;
#pragma unroll
  for (int j = 0; j < VC; ++j) {
    float s[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float s0 = o[j * 8 + i][0] + o[j * 8 + i][2], s1 = o[j * 8 + i][1] + o[j * 8 + i][3];
      s[i] = (upper ? s1 : s0) + __shfl_xor_sync(0xffffffffu, upper ? s0 : s1, 16);
      special[i & 3] = fmaf(s[i], 0.f, special[i & 3]);
    }
    float4* to = reinterpret_cast<float4*>(&s_mrg.acc[warp][(g & 3) * (D + 4) + j * 64 + (2 * c + (upper ? 1 : 0)) * 8]);
    to[0] = make_float4(s[0], s[1], s[2], s[3]);
    to[1] = make_float4(s[4], s[5], s[6], s[7]);
  }
  if (__any_sync(0xffffffffu, (special[0] + special[1]) + (special[2] + special[3]) != 0.f)) {
    __syncwarp();
#pragma unroll 1
    for (int j = 0; j < min(GT, p.group - g0); ++j) {
      const float mj = __shfl_sync(0xffffffffu, m, j * 4);
      dec_sum_special<T, D, PAGED, WARPS>(p, b, h, static_cast<const T*>(p.q) + (hq0 + j) * D, row0, lo + warp * 16, hi,
                                   mj == -INFINITY ? 0.f : mj - X::kShift, &s_mrg.acc[warp][j * (D + 4)]);
    }
  }
  if (g < 4 && c == 0) {
    s_mrg.m[warp][g] = dec_none(m);
    s_mrg.z[warp][g] = z;
  }
  __syncthreads();
  dec_finish<D, GT, WARPS>(s_mrg, p, C, rank, hq0, p.group - g0);
}

}  // namespace pkv
