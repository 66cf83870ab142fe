// Window-score kernels on the plain fp32 pipes (Section 4.2.2, Eq. 2 and Eq. 3).
//
// These cover every dtype / shape the boundary admits (fp32 inputs, any window, any group size) and are the path of
// small fp32 problems.  The tensor-core kernels in pkv_score_tc.cuh take over for 16-bit inputs when their shape rules
// hold.
//
// The score of a key mixes softmax rows that each have their own normaliser, so the normalisers must be known before
// any score can be formed:
//   logit_tiles<STATS>   x_ri = q_r . k_i * log2(e) / sqrt(d) of a block of window rows and a chunk of keys, tile by tile;
//                        per row the maximum and the sum of 2^(x - max) -> partial (max, sum), and x itself to the
//                        workspace when that has room for it (w.logits)
//   scores_of_logits     s_i = sum_r 2^(x_ri - lse2[r] - log2 G) from the stored x; merges a head's partials first
//   logit_tiles<SCORES>  the same sum straight from the tiles, with the normalisers known (the caller's, or those of
//                        combine_stats): when x was not stored
// Both ways form x with the same sequence of operations (one multiply-add chain over the channels per logit).
//
// What bounds it: 2 R n d flops per KV head on the fp32 pipe (128 multiply-adds per clock and SM).  Storing x (4 R n
// bytes, mostly in the L2) costs a quarter of forming it again.  A tile is a register-blocked product: 256 threads with
// 8 x 4 (4 x 4) logits each, fed by 16-byte shared-memory reads of channel-major Q and K, two logits per packed
// multiply-add, so that the pipe and not the reads are the limit.
#pragma once

#include "pkv_common.cuh"

namespace pkv {

constexpr int kGenThreads = 256;
constexpr int kGenMinTile = 64;      // fewest keys per tile (a chunk of partial statistics is at least one tile)
constexpr int kGenSumThreads = 256;  // scores_of_logits: threads per CTA,
constexpr int kGenSumKeys = 256;     // keys per CTA (four per thread),
constexpr int kGenSumGroups = kGenSumThreads * 4 / kGenSumKeys;   // and groups of threads that share the rows

struct ScoreParams {
  TensorView q, k;
  SeqTable seq;                          // stat_off / score_off count chunks of chunk_tiles tiles
  int32_t num_kv_heads, group, rows;     // rows = group * alpha
  float scale_log2;                      // log2(e) / sqrt(d)
  float2* partial;                       // [sum_b chunks_b][slots_per_chunk][H_kv][rows] (max, sum)
  int32_t slots_per_chunk;               // partial slots each chunk writes (1 here, 2 for the tensor-core sweep)
  float* lse2;                           // [batch][H_kv][rows]
  const float* lse_in;                   // normalisers the score sweep reads: lse2, or the caller's
  float lse_scale, lse_add;              // applied on load: (1, 0), or (log2 e, log2 G) for natural-log input
  float* scores;                         // [batch][H_kv][ld]
  int64_t ld_scores;
  int32_t stats_only;                    // host side: stop after the row normalisers (no score sweep)
  int32_t stat_grid;                     // 0: partial is [chunk][slot][H_kv][rows] (fp32-pipe sweep).  > 0: CTAs of
                                         // the tensor-core sweep, which writes [segment][slot][rows] with segment =
                                         // CTA + head for every run of a CTA over one head's chunks
  float* logits;                         // fp32-pipe path: [batch][H_kv][rows][ld_logits] x values, or null
  int64_t ld_logits;
  int32_t chunk_tiles;                   // tiles per chunk (1 when there are several row blocks)
  float log2_group;
};

// Four consecutive channels of a row as floats.
__device__ __forceinline__ float4 gen_load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 gen_load4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ float4 gen_load4(const __half* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x)), b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// Channel-major tile in shared memory: element (channel c, column x) of a tile of W columns.  Columns are exchanged in
// groups of four by a function of the channel, so that both the transposing stores (eight lanes along the channels,
// four along the columns) and the 16-byte reads along the columns touch every bank once.
template <int W>
__device__ __forceinline__ int gen_at(int c, int x) { return c * W + (x ^ (((c >> 2) & 7) << 2)); }

// Fills a channel-major tile from `count` rows (row(x) = address of row x; the columns from `count` to W become zero).
template <int W, int D, typename F>
__device__ __forceinline__ void gen_fill(float* tile, int count, F&& row) {
  constexpr int kSteps = W * D / 4 / kGenThreads, kBatch = kSteps < 4 ? kSteps : 4;
  static_assert(W * D / 4 % kGenThreads == 0, "tile of whole steps");
  const int dq = threadIdx.x & 7;                            // 32 channels = 8 lanes of 4
#pragma unroll
  for (int s0 = 0; s0 < kSteps; s0 += kBatch) {
    float4 f[kBatch];
#pragma unroll
    for (int s = 0; s < kBatch; ++s) {
      const int e = (s0 + s) * (kGenThreads / 8) + threadIdx.x / 8;        // (channel block of 32, column), column fastest
      const int x = e % W, cb = e / W;
      f[s] = x < count ? gen_load4(row(x) + cb * 32 + dq * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int s = 0; s < kBatch; ++s) {
      const int e = (s0 + s) * (kGenThreads / 8) + threadIdx.x / 8;
      const int x = e % W, c = (e / W) * 32 + dq * 4;
      tile[gen_at<W>(c, x)] = f[s].x;
      tile[gen_at<W>(c + 1, x)] = f[s].y;
      tile[gen_at<W>(c + 2, x)] = f[s].z;
      tile[gen_at<W>(c + 3, x)] = f[s].w;
    }
  }
}

// grid (chunks over all sequences, H_kv), block kGenThreads, dynamic shared memory gen_smem_bytes.
// ROWS x KEYS: window rows and keys of a tile; TR rows x 4 keys per thread.
template <int D, int ROWS, int KEYS>
__host__ __device__ constexpr int gen_smem_bytes() { return (ROWS + KEYS) * D * 4; }

template <typename T, int D, int ROWS, int KEYS, bool SCORES>
__global__ void __launch_bounds__(kGenThreads, 2) logit_tiles_kernel(const ScoreParams p) {
  constexpr int KT = KEYS / 4;                               // threads along the keys
  constexpr int RT = kGenThreads / KT;                       // threads along the rows
  constexpr int TR = ROWS / RT;                              // rows per thread
  static_assert(KT <= 32 && TR % 4 == 0, "a warp holds whole rows of threads");
  extern __shared__ __align__(16) float gen_smem[];
  float* qs = gen_smem;                                      // channel-major [D][ROWS]
  float* ks = gen_smem + ROWS * D;                           // channel-major [D][KEYS]
  __shared__ float lse_s[SCORES ? ROWS : 1];
  __shared__ __align__(16) float part[SCORES ? RT : 1][SCORES ? KEYS : 4];
  pdl_trigger();
  const int32_t* off = SCORES ? p.seq.score_off : p.seq.stat_off;
  const int h = blockIdx.y, b = find_sequence(off, p.seq.batch, blockIdx.x);
  const int n = p.seq.n[b], alpha = p.seq.alpha, P = p.seq.prefix[b];
  const int keys = SCORES ? P : n;
  const int tile0 = (blockIdx.x - off[b]) * p.chunk_tiles, tile1 = min(tile0 + p.chunk_tiles, (keys + KEYS - 1) / KEYS);
  const T* kbase = static_cast<const T*>(p.k.ptr) + b * p.k.sb + h * p.k.sh;
  const T* qbase = static_cast<const T*>(p.q.ptr) + b * p.q.sb + static_cast<int64_t>(h * p.group) * p.q.sh;
  const int tk = threadIdx.x % KT, tr = threadIdx.x / KT;
  const int blocks = (p.rows + ROWS - 1) / ROWS;
  const int64_t head = static_cast<int64_t>(b) * p.num_kv_heads + h;
  pdl_wait();

  float m[TR], z[TR];                                        // STATS: per row over this thread's keys of the chunk
#pragma unroll
  for (int i = 0; i < TR; ++i) { m[i] = -INFINITY; z[i] = 0.f; }
  for (int t = tile0; t < tile1; ++t) {
    const int key0 = t * KEYS;
    float sum[4] = {0.f, 0.f, 0.f, 0.f};                     // SCORES: of this thread's keys
    for (int rb = 0; rb < blocks; ++rb) {
      const int r0 = rb * ROWS;
      __syncthreads();                                       // the tiles before have been read
      if (blocks > 1 || t == tile0) {
        gen_fill<ROWS, D>(qs, min(ROWS, p.rows - r0), [&](int x) {
          const int r = r0 + x;
          return qbase + (r / alpha) * p.q.sh + (r % alpha) * p.q.st;
        });
        if (SCORES)
          for (int x = threadIdx.x; x < ROWS; x += kGenThreads)
            lse_s[x] = r0 + x < p.rows ? fmaf(p.lse_in[head * p.rows + r0 + x], p.lse_scale, p.lse_add) : INFINITY;
      }
      if (rb == 0) gen_fill<KEYS, D>(ks, min(KEYS, n - key0), [&](int x) { return kbase + static_cast<int64_t>(key0 + x) * p.k.st; });
      __syncthreads();
      unsigned long long acc[TR / 2][4];                     // pairs of rows: the queries come in pairs as they are, only the
#pragma unroll                                               // four keys have to be doubled
      for (int i = 0; i < TR / 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll 32
      for (int c = 0; c < D; ++c) {
        const float4 kf = *reinterpret_cast<const float4*>(ks + gen_at<KEYS>(c, tk * 4));
        const unsigned long long k2[4] = {pack2(kf.x, kf.x), pack2(kf.y, kf.y), pack2(kf.z, kf.z), pack2(kf.w, kf.w)};
#pragma unroll
        for (int i = 0; i < TR; i += 4) {
          const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(qs + gen_at<ROWS>(c, tr * TR + i));
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            acc[i / 2][j] = fma2(q.x, k2[j], acc[i / 2][j]);
            acc[i / 2 + 1][j] = fma2(q.y, k2[j], acc[i / 2 + 1][j]);
          }
        }
      }
      const int i0 = key0 + tk * 4;                          // this thread's keys
#pragma unroll
      for (int i = 0; i < TR; ++i) {
        const int r = r0 + tr * TR + i;
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float even, odd;
          unpack2(acc[i / 2][j], even, odd);
          x[j] = (i & 1 ? odd : even) * p.scale_log2;
        }
        if (SCORES) {
#pragma unroll
          for (int j = 0; j < 4; ++j) sum[j] += exp2f(x[j] - lse_s[tr * TR + i]);
          continue;
        }
        if (r >= p.rows) continue;
        if (p.logits && i0 < P)
          *reinterpret_cast<float4*>(p.logits + (head * p.rows + r) * p.ld_logits + i0) = make_float4(x[0], x[1], x[2], x[3]);
        const int last = min(P + r % alpha, n - 1);          // row (g, j) sees keys 0 .. P + j that exist here
        if (i0 + 3 > last) {
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = i0 + j <= last ? x[j] : -INFINITY;
        }
        const float mn = fmaxf(fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3])), m[i]);
        if (mn > -INFINITY) {
          z[i] = z[i] * exp2f(m[i] - mn) + ((exp2f(x[0] - mn) + exp2f(x[1] - mn)) + (exp2f(x[2] - mn) + exp2f(x[3] - mn)));
          m[i] = mn;
        }
      }
      if (!SCORES && (blocks > 1 || t + 1 == tile1)) {       // the rows' statistics over the chunk: merge the threads along the keys
#pragma unroll
        for (int i = 0; i < TR; ++i) {
#pragma unroll
          for (int o = 1; o < KT; o <<= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, m[i], o), z2 = __shfl_xor_sync(0xffffffffu, z[i], o);
            const float mm = fmaxf(m[i], m2);
            if (mm > -INFINITY) z[i] = z[i] * exp2f(m[i] - mm) + z2 * exp2f(m2 - mm);
            m[i] = mm;
          }
          const int r = r0 + tr * TR + i;
          if (tk == 0 && r < p.rows)
            p.partial[(static_cast<int64_t>(blockIdx.x) * p.num_kv_heads + h) * p.rows + r] = make_float2(m[i], z[i]);
          m[i] = -INFINITY;
          z[i] = 0.f;
        }
      }
    }
    if (SCORES) {                                            // the rows of a key are spread over RT threads
      *reinterpret_cast<float4*>(&part[tr][tk * 4]) = make_float4(sum[0], sum[1], sum[2], sum[3]);
      __syncthreads();
      for (int x = threadIdx.x; x < KEYS; x += kGenThreads) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < RT; ++q) s += part[q][x];
        if (key0 + x < P) p.scores[head * p.ld_scores + key0 + x] = s;
      }
    }
  }
}

// grid (blocks of kGenSumKeys prefix keys of the longest sequence, H_kv, batch), block kGenSumThreads, dynamic shared
// memory rows floats: scores from stored logits.  Latency is what it has to hide (a thread's loads are strided by whole
// rows): four keys per thread, the rows dealt round to the CTA's four groups of threads in batches of eight loads, the
// groups' sums added in a fixed order.  The row normalisers are merged from the partials by every CTA for itself (a few
// hundred kilobytes from the L2), which saves a launch between the two.
__global__ void __launch_bounds__(kGenSumThreads) scores_of_logits_kernel(const ScoreParams p) {
  extern __shared__ float lse_all[];
  __shared__ float4 part[kGenSumGroups - 1][kGenSumKeys / 4];
  pdl_trigger();
  const int h = blockIdx.y, b = blockIdx.z, P = p.seq.prefix[b];
  const int kt = threadIdx.x % (kGenSumKeys / 4), grp = threadIdx.x / (kGenSumKeys / 4);
  const int i0 = blockIdx.x * kGenSumKeys + kt * 4;
  pdl_wait();
  if (blockIdx.x * kGenSumKeys >= P) return;
  const int64_t head = static_cast<int64_t>(b) * p.num_kv_heads + h;
  const int t0 = p.seq.stat_off[b], t1 = p.seq.stat_off[b + 1];
  const int64_t step = static_cast<int64_t>(p.num_kv_heads) * p.rows;
  for (int r = threadIdx.x; r < p.rows; r += kGenSumThreads) {
    const float2* src = p.partial + static_cast<int64_t>(h) * p.rows + r;
    float m = -INFINITY, z = 0.f;
    for (int t = t0; t < t1; t += 8) {
      float2 pz[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) pz[u] = t + u < t1 ? __ldcg(src + (t + u) * step) : make_float2(-INFINITY, 0.f);
      float mn = m;
#pragma unroll
      for (int u = 0; u < 8; ++u) mn = fmaxf(mn, pz[u].x);
      if (mn > -INFINITY) {
        z *= exp2f(m - mn);
#pragma unroll
        for (int u = 0; u < 8; ++u) z += pz[u].y * exp2f(pz[u].x - mn);
        m = mn;
      }
    }
    lse_all[r] = m + log2f(z) + p.log2_group;
  }
  __syncthreads();
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  if (i0 < P) {
    const float* x = p.logits + head * p.rows * p.ld_logits + i0;
    for (int r0 = grp; r0 < p.rows; r0 += 8 * kGenSumGroups) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = r0 + u * kGenSumGroups;
        v[u] = r < p.rows ? __ldcg(reinterpret_cast<const float4*>(x + r * p.ld_logits)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = r0 + u * kGenSumGroups;
        const float l = r < p.rows ? lse_all[r] : INFINITY;
        s[0] += exp2f(v[u].x - l);
        s[1] += exp2f(v[u].y - l);
        s[2] += exp2f(v[u].z - l);
        s[3] += exp2f(v[u].w - l);
      }
    }
  }
  if (grp > 0) part[grp - 1][kt] = make_float4(s[0], s[1], s[2], s[3]);
  __syncthreads();
  if (grp > 0) return;
#pragma unroll
  for (int q = 0; q < kGenSumGroups - 1; ++q) {
    const float4 o = part[q][kt];
    s[0] += o.x; s[1] += o.y; s[2] += o.z; s[3] += o.w;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (i0 + j < P) p.scores[head * p.ld_scores + i0 + j] = s[j];
}

// grid (ceil(rows / 32), H_kv, batch), block 1024: merge the chunk partials of each window row.
// Thread (rl, sg) = (tid % 32, tid / 32) takes row r0 + rl and every 32nd partial slot starting at sg, so
// a warp reads 32 consecutive rows of one slot (256 contiguous bytes); loads are issued four at a time
// before they are used.  The 32 slot groups of a row are merged through shared memory.
// extra_log2 = log2(G) folds the mean over the group's query heads into the normaliser.
constexpr int kCombineThreads = 1024;
__global__ void __launch_bounds__(kCombineThreads) combine_stats_kernel(const ScoreParams p, float extra_log2) {
  __shared__ float sm[32][33], sz[32][33];
  pdl_trigger();
  pdl_wait();
  const int h = blockIdx.y, b = blockIdx.z;
  const int rl = threadIdx.x & 31, sg = threadIdx.x >> 5;
  const int r = blockIdx.x * 32 + rl;
  int t0 = p.seq.stat_off[b] * p.slots_per_chunk, t1 = p.seq.stat_off[b + 1] * p.slots_per_chunk;
  int64_t slot_stride = static_cast<int64_t>(p.num_kv_heads) * p.rows;
  int64_t first = static_cast<int64_t>(h) * p.rows;
  if (p.stat_grid > 0) {
    // The sweep's CTAs take contiguous item ranges (items ordered sequence, head, chunk): the first `rem`
    // CTAs per + 1 items, the others per.  This head's items fall to CTAs c0..c1, one segment each.
    const int nc = p.seq.stat_off[b + 1] - p.seq.stat_off[b];
    const int total = p.num_kv_heads * p.seq.stat_off[p.seq.batch];
    const int per = total / p.stat_grid, rem = total % p.stat_grid;
    const int edge = rem * (per + 1);
    const int i0 = p.num_kv_heads * p.seq.stat_off[b] + h * nc, i1 = i0 + nc - 1;
    const int c0 = i0 < edge ? i0 / (per + 1) : rem + (i0 - edge) / per;
    const int c1 = i1 < edge ? i1 / (per + 1) : rem + (i1 - edge) / per;
    const int hg = b * p.num_kv_heads + h;
    t0 = (c0 + hg) * p.slots_per_chunk;
    t1 = (c1 + hg + 1) * p.slots_per_chunk;
    slot_stride = p.rows;
    first = 0;
  }
  float m = -INFINITY, z = 0.f;
  if (r < p.rows) {
    const float2* base = p.partial + first + r;
    for (int t = t0 + sg; t < t1; t += 4 * 32) {
      float2 pz[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        pz[u] = t + 32 * u < t1 ? base[(t + 32 * u) * slot_stride] : make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (pz[u].x > -INFINITY) {                 // (-inf, 0) marks a slot that saw no key of this row
          const float mn = fmaxf(m, pz[u].x);
          z = z * exp2f(m - mn) + pz[u].y * exp2f(pz[u].x - mn);
          m = mn;
        }
    }
  }
  sm[sg][rl] = m;
  sz[sg][rl] = z;
  __syncthreads();
  if (sg == 0 && r < p.rows) {
    float mm = -INFINITY;
    for (int g = 0; g < 32; ++g) mm = fmaxf(mm, sm[g][rl]);
    float zz = 0.f;
    for (int g = 0; g < 32; ++g)
      if (sm[g][rl] > -INFINITY) zz += sz[g][rl] * exp2f(sm[g][rl] - mm);
    p.lse2[(static_cast<int64_t>(b) * p.num_kv_heads + h) * p.rows + r] = mm + log2f(zz) + extra_log2;
  }
}

}  // namespace pkv
