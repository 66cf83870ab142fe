// Window-score kernels on the plain fp32 pipes (Section 4.2.2, Eq. 2 and Eq. 3).
//
// These cover every dtype / shape the boundary admits (fp32 inputs, any window, any group size) and are the path of
// fp32 problems of few window rows, of calls without room for the logits and of handed-in normalisers.  The tensor-core kernels in
// pkv_score_tc.cuh take over for 16-bit inputs when their shape rules hold, those in pkv_score_split.cuh for fp32 ones of more
// than 32 window rows.
//
// The score of a key mixes softmax rows that each have their own normaliser, so the normalisers must be known before
// any score can be formed:
//   logit_tiles<STATS>   x_ri = q_r . k_i * log2(e) / sqrt(d) of a block of window rows and a chunk of keys, tile by tile;
//                        per row and tile the maximum and the sum of 2^(x - max) -> partial (max, sum), and x itself to
//                        the workspace when that has room for it (w.logits)
//   scores_of_logits     s_i = sum_r 2^(x_ri - lse2[r] - log2 G) from the stored x; merges a head's partials first
//   logit_tiles<SCORES>  the same sum straight from the tiles, with the normalisers known (the caller's, or those of
//                        combine_stats): when x was not stored
// Both ways form x with the same sequence of operations.
//
// What bounds it: 2 R n d flops per KV head on the fp32 pipe (a loop of packed multiply-adds reaches 63 TFLOP/s on this
// device, scalar ones 50).  Storing x (4 R n bytes, mostly in the L2) costs a quarter of forming it again.  A tile is a
// register-blocked product: 256 threads with 8 x 8 (4 x 8, 4 x 4) logits each.  At 8 x 4 the 16-byte shared-memory reads
// (four wavefronts each) and not the multiply-adds were the limit, whichever way the operands lay.
#pragma once

#include "pkv_common.cuh"

namespace pkv {

constexpr int kGenThreads = 256;
constexpr int kGenTile = 128;        // keys per tile: one (max, sum) per row and tile
constexpr int kGenSumThreads = 256;  // scores_of_logits: threads per CTA,
constexpr int kGenSumKeys = 256;     // keys per CTA (four per thread),
constexpr int kGenSumGroups = kGenSumThreads * 4 / kGenSumKeys;   // and groups of threads that share the rows

struct ScoreParams {
  TensorView q, k;
  SeqTable seq;                          // stat_off / score_off count chunks of chunk_tiles tiles
  int32_t num_kv_heads, group, rows;     // rows = group * alpha
  float scale_log2;                      // log2(e) / sqrt(d)
  float2* partial;                       // [sum_b tiles_b][H_kv][rows] (max, sum), or see stat_grid
  float* lse2;                           // [batch][H_kv][rows]
  const float* lse_in;                   // normalisers the score sweep reads: lse2, or the caller's
  float lse_scale, lse_add;              // applied on load: (1, 0), or (log2 e, log2 G) for natural-log input
  float* scores;                         // [batch][H_kv][ld]
  int64_t ld_scores;
  int32_t stats_only;                    // host side: stop after the row normalisers (no score sweep)
  int32_t stat_grid;                     // 0: partial is [tile][H_kv][rows] (fp32-pipe sweep).  > 0: CTAs of
                                         // a tensor-core sweep, which writes [segment][rows] with segment =
                                         // CTA + head for every run of a CTA over one head's chunks (fp32 inputs:
                                         // over the tiles of one unit, a head's block of 128 rows)
  float* logits;                         // x values kept between two kernels, or null: [batch][H_kv][rows][ld_logits] (fp32
                                         // pipe), [batch][H_kv][ld_logits][rows] (fp32 inputs on the tensor cores)
  int64_t ld_logits;
  int32_t chunk_tiles;                   // tiles per CTA (1 when there are several row blocks)
  float log2_group;
  int32_t per_unit;                      // pkv_score_split.cuh: CTAs per unit of one length, or 0
  int32_t withhold;                      // ... test aid: CTA 0 never hands over its last K tile (its waits then run out)
  long long wait_clocks;                 // ... bound of any one wait, in SM clocks
  uint32_t* status;
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

constexpr int kGenSlice = 32;        // channels of K in shared memory at a time (two buffers)

// 32 channels of W rows, global memory -> registers -> channel-major tile: eight lanes take a row's 32 channels.
template <int W>
struct GenSlice {
  static constexpr int kSteps = W * kGenSlice / 4 / kGenThreads;
  static_assert(W * kGenSlice / 4 % kGenThreads == 0, "slice of whole steps");
  float4 f[kSteps];
  // row(x) = address of the first of the 32 channels of row x; rows from `count` on are zero
  template <typename F>
  __device__ __forceinline__ void load(int count, F&& row) {
#pragma unroll
    for (int s = 0; s < kSteps; ++s) {
      const int x = s * (kGenThreads / 8) + threadIdx.x / 8;
      f[s] = x < count ? gen_load4(row(x) + (threadIdx.x & 7) * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ __forceinline__ void store(float* tile) const {       // tile: the slice's first channel
    const int c = (threadIdx.x & 7) * 4;
#pragma unroll
    for (int s = 0; s < kSteps; ++s) {
      const int x = s * (kGenThreads / 8) + threadIdx.x / 8;
      tile[gen_at<W>(c, x)] = f[s].x;
      tile[gen_at<W>(c + 1, x)] = f[s].y;
      tile[gen_at<W>(c + 2, x)] = f[s].z;
      tile[gen_at<W>(c + 3, x)] = f[s].w;
    }
  }
};

// grid (chunks over all sequences, H_kv), block kGenThreads, dynamic shared memory gen_smem_bytes.
// ROWS x KEYS: window rows and keys of a tile; TR rows x TK keys per thread, in groups of four.
template <int D, int ROWS, int KEYS>
__host__ __device__ constexpr int gen_smem_bytes() { return (ROWS * D + 2 * KEYS * kGenSlice) * 4; }

template <typename T, int D, int ROWS, int KEYS, int TR, int TK, bool SCORES>
__global__ void __launch_bounds__(kGenThreads, 2) logit_tiles_kernel(const ScoreParams p) {
  constexpr int KT = KEYS / TK;                              // threads along the keys
  constexpr int RT = kGenThreads / KT;                       // threads along the rows
  constexpr int SLICES = D / kGenSlice;
  static_assert(KT <= 32 && RT * TR == ROWS && TR % 4 == 0 && TK % 4 == 0, "whole rows of threads in a warp");
  extern __shared__ __align__(16) float gen_smem[];
  float* qs = gen_smem;                                      // channel-major [D][ROWS]
  float* ks = gen_smem + ROWS * D;                           // channel-major [2][kGenSlice][KEYS]
  __shared__ float lse_s[SCORES ? ROWS : 1];
  __shared__ float part[SCORES ? RT : 1][SCORES ? KEYS : 1];
  pdl_trigger();
  const int32_t* off = SCORES ? p.seq.score_off : p.seq.stat_off;
  const int h = blockIdx.y, b = find_sequence(off, p.seq.batch, blockIdx.x);
  const int n = p.seq.n[b], alpha = p.seq.alpha, P = p.seq.prefix[b];
  const int keys = SCORES ? P : n;
  const int tiles = (keys + KEYS - 1) / KEYS;
  const int tile0 = (blockIdx.x - off[b]) * p.chunk_tiles, tile1 = min(tile0 + p.chunk_tiles, tiles);
  const int64_t tile_id = (SCORES ? 0 : p.seq.tile_off[b]) + tile0;
  const T* kbase = static_cast<const T*>(p.k.ptr) + b * p.k.sb + h * p.k.sh;
  const T* qbase = static_cast<const T*>(p.q.ptr) + b * p.q.sb + static_cast<int64_t>(h * p.group) * p.q.sh;
  const int tk = threadIdx.x % KT, tr = threadIdx.x / KT;
  const int blocks = (p.rows + ROWS - 1) / ROWS;
  const int64_t head = static_cast<int64_t>(b) * p.num_kv_heads + h;
  auto key_of = [&](int j) { return (j / 4) * (KT * 4) + tk * 4 + j % 4; };        // column of a tile
  auto row_of = [&](int i) { return (i / 4) * (RT * 4) + tr * 4 + i % 4; };
  const int steps = (tile1 - tile0) * SLICES;
  GenSlice<KEYS> next;
  auto load_slice = [&](int it) {                            // slice it of the chunk
    const int key0 = (tile0 + it / SLICES) * KEYS;
    const T* base = kbase + static_cast<int64_t>(key0) * p.k.st + (it % SLICES) * kGenSlice;
    next.load(min(KEYS, n - key0), [&](int x) { return base + x * p.k.st; });
  };
  pdl_wait();

  float sum[SCORES ? TK : 1];                                // SCORES: of this thread's keys, over the row blocks
#pragma unroll
  for (int j = 0; j < (SCORES ? TK : 1); ++j) sum[j] = 0.f;
  for (int rb = 0; rb < blocks; ++rb) {
    const int r0 = rb * ROWS;
    if (rb > 0) __syncthreads();                             // the block before has been read
    load_slice(0);
#pragma unroll
    for (int s = 0; s < SLICES; ++s) {
      GenSlice<ROWS> q;
      q.load(min(ROWS, p.rows - r0), [&](int x) {
        const int r = r0 + x;
        return qbase + (r / alpha) * p.q.sh + (r % alpha) * p.q.st + s * kGenSlice;
      });
      q.store(qs + s * kGenSlice * ROWS);
    }
    if (SCORES)
      for (int x = threadIdx.x; x < ROWS; x += kGenThreads)
        lse_s[x] = r0 + x < p.rows ? fmaf(p.lse_in[head * p.rows + r0 + x], p.lse_scale, p.lse_add) : INFINITY;
    next.store(ks);
    __syncthreads();
    unsigned long long acc[TR / 2][TK];                      // pairs of rows: the queries come in pairs as they are, the
#pragma unroll                                               // keys are doubled
    for (int i = 0; i < TR / 2; ++i)
#pragma unroll
      for (int j = 0; j < TK; ++j) acc[i][j] = 0ull;
    for (int it = 0; it < steps; ++it) {
      if (it + 1 < steps) load_slice(it + 1);                // arrives under this slice's multiply-adds
      const float* kc = ks + (it & 1) * (kGenSlice * KEYS);
      const float* qc = qs + (it % SLICES) * (kGenSlice * ROWS);
#pragma unroll 8
      for (int c = 0; c < kGenSlice; ++c) {
        ulonglong2 q[TR / 4];
#pragma unroll
        for (int i = 0; i < TR / 4; ++i) q[i] = *reinterpret_cast<const ulonglong2*>(qc + gen_at<ROWS>(c, i * RT * 4 + tr * 4));
#pragma unroll
        for (int g = 0; g < TK / 4; ++g) {
          const float4 kf = *reinterpret_cast<const float4*>(kc + gen_at<KEYS>(c, g * KT * 4 + tk * 4));
          const unsigned long long k2[4] = {pack2(kf.x, kf.x), pack2(kf.y, kf.y), pack2(kf.z, kf.z), pack2(kf.w, kf.w)};
#pragma unroll
          for (int i = 0; i < TR / 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              acc[2 * i][4 * g + j] = fma2(q[i].x, k2[j], acc[2 * i][4 * g + j]);
              acc[2 * i + 1][4 * g + j] = fma2(q[i].y, k2[j], acc[2 * i + 1][4 * g + j]);
            }
        }
      }
      if (it % SLICES == SLICES - 1) {                       // the tile's logits are complete
        const int t = tile0 + it / SLICES, key0 = t * KEYS;
        const bool masked = key0 + KEYS - 1 > min(P, n - 1); // some key of the tile is hidden from some row
#pragma unroll
        for (int i = 0; i < TR; ++i) {
          const int r = r0 + row_of(i);
          float x[TK];
#pragma unroll
          for (int j = 0; j < TK; ++j) {
            float even, odd;
            unpack2(acc[i / 2][j], even, odd);
            x[j] = (i & 1 ? odd : even) * p.scale_log2;
          }
          if (SCORES) {
#pragma unroll
            for (int j = 0; j < TK; ++j) sum[SCORES ? j : 0] += exp2f(x[j] - lse_s[SCORES ? row_of(i) : 0]);
            continue;
          }
          if (p.logits && r < p.rows) {
            float* to = p.logits + (head * p.rows + r) * p.ld_logits + key0;
#pragma unroll
            for (int j = 0; j < TK; j += 4)                  // within the row: ld_logits is a multiple of every tile
              *reinterpret_cast<float4*>(to + key_of(j)) = make_float4(x[j], x[j + 1], x[j + 2], x[j + 3]);
          }
          if (masked) {
            const int last = min(P + r % alpha, n - 1);      // row (g, j) sees keys 0 .. P + j that exist here
#pragma unroll
            for (int j = 0; j < TK; ++j) x[j] = key0 + key_of(j) <= last ? x[j] : -INFINITY;
          }
          float m = x[0];
#pragma unroll
          for (int j = 1; j < TK; ++j) m = fmaxf(m, x[j]);
#pragma unroll
          for (int o = 1; o < KT; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
          const float ref = m == -INFINITY ? 0.f : m;        // arguments at most 0, one of them 0: what flushes to zero does
          float z = 0.f;                                     // not count
#pragma unroll
          for (int j = 0; j < TK; ++j) z += ex2(x[j] - ref);
#pragma unroll
          for (int o = 1; o < KT; o <<= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
          if (tk == 0 && r < p.rows)
            p.partial[((tile_id + it / SLICES) * p.num_kv_heads + h) * p.rows + r] = make_float2(m, z);
        }
#pragma unroll
        for (int i = 0; i < TR / 2; ++i)
#pragma unroll
          for (int j = 0; j < TK; ++j) acc[i][j] = 0ull;
        if (SCORES && rb + 1 == blocks) {                    // the rows of a key are spread over RT threads
#pragma unroll
          for (int j = 0; j < TK; ++j) {
            part[SCORES ? tr : 0][SCORES ? key_of(j) : 0] = sum[SCORES ? j : 0];
            sum[SCORES ? j : 0] = 0.f;
          }
          __syncthreads();
          for (int x = threadIdx.x; x < KEYS; x += kGenThreads) {
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < RT; ++q) s += part[SCORES ? q : 0][SCORES ? x : 0];
            if (key0 + x < P) p.scores[head * p.ld_scores + key0 + x] = s;
          }
        }
      }
      if (it + 1 < steps) next.store(ks + ((it + 1) & 1) * (kGenSlice * KEYS));
      __syncthreads();
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
  const int t0 = p.seq.tile_off[b], t1 = p.seq.tile_off[b + 1];
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
  int t0 = p.seq.tile_off[b], t1 = p.seq.tile_off[b + 1];   // fp32-pipe path: one slot per tile
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
    t0 = c0 + hg;
    t1 = c1 + hg + 1;
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
