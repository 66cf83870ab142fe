// Window logits of fp32 inputs on the sm_100a tensor cores (Section 4.2.2, Eq. 2): every fp32 value is the exact sum of
// three bfloat16 values (8 + 8 + 8 significant bits, rounded to nearest, remainders exact), and of the nine products of
// two such triples the six largest are formed, with fp32 accumulation:
//
//   q . k = sum (q_hi + q_mid + q_lo) (k_hi + k_mid + k_lo)  ~  hh + (hm + mh) + (hl + mm + lh)
//
// What is left out, (ml + lm) + ll, is at most about 2^-24 of a product of two magnitudes, as much as the rounding of one fp32
// multiply-add (a middle part is up to 2^-8 of its value, a low part up to 2^-17).  The small products come first and each half of the channels has an accumulator of its own, so that a logit goes through
// few roundings at full size (the accumulator of the tensor cores cuts off, it does not round).
//
//   split_logits_kernel     logits (key-major: the window rows of a key are consecutive) and row statistics, one segment
//                           per run of a CTA over the tiles of a (sequence, KV head, block of 128 rows)
//   split_scores_kernel     merges a head's segments, then s_i = sum_r 2^(x_ri - lse2[r] - log2 G) from the stored logits
//
// Why: 2 R n d flops per KV head are the bound of the fp32 pipe (8101 keys x 8 heads x 128 rows x 128 channels: 34 us at the
// 63 TFLOP/s that it reaches); six products on the tensor cores take 8 us.  Scores of that shape, both kernels: 79 us on
// the fp32 pipe, 33 here; the layer call 101 -> 54.  Error of the scores against 64 bits (2-norm / largest, relative): 2.1e-7 /
// 8.6e-7 on the fp32 pipe, 1.5e-7 / 5.4e-7 here, and no larger at ten other shapes (16 to 384 rows, d = 64 and 128).
// What is left: the first tile waits some 4 us for Q's parts, a tile takes some 2300 clocks where its MMAs take 1536, and the second
// kernel reads the logits at 3.3 TB/s out of the L2 (10 us).
//
// Warps 0..7 load a tile of 64 keys into registers, split it and store the parts swizzled as the MMAs want them (the loads of
// the next tile are under way while they wait for room); warp 16 issues the MMAs; warps 8..15 take the logits out of TMEM, a
// thread per window row, in two teams that take the tiles in turn (all of them on every tile: 1.8 us a tile, not 1.2).
// Tiles of 64 keys and not 128: two stages of parts fit beside Q's, and the tiles spread more evenly over the CTAs.
//
// Infinities, NaN and magnitudes of 2^59 or more raise a flag for their tile, whose logits are then formed by plain fp32
// multiply-adds, once the CTA is through with the others (sp_plain_tiles).  Below that nothing overflows that the
// multiply-adds would not: the parts of 128 products add up to less than 2^126 in magnitude.  (Parts have either sign: of
// products near 2^128 some would become infinities of opposite signs, and NaN of a logit that is -inf.)  And parts that
// are subnormal and lost change no logit by more than 2^-59.
#pragma once

#include "pkv_score_generic.cuh"
#include "pkv_score_tc.cuh"

namespace pkv {

constexpr int kSpThreads = 544;             // 8 warps that split, 8 that take the logits, the MMA issuer
constexpr int kSpConverters = 256;
constexpr int kSpKeys = 64;                 // keys of a tile: the N of an MMA
constexpr int kSpRows = 128;                // window rows of a block: the M
constexpr int kSpStages = 2;                // of K parts, and of accumulators
constexpr int kSpAccs = 2;                  // accumulators of a tile, each for its share of the channels
constexpr int kSpMaxGrid = 256;
constexpr int kSpPrefetch = 8;              // K tiles (32 KB each at d = 128) on their way into the L2 ahead of their use
constexpr int kSpMaxTiles = 32768;          // of a CTA: a bit for each (with one CTA 256 MB of logits take at most 31800, of 33 rows each)
constexpr float kSpMost = 5.7646075230342349e17f;              // 2^59
constexpr int kSpSumKeys = 128;             // split_scores_kernel: keys per CTA
constexpr int kSpSumThreads = 256;

template <int D>
struct SpSmem {
  static constexpr int kQPart = kSpRows * D * 2;               // bytes of one part
  static constexpr int kKPart = kSpKeys * D * 2;
  static constexpr int kQOff = 0;
  static constexpr int kKOff = 3 * kQPart;
  static constexpr int kMiscOff = kKOff + kSpStages * 3 * kKPart;
  static constexpr int kMiscBytes = 2048 + kSpMaxTiles / 8;
  static constexpr int kTotal = kMiscOff + kMiscBytes + 1024;  // + slack for manual 1024-byte alignment
};

// Where the runs of the CTAs over unit (sequence, head, row block) number `unit` went: segments [s0, s1).
__device__ __forceinline__ void sp_segments(const ScoreParams& p, int b, int unit_in_seq, int units, int& s0, int& s1) {
  if (p.per_unit > 0) {
    s0 = (b * units + unit_in_seq) * (p.per_unit + 1);
    s1 = s0 + p.per_unit;
    return;
  }
  const int nc = p.seq.stat_off[b + 1] - p.seq.stat_off[b];
  const int total = units * p.seq.stat_off[p.seq.batch];
  const int per = total / p.stat_grid, rem = total % p.stat_grid, edge = rem * (per + 1);
  const int i0 = units * p.seq.stat_off[b] + unit_in_seq * nc, i1 = i0 + nc - 1;
  const int c0 = i0 < edge ? i0 / (per + 1) : rem + (i0 - edge) / per;
  const int c1 = i1 < edge ? i1 / (per + 1) : rem + (i1 - edge) / per;
  s0 = c0 + b * units + unit_in_seq;
  s1 = c1 + b * units + unit_in_seq + 1;
}

// What a thread has seen of the values it split: the largest magnitude, and a zero that infinities and NaN turn into NaN.
struct SpSeen {
  float most = 0.f;
  unsigned long long zero = 0ull;
  __device__ __forceinline__ bool special() const {
    float a, b;
    unpack2(zero, a, b);
    return !(most < kSpMost) || !(a == 0.f) || !(b == 0.f);
  }
};

// Eight consecutive channels of a row -> their three parts, eight bfloat16 each.
__device__ __forceinline__ void sp_split8(const float4& a, const float4& b, uint4& hi, uint4& mid, uint4& lo, SpSeen& seen) {
  const float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  uint32_t h[4], m[4], l[4];
  auto bf16x2 = [](float low, float high) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(low, high);
    return *reinterpret_cast<const uint32_t*>(&v);
  };
  auto widen = [](uint32_t u) { return pack2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)); };
  const unsigned long long minus = pack2(-1.f, -1.f);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    unsigned long long r = pack2(x[2 * i], x[2 * i + 1]);
    float r0, r1;
    seen.most = fmaxf(seen.most, fmaxf(fabsf(x[2 * i]), fabsf(x[2 * i + 1])));
    seen.zero = fma2(r, 0ull, seen.zero);
    h[i] = bf16x2(x[2 * i], x[2 * i + 1]);
    r = fma2(widen(h[i]), minus, r);                           // exact
    unpack2(r, r0, r1);
    m[i] = bf16x2(r0, r1);
    r = fma2(widen(m[i]), minus, r);
    unpack2(r, r0, r1);
    l[i] = bf16x2(r0, r1);
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  mid = make_uint4(m[0], m[1], m[2], m[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}
__device__ __forceinline__ void sp_store16(uint32_t to, const uint4& v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(to), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// Keys of a unit's head; window row r of it (of its KV head, over all blocks).
__device__ __forceinline__ const float* sp_keys(const ScoreParams& p, const TcItem& w, int blocks) {
  return static_cast<const float*>(p.k.ptr) + w.b * p.k.sb + (w.h / blocks) * p.k.sh;
}
__device__ __forceinline__ const float* sp_q_row(const ScoreParams& p, const TcItem& w, int blocks, int r) {
  const int alpha = p.seq.alpha;
  return static_cast<const float*>(p.q.ptr) + w.b * p.q.sb + static_cast<int64_t>((w.h / blocks) * p.group + r / alpha) * p.q.sh +
         (r % alpha) * p.q.st;
}

// The flagged tiles of a CTA, after all others: logits by multiply-adds, each summed in the order of its channels as on the fp32
// pipe, and their row statistics added to those of the CTA's runs.  By all threads, with the shared memory that the parts have
// left: a unit's window rows channel-major, a tile's keys row-major, two window rows and eight keys per thread.
// Scores of 8101 keys x 8 heads x 128 rows with every tile flagged: 115 us, one tile in a head 43 (none: 33, the fp32 pipe 79).  In the epilogue's
// own loop, a window row and a key at a time, 4430 and 660; eight keys at a time 445, and every call 0.9 us longer by the registers.
template <int D>
__device__ __forceinline__ void sp_plain_tiles(const ScoreParams& p, float* qs, float* ks, float2* part, const uint32_t* flagged, int item0,
                                               int ntiles) {
  constexpr int kThreads = 512, kGroups = 8, kKeys = kSpKeys / kGroups;        // groups of threads, each with its keys
  static_assert(kSpRows / 2 * kGroups == kThreads, "two rows per thread");
  const int tid = threadIdx.x, row = tid % (kSpRows / 2) * 2, kg = tid / (kSpRows / 2);
  const int blocks = (p.rows + kSpRows - 1) / kSpRows, units = p.num_kv_heads * blocks;
  const int32_t* off = p.seq.stat_off;
  int cur_b = -1, cur_h = -1;
  TcItem w = tc_item(off, p.seq.batch, units, item0);
  for (int it = 0; it < ntiles; ++it, tc_next<false>(off, p.seq.batch, units, w)) {
    if (!((flagged[it >> 5] >> (it & 31)) & 1u)) continue;
    const int r0 = (w.h % blocks) * kSpRows, n = p.seq.n[w.b], key0 = w.c * kSpKeys;
    __syncthreads();                                           // the tile before has been read
    if (tid < kThreads) {
      if (w.b != cur_b || w.h != cur_h) {
        const int x = tid % kSpRows;
        for (int c = tid / kSpRows * 4; c < D; c += kThreads / kSpRows * 4) {
          const float4 f = r0 + x < p.rows ? *reinterpret_cast<const float4*>(sp_q_row(p, w, blocks, r0 + x) + c) : make_float4(0.f, 0.f, 0.f, 0.f);
          qs[c * kSpRows + x] = f.x;
          qs[(c + 1) * kSpRows + x] = f.y;
          qs[(c + 2) * kSpRows + x] = f.z;
          qs[(c + 3) * kSpRows + x] = f.w;
        }
      }
      for (int i = tid; i < kSpKeys * D / 4; i += kThreads) {
        const int key = key0 + i / (D / 4);
        reinterpret_cast<float4*>(ks)[i] = key < n ? *reinterpret_cast<const float4*>(sp_keys(p, w, blocks) + key * p.k.st + i % (D / 4) * 4)
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    cur_b = w.b;
    cur_h = w.h;
    __syncthreads();
    if (tid < kThreads) {
      unsigned long long x2[kKeys] = {};
#pragma unroll 2
      for (int c = 0; c < D; c += 4) {
        unsigned long long q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = *reinterpret_cast<const unsigned long long*>(qs + (c + u) * kSpRows + row);
#pragma unroll
        for (int j = 0; j < kKeys; ++j) {
          const float4 k = *reinterpret_cast<const float4*>(ks + (kg * kKeys + j) * D + c);
          x2[j] = fma2(q[0], pack2(k.x, k.x), x2[j]);
          x2[j] = fma2(q[1], pack2(k.y, k.y), x2[j]);
          x2[j] = fma2(q[2], pack2(k.z, k.z), x2[j]);
          x2[j] = fma2(q[3], pack2(k.w, k.w), x2[j]);
        }
      }
      const int first = key0 + kg * kKeys;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = r0 + row + i, last = min(p.seq.prefix[w.b] + r % p.seq.alpha, n - 1);
        float* to = p.logits + ((static_cast<int64_t>(w.b) * p.num_kv_heads + w.h / blocks) * p.ld_logits + first) * p.rows + r;
        float x[kKeys], m = -INFINITY, z = 0.f;
#pragma unroll
        for (int j = 0; j < kKeys; ++j, to += p.rows) {
          float even, odd;
          unpack2(x2[j], even, odd);
          x[j] = (i == 0 ? even : odd) * p.scale_log2;
          if (r < p.rows) *to = x[j];                          // (within the padded length)
          if (first + j > last) x[j] = -INFINITY;
          m = fmaxf(m, x[j]);
        }
        const float ref = m == -INFINITY ? 0.f : m;
#pragma unroll
        for (int j = 0; j < kKeys; ++j) z += ex2(x[j] - ref);
        part[kg * kSpRows + row + i] = make_float2(m, z);
      }
    }
    __syncthreads();
    if (tid < kSpRows && r0 + tid < p.rows) {
      float2* of_run = p.partial + (static_cast<int64_t>(blockIdx.x) + w.b * units + w.h) * p.rows + r0 + tid;
      float2 s = *of_run;
#pragma unroll
      for (int g = 0; g < kGroups; ++g) {
        const float2 o = part[g * kSpRows + tid];
        const float mn = fmaxf(s.x, o.x), ref = mn == -INFINITY ? 0.f : mn;
        s = make_float2(mn, s.y * ex2(s.x - ref) + o.y * ex2(o.x - ref));
      }
      *of_run = s;
    }
  }
}

// grid: at most one CTA per SM, block kSpThreads, dynamic shared memory SpSmem<D>::kTotal.
template <int D>
__global__ void __launch_bounds__(kSpThreads, 1) split_logits_kernel(const __grid_constant__ ScoreParams p) {
  using L = SpSmem<D>;
  constexpr int kChunks = D / 8;                               // 16-byte chunks of a part's row
  constexpr int kSteps = kSpKeys * kChunks / kSpConverters;    // chunks of a K tile per converter thread
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + (-smem_u32(smem_raw) & 1023u);   // (an offset, so that accesses stay known as shared memory)
  uint8_t* misc = smem + L::kMiscOff;
  uint64_t* bars = reinterpret_cast<uint64_t*>(misc);          // k_full, k_empty, t_full, t_empty (two of each), x_full, x_empty
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc + 192);                                      // (one a quarter)
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 196);
  volatile int* any_flagged = reinterpret_cast<volatile int*>(misc + 200);
  volatile int* special = reinterpret_cast<volatile int*>(misc + 256);         // [8]: tiles with values that are not split
  volatile int* q_special = reinterpret_cast<volatile int*>(misc + 288);       // [8]: the same of the units' window rows
  float2* halves = reinterpret_cast<float2*>(misc + 1024);                     // [128] statistics of the second team
  uint32_t* flagged = reinterpret_cast<uint32_t*>(misc + 2048);                // a bit per tile of this CTA
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = smem_u32(bars), smem0 = smem_u32(smem);
  auto k_full = [&](int s) { return bar0 + 8u * s; };
  auto k_empty = [&](int s) { return bar0 + 8u * (2 + s); };
  auto t_full = [&](int s) { return bar0 + 8u * (4 + s); };
  auto t_empty = [&](int s) { return bar0 + 8u * (6 + s); };
  auto x_full = [&](int q) { return bar0 + 8u * (8 + q); };
  auto x_empty = [&](int q) { return bar0 + 8u * (12 + q); };
  const uint32_t q_full = bar0 + 8u * 16;

  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSpStages; ++s) {
      mbar_init(k_full(s), kSpConverters / 32);
      mbar_init(k_empty(s), 1);
      mbar_init(t_full(s), 1);
      mbar_init(t_empty(s), 4);
    }
    for (int q = 0; q < 4; ++q) { mbar_init(x_full(q), 1); mbar_init(x_empty(q), 1); }
    mbar_init(q_full, 2 * kSpConverters / 32);
    *abort_flag = *any_flagged = 0;
    for (int i = 0; i < 8; ++i) special[i] = q_special[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < kSpMaxTiles / 32; i += kSpThreads) flagged[i] = 0;
  constexpr uint32_t kCols = kSpStages * kSpAccs * kSpKeys;
  if (warp == 16) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // this CTA's contiguous range of tiles; a unit is a block of rows of a KV head of a sequence
  const int blocks = (p.rows + kSpRows - 1) / kSpRows, units = p.num_kv_heads * blocks;
  const int32_t* off = p.seq.stat_off;
  const int total = units * off[p.seq.batch];
  const int per = total / gridDim.x, rem = total % gridDim.x;
  int item0 = blockIdx.x * per + min(static_cast<int>(blockIdx.x), rem);
  int ntiles = per + (static_cast<int>(blockIdx.x) < rem ? 1 : 0);
  if (p.per_unit > 0) {
    const int nc = off[1], part = blockIdx.x % p.per_unit, first = part * nc / p.per_unit;
    item0 = blockIdx.x / p.per_unit * nc + first;
    ntiles = (part + 1) * nc / p.per_unit - first;
  }
  const int alpha = p.seq.alpha;
  // Chunk c of row x of a part of `rows` rows: 64 channels to a row of 128 bytes, its 16-byte chunks exchanged by the row.
  auto place = [](int rows, int x, int c) { return (c >> 3) * rows * 128 + x * 128 + (((c & 7) ^ (x & 7)) << 4); };
  // Chunks [begin, end) of the window rows of w's unit, by 256 threads; returns whether this thread saw a value that is not split.
  auto convert_q = [&](const TcItem& w, int tid, int begin, int end) -> bool {
    constexpr int kBatch = 2;
    static_assert(kSpRows * kChunks / 2 % (kBatch * kSpConverters) == 0, "halves in whole steps");
    const int r0 = (w.h % blocks) * kSpRows;
    SpSeen seen;
#pragma unroll 1
    for (int i0 = begin + tid; i0 < end; i0 += kBatch * kSpConverters) {
      float4 f[kBatch][2];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int x = (i0 + u * kSpConverters) / kChunks, c = (i0 + u * kSpConverters) % kChunks;
        f[u][0] = f[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + x < p.rows) {
          const float4* src = reinterpret_cast<const float4*>(sp_q_row(p, w, blocks, r0 + x) + c * 8);
          f[u][0] = src[0];
          f[u][1] = src[1];
        }
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int x = (i0 + u * kSpConverters) / kChunks, c = (i0 + u * kSpConverters) % kChunks;
        uint4 hi, mid, lo;
        sp_split8(f[u][0], f[u][1], hi, mid, lo, seen);
        const uint32_t to = smem0 + L::kQOff + place(kSpRows, x, c);
        sp_store16(to, hi);
        sp_store16(to + L::kQPart, mid);
        sp_store16(to + 2 * L::kQPart, lo);
      }
    }
    return seen.special();
  };
  // K tiles into the L2: the first ones while the kernels ahead finish, then each as many tiles ahead of its use.
  auto prefetch_tile = [&](const TcItem& w) {
    const int key = w.c * kSpKeys + static_cast<int>(threadIdx.x) / (D / 32);
    if (threadIdx.x < kSpKeys * (D / 32) && key < p.seq.n[w.b])
      asm volatile("prefetch.global.L2 [%0];" ::"l"(sp_keys(p, w, blocks) + key * p.k.st + threadIdx.x % (D / 32) * 32));
  };
  static_assert(kSpKeys * (D / 32) <= kSpConverters, "a line per thread");
  TcItem ahead = tc_item(off, p.seq.batch, units, item0);
  if (warp >= 8 && warp < 16)
    for (int i = threadIdx.x - kSpConverters; i < kSpRows * (D / 32); i += kSpConverters) {
      const int r = (ahead.h % blocks) * kSpRows + i / (D / 32);
      if (r < p.rows) asm volatile("prefetch.global.L2 [%0];" ::"l"(sp_q_row(p, ahead, blocks, r) + i % (D / 32) * 32));
    }
  if (warp < 8)
    for (int it = 0; it < min(ntiles, kSpPrefetch); ++it, tc_next<false>(off, p.seq.batch, units, ahead)) prefetch_tile(ahead);
  pdl_wait();

  const long long limit = p.wait_clocks;
  if (warp < 8) {
    // =========================================================== converters
    TcItem w = tc_item(off, p.seq.batch, units, item0);
    float4 f[kSteps][2];
    auto load_tile = [&](const TcItem& t) {
      constexpr int kRows = kSpConverters / kChunks;           // per step
      const int n = p.seq.n[t.b], key0 = t.c * kSpKeys + threadIdx.x / kChunks;
      const float* base = sp_keys(p, t, blocks) + key0 * p.k.st + threadIdx.x % kChunks * 8;
#pragma unroll
      for (int s = 0; s < kSteps; ++s) {
        if (key0 + s * kRows < n) {
          const float4* src = reinterpret_cast<const float4*>(base + s * kRows * p.k.st);
          f[s][0] = src[0];
          f[s][1] = src[1];
        } else {
          f[s][0] = f[s][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    };
    if (ntiles > 0) load_tile(w);
    int cur_b = w.b, cur_h = w.h, runs = 0;
    bool ok = true;
    auto have_q = [&](int parts) {                             // of the sixteen arrivals that a unit's rows take
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0)
        for (int i = 0; i < parts; ++i) mbar_arrive(q_full);
    };
    if (ntiles > 0) {                                          // the first unit's rows: half of them the epilogue's, which has time then
      if (convert_q(w, threadIdx.x, kSpRows * kChunks / 2, kSpRows * kChunks)) q_special[0] = 1;
      have_q(1);
    }
    for (int it = 0; it < ntiles; ++it) {
      const int s = it % kSpStages;
      if (w.b != cur_b || w.h != cur_h) {                      // another unit: its window rows, once the MMAs of the last are done
        ok = mbar_wait(k_empty((it - 1) % kSpStages), ((it - 1) / kSpStages) & 1, abort_flag, limit);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        cur_b = w.b; cur_h = w.h;
        ++runs;
        // (the epilogue is at most three tiles behind)
        if (threadIdx.x == 0) q_special[(runs + 4) & 7] = 0;
        if (convert_q(w, threadIdx.x, 0, kSpRows * kChunks)) q_special[runs & 7] = 1;
        have_q(2);
      }
      ok = mbar_wait(k_empty(s), ((it / kSpStages) & 1) ^ 1, abort_flag, limit);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      // (the MMAs that have made room here waited for the epilogue of four tiles ago, which was the last to read that flag)
      if (threadIdx.x == 0) special[(it + 4) & 7] = 0;
      SpSeen seen;
#pragma unroll
      for (int j = 0; j < kSteps; ++j) {
        const int i = j * kSpConverters + threadIdx.x;
        uint4 hi, mid, lo;
        sp_split8(f[j][0], f[j][1], hi, mid, lo, seen);
        const uint32_t to = smem0 + L::kKOff + s * 3 * L::kKPart + place(kSpKeys, i / kChunks, i % kChunks);
        sp_store16(to, hi);
        sp_store16(to + L::kKPart, mid);
        sp_store16(to + 2 * L::kKPart, lo);
      }
      if (seen.special()) special[it & 7] = 1;
      tc_next<false>(off, p.seq.batch, units, w);
      if (it + 1 < ntiles) load_tile(w);
      if (it + kSpPrefetch < ntiles) {
        prefetch_tile(ahead);
        tc_next<false>(off, p.seq.batch, units, ahead);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0 && !(p.withhold && blockIdx.x == 0 && it + 1 == ntiles)) mbar_arrive(k_full(s));
    }
  } else if (warp == 16) {
    // =========================================================== MMA issuer
    if (elect_one()) {
      const uint32_t idesc = instr_desc_16bit(kSpRows, kSpKeys, 0);
      const uint32_t q_addr = smem_u32(smem + L::kQOff);
      // (part of Q, part of K), the smallest products first
      constexpr int kTerms = 6;
      const int tq[kTerms] = {2, 1, 0, 1, 0, 0}, tk[kTerms] = {0, 1, 2, 0, 1, 0};
      bool ok = true;
      int cur_b = -1, cur_h = -1, runs = 0;
      TcItem w = tc_item(off, p.seq.batch, units, item0);
      for (int it = 0; it < ntiles && ok; ++it, tc_next<false>(off, p.seq.batch, units, w)) {
        const int s = it % kSpStages;
        if (w.b != cur_b || w.h != cur_h) {
          ok = mbar_wait(q_full, runs & 1, abort_flag, limit);
          if (!ok) break;
          ++runs;
          cur_b = w.b; cur_h = w.h;
        }
        ok = mbar_wait(k_full(s), (it / kSpStages) & 1, abort_flag, limit) &&
             mbar_wait(t_empty(s), ((it / kSpStages) & 1) ^ 1, abort_flag, limit);
        if (!ok) break;
        tc_fence_after();
        const uint32_t k_addr = smem_u32(smem + L::kKOff) + s * 3 * L::kKPart;
#pragma unroll
        for (int a = 0; a < kSpAccs; ++a) {
          const uint32_t d_addr = tmem_base + (s * kSpAccs + a) * kSpKeys;
#pragma unroll
          for (int t = 0; t < kTerms; ++t)
#pragma unroll
            for (int k0 = 0; k0 < D / 16 / kSpAccs; ++k0) {
              const int kk = a * (D / 16 / kSpAccs) + k0;
              const uint32_t qa = q_addr + tq[t] * L::kQPart + (kk / 4) * kSpRows * 128 + (kk % 4) * 32;
              const uint32_t ka = k_addr + tk[t] * L::kKPart + (kk / 4) * kSpKeys * 128 + (kk % 4) * 32;
              tc_mma_f16kind(d_addr, smem_desc_sw128(qa), smem_desc_sw128(ka), idesc, t > 0 || k0 > 0);
            }
        }
        tc_commit(t_full(s));
        tc_commit(k_empty(s));
      }
    }
  } else {
    // =========================================================== epilogue: two teams of four warps, each with an accumulator stage,
    // take the tiles in turn; thread = window row
    const int quarter = warp & 3, team = (warp - 8) >> 2;
    const int lane_row = quarter * 32 + lane;
    float m = -INFINITY, z = 0.f;
    uint32_t runs = 0;                                         // over units so far
    TcItem w = tc_item(off, p.seq.batch, units, item0);
    bool ok = true;
    if (ntiles > 0) {
      if (convert_q(w, threadIdx.x - kSpConverters, 0, kSpRows * kChunks / 2)) q_special[0] = 1;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(q_full);
    }
    int cur_b = -1, cur_h = -1, r = 0, n = 0, last = 0;        // of the unit: this thread's row, the last key it sees
    float* lrow = nullptr;                                     // ... its logits of key 0
    const unsigned long long scale = pack2(p.scale_log2, p.scale_log2);
    for (int it = 0; it < ntiles; ++it) {
      if (w.b != cur_b || w.h != cur_h) {
        cur_b = w.b; cur_h = w.h;
        const int h = w.h / blocks;
        r = (w.h - h * blocks) * kSpRows + lane_row;
        n = p.seq.n[w.b];
        last = min(p.seq.prefix[w.b] + r % alpha, n - 1);      // row (g, j) sees keys 0 .. P + j
        lrow = p.logits + (static_cast<int64_t>(w.b) * p.num_kv_heads + h) * p.ld_logits * p.rows + r;
      }
      const bool live = r < p.rows;
      if (it % kSpStages == team) {
        ok = mbar_wait(t_full(team), (it / kSpStages) & 1, abort_flag, limit);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const bool plain = special[it & 7] | q_special[runs & 7];              // left to sp_plain_tiles
        if (plain) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(t_empty(team));
            atomicOr(&flagged[it >> 5], 1u << (it & 31));
            *any_flagged = 1;
          }
        }
#pragma unroll 1
        for (int half = plain ? 2 : 0; half < 2; ++half) {
          const int key0 = w.c * kSpKeys + half * 32;
          const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + team * kSpAccs * kSpKeys + half * 32;
          unsigned long long x2[16];
#pragma unroll
          for (int a = 0; a < kSpAccs; ++a) {
            uint32_t v0[16], v1[16];
            tc_ld16(taddr + a * kSpKeys, v0);
            tc_ld16(taddr + a * kSpKeys + 16, v1);
            tc_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const unsigned long long y0 = pack2(__uint_as_float(v0[2 * j]), __uint_as_float(v0[2 * j + 1]));
              const unsigned long long y1 = pack2(__uint_as_float(v1[2 * j]), __uint_as_float(v1[2 * j + 1]));
              x2[j] = a == 0 ? y0 : add2(x2[j], y0);
              x2[8 + j] = a == 0 ? y1 : add2(x2[8 + j], y1);
            }
          }
          float x[32];
#pragma unroll
          for (int j = 0; j < 16; ++j) unpack2(mul2(x2[j], scale), x[2 * j], x[2 * j + 1]);
          if (half == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(t_empty(team));
          }
          if (live) {                                          // (within the padded length)
            float* to = lrow + static_cast<int64_t>(key0) * p.rows;
#pragma unroll
            for (int j = 0; j < 32; ++j, to += p.rows) *to = x[j];
          }
          if (key0 + 31 > min(p.seq.prefix[w.b], n - 1)) {     // some key is hidden from some row
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (key0 + j > last) x[j] = -INFINITY;
          }
          float gm = x[0];
#pragma unroll
          for (int j = 1; j < 32; ++j) gm = fmaxf(gm, x[j]);
          const float mn = fmaxf(m, gm), ref = mn == -INFINITY ? 0.f : mn;     // (a NaN among the logits shows in z)
          const unsigned long long minus = pack2(-ref, -ref);
          unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float d0, d1;
            unpack2(add2(pack2(x[2 * j], x[2 * j + 1]), minus), d0, d1);
            acc[j & 3] = add2(acc[j & 3], pack2(ex2(d0), ex2(d1)));
          }
          z = z * ex2(m - ref) + sum_pairs(acc);
          m = mn;
        }
      }
      const TcItem was = w;
      tc_next<false>(off, p.seq.batch, units, w);
      if (it + 1 == ntiles || w.b != was.b || w.h != was.h) {  // the run is over: the two teams meet
        if (team == 1) {
          ok = mbar_wait(x_empty(quarter), (runs & 1) ^ 1, abort_flag, limit);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          halves[lane_row] = make_float2(m, z);
          __syncwarp();
          if (lane == 0) mbar_arrive(x_full(quarter));
        } else {
          ok = mbar_wait(x_full(quarter), runs & 1, abort_flag, limit);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          const float2 o = halves[lane_row];
          __syncwarp();
          if (lane == 0) mbar_arrive(x_empty(quarter));
          const float mn = fmaxf(m, o.x), ref = mn == -INFINITY ? 0.f : mn;
          if (live)
            p.partial[(static_cast<int64_t>(blockIdx.x) + was.b * units + was.h) * p.rows + r] =
                make_float2(mn, z * ex2(m - ref) + o.y * ex2(o.x - ref));
        }
        ++runs;
        m = -INFINITY;
        z = 0.f;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*any_flagged && !*abort_flag)
    sp_plain_tiles<D>(p, reinterpret_cast<float*>(smem + L::kQOff), reinterpret_cast<float*>(smem + L::kKOff),
                      reinterpret_cast<float2*>(smem + L::kKOff + kSpKeys * D * 4), flagged, item0, ntiles);
  if (threadIdx.x == 0 && *abort_flag) atomicOr(p.status, kStatusWaitExpired);
  if (warp == 16) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kCols) : "memory");
  }
}

// grid (blocks of kSpSumKeys prefix keys of the longest sequence, H_kv, batch), block kSpSumThreads, dynamic shared memory
// rows floats.  A warp takes eight keys at a time, its lanes the rows of a key (consecutive in memory): 32 loads in flight per
// lane at 128 rows, and nine exchanges for the eight sums.
__global__ void __launch_bounds__(kSpSumThreads, 4) split_scores_kernel(const ScoreParams p) {
  extern __shared__ float lse_all[];
  pdl_trigger();
  const int h = blockIdx.y, b = blockIdx.z, P = p.seq.prefix[b];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blocks = (p.rows + kSpRows - 1) / kSpRows;
  // 1, 2, 4 or 8 adjacent lanes share a row's segments; where they lie is worked out ahead of the wait
  const int per_row = p.rows > 128 ? 1 : (p.rows > 64 ? 2 : (p.rows > 32 ? 4 : 8)), part = threadIdx.x % per_row;
  auto segments = [&](int r, int& s0, int& s1) {
    s0 = s1 = 0;
    if (r < p.rows) sp_segments(p, b, h * blocks + r / kSpRows, p.num_kv_heads * blocks, s0, s1);
  };
  int s0, s1;
  segments(threadIdx.x / per_row, s0, s1);
  pdl_wait();
  if (blockIdx.x * kSpSumKeys >= P) return;
  const int64_t head = static_cast<int64_t>(b) * p.num_kv_heads + h;
  auto load_segments = [&](int r, int t, float2 (&pz)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u)
      pz[u] = t + u * per_row < s1 ? __ldcg(p.partial + static_cast<int64_t>(t + u * per_row) * p.rows + r) : make_float2(-INFINITY, 0.f);
  };
  // the segments first, then, on their way while those are merged, the first eight keys' logits
  float2 pz[8];
  load_segments(threadIdx.x / per_row, s0 + part, pz);
  float v[8][4];
  auto load = [&](const float* x, int r0) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j][q] = r0 + 32 * q < p.rows ? __ldcg(x + j * p.rows + r0 + 32 * q) : 0.f;
  };
  bool first = true;
  if (blockIdx.x * kSpSumKeys + warp * 8 >= P) first = false;
  else load(p.logits + (head * p.ld_logits + blockIdx.x * kSpSumKeys + warp * 8) * p.rows, lane);
  for (int r0 = 0; r0 < p.rows; r0 += kSpSumThreads / per_row) {
    const int r = r0 + threadIdx.x / per_row;
    float m = -INFINITY, z = 0.f;
    if (r0 > 0) {
      segments(r, s0, s1);
      load_segments(r, s0 + part, pz);
    }
    for (int t = s0 + part; t < s1;) {
      float mn = m;
#pragma unroll
      for (int u = 0; u < 8; ++u) mn = fmaxf(mn, pz[u].x);
      const float ref = mn == -INFINITY ? 0.f : mn;
      z *= exp2f(m - ref);
#pragma unroll
      for (int u = 0; u < 8; ++u) z += pz[u].y * exp2f(pz[u].x - ref);
      m = mn;
      t += 8 * per_row;
      if (t < s1) load_segments(r, t, pz);
    }
    for (int o = 1; o < per_row; o <<= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, o), z2 = __shfl_xor_sync(0xffffffffu, z, o);
      const float mn = fmaxf(m, m2), ref = mn == -INFINITY ? 0.f : mn;
      z = z * exp2f(m - ref) + z2 * exp2f(m2 - ref);
      m = mn;
    }
    if (r < p.rows && part == 0) lse_all[r] = m + log2f(z) + p.log2_group;
  }
  __syncthreads();
  for (int i0 = blockIdx.x * kSpSumKeys + warp * 8; i0 < min(P, static_cast<int>(blockIdx.x + 1) * kSpSumKeys);
       i0 += kSpSumThreads / 32 * 8, first = false) {
    const float* x = p.logits + (head * p.ld_logits + i0) * p.rows;            // (eight keys lie within the padded length)
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int r0 = lane; r0 < p.rows; r0 += 128) {
      if (!first || r0 >= 128) load(x, r0);
      // 2^x without the scaling that a subnormal result needs, where none comes out (as good as always)
      float least = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float l = r0 + 32 * q < p.rows ? lse_all[r0 + 32 * q] : 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          v[j][q] -= l;
          least = fminf(least, v[j][q]);
        }
      }
      if (least < -126.f) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j][q] = exp2f(v[j][q]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j][q] = ex2(v[j][q]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float there = r0 + 32 * q < p.rows ? 1.f : 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] = fmaf(v[j][q], there, s[j]);
      }
    }
    int cnt = 8;
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) {                        // lane bit o picks the half of the keys a lane keeps
      const int rest = cnt / 2;
      const bool upper = (lane & o) != 0;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < rest) {
          const float send = upper ? s[j] : s[j + rest], keep = upper ? s[j + rest] : s[j];
          s[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      cnt = rest;
    }
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
    const int i = i0 + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    if ((lane & 3) == 0 && i < P) p.scores[head * p.ld_scores + i] = s[0];
  }
}

}  // namespace pkv
