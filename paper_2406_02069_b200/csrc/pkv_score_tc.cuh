// Window-score kernels on the sm_100a tensor cores (Section 4.2.2, Eq. 2 and Eq. 3), bf16 or fp16 inputs.
//
// Two sweeps over K, because the score of a key sums softmax rows that each have
// their own normaliser (known only after a whole row has been seen):
//
//   sweep A  D[row r][key i] = Q K^T   (A operand = 128 window rows, B operand = 128-key tile)
//            TMEM lane = window row, so each epilogue thread owns one row and keeps its
//            reference exponent and sum of 2^x privately: no cross-thread reduction at all.
//   sweep B  D[key i][row r] = K Q^T   (A operand = 128-key tile, B operand = all window rows)
//            TMEM lane = key, so each epilogue thread owns one key and sums
//            2^(x_ri - lse2_r) over the rows r, reading lse2 from shared memory.
//
// x = (q . k) * log2(e) / sqrt(d).  Operands arrive by plain per-CTA TMA loads into
// 128-byte-swizzled shared memory; tcgen05.mma accumulates in TMEM (four
// accumulator stages of up to 128 columns); epilogue warps read TMEM with tcgen05.ld.
// Warp roles: warp 0 = TMA producer of K, warp 1 = MMA issuer and TMEM owner, warp 2 = TMA producer of Q, warp 3 = row
// statistics on their way out of sweep A and into sweep B, warps 4..19 = epilogue, four per scheduler: the exponentials (16 per
// clock per SM on their unit, a quarter of them on the FMA pipe) are the longest of the resources a tile needs, but no unit
// is the bound (see the split below: 0 to 4 pairs of eight make a few per cent).  The 16 epilogue
// warps form four groups (TMEM lane quarter = warp % 4, group = (warp - 4) / 4), each with
// an accumulator stage of its own, refilled while the other three compute.  CTAs are persistent: each takes a contiguous range of (sequence,
// KV head, key chunk) work items.
//
// Every wait on an mbarrier is bounded.  Sweep B's epilogue waits for sweep A, whose time that bound says nothing about, so
// the roles that wait for the epilogue wait for sweep A first (pdl_wait).  A wait that runs out sets an abort flag in
// shared memory and a status bit in the workspace; all roles then leave their loops,
// the producer drains the copies it still has in flight, TMEM is released and the
// kernel returns.
#pragma once

#include <cuda.h>

#include <type_traits>

#include "pkv_common.cuh"

namespace pkv {

constexpr int kTcThreads = 640;         // 20 warps: producer of K, MMA issuer, producer of Q, statistics, 16 epilogue
constexpr int kTcEpiWarp0 = 4;          // first epilogue warp
constexpr int kTcEpiWarps = 16;         // four per scheduler, which is what keeps the exp unit fed
constexpr int kTcTileKeys = 128;        // keys per K tile: the N of sweep A's MMAs, the M of sweep B's
constexpr int kTcStageCols = 128;       // TMEM columns of an accumulator stage
constexpr int kTcStages = 4;            // accumulator stages, one per group of epilogue warps
constexpr int kTcKBytes = 128 * 1024;   // shared memory given to K stages (4 x 32 KB at d = 128)
constexpr int kTcMaxGrid = 256;         // CTAs of a sweep at most (the workspace holds a partial segment per CTA)
constexpr int kTcPrefetchBytes = 128 * 1024;   // of K per CTA into the L2 ahead of the wait: what the start needs (more gains nothing)
constexpr int kTcMaxRows = 256;         // window rows (G * alpha) the tensor-core path takes
constexpr long long kTcWaitCycles = 1ll << 31;   // bound of any one wait, in SM clocks

struct TcParams {
  SeqTable seq;                 // stat_off / score_off count key tiles (of all keys / of the prefix)
  int32_t num_kv_heads, group, rows;      // rows = group * alpha (R)
  int32_t rows_pad;             // R rounded up to 32
  int32_t fp16;                 // 1: Q and K hold binary16, 0: bfloat16 (both operands always share the type)
  int32_t early;                // 1: start reading Q and K at once.  Sweep A: the caller vouches for them
                                // (PKV_FLAG_INPUTS_FINAL) and they are not outputs of a library kernel that may still
                                // run.  Sweep B behind a sweep A of the same call: A has waited for them
  int32_t prefetch_tiles;       // K tiles a CTA brings into the L2 while it waits for the kernels ahead
  int32_t withhold;             // test aid: CTA 0 of sweep A never loads its last K tile (its waits then run out)
  long long wait_clocks;        // bound of any one wait, in SM clocks
  int32_t row_blocks;           // ceil(R / 128): M-blocks of sweep A
  float scale_log2;             // log2(e) / sqrt(d)
  float2* partial;              // sweep A out: [segment][R] (reference exponent, sum); a segment is one CTA's run over one
                                // (sequence, head)
  const float* lse2;            // sweep B in:  [batch][H_kv][R] row normalisers (log of the row's sum of exps)
  float lse_scale, lse_add;     // lse2_r = lse2[r] * lse_scale + lse_add: (1, 0) for the library's own sweep A,
                                // (log2 e, log2 G) for natural-log normalisers handed in by the caller
  int32_t merge;                // sweep B: 1 = lse2 is not read; every CTA merges the partials of sweep A for the
                                // heads it works on (no merge kernel between the sweeps)
  int32_t stat_grid;            // CTAs sweep A ran with (which segments belong to a head follows from it)
  float log2_group;             // log2 G, added to the merged normalisers
  float* scores;                // sweep B out: [batch][H_kv][ld]
  int64_t ld_scores;
  uint32_t* status;
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Non-blocking test of a barrier phase.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Hardware-suspended wait for a barrier phase: the thread sleeps until the phase completes or the time hint (in
// nanoseconds) has passed, whichever comes first; returns false in the second case.  The hint matters: with the
// default (short) limit the waiting warps of this kernel spent a fifth of all issued instructions on re-trying.
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(20000u)
      : "memory");
  return ok != 0;
}
// Bounded wait.  The thread is suspended by the hardware between checks (no sleeping in software, which
// would add its wake-up latency to every hand-off of the pipeline).  Gives up after `limit` SM
// clocks (kTcWaitCycles, of the order of a second, unless a test lowers it) or when another thread gave up (abort flag); returns false then.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, long long limit) {
  if (mbar_try(bar, parity)) return true;
  const long long start = clock64();
  for (;;) {
    if (mbar_try(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - start > limit) break;
  }
  *abort_flag = 1;
  return false;
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                            int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}

// The same with a cache policy for the lines it brings into the L2.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3,
                                            uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_evict_first() {
  uint64_t policy;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  return policy;
}
// Brings a box of a tensor into the L2.
__device__ __forceinline__ void tma_prefetch_4d(const CUtensorMap* map, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global [%0, {%1, %2, %3, %4}];" ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0),
               "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}

// One lane of a converged warp, the same one each time.  The role of the MMA issuer is entered through it: an MMA takes its
// descriptors from uniform registers, and behind a test of the lane number the compiler does not know that there is one
// thread only and wraps every MMA in a loop over the lanes (some 100 clocks an MMA: 32k-token layer 62.6 us, 59.8 with this).
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok));
  return ok != 0;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma_f16kind(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The special-function unit evaluates 16 exponentials per clock per SM, which is what bounds both
// sweeps when every 2^x goes through it.  A fixed share of the exponentials is therefore evaluated on
// the FMA pipe instead, two at a time with the packed fp32 instructions.  Of every eight consecutive
// pairs of values (16 accumulator columns), kTcPolyPairs go this way, spread evenly over the eight.  Measured at 0 / 1 / 2 /
// 3 / 4 of 8: one layer of 131072 tokens (at the board's power cap) 211 / 206 / 209 / 213 / 223 us, 32768 tokens 54.8 / 53.6
// / 54.0 / 53.5 / 55.1 us, 32 ragged layers 2.71 / 2.70 / 2.76 / 2.82 / 2.87 ms.  2 rather than 1: which columns take the cubic
// moves the scores by 2e-6, enough to exchange positions at the edge of a list now and then, and stays as it was.
#ifndef PKV_POLY_PAIRS
#define PKV_POLY_PAIRS 2
#endif
constexpr int kTcPolyPairs = PKV_POLY_PAIRS;    // 0 = every exponential on the special-function unit
__host__ __device__ constexpr bool tc_pair_is_poly(int pair) {
  return ((pair % 8 + 1) * kTcPolyPairs) / 8 != ((pair % 8) * kTcPolyPairs) / 8;
}

__device__ __forceinline__ float fma_sat(float a, float b, float c) {   // a * b + c clamped to [0, 1]
  float d;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// acc + (2^x0, 2^x1), evaluated on the FMA pipe.
//   y = sat((x + 126) / 253)            one instruction rescales x and clamps it to [-126, 127], so that the
//                                       exponent arithmetic below cannot wrap (-inf and NaN give y = 0)
//   t = 253 y + (1.5 * 2^23 + 1)        rounds to an integer: the low mantissa bits of t hold n + 127, n = round(x)
//   f = 253 y + (1.5 * 2^23 + 1 - t)    = x - n in [-0.5, 0.5]
//   2^f by a cubic minimax polynomial (largest relative error 7.5e-5, far inside the 2e-3 the scores are held to);
//   2^n is the float whose exponent field is n + 127, i.e. t << 23;  result = acc + 2^f * 2^n.
__device__ __forceinline__ unsigned long long ex2_poly_add(float x0, float x1, unsigned long long acc) {
  const float kMagic1 = 12582913.0f;
  const float y0 = fma_sat(x0, 1.0f / 253.0f, 126.0f / 253.0f), y1 = fma_sat(x1, 1.0f / 253.0f, 126.0f / 253.0f);
  const unsigned long long y = pack2(y0, y1), k253 = pack2(253.0f, 253.0f), km = pack2(kMagic1, kMagic1);
  const unsigned long long t = fma2(y, k253, km);
  const unsigned long long g = fma2(t, pack2(-1.0f, -1.0f), km);
  const unsigned long long f = fma2(y, k253, g);
  unsigned long long q = fma2(f, pack2(0.0551716685295105f, 0.0551716685295105f),
                              pack2(0.2426111251115799f, 0.2426111251115799f));
  q = fma2(q, f, pack2(0.6932609677314758f, 0.6932609677314758f));
  q = fma2(q, f, pack2(0.9999280571937561f, 0.9999280571937561f));
  float t0, t1;
  unpack2(t, t0, t1);
  const unsigned long long scale = pack2(__int_as_float(__float_as_int(t0) << 23), __int_as_float(__float_as_int(t1) << 23));
  return fma2(q, scale, acc);
}

// acc[j % 4] += (2^x0, 2^x1) for the eight packed pairs xs[j] of one 16-column chunk, each pair by the unit its
// position selects.
__device__ __forceinline__ void ex2_accumulate8(const unsigned long long (&xs)[8], unsigned long long (&acc)[4]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    float x0, x1;
    unpack2(xs[j], x0, x1);
    if (tc_pair_is_poly(j)) acc[j & 3] = ex2_poly_add(x0, x1, acc[j & 3]);
    else acc[j & 3] = add2(acc[j & 3], pack2(ex2(x0), ex2(x1)));
  }
}

// Sweep A, 16 logits of one window row, fast path: acc += 2^(v_j * c2 - m) in four packed pairs of partial sums.
// m is a reference exponent, not necessarily the running maximum; the caller adds the partial sums up once per
// unit and falls back to rowstats_rescue when the total is not a moderate finite number.
__device__ __forceinline__ void rowstats_accumulate(const uint32_t (&v)[16], unsigned long long cc,
                                                    unsigned long long mm, unsigned long long (&acc)[4]) {
  unsigned long long xs[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) xs[j] = fma2(pack2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])), cc, mm);
  ex2_accumulate8(xs, acc);
}
__device__ __forceinline__ float sum_pairs(const unsigned long long (&acc)[4]) {
  float a[8];
#pragma unroll
  for (int q = 0; q < 4; ++q) unpack2(acc[q], a[2 * q], a[2 * q + 1]);
  return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}
// Sweep A, slow path for the same 16 logits: moves the reference exponent up to a whole number at or above the
// running maximum first (a logit some 60 binades above the reference, or one that is not finite).
// `live` is false for threads that only keep the warp's loads aligned.
__device__ __forceinline__ void rowstats_rescue(const uint32_t (&v)[16], float c2, bool live, float& m, float& z) {
  if (!live) return;
  float gm = __uint_as_float(v[0]);
#pragma unroll
  for (int j = 1; j < 16; ++j) gm = fmaxf(gm, __uint_as_float(v[j]));
  const float mn = fmaxf(m, ceilf(gm * c2));
  z *= ex2(m - mn);
  m = mn;
  float g = 0.f;
#pragma unroll
  for (int j = 0; j < 16; ++j) g += ex2(fmaf(__uint_as_float(v[j]), c2, -m));
  z += g;
}

// Sweep B, 16 window rows of one key: acc += 2^(v_j * c2 + nlse_j); nlse = -lse2 sits in shared memory
// (negated when it was loaded), acc holds four packed pairs of partial sums.
__device__ __forceinline__ void score_group(const uint32_t (&v)[16], unsigned long long cc, const float* nlse,
                                            unsigned long long (&acc)[4]) {
  unsigned long long xs[8];
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const ulonglong2 l = *reinterpret_cast<const ulonglong2*>(nlse + 2 * j);   // four floats as two packed pairs
    xs[j] = fma2(pack2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])), cc, l.x);
    xs[j + 1] = fma2(pack2(__uint_as_float(v[2 * j + 2]), __uint_as_float(v[2 * j + 3])), cc, l.y);
  }
  ex2_accumulate8(xs, acc);
}

// Shared-memory matrix descriptor of a K-major bf16 operand whose rows are 128 bytes wide and
// stored with the 128-byte swizzle: 8-row groups are 1024 bytes apart.  `addr` is the byte address
// of the first row, plus 32 bytes per 16-element step along the contraction dimension.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);          // start address
  d |= static_cast<uint64_t>(1) << 16;                         // leading byte offset (unused with swizzle), 16 B
  d |= static_cast<uint64_t>(1024 >> 4) << 32;                 // stride byte offset: 1024 B between 8-row groups
  d |= static_cast<uint64_t>(1) << 46;                         // descriptor version of this architecture
  d |= static_cast<uint64_t>(2) << 61;                         // 128-byte swizzle
  return d;
}
// Instruction descriptor: 16-bit x 16-bit -> fp32, both operands K-major and of one type (format code 1 =
// bf16, 0 = fp16, for A at bit 7 and B at bit 10), M x N tile.
__device__ __forceinline__ uint32_t instr_desc_16bit(int M, int N, int fp16) {
  const uint32_t fmt = fp16 ? 0u : 1u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}

// Work item -> (sequence, head, chunk).  Items are ordered sequence, head, chunk (in the sweeps a chunk is a key tile).
struct TcItem { int b, h, c, nchunks; };
__device__ __forceinline__ TcItem tc_item(const int32_t* off, int batch, int heads, int id) {
  int b = 0;
  while (b + 1 < batch && id >= heads * off[b + 1]) ++b;
  const int local = id - heads * off[b];
  const int nc = off[b + 1] - off[b];
  return TcItem{b, local / nc, local % nc, nc};
}

// Sweep A: row r of a finished run, from the (reference, sum of 2^(x - reference)) pairs that the epilogue warps hold of it
// ([4 groups][128 lanes]; one pair per group that works on the row's block and per copy of the rows; (-inf, 0): no key).
__device__ __forceinline__ float2 run_row(const float2* runs, int r, bool two_blocks, int copies) {
  float m = -INFINITY, z = 0.f;
  const int step = two_blocks ? 2 : 1, first = two_blocks ? r >> 7 : 0;
  for (int c = 0; c < copies; ++c) {
    const float2* at = runs + c * (128 / copies) + (r & 127);
    float2 o[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) o[g] = first + g * step < 4 ? at[(first + g * step) * 128] : make_float2(-INFINITY, 0.f);
    const float mn = fmaxf(m, fmaxf(fmaxf(o[0].x, o[1].x), fmaxf(o[2].x, o[3].x)));
    if (mn > -INFINITY) {
      z = z * ex2(m - mn) + ((o[0].y * ex2(o[0].x - mn) + o[1].y * ex2(o[1].x - mn)) +
                             (o[2].y * ex2(o[2].x - mn) + o[3].y * ex2(o[3].x - mn)));
      m = mn;
    }
  }
  return make_float2(m, z);
}

// Segments t, t + per_row, ... < s1 of sweep A's partials, of U rows from r on, r_step apart, in batches of Q loads:
// (reference, sum) added to m, z.  How many are loaded at a time does not change a bit of the result as long as one batch
// holds them all, or Q is the same.  The loads are unconditional (of the last row and segment where there is none), so
// that all of a batch are in flight.
template <int U, int Q>
__device__ __forceinline__ void tc_fold_segments(const float2* partial, int r, int r_step, int rows, int t, int s1, int per_row,
                                                 float* m, float* z) {
  for (; t < s1; t += Q * per_row) {
    float2 pz[U][Q];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int q = 0; q < Q; ++q)
        pz[u][q] = __ldcg(partial + static_cast<int64_t>(min(t + q * per_row, s1 - 1)) * rows + min(r + u * r_step, rows - 1));
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float mn = m[u];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        if (q > 0 && t + q * per_row >= s1) pz[u][q] = make_float2(-INFINITY, 0.f);
        mn = fmaxf(mn, pz[u][q].x);
      }
      if (mn > -INFINITY) {                                    // (-inf, 0) marks a segment that saw no key of this row
        z[u] = __fmul_rn(z[u], ex2(m[u] - mn));
#pragma unroll
        for (int q = 0; q < Q; ++q) z[u] = fmaf(pz[u][q].y, ex2(pz[u][q].x - mn), z[u]);
        m[u] = mn;
      }
    }
  }
}

// Two lanes' (reference, sum) of one row; the first operand is the one of the lower lane.
__device__ __forceinline__ float2 tc_merge_pair(float2 a, float2 b) {
  const float mm = fmaxf(a.x, b.x);
  return make_float2(mm, __fadd_rn(a.x > -INFINITY ? __fmul_rn(a.y, ex2(a.x - mm)) : 0.f,
                                   b.x > -INFINITY ? __fmul_rn(b.y, ex2(b.x - mm)) : 0.f));
}

// What PER_ROW lanes with at most Q segments each make of a row, by one lane.
template <int PER_ROW, int Q>
__device__ __forceinline__ float2 tc_merge_row(const float2* row, int rows, int s0, int s1) {
  float2 pz[Q][PER_ROW];
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int i = 0; i < PER_ROW; ++i) pz[q][i] = __ldcg(row + static_cast<int64_t>(min(s0 + q * PER_ROW + i, s1 - 1)) * rows);
  float2 lane[PER_ROW];
#pragma unroll
  for (int i = 0; i < PER_ROW; ++i) {
    lane[i] = s0 + i < s1 ? pz[0][i] : make_float2(-INFINITY, 0.f);
    if (Q == 2 && s0 + PER_ROW + i < s1) {
      const float mn = fmaxf(lane[i].x, pz[Q - 1][i].x);
      if (mn > -INFINITY)
        lane[i] = make_float2(mn, fmaf(pz[Q - 1][i].y, ex2(pz[Q - 1][i].x - mn), __fmul_rn(lane[i].y, ex2(lane[i].x - mn))));
    }
  }
#pragma unroll
  for (int o = 1; o < PER_ROW; o <<= 1)
#pragma unroll
    for (int i = 0; i < PER_ROW; i += 2 * o) lane[i] = tc_merge_pair(lane[i], lane[i + o]);
  return lane[0];
}

// Sweep A's partials of a head -> its negated row normalisers in dst (-inf for the padding rows), by THREADS threads (the sixteen
// epilogue warps, eight or one).  Every CTA that works on a head merges it for itself, and equal keys must get equal scores whichever CTA has them, so the additions come in the same order whoever does
// it: 2 to 16 lanes per row by the number of rows alone, each with every per_row-th segment, then pairwise.  A single warp
// does the same with a lane per row where the head has few segments (what it has to save there are instructions, beside
// four warps of the epilogue on its scheduler), else in sixteen steps, four at a time if it can (L2 latencies).
template <int THREADS, bool ACCURATE, typename Params>
__device__ __forceinline__ void tc_merge_head(const Params& p, int b, int h, int tid, float* dst) {
  constexpr int kSteps = kTcEpiWarps * 32 / THREADS;           // of THREADS / per_row rows
  const int rows_p2 = p.rows_pad <= 32 ? 32 : (p.rows_pad <= 64 ? 64 : (p.rows_pad <= 128 ? 128 : 256));
  const int per_row = kTcEpiWarps * 32 / rows_p2, r_step = THREADS / per_row;
  const int hg = b * p.num_kv_heads + h;
  // sweep A's CTAs took contiguous item ranges (items ordered sequence, head, chunk): the first `rem`
  // CTAs per + 1 items, the others per; this head's items fell to CTAs c0..c1, one segment each
  const int nc = p.seq.stat_off[b + 1] - p.seq.stat_off[b];
  const int total_a = p.num_kv_heads * p.seq.stat_off[p.seq.batch];
  const int per_a = total_a / p.stat_grid, rem_a = total_a % p.stat_grid, edge = rem_a * (per_a + 1);
  const int i0 = p.num_kv_heads * p.seq.stat_off[b] + h * nc, i1 = i0 + nc - 1;
  const int c0 = i0 < edge ? i0 / (per_a + 1) : rem_a + (i0 - edge) / per_a;
  const int c1 = i1 < edge ? i1 / (per_a + 1) : rem_a + (i1 - edge) / per_a;
  const int s0 = c0 + hg, s1 = c1 + hg + 1;
  const int part = tid % per_row;
  pdl_wait();                                                  // the partials are written by the kernel before
  // log2f costs the warp that merges ahead of sweep B's epilogue some instructions (three steps of two sequences at head size
  // 64: 33.7 -> 34.2 us); the exponentials of the score sweeps are not as exact as __log2f
  auto log_of = [](float x) { return ACCURATE ? log2f(x) : __log2f(x); };
  // U steps from `step` on, segments in batches of Q
  auto some = [&](int step, auto u_const, auto q_const) {
    constexpr int U = decltype(u_const)::value, Q = decltype(q_const)::value;
    const int r0 = step * r_step + tid / per_row;
    float m[U], z[U];
#pragma unroll
    for (int u = 0; u < U; ++u) { m[u] = -INFINITY; z[u] = 0.f; }
    tc_fold_segments<U, Q>(p.partial, r0, r_step, p.rows, s0 + part, s1, per_row, m, z);
    for (int o = 1; o < per_row; o <<= 1) {
#pragma unroll
      for (int u = 0; u < U; ++u) {                            // both partners of a pair compute the same merged value
        const float2 both = tc_merge_pair(make_float2(m[u], z[u]), make_float2(__shfl_xor_sync(0xffffffffu, m[u], o),
                                                                               __shfl_xor_sync(0xffffffffu, z[u], o)));
        m[u] = both.x;
        z[u] = both.y;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = r0 + u * r_step;
      if (part == 0) dst[r] = r < p.rows ? -(m[u] + log_of(z[u]) + p.log2_group) : -INFINITY;
    }
  };
  using std::integral_constant;
  if constexpr (kSteps == 1) {
    some(0, integral_constant<int, 1>{}, integral_constant<int, 10>{});
  } else {
    auto lane_a_row = [&](auto lanes, auto q_const) {
#pragma unroll 1
      for (int r = tid; r < rows_p2; r += THREADS) {
        const float2 mz = tc_merge_row<decltype(lanes)::value, decltype(q_const)::value>(p.partial + min(r, p.rows - 1), p.rows, s0, s1);
        dst[r] = r < p.rows ? -(mz.x + log_of(mz.y) + p.log2_group) : -INFINITY;
      }
    };
    if (s1 - s0 <= min(2 * per_row, 16)) {
      if (per_row == 2) lane_a_row(integral_constant<int, 2>{}, integral_constant<int, 2>{});
      else if (per_row == 4) lane_a_row(integral_constant<int, 4>{}, integral_constant<int, 2>{});
      else if (per_row == 8) lane_a_row(integral_constant<int, 8>{}, integral_constant<int, 2>{});
      else lane_a_row(integral_constant<int, 16>{}, integral_constant<int, 1>{});
    } else if (s1 - s0 <= 5 * per_row) {
      constexpr int kAtOnce = kSteps < 4 ? kSteps : 4;
#pragma unroll 1
      for (int step = 0; step < kSteps; step += kAtOnce) some(step, integral_constant<int, kAtOnce>{}, integral_constant<int, 5>{});
    } else {
#pragma unroll 1
      for (int step = 0; step < kSteps; ++step) some(step, integral_constant<int, 1>{}, integral_constant<int, 10>{});
    }
  }
}

// Sweep B: the same from the caller's values (or the merge kernel's), or from sweep A's partials.
template <int THREADS>
__device__ __forceinline__ void tc_normalisers(const TcParams& p, int b, int h, int tid, float* dst) {
  if (p.merge) {
    tc_merge_head<THREADS, false>(p, b, h, tid, dst);
    return;
  }
  const int rows_p2 = p.rows_pad <= 32 ? 32 : (p.rows_pad <= 64 ? 64 : (p.rows_pad <= 128 ? 128 : 256));
  const float* lse2 = p.lse2 + (static_cast<int64_t>(b) * p.num_kv_heads + h) * p.rows;
  pdl_wait();                                                  // normalisers may be written by a kernel before
  for (int r = tid; r < rows_p2; r += THREADS) dst[r] = r < p.rows ? -fmaf(lse2[r], p.lse_scale, p.lse_add) : -INFINITY;
}

// The item behind (REVERSE: before) w; behind the last one w stays on its sequence.
template <bool REVERSE>
__device__ __forceinline__ void tc_next(const int32_t* off, int batch, int heads, TcItem& w) {
  if (REVERSE) {
    if (--w.c >= 0) return;
    if (--w.h < 0) {
      w.h = heads - 1;
      if (w.b > 0) { --w.b; w.nchunks = off[w.b + 1] - off[w.b]; }
    }
    w.c = w.nchunks - 1;
  } else {
    if (++w.c < w.nchunks) return;
    w.c = 0;
    if (++w.h == heads) {
      w.h = 0;
      if (w.b + 1 < batch) { ++w.b; w.nchunks = off[w.b + 1] - off[w.b]; }
    }
  }
}

// Dynamic shared memory carve-up (bytes), all regions 1024-aligned.
template <int D>
struct TcSmem {
  static constexpr int kHalves = D / 64;                       // 64-element (128-byte) column blocks
  static constexpr int kQBytes = kTcMaxRows * D * 2;
  static constexpr int kQOff = 0;
  static constexpr int kKOff = kQBytes;
  static constexpr int kMiscOff = kKOff + kTcKBytes;
  static constexpr int kMiscBytes = 20 * 1024;                 // barriers, exchange buffers, per-warp lse2 copies
  static constexpr int kTotal = kMiscOff + kMiscBytes + 1024;  // + slack for manual 1024-byte alignment
};

// SWEEP 0 = row statistics (A), 1 = scores (B).
template <int D, int SWEEP>
__global__ void __launch_bounds__(kTcThreads, 1)
score_tc_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                const TcParams p) {
  using L = TcSmem<D>;
  constexpr int kTileKeys = kTcTileKeys;
  // Sweep B walks each CTA's items and tiles from the last to the first: sweep A has just read the same keys in
  // ascending order, so the end of every range is what the L2 still holds.
  constexpr bool kReverse = SWEEP == 1;
  constexpr int kStageBytes = kTileKeys * D * 2;               // one K tile in shared memory
  constexpr int kKStages = kTcKBytes / kStageBytes >= 4 ? 4 : kTcKBytes / kStageBytes;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + (-smem_u32(smem_raw) & 1023u);   // (an offset, so that accesses stay known as shared memory)
  uint8_t* q_s = smem + L::kQOff;
  uint8_t* k_s = smem + L::kKOff;
  uint8_t* misc = smem + L::kMiscOff;
  uint64_t* bars = reinterpret_cast<uint64_t*>(misc);          // [0..3] k_full, [4..7] k_empty, [8..11] t_full,
                                                               // [12..15] t_empty, [16..17] q_full, [18..19] q_empty,
                                                               // [20..21] x_full, [22..23] x_empty, [24..25] n_full,
                                                               // [26..27] n_empty, [28] meet
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc + 256);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 260);
  float* xch = reinterpret_cast<float*>(misc + 1024);          // sweep B: [2][128] partial sums handed between groups
  float* lse_all = reinterpret_cast<float*>(misc + 4096);      // sweep B: [2][256] -lse2 of the current / next head
  float2* run_all = reinterpret_cast<float2*>(misc + 8192);    // sweep A: [2][4 groups][128 lanes] (reference, sum) of a run

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = smem_u32(bars);
  auto k_full = [&](int s) { return bar0 + 8u * s; };
  auto k_empty = [&](int s) { return bar0 + 8u * (4 + s); };
  auto t_full = [&](int s) { return bar0 + 8u * (8 + s); };
  auto t_empty = [&](int s) { return bar0 + 8u * (12 + s); };
  auto q_full = [&](int s) { return bar0 + 8u * (16 + s); };
  auto q_empty = [&](int s) { return bar0 + 8u * (18 + s); };
  auto x_full = [&](int s) { return bar0 + 8u * (20 + s); };
  auto x_empty = [&](int s) { return bar0 + 8u * (22 + s); };
  // n: the buffers that go through warp 3, the runs' statistics in sweep A, the heads' normalisers in sweep B
  auto n_full = [&](int s) { return bar0 + 8u * (24 + s); };
  auto n_empty = [&](int s) { return bar0 + 8u * (26 + s); };
  const uint32_t meet = bar0 + 8u * 28;

  // A unit of work is an accumulator stage of up to 128 columns: one K tile and up to 128 window rows.  With more rows a
  // tile makes two units: sweep A takes the rows in blocks of 128, sweep B in halves (columns [0, split) and [split, R)).
  // Each of the four groups of epilogue warps owns one stage and takes every fourth unit, so that three groups compute
  // while the stage of the fourth is filled.  (Two stages of 256 columns with a pair of groups each left a pair idle for
  // the 1400 clocks of the refill: 75 us of sweep A for 131072 keys x 256 rows x 8 heads, 68 with these.)
  const bool two_blocks = p.row_blocks == 2;
  const int split_b = two_blocks ? ((p.rows_pad / 2) + 31) & ~31 : p.rows_pad;
  // Sweep A: with 64 (32) rows or fewer the window rows stand two (four) times in the 128 rows of the Q tile, and each
  // copy's lanes take their share of the key columns: otherwise the sub-partitions of the padding rows would idle.
  const int copies = SWEEP == 1 || p.rows > 64 ? 1 : (p.rows > 32 ? 2 : 4);
  const int copy_rows = 128 / copies;
  // Up to 128 rows: Q tiles of two heads, so that a CTA's next head is in place when its turn comes.
  const int q_slots = p.rows <= 128 ? 2 : 1;

  // ---- set-up (shared memory and TMEM only: it may overlap the tail of the preceding kernel)
  // Sweep A lets sweep B start once it knows itself that Q and K are complete, so that B can read them at once.
  if (SWEEP == 1 || p.early) pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < 4; ++s) { mbar_init(k_full(s), 1); mbar_init(k_empty(s), 1); }
    for (int s = 0; s < kTcStages; ++s) { mbar_init(t_full(s), 1); mbar_init(t_empty(s), 4); }
    for (int s = 0; s < 2; ++s) { mbar_init(q_full(s), 1); mbar_init(q_empty(s), 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(x_full(s), 4); mbar_init(x_empty(s), 4); }
    for (int s = 0; s < 2; ++s) {
      mbar_init(n_full(s), SWEEP == 0 ? kTcEpiWarps : 1);
      mbar_init(n_empty(s), SWEEP == 0 ? 1 : kTcEpiWarps);
    }
    mbar_init(meet, kTcEpiWarps);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // rows of the Q tile beyond R stay zero for the whole kernel (TMA only ever writes R rows)
  for (int i = threadIdx.x; i < L::kQBytes / 16; i += kTcThreads) reinterpret_cast<uint4*>(q_s)[i] = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // ---- this CTA's contiguous range of key tiles
  const int32_t* off = SWEEP == 0 ? p.seq.stat_off : p.seq.score_off;
  const int total = p.num_kv_heads * off[p.seq.batch];
  const int per = total / gridDim.x, rem = total % gridDim.x;
  const int item0 = blockIdx.x * per + min(static_cast<int>(blockIdx.x), rem);
  const int item1 = item0 + per + (static_cast<int>(blockIdx.x) < rem ? 1 : 0);
  const int ntiles = item1 - item0;
  auto first_tile = [&]() { return tc_item(off, p.seq.batch, p.num_kv_heads, kReverse ? item1 - 1 : item0); };
  auto next_tile = [&](TcItem& w) { tc_next<kReverse>(off, p.seq.batch, p.num_kv_heads, w); };

  // Copies and MMAs touch only the caller's Q and K.  With `early` they start at once, beside the tail of the kernels
  // ahead in the stream; then sweep A waits just before its first write (its partials), sweep B just before it reads
  // the row normalisers, and both wait again before they end.  Without it the kernel waits here, and spends
  // the time on bringing its first K tiles into the L2: a prefetch hands no data to anybody, so it does not matter
  // whether the kernels ahead still write them.
  if (!p.early) {
    if (warp == 0 && lane == 0) {
      TcItem w = first_tile();
      for (int half = 0; half < L::kHalves; ++half) tma_prefetch_4d(&q_map, half * 64, 0, w.h * p.group, w.b);
      for (int it = 0; it < min(ntiles, p.prefetch_tiles); ++it, next_tile(w))
        for (int half = 0; half < L::kHalves; ++half) tma_prefetch_4d(&k_map, half * 64, w.c * kTileKeys, w.h, w.b);
    }
    pdl_wait();
    if (SWEEP == 0) pdl_trigger();
  }

  if (warp == 0) {
    // =========================================================== TMA producer of K
    if (lane == 0) {
      uint32_t it = 0;                                         // K tiles
      // behind a sweep A this is the last time a tile is read
      const uint64_t policy = l2_evict_first();
      bool ok = true;
      TcItem w = first_tile();
      for (; static_cast<int>(it) < ntiles; ++it, next_tile(w)) {
        const int s = it % kKStages;
        if (SWEEP == 1 && it == static_cast<uint32_t>(kKStages + kTcStages / p.row_blocks)) pdl_wait();
        ok = mbar_wait(k_empty(s), ((it / kKStages) & 1) ^ 1, abort_flag, p.wait_clocks);
        if (!ok) break;
        if (SWEEP == 0 && p.withhold && blockIdx.x == 0 && static_cast<int>(it) + 1 == ntiles) continue;   // test aid: never arrives
        mbar_expect_tx(k_full(s), kStageBytes);
        for (int half = 0; half < L::kHalves; ++half) {
          const uint32_t dst = smem_u32(k_s) + s * kStageBytes + half * kTileKeys * 128;
          if (SWEEP == 1 && p.merge) tma_load_4d(dst, &k_map, k_full(s), half * 64, w.c * kTileKeys, w.h, w.b, policy);
          else tma_load_4d(dst, &k_map, k_full(s), half * 64, w.c * kTileKeys, w.h, w.b);
        }
      }
      if (!ok) {
        // drain: wait (bounded) for the copies still in flight before shared memory is given up
        const uint32_t first = it > kKStages ? it - kKStages : 0;
        for (uint32_t j = first; j < it; ++j)
          for (uint32_t spin = 0; spin < (1u << 16) && !mbar_test(k_full(j % kKStages), (j / kKStages) & 1); ++spin)
            __nanosleep(64);
      }
    }
  } else if (warp == 2) {
    // =========================================================== TMA producer of Q, one tile per head
    if (lane == 0) {
      uint32_t heads = 0;
      int cur_b = -1, cur_h = -1;
      bool ok = true;
      TcItem w = first_tile();
      for (int ii = 0; ii < ntiles; ++ii, next_tile(w)) {
        if (w.b == cur_b && w.h == cur_h) continue;
        cur_b = w.b; cur_h = w.h;
        const uint32_t slot = heads % q_slots, round = heads / q_slots;
        if (SWEEP == 1 && heads == static_cast<uint32_t>(q_slots)) pdl_wait();
        ok = mbar_wait(q_empty(slot), (round & 1) ^ 1, abort_flag, p.wait_clocks);
        if (!ok) break;
        mbar_expect_tx(q_full(slot), static_cast<uint32_t>(copies * p.rows) * D * 2);
        for (int half = 0; half < L::kHalves; ++half)
          for (int c = 0; c < copies; ++c)
            tma_load_4d(smem_u32(q_s) + half * kTcMaxRows * 128 + (slot * 128 + c * copy_rows) * 128, &q_map, q_full(slot),
                        half * 64, 0, w.h * p.group, w.b);
        ++heads;
      }
      if (!ok)
        for (uint32_t j = heads > 2 ? heads - 2 : 0; j < heads; ++j)
          for (uint32_t spin = 0; spin < (1u << 16) && !mbar_test(q_full(j % q_slots), (j / q_slots) & 1); ++spin)
            __nanosleep(64);
    }
  } else if (warp == 1) {
    // =========================================================== MMA issuer
    if (elect_one()) {
      uint32_t it = 0, u = 0, heads = 0;                       // it counts K tiles, u accumulator units
      int cur_b = -1, cur_h = -1;
      bool ok = true;
      const uint32_t idesc0 = SWEEP == 0 ? instr_desc_16bit(128, kTileKeys, p.fp16) : instr_desc_16bit(kTileKeys, split_b, p.fp16);
      const uint32_t idesc1 = SWEEP == 0 || !two_blocks ? idesc0 : instr_desc_16bit(kTileKeys, p.rows_pad - split_b, p.fp16);
      uint32_t slot = 0;
      TcItem w = first_tile();
      for (; static_cast<int>(it) < ntiles && ok; ++it) {
        if (w.b != cur_b || w.h != cur_h) {
          slot = heads % q_slots;
          ok = mbar_wait(q_full(slot), (heads / q_slots) & 1, abort_flag, p.wait_clocks);
          if (!ok) break;
          ++heads;
          cur_b = w.b; cur_h = w.h;
        }
        {
          const int s = it % kKStages;
          ok = mbar_wait(k_full(s), (it / kKStages) & 1, abort_flag, p.wait_clocks);
          if (!ok) break;
          const uint32_t k_addr = smem_u32(k_s) + s * kStageBytes;
          const uint32_t q_addr = smem_u32(q_s) + slot * 128 * 128;
          for (int rb = 0; rb < p.row_blocks && ok; ++rb, ++u) {
            const int ts = u % kTcStages;
            if (SWEEP == 1 && u == kTcStages) pdl_wait();
            ok = mbar_wait(t_empty(ts), ((u / kTcStages) & 1) ^ 1, abort_flag, p.wait_clocks);
            if (!ok) break;
            tc_fence_after();
            const uint32_t d_addr = tmem_base + ts * kTcStageCols;
            const uint32_t idesc = rb == 0 ? idesc0 : idesc1;
            const int row_at = SWEEP == 0 ? rb * 128 : rb * split_b;     // first window row of the unit
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint32_t qa = q_addr + (kk / 4) * kTcMaxRows * 128 + row_at * 128 + (kk % 4) * 32;
              const uint32_t ka = k_addr + (kk / 4) * kTileKeys * 128 + (kk % 4) * 32;
              if (SWEEP == 0) tc_mma_f16kind(d_addr, smem_desc_sw128(qa), smem_desc_sw128(ka), idesc, kk > 0);
              else tc_mma_f16kind(d_addr, smem_desc_sw128(ka), smem_desc_sw128(qa), idesc, kk > 0);
            }
            tc_commit(t_full(ts));
          }
          if (ok) tc_commit(k_empty(s));
        }
        // does the next tile belong to another head?  then Q may be overwritten after these MMAs
        next_tile(w);
        if (ok && (w.b != cur_b || w.h != cur_h || static_cast<int>(it) + 1 == ntiles)) tc_commit(q_empty(slot));
      }
    }
  } else if (warp == 3) {
    // =========================================================== statistics between the sweeps, off the epilogue's path
    // Sweep A: merges what the sixteen warps hold of a finished run and writes one (reference, sum) per window row, to
    // the segment numbered blockIdx.x + head: along the item order either the CTA or the head advances from one run to
    // the next, so the numbers are distinct, and a head's segments follow from the CTAs its items fall to.
    // Sweep B: the normalisers of the CTA's second and later heads, while the epilogue works on the head before.
    uint32_t heads = 0;
    int cur_b = -1, cur_h = -1;
    bool ok = true;
    if (SWEEP == 0) pdl_wait();                                // the partials of the call before have been read
    auto finish = [&](int b, int h) {
      if (SWEEP == 0) {
        const uint32_t buf = heads & 1u;
        ok = mbar_wait(n_full(buf), (heads >> 1) & 1, abort_flag, p.wait_clocks);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return;
        const float2* runs = run_all + buf * 512;
        const int64_t seg = static_cast<int64_t>(blockIdx.x) + b * p.num_kv_heads + h;
        for (int r = lane; r < p.rows; r += 32) p.partial[seg * p.rows + r] = run_row(runs, r, two_blocks, copies);
        __syncwarp();
        if (lane == 0) mbar_arrive(n_empty(buf));
      } else if (heads > 0) {
        const uint32_t buf = heads & 1u;
        if (heads > 1) {
          ok = mbar_wait(n_empty(buf), ((heads >> 1) & 1) ^ 1, abort_flag, p.wait_clocks);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) return;
        }
        tc_normalisers<32>(p, b, h, lane, lse_all + buf * 256);
        __syncwarp();
        if (lane == 0) mbar_arrive(n_full(buf));
      }
      ++heads;
    };
    TcItem w = first_tile();
    for (int ii = 0; ii < ntiles && ok; ++ii, next_tile(w)) {
      if (w.b == cur_b && w.h == cur_h) continue;
      if (SWEEP == 0 && ii > 0) finish(cur_b, cur_h);          // a run that has ended; the last one is the epilogue's
      cur_b = w.b; cur_h = w.h;
      if (SWEEP == 1) finish(w.b, w.h);
    }
  } else {
    // =========================================================== epilogue
    const int e = warp - kTcEpiWarp0;
    const int quarter = warp & 3;               // TMEM lanes 32*quarter .. +31 are this warp's
    const int grp = e >> 2;                     // 0..3
    const int blk = two_blocks ? grp & 1 : 0;   // row block (half) of its units
    const int par = grp >> 1;                   // two blocks: parity of its K tiles
    const int lane_row = quarter * 32 + lane;   // TMEM lane of this thread
    const float c2 = p.scale_log2;
    uint32_t u = 0, mine = 0;                   // units seen by the CTA / read by this group
    uint32_t heads = 0;                         // (sequence, head) changes so far
    const float* lse_s = lse_all;               // sweep B: the current head's -lse2
    int cur_b = -1, cur_h = -1;
    bool ok = true;
    // Sweep A: a thread's (reference, sum) runs on over consecutive work items of one (sequence, head), then goes to warp 3
    // (the CTA's last one, which the end of the kernel waits for, is merged by all epilogue warps together).
    float m = -INFINITY, z = 0.f;
    auto flush_run = [&]() -> bool {            // hands run number heads - 1 over
      const uint32_t run = heads - 1, buf = run & 1u;
      bool good = mbar_wait(n_empty(buf), ((run >> 1) & 1) ^ 1, abort_flag, p.wait_clocks);
      good = __all_sync(0xffffffffu, good);
      if (!good) return false;
      run_all[buf * 512 + grp * 128 + lane_row] = make_float2(m, z);
      __syncwarp();
      if (lane == 0) mbar_arrive(n_full(buf));
      m = -INFINITY;
      z = 0.f;
      return true;
    };
    TcItem w = first_tile();
    int n = 0, P = 0;
    const int alpha = p.seq.alpha;
    float* srow = nullptr;                      // sweep B: the head's scores
    for (int ii = 0; ii < ntiles && ok; ++ii, next_tile(w)) {
      const bool new_head = w.b != cur_b || w.h != cur_h;
      if (new_head) { n = p.seq.n[w.b]; P = p.seq.prefix[w.b]; }
      if (SWEEP == 0) {
        // thread -> window row (and, with copies of the rows, share of the columns), the same in all units of the group: a
        // thread keeps one (reference, sum) per run of work items.
        const int r = blk * 128 + lane_row % copy_rows;
        const int last_visible = min(P + (r % alpha), n - 1); // row (g, j) sees keys 0 .. P + j that exist here
        const int cols = 128 / copies;                        // this thread's key columns of a unit
        const int col0 = (lane_row / copy_rows) * cols;
        // a warp whose 32 TMEM lanes are all padding rows has nothing to evaluate
        const bool warp_has_rows = blk * 128 + (quarter * 32) % copy_rows < p.rows;
        if (new_head) {
          if (heads > 0) ok = flush_run();
          if (!ok) break;
          cur_b = w.b; cur_h = w.h;
          ++heads;
        }
        {
          for (int rb = 0; rb < p.row_blocks && ok; ++rb, ++u) {
            if (static_cast<int>(u % kTcStages) != grp) continue;        // another group's unit
            ok = mbar_wait(t_full(grp), (u / kTcStages) & 1, abort_flag, p.wait_clocks);
            ok = __all_sync(0xffffffffu, ok);                 // whole warp proceeds together or not at all
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + grp * kTcStageCols + col0;
            const int key_base = w.c * kTileKeys + col0;
            if (!warp_has_rows) {
              // only the hand-shake below
            } else if (key_base + cols - 1 <= min(P, n - 1)) {   // every key visible to every row: no mask
              // fast path over the columns; the sums are only looked at once, at the end
              // 16-column loads, double buffered: the next load is in flight while a chunk is evaluated
              uint32_t va[16], vb[16];
              tc_ld16(taddr, va);
              if (m == -INFINITY) {                           // a new run: any of the row's logits will do as the reference
                tc_wait_ld();
                float gm = __uint_as_float(va[0]);
#pragma unroll
                for (int j = 1; j < 16; ++j) gm = fmaxf(gm, __uint_as_float(va[j]));
                m = ceilf(gm * c2);
              }
              const unsigned long long cc = pack2(c2, c2), mm = pack2(-m, -m);
              unsigned long long acc[4] = {pack2(0.f, 0.f), pack2(0.f, 0.f), pack2(0.f, 0.f), pack2(0.f, 0.f)};
              if (copies == 1) {
#pragma unroll
                for (int cg = 0; cg < 128; cg += 32) {
                  tc_wait_ld();
                  tc_ld16(taddr + cg + 16, vb);
                  rowstats_accumulate(va, cc, mm, acc);
                  tc_wait_ld();
                  if (cg + 32 < 128) tc_ld16(taddr + cg + 32, va);
                  rowstats_accumulate(vb, cc, mm, acc);
                }
              } else {
                for (int cg = 0; cg < cols; cg += 32) {
                  tc_wait_ld();
                  tc_ld16(taddr + cg + 16, vb);
                  rowstats_accumulate(va, cc, mm, acc);
                  tc_wait_ld();
                  if (cg + 32 < cols) tc_ld16(taddr + cg + 32, va);
                  rowstats_accumulate(vb, cc, mm, acc);
                }
              }
              const float g = sum_pairs(acc);
              const bool good = g < 1.0e18f;                  // false for inf and NaN too
              if (good) z += g;
              if (!__all_sync(0xffffffffu, good)) {           // rare: the warp reads its columns again, slow path
                for (int cg = 0; cg < cols; cg += 16) {
                  tc_ld16(taddr + cg, va);
                  tc_wait_ld();
                  rowstats_rescue(va, c2, !good, m, z);
                }
              }
            } else {
              for (int cg = 0; cg < cols; cg += 16) {
                uint32_t v[16];
                tc_ld16(taddr + cg, v);
                tc_wait_ld();
                float gm = -INFINITY;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                  const bool vis = key_base + cg + j <= last_visible;
                  const float x = vis ? __uint_as_float(v[j]) * c2 : -INFINITY;
                  v[j] = __float_as_uint(x);
                  gm = fmaxf(gm, x);
                }
                if (gm > -INFINITY) {
                  const float mn = fmaxf(m, ceilf(gm));
                  z *= ex2(m - mn);
                  m = mn;
                  float a0 = 0.f;
#pragma unroll
                  for (int j = 0; j < 16; ++j) a0 += ex2(__uint_as_float(v[j]) - m);
                  z += a0;
                }
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(t_empty(grp));
          }
        }
        if (!ok) break;
      } else {
        // thread -> key.  The head's normalisers, negated (the epilogue adds them), sit in one of two buffers that alternate
        // from head to head.  The first one is filled by the sixteen warps together, which then meet; the others by warp 3,
        // ahead of time.  They come from the caller (or the merge kernel), or straight from sweep A's partials of the head,
        // which every CTA that works on it merges for itself, always in the same order (see tc_merge_head).
        if (new_head) {
          const uint32_t buf = heads & 1u;
          if (heads == 0) {
            tc_normalisers<kTcEpiWarps * 32>(p, w.b, w.h, e * 32 + lane, lse_all);
            __syncwarp();
            if (lane == 0) mbar_arrive(meet);
            ok = mbar_wait(meet, 0, abort_flag, p.wait_clocks);
          } else {
            __syncwarp();
            if (lane == 0) mbar_arrive(n_empty(buf ^ 1u));    // done with the head before
            ok = mbar_wait(n_full(buf), buf == 1u ? (heads >> 1) & 1 : ((heads >> 1) & 1) ^ 1, abort_flag, p.wait_clocks);
          }
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          lse_s = lse_all + buf * 256;
          cur_b = w.b; cur_h = w.h;
          srow = p.scores + (static_cast<int64_t>(w.b) * p.num_kv_heads + w.h) * p.ld_scores;
          ++heads;
        }
        const float* nlse = lse_s + (blk ? split_b : 0);
        const int cols = blk ? p.rows_pad - split_b : split_b;
        // a key's rows are summed in two halves whether one group or two of them take its tile: the same rounding either way
        const int split_sum = two_blocks ? 0 : ((p.rows_pad / 2) + 31) & ~31;
        const bool ours = (u + blk) % kTcStages == static_cast<uint32_t>(grp);   // or another group's unit
        const uint32_t phase = (u / kTcStages) & 1;
        u += p.row_blocks;
        if (ours) {
          ok = mbar_wait(t_full(grp), phase, abort_flag, p.wait_clocks);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
          const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + grp * kTcStageCols;
          unsigned long long acc[4] = {pack2(0.f, 0.f), pack2(0.f, 0.f), pack2(0.f, 0.f), pack2(0.f, 0.f)};
          const unsigned long long cc = pack2(c2, c2);
          float head_sum = 0.f;
          {
            uint32_t va[16], vb[16];
            tc_ld16(taddr, va);
            for (int cg = 0; cg < cols; cg += 32) {
              tc_wait_ld();
              tc_ld16(taddr + cg + 16, vb);
              score_group(va, cc, nlse + cg, acc);
              tc_wait_ld();
              if (cg + 32 < cols) tc_ld16(taddr + cg + 32, va);
              score_group(vb, cc, nlse + cg + 16, acc);
              if (cg + 32 == split_sum) {
                head_sum = sum_pairs(acc);
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] = 0ull;
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(t_empty(grp));
          float sum = head_sum + sum_pairs(acc);
          if (two_blocks) {                                   // the second half's group hands its partial sum to the first's
            if (blk == 1) {
              ok = mbar_wait(x_empty(par), (mine & 1) ^ 1, abort_flag, p.wait_clocks);
              ok = __all_sync(0xffffffffu, ok);
              if (!ok) break;
              xch[par * 128 + lane_row] = sum;
              __syncwarp();
              if (lane == 0) mbar_arrive(x_full(par));
            } else {
              ok = mbar_wait(x_full(par), mine & 1, abort_flag, p.wait_clocks);
              ok = __all_sync(0xffffffffu, ok);
              if (!ok) break;
              sum += xch[par * 128 + lane_row];
              __syncwarp();
              if (lane == 0) mbar_arrive(x_empty(par));
            }
          }
          ++mine;
          const int i = w.c * kTileKeys + lane_row;
          if (blk == 0 && i < P) srow[i] = sum;
        }
      }
    }
    if (SWEEP == 0 && ok && heads > 0 && flush_run()) {       // the CTA's last run
      const uint32_t run = heads - 1;
      if (mbar_wait(n_full(run & 1u), (run >> 1) & 1, abort_flag, p.wait_clocks)) {
        pdl_wait();                                           // the partials of the call before have been read
        const int r = e * 32 + lane;
        if (r < p.rows)
          p.partial[(static_cast<int64_t>(blockIdx.x) + cur_b * p.num_kv_heads + cur_h) * p.rows + r] =
              run_row(run_all + (run & 1u) * 512, r, two_blocks, copies);
      }
    }
  }

  // ---- teardown
  pdl_wait();                                                  // never finish before the kernels ahead in the stream
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicOr(p.status, kStatusWaitExpired);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

}  // namespace pkv
