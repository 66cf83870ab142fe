// Fused max-pool + per-head top-k + window retention (+ optional eviction by gather), Section 4.2.2.
//
// One thread-block cluster per (sequence, KV head).  The prefix positions are
// split into contiguous slices, one per CTA of the cluster, and inside a CTA into
// contiguous runs, one per warp, so that position order is (CTA rank, warp, order
// inside the warp's run).
//
//  1. Every CTA stages its slice of raw scores in shared memory (coalesced), pools
//     them (halo of (w-1)/2 scores on both sides, clipped to the prefix) into
//     order-preserving 32-bit keys held in registers.
//  2. Candidate filter.  Every thread remembers the largest key it produced.  The
//     k-th largest of those per-thread maxima is a lower bound of the k-th largest
//     key (k distinct keys >= it exist); its top 22 bits are found with two CTA-local
//     11-bit histogram passes.  The CTA writes the (key, position) pairs of its slice
//     that reach the bound, in position order, to its region of a scratch buffer in
//     global memory.  Typically a few times k pairs survive in the whole cluster; in
//     the worst case (all keys equal, or k larger than the thread count) all do.
//  3. After one cluster barrier CTA 0 alone finishes: it concatenates the regions
//     (they are already in position order), finds the k-th largest key T by a
//     most-significant-digit radix search in three passes (11, 11, 10 bits) over the
//     candidates, and emits
//       kept = { i : key_i > T } plus the leftmost (k - |{key > T}|) positions with key_i == T
//     in ascending position; the alpha window positions follow.
//  4. After a second cluster barrier all CTAs of the cluster copy the kept rows of K
//     and V (when asked to).
//
// Ties therefore go to the smaller position and the list is canonical.  Only
// block and cluster barriers are used for synchronisation (no flag spinning).
#pragma once

#include <cooperative_groups.h>

#include "pkv_common.cuh"
#include "pkv_paged.cuh"

namespace pkv {

namespace cg = cooperative_groups;

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelMaxCluster = 8;
constexpr int kSelBins = 2048;
constexpr int kSelSliceCap = 16384;        // positions a CTA can hold in shared memory (6 bytes each)
constexpr int kSelRunMax = kSelSliceCap / kSelWarps;   // positions per warp in that case
constexpr int kSelPerLane = kSelRunMax / 32;           // ... and per lane
constexpr int kSelHalo = 16;               // largest pool radius the shared-memory path stages

struct SelectParams {
  const float* scores;      // [batch][H_kv][ld]
  int64_t ld_scores;
  int32_t* indices;         // packed rows
  SeqTable seq;
  int32_t num_kv_heads;
  int32_t pool_radius;      // (w - 1) / 2
  int32_t cached;           // 1: the pool radius fits kSelHalo, slices are staged in shared memory round by round
  int32_t smem_pairs;       // (key, position) pairs CTA 0 can hold in its dynamic shared memory
  uint2* cand;              // scratch: [batch * H_kv][cand_stride] candidate pairs, one region per CTA rank
  int64_t cand_stride;      // >= cluster * slice
  uint32_t* cand_cnt;       // scratch: [batch * H_kv][kSelMaxCluster] pairs written per region
  uint32_t* status;
  // Optional fused eviction by gather (k_out == nullptr: indices only).  Once a head's list is complete
  // the cluster that produced it copies the listed rows of K and V into the packed cache.
  TensorView k, v;
  void* k_out;
  void* v_out;
  int32_t elem_bytes;       // 4 or 2
  int32_t pieces;           // 16-byte pieces per row = d * elem_bytes / 16
  int32_t log_pieces;       // log2 of that
  int32_t vec;              // score rows start on 16-byte boundaries
  int32_t max_slice;        // positions of the longest slice of the launch
  int32_t raw_floats;       // floats of the staged scores in shared memory (a multiple of 4)
  int32_t inbox;            // keys that a CTA has room for from each CTA of its cluster (a multiple of 4)
  int32_t common_rows;      // lists of more rows than this take one bound for the whole cluster
  int32_t paged;            // kept rows go to page slots of k_out / v_out through pt instead of packed rows
  PageTable pt;
};

// Monotone map float -> uint32 (larger float, larger key).  -0 is folded into +0 first.
__device__ __forceinline__ uint32_t ordered_key(float x) {
  const uint32_t u = __float_as_uint(x + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The mean pool decides a top-k, so its rounding is fixed: float additions from the left-most position of the
// window to the right-most, then one float division by the width.
__device__ __forceinline__ uint32_t pooled_key(const float* s, int i, int P, int radius, int avg) {
  const int lo = max(0, i - radius), hi = min(P - 1, i + radius);
  float best = s[lo];
  if (avg) {
    for (int t = lo + 1; t <= hi; ++t) best = __fadd_rn(best, s[t]);
    best = __fdiv_rn(best, static_cast<float>(2 * radius + 1));
  } else {
    for (int t = lo + 1; t <= hi; ++t) best = fmaxf(best, s[t]);
  }
  return ordered_key(best);
}

// Copies the rows named by one head's finished list into the packed cache: 16 bytes of K and of V per thread
// and piece.  `first` / `stride` spread the pieces over the threads of the cluster.  Kept out of line so that
// its registers are allocated apart from the selection's.  Long lists (large budgets move hundreds of
// megabytes here) take four pieces per step with the index loads, the row loads and the stores issued as
// batches; a one-piece loop would be bound by its latency chain.
__device__ __noinline__ void gather_listed_rows(const int32_t* out, const char* kb, const char* vb, int64_t k_step,
                                                int64_t v_step, uint4* k_dst, uint4* v_dst, int64_t row0, int total,
                                                int pieces, int first, int stride) {
  constexpr int kUnroll = 4;
  int g0 = first;
  {
    for (; g0 + (kUnroll - 1) * stride < total; g0 += kUnroll * stride) {
      int piece[kUnroll], pos[kUnroll];
      int64_t dst[kUnroll];
      uint4 val[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int g = g0 + u * stride;
        const int row = g / pieces;
        piece[u] = g - row * pieces;
        pos[u] = __ldcg(out + row);                           // written by other CTAs of the cluster: skip L1
        dst[u] = (row0 + row) * pieces + piece[u];
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        val[u] = reinterpret_cast<const uint4*>(kb + pos[u] * k_step)[piece[u]];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) k_dst[dst[u]] = val[u];
      if (v_dst) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
          val[u] = reinterpret_cast<const uint4*>(vb + pos[u] * v_step)[piece[u]];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) v_dst[dst[u]] = val[u];
      }
    }
  }
  for (; g0 < total; g0 += stride) {
    const int row = g0 / pieces, piece = g0 - row * pieces;
    const int pos = __ldcg(out + row);
    const int64_t dst = (row0 + row) * pieces + piece;
    k_dst[dst] =
        reinterpret_cast<const uint4*>(kb + pos * k_step)[piece];
    if (v_dst)
      v_dst[dst] =
          reinterpret_cast<const uint4*>(vb + pos * v_step)[piece];
  }
}

// grid (cluster * H_kv, batch), cluster (cluster, 1, 1), block kSelThreads,
// dynamic shared memory (6 bytes per slice position + 8 * kSelHalo) when cached, else none.
// A slice longer than kSelSliceCap is taken in several rounds.
// GROUPS: maxima each thread keeps for the lower bound of step 2 (1 for small budgets, 8 when k nears or
// passes the thread count, so that the bound stays tight).
template <bool AVG, int GROUPS>
__global__ void __launch_bounds__(kSelThreads, 1) pool_select_kernel(const SelectParams p) {
  constexpr int THREADS = kSelThreads, WARPS = kSelWarps;
  constexpr int CAP = kSelSliceCap;                              // positions a CTA holds per round
  constexpr int PER_LANE = kSelPerLane;
  constexpr int BPT = kSelBins / THREADS;                        // histogram bins every thread scans
  extern __shared__ __align__(16) uint32_t sel_smem[];      // [halo | slice | halo] raw scores; later CTA 0's pairs
  __shared__ uint32_t hist[2][kSelBins];                    // per-pass digit histogram (double buffered)
  __shared__ uint32_t warp_sum[WARPS];
  __shared__ uint32_t warp_gt[WARPS], warp_eq[WARPS];
  __shared__ uint32_t sel_digit, sel_above, bound_digit;

  pdl_trigger();
  pdl_wait();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = cluster.dim_blocks().x;
  const int rank = cluster.block_rank();
  const int h = blockIdx.x / C, b = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = (1u << lane) - 1u;

  const int n = p.seq.n[b], alpha = p.seq.alpha, P = n - alpha;
  const int count = p.seq.count[b];
  const int k = count - alpha;                              // prefix rows to keep, 0 <= k <= P
  int32_t* out = p.indices + p.seq.row_off[b] + static_cast<int64_t>(h) * count;
  const bool selecting = k > 0 && k < P;                    // uniform over the cluster

  // The window positions close the list (Section 4.2.1: always retained).
  if (rank == 0)
    for (int j = tid; j < alpha; j += THREADS) out[k + j] = P + j;
  if (k >= P) {                                             // nothing to evict: identity list
    for (int i = rank * THREADS + tid; i < P; i += C * THREADS) out[i] = i;
  }

  const int64_t head = static_cast<int64_t>(b) * p.num_kv_heads + h;
  const int slice = ((P + C - 1) / C + 31) & ~31;           // multiple of 32 positions per CTA
  uint2* regions = p.cand + head * p.cand_stride;           // region of CTA c starts at c * slice
  uint32_t* counts = p.cand_cnt + head * kSelMaxCluster;
  for (int i = tid; i < 2 * kSelBins; i += THREADS) (&hist[0][0])[i] = 0;

  if (selecting) {
    const float* s = p.scores + head * p.ld_scores;
    const int lo = min(P, rank * slice), hi = min(P, lo + slice);
    const int radius = p.pool_radius;
    uint2* region = regions + static_cast<int64_t>(rank) * slice;
    if (p.cached) {                                         // the pool's reach fits the staged halo
      // The slice is taken in rounds of at most CAP positions (one round up to 131072 keys per head
      // with a cluster of 8).  Round: stage raw scores with a halo (outside the prefix: -inf for the max, 0
      // for the mean), pool them into one key per lane and step.
      float* raw = reinterpret_cast<float*>(sel_smem + kSelHalo);
      const float outside = AVG ? 0.0f : -INFINITY;
      const float width = static_cast<float>(2 * radius + 1);
      const int rounds = (hi - lo + CAP - 1) / CAP;
      const int run = ((min(slice, CAP) / WARPS) + 31) & ~31;   // positions per warp and round
      uint32_t pk[PER_LANE];
      int wlo = hi, whi = hi;
      auto pool_round = [&](int r) {
        const int rlo = lo + r * CAP, rhi = min(hi, rlo + CAP);
        __syncthreads();                         // the previous round's readers are done
        for (int i = rlo - kSelHalo + tid; i < rhi + kSelHalo; i += THREADS)
          raw[i - rlo] = (i >= 0 && i < P) ? s[i] : outside;
        __syncthreads();
        wlo = min(rhi, rlo + warp * run);
        whi = min(rhi, wlo + run);
#pragma unroll
        for (int it = 0; it < PER_LANE; ++it) {
          const int i = wlo + it * 32 + lane;
          pk[it] = 0;
          if (i < whi) {
            float best;
            if (AVG) {                                      // left to right; adding the zeros outside changes nothing
              best = raw[i - rlo - radius];
              for (int t = 1 - radius; t <= radius; ++t) best = __fadd_rn(best, raw[i - rlo + t]);
              best = __fdiv_rn(best, width);
            } else {
              best = raw[i - rlo];
              for (int t = 1; t <= radius; ++t) best = fmaxf(best, fmaxf(raw[i - rlo - t], raw[i - rlo + t]));
            }
            pk[it] = ordered_key(best);
          }
        }
      };
      // ---- 1. every thread's largest pooled keys over the whole slice: one per group of its positions
      //         (position step `it` belongs to group it mod GROUPS)
      uint32_t tmax[GROUPS];
#pragma unroll
      for (int g = 0; g < GROUPS; ++g) tmax[g] = 0;
#pragma unroll
      for (int it = 0; it < PER_LANE; ++it) pk[it] = 0;
      for (int r = 0; r < rounds; ++r) {
        pool_round(r);
#pragma unroll
        for (int it = 0; it < PER_LANE; ++it) tmax[it % GROUPS] = max(tmax[it % GROUPS], pk[it]);
      }
      // ---- 2. lower bound of the k-th largest key: the k-th largest of these maxima (maxima of disjoint
      //         groups of positions, so at least k keys are no smaller), resolved to its top 22 bits by two
      //         CTA-local histogram passes
      uint32_t bprefix = 0, bmask = 0, brem = static_cast<uint32_t>(k);
      for (int bp = 0; bp < 2; ++bp) {
        const int shift = bp == 0 ? 21 : 10;
        // maxima that left the searched prefix do not take part in the second pass
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
          const uint32_t digit = ((tmax[g] & bmask) == bprefix) ? ((tmax[g] >> shift) & 2047u) : kSelBins;
          const uint32_t peers = __match_any_sync(0xffffffffu, digit);
          if (digit < kSelBins && lane == __ffs(peers) - 1) atomicAdd(&hist[1][digit], __popc(peers));
        }
        __syncthreads();
        uint32_t bins[BPT];                                 // every thread owns BPT adjacent digits
#pragma unroll
        for (int j = 0; j < BPT; ++j) bins[j] = hist[1][BPT * tid + j];
        uint32_t mine = 0;
#pragma unroll
        for (int j = 0; j < BPT; ++j) mine += bins[j];
        uint32_t incl = mine;
        for (int off = 1; off < 32; off <<= 1) {
          const uint32_t u = __shfl_down_sync(0xffffffffu, incl, off);
          if (lane + off < 32) incl += u;
        }
        if (lane == 0) warp_sum[warp] = incl;
        if (tid == 0) { bound_digit = kSelBins; sel_above = 0; }   // kSelBins: fewer than brem maxima in play
        __syncthreads();
        uint32_t higher = incl - mine;
        for (int w2 = warp + 1; w2 < WARPS; ++w2) higher += warp_sum[w2];
        if (higher < brem && brem <= higher + mine) {
          uint32_t above = higher;                          // from the thread's highest digit down
#pragma unroll
          for (int j = BPT - 1; j >= 0; --j) {
            if (above < brem && brem <= above + bins[j]) { bound_digit = BPT * tid + j; sel_above = above; }
            above += bins[j];
          }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < BPT; ++j) hist[1][BPT * tid + j] = 0;
        const uint32_t bd = bound_digit;
        if (bd == kSelBins) {                               // cannot bound (k exceeds the number of maxima): keep all
          if (bp == 0) { bprefix = 0; bmask = 0; }
          __syncthreads();
          break;
        }
        bprefix |= bd << shift;
        bmask |= 2047u << shift;
        brem -= sel_above;
        __syncthreads();                                    // histogram zeroed, bound_digit consumed
      }
      const uint32_t bound = bprefix;                       // lower edge of the resolved digits
      // ---- 2b. candidates (keys >= bound) of every round, in position order, to this CTA's region
      uint32_t filled = 0;
      for (int r = 0; r < rounds; ++r) {
        pool_round(r);
        uint32_t wc = 0;
#pragma unroll
        for (int it = 0; it < PER_LANE; ++it) {
          const int i = wlo + it * 32 + lane;
          wc += __popc(__ballot_sync(0xffffffffu, i < whi && pk[it] >= bound));
        }
        if (lane == 0) warp_gt[warp] = wc;
        __syncthreads();
        uint32_t base = filled, all_cand = 0;
        for (int w2 = 0; w2 < WARPS; ++w2) {
          if (w2 < warp) base += warp_gt[w2];
          all_cand += warp_gt[w2];
        }
#pragma unroll
        for (int it = 0; it < PER_LANE; ++it) {
          const int i = wlo + it * 32 + lane;
          const bool c = i < whi && pk[it] >= bound;
          const uint32_t bal = __ballot_sync(0xffffffffu, c);
          if (c) region[base + __popc(bal & lt)] = make_uint2(pk[it], static_cast<uint32_t>(i));
          base += __popc(bal);
        }
        filled += all_cand;
      }
      if (tid == 0) counts[rank] = filled;
    } else {
      // a very wide pool: every position is a candidate
      for (int i = lo + tid; i < hi; i += THREADS) region[i - lo] = make_uint2(pooled_key(s, i, P, radius, AVG ? 1 : 0), i);
      if (tid == 0) counts[rank] = hi - lo;
    }
  }
  if (C == 1) __syncthreads(); else cluster.sync();         // every region and its count are written

  if (selecting && rank == 0) {
    // ---- 3. CTA 0: concatenate the regions, radix search, emit
    uint32_t pre[kSelMaxCluster + 1];
    pre[0] = 0;
#pragma unroll
    for (int c = 0; c < kSelMaxCluster; ++c) pre[c + 1] = pre[c] + (c < C ? __ldcg(counts + c) : 0u);
    const int N = static_cast<int>(pre[kSelMaxCluster]);
    auto fetch = [&](int j) -> uint2 {                      // pair j of the concatenation, from global memory
      int c = 0;
#pragma unroll
      for (int q = 1; q < kSelMaxCluster; ++q) c += static_cast<uint32_t>(j) >= pre[q] ? 1 : 0;
      return __ldcg(regions + static_cast<int64_t>(c) * slice + (j - static_cast<int>(pre[c])));
    };
    uint2* flat = reinterpret_cast<uint2*>(sel_smem);
    const int held = min(N, p.smem_pairs);
    for (int j = tid; j < held; j += THREADS) flat[j] = fetch(j);
    __syncthreads();
    auto item = [&](int j) -> uint2 { return j < held ? flat[j] : fetch(j); };

    uint32_t prefix = 0, mask = 0, remaining = k;
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
      const uint32_t dmask = pass == 2 ? 1023u : 2047u;
      uint32_t* hcur = hist[pass & 1];
      for (int j0 = warp * 32; j0 < N; j0 += THREADS) {
        const int j = j0 + lane;
        uint32_t digit = kSelBins;                          // kSelBins = does not take part
        if (j < N) {
          const uint32_t key = item(j).x;
          if ((key & mask) == prefix) digit = (key >> shift) & dmask;
        }
        const uint32_t peers = __match_any_sync(0xffffffffu, digit);
        if (digit < kSelBins && lane == __ffs(peers) - 1) atomicAdd(&hcur[digit], __popc(peers));
      }
      __syncthreads();
      uint32_t bins[BPT];                                   // every thread owns BPT adjacent digits
      uint32_t mine = 0;
#pragma unroll
      for (int j = 0; j < BPT; ++j) {
        bins[j] = hcur[BPT * tid + j];
        hist[(pass + 1) & 1][BPT * tid + j] = 0;            // next pass's buffer
        mine += bins[j];
      }
      uint32_t incl = mine;                                 // keys in this and the higher threads of the warp
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t u = __shfl_down_sync(0xffffffffu, incl, off);
        if (lane + off < 32) incl += u;
      }
      if (lane == 0) warp_sum[warp] = incl;
      __syncthreads();
      uint32_t higher = incl - mine;
      for (int w2 = warp + 1; w2 < WARPS; ++w2) higher += warp_sum[w2];
      if (higher < remaining && remaining <= higher + mine) {  // exactly one thread: the k-th key is in its digits
        uint32_t above = higher;                            // from the thread's highest digit down
#pragma unroll
        for (int j = BPT - 1; j >= 0; --j) {
          if (above < remaining && remaining <= above + bins[j]) { sel_digit = BPT * tid + j; sel_above = above; }
          above += bins[j];
        }
      }
      __syncthreads();
      prefix |= sel_digit << shift;
      mask |= dmask << shift;
      remaining -= sel_above;
      __syncthreads();                                      // sel_* are rewritten next pass
    }
    const uint32_t T = prefix;                              // the k-th largest key
    const uint32_t need_eq = remaining;                     // ties at T to take, from the left

    // keys above / at the threshold, warp by warp over contiguous chunks of the concatenation
    const int chunk = (((N + WARPS - 1) / WARPS) + 31) & ~31;
    const int j_lo = min(N, warp * chunk), j_hi = min(N, j_lo + chunk);
    uint32_t ngt = 0, neq = 0;
    for (int j0 = j_lo; j0 < j_hi; j0 += 32) {
      const int j = j0 + lane;
      const uint32_t key = j < j_hi ? item(j).x : 0u;
      ngt += __popc(__ballot_sync(0xffffffffu, j < j_hi && key > T));
      neq += __popc(__ballot_sync(0xffffffffu, j < j_hi && key == T));
    }
    if (lane == 0) { warp_gt[warp] = ngt; warp_eq[warp] = neq; }
    __syncthreads();
    uint32_t gt_before = 0, eq_before = 0;
    for (int w2 = 0; w2 < warp; ++w2) { gt_before += warp_gt[w2]; eq_before += warp_eq[w2]; }
    if (tid == THREADS - 1) {                           // the last thread can see the grand total
      if (gt_before + ngt + min(eq_before + neq, need_eq) != static_cast<uint32_t>(k))
        atomicOr(p.status, kStatusSelectMismatch);
    }
    // rank of a kept position = (#greater before it) + min(#equal before it, need_eq)
    for (int j0 = j_lo; j0 < j_hi; j0 += 32) {
      const int j = j0 + lane;
      const uint2 kv = j < j_hi ? item(j) : make_uint2(0u, 0u);
      const bool is_gt = j < j_hi && kv.x > T, is_eq = j < j_hi && kv.x == T;
      const uint32_t bg = __ballot_sync(0xffffffffu, is_gt), be = __ballot_sync(0xffffffffu, is_eq);
      const uint32_t g = gt_before + __popc(bg & lt), e = eq_before + __popc(be & lt);
      if (is_gt || (is_eq && e < need_eq)) out[g + min(e, need_eq)] = static_cast<int32_t>(kv.y);
      gt_before += __popc(bg);
      eq_before += __popc(be);
    }
  }
  if (C == 1) __syncthreads(); else cluster.sync();         // the list is complete

  // ---- 5. eviction by gather (appendix on torch.gather), spread over the cluster
  if (p.k_out != nullptr) {
    const char* kb = static_cast<const char*>(p.k.ptr) + (b * p.k.sb + h * p.k.sh) * p.elem_bytes;
    const char* vb = static_cast<const char*>(p.v.ptr) + (b * p.v.sb + h * p.v.sh) * p.elem_bytes;
    const int64_t row0 = p.seq.row_off[b] + static_cast<int64_t>(h) * count;
    const int total = count * p.pieces, stride = C * THREADS;
    if (total >= 8 * stride) {                              // a long list: the batched copy
      gather_listed_rows(out, kb, vb, p.k.st * p.elem_bytes, p.v.st * p.elem_bytes, static_cast<uint4*>(p.k_out),
                         static_cast<uint4*>(p.v_out), row0, total, p.pieces, rank * THREADS + tid, stride);
    } else {
      for (int g = rank * THREADS + tid; g < total; g += stride) {
        const int row = g / p.pieces, piece = g - row * p.pieces;
        const int pos = __ldcg(out + row);                  // written by other CTAs of the cluster: skip L1
        const int64_t dst = (row0 + row) * p.pieces + piece;
        static_cast<uint4*>(p.k_out)[dst] =
            reinterpret_cast<const uint4*>(kb + static_cast<int64_t>(pos) * p.k.st * p.elem_bytes)[piece];
        if (p.v_out)
          static_cast<uint4*>(p.v_out)[dst] =
              reinterpret_cast<const uint4*>(vb + static_cast<int64_t>(pos) * p.v.st * p.elem_bytes)[piece];
      }
    }
  }
}

// ------------------------------------------------------------------ rows of at most kSelMaxCluster * 16384 positions
//
// The kernel is a chain of short phases, bound by their latencies (loads, block and cluster barriers), not by a unit.
// What shortens the chain:
//   * a thread takes runs of eight consecutive positions, so pooling is a handful of 16-byte shared-memory reads (the
//     staged scores are padded by 16 bytes per 128 so that these do not conflict) and position order is thread order;
//   * the lower bound of the k-th key comes from one histogram pass over the runs' maxima on an absolute scale.  A run
//     counts with the number of its positions that hold its maximum (pooled scores come in plateaus), so that the bound
//     lets through about k positions.  Short lists take a bound per CTA (about k candidates each); for long ones the
//     CTAs' histograms are added up first, one cluster barrier more, and about k candidates are left in all;
//   * every CTA of the cluster finishes on its own: it is sent the candidates of all (distributed shared memory), finds
//     the threshold, and emits and copies the rows of its own slice.  There is one full cluster barrier (up to three
//     when the list is long) and no trip through global memory;
//   * the exact threshold is searched inside [largest bound of the CTAs, largest key], ten bits a pass, and finished by
//     a warp as soon as at most 32 candidates are left in the bin (mostly after the first pass).
constexpr int kSelBinsLin = 1024;          // bins of a linear histogram: ten bits of the key range
constexpr int kSelRun = 8;                 // consecutive positions of a thread
constexpr int kSelClusterSlice = 8192;     // a cluster doubles (up to 8 CTAs) while its slices are longer than this
constexpr int kSelCopyBytes = 128 << 10;   // ... or while a CTA would copy more than this and SMs are idle
constexpr int kSelCommonCandidates = 4096; // more expected candidates (k per CTA) than this: one bound for the cluster
constexpr int kSelCrowd = 1024;            // candidates of a CTA beyond 2 k that its bound may let through before it is refined
constexpr int kSelEvenRows = 1024;         // lists of at least this many rows are copied by the whole cluster evenly

// Position i of the staged scores in shared memory: four floats of padding after every 32.
__device__ __forceinline__ int sel_pad(int i) { return i + ((i >> 5) << 2); }

// The largest bin d with (sum of bins >= d) >= want, and what lies above it; false when all bins together hold less.
// Called by the whole block after a barrier behind the last update; `rows` is scratch (32 words); one barrier inside.
template <int THREADS>
__device__ __forceinline__ bool sel_find_from_top(const uint32_t* hist, uint32_t* rows, uint32_t want, uint32_t& digit,
                                                  uint32_t& above) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kRowsPerWarp = kSelBinsLin / THREADS;       // a row: 32 bins
#pragma unroll
  for (int r = 0; r < kRowsPerWarp; ++r) {
    const int row = warp + r * (THREADS / 32);
    const uint32_t sum = __reduce_add_sync(0xffffffffu, hist[row * 32 + lane]);
    if (lane == 0) rows[row] = sum;
  }
  __syncthreads();
  // suffix sums over the 32 rows, then over the bins of the row the searched one lies in
  auto suffix = [&](uint32_t x) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t u = __shfl_down_sync(0xffffffffu, x, off);
      if (lane + off < 32) x += u;
    }
    return x;
  };
  const uint32_t rs = suffix(rows[lane]);
  const uint32_t rmask = __ballot_sync(0xffffffffu, rs >= want);
  if (rmask == 0) return false;
  const int row = 31 - __clz(rmask);
  const uint32_t past = row == 31 ? 0u : __shfl_sync(0xffffffffu, rs, row + 1);
  const uint32_t bin = hist[row * 32 + lane];
  const uint32_t bs = suffix(bin) + past;
  const int b = 31 - __clz(__ballot_sync(0xffffffffu, bs >= want));
  digit = static_cast<uint32_t>(row * 32 + b);
  above = __shfl_sync(0xffffffffu, bs - bin, b);
  return true;
}

// Bin of a key for the candidate bound: an absolute scale (the same in every CTA of a cluster), 32 bins an octave over the
// 32 octaves below 2^6 (scores lie between 0 and alpha); what lies below or above goes to the first and last bin.
constexpr uint32_t kSelBinBase = 0x80000000u | ((127u + 6u - 32u) << 23);      // key of 2^-26
__device__ __forceinline__ uint32_t sel_bin(uint32_t key) {
  return key < kSelBinBase ? 0u : min((key - kSelBinBase) >> 18, static_cast<uint32_t>(kSelBinsLin - 1));
}
__device__ __forceinline__ uint32_t sel_bin_edge(uint32_t bin) { return bin == 0 ? 0u : kSelBinBase + (bin << 18); }

// Pooled keys of eight consecutive positions; x[4 + j] is position j of the run.
template <int R, bool AVG>
__device__ __forceinline__ void sel_pool8(const float (&x)[16], uint32_t (&key)[kSelRun]) {
#pragma unroll
  for (int j = 0; j < kSelRun; ++j) {
    float best = x[4 + j - R];
#pragma unroll
    for (int t = 1 - R; t <= R; ++t) best = AVG ? __fadd_rn(best, x[4 + j + t]) : fmaxf(best, x[4 + j + t]);
    if (AVG) best = __fdiv_rn(best, static_cast<float>(2 * R + 1));
    key[j] = ordered_key(best);
  }
}

template <bool AVG>
__device__ __forceinline__ void sel_pool_run(const float* raw, int at, int radius, uint32_t (&key)[kSelRun]) {
  if (radius <= 4) {
    float x[16];                                             // positions at - 4 .. at + 11
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float4 f = *reinterpret_cast<const float4*>(raw + sel_pad(at - 4 + 4 * c));
      x[4 * c] = f.x; x[4 * c + 1] = f.y; x[4 * c + 2] = f.z; x[4 * c + 3] = f.w;
    }
    switch (radius) {
      case 0: sel_pool8<0, AVG>(x, key); break;
      case 1: sel_pool8<1, AVG>(x, key); break;
      case 2: sel_pool8<2, AVG>(x, key); break;
      case 3: sel_pool8<3, AVG>(x, key); break;
      default: sel_pool8<4, AVG>(x, key); break;
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < kSelRun; ++j) {
    float best = raw[sel_pad(at + j - radius)];
    for (int t = 1 - radius; t <= radius; ++t) {
      const float v = raw[sel_pad(at + j + t)];
      best = AVG ? __fadd_rn(best, v) : fmaxf(best, v);
    }
    if (AVG) best = __fdiv_rn(best, static_cast<float>(2 * radius + 1));
    key[j] = ordered_key(best);
  }
}

// Candidates beyond all use: the scale of sel_bin has 32 bins an octave between 2^-26 and 2^6, so a flat row (its keys share a
// few bins) or scores on another scale (which share the first or last one) can have every position above the bound.  Every
// candidate is sent to and ranked by all CTAs of the cluster, some 2 us per 1000 of them.  Here the range from the smallest
// to the largest candidate is divided, ten bits at a time, until the bound lets through little more than k, and the list
// is closed up.  131040 positions, k = 96: flat rows 93 -> 20 us, scores near 1e-12 147 -> 22 us
// (rows spread over the scale: 12).
// Called by the whole block (common: by the whole cluster) behind a barrier; ends with one.  Out of line: the registers of
// the ordinary way are not to be shared with it.  minima: scratch, a word per warp; maxima: the warps' largest keys.
// Returns the number of candidates left and the new bound.
template <int THREADS, int RUNS>
__device__ __noinline__ uint2 sel_refine(uint32_t* list_key, uint16_t* list_pos, int M, uint32_t k, uint32_t* hist, uint32_t* rows,
                                         uint32_t* minima, uint32_t* maxima, bool common) {
  constexpr int WARPS = THREADS / 32, E = RUNS * kSelRun;
  cg::cluster_group cluster = cg::this_cluster();
  const int C = cluster.dim_blocks().x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t full = 0xffffffffu, lt = (1u << lane) - 1u;
  // a warp takes consecutive entries, 32 * per of them; entry j * 32 + lane of these is this lane's j-th
  const int per = (M + THREADS - 1) / THREADS, first = warp * per * 32 + lane;
  auto mine = [&](int j) { return j < per && first + j * 32 < M; };
  uint32_t key[E], least = 0xffffffffu;
#pragma unroll
  for (int j = 0; j < E; ++j) {
    key[j] = mine(j) ? list_key[first + j * 32] : 0u;
    if (mine(j)) least = min(least, key[j]);
  }
  least = __reduce_min_sync(full, least);
  if (lane == 0) minima[warp] = least;
  if (common) cluster.sync(); else __syncthreads();         // (and everybody has read the counts before)
  uint32_t bound = 0xffffffffu, top = 0;                    // the smallest and the largest candidate
  for (int c = 0; c < (common ? C : 1); ++c)
    if (lane < WARPS) {
      bound = min(bound, common ? cluster.map_shared_rank(minima, c)[lane] : minima[lane]);
      top = max(top, common ? cluster.map_shared_rank(maxima, c)[lane] : maxima[lane]);
    }
  bound = __reduce_min_sync(full, bound);
  top = __reduce_max_sync(full, top);
  uint32_t span = 0xffffffffu, want = k;
  int shift = max(0, 22 - __clz(top - bound));
  uint32_t* counts = hist + (common ? kSelBinsLin : 0);
  for (;;) {
    for (int i = tid; i < 2 * kSelBinsLin; i += THREADS) hist[i] = 0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < E; ++j)
      if (mine(j) && key[j] >= bound && key[j] - bound <= span) atomicAdd(&hist[(key[j] - bound) >> shift], 1u);
    if (common) {
      cluster.sync();
      for (int i = tid; i < kSelBinsLin; i += THREADS) {
        uint32_t sum = 0;
        for (int c = 0; c < C; ++c) sum += cluster.map_shared_rank(hist, c)[i];
        counts[i] = sum;
      }
    }
    __syncthreads();
    uint32_t digit = 0, above = 0;
    sel_find_from_top<THREADS>(counts, rows, want, digit, above);
    bound += digit << shift;
    want -= above;
    if (shift == 0 || k - want + counts[digit] <= k + k / 4 + 128) break;
    span = (1u << shift) - 1u;
    shift = max(0, shift - 10);
    if (common) cluster.sync(); else __syncthreads();       // everybody has read the counts
  }
  uint32_t left = 0;
#pragma unroll
  for (int j = 0; j < E; ++j) left += __popc(__ballot_sync(full, mine(j) && key[j] >= bound));
  uint32_t pos[E / 2];                                      // (read before anybody writes)
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const uint32_t x = mine(j) ? list_pos[first + j * 32] : 0u;
    pos[j / 2] = j & 1 ? pos[j / 2] | x << 16 : x;
  }
  if (common) cluster.sync(); else __syncthreads();         // the others have read this CTA's minima
  if (lane == 0) minima[warp] = left;
  __syncthreads();
  const uint32_t sum = lane < WARPS ? minima[lane] : 0u;
  uint32_t to = __reduce_add_sync(full, lane < warp ? sum : 0u);
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const bool stays = mine(j) && key[j] >= bound;
    const uint32_t all = __ballot_sync(full, stays);
    if (stays) {
      list_key[to + __popc(all & lt)] = key[j];
      list_pos[to + __popc(all & lt)] = static_cast<uint16_t>(pos[j / 2] >> (16 * (j & 1)));
    }
    to += __popc(all);
  }
  __syncthreads();
  return make_uint2(__reduce_add_sync(full, sum), bound);
}

// Dynamic shared memory of an instance for slices of `slice` positions (a multiple of 32).
__host__ __device__ constexpr size_t sel_smem_floats(int slice) { return static_cast<size_t>(slice + 2 * kSelHalo) * 9 / 8 + 4; }
constexpr size_t kSelSmemMax = 208 * 1024;
// Staged scores, the CTA's candidates (4-byte keys, 2-byte offsets in the slice), keys from the cluster.
__host__ __device__ constexpr size_t sel_smem_bytes(int slice, int cluster, int inbox) {
  return (sel_smem_floats(slice) + static_cast<size_t>(slice) + static_cast<size_t>(slice) / 2 + static_cast<size_t>(cluster) * inbox) * 4;
}

// grid (cluster * H_kv, batch), cluster (cluster, 1, 1), block THREADS, dynamic shared memory sel_smem_bytes.
// RUNS runs of eight positions per thread: a CTA takes at most THREADS * RUNS * 8 positions.
template <int THREADS, int RUNS, bool AVG>
__global__ void __launch_bounds__(THREADS, THREADS == 1024 ? 1 : 2) select_kernel(const SelectParams p) {
  constexpr int WARPS = THREADS / 32;
  constexpr bool kLong = THREADS > 256;                     // long slices: see the threshold search
  extern __shared__ __align__(16) uint8_t sel_dyn[];
  __shared__ __align__(16) uint32_t hist[2][kSelBinsLin];                 // [0]: read by the whole cluster when the bound is a common one
  __shared__ __align__(16) uint32_t local[2][kSelBinsLin];  // threshold search
  __shared__ uint32_t rows[32];
  __shared__ uint32_t warp_a[WARPS], warp_b[WARPS], warp_c[WARPS], warp_d[WARPS];
  __shared__ __align__(16) uint32_t few[32];
  __shared__ uint32_t few_n;
  __shared__ uint2 found;                                   // threshold, ties at it that are taken
  __shared__ uint4 pub[kSelMaxCluster];                     // every CTA's number of candidates, bound, largest key

  pdl_trigger();
  cg::cluster_group cluster = cg::this_cluster();
  const int C = cluster.dim_blocks().x, rank = cluster.block_rank();
  const int h = blockIdx.x / C, b = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t full = 0xffffffffu, lt = (1u << lane) - 1u;

  const int n = p.seq.n[b], alpha = p.seq.alpha, P = n - alpha;
  const int count = p.seq.count[b], k = count - alpha;      // prefix rows to keep, 0 <= k <= P
  const bool selecting = k > 0 && k < P;                    // uniform over the cluster
  const int slice = ((P + C - 1) / C + 31) & ~31;           // positions of a CTA, a multiple of 32
  const int lo = min(P, rank * slice), len = min(P, lo + slice) - lo;
  const int64_t head = static_cast<int64_t>(b) * p.num_kv_heads + h;
  const int64_t row0 = p.seq.row_off[b] + static_cast<int64_t>(h) * count;
  int32_t* out = p.indices + row0;
  float* raw = reinterpret_cast<float*>(sel_dyn);           // staged scores; later the positions this CTA keeps
  uint32_t* list_key = reinterpret_cast<uint32_t*>(raw + p.raw_floats);                 // own candidates in position order
  uint16_t* list_pos = reinterpret_cast<uint16_t*>(list_key + p.max_slice);                // ... offsets in the slice
  uint32_t* inbox = list_key + p.max_slice + p.max_slice / 2;                           // [C][p.inbox] everybody's keys
  if (C > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");              // this CTA's inbox may be written

  // (hist[1] is written before it is read.)  Short slices do without the zeros in few[], and clear by words: 0.1 to 0.3 us of a layer
  // call of 512 to 1800 positions.
  if constexpr (kLong) {
    for (int i = tid; i < kSelBinsLin / 4; i += THREADS) {
      reinterpret_cast<uint4*>(hist[0])[i] = make_uint4(0, 0, 0, 0);
      reinterpret_cast<uint4*>(local[0])[i] = make_uint4(0, 0, 0, 0);
    }
    if (tid < 32) few[tid] = 0;
  } else {
    for (int i = tid; i < kSelBinsLin; i += THREADS) hist[0][i] = local[0][i] = 0;
  }
  if (tid == 0) few_n = 0;
  pdl_wait();

  // the rows this CTA copies: entries [own0, own1) of the head's list, positions in kept[]; the window closes the list
  int own0 = 0, own1 = 0;
  int32_t* kept = reinterpret_cast<int32_t*>(raw);
  if (selecting) {
    // ---- stage the slice with a halo (outside the prefix: what the pool ignores)
    {
      const float* s = p.scores + head * p.ld_scores;
      const float outside = AVG ? 0.0f : -INFINITY;
      constexpr int V = RUNS * 2 + 1;                       // 16-byte pieces per thread, halo included
      const int pieces = (len + 2 * kSelHalo + 3) / 4;
      float4 f[V];
#pragma unroll
      for (int j = 0; j < V; ++j) {
        const int v = tid + j * THREADS, i = lo - kSelHalo + 4 * v;
        if (v < pieces) {
          if (p.vec && i >= 0 && i + 3 < P) {
            f[j] = __ldcg(reinterpret_cast<const float4*>(s + i));
          } else {
            f[j].x = i >= 0 && i < P ? s[i] : outside;
            f[j].y = i + 1 >= 0 && i + 1 < P ? s[i + 1] : outside;
            f[j].z = i + 2 >= 0 && i + 2 < P ? s[i + 2] : outside;
            f[j].w = i + 3 >= 0 && i + 3 < P ? s[i + 3] : outside;
          }
        }
      }
#pragma unroll
      for (int j = 0; j < V; ++j) {
        const int v = tid + j * THREADS;
        if (v < pieces) *reinterpret_cast<float4*>(raw + sel_pad(4 * v)) = f[j];
      }
    }
    __syncthreads();

    // ---- pool, and each run's largest key with the number of its positions that hold it
    uint32_t key[RUNS][kSelRun], tmax[RUNS], weight[RUNS];
    uint32_t mx = 0;
#pragma unroll
    for (int r = 0; r < RUNS; ++r) {
      const int at = (r * THREADS + tid) * kSelRun;
      tmax[r] = 0;
      weight[r] = 0;
      if (at < len) {
        sel_pool_run<AVG>(raw, kSelHalo + at, p.pool_radius, key[r]);
#pragma unroll
        for (int j = 0; j < kSelRun; ++j)
          if (at + j < len) tmax[r] = max(tmax[r], key[r][j]);
#pragma unroll
        for (int j = 0; j < kSelRun; ++j)
          if (at + j < len && key[r][j] == tmax[r]) ++weight[r];
        mx = max(mx, tmax[r]);
        atomicAdd(&hist[0][sel_bin(tmax[r])], weight[r]);
      }
    }
    mx = __reduce_max_sync(full, mx);
    if (lane == 0) warp_a[warp] = mx;

    // ---- lower bound of the k-th key, candidates in position order
    const bool common = C > 1 && k > p.common_rows;         // uniform over the cluster
    if (C > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");              // every CTA has started
    if (common) {
      cluster.sync();
      for (int i = tid; i < kSelBinsLin; i += THREADS) {
        uint32_t sum = 0;
#pragma unroll
        for (int c = 0; c < kSelMaxCluster; ++c) sum += c < C ? cluster.map_shared_rank(&hist[0][0], c)[i] : 0u;
        hist[1][i] = sum;
      }
    }
    __syncthreads();
    uint32_t bound = 0;
    bool crowded = false;                                   // common bound: many more candidates than wanted (the runs stand for
    {                                                       // them; without one the CTA counts them below)
      uint32_t digit, above;
      if (sel_find_from_top<THREADS>(hist[common ? 1 : 0], rows, static_cast<uint32_t>(k), digit, above)) {
        bound = sel_bin_edge(digit);
        crowded = common && above + hist[1][digit] > 2u * k + kSelCrowd / 2 * C;
      } else if (common || k < len) {                       // the plateaus do not add up to k: count every position
        if (common) cluster.sync(); else __syncthreads();   // everybody has read the first counts
        for (int i = tid; i < 2 * kSelBinsLin; i += THREADS) (&hist[0][0])[i] = 0;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < RUNS; ++r) {
          const int at = (r * THREADS + tid) * kSelRun;
#pragma unroll
          for (int j = 0; j < kSelRun; ++j)
            if (at + j < len) atomicAdd(&hist[0][sel_bin(key[r][j])], 1u);
        }
        if (common) {
          cluster.sync();
          for (int i = tid; i < kSelBinsLin; i += THREADS) {
            uint32_t sum = 0;
#pragma unroll
            for (int c = 0; c < kSelMaxCluster; ++c) sum += c < C ? cluster.map_shared_rank(&hist[0][0], c)[i] : 0u;
            hist[1][i] = sum;
          }
        }
        __syncthreads();
        if (sel_find_from_top<THREADS>(hist[common ? 1 : 0], rows, static_cast<uint32_t>(k), digit, above)) bound = sel_bin_edge(digit);
      }
    }
    uint32_t c2 = 0;                                        // candidates of the runs, 16 bits each
#pragma unroll
    for (int r = 0; r < RUNS; ++r) {
      const int at = (r * THREADS + tid) * kSelRun;
#pragma unroll
      for (int j = 0; j < kSelRun; ++j)
        if (at + j < len && key[r][j] >= bound) c2 += 1u << (16 * r);
    }
    uint32_t incl = c2;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t u = __shfl_up_sync(full, incl, off);
      if (lane >= off) incl += u;
    }
    if (lane == 31) warp_c[warp] = incl;
    __syncthreads();
    uint32_t wsum = lane < WARPS ? warp_c[lane] : 0u;
    const uint32_t before = __reduce_add_sync(full, lane < warp ? wsum : 0u), all = __reduce_add_sync(full, wsum);
    int M = static_cast<int>((all & 0xffffu) + (all >> 16));
    {
      const uint32_t base2 = before + incl - c2;
#pragma unroll
      for (int r = 0; r < RUNS; ++r) {
        const int at = (r * THREADS + tid) * kSelRun;
        uint32_t to = r == 0 ? (base2 & 0xffffu) : (all & 0xffffu) + (base2 >> 16);
        if ((c2 >> (16 * r)) & 0xffffu) {
#pragma unroll
          for (int j = 0; j < kSelRun; ++j)
            if (at + j < len && key[r][j] >= bound) {
              list_key[to] = key[r][j];
              list_pos[to++] = static_cast<uint16_t>(at + j);
            }
        }
      }
    }
    mx = __reduce_max_sync(full, warp_a[lane & (WARPS - 1)]);
    __syncthreads();
    if constexpr (THREADS * RUNS > 512) {                   // (up to 4096 candidates of one CTA are ranked in 10 us all the same)
      if (!common) crowded = k < len && M > 2 * k + kSelCrowd;
      if (crowded) {
        const uint2 refined = sel_refine<THREADS, RUNS>(list_key, list_pos, M, k, &hist[0][0], rows, warp_c, warp_a, common);
        M = static_cast<int>(refined.x);
        bound = refined.y;
      }
    }
    // every CTA gets everybody's keys: stores into the others' shared memory, which nobody waits for until the barrier
    // (reading them there after it cost 2 to 3 us)
    if (tid < C) {
      const uint4 mine = make_uint4(static_cast<uint32_t>(M), bound, mx, 0u);
      if (C == 1) pub[0] = mine; else cluster.map_shared_rank(&pub[0], tid)[rank] = mine;
    }
    if (C > 1)
      for (int i = tid; i < min(M, p.inbox); i += THREADS) {
        const uint32_t x = list_key[i];
        for (int c = 0; c < C; ++c)
          if (c != rank) cluster.map_shared_rank(inbox, c)[rank * p.inbox + i] = x;
      }
    if (C == 1) __syncthreads(); else cluster.sync();       // candidates of the whole cluster are in place

    // ---- the threshold T (k-th largest key) and how many ties at T are taken
    uint32_t base = 0, top = 0;                             // at least k keys of some CTA, so of all, reach its bound
#pragma unroll
    for (int c = 0; c < kSelMaxCluster; ++c)
      if (c < C) {
        const uint4 o = pub[c];
        base = max(base, o.y);
        top = max(top, o.z);
      }
    // Key i of CTA c; a CTA whose candidates did not fit its place in the inbox is asked for the rest.  The warps are
    // dealt round to the CTAs: warp w takes CTA w % C, 32 keys at a time.
    auto key_at = [&](int c, int i) -> uint32_t {
      if (c == rank) return list_key[i];
      return i < p.inbox ? inbox[c * p.inbox + i] : cluster.map_shared_rank(list_key, c)[i];
    };
    const int my_c = warp & (C - 1), my_first = (warp / C) * 32 + lane, my_step = (WARPS / C) * 32;
    const int my_n = static_cast<int>(pub[my_c].x);
    // Most candidates lie within an octave of the bound and a few far above it: the first pass divides the lowest eighth of
    // the range, what lies above counts in its last bin.  (Over the whole range a bin held some 50 of 3600 candidates, and
    // a second pass followed.)
    // In short slices the whole range is divided and every warp ranks the last ones for itself, two barriers less (1146 to 1989
    // positions: layer calls of 20.5 to 24.2 us take 0.7 to 0.9 more the other way).
    uint32_t want = static_cast<uint32_t>(k), T = 0, need_eq = 0;
    int shift = max(0, 22 - (kLong ? 3 : 0) - __clz(top - base));
    uint32_t span = 0xffffffffu;                            // keys base .. base + span take part
    for (int pass = 0;; ++pass) {
      uint32_t* hc = local[pass & 1];
      for (int i = my_first; i < my_n; i += my_step) {
        const uint32_t x = key_at(my_c, i);
        if (x >= base && x - base <= span) atomicAdd(&hc[kLong ? min((x - base) >> shift, kSelBinsLin - 1u) : (x - base) >> shift], 1u);
      }
      __syncthreads();
      uint32_t digit = 0, above = 0;
      sel_find_from_top<THREADS>(hc, rows, want, digit, above);
      const bool beyond = kLong && digit == kSelBinsLin - 1u && min(span, top - base) >> shift > digit;      // in what was put together
      want -= above;
      base += digit << shift;
      const uint32_t in_bin = hc[digit];
      // All but a few of the rows to copy are known: in short slices they go into the L2 ahead of the copy.  Not in the other
      // instances, where the prefetches cost more than they save, the search's own accesses queueing behind them: 4096 keys 28.8 us,
      // 28.1 without; 32768 keys 51.6, 50.9; three steps of 2 x 10000 keys 32.9, 32.2.
      if constexpr (!kLong) {
        if (pass == 0 && p.k_out != nullptr) {
          const int64_t ks = p.k.st * p.elem_bytes, vs = p.v.st * p.elem_bytes;
          const char* kb = static_cast<const char*>(p.k.ptr) + (b * p.k.sb + h * p.k.sh + static_cast<int64_t>(lo) * p.k.st) * p.elem_bytes;
          const char* vb = static_cast<const char*>(p.v.ptr) + (b * p.v.sb + h * p.v.sh + static_cast<int64_t>(lo) * p.v.st) * p.elem_bytes;
          for (int i = tid; i < M; i += THREADS)
            if (list_key[i] >= base)
              for (int c = 0; c < p.pieces * 16; c += 128) {
                asm volatile("prefetch.global.L2 [%0];" ::"l"(kb + list_pos[i] * ks + c));
                asm volatile("prefetch.global.L2 [%0];" ::"l"(vb + list_pos[i] * vs + c));
              }
        }
      }
      if (shift == 0 && !beyond) {
        T = base;
        need_eq = want;
        break;
      }
      if (in_bin <= 32u) {                                  // few enough for a warp: rank them by counting
        const uint32_t width = beyond ? 0xffffffffu : (1u << shift) - 1u;
        for (int i = my_first; i < my_n; i += my_step) {
          const uint32_t x = key_at(my_c, i);
          if (x >= base && x - base <= width) few[atomicAdd(&few_n, 1u)] = x;
        }
        __syncthreads();
        if constexpr (!kLong) {
          const uint32_t x = lane < static_cast<int>(in_bin) ? few[lane] : 0u;
          uint32_t gt = 0, ge = 0;
          for (int q = 0; q < static_cast<int>(in_bin); ++q) {
            const uint32_t o = __shfl_sync(full, x, q);
            gt += o > x ? 1u : 0u;
            ge += o >= x ? 1u : 0u;
          }
          const uint32_t hit = __ballot_sync(full, lane < static_cast<int>(in_bin) && gt < want && want <= ge);
          T = __shfl_sync(full, x, __ffs(hit) - 1);
          need_eq = want - __shfl_sync(full, gt, __ffs(hit) - 1);
          break;
        }
        if (warp == 0) {                                    // (all for themselves with shuffles: 0.5 us more at 1024 threads)
          const uint32_t x = few[lane];                     // (zeros behind the last one)
          uint32_t gt = 0, ge = 0;
#pragma unroll
          for (int q = 0; q < 32; q += 4) {
            const uint4 o = *reinterpret_cast<const uint4*>(few + q);
            gt += (o.x > x ? 1u : 0u) + (o.y > x ? 1u : 0u) + (o.z > x ? 1u : 0u) + (o.w > x ? 1u : 0u);
            ge += (o.x >= x ? 1u : 0u) + (o.y >= x ? 1u : 0u) + (o.z >= x ? 1u : 0u) + (o.w >= x ? 1u : 0u);
          }
          const uint32_t hit = __ballot_sync(full, lane < static_cast<int>(in_bin) && gt < want && want <= ge);
          if (lane == __ffs(hit) - 1) found = make_uint2(x, want - gt);
        }
        __syncthreads();
        T = found.x;
        need_eq = found.y;
        break;
      }
      span = beyond ? 0xffffffffu : (1u << shift) - 1u;
      shift = beyond ? max(0, 22 - __clz(top - base)) : max(0, shift - 10);
      for (int i = tid; i < kSelBinsLin; i += THREADS) local[(pass + 1) & 1][i] = 0;
      __syncthreads();
    }

    // ---- emit: kept = keys above T and the leftmost need_eq of those at T.  Counted over the candidates of the CTAs
    //      before this one (where its part of the list starts) and over its own, warp by warp in contiguous chunks
    uint32_t pgt = 0, peq = 0;
    if (my_c < rank)
      for (int i = my_first; i < my_n; i += my_step) {
        const uint32_t x = key_at(my_c, i);
        pgt += x > T ? 1u : 0u;
        peq += x == T ? 1u : 0u;
      }
    pgt = __reduce_add_sync(full, pgt);
    peq = __reduce_add_sync(full, peq);
    const int chunk = (((M + WARPS - 1) / WARPS) + 31) & ~31;
    const int j_lo = min(M, warp * chunk), j_hi = min(M, j_lo + chunk);
    uint32_t ngt = 0, neq = 0;
    for (int j0 = j_lo; j0 < j_hi; j0 += 32) {
      const int j = j0 + lane;
      const uint32_t x = j < j_hi ? list_key[j] : 0u;
      ngt += __popc(__ballot_sync(full, j < j_hi && x > T));
      neq += __popc(__ballot_sync(full, j < j_hi && x == T));
    }
    if (lane == 0) { warp_a[warp] = pgt; warp_b[warp] = peq; warp_c[warp] = ngt; warp_d[warp] = neq; }
    __syncthreads();
    const bool has = lane < WARPS;
    const uint32_t gt0 = __reduce_add_sync(full, has ? warp_a[lane & (WARPS - 1)] : 0u);
    const uint32_t eq0 = __reduce_add_sync(full, has ? warp_b[lane & (WARPS - 1)] : 0u);
    const uint32_t wg = has ? warp_c[lane & (WARPS - 1)] : 0u, we = has ? warp_d[lane & (WARPS - 1)] : 0u;
    const uint32_t gt_all = gt0 + __reduce_add_sync(full, wg), eq_all = eq0 + __reduce_add_sync(full, we);
    uint32_t gt_before = gt0 + __reduce_add_sync(full, lane < warp ? wg : 0u);
    uint32_t eq_before = eq0 + __reduce_add_sync(full, lane < warp ? we : 0u);
    own0 = static_cast<int>(gt0 + min(eq0, need_eq));
    own1 = static_cast<int>(gt_all + min(eq_all, need_eq));
    if (rank == C - 1 && tid == 0 && own1 != k) atomicOr(p.status, kStatusSelectMismatch);
    for (int j0 = j_lo; j0 < j_hi; j0 += 32) {
      const int j = j0 + lane;
      const uint2 kv = j < j_hi ? make_uint2(list_key[j], static_cast<uint32_t>(lo) + list_pos[j]) : make_uint2(0u, 0u);
      const bool is_gt = j < j_hi && kv.x > T, is_eq = j < j_hi && kv.x == T;
      const uint32_t bg = __ballot_sync(full, is_gt), be = __ballot_sync(full, is_eq);
      const uint32_t g = gt_before + __popc(bg & lt), e = eq_before + __popc(be & lt);
      if (is_gt || (is_eq && e < need_eq)) {
        const int at = static_cast<int>(g + min(e, need_eq));
        out[at] = static_cast<int32_t>(kv.y);
        kept[at - own0] = static_cast<int32_t>(kv.y);       // over the scores, which nobody reads any more
      }
      gt_before += __popc(bg);
      eq_before += __popc(be);
    }
    if (C > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");   // done with the others' memory
  } else if (C > 1) {
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
  if (!selecting && k >= P) {                               // nothing to evict: this CTA's share of the identity list
    own0 = lo;
    own1 = lo + len;
    for (int i = tid; i < len; i += THREADS) out[lo + i] = lo + i;
  }
  // The window positions close the list (Section 4.2.1: always retained).
  if (rank == C - 1)
    for (int j = tid; j < alpha; j += THREADS) out[k + j] = P + j;

  // ---- eviction by gather (appendix on torch.gather).  Every CTA copies the rows of its own slice, unless the list is
  //      long: then it is dealt out evenly (kept rows may crowd into one slice)
  if (p.k_out == nullptr) {
    if (selecting && C > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    return;
  }
  const bool even = C > 1 && selecting && k >= kSelEvenRows;
  if (even) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");        // the list is complete
  else __syncthreads();                                     // kept[] is complete
  const char* kb = static_cast<const char*>(p.k.ptr) + (b * p.k.sb + h * p.k.sh) * p.elem_bytes;
  const char* vb = static_cast<const char*>(p.v.ptr) + (b * p.v.sb + h * p.v.sh) * p.elem_bytes;
  const int64_t k_step = p.k.st * p.elem_bytes, v_step = p.v.st * p.elem_bytes;
  const int first = even ? 0 : own0;                        // list entries [first, first + listed), then the window
  const int listed = even ? k : own1 - own0;
  const int total = (listed + (even || rank == C - 1 ? alpha : 0)) << p.log_pieces;
  const int start = even ? rank * THREADS + tid : tid, stride = even ? C * THREADS : THREADS;
  constexpr int U = 4;
  for (int g0 = start; g0 < total; g0 += U * stride) {
    uint4 kv[U], vv[U];
    int64_t dst[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int g = g0 + u * stride;
      dst[u] = -1;
      if (g >= total) continue;
      const int r = g >> p.log_pieces, piece = g & ((1 << p.log_pieces) - 1);
      const int pos = r >= listed ? P + (r - listed) : (!selecting ? first + r : (even ? __ldcg(out + r) : kept[r]));
      const int dr = r >= listed ? k + (r - listed) : first + r;
      int64_t to = row0 + dr;
      if (p.paged) {
        to = paged_row(p.pt, b, h, dr);
        if (to < 0) {
          if (piece == 0) atomicOr(p.status, kStatusBadPage);
          continue;
        }
      }
      dst[u] = (to << p.log_pieces) + piece;
      kv[u] = reinterpret_cast<const uint4*>(kb + pos * k_step)[piece];
      vv[u] = reinterpret_cast<const uint4*>(vb + pos * v_step)[piece];
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (dst[u] >= 0) {
        static_cast<uint4*>(p.k_out)[dst[u]] = kv[u];
        static_cast<uint4*>(p.v_out)[dst[u]] = vv[u];
      }
  }
  if (selecting && C > 1 && !even) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

}  // namespace pkv
