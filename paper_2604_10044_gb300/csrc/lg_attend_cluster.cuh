// Decode attention by thread-block clusters that merge their split-K partials through distributed
// shared memory, for bf16 caches (lg_attend_cluster.cu, tensor cores) and fp32 ones
// (lg_attend_cluster_f32.cu).  lg_attend_mma.cu and lg_attend.cu hold the passes for batches and
// calls past its limits.
//
// What bounds a call: a long one the memory, a short one (a layer at one sequence: 64 KB a CTA)
// latency.  The persistent pass pays for its work sharing there: a kernel before it that resets
// its counters, a claim per chunk, and a merge through L2 (partials, an arrival count, partials
// again, one warp for all heads of a group).  Here each cluster owns a run of whole (layer,
// sequence, kv-head) groups, about the same number of tiles each, and splits the run's tiles
// evenly over its CTAs, so every CTA streams one contiguous range of tiles through a ring of
// tensor copies.  A group that lies within one CTA is finished there.  The (at most two) groups
// a CTA shares with its neighbours are folded over its warps, and the folded pieces {M, l, u,
// sigma, o[32]} go straight into the shared memory of the CTAs that own them (the sharing CTAs own
// a group's pieces in turn), each store counting its bytes on the owner's barrier; the owner
// merges once all have arrived (a cluster barrier in its place waits for the stores'
// acknowledgements first: 5.74 -> 5.58 us a layer at one sequence of 1024 rows, 32 sequences of
// 128 9.70 -> 9.09).  No counters, no partials in memory, no other launch.  Uneven lengths cost
// little while groups outnumber the clusters: a CTA with less to read leaves its bandwidth to the
// others (one CTA streams up to 90 GB/s, 1.8 times its even share).  A few long groups, which have
// at most 8 CTAs each, are the general passes' (lg_attend_rule.cuh).
//
// GB300, one layer of 28 (append and attention, called one by one in a graph), one sequence of
// 1024 rows, 16/8 heads of 128: 12.0 -> 5.6 us.  Of a CTA's 4.1 us after its wait, 1.6 go to its
// first copies, 0.7 to the tile, 0.8 to the fold, 0.4 to the pieces' way and 0.4 to the merge
// (clock64 at each phase).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <atomic>

#include "lg_attend_rule.cuh"
#include "lg_common.cuh"
#include "lg_internal.h"
#include "lg_mma_tile.cuh"

namespace lg {

namespace {

constexpr int kClusterSeqs = 64;  // batch at most (two sequences a lane in the prologue's scan)

// What differs between the element types: the tile and the ring, and a consumer warp's work.
//   kTile rows a tile, kBoxes boxes of kBoxCols columns per tensor, kStages stages in the ring
//   kWarps consumer warps, which share every tile
//   begin(the query rows, whether it is the segment's first tile), update(a tile), join() (the
//   lanes' sums) and store(to, or added to, a row of D + 4 floats per head: o, then {M, l, u,
//   sigma}); with kFlushTiles > 0 a segment's sums are stored every so many tiles
template <typename T, int D, int G>
struct Pass;

template <typename T, int D, int G>
struct ClusterCfg {
  using P = Pass<T, D, G>;
  static constexpr int kSize = Elem<T>::kSize;
  static constexpr int kWarps = P::kWarps, kStages = P::kStages;
  static constexpr int kThreads = (kWarps + 1) * 32;
  static constexpr int kBoxBytes = P::kTile * P::kBoxCols * kSize;
  static constexpr int kStageBytes = 2 * P::kBoxes * kBoxBytes;
  static constexpr int kTileBytes = 2 * P::kTile * D * kSize;
  static_assert(kStageBytes == kTileBytes && P::kBoxCols * kSize == 128, "whole rows");
  static constexpr int kQBytes = G * D * kSize;         // a group's query rows
  static constexpr int kRow = D + 4;                    // one head's o, then {M, l, u, sigma}
  static constexpr int kWarpFloats = kWarps * G * kRow;  // one segment's warp partials
  // a group's output in units of 32 elements of a head: unit u is elements 32 (u / G) ... of
  // head u mod G
  static constexpr int kUnits = G * (D / 32);
  // the fold of a segment: kTasks warps, each kTaskUnits units of one head, for which the weights
  // of the warps' partials are formed once (Pass::kFoldUnits units at most: same-box A/B of 1
  // against 4, the fp32 layer of 4 sequences of 8191 rows 47.5 -> 45.6 us, the bf16 one of 16384
  // rows 17.2 -> 17.7, its tile loop short of registers)
  static constexpr int split() {
    int s = 1;
    while (2 * s <= D / 32 && (G * 2 * s <= kWarps || D / 32 / s > P::kFoldUnits)) s *= 2;
    return s;
  }
  static constexpr int kTasks = G * split(), kTaskUnits = D / 32 / split();
  static constexpr int kUnit = 36;                      // floats of a unit's partial: o, then stats
  // a CTA owns every np-th unit of a group shared by np CTAs and receives np partials of each
  static constexpr int recv_max() {
    int m = 0;
    for (int np = 2; np <= kMaxCluster; ++np) {
      const int r = (kUnits + np - 1) / np * np;
      if (r > m) m = r;
    }
    return m;
  }
  static constexpr int kRecvFloats = recv_max() * kUnit;
  static constexpr int kSmem = kStages * kStageBytes + 2 * kQBytes +
                               (kWarpFloats + 2 * kRecvFloats) * (int)sizeof(float) + 1024;
  static_assert(kSmem + 1024 <= 227 * 1024, "shared memory of a CTA, with its static arrays");
};

__device__ __forceinline__ int cluster_rank() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the cluster's barrier (every thread; whole warps, converged): release at the arrival, acquire
// at the wait, cluster scope
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared-memory address of the same variable in another CTA of the cluster, and stores to it
__device__ __forceinline__ uint32_t peer_addr(const void *p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  return a;
}
// (each counts its bytes on the barrier, which lies in the same CTA as the address)
__device__ __forceinline__ void peer_st(uint32_t addr, float v, uint32_t bar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(addr),
      "f"(v), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void peer_st4(uint32_t addr, float4 v, uint32_t bar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, "
      "[%5];" ::"r"(addr),
      "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
      : "memory");
}

// keeps the barrier's current phase from ever completing (a byte more than will arrive)
__device__ __forceinline__ void mbar_hold(uint64_t *bar) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar))
               : "memory");
}

template <int kThreads>
__device__ __forceinline__ void named_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kThreads) : "memory");
}
template <int kThreads>
__device__ __forceinline__ void named_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kThreads) : "memory");
}

// floor(x / d) for 0 <= x < 2^24, d >= 1 and a quotient below 2^20: in floats it is off by at most
// one (the integer division's longer chain sat on the way to the first copy)
__device__ __forceinline__ int quick_div(int x, int d) {
  int q = (int)__fdividef((float)x, (float)d);
  q -= q * d > x;
  q += (q + 1) * d <= x;
  return q;
}

// One (layer, sequence, kv-head) group among the call's tiles, numbered layer by layer, sequence
// by sequence, kv-head by kv-head.
struct TileGroup {
  int lloc, b, kvh;
  int start, tiles;  // its first tile and their number
};

// The call's tiles: pre[b] tiles in the sequences before b (of one kv-head of one layer), total
// over the batch, rows to a tile.
struct TileSpace {
  const int *len, *pre;  // [batch]
  int batch, H_kv, n_layers, total, rows;
  __device__ __forceinline__ int tiles(int b) const { return (len[b] + rows - 1) / rows; }
  __device__ __forceinline__ TileGroup find(int t) const {
    TileGroup g;
    const int per_layer = total * H_kv;
    g.lloc = n_layers > 1 ? quick_div(t, per_layer) : 0;
    const int r = t - g.lloc * per_layer;
    int b = 0;
    if (batch > 1) {
#pragma unroll
      for (int st = kClusterSeqs / 2; st >= 1; st >>= 1)
        if (b + st < batch && pre[b + st] * H_kv <= r) b += st;
    }
    g.b = b;
    g.tiles = tiles(b);
    const int r0 = pre[b] * H_kv;
    g.kvh = quick_div(r - r0, g.tiles);
    g.start = g.lloc * per_layer + r0 + g.kvh * g.tiles;
    return g;
  }
  __device__ __forceinline__ void next(TileGroup &g) const {
    g.start += g.tiles;
    if (++g.kvh < H_kv) return;
    g.kvh = 0;
    do {
      if (++g.b == batch) {
        g.b = 0;
        ++g.lloc;
      }
      g.tiles = tiles(g.b);
    } while (g.tiles == 0);
  }
};

// The first tile of cluster k's run among n_cl (of T tiles): an even share of the tiles, rounded
// to the nearest group boundary.
__device__ __forceinline__ int run_bound(const TileSpace &ts, int T, int k, int n_cl) {
  const int x = (int)((unsigned)T * (unsigned)k / (unsigned)n_cl);
  if (x <= 0 || x >= T) return x;
  const TileGroup g = ts.find(x);
  return 2 * (x - g.start) < g.tiles ? g.start : g.start + g.tiles;
}

// out and statistics of one head from its merged sums (a warp's 32 elements of the output)
template <typename T, int D>
__device__ __forceinline__ void finish(const AttendArgs &a, int64_t head, int e, bool first,
                                       float M, float l, float u, float sg, float o) {
  const float inv_l = 1.f / l;
  Elem<T>::store(a.out, head * D + e, o * inv_l);
  if (first) {
    constexpr float kLn2 = 0.69314718055994530942f;
    *reinterpret_cast<float4 *>(a.stats + head * 4) =
        make_float4(M * kLn2, l, logf(l) - u * kLn2 * inv_l, sg * inv_l);
    if (a.final_ml) {
      a.final_ml[head * 2] = M;
      a.final_ml[head * 2 + 1] = l;
    }
  }
}

// whether the general pass is the faster for a call's lengths: the longest of each lane's two
// sequences, tiles of all of them (not inlined: few calls ask, and the others' way to their first
// copies stays as short as it was)
template <typename T, int D, int G>
__device__ __noinline__ bool leave_to_general(int groups, int rows, int batch, int total,
                                              int chunk_rows, int max_chunks, int sms, int ctas,
                                              int n_cl) {
  const CallShape s = call_shape({Elem<T>::kDtype == LG_BF16, D, G, Pass<T, D, G>::kTile}, groups,
                                 __reduce_max_sync(0xffffffffu, rows), chunk_rows, max_chunks, sms);
  return general_gains_us(s, batch, total, total == s.tiles * batch, ctas, n_cl) > 0.f;
}

}  // namespace

template <typename T, int D, int G>
__global__ void __launch_bounds__(ClusterCfg<T, D, G>::kThreads, 1)
attend_cluster_kernel(const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmV, AttendArgs a, int ctas, int n_cl,
                      int rows_total) {
  using P = Pass<T, D, G>;
  using Cl = ClusterCfg<T, D, G>;
  constexpr int kWarps = Cl::kWarps, kRow = Cl::kRow, kTile = P::kTile;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[Cl::kStages];
  __shared__ __align__(8) uint64_t empty_bar[Cl::kStages];
  __shared__ __align__(8) uint64_t recv_bar[2];  // a slot's pieces have arrived
  __shared__ __align__(8) uint64_t q_full[2], q_empty[2];  // query rows of segment i in buffer i & 1
  __shared__ int s_len[kClusterSeqs], s_pre[kClusterSeqs], s_off[kClusterSeqs];
  __shared__ int s_total, s_c0, s_c1, s_skip;
  __shared__ int s_todo;  // besides the tiles: 1 empty sequences, 2 the general pass's counters
  __shared__ int s_stop;  // bit 0: the status was set before this call, bit 1: a wait ran out
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *qbuf = smem + Cl::kStages * Cl::kStageBytes;  // [2][G][D]
  float *part = reinterpret_cast<float *>(qbuf + 2 * Cl::kQBytes);  // [warp][G][kRow]
  float *recv = part + Cl::kWarpFloats;  // [2][recv_max][kUnit]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = cluster_rank(), cluster = quick_div(blockIdx.x, ctas);
  // the producer's early look at the lengths and offsets (see there), two sequences a lane
  int early_n[2] = {0, 0}, early_off[2] = {0, 0};
  if (warp == kWarps) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (2 * lane + k < a.batch) {
        early_n[k] = __ldcg(a.len + 2 * lane + k);
        early_off[k] = (int)__ldcg(a.seq_off + 2 * lane + k);
      }
  }
  if (threadIdx.x == kWarps * 32) {
    for (int s = 0; s < Cl::kStages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], kWarps);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&q_full[s], 1);
      mbar_init(&q_empty[s], kWarps);
      mbar_init(&recv_bar[s], 1);
    }
    mbar_fence_init();
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmK)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmV)) : "memory");
  }
  __syncwarp();
  // waited for before the first store to a peer: every CTA has started and set up its barriers
  cluster_arrive();
  auto stopped = [&] { return *(volatile int *)&s_stop; };
  TileSpace ts;
  ts.len = s_len;
  ts.pre = s_pre;
  ts.batch = a.batch;
  ts.H_kv = a.H_kv;
  ts.n_layers = a.n_layers;
  ts.rows = kTile;

  if (warp == kWarps) {
    // ------------------------------------------------------------ producer
    // (this warp alone reads the lengths and forms the ranges: the others pick them up from
    // shared memory while its first copies are in flight)
    uint64_t evict_first, evict_normal;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(evict_first));
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(evict_normal));
    // The groups of this cluster if all have as many tiles: [gi0, gi1), and the first one's place
    // (known before the lengths are: a group's share of the tiles is then its share of the groups)
    const int groups = a.n_layers * a.batch * a.H_kv;
    const int gi0 = quick_div(groups * cluster, n_cl), gi1 = quick_div(groups * (cluster + 1), n_cl);
    TileGroup g;
    {
      const int lb = quick_div(gi0, a.H_kv);
      g.kvh = gi0 - lb * a.H_kv;
      g.lloc = quick_div(lb, a.batch);
      g.b = lb - g.lloc * a.batch;
    }
    // cache row of slot 0 of a group's layer and kv-head (the first group's before the wait)
    auto stream_row = [&](const TileGroup &g) {
      return (int)(((int64_t)(a.layer0 + g.lloc) * a.H_kv + g.kvh) * a.S_total);
    };
    int row0 = stream_row(g);
    const int first_kvh = g.kvh, first_lloc = g.lloc;
    // Before the wait, the lengths as they are now (past L1) give the range this CTA will most
    // likely have, if they all agree (a few instructions then).  Its first tiles are requested into
    // L2, a hint: in a step the kernel before is a short one (the append), beside which the memory
    // idled.  In a call of few tiles a CTA, bound by latency, the copies of its first segment are
    // then issued right after the wait, beside the read of the lengths that count; if those give
    // another range, the copies are dropped (the consumers pass over their stages).  What is read
    // early decides only which rows are fetched first.  (GB300, layers one by one in a graph: 1
    // sequence of 1024 rows 6.39 us, 6.06 with the L2 requests, 5.73 with the early copies; 8 of
    // 4096 rows 25.7, 23.5 and, as longer calls gain nothing from them, 24.0.)
    int guess_t[2], guess_tiles = 0, guess_row = 0, guess_off = 0;
    TileGroup guess = g;  // the first segment's group; guess_tiles of its tiles, from guess_row on
    {
#pragma unroll
      for (int k = 0; k < 2; ++k)
        guess_t[k] = (max(min(early_n[k], a.max_len), 0) + kTile - 1) / kTile;
      const int tiles = __shfl_sync(0xffffffffu, guess_t[0], 0);
      const bool same = (2 * lane >= a.batch || guess_t[0] == tiles) &&
                        (2 * lane + 1 >= a.batch || guess_t[1] == tiles);
      if (__all_sync(0xffffffffu, same) && tiles > 0) {
        const int len = (gi1 - gi0) * tiles;
        const int u = quick_div(len * rank, ctas), end = quick_div(len * (rank + 1), ctas);
        const int skip = quick_div(u, tiles);
        if (skip > 0) {
          const int gi = gi0 + skip, lb = quick_div(gi, a.H_kv);
          guess.kvh = gi - lb * a.H_kv;
          guess.lloc = quick_div(lb, a.batch);
          guess.b = lb - guess.lloc * a.batch;
        }
        const int off0 = __shfl_sync(0xffffffffu, early_off[0], guess.b >> 1);
        const int off1 = __shfl_sync(0xffffffffu, early_off[1], guess.b >> 1);
        guess_off = guess.b & 1 ? off1 : off0;
        const int64_t row = (int64_t)stream_row(guess) + guess_off +
                            (int64_t)(u - skip * tiles) * kTile;
        int ahead = 0;
        if (row >= 0 && row < rows_total) {
          guess_row = (int)row;
          ahead = min(min(end, (skip + 1) * tiles) - u, Cl::kStages);
          if (end - u <= Cl::kStages) guess_tiles = ahead;
        }
        // box and tile of this lane
        const int x = lane % (2 * P::kBoxes), i = lane / (2 * P::kBoxes);
        if (i < ahead)
          tma_prefetch_2d(x < P::kBoxes ? &tmK : &tmV, x % P::kBoxes * P::kBoxCols,
                          guess_row + i * kTile);
      }
      __syncwarp();
    }
    auto head_first = [&](const TileGroup &g) {
      return ((int64_t)g.lloc * a.batch + g.b) * a.H_q + (int64_t)g.kvh * G;
    };
    const int64_t guess_head0 = head_first(guess);
    auto copy_tile = [&](int st, int row, uint64_t policy) {
      unsigned char *stage = smem + (size_t)st * Cl::kStageBytes;
      mbar_arrive_expect_tx(&full_bar[st], Cl::kStageBytes);
#pragma unroll
      for (int h = 0; h < P::kBoxes; ++h) {
        tma_load_2d(stage + h * Cl::kBoxBytes, &tmK, h * P::kBoxCols, row, &full_bar[st], policy);
        tma_load_2d(stage + (P::kBoxes + h) * Cl::kBoxBytes, &tmV, h * P::kBoxCols, row,
                    &full_bar[st], policy);
      }
    };
    auto copy_q = [&](int qb, int64_t head0) {
      mbar_arrive_expect_tx(&q_full[qb], Cl::kQBytes);
      bulk_load(qbuf + qb * Cl::kQBytes, (const unsigned char *)a.q + head0 * D * Cl::kSize,
                Cl::kQBytes, &q_full[qb]);
    };
    // K/V are streamed once; a call that fits beside the rest of the step stays in L2
    auto tile_policy = [&](int total) {
      return total * a.H_kv * a.n_layers <= kL2KeepBytes / Cl::kTileBytes ? evict_normal
                                                                           : evict_first;
    };
    const uint64_t guess_policy = tile_policy(guess_t[0] * a.batch);
    pdl_enter();
    // lengths and the tiles before each sequence, two sequences a lane (requested before the early
    // copies are issued, first used after)
    int n[2], t[2], any_empty = 0;
    int64_t off[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int b = 2 * lane + k;
      n[k] = b < a.batch ? a.len[b] : -1;
      off[k] = b < a.batch ? a.seq_off[b] : 0;
    }
    const int32_t status = lane == 0 && a.status ? *(volatile const int32_t *)a.status : 0;
    if (lane == 0 && guess_tiles > 0) {
      for (int i = 0; i < guess_tiles; ++i) copy_tile(i, guess_row + i * kTile, guess_policy);
      copy_q(0, guess_head0);
    }
    __syncwarp();
    const int bad = __shfl_sync(0xffffffffu, status, 0);
    bool hit = guess_tiles > 0 && !bad;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (2 * lane + k < a.batch) s_off[2 * lane + k] = (int)off[k];
      hit = hit && (int)off[k] == early_off[k];
      // (a negative length is an error over fp32 rows and reads as none over bf16 ones, as in the
      // general passes)
      if (n[k] > a.max_len ||
          (Elem<T>::kDtype == LG_F32 && n[k] < 0 && 2 * lane + k < a.batch)) {
        set_status(a.status, LG_ERR_CAPACITY);
        n[k] = -1;
        hit = false;
      }
      any_empty |= n[k] == 0;
      n[k] = max(n[k], 0);
      t[k] = (n[k] + kTile - 1) / kTile;
      hit = hit && (2 * lane + k >= a.batch || t[k] == guess_t[k]);
    }
    hit = __all_sync(0xffffffffu, hit);
    const int t_first = __shfl_sync(0xffffffffu, t[0], 0);
    const bool same = (2 * lane >= a.batch || t[0] == t_first) &&
                      (2 * lane + 1 >= a.batch || t[1] == t_first);
    int c0 = 0, c1 = 0, u0 = 0, u1 = 0;
    if (__all_sync(0xffffffffu, same)) {
      ts.total = t_first * a.batch;
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (2 * lane + k < a.batch) {
          s_len[2 * lane + k] = n[k];
          s_pre[2 * lane + k] = (2 * lane + k) * t_first;
        }
      c0 = gi0 * t_first;
      c1 = gi1 * t_first;
      u0 = c0 + quick_div((c1 - c0) * rank, ctas);
      u1 = c0 + quick_div((c1 - c0) * (rank + 1), ctas);
      g.tiles = t_first;
      g.start = c0;
      __syncwarp();
      while (g.start + t_first <= u0 && u0 < u1) ts.next(g);
    } else {
      int upto = t[0] + t[1];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += x;
      }
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (2 * lane + k < a.batch) {
          s_len[2 * lane + k] = n[k];
          s_pre[2 * lane + k] = upto - t[0] - t[1] + (k ? t[0] : 0);
        }
      ts.total = __shfl_sync(0xffffffffu, upto, 31);
      __syncwarp();
      const int all = ts.total * a.H_kv * a.n_layers;
      // this cluster's run of groups [c0, c1) (even lanes form its start, odd lanes its end)
      const int x = run_bound(ts, all, cluster + (lane & 1), n_cl);
      c0 = __shfl_sync(0xffffffffu, x, 0);
      c1 = __shfl_sync(0xffffffffu, x, 1);
      u0 = c0 + quick_div((c1 - c0) * rank, ctas);
      u1 = c0 + quick_div((c1 - c0) * (rank + 1), ctas);
      if (u0 < u1) g = ts.find(u0);
    }
    any_empty = __any_sync(0xffffffffu, any_empty);
    bool general = false;
    if (a.gate) {
      // the general pass follows: one of the two runs, by the lengths (the same in every CTA)
      general = leave_to_general<T, D, G>(groups, max(n[0], n[1]), a.batch, ts.total, a.chunk_rows,
                                          a.max_chunks, a.sms, ctas, n_cl);
      if (!general && blockIdx.x == 0 && lane == 0) *a.gate = -1;
      if (general) {
        c0 = c1 = u0 = u1 = 0;
        hit = false;
      }
    }
    if (lane == 0) {
      s_total = ts.total;
      s_c0 = c0;
      s_c1 = c1;
      s_todo = bad ? 0 : general ? 2 : any_empty;
      s_skip = hit ? 0 : guess_tiles;
      s_stop = bad != 0;
    }
    __syncwarp();
    named_arrive<Cl::kThreads>(1);
    if (lane == 0 && u0 < u1 && !bad) {
      const uint64_t policy = tile_policy(ts.total);
      auto timed_out = [&](uint64_t *bar, uint32_t parity) {
        if (mbar_wait(bar, parity)) return false;
        set_status(a.status, LG_ERR_TIMEOUT);
        return true;
      };
      // stages used so far, segments begun so far (a dropped guess counts as one)
      uint32_t it = guess_tiles, seg = guess_tiles > 0 && !hit;
      bool ok = true, begun = hit;
      for (int t = hit ? u0 + guess_tiles : u0; t < u1 && ok; ++seg) {
        const int end = min(g.start + g.tiles, u1);
        if (seg > 0 || g.kvh != first_kvh || g.lloc != first_lloc) row0 = stream_row(g);
        const int row = row0 + s_off[g.b] - g.start * kTile;
        for (; t < end; ++t, ++it) {
          const int st = it % Cl::kStages;
          if (it >= (uint32_t)Cl::kStages &&
              timed_out(&empty_bar[st], ((it / Cl::kStages) - 1) & 1)) {
            ok = false;
            break;
          }
          copy_tile(st, row + t * kTile, policy);
          if (!begun) {
            const int qb = seg & 1;
            if (seg >= 2 && timed_out(&q_empty[qb], ((seg >> 1) - 1) & 1)) {
              ok = false;
              break;
            }
            copy_q(qb, head_first(g));
            begun = true;
          }
        }
        begun = false;
        if (ok && t < u1) ts.next(g);
      }
    }
    __syncwarp();
    cluster_wait();
    return;
  }

  // -------------------------------------------------------------- consumers
  pdl_enter();
  named_sync<Cl::kThreads>(1);
  cluster_wait();
  ts.total = s_total;
  // this CTA's tiles [u0, u1): an even share of the cluster's (read again for each use: registers
  // are short)
  auto first_tile = [&](int r) {
    const int c0 = *(volatile int *)&s_c0, c1 = *(volatile int *)&s_c1;
    return c0 + quick_div((c1 - c0) * r, ctas);
  };
  // The CTAs of the cluster that share a group: lane r stands for CTA r (np of them, mine before
  // this one).  CTA number i of them owns units i, i + np, ... of the group.
  struct Sharers {
    int lo, nth;   // lane r: CTA r's first tile, its number among the sharers (-1: none)
    int mine, np;
  };
  auto sharers = [&](const TileGroup &g) {
    Sharers s;
    s.lo = first_tile(min(lane, ctas));
    const int hi = first_tile(min(lane + 1, ctas));
    const bool in = lane < ctas && s.lo < hi && s.lo < g.start + g.tiles && hi > g.start;
    const unsigned mask = __ballot_sync(0xffffffffu, in);
    s.nth = in ? __popc(mask & ((1u << lane) - 1u)) : -1;
    s.mine = __popc(mask & ((1u << rank) - 1u));
    s.np = __popc(mask);
    return s;
  };
  struct UnitAddr {
    uint32_t data, bar;
  };
  // where this CTA's partial of a group's unit goes: the owner, sharer number un % np, and its
  // slot of this group
  auto unit_addr = [&](const Sharers &sh, const TileGroup &g, int un) {
    const int j = quick_div(un, sh.np);
    const int owner = __ffs(__ballot_sync(0xffffffffu, sh.nth == un - j * sh.np)) - 1;
    const int slot = __shfl_sync(0xffffffffu, sh.lo, owner) >= g.start ? 0 : 1;
    UnitAddr u;
    u.data = peer_addr(recv + slot * Cl::kRecvFloats + (j * sh.np + sh.mine) * Cl::kUnit, owner);
    u.bar = peer_addr(&recv_bar[slot], owner);
    return u;
  };
  const int u0 = first_tile(rank), u1 = first_tile(rank + 1);
  TileGroup g = {};
  if (u0 < u1) g = ts.find(u0);
  if (s_todo == 2) {
    // the call is left to the general pass: its counters (the gate is their first) to zero and the
    // direction word flipped, as zero_counters_kernel does
    const int words = 1 + a.n_layers * a.batch * a.H_kv;
    for (int i = blockIdx.x * kWarps * 32 + threadIdx.x; i <= words; i += gridDim.x * kWarps * 32)
      a.counter[i] = i < words ? 0 : a.counter[i] ^ 1;
  } else if (s_todo == 1) {
    // empty sequences: zero output, m = -inf, l = H = S = 0
    for (int i = blockIdx.x; i < a.n_layers * a.batch * a.H_kv; i += gridDim.x) {
      const int lb = i / a.H_kv;
      if (a.len[lb % a.batch] != 0) continue;
      const int64_t head0 = (int64_t)lb * a.H_q + (int64_t)(i % a.H_kv) * G;
      for (int x = threadIdx.x; x < G * D; x += kWarps * 32)
        Elem<T>::store(a.out, head0 * D + x, 0.f);
      if (threadIdx.x < G * 4)
        a.stats[head0 * 4 + threadIdx.x] = threadIdx.x % 4 == 0 ? -INFINITY : 0.f;
    }
  }
  // groups in the slots: 0 for a segment that starts at u0, 1 for another that ends at u1
  // (np 0: not in use; mine and np as above, the group's first head)
  struct Slot {
    int mine, np, head0;
  };
  Slot slot0 = {}, slot1 = {};
  P pass;
  uint32_t it = 0, seg = 0;
  // With the status set nothing is read or written, but a CTA still passes its (meaningless)
  // pieces on: the status may have been set by another CTA of this launch, and its peers wait.
  const bool bad = stopped() & 1;
  // The waits of one lane: at the limit a warp's lanes may see a barrier differently, and what
  // follows has shuffles and matrix instructions of all lanes, so nothing branches on them.  After
  // the first that runs out no copy is waited for, what is late is worked on as it is, and no stage
  // or query buffer gets back to the producer, which would arm a barrier that may be in use (held
  // here, off every tile's way: a look at s_stop before each copy cost one fp32 sequence of 9000
  // rows 10.7 -> 11.3 us).
  auto ran_out = [&] {
    set_status(a.status, LG_ERR_TIMEOUT);
    atomicOr(&s_stop, 2);
    for (int s = 0; s < Cl::kStages; ++s) mbar_hold(&empty_bar[s]);
    for (int s = 0; s < 2; ++s) mbar_hold(&q_empty[s]);
  };
  auto landed = [&](uint64_t *bar, uint32_t parity) {
    if (!mbar_try_wait(bar, parity) && !stopped() && !mbar_wait(bar, parity)) ran_out();
  };
  if (s_skip > 0) {
    // a dropped guess: its stages and queries pass unused
    bool in = mbar_wait(&q_full[0], 0);
    for (; it < (uint32_t)s_skip; ++it) {
      in = in && mbar_wait(&full_bar[it], 0);
      if (!in) ran_out();
      if (lane == 0) mbar_arrive(&empty_bar[it]);
    }
    if (lane == 0) mbar_arrive(&q_empty[0]);
    seg = 1;
  }
  for (int t = u0; t < u1; ++seg) {
    const int start = t, end = min(g.start + g.tiles, u1);
    const int n = s_len[g.b];
    const int suffix_lo = n - min(a.suffix_w, n);
    // (32 bits hold every row and head of a call: the limits of attend_cluster_takes)
    const int lrow = (g.lloc * a.H_kv + g.kvh) * (int)a.S_total + s_off[g.b];
    const int qb = seg & 1;
    // who shares the group and where this warp's first unit goes, formed while the first copies
    // are in flight (after the tiles they would sit on the way to the merge)
    const bool whole = start == g.start && end == g.start + g.tiles;
    const int head0 = (g.lloc * a.batch + g.b) * a.H_q + g.kvh * G;
    Sharers sh = {};
    UnitAddr dst0 = {};
    auto place_units = [&] {
      if (whole) return;
      sh = sharers(g);
      if (threadIdx.x == 0)  // the pieces of its units: np times (32 + 4) floats each
        mbar_arrive_expect_tx(&recv_bar[start == u0 ? 0 : 1],
                              quick_div(Cl::kUnits - sh.mine + sh.np - 1, sh.np) * sh.np *
                                  Cl::kUnit * (int)sizeof(float));
      dst0 = unit_addr(sh, g, warp / G * Cl::kTaskUnits * G + warp % G);
    };
    if (P::kEarlyUnits) place_units();
    // (all of the segment at once, or kFlushTiles tiles at a time)
    do {
      const int from = t, stop = P::kFlushTiles ? min(end, t + P::kFlushTiles) : end;
      landed(&q_full[qb], (seg >> 1) & 1);
      pass.begin(qbuf + qb * Cl::kQBytes, from == start, a.qscale, lane);
      for (; t < stop; ++t, ++it) {
        const int st = it % Cl::kStages;
        landed(&full_bar[st], (it / Cl::kStages) & 1);
        const int r0 = (t - g.start) * kTile;
        float *logits = a.logits && !bad ? a.logits + (int64_t)(lrow + r0) * G : nullptr;
        pass.update(smem + (size_t)st * Cl::kStageBytes, min(kTile, n - r0), suffix_lo - r0, logits,
                    a.qscale, warp, lane);
        if (lane == 0) mbar_arrive(&empty_bar[st]);
      }
      if (t == end && lane == 0) mbar_arrive(&q_empty[qb]);
      // the segment's warp partials folded: a whole group is finished here, a part of a group goes
      // to the owners of its units
      pass.join();
      if (from == start && start != u0) named_sync<kWarps * 32>(2);  // the segment before is folded
      pass.store(part + warp * G * kRow, from != start, lane);
    } while (P::kFlushTiles && t < end);
    if (!P::kEarlyUnits) place_units();
    named_sync<kWarps * 32>(2);
#pragma unroll 1
    for (int task = warp; task < Cl::kTasks; task += kWarps) {
      const int h = task % G, first_slice = task / G * Cl::kTaskUnits;
      float f[kWarps], M = -INFINITY, l = 0.f, u = 0.f, sg = 0.f;
      {
        float4 w4[kWarps];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
          w4[w] = *reinterpret_cast<const float4 *>(part + (w * G + h) * kRow + D);
          M = fmaxf(M, w4[w].x);
        }
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
          // a warp that saw no row of this segment has l = u = 0 and M = -inf: no weight
          const float dm = fmaxf(w4[w].x - M, -1e30f);
          f[w] = exp2f(dm);
          l += f[w] * w4[w].y;
          u += f[w] * (w4[w].z + dm * w4[w].y);
          sg += f[w] * w4[w].w;
        }
      }
#pragma unroll
      for (int k = 0; k < Cl::kTaskUnits; ++k) {
        const int slice = first_slice + k, un = slice * G + h, e = slice * 32 + lane;
        float o = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) o += f[w] * part[(w * G + h) * kRow + e];
        if (whole) {
          if (!bad) finish<T, D>(a, head0 + h, e, slice == 0 && lane == 0, M, l, u, sg, o);
        } else {
          const UnitAddr dst = k == 0 && task == warp ? dst0 : unit_addr(sh, g, un);
          peer_st(dst.data + lane * 4, o, dst.bar);
          if (lane == 0) peer_st4(dst.data + 32 * 4, make_float4(M, l, u, sg), dst.bar);
        }
      }
    }
    if (!whole) (start == u0 ? slot0 : slot1) = Slot{sh.mine, sh.np, head0};
    if (t < u1) ts.next(g);
  }
#pragma unroll 1
  for (int slot = 0; slot < 2; ++slot) {
    const int mine = slot ? slot1.mine : slot0.mine, np = slot ? slot1.np : slot0.np;
    const int head0 = slot ? slot1.head0 : slot0.head0;
    if (np == 0) continue;
    if (!mbar_wait_cluster(&recv_bar[slot], 0)) ran_out();
    if (bad) continue;
#pragma unroll 1
    for (int j = warp; j * np + mine < Cl::kUnits; j += kWarps) {
      const int un = j * np + mine;
      const float *src = recv + slot * Cl::kRecvFloats + j * np * Cl::kUnit;
      float4 s4[kMaxCluster];
      float so[kMaxCluster];
      float M = -INFINITY;
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r) {
        s4[r] = r < np ? *reinterpret_cast<const float4 *>(src + r * Cl::kUnit + 32)
                       : make_float4(-INFINITY, 0.f, 0.f, 0.f);
        so[r] = r < np ? src[r * Cl::kUnit + lane] : 0.f;
        M = fmaxf(M, s4[r].x);
      }
      float l = 0.f, u = 0.f, sg = 0.f, o = 0.f;
#pragma unroll
      for (int r = 0; r < kMaxCluster; ++r) {
        const float dm = fmaxf(s4[r].x - M, -1e30f);
        const float f = exp2f(dm);
        l += f * s4[r].y;
        u += f * (s4[r].z + dm * s4[r].y);
        sg += f * s4[r].w;
        o += f * so[r];
      }
      finish<T, D>(a, head0 + un % G, un / G * 32 + lane, un < G && lane == 0, M, l, u, sg, o);
    }
  }
  __syncwarp();
  if (stopped() & 2) {
    // A peer may still be about to send pieces into this CTA's shared memory (every CTA sends
    // them, late or not): it stays until every thread of the cluster has ended or come here.
    cluster_arrive();
    cluster_wait();
    linger();
  }
}

namespace {

constexpr int kMaxDev = 64;

template <typename T, int D, int G>
struct ClusterLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  ClusterLaunch(int clusters, int ctas, cudaStream_t s) {
    cfg.gridDim = clusters * ctas;
    cfg.blockDim = ClusterCfg<T, D, G>::kThreads;
    cfg.dynamicSmemBytes = ClusterCfg<T, D, G>::kSmem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
  }
};

// How many clusters of each size the current device holds at once, looked up once per device and
// kernel (a function of the kernel's shared memory alone).
template <typename T, int D, int G>
cudaError_t resident_clusters(int (&n)[kNumSizes]) {
  static std::atomic<int> known[kMaxDev][kNumSizes];  // 0: not looked up yet
  int dev = 0;
  LG_TRY(cudaGetDevice(&dev));
  for (int i = 0; i < kNumSizes; ++i) {
    n[i] = dev < kMaxDev ? known[dev][i].load(std::memory_order_relaxed) : 0;
    if (n[i] > 0) continue;
    auto kern = attend_cluster_kernel<T, D, G>;
    LG_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                ClusterCfg<T, D, G>::kSmem));
    ClusterLaunch<T, D, G> l(1, kSizes[i], nullptr);
    l.cfg.numAttrs = 1;
    LG_TRY(cudaOccupancyMaxActiveClusters(&n[i], kern, &l.cfg));
    if (n[i] < 1) n[i] = 1;
    if (dev < kMaxDev) known[dev][i].store(n[i], std::memory_order_relaxed);
  }
  return cudaSuccess;
}

template <typename T, int D, int G>
constexpr PassKind pass_kind() {
  return {Elem<T>::kDtype == LG_BF16, D, G, Pass<T, D, G>::kTile};
}

template <typename T, int D, int G>
cudaError_t launch_cluster_typed(AttendArgs &a, int64_t rows_total, bool *general,
                                 cudaStream_t s) {
  int resident[kNumSizes];
  LG_TRY((resident_clusters<T, D, G>(resident)));
  a.sms = resident[kNumSizes - 1];  // one CTA an SM
  const CallShape shape = call_shape(pass_kind<T, D, G>(), a.n_layers * a.batch * a.H_kv, a.max_len,
                                     a.chunk_rows, a.max_chunks, a.sms);
  const AttendChoice ch = attend_choose(
      shape, a.batch, fminf(1.f, (float)a.S_total / ((float)a.batch * (float)a.max_len)), resident);
  *general = ch.pass != kClusterPass;
  if (ch.pass == kGeneralPass) return cudaSuccess;
  if (ch.pass == kEitherPass) a.gate = a.counter;
  CUtensorMap mk, mv;
  if (!make_kv_map(&mk, a.K, Elem<T>::kDtype, D, rows_total, Pass<T, D, G>::kTile) ||
      !make_kv_map(&mv, a.V, Elem<T>::kDtype, D, rows_total, Pass<T, D, G>::kTile))
    return cudaErrorInvalidValue;
  auto kern = attend_cluster_kernel<T, D, G>;
  LG_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              ClusterCfg<T, D, G>::kSmem));
  ClusterLaunch<T, D, G> l(ch.clusters, ch.ctas, s);
  return cudaLaunchKernelEx(&l.cfg, kern, mk, mv, a, ch.ctas, ch.clusters, (int)rows_total);
}

template <typename T, int D>
cudaError_t launch_cluster_d(AttendArgs &a, int g, int64_t rows_total, bool *general,
                             cudaStream_t s) {
  switch (g) {
    case 1: return launch_cluster_typed<T, D, 1>(a, rows_total, general, s);
    case 2: return launch_cluster_typed<T, D, 2>(a, rows_total, general, s);
    case 3: return launch_cluster_typed<T, D, 3>(a, rows_total, general, s);
    case 4: return launch_cluster_typed<T, D, 4>(a, rows_total, general, s);
    case 5: return launch_cluster_typed<T, D, 5>(a, rows_total, general, s);
    case 6: return launch_cluster_typed<T, D, 6>(a, rows_total, general, s);
    case 7: return launch_cluster_typed<T, D, 7>(a, rows_total, general, s);
    case 8: return launch_cluster_typed<T, D, 8>(a, rows_total, general, s);
  }
  return cudaErrorInvalidValue;
}

// the pass over a cache of rows_total rows of T; *general set: the general pass is to be launched,
// alone, or after it with a.gate set
template <typename T>
cudaError_t launch_cluster(AttendArgs &a, int d, int g, int64_t rows_total, bool *general,
                           cudaStream_t s) {
  if (d == 128) return launch_cluster_d<T, 128>(a, g, rows_total, general, s);
  if (d == 64) return launch_cluster_d<T, 64>(a, g, rows_total, general, s);
  return cudaErrorInvalidValue;
}

}  // namespace

}  // namespace lg
