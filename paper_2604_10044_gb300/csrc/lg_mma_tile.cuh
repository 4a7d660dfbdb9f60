// Pieces shared by the two tensor-core attention passes (lg_attend_mma.cu: persistent CTAs over
// the whole call; lg_attend_cluster.cu: clusters for short calls): the tile layout, the tensor
// copies and matrix instructions, and one consumer warp's work on a tile.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "lg_common.cuh"
#include "lg_internal.h"

namespace lg {

constexpr int kTileRows = 128;              // rows per tile (TMA box height)
constexpr int kBoxBytes = kTileRows * 128;  // one box: 128 rows x 64 bf16
constexpr int kConsumerWarps = 4;
constexpr int kStagedSeqs = 256;     // lengths and offsets kept in shared memory up to this batch
constexpr int kL2KeepBytes = 32 << 20;  // K/V a short pass leaves in L2 at normal priority

template <int D>
struct MmaCfg {
  static constexpr int kHalves = D / 64;                      // boxes per row
  static constexpr int kStageBytes = 2 * kHalves * kBoxBytes;  // K and V
  static constexpr int kStages = D == 128 ? 3 : 6;
  static constexpr int kRingBytes = kStages * kStageBytes;
  // ticket buffers: room for one buffer of 8 heads; fewer heads fit more buffers
  static constexpr int kMergeBytes = kConsumerWarps * 8 * (D + 8) * 4;
  static constexpr int kQBytes = 8 * D * 2;  // a stage's query rows (up to 8 heads), bf16
  static constexpr int kSmem = kRingBytes + kMergeBytes + kStages * kQBytes + 1024;  // + slack
  static constexpr int kKSteps = D / 16;
};

// 2-D tensor copy of one box into shared memory, completing on `bar`, with an L2 eviction
// policy (createpolicy) for the lines it brings in.
__device__ __forceinline__ void tma_load_2d(void *smem_dst, const CUtensorMap *map, int x,
                                                 int y, uint64_t *bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(smem_addr(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_addr(bar)), "l"(policy)
      : "memory");
}

// the same box requested into L2 only: a hint, nothing is read from it
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap *map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y)
               : "memory");
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2,
                                        uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}

__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t &r0, uint32_t &r1,
                                              uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}

__device__ __forceinline__ void mma_bf16(float *d, uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm(  // not volatile: the compiler may place it among the loads of other fragments
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, "
      "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// the same into fresh sums
__device__ __forceinline__ void mma_bf16_zero(float *d, uint32_t a0, uint32_t a1, uint32_t a2,
                                              uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, "
      "{%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
  uint32_t d;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

// byte offset of 16-byte chunk c8 (0..7) of row r in a 128-byte-swizzled box
__device__ __forceinline__ uint32_t swz(int r, int c8) {
  return (uint32_t)(r * 128 + ((c8 ^ (r & 7)) << 4));
}

// One consumer warp's running sums over its rows (accumulator fragments of S^T and o^T: this
// thread holds heads 2 t4 and 2 t4 + 1, t4 = lane & 3, and of o the elements 16 eb + g (+8),
// g = lane >> 2): maxima in log2 units, normalisers, sum p (s - m), suffix mass.
template <int D>
struct WarpSums {
  float o[D / 16][4];
  float m2[2], l2[2], u2[2], sg2[2];

  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int eb = 0; eb < D / 16; ++eb) o[eb][0] = o[eb][1] = o[eb][2] = o[eb][3] = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      m2[h] = -INFINITY;
      l2[h] = u2[h] = sg2[h] = 0.f;
    }
  }

  // the scalars summed over the lanes of one t4 (their rows are disjoint)
  __device__ __forceinline__ void join_lanes() {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int off = 4; off <= 16; off <<= 1) {
        l2[h] += __shfl_xor_sync(0xffffffffu, l2[h], off);
        u2[h] += __shfl_xor_sync(0xffffffffu, u2[h], off);
        sg2[h] += __shfl_xor_sync(0xffffffffu, sg2[h], off);
      }
    }
  }

  // the warp's partial of G heads: o as [head][D + 4] (the padding spreads the stores over all
  // banks), {M, l, u, sigma} as [head][kStat] from sb on
  template <int G, int kStat>
  __device__ __forceinline__ void store(float *ob, float *sb, int lane) const {
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int h2 = 0; h2 < 2; ++h2) {
      const int h = 2 * t4 + h2;
      if (h < G) {
#pragma unroll
        for (int eb = 0; eb < D / 16; ++eb) {
          ob[h * (D + 4) + eb * 16 + g] = o[eb][h2];
          ob[h * (D + 4) + eb * 16 + g + 8] = o[eb][h2 + 2];
        }
        if (g == 0)
          *reinterpret_cast<float4 *>(sb + h * kStat) = make_float4(m2[h2], l2[h2], u2[h2], sg2[h2]);
      }
    }
  }
};

// B fragments of q^T: head g (zero for padded heads), d = 16 ks + 2 t4 (+1, +8, +9)
template <int D, int G>
__device__ __forceinline__ void load_q(uint32_t (&qf)[D / 16][2], const unsigned char *qrows,
                                       int lane) {
  const int g = lane >> 2, t4 = lane & 3;
  const uint32_t *qp = reinterpret_cast<const uint32_t *>(qrows) + g * (D / 2);
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks) {
    qf[ks][0] = g < G ? qp[ks * 8 + t4] : 0u;
    qf[ks][1] = g < G ? qp[ks * 8 + 4 + t4] : 0u;
  }
}

// One consumer warp's MB blocks of 16 rows of a tile in `stage` (K boxes, then V boxes): logits,
// online softmax, sums and o^T.  tile_rows: rows of the tile in use; rows from `suffix` on (tile row
// numbers) count toward the suffix mass; logits: nullable, the tile's first row [rows][G].
// kFresh: a block's products go into sums of their own, which are then added to o.  The matrix
// unit truncates where an addition rounds, so a chain of its additions falls short in proportion
// to its length: with a segment's 342 blocks in one chain (2 sequences of 131071 rows, 8 heads a
// group, clusters of 6) the output was 1.28e-5 of its norm off the 64-bit value before its rounding
// to bf16, with this 2.36e-6; the persistent pass, whose chunks of 8 tiles keep the chains short,
// has 2.40e-6 there (most of it P's two bf16 parts).  The additions follow all of a block's products,
// so that none waits for its own (added after every four fragments: 18.6 us below).  It costs nothing
// at one tile a CTA, 0 to 1.5 % of most calls and 2.5 % where a CTA's own work bounds the call (1
// sequence of 16384 rows, 4 heads: 17.9 -> 18.3 us); flushes to shared memory every 16 blocks cost
// more (the long call above 157.0 -> 159.5 us, against 156.9).
template <int D, int G, int MB, bool kFresh>
__device__ __forceinline__ void tile_update(WarpSums<D> &acc, const uint32_t (&qf)[D / 16][2],
                                            unsigned char *stage, int tile_rows, int suffix,
                                            float *logits, float qscale, int warp, int lane) {
  using C = MmaCfg<D>;
  const int g = lane >> 2, t4 = lane & 3;
  const int mrow = lane & 7, msel = lane >> 3;  // ldmatrix: row within 8x8, matrix index
  float (&o)[D / 16][4] = acc.o;
  float (&m2)[2] = acc.m2, (&l2)[2] = acc.l2, (&u2)[2] = acc.u2, (&sg2)[2] = acc.sg2;
  const uint32_t kbase = smem_addr(stage);
  const uint32_t vbase = kbase + C::kHalves * kBoxBytes;
  constexpr int kRows = 16 * MB;
  const int r_w = warp * kRows;  // this warp's first row in the tile
  if (tile_rows < r_w + kRows) {
    // ragged tail: zero the V rows past the end so that 0 * stale stays 0
    for (int idx = lane; idx < kRows * C::kHalves * 8; idx += 32) {
      const int rr = r_w + idx / (C::kHalves * 8);
      const int hc = idx % (C::kHalves * 8);
      if (rr >= tile_rows)
        *reinterpret_cast<uint4 *>(stage + (C::kHalves + hc / 8) * kBoxBytes + rr * 128 +
                                   (hc % 8) * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncwarp();
  }

  // S^T for the warp's 16-row blocks (two accumulators a block: half the dependent chain)
  float s[MB][4], s1[MB][4];
#pragma unroll
  for (int mb = 0; mb < MB; ++mb) {
#pragma unroll
    for (int j = 0; j < 4; ++j) s[mb][j] = s1[mb][j] = 0.f;
    const int r = r_w + mb * 16 + (msel & 1) * 8 + mrow;
    uint32_t ka[C::kKSteps][4];
#pragma unroll
    for (int ks = 0; ks < C::kKSteps; ++ks)
      ldsm_x4(kbase + (ks >> 2) * kBoxBytes + swz(r, (ks & 3) * 2 + (msel >> 1)), ka[ks][0],
              ka[ks][1], ka[ks][2], ka[ks][3]);
#pragma unroll
    for (int ks = 0; ks < C::kKSteps; ks += 2) {
      mma_bf16(s[mb], ka[ks][0], ka[ks][1], ka[ks][2], ka[ks][3], qf[ks][0], qf[ks][1]);
      mma_bf16(s1[mb], ka[ks + 1][0], ka[ks + 1][1], ka[ks + 1][2], ka[ks + 1][3], qf[ks + 1][0],
               qf[ks + 1][1]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) s[mb][j] += s1[mb][j];
  }
  // scale to log2 units, mask rows past the end; tile max per head (heads 2 t4, 2 t4 + 1)
  float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
  for (int mb = 0; mb < MB; ++mb)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int rl = r_w + mb * 16 + g + (j >> 1) * 8;  // row within the tile
      const bool valid = rl < tile_rows;
      s[mb][j] = valid ? s[mb][j] * qscale : -INFINITY;
      mx[j & 1] = fmaxf(mx[j & 1], s[mb][j]);
    }
  // (a lane's own maxima tell whether any head's rises; only then are they joined)
  const bool raise = mx[0] > m2[0] || mx[1] > m2[1];
  if (__any_sync(0xffffffffu, raise)) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 4));
      mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 8));
      mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 16));
    }
    float corr[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float mn = fmaxf(m2[h], mx[h]);
      corr[h] = mn == m2[h] ? 1.f : exp2f(m2[h] - mn);
      u2[h] = l2[h] > 0.f ? corr[h] * (u2[h] + (m2[h] - mn) * l2[h]) : 0.f;
      l2[h] *= corr[h];
      sg2[h] *= corr[h];
      m2[h] = mn;
    }
#pragma unroll
    for (int eb = 0; eb < C::kKSteps; ++eb) {
      o[eb][0] *= corr[0];
      o[eb][1] *= corr[1];
      o[eb][2] *= corr[0];
      o[eb][3] *= corr[1];
    }
  }
  // probabilities, sums, and P^T fragments
  uint32_t pb[MB][2], pl[MB][2];
#pragma unroll
  for (int mb = 0; mb < MB; ++mb) {
    float p[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int h = j & 1;
      const int rl = r_w + mb * 16 + g + (j >> 1) * 8;
      const bool valid = rl < tile_rows;
      p[j] = valid ? exp2f(s[mb][j] - m2[h]) : 0.f;
      if (valid) {
        l2[h] += p[j];
        u2[h] += p[j] * (s[mb][j] - m2[h]);
        if (rl >= suffix) sg2[h] += p[j];
      }
    }
    if (logits) {
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int rl = r_w + mb * 16 + g + half * 8;
        if (rl < tile_rows) {
          float *dst = logits + (int64_t)rl * G;
          if (G % 2 == 0) {
            // heads 2 t4 and 2 t4 + 1 side by side: one 8-byte store (rows of an even G
            // start 8-byte aligned)
            if (2 * t4 < G)
              *reinterpret_cast<float2 *>(dst + 2 * t4) =
                  make_float2(s[mb][half * 2], s[mb][half * 2 + 1]);
          } else {
            if (2 * t4 < G) dst[2 * t4] = s[mb][half * 2];
            if (2 * t4 + 1 < G) dst[2 * t4 + 1] = s[mb][half * 2 + 1];
          }
        }
      }
    }
    // P = hi + lo, both bf16: the P.V product keeps ~16 mantissa bits of P
    const uint32_t h01 = pack_bf16(p[0], p[1]), h23 = pack_bf16(p[2], p[3]);
    const float2 f01 = bf16x2_to_float2(h01), f23 = bf16x2_to_float2(h23);
    pb[mb][0] = movmatrix_trans(h01);  // rows 0-7 of the block
    pb[mb][1] = movmatrix_trans(h23);  // rows 8-15
    pl[mb][0] = movmatrix_trans(pack_bf16(p[0] - f01.x, p[1] - f01.y));
    pl[mb][1] = movmatrix_trans(pack_bf16(p[2] - f23.x, p[3] - f23.y));
  }
  // o^T += V^T P^T (four fragments at a time: their loads, the products with P's high parts, then
  // with its low parts, so that no product waits for the one before it)
#pragma unroll
  for (int mb = 0; mb < MB; ++mb) {
    const int r = r_w + mb * 16 + (msel >> 1) * 8 + mrow;
    float fresh[C::kKSteps][4];
#pragma unroll
    for (int e0 = 0; e0 < C::kKSteps; e0 += 4) {
      uint32_t va[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        ldsm_x4_trans(vbase + (e0 >> 2) * kBoxBytes + swz(r, j * 2 + (msel & 1)), va[j][0],
                      va[j][1], va[j][2], va[j][3]);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (kFresh)
          mma_bf16_zero(fresh[e0 + j], va[j][0], va[j][1], va[j][2], va[j][3], pb[mb][0], pb[mb][1]);
        else
          mma_bf16(o[e0 + j], va[j][0], va[j][1], va[j][2], va[j][3], pb[mb][0], pb[mb][1]);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        mma_bf16(kFresh ? fresh[e0 + j] : o[e0 + j], va[j][0], va[j][1], va[j][2], va[j][3],
                 pl[mb][0], pl[mb][1]);
    }
    if (kFresh) {
#pragma unroll
      for (int eb = 0; eb < C::kKSteps; ++eb)
#pragma unroll
        for (int k = 0; k < 4; ++k) o[eb][k] += fresh[eb][k];
    }
  }
  __syncwarp();
  if (tile_rows < r_w + kRows) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// tensor map of one cache tensor [rows][d] of a dtype: boxes of box_rows rows x 128 bytes
bool make_kv_map(CUtensorMap *m, const void *base, int dtype, int d, int64_t rows, int box_rows);

}  // namespace lg
