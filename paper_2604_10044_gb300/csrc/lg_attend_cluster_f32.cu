// The cluster pass (lg_attend_cluster.cuh) over fp32 caches, in packed fp32 FMAs.
//
// A row is spread over kLpr lanes of 4 to 16 elements each, kRpw rows a warp step: the query
// slices and the output stay in registers (fewer elements a lane for more heads), so shared
// memory is read for K and V only.  A transposed butterfly leaves each lane with the full logit
// of one head, that lane runs the online softmax for its head and row group, and the
// probabilities are passed back by shuffles.  Up to 4 heads the memory bounds a call; at 5 to 8
// the chains of dependent shuffles and FMAs do, of which two to four rows run side by side.
// GB300, one layer (append and attention), 268 MB, 4 sequences of 8191 rows, 8 kv-heads of 128,
// against the chunk kernel with its separate combine: 1 head a group 80.8 -> 43.6 us, 4 heads
// 91.1 -> 46.8, 8 heads 108.0 -> 76.6.  Not kept: a lane a row with the query rows broadcast from
// shared memory (its datapath moves 512 bytes for a broadcast too: 54 and 80 us at 4 and 8 heads).
#include "lg_attend_cluster.cuh"

namespace lg {

namespace {

constexpr int kF32TileMin = 32;

template <int D, int G>
struct Pass<float, D, G> {
  // (64-row tiles of 5 to 8 heads leave no room for a third stage)
  static constexpr int kTile = G <= 4 ? 64 : kF32TileMin, kBoxCols = 32, kBoxes = D / 32;
  static constexpr int kStages = (G <= 4 ? 3 : 5) * 128 / D;
  static constexpr int kWarps = 8;
  static constexpr int kFoldUnits = 4;
  static constexpr float kTileUs = (G <= 4 ? 1.f : 1.2f) * D / 128.f;
  static constexpr int kBox = kTile * 128;       // bytes of a box
  static constexpr int kEpl = G <= 2 ? 16 : (G <= 4 ? 8 : 4);  // elements of a lane
  static constexpr int kCh = kEpl / 4;           // 16-byte chunks of a lane
  static constexpr int kLpr = D / kEpl;          // lanes of a row: 4 to 32
  static constexpr int kRpw = 32 / kLpr;         // rows of a warp step
  static constexpr int kRows = kTile / kWarps;   // a warp's rows of a tile
  // warp steps done together, so that one row's chain of shuffles overlaps another's
  static constexpr int kMaxSteps = G <= 4 ? 2 : 4;
  static constexpr int kSteps = kRows / kRpw < kMaxSteps ? kRows / kRpw : kMaxSteps;
  static constexpr int kGP = pow2_ceil(G);
  static constexpr int kDup = kLpr / kGP;        // lanes that hold the same head's logit
  static_assert(kGP <= kLpr && kRows % (kSteps * kRpw) == 0, "lanes for the heads, whole steps");

  float2 q[G][kCh][2], o[G][kCh][2];
  float m, l, u, sg;  // of head (lane % kLpr) / kDup over this lane's row group

  // chunk j of this lane, a multiple of 4 elements: the lanes of a row side by side, so that
  // eight lanes read 128 bytes of different banks (with four lanes a row, odd rows take the
  // other half of a box first)
  __device__ __forceinline__ static int chunk(int j, int lane) {
    const int li = lane % kLpr;
    return kLpr == 4 ? (j ^ ((lane / kLpr) & 1)) * kLpr + li : j * kLpr + li;
  }
  __device__ __forceinline__ static float4 load(const unsigned char *boxes, int row, int ch) {
    return *reinterpret_cast<const float4 *>(boxes + (ch >> 3) * kBox + row * 128 +
                                             (((ch & 7) ^ (row & 7)) << 4));
  }

  __device__ __forceinline__ void begin(const unsigned char *qrows, float qscale, int lane) {
    const float4 *q4 = reinterpret_cast<const float4 *>(qrows);
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int j = 0; j < kCh; ++j) {
        const float4 v = q4[g * (D / 4) + chunk(j, lane)];
        q[g][j][0] = make_float2(v.x * qscale, v.y * qscale);
        q[g][j][1] = make_float2(v.z * qscale, v.w * qscale);
        o[g][j][0] = o[g][j][1] = make_float2(0.f, 0.f);
      }
    m = -INFINITY;
    l = u = sg = 0.f;
  }

  __device__ __forceinline__ void update(unsigned char *stage, int tile_rows, int suffix,
                                         float *logits, float, int warp, int lane) {
    const int li = lane % kLpr, hd = li / kDup, gbase = lane - li;
#pragma unroll
    for (int s0 = 0; s0 < kRows; s0 += kSteps * kRpw) {
      int r[kSteps];  // this lane's rows in the tile
      bool live[kSteps];
      float part[kSteps][kGP];
#pragma unroll
      for (int i = 0; i < kSteps; ++i) {
        r[i] = warp * kRows + s0 + i * kRpw + lane / kLpr;
        live[i] = r[i] < tile_rows && hd < G;
        float4 k[kCh];
#pragma unroll
        for (int j = 0; j < kCh; ++j) k[j] = load(stage, r[i], chunk(j, lane));
#pragma unroll
        for (int g = 0; g < kGP; ++g) {
          float2 acc = make_float2(0.f, 0.f);
          if (g < G) {
#pragma unroll
            for (int j = 0; j < kCh; ++j) {
              acc = __ffma2_rn(q[g][j][0], make_float2(k[j].x, k[j].y), acc);
              acc = __ffma2_rn(q[g][j][1], make_float2(k[j].z, k[j].w), acc);
            }
          }
          part[i][g] = acc.x + acc.y;
        }
      }
      HeadReduce<kGP, kLpr / 2>::run_all(part, lane);
      // part[i][0]: the logit of head hd for row r[i], log2 units
      float mn = m;
#pragma unroll
      for (int i = 0; i < kSteps; ++i)
        if (live[i]) mn = fmaxf(mn, part[i][0]);
      if (__any_sync(0xffffffffu, mn > m)) {
        const float corr = mn == m ? 1.f : exp2f(m - mn);  // -inf -> 0
        u = l > 0.f ? corr * (u + (m - mn) * l) : 0.f;
        l *= corr;
        sg *= corr;
        m = mn;
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const float cg = __shfl_sync(0xffffffffu, corr, gbase + g * kDup);
          const float2 c2 = make_float2(cg, cg);
#pragma unroll
          for (int j = 0; j < kCh; ++j) {
            o[g][j][0] = __fmul2_rn(o[g][j][0], c2);
            o[g][j][1] = __fmul2_rn(o[g][j][1], c2);
          }
        }
      }
      // rows past the end hold stale shared memory: they must not touch the sums
      float p[kSteps];
#pragma unroll
      for (int i = 0; i < kSteps; ++i) {
        const float s = part[i][0];
        p[i] = live[i] ? exp2f(s - m) : 0.f;
        if (live[i]) {
          l += p[i];
          u += p[i] * (s - m);
          if (r[i] >= suffix) sg += p[i];
          if (logits && li % kDup == 0) logits[(int64_t)r[i] * G + hd] = s;
        }
      }
#pragma unroll
      for (int i = 0; i < kSteps; ++i) {
        float4 v[kCh];
#pragma unroll
        for (int j = 0; j < kCh; ++j)
          v[j] = r[i] < tile_rows ? load(stage + kBoxes * kBox, r[i], chunk(j, lane))
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const float pg = __shfl_sync(0xffffffffu, p[i], gbase + g * kDup);
          const float2 p2 = make_float2(pg, pg);
#pragma unroll
          for (int j = 0; j < kCh; ++j) {
            o[g][j][0] = __ffma2_rn(p2, make_float2(v[j].x, v[j].y), o[g][j][0]);
            o[g][j][1] = __ffma2_rn(p2, make_float2(v[j].z, v[j].w), o[g][j][1]);
          }
        }
      }
    }
    __syncwarp();
  }

  // the row groups' sums on every lane, against the warp's maximum of each head
  __device__ __forceinline__ void join() {
    const int lane = threadIdx.x & 31, gbase = lane - lane % kLpr;
    float M = m;
#pragma unroll
    for (int x = kLpr; x < 32; x <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, x));
    // (a group that saw no row has l = u = 0 and no weight)
    const float dm = fmaxf(m - M, -1e30f), f = exp2f(dm);
    u = f * (u + dm * l);
    l *= f;
    sg *= f;
    m = M;
#pragma unroll
    for (int x = kLpr; x < 32; x <<= 1) {
      l += __shfl_xor_sync(0xffffffffu, l, x);
      u += __shfl_xor_sync(0xffffffffu, u, x);
      sg += __shfl_xor_sync(0xffffffffu, sg, x);
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float fg = __shfl_sync(0xffffffffu, f, gbase + g * kDup);
#pragma unroll
      for (int j = 0; j < kCh; ++j)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          o[g][j][k].x *= fg;
          o[g][j][k].y *= fg;
        }
#pragma unroll
      for (int x = kLpr; x < 32; x <<= 1) {
        // the neighbour row of four-lane rows holds its chunks in the other order
        const int flip = kLpr == 4 && x == kLpr ? 1 : 0;
        float2 t[kCh][2];
#pragma unroll
        for (int j = 0; j < kCh; ++j)
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            t[j][k].x = __shfl_xor_sync(0xffffffffu, o[g][j ^ flip][k].x, x);
            t[j][k].y = __shfl_xor_sync(0xffffffffu, o[g][j ^ flip][k].y, x);
          }
#pragma unroll
        for (int j = 0; j < kCh; ++j)
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            o[g][j][k].x += t[j][k].x;
            o[g][j][k].y += t[j][k].y;
          }
      }
    }
  }

  __device__ __forceinline__ void store(float *rows, int lane) {
    if (lane < kLpr) {
#pragma unroll
      for (int g = 0; g < G; ++g)
#pragma unroll
        for (int j = 0; j < kCh; ++j)
          *reinterpret_cast<float4 *>(rows + g * (D + 4) + 4 * chunk(j, lane)) =
              make_float4(o[g][j][0].x, o[g][j][0].y, o[g][j][1].x, o[g][j][1].y);
      const int hd = lane / kDup;
      if (lane % kDup == 0 && hd < G)
        *reinterpret_cast<float4 *>(rows + hd * (D + 4) + D) = make_float4(m, l, u, sg);
    }
  }
};

}  // namespace

int cluster_f32_tile_rows() { return kF32TileMin; }

cudaError_t launch_attend_cluster_f32(const AttendArgs &a, int d, int g, int64_t rows_total,
                                      cudaStream_t s) {
  return launch_cluster<float>(a, d, g, rows_total, s);
}

}  // namespace lg
