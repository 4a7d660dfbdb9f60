// The cluster pass (lg_attend_cluster.cuh) over fp32 caches, in packed fp32 FMAs.
//
// A row is spread over kLpr lanes of 4 to 16 elements each, kRpw rows a warp step: the query
// slices and the output stay in registers (fewer elements a lane for more heads), so shared
// memory is read for K and V only.  A transposed butterfly leaves each lane with the full logit
// of one head, that lane runs the online softmax for its head and row group, and the
// probabilities are passed back by shuffles.  Up to 4 heads the memory bounds a call; at 5 to 8
// the chains of dependent shuffles and FMAs do, of which two to four rows run side by side.
// GB300, one layer (append and attention), 268 MB, 4 sequences of 8191 rows, 8 kv-heads of 128,
// against the chunk kernel with its separate combine: 1 head a group 80.8 -> 41.5 us, 4 heads
// 91.1 -> 44.9, 8 heads 108.0 -> 72.5 (77.7 with the chunk kernel launched after it, as lengths in
// such slots can make that the faster).  Not kept: a lane a row with the query rows broadcast from
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
  static constexpr bool kEarlyUnits = false;  // (six registers that the tiles' loop lacks)
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
  // A flush every so many tiles (32 of a lane's rows) adds the sums to the warp's partial in shared
  // memory, which keeps the chains of dependent roundings short: a lane takes hundreds of rows of a
  // long call.  Distance of the output from 64 bits (2-norm, normal rows; the chunk kernel /
  // without flushes / with): 4 sequences of 8191, 4 heads 2.65e-7 / 2.82e-7 / 2.16e-7, one of
  // 131071, 8 heads 4.4e-7 / 8.4e-7 / 2.6e-7.  It cost 2 % of the time when it came (44.4 -> 45.4 us, above).
  static constexpr int kFlushTiles = 32 * kRpw / kRows;
  static_assert(kGP <= kLpr && kRows % (kSteps * kRpw) == 0, "lanes for the heads, whole steps");

  static constexpr int kKept = D / 64;  // pairs of a head that a lane keeps when they are joined
  struct __align__(8 * kKept) Pairs {
    float2 p[kKept];
  };

  float2 q[G][kCh][2], o[G][2 * kCh];
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

  __device__ __forceinline__ void begin(const unsigned char *qrows, bool first, float qscale,
                                        int lane) {
    const float4 *q4 = reinterpret_cast<const float4 *>(qrows);
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int j = 0; j < kCh; ++j) {
        const float4 v = q4[g * (D / 4) + chunk(j, lane)];
        q[g][j][0] = make_float2(v.x * qscale, v.y * qscale);
        q[g][j][1] = make_float2(v.z * qscale, v.w * qscale);
        o[g][2 * j] = o[g][2 * j + 1] = make_float2(0.f, 0.f);
      }
    if (first) m = -INFINITY;  // else it runs on
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
            o[g][2 * j] = __fmul2_rn(o[g][2 * j], c2);
            o[g][2 * j + 1] = __fmul2_rn(o[g][2 * j + 1], c2);
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
            o[g][2 * j] = __ffma2_rn(p2, make_float2(v[j].x, v[j].y), o[g][2 * j]);
            o[g][2 * j + 1] = __ffma2_rn(p2, make_float2(v[j].z, v[j].w), o[g][2 * j + 1]);
          }
        }
      }
    }
    __syncwarp();
  }

  // The row groups' sums, against the warp's maximum of each head: l, u and sg on every lane, of o
  // the pairs that the lane keeps (o[g][0 .. kKept)).
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
      float2(&v)[2 * kCh] = o[g], sum[kCh];
#pragma unroll
      for (int c = 0; c < 2 * kCh; ++c) v[c] = __fmul2_rn(v[c], make_float2(fg, fg));
      // each level, a lane hands half of its pairs to the other row group's lane
#pragma unroll
      for (int x = kLpr, half = kCh; x < 32; x <<= 1, half >>= 1) {
        const bool up = lane & x;
        // the neighbour row of four-lane rows holds its chunks in the other order
        const int flip = kLpr == 4 && x == kLpr ? 2 : 0;
#pragma unroll
        for (int c = 0; c < kCh; ++c)
          if (c < half) {
            const float2 send = up ? v[c ^ flip] : v[(c ^ flip) + half];
            const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, send.x, x),
                                           __shfl_xor_sync(0xffffffffu, send.y, x));
            sum[c] = __fadd2_rn(up ? v[c + half] : v[c], got);
          }
#pragma unroll
        for (int c = 0; c < kCh; ++c)
          if (c < half) v[c] = sum[c];
      }
    }
  }

  // the joined sums to the warp's partial, or added to the sums of earlier tiles there
  __device__ __forceinline__ void store(float *rows, bool add, int lane) {
    const int gbase = lane - lane % kLpr, hd = lane % kLpr / kDup;
    float f = 0.f;
    if (add && hd < G) {
      const float4 h = *reinterpret_cast<const float4 *>(rows + hd * (D + 4) + D);
      const float dm = fmaxf(h.x - m, -1e30f);  // the maximum runs on: h.x <= m
      f = exp2f(dm);
      l += f * h.y;
      u += f * (h.z + dm * h.y);
      sg += f * h.w;
    }
    // where this lane's pairs lie
    int c = 0;
#pragma unroll
    for (int x = kLpr, half = kCh; x < 32; x <<= 1, half >>= 1) c += lane & x ? half : 0;
    float *at = rows + 4 * chunk(c >> 1, lane) + 2 * (c & 1);
#pragma unroll
    for (int g = 0; g < G; ++g, at += D + 4) {
      const float fg = __shfl_sync(0xffffffffu, f, gbase + g * kDup);
      float2 v[kKept];
#pragma unroll
      for (int i = 0; i < kKept; ++i) v[i] = o[g][i];
      if (add) {
        const Pairs h = *reinterpret_cast<const Pairs *>(at);
#pragma unroll
        for (int i = 0; i < kKept; ++i) v[i] = __ffma2_rn(make_float2(fg, fg), h.p[i], v[i]);
      }
      Pairs w;
#pragma unroll
      for (int i = 0; i < kKept; ++i) w.p[i] = v[i];
      *reinterpret_cast<Pairs *>(at) = w;
    }
    __syncwarp();  // every lane has read its head's earlier sums
    if (lane < kLpr && lane % kDup == 0 && hd < G)
      *reinterpret_cast<float4 *>(rows + hd * (D + 4) + D) = make_float4(m, l, u, sg);
    __syncwarp();
  }
};

}  // namespace

int cluster_f32_tile_rows() { return kF32TileMin; }

cudaError_t launch_attend_cluster_f32(AttendArgs &a, int d, int g, int64_t rows_total,
                                      bool *general, cudaStream_t s) {
  return launch_cluster<float>(a, d, g, rows_total, general, s);
}

}  // namespace lg
