// The cluster pass (lg_attend_cluster.cuh) over bf16 caches, on tensor cores, and the rule that
// sends a call to it.
#include "lg_attend_cluster.cuh"

namespace lg {

namespace {

template <int D, int G>
struct Pass<__nv_bfloat16, D, G> {
  static constexpr int kTile = kTileRows, kBoxCols = 64, kBoxes = D / 64;
  static constexpr int kStages = MmaCfg<D>::kStages;
  // eight consumer warps of 16 rows of a tile, or four of 32: at one tile a CTA the pass waits
  // for a warp's chain of dependent instructions, which eight warps shorten (G > 4 lacks the
  // shared memory for eight partials)
  static constexpr int kWarps = G <= 4 ? 8 : 4;
  static constexpr int kBlocks = kTile / 16 / kWarps;  // 16-row blocks of a warp
  static constexpr int kFoldUnits = 1;
  static constexpr bool kEarlyUnits = true;
  // No flush: o takes one rounded addition per 16 rows (kFresh in lg_mma_tile.cuh), l, u and sigma
  // one per row of a lane (two rows a block and head), so that 2 sequences of 131071 rows have l
  // 2.2e-7 off its 64-bit value where the persistent pass has 3.0e-7.
  static constexpr int kFlushTiles = 0;

  WarpSums<D> acc;
  uint32_t qf[D / 16][2];

  __device__ __forceinline__ void begin(const unsigned char *q, bool, float, int lane) {
    acc.reset();
    load_q<D, G>(qf, q, lane);
  }
  __device__ __forceinline__ void update(unsigned char *stage, int tile_rows, int suffix,
                                         float *logits, float qscale, int warp, int lane) {
    tile_update<D, G, kBlocks, true>(acc, qf, stage, tile_rows, suffix, logits, qscale, warp, lane);
  }
  __device__ __forceinline__ void join() { acc.join_lanes(); }
  __device__ __forceinline__ void store(float *rows, bool, int lane) {
    acc.template store<G, D + 4>(rows, rows + D, lane);
  }
};

}  // namespace

// The limits of its tables and integers: the batch (two sequences a lane), the groups (a group
// number times a cluster number in a float's 24 bits) and the tiles (a cluster's tiles times a CTA
// number in 24 bits).  Within them attend_choose (lg_attend_rule.cuh) compares it with the general
// pass.
bool attend_cluster_takes(const AttendArgs &a, int tile_rows, int64_t rows_total) {
  const int64_t groups = (int64_t)a.n_layers * a.batch * a.H_kv;
  const int64_t tiles = groups * ((a.max_len + tile_rows - 1) / tile_rows);
  return a.batch <= kClusterSeqs && groups <= 1 << 16 && tiles < 1 << 20 &&
         rows_total < (int64_t)1 << 31;
}

cudaError_t launch_attend_cluster(AttendArgs &a, int d, int g, int64_t rows_total,
                                  bool *general, cudaStream_t s) {
  return launch_cluster<__nv_bfloat16>(a, d, g, rows_total, general, s);
}

}  // namespace lg
