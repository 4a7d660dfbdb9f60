// Which pass a call of lg_decode_attend takes: estimates of the cluster pass's time
// (lg_attend_cluster.cuh) and of the general passes' (lg_attend_mma.cu for bf16 caches, the chunk
// kernel of lg_attend.cu for fp32 ones).
//
// The host sees sizes only: max_len bounds the lengths, and S_total says how many rows the cache
// has for them.  Sequences kept in equal slots look like equal lengths, whatever they are.  Most
// calls lose little by clusters for any lengths; for the others the host launches both, and the
// cluster pass, which reads the lengths anyway, decides (attend_choose below).  Eight slots of
// 131072 rows, 2 kv-heads, 4 heads a group, bf16, us a call (the general pass alone / clusters alone
// / both): all full 177 / 153 / 157, one full and seven of 300 rows 57 / 121 / 60; 16 slots of 56396
// rows, 1 head, fp32, the same 303 / 254 / 260 and 76 / 138 / 83.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define LG_HD __host__ __device__ __forceinline__
#else
#define LG_HD inline
#endif

namespace lg {

constexpr int kMaxCluster = 8;             // CTAs of a cluster at most (portable)
constexpr int kSizes[] = {8, 6, 4, 2, 1};  // cluster sizes used (5 and 7 fit no better than 4 and 6
                                           // beside the GPU's clusters of SMs)
constexpr int kNumSizes = sizeof(kSizes) / sizeof(kSizes[0]);

// What the estimates need to know of a kernel.
struct PassKind {
  bool bf16;
  int d, g;       // head size, heads of a group
  int tile_rows;  // the cluster pass's tile
  LG_HD float tile_bytes() const { return (float)(2 * tile_rows * d * (bf16 ? 2 : 4)); }
  // one CTA's time for a tile
  LG_HD float tile_us() const {
    if (bf16) return d == 128 ? (g <= 4 ? 0.66f : 0.76f) : (g <= 4 ? 0.47f : 0.63f);
    return d == 128 ? (g <= 2 ? 0.66f : g <= 4 ? 1.13f : 1.07f)
                    : (g <= 2 ? 0.38f : g <= 4 ? 0.62f : 0.69f);
  }
  // and for a segment's fold (short groups: the fold's latency hides behind the next one's copies)
  LG_HD float segment_us(int tiles) const {
    return tiles < 8 || !bf16 ? 1.f : 0.4f + 0.35f * (float)g;
  }
};

// One call: its (layer, sequence, kv-head) groups, the rows and tiles of a longest one, the chunk
// kernel's rows a chunk, the chunks a group that the workspace holds, the GPU's SMs.
struct CallShape {
  PassKind kind;
  int groups, rows, tiles, chunk_rows, max_chunks, sms;
  // HBM's time for so many tiles (7.3 TB/s, as long passes read)
  LG_HD float mem_us(float n_tiles) const { return n_tiles * kind.tile_bytes() / 7.3e6f; }
};
LG_HD CallShape call_shape(const PassKind &kind, int groups, int rows, int chunk_rows,
                           int max_chunks, int sms) {
  const int tiles = (rows + kind.tile_rows - 1) / kind.tile_rows;
  return {kind, groups, rows, tiles, chunk_rows, max_chunks, sms};
}

constexpr float kCallUs = 5.f;

// The cluster pass with K clusters of c CTAs.  Equal lengths: each takes groups / K groups and then
// groups mod K of them one more; either phase is bound by the memory or by the CTAs.  Ragged ones,
// of `mean` of the longest on average: the clusters' runs are even but for a part of a longest group
// on one cluster, and no group has more than c CTAs.  Larger clusters stream a little better (about
// a percent per halving on passes of half a millisecond).
LG_HD float cluster_us(const CallShape &s, int c, int k, bool equal, float mean) {
  const float tile_us = s.kind.tile_us(), seg_us = s.kind.segment_us(s.tiles);
  const float cta = (float)s.tiles / (float)c * tile_us;  // a longest group's tiles on one of its CTAs
  float us;
  if (equal) {
    const int q = s.groups / k, r = s.groups % k;
    us = fmaxf(s.mem_us((float)k * (float)q * (float)s.tiles),
               (float)q * cta + seg_us * (float)(q - 1) / (float)c);
    if (r) us += fmaxf(s.mem_us((float)r * (float)s.tiles), cta + seg_us / (float)c);
  } else {
    const float total = mean * (float)s.groups * (float)s.tiles;
    const float even = (total * tile_us + (float)s.groups * seg_us) / (float)(k * c);
    us = fmaxf(fmaxf(s.mem_us(total), even) + 0.35f * cta, cta);
  }
  // a CTA's last segments: where it has several tiles of a group, of which it shares some
  if (s.tiles >= 8) us += seg_us * (c > 1 ? 2.f : 1.f);
  return kCallUs + (1.f + 0.0125f * log2f((float)kMaxCluster / (float)c)) * us;
}

// The general pass, for lengths of `mean` of the longest on average.  bf16: the persistent pass's
// chunks are about an eighth of a CTA's share, 3 to 16 a CTA, no more than max_chunks a group (what
// the workspace holds); one warp merges a group's, head by head, and those past a group's length are
// claimed all the same.  fp32: the chunk kernel (more arithmetic the more heads; one CTA reads its
// chunk at 25 GB/s) and its combine, which walks a group's chunks one by one (their partials still
// in L2 after a short pass).  Over 450 calls of long groups with any lengths in equal slots (one or
// more full ones among short ones, falling, log-uniform and equal ones) it is off by 10 % in bf16
// and 13 % in fp32 (standard deviations), the cluster pass's estimate by 8 and 10 %.
LG_HD float general_us(const CallShape &s, float mean, int max_chunks) {
  const float g = (float)s.kind.g, total = mean * (float)s.groups * (float)s.tiles;
  const float mem = s.mem_us(total);
  if (s.kind.bf16) {
    const float share = total / (float)s.sms;
    const float chunk = fmaxf(fmaxf(share / fminf(16.f, fmaxf(3.f, share / 8.f)), 1.f),
                              (float)s.tiles / (float)max_chunks);
    const float per_group = (float)s.tiles / chunk;
    return 12.f + 1.03f * mem + 0.07f * g * per_group +
           0.7f / (float)s.sms * (1.f - mean) * (float)s.groups * per_group;
  }
  const int chunk = s.chunk_rows < s.rows ? s.chunk_rows : s.rows;
  return 12.f + (8.f + 3.f * g) * fminf(1.f, mem / 30.f) +
         fmaxf((1.03f + 0.045f * g) * mem, (float)(chunk * s.kind.d) * (8.f * 4e-5f)) +
         (mem < 15.f ? 0.23f : 0.42f) * (float)s.rows / (float)s.chunk_rows;
}

// By how much the general pass is the faster one (us) for the lengths of a call: rows of the longest
// sequence in s, tiles of all of them (of one kv-head of one layer), and whether they all have as
// many tiles.
LG_HD float general_gains_us(const CallShape &s, int batch, int tiles, bool equal, int c, int k) {
  if (s.tiles == 0) return 0.f;
  const float mean = (float)tiles / ((float)batch * (float)s.tiles);
  // (less 5 % of the cluster pass's time: of two equals that one runs)
  return 0.95f * cluster_us(s, c, k, equal, mean) - general_us(s, mean, s.max_chunks);
}
// The gain that is worth launching both passes for, which costs a call 4 us in bf16 and 5 in fp32
// (the one that does not run still starts, after the other).
constexpr float kWorthBothUs = 15.f;

enum AttendPass { kClusterPass, kGeneralPass, kEitherPass };

struct AttendChoice {
  AttendPass pass;
  int ctas, clusters;  // of the cluster pass
};

// `fill`: S_total / (batch * max_len), at most 1.  A batch with fill above 0.9 may have equal
// lengths or any others, so it is judged as equal ones and, half as much, as ragged ones of 0.35 of
// the longest on average (as log-uniform ones are); below, as ragged ones of fill on average.  The
// general pass is the faster with few long groups, which have at most 8 CTAs each in the cluster
// pass and the whole GPU there, and, of fp32 calls, with 5 to 8 heads a group, bound by a CTA's
// arithmetic.  Smaller clusters fill the GPU better (152 SMs hold 15, 23, 36, 76, 152 clusters of 8,
// 6, 4, 2, 1), larger ones split a group further.
// Measured per call (append and attention, one layer, us, 128 elements; sizes 8 / 6 / 4 / 2 / 1,
// general): bf16, equal lengths, 1 sequence of 131071 rows, 2 kv-heads, 1 head a group 74 / 97 /
// 142 / 277 / 540, 45; the same with 8 heads 102 / 132 / 192 / 374 / 727, 136; 2 of 66791, 8 kv-heads
// 107 / 80 / 91 / 150 / 284, 90; ragged, 8 up to 124643, 2 kv-heads 84 / 101 / 140 / 264 / 522, 73;
// the same with 7 heads 103 / 132 / 189 / 367 / 717, 109; 48 up to 17000, 4 kv-heads 87 / 88 / 91 /
// 99 / 106, 99.  fp32, 6 of 9036, 8 kv-heads, 4 heads 88 / 93 / 93 / 88 / 165, 109; the same with 8
// heads 158 / 158 / 159 / 158 / 307, 134; ragged, 11 up to 88235, 2 kv-heads, 1 head 134 / 158 / 211
// / 394 / 773, 173; the same with 7 heads 380 / 505 / 751 / 1488 / 2965, 232.  Over 130 such calls
// the choice is 2 % off the best one's time on average.
//
// With the cluster pass chosen, lengths that leave it few long groups (1, 2, 4, ... full slots among
// empty ones) may still make the general pass the faster: where it gains enough by any of them, the
// call gets both, of which the one that is the faster for its lengths runs.
inline AttendChoice attend_choose(const CallShape &s, int batch, float fill,
                                  const int (&resident)[kNumSizes]) {
  const float w_equal = batch == 1 || fill > 0.9f ? 1.f : 0.f;
  const float w_ragged = batch == 1 ? 0.f : (w_equal > 0.f ? 0.5f : 1.f);
  const float mean = w_equal > 0.f ? 0.35f : fill;
  AttendChoice best = {kClusterPass, 1, 1};
  float best_us = 0.f;
  for (int i = 0; i < kNumSizes; ++i) {
    const int c = kSizes[i], k = resident[i] < s.groups ? resident[i] : s.groups;
    const float us = w_equal * cluster_us(s, c, k, true, 1.f) +
                     w_ragged * cluster_us(s, c, k, false, mean);
    if (best_us == 0.f || us < best_us) {
      best_us = us;
      best = {kClusterPass, c, k};
    }
  }
  // (without the workspace's limit: these weights, the estimates and the 1.05 were fitted together
  // without it, and with it one call in ten, most of them faster by clusters, would change sides)
  constexpr int kAny = 1 << 30;
  if (w_equal * general_us(s, 1.f, kAny) + w_ragged * general_us(s, mean, kAny) < 1.05f * best_us) {
    best.pass = kGeneralPass;
  } else {
    for (int full = 1; full < batch; full *= 2)
      if (general_gains_us(s, batch, full * s.tiles, false, best.ctas, best.clusters) > kWorthBothUs)
        best.pass = kEitherPass;
  }
  return best;
}

}  // namespace lg
