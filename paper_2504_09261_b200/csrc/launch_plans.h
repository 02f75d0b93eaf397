// How launches are cut up: host rules on the sizes of a step, apart from the code that launches.
#pragma once

#include <stddef.h>

#include <algorithm>

namespace hack {

// K and V rows of a head up to which the selection moves the rows itself (select_kernels.cu).
constexpr size_t kSmallMoveBytes = 384 * 1024;

// ---------------------------------------------------------------- selection with the moves (select_kernels.cu)
// CTAs per head.  A cluster moves a head's rows faster than one CTA, which reads and writes its own at 40 GB/s, but every
// cluster has to find a place at once (148 SMs take 33 of 4 CTAs: 37 heads x 64, 324 queries 67.8 us a step with one CTA, 72.2 with
// four).  The CTAs of the attention behind it take their SMs while it runs.  At head_dim 128 an SM holds one of them either way
// (us a step with one, two and four CTAs: 16 heads, 324 queries 50.4, 48.1 and 45.8, 26 heads 67.3, 65.1 and 63.0, 37 heads 80.4,
// 77.9 and, in a second wave, 81.5).  At head_dim 64 two of them meet on an SM if the launch leaves too few, so there it
// leaves one each of attention_ctas (8 heads, 196 queries, 64 CTAs 23.0, 23.0 and 21.5; 16 heads, 112 CTAs 33.3, 31.7 and 36.4, 256
// queries, 128 CTAs 28.4, 30.5 and 30.0; 26 heads, 182 CTAs 28.4, 32.3 and 34.3), unless there are two for every SM anyway (33
// heads, 324 queries, 363 CTAs 60.2, 56.3 and 55.5; 45 heads, 256 queries, 360 CTAs 57.7 and 55.2).
template <typename Places>
int move_ctas(int heads, int attention_ctas, int sms, Places places) {
  int cl = 1;
  const int beside = attention_ctas < 2 * sms ? attention_ctas : 0;
  while (cl < 4 && heads * cl * 2 + beside <= sms && heads <= places(2 * cl)) cl *= 2;
  return cl;
}

// ---------------------------------------------------------------- attention of fp32 caches (attend_simt.cu)
namespace simt {

constexpr int kBQ = 32;              // query rows per CTA
constexpr int kBK = 32;              // keys per tile
constexpr int kGroups = 4;           // groups of 64 threads, each with its own key tiles

#if defined(__CUDACC__)
#define HACK_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define HACK_HOST_DEVICE inline
#endif

// A launch whose query tiles are shared out evenly: the tiles of the first type's heads, then the others', laid
// end to end, a tile of r rounds (a key tile per group each) as 2 r + 1 half rounds, the first of which stands for its
// loads and its merge.  CTA i takes the half rounds [i * span, (i + 1) * span).
struct Shares {
  int n_qt, n_first;              // query tiles per head; of the first type's heads together
  int rounds[2];                  // of a query tile of the first type, of the other one
  int span, total;                // half rounds of a CTA, of the launch
};
HACK_HOST_DEVICE int tile_begin(const Shares& sh, int tile) {
  const int n = tile < sh.n_first ? tile : sh.n_first;
  return n * (2 * sh.rounds[0] + 1) + (tile - n) * (2 * sh.rounds[1] + 1);
}

// Rounds until `slots` CTAs at a time have done the tiles one by one, those of the first type first.
inline float rounds_one_by_one(const Shares& sh, int tiles, int slots) {
  struct Group { float at; int n; } g[16] = {{0.f, slots}};
  int groups = 1;
  float end = 0.f;
  for (int type = 0; type < 2; ++type)
    for (int left = type == 0 ? sh.n_first : tiles - sh.n_first; left > 0;) {
      int e = 0;                                             // the places that are free first
      for (int i = 1; i < groups; ++i)
        if (g[i].at < g[e].at) e = i;
      const int take = std::min(left, g[e].n);
      const float at = g[e].at + sh.rounds[type] + 0.5f;
      g[e].n -= take;
      if (g[e].n == 0) g[e] = g[--groups];
      if (groups == 16) return 1e30f;
      g[groups++] = {at, take};
      end = std::max(end, at);
      left -= take;
    }
  return end;
}

struct SimtPlan {
  int cluster;                    // CTAs per query tile
  bool shared;                    // CTAs with equal shares
  int ctas;
  Shares sh;
};

// kept, heads_of: keys per head and heads of either type.
inline SimtPlan simt_plan(int head_dim, int n_new, const int* kept, const int* heads_of, int sms) {
  const int n_qt = (n_new + kBQ - 1) / kBQ, heads = heads_of[0] + heads_of[1];
  SimtPlan p{1, false, 0, {}};
  // Cluster size: the shortest estimate of the launch in key tiles of a group.  A CTA costs its share of
  // the tiles and about three more (start, merge); a launch past one wave lasts as long as all of them
  // spread over the SMs plus half of its longest CTA.  Steps of 16 heads x 100 queries x 64: 33.2 -> 30.8 us
  // with two CTAs per query tile, 256 queries 49.5 -> 39.3; 324 queries x 128: 85 -> 75 by the order of the
  // heads alone; 4 CTAs per tile 310 -> 464 where the launch is long anyway (1 024 queries, 1 717 keys).
  float best = 0.f;
  for (int c = 1; c <= 4; c *= 2) {
    float total = 0.f, longest = 0.f;
    for (int t = 0; t < 2; ++t) {
      if (heads_of[t] == 0) continue;
      const float one = 3.f + (float)(((kept[t] + kBK - 1) / kBK + c * kGroups - 1) / (c * kGroups));
      total += one * heads_of[t] * n_qt * c;
      longest = std::max(longest, one);
    }
    const float cost = n_qt * c * heads <= sms ? longest : std::max(longest, total / sms + 0.5f * longest);
    if (c == 1 || cost < best) {
      best = cost;
      p.cluster = c;
    }
  }
  p.ctas = n_qt * heads * p.cluster;
  if (p.cluster > 1) return p;
  const int first_type = kept[1] > kept[0];
  const int slots = sms * (head_dim == 64 ? 2 : 1);
  Shares& sh = p.sh;
  sh.n_qt = n_qt;
  sh.n_first = n_qt * heads_of[first_type];
  for (int i = 0; i < 2; ++i) {
    const int type = i == 0 ? first_type : 1 - first_type;
    sh.rounds[i] = ((kept[type] + kBK - 1) / kBK + kGroups - 1) / kGroups;
  }
  // A query tile per CTA, the longer ones first, or equal shares, whichever ends earlier; parts of a tile that meet
  // in memory cost about a round.  16 heads x 128, us a step: 324 queries (176 tiles) 70 against 77, 576 queries
  // (288 tiles) 170 against 138, 1 024 queries (512 tiles) 300 against 267.
  // At head_dim 64 the two CTAs of an SM take turns on the FMA pipe, so that an SM is one place that does two
  // spans, and a start and a merge cost more against the shorter rounds.  Shares and a tile per CTA, us a step: 176
  // tiles of 8 rounds 57.5 and 62.5, 352 of 17 171 and 188, 768 of 11 238 and 247, but 407 of 8 104 and 92, 465 of 4 65.2
  // and 60.9, 2 046 of 17 885 and 831.  Behind a compaction with launches of its own, whose last CTAs still hold SMs, tiles
  // of the longer type may meet on one SM: 88 tiles of 8 rounds and 88 of 2 62.7 and 79; behind the selection that moves the
  // rows itself they do not: 91 of 5 and 91 of 2 50.4 and 47.9.
  sh.total = tile_begin(sh, n_qt * heads);
  sh.span = (sh.total + slots - 1) / slots;
  const float by_share = head_dim == 64 ? 1.06f * sh.span + 4.5f : 0.5f * sh.span + 1.f;
  float by_tile = rounds_one_by_one(sh, n_qt * heads, sms);
  if (head_dim == 64 && (size_t)kept[first_type] * head_dim * 8 > kSmallMoveBytes)
    by_tile = std::max(by_tile, 2.f * (sh.rounds[0] + 0.5f));
  p.shared = n_qt * heads > sms && by_tile > by_share;
  p.ctas = p.shared ? (sh.total + sh.span - 1) / sh.span : n_qt * heads;
  return p;
}

}  // namespace simt
}  // namespace hack
