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
// heads, 324 queries, 363 CTAs 60.2, 56.3 and 55.5; 45 heads, 256 queries, 360 CTAs 57.7 and 55.2) or they come in clusters, one on an
// SM (attention_ctas 0; 12 heads, a whole loop of 680 tokens 123.8 with two and one at its last scales, 121.2 with four).  In loops of one or two layers
// four CTAs for 16 heads are 1 % faster, in loops of four and more 1 to 2 % slower.
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

// ---------------------------------------------------------------- small steps in one launch (step_small.cu, step_small_f32.cu)
namespace small_step {

constexpr int kStepWarps = 8;
constexpr int kStepThreads = kStepWarps * 32;
constexpr int kMaxRows = 768;                   // candidates of a head, at most
constexpr int kMaxTiles = 8;                    // query tiles of a CTA
constexpr int kMaxCtas = 8;                     // CTAs per head
constexpr size_t kSmemCta = 216 * 1024;         // dynamic shared memory beside the static tables ...
constexpr size_t kSmemHalf = 108 * 1024;        // ... and with two CTAs on an SM

struct StepShape {
  int ctas;        // CTAs per head
  int tiles;       // query tiles per CTA: 1, 2, 4 or 8; the CTA's 8 warps share the keys of a tile 8 / tiles ways
  int log_splits;  // log2(8 / tiles)
  int rows;        // candidate rows shared memory has room for
};

// What the rules know of a step; arrays by head type, structural heads first (as the launches take them).
struct StepSizes {
  int head_dim, n_new;
  const int *heads_of, *cand, *kept, *trig;
  int sms;
};

// The CTAs of a head and their query tiles: as many CTAs per head as leave every CTA an SM, at least what its
// queries need; clusters of seven and eight only where they are few (16 clusters of 8 CTAs do not find a
// place at once beside each other: 100 queries, 16 heads, bf16: 7 CTAs 8.5 us, 4 CTAs 7.9; 169 queries:
// 6 CTAs 8.2, 3 CTAs 10.3).
inline void split_queries(StepShape& s, int heads, int tiles, int sms, int at_most = kMaxCtas) {
  auto split = [&](int most) {
    int want = sms / heads < tiles ? sms / heads : tiles;
    want = want < 1 ? 1 : want > most ? most : want;
    for (s.tiles = 1; s.tiles < kMaxTiles && s.tiles * want < tiles; s.tiles *= 2) {}
    s.ctas = (tiles + s.tiles - 1) / s.tiles;
  };
  split(at_most);
  if (s.ctas > 6 && heads * s.ctas * 2 > sms) split(kMaxCtas / 2);
  for (s.log_splits = 0; s.tiles << s.log_splits < kStepWarps; ++s.log_splits) {}
}

// The clusters of split_queries are meant to run at once, but may not all find a place (the SMs of a processing cluster are
// no multiple of every size: 148 SMs take 45 clusters of 3, 33 of 4, 22 of 6).  Returns the heads that have to wait for a
// first one to end; if there are any, `smaller` is the shape of the largest clusters that all find a place and fit shared
// memory (ctas 0: there is none, -1: it does not fit).
template <typename Smem, typename Places>
int split_and_place(StepShape& s, StepShape& smaller, int heads, int tiles, int sms, Smem smem, Places places) {
  auto missing = [&](const StepShape& of) {
    const size_t bytes = smem(of);
    if (heads * of.ctas > sms || bytes > kSmemCta) return 0;
    const int n = places(of.ctas, bytes <= kSmemHalf ? kSmemHalf : kSmemCta);
    return heads > n ? heads - n : 0;
  };
  split_queries(s, heads, tiles, sms);
  smaller = s;
  const int waiting = missing(s);
  bool found = false, fits = true;
  for (int most = s.ctas - 1; waiting > 0 && most >= 1 && !found && fits; --most) {
    split_queries(smaller, heads, tiles, sms, most);
    fits = smem(smaller) <= kSmemCta;
    found = fits && smaller.ctas < s.ctas && missing(smaller) == 0;
  }
  if (!found) smaller.ctas = fits ? 0 : -1;
  return waiting;
}

// Microseconds of a bf16 step in one launch and in the two it stands for (compression, then attention).  Both forms were
// fitted to 287 steps of 8 to 256 heads, 16 to 400 queries and 50 to 700 candidates (rms 8 and 6 %).  two_waves: the same in one
// launch of which `waiting` heads, the last ones, start when the first clusters end (23 to 49 heads, 81 to 361 queries,
// within 10 % where shared memory holds one CTA).
struct StepTimes { float here, two_waves, apart; };
inline StepTimes step_times(const StepSizes& z, const StepShape& s, int per_sm, int waiting) {
  constexpr int kTile = 16;                     // keys a warp weighs at a time
  const float sms = (float)z.sms, heads = (float)(z.heads_of[0] + z.heads_of[1]), ctas = heads * s.ctas;
  const float turn = z.head_dim == 64 ? 0.92f : 1.81f;
  const int keys = 2 * kTile << s.log_splits;   // of a turn
  float longest = 0.f, mean = 0.f, work = 0.f, ranked = 0.f, last = 0.f;
  for (int t = 0; t < 2; ++t) {
    if (z.heads_of[t] == 0) continue;
    const float start = 2.1f + (z.trig[t] && z.kept[t] < z.cand[t] ? 3.5f : 0.f) + 0.031f * (z.cand[t] * z.head_dim * 4 / 1000.f);
    const float us = start + turn * ((z.kept[t] + keys - 1) / keys);
    longest = std::max(longest, us);
    mean += us * z.heads_of[t] / heads;
    work += (float)z.heads_of[t] * ((z.n_new + 127) / 128) * (1 + (z.kept[t] + 127) / 128);
    if (z.trig[t]) ranked = std::max(ranked, z.cand[t] / 128.f);
    if (t == 0 || z.heads_of[1] >= waiting) last = start + turn * z.kept[t] / keys;
  }
  StepTimes us;
  // two CTAs on an SM slow each other down by two thirds
  us.here = std::max(longest * (per_sm == 2 ? 1.f + 0.67f * std::min(1.f, std::max(0.f, ctas / sms - 1.f)) : 1.f),
                     ctas > sms * per_sm ? mean * (ctas / (sms * per_sm) * (per_sm == 2 ? 1.67f : 1.f) + 0.3f) : 0.f);
  us.two_waves = std::max(longest, 1.8f * last);
  us.apart = z.head_dim == 64 ? 10.8f + (1.58f * heads + 0.92f * work) / sms + 1.57f * ranked
                              : 11.9f + (3.92f * heads + 1.13f * work) / sms + 1.94f * ranked;
  return us;
}

// The shape of a bf16 step in one launch (s.rows is given); false: two launches are the faster ones.  turns: key tiles of a warp.
// This side has become faster since the fit where every CTA has an SM and a cluster is smaller than eight, so there it
// is taken up to a tenth past the line, to 256 queries: 13 heads x 128, 121 queries 20.5 -> 15.7 us, 36 heads, 169 queries
// 22.2 -> 18.4, 52 heads x 64, 196 queries 22.5 -> 19.1.  Elsewhere it keeps a margin of a tenth (81 heads x 64, 169 queries
// 20.5 against 24.6; 18 heads, 400 queries 21.2 against 22.5; at 289 and 324 queries, 26 and 22 heads x 64, 13.6-16.4 against
// 16.1-19.5, either margin takes it).  16 heads x 64, 36 queries, 91 candidates: 5.9 against 12.6;
// 256 heads: 9.3 against 18.2; 100 queries, 168 and 255 candidates: 7.3 against 12.8 (16 heads), 20.2 against
// 19.9 (256 heads: not taken); 16 heads x 128, 36 queries, 91 candidates: 7.5 against 15.0; 256 heads: 18.6
// against 25.2.
// Where clusters would have to wait, smaller ones usually are faster (46 heads x 128, 81 queries 17.1 -> 12.3 us; 35 heads, 121
// queries 17.4 -> 13.0; 24 heads, 81 queries 16.0 -> 10.2), but not if the heads that wait are contextual ones of few
// keys: 46 heads x 128, 144 queries, 174 candidates, clusters of 3, of 2, two launches: 16.1, 17.9 and 17.4 us with 23 keys, 17.1,
// 17.9 and 17.7 with 43, 19.5, 17.9 and 18.9 with 87.  (At head_dim 64 with a margin: 24 heads, 324 queries, 435 candidates 18.0
// against 16.4 for two launches.)
template <typename Smem, typename Places>
bool step_shape_bf16(const StepSizes& z, StepShape& s, int tiles, int turns, Smem smem, Places places) {
  const int heads = z.heads_of[0] + z.heads_of[1];
  StepShape smaller;
  const int waiting = split_and_place(s, smaller, heads, tiles, z.sms, smem, places);
  auto times = [&](const StepShape& of) { return step_times(z, of, z.head_dim == 64 && turns <= 4 && smem(of) <= kSmemHalf ? 2 : 1, waiting); };
  if (smem(s) > kSmemCta) return false;
  if (waiting > 0) {
    const StepTimes us = times(s);
    if (smaller.ctas <= 0 || us.two_waves < 0.95f * times(smaller).here) return us.two_waves * (z.head_dim == 64 ? 1.1f : 1.f) < us.apart;
    s = smaller;
  }
  const StepTimes us = times(s);
  return us.here * (heads * s.ctas <= z.sms && s.ctas < kMaxCtas && z.n_new <= 256 ? 0.9f : 1.1f) < us.apart;
}

// The same for a step of an fp32 cache: every head of up to 128 candidates; longer ones only where every CTA has an SM to itself
// (120 heads x 64, 260 candidates, 240 CTAs: 37.0 against 42.1 us; 120 heads, 155 candidates, 120 CTAs: 30.7 -> 19.0).
// Where clusters would have to wait, both shapes by lines through what they took (23 to 48 heads, 81 to 169 queries, 102 to 311
// candidates; 4 %): 23 heads x 64, 169 queries, 311 candidates, clusters of 6 and of 3: 26.7 and 39.9 us with 24 keys in the heads that
// wait, 35.3 and 39.9 with 103, 41.0 and 40.2 with 155; 36 heads x 128, 100 queries, clusters of 4 and of 2: 30.2 and 32.5 with
// 18 keys, 42.6 and 32.8 with 90.  Where the smaller ones do not fit shared memory the launches of their own are faster (27
// heads x 128, 144 queries 35.1 against 35 to 47).
template <typename Smem, typename Places>
bool step_shape_f32(const StepSizes& z, StepShape& s, int tiles, Smem smem, Places places) {
  const int heads = z.heads_of[0] + z.heads_of[1], cand = std::max(z.heads_of[0] ? z.cand[0] : 0, z.heads_of[1] ? z.cand[1] : 0);
  StepShape smaller;
  const int waiting = split_and_place(s, smaller, heads, tiles, z.sms, smem, places);
  if (waiting > 0) {
    const int kept = std::max(z.heads_of[0] ? z.kept[0] : 0, z.heads_of[1] ? z.kept[1] : 0);
    const int last = z.kept[z.heads_of[1] >= waiting ? 1 : 0];
    const int keys = 32 << s.log_splits, keys_smaller = 32 << smaller.log_splits;   // of a turn of the warps
    const int more = (last + keys - 1) / keys - 1, turns = (kept + keys_smaller - 1) / keys_smaller;
    const float part = (float)last / keys, past = cand > 128 ? 3.f : 0.f;
    const float two_waves = z.head_dim == 64 ? 18.3f + 0.02f * cand + 4.5f * part + 3.f * more : 27.7f + 6.7f * part + 4.5f * more + 2.f * past;
    const float one_wave = z.head_dim == 64 ? 9.3f + 3.05f * turns : 15.3f + 4.3f * turns + past;
    const bool evicts = z.trig[0] || z.trig[1];
    if (smaller.ctas < 0) return false;
    if (smaller.ctas > 0 && (!evicts || 1.03f * two_waves > one_wave)) s = smaller;
  }
  return smem(s) <= kSmemCta && (cand <= 128 || heads * s.ctas <= z.sms);
}

}  // namespace small_step
}  // namespace hack
