// One step of a bf16 cache that evicts, in ONE launch, for heads whose candidates fit into the shared
// memory of an SM: scores (Eq. 9), selection (Eq. 10 / 11), attention over the survivors and the
// compaction of the cache.
//
// A cluster of one to eight CTAs owns one (batch, head).  Every CTA brings all candidate rows (stored,
// then new; K first, V behind it) into its shared memory with cp.async, the observation rows and its own
// queries with them.  Every CTA forms the same scores and the same list for itself: a few hundred rows
// against 32 observation rows are less than an exchange between CTAs costs.  Then the CTAs share the
// queries, 16 per matrix row tile; keys and values are gathered by ldmatrix through the list, so that
// nothing is compacted before it is attended over.  Last, the CTAs write the survivors that change their
// place, and the surviving new rows, from shared memory to the cache: a cluster barrier has told them that
// all of them hold the old rows.  Heads of a type that evicts nothing in this step skip the selection and
// append.
//
// What bounds it is latency: launch, one trip to memory, some ten block barriers.  The two launches it
// stands for (compression on tcgen05, then attention) wait for each other and each pay a launch, a trip to
// memory and a tail.
// Step of 16 heads x 64, 36 queries, 91 candidates: 12.6 -> 5.9 us (169 queries, 237 candidates: 14.6 -> 7.6);
// 256 heads: 18.2 -> 9.3.  More work per head goes to the two launches (step_shape_bf16).  The cluster
// barrier without memory ordering took 0.45 us off a step, the merge in a form per number of warps 0.25.
// Rounded probabilities (one product instead of two) where the larger kernel's would be rounded as well:
// 5 to 15 % slower from eight turns on, the rounding costs more issue slots than the products.
#include <algorithm>
#include <type_traits>

#include "hack_internal.h"
#include "step_small.cuh"
#include "tc_ptx.cuh"

namespace hack {
namespace {

using namespace ptx;
using namespace small_step;

constexpr int kTile = 16;                       // queries per row tile, keys per warp and turn
constexpr int kMaxTurns = kMaxRows / (kStepWarps * kTile);   // key tiles of a warp whose logits it can hold: 6

// Bytes in front of the small tables: K and V rows (later the warps' unnormalised outputs), observation
// rows, queries.
template <int D>
__host__ __device__ constexpr size_t kv_bytes(int rows) {
  return (size_t)rows * D * 4 > (size_t)kStepWarps * kTile * D * 4 ? (size_t)rows * D * 4 : (size_t)kStepWarps * kTile * D * 4;
}
template <int D>
size_t step_smem(const StepShape& s) {
  return kv_bytes<D>(s.rows) + (size_t)kMaxObs * D * 2 + (size_t)s.tiles * kTile * D * 2 + (size_t)s.rows * 3 * sizeof(int32_t);
}

// Two fp32 numbers as a sum of two packed pairs of bf16.
__device__ __forceinline__ void split_pair(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - __low2float(h), y - __high2float(h));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// kTurns: key tiles per warp that the head types which evict can need
template <int D, int kTurns>
__global__ void __launch_bounds__(kStepThreads, D == 64 && kTurns < kMaxTurns ? 2 : 1)
step_small_kernel(const StepArgs a, const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k_new,
                  const __nv_bfloat16* __restrict__ v_new, __nv_bfloat16* __restrict__ out, const StepShape sp) {
  constexpr int PIECES = D / 8;                 // 16-byte pieces per row
  constexpr uint32_t ROWB = D * 2;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ float2 stats[kStepWarps][kMaxObs];
  __shared__ PickShared ps;
  __shared__ float2 row_ml[kStepWarps][kTile];

  const int bh = a.head_order[blockIdx.y], rank = blockIdx.x;   // structural heads (the longer ones) first
  const int ctx = a.is_ctx[bh % a.n_heads];
  const int stored = a.stored[ctx], n_new = a.n_new, cand = a.cand[ctx], n_keep = a.kept[ctx];
  const bool evicts = a.trig[ctx] && n_keep < cand;
  const size_t off = a.row_off[bh];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  __nv_bfloat16* kc = static_cast<__nv_bfloat16*>(a.k_plane) + off * D;
  __nv_bfloat16* vc = static_cast<__nv_bfloat16*>(a.v_plane) + off * D;
  const __nv_bfloat16* kn = k_new + (size_t)bh * n_new * D;
  const __nv_bfloat16* vn = v_new + (size_t)bh * n_new * D;
  const __nv_bfloat16* qn = q + (size_t)bh * n_new * D;
  const uint32_t k_sm = smem_u32(sm), v_sm = k_sm + (uint32_t)sp.rows * ROWB;
  const uint32_t obs_sm = k_sm + (uint32_t)kv_bytes<D>(sp.rows), q_sm = obs_sm + kMaxObs * ROWB;
  uint32_t* key = reinterpret_cast<uint32_t*>(sm + (q_sm - k_sm) + (size_t)sp.tiles * kTile * ROWB);   // [rows]
  int32_t* list = reinterpret_cast<int32_t*>(key + sp.rows);                                          // [rows]
  int32_t* pos = list + sp.rows;                                                                      // [rows]
  // 16-byte piece c of row r: the pieces of eight consecutive rows fall into different banks
  auto at = [](int r, int c) { return (uint32_t)r * ROWB + (uint32_t)((c ^ (r & 7)) << 4); };
  auto fetch = [](uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  };
  pick_init(ps);
  pdl_wait();

  // ------------------------------------------------------------------ rows into shared memory
  for (int v = tid; v < cand * PIECES; v += kStepThreads) {
    const int r = v / PIECES, c = v % PIECES;
    fetch(k_sm + at(r, c), (r < stored ? kc + (size_t)r * D : kn + (size_t)(r - stored) * D) + c * 8);
  }
  if (evicts) {
    for (int v = tid; v < kMaxObs * PIECES; v += kStepThreads) {
      const int r = v / PIECES, c = v % PIECES;                // rows past the last repeat it and weigh nothing
      fetch(obs_sm + at(r, c), qn + (size_t)obs_row(a, min(r, a.n_obs_rows - 1)) * D + c * 8);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int v = tid; v < cand * PIECES; v += kStepThreads) {
    const int r = v / PIECES, c = v % PIECES;
    fetch(v_sm + at(r, c), (r < stored ? vc + (size_t)r * D : vn + (size_t)(r - stored) * D) + c * 8);
  }
  const int q_first = rank * sp.tiles * kTile;
  for (int v = tid; v < sp.tiles * kTile * PIECES; v += kStepThreads) {
    const int r = v / PIECES, c = v % PIECES;
    fetch(q_sm + at(r, c), qn + (size_t)min(q_first + r, n_new - 1) * D + c * 8);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");

  // ------------------------------------------------------------------ scores and list
  if (evicts) {
    for (int j = tid; j < cand; j += kStepThreads) pos[j] = j < stored ? a.pos_plane[off + j] : a.pos_base + (j - stored);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    // a warp has key tiles warp, warp + 8, ... against all observation rows
    const int key_tiles = (cand + kTile - 1) / kTile;
    float z[kMaxTurns][2][2][4];                // [turn][rows 0-15, 16-31][keys 0-7, 8-15][fragment]
#pragma unroll
    for (int t = 0; t < kTurns; ++t)
#pragma unroll
      for (int e = 0; e < 16; ++e) z[t][e >> 3][(e >> 2) & 1][e & 3] = 0.f;
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
      uint32_t qa[2][4];
      ldsm4(obs_sm + at(lane & 15, 2 * kk + (lane >> 4)), qa[0]);
      ldsm4(obs_sm + at(16 + (lane & 15), 2 * kk + (lane >> 4)), qa[1]);
#pragma unroll
      for (int t = 0; t < kTurns; ++t) {
        uint32_t b[4];                          // a tile past the end is the last one again, and masked below
        ldsm4(k_sm + at(min(t * kStepWarps + warp, key_tiles - 1) * kTile + (lane & 7) + ((lane >> 4) << 3), 2 * kk + ((lane >> 3) & 1)), b);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
          mma16816(z[t][mt][0], qa[mt], b[0], b[1]);
          mma16816(z[t][mt][1], qa[mt], b[2], b[3]);
        }
      }
    }
    const float cs = a.sm_scale * 1.4426950408889634f;        // log2 units
    // the warp's own (max, sum-exp) of every row; the exponentials stay in registers
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float m = -INFINITY;
#pragma unroll
        for (int t = 0; t < kTurns; ++t)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = (t * kStepWarps + warp) * kTile + (e >> 1) * 8 + 2 * (lane & 3) + (e & 1);
            float& x = z[t][mt][e >> 1][2 * h + (e & 1)];
            x = j < cand ? x * cs : -INFINITY;
            m = fmaxf(m, x);
          }
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        const float ref = m == -INFINITY ? 0.f : m;           // a warp without keys
        float l = 0.f;
#pragma unroll
        for (int t = 0; t < kTurns; ++t)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float& x = z[t][mt][e >> 1][2 * h + (e & 1)];
            x = ex2(x - ref);
            l += x;
          }
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
        if ((lane & 3) == 0) stats[warp][mt * 16 + h * 8 + (lane >> 2)] = make_float2(m, l);
      }
    __syncthreads();
    // lane r: the whole head's statistics of row r, as the factor exp2(m_warp - m) / l of this warp's terms
    float f;
    {
      float2 st[kStepWarps];
      float top = -INFINITY, sum = 0.f;
#pragma unroll
      for (int w = 0; w < kStepWarps; ++w) { st[w] = stats[w][lane]; top = fmaxf(top, st[w].x); }
#pragma unroll
      for (int w = 0; w < kStepWarps; ++w) sum = fmaf(ex2(st[w].x - top), st[w].y, sum);
      f = lane < a.n_obs_rows ? ex2(stats[warp][lane].x - top) / sum : 0.f;
    }
    float fr[2][2];
#pragma unroll
    for (int e = 0; e < 4; ++e) fr[e >> 1][e & 1] = __shfl_sync(0xffffffffu, f, (e >> 1) * 16 + (e & 1) * 8 + (lane >> 2));
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int t = 0; t < kTurns; ++t) {
      const int kt = t * kStepWarps + warp;
      if (kt < key_tiles) {
        float s[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          s[e] = 0.f;
#pragma unroll
          for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) s[e] = fmaf(z[t][mt][e >> 1][2 * h + (e & 1)], fr[mt][h], s[e]);
        }
        // the sum over the eight lanes of a column: a lane hands half of its columns on, then adds
        const bool up = lane & 4, upper = lane & 8;
        const float s0 = (up ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, up ? s[0] : s[2], 4);
        const float s1 = (up ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, up ? s[1] : s[3], 4);
        float sc = (upper ? s1 : s0) + __shfl_xor_sync(0xffffffffu, upper ? s0 : s1, 8);
        sc += __shfl_xor_sync(0xffffffffu, sc, 16);
        const int j = kt * kTile + (up ? 8 : 0) + 2 * (lane & 3) + (upper ? 1 : 0);
        if (lane < 16 && j < cand) {
          const bool fixed = is_protected(a, ctx, j);
          const uint32_t k = fixed ? 0xffffffffu : order_key(sc);
          key[j] = k;
          if (!fixed) { lo = min(lo, k); hi = max(hi, k); }
        }
      }
    }
    pick<(kTurns * kStepWarps * kTile + kStepThreads - 1) / kStepThreads>(a, ps, key, list, cand, n_keep, lo, hi);
  } else {
    for (int j = tid; j < n_keep; j += kStepThreads) list[j] = j;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // this CTA has read what it needs of the cache: its loads have landed, so no memory ordering is asked for
  if (sp.ctas > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

  // ------------------------------------------------------------------ attention over the list
  const int splits = 1 << sp.log_splits, tile = warp >> sp.log_splits, split = warp & (splits - 1);
  const float cs = a.sm_scale * 1.4426950408889634f;
  float m[2] = {kNoLogit, kNoLogit}, l[2] = {0.f, 0.f};     // rows lane / 4 and lane / 4 + 8; l: this thread's share
  float o[D / 8][4];
#pragma unroll
  for (int n = 0; n < D / 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
  // KT key tiles of 16 at a time: two where the warp has as many (the chain of a turn is then paid half as often)
  auto attend = [&](auto kt_c) {
    constexpr int KT = decltype(kt_c)::value;
    uint32_t qa[D / 16][4];
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) ldsm4(q_sm + at(tile * kTile + (lane & 15), 2 * kk + (lane >> 4)), qa[kk]);
    for (int j0 = split * KT * kTile; j0 < n_keep; j0 += splits * KT * kTile) {
      int kr[KT], vr[KT];
      float s[2 * KT][4] = {};
#pragma unroll
      for (int u = 0; u < KT; ++u) {
        kr[u] = list[min(j0 + u * kTile + (lane & 7) + ((lane >> 4) << 3), n_keep - 1)];
        vr[u] = list[min(j0 + u * kTile + (lane & 15), n_keep - 1)];
      }
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk)
#pragma unroll
        for (int u = 0; u < KT; ++u) {
          uint32_t b[4];                        // keys 0-7 and 8-15, each with the two halves of the k-step
          ldsm4(k_sm + at(kr[u], 2 * kk + ((lane >> 3) & 1)), b);
          mma16816(s[2 * u], qa[kk], b[0], b[1]);
          mma16816(s[2 * u + 1], qa[kk], b[2], b[3]);
        }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float mt = m[h];
#pragma unroll
        for (int e = 0; e < 4 * KT; ++e) {
          const int j = j0 + (e >> 1) * 8 + 2 * (lane & 3) + (e & 1);
          float& x = s[e >> 1][2 * h + (e & 1)];
          x = j < n_keep ? x * cs : -INFINITY;
          mt = fmaxf(mt, x);
        }
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 1));
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 2));
        const float corr = ex2(m[h] - mt);                    // 0 in the first turn
        m[h] = mt;
        float add = 0.f;
#pragma unroll
        for (int e = 0; e < 4 * KT; ++e) {
          float& x = s[e >> 1][2 * h + (e & 1)];
          x = ex2(x - mt);
          add += x;
        }
        l[h] = l[h] * corr + add;
#pragma unroll
        for (int n = 0; n < D / 8; ++n) { o[n][2 * h] *= corr; o[n][2 * h + 1] *= corr; }
      }
#pragma unroll
      for (int u = 0; u < KT; ++u) {
        uint32_t ph[4], pl[4];
        split_pair(s[2 * u][0], s[2 * u][1], ph[0], pl[0]);
        split_pair(s[2 * u][2], s[2 * u][3], ph[1], pl[1]);
        split_pair(s[2 * u + 1][0], s[2 * u + 1][1], ph[2], pl[2]);
        split_pair(s[2 * u + 1][2], s[2 * u + 1][3], ph[3], pl[3]);
#pragma unroll
        for (int nn = 0; nn < D / 16; ++nn) {
          uint32_t b[4];                        // 16 dimensions: two n-tiles, each with both halves of the 16 keys
          ldsm4_trans(v_sm + at(vr[u], 2 * nn + (lane >> 4)), b);
          mma16816(o[2 * nn], ph, b[0], b[1]);
          mma16816(o[2 * nn + 1], ph, b[2], b[3]);
          mma16816(o[2 * nn], pl, b[0], b[1]);
          mma16816(o[2 * nn + 1], pl, b[2], b[3]);
        }
      }
    }
  };
  if (q_first + tile * kTile < n_new) {
    if (n_keep > splits * kTile) attend(std::integral_constant<int, 2>());
    else attend(std::integral_constant<int, 1>());
  }

  // ------------------------------------------------------------------ survivors to their places in the cache
  if (sp.ctas > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  {
    const int share = (n_keep + sp.ctas - 1) / sp.ctas, r0 = rank * share, r1 = min(n_keep, r0 + share);
    uint4* kd = reinterpret_cast<uint4*>(kc);
    uint4* vd = reinterpret_cast<uint4*>(vc);
    for (int v = r0 * PIECES + tid; v < r1 * PIECES; v += kStepThreads) {
      const int r = v / PIECES, c = v % PIECES, src = list[r];
      // stored rows that stay where they are need not be touched
      if ((src != r || src >= stored) && dbg_ok(src >= r && src < cand && r < a.cap[ctx], a.status, 13)) {
        kd[(size_t)r * PIECES + c] = *reinterpret_cast<const uint4*>(sm + at(src, c));
        vd[(size_t)r * PIECES + c] = *reinterpret_cast<const uint4*>(sm + (size_t)sp.rows * ROWB + at(src, c));
        if (c == 0) a.pos_plane[off + r] = evicts ? pos[src] : a.pos_base + (src - stored);
      }
    }
  }

  // ------------------------------------------------------------------ merge of the warps that share a query tile
  __syncthreads();                              // nothing reads K and V any more
  const int g = lane >> 2;
  float* ob = reinterpret_cast<float*>(sm) + (size_t)warp * kTile * D;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float lh = l[h];
    lh += __shfl_xor_sync(0xffffffffu, lh, 1);
    lh += __shfl_xor_sync(0xffffffffu, lh, 2);
    if ((lane & 3) == 0) row_ml[warp][g + 8 * h] = make_float2(m[h], lh);
#pragma unroll
    for (int n = 0; n < D / 8; ++n) {
      const int u = (4 * n + (lane & 3)) ^ ((g & 3) << 2);
      *reinterpret_cast<float2*>(ob + (g + 8 * h) * D + 2 * u) = make_float2(o[n][2 * h], o[n][2 * h + 1]);
    }
  }
  __syncthreads();
  // four columns per thread; a form per number of warps, so that all loads of a row are in flight at once
  auto combine = [&](auto splits_c) {
    constexpr int S = decltype(splits_c)::value;
    for (int v = tid; v < sp.tiles * kTile * (D / 4); v += kStepThreads) {
      const int row = v / (D / 4), c = v % (D / 4), r = row % kTile, w0 = row / kTile * S;
      if (q_first + row >= n_new) break;
      float2 ml[S], f[S][2];
      float top = -INFINITY, sum = 0.f, acc[4] = {};
#pragma unroll
      for (int w = 0; w < S; ++w) {
        ml[w] = row_ml[w0 + w][r];
        const float* src = reinterpret_cast<const float*>(sm) + (size_t)(w0 + w) * kTile * D + r * D;
#pragma unroll
        for (int e = 0; e < 2; ++e) f[w][e] = *reinterpret_cast<const float2*>(src + 2 * ((2 * c + e) ^ ((r & 3) << 2)));
      }
#pragma unroll
      for (int w = 0; w < S; ++w) top = fmaxf(top, ml[w].x);
#pragma unroll
      for (int w = 0; w < S; ++w) {
        const float wt = ex2(ml[w].x - top);    // 0 for a warp without keys
        sum = fmaf(wt, ml[w].y, sum);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          acc[2 * e] = fmaf(wt, f[w][e].x, acc[2 * e]);
          acc[2 * e + 1] = fmaf(wt, f[w][e].y, acc[2 * e + 1]);
        }
      }
      const float inv = 1.f / sum;
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(acc[0] * inv, acc[1] * inv), h1 = __floats2bfloat162_rn(acc[2] * inv, acc[3] * inv);
      *reinterpret_cast<uint2*>(out + ((size_t)bh * n_new + q_first + row) * D + c * 4) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
    }
  };
  if (sp.log_splits == 3) combine(std::integral_constant<int, 8>());
  else if (sp.log_splits == 2) combine(std::integral_constant<int, 4>());
  else if (sp.log_splits == 1) combine(std::integral_constant<int, 2>());
  else combine(std::integral_constant<int, 1>());
}

template <int D>
int launch_t(const StepArgs& a, const void* q, const void* k_new, const void* v_new, void* out, cudaStream_t st) {
  const int heads = a.batch * a.n_heads, tiles = (a.n_new + kTile - 1) / kTile;
  const int cand = std::max(a.heads_of[0] ? a.cand[0] : 0, a.heads_of[1] ? a.cand[1] : 0);
  if (cand > kMaxRows || tiles > kMaxTiles * kMaxCtas) return 0;
  StepShape s;
  s.rows = (cand + kTile - 1) / kTile * kTile;
  const int ranked = std::max(a.trig[0] ? a.cand[0] : 0, a.trig[1] ? a.cand[1] : 0);
  const int turns = (ranked + kStepWarps * kTile - 1) / (kStepWarps * kTile);
  const StepSizes sizes{D, a.n_new, a.heads_of, a.cand, a.kept, a.trig, sm_count()};
  auto go = [&](auto kern) {
    if (!allow_dynamic_smem(kern, kSmemCta)) return -1;
    const auto places = [&](int ctas, size_t smem) { return cluster_places(reinterpret_cast<const void*>(kern), ctas, kStepThreads, smem); };
    if (!step_shape_bf16(sizes, s, tiles, turns, step_smem<D>, places)) return 0;
    return launch_step<__nv_bfloat16>(kern, a, s, step_smem<D>(s), q, k_new, v_new, out, st);
  };
  if (turns <= 1) return go(step_small_kernel<D, 1>);
  if (turns <= 2) return go(step_small_kernel<D, 2>);
  if constexpr (D == 64) {                      // at head_dim 128 shared memory holds fewer rows than four turns rank
    if (turns > 4) return go(step_small_kernel<D, kMaxTurns>);
  }
  return go(step_small_kernel<D, 4>);
}

}  // namespace

int launch_step_small(const StepArgs& a, int dtype, const void* q, const void* k_new, const void* v_new, void* out, cudaStream_t st) {
  const bool any = a.trig[0] || a.trig[1];
  if (a.score_accumulate || (any && a.obs_full)) return 0;
  if (dtype == HACK_F32) return launch_step_small_f32(a, q, k_new, v_new, out, st);
  if (!any) return 0;                           // append_attend_mma_kernel has no list to go through
  return a.head_dim == 128 ? launch_t<128>(a, q, k_new, v_new, out, st) : launch_t<64>(a, q, k_new, v_new, out, st);
}

}  // namespace hack
