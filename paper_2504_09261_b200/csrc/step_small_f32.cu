// One step of an fp32 cache that evicts, in ONE launch: the form of step_small.cu on the FMA pipe.
//
// A cluster of one to eight CTAs owns one (batch, head); every CTA holds all candidate rows in shared
// memory, ranks them for itself, serves its share of the queries through the list and writes its share of
// the rows that move.  Scores: a warp has 8 of the 32 observation rows and every other group of 32 keys, a
// lane one key of each group, so that a key row is read once for 8 products and the observation rows are
// broadcasts; rows are padded by 16 bytes, which spreads the lanes over the banks.  Attention: a warp has 8
// queries and, as above, 32 keys a turn; for the second product the probabilities go through shared
// memory and a lane owns D / 32 output columns.
// The three launches it stands for (scores, selection with compaction, attention) take 20 us however little
// there is to do, each a launch and a trip to memory behind the one before.
// Step of 16 heads x 64, 36 queries, 91 candidates: 19.6 -> 10.8 us; 64 heads: 24.3 -> 13.9; 16 heads x 128: 26.6 -> 14.4.
#include <algorithm>
#include <type_traits>

#include "hack_internal.h"
#include "step_small.cuh"
#include "tc_ptx.cuh"

namespace hack {
namespace {

using namespace ptx;
using namespace small_step;

constexpr int kRows = 8;                        // observation rows, or queries, of a warp
constexpr int kKeys = 32;                       // keys of a warp and turn: one per lane
constexpr int kObsGroups = kMaxObs / kRows;     // 4: the 8 warps are 4 groups of rows x 2 of keys
constexpr int kKeyWarps = kStepWarps / kObsGroups;
constexpr int kMaxTurns = 5;                    // groups of 32 keys of a warp whose logits it holds
// Candidates up to which a step is served: every CTA of a head ranks all of them on the FMA pipe.  16 heads x 64,
// 260 candidates 24.6 -> 20.0 us, 64 heads 32.5 -> 26.8; 329 candidates 25.7 against 23.6, 64 heads 33.5 against 48.2.
constexpr int kMaxCand = kMaxTurns * kKeyWarps * kKeys;   // 320
constexpr float kLog2e = 1.4426950408889634f;

// Steps that evict nothing: 16 heads x 64, 25 queries and 55 keys 9.1 -> 5.2 us, 64 heads 18.6 -> 6.2 (against a warp per
// query); 36 queries, 91 keys 8.2 -> 5.7, 120 heads 12.9 -> 11.8 (against copy and attend_simt_kernel); 155 keys 9.8
// against 9.3, 30 heads 10.3 against 10.8; 4 queries, 5 keys 3.2 against 4.1.
constexpr int kMaxAppend = 96, kMinAppend = 12;

template <int D>
struct Layout {
  static constexpr int kKeyFloats = D + 4;      // padded key row
  size_t v, obs, q, part, key, list, pos, total;   // byte offsets; the warps' outputs take the place of the keys
  __host__ __device__ Layout(int rows, int tiles) {
    const size_t k_bytes = (size_t)rows * kKeyFloats * 4, o_bytes = (size_t)kStepWarps * kRows * D * 4;
    v = k_bytes > o_bytes ? k_bytes : o_bytes;
    obs = v + (size_t)rows * D * 4;
    q = obs + (size_t)kMaxObs * D * 4;
    part = q + (size_t)tiles * kRows * D * 4;
    key = part + (size_t)rows * kObsGroups * 4;
    list = key + (size_t)rows * 4;
    pos = list + (size_t)rows * 4;
    total = pos + (size_t)rows * 4;
  }
};

// Reduction of eight values over the 32 lanes of a warp; every lane receives all eight results.
template <typename Op>
__device__ __forceinline__ void reduce8(float (&x)[kRows], Op op) {
  const int lane = threadIdx.x & 31;
  float y[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {                 // a lane hands half of its values on and keeps the other half
    const bool up = lane & 16;
    const float got = __shfl_xor_sync(0xffffffffu, up ? x[i] : x[i + 4], 16);
    y[i] = op(up ? x[i + 4] : x[i], got);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool up = lane & 8;
    const float got = __shfl_xor_sync(0xffffffffu, up ? y[i] : y[i + 2], 8);
    y[i] = op(up ? y[i + 2] : y[i], got);
  }
  const bool up = lane & 4;
  const float got = __shfl_xor_sync(0xffffffffu, up ? y[0] : y[1], 4);
  float r = op(up ? y[1] : y[0], got);
  r = op(r, __shfl_xor_sync(0xffffffffu, r, 2));
  r = op(r, __shfl_xor_sync(0xffffffffu, r, 1));
#pragma unroll
  for (int i = 0; i < kRows; ++i) x[i] = __shfl_sync(0xffffffffu, r, ((i >> 2) & 1) * 16 + ((i >> 1) & 1) * 8 + (i & 1) * 4);
}

// kTurns: groups of 32 keys per warp that the head types which evict can need
template <int D, int kTurns>
__global__ void __launch_bounds__(kStepThreads, kTurns <= 2 ? 2 : 1)
step_small_f32_kernel(const StepArgs a, const float* __restrict__ q, const float* __restrict__ k_new,
                      const float* __restrict__ v_new, float* __restrict__ out, const StepShape sp) {
  constexpr int PIECES = D / 4, KF = Layout<D>::kKeyFloats, PAIRS = D / 64;   // 16-byte pieces; column pairs per lane
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ PickShared ps;
  __shared__ float2 stats[kKeyWarps][kMaxObs];
  __shared__ __align__(16) float prob[kStepWarps][kRows][kKeys];
  __shared__ float2 row_ml[kStepWarps][kRows];

  const int bh = a.head_order[blockIdx.y], rank = blockIdx.x;   // structural heads (the longer ones) first
  const int ctx = a.is_ctx[bh % a.n_heads];
  const int stored = a.stored[ctx], n_new = a.n_new, cand = a.cand[ctx], n_keep = a.kept[ctx];
  const bool evicts = a.trig[ctx] && n_keep < cand;
  const size_t off = a.row_off[bh];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Layout<D> lay(sp.rows, sp.tiles);
  float* kc = static_cast<float*>(a.k_plane) + off * D;
  float* vc = static_cast<float*>(a.v_plane) + off * D;
  const float* kn = k_new + (size_t)bh * n_new * D;
  const float* vn = v_new + (size_t)bh * n_new * D;
  const float* qn = q + (size_t)bh * n_new * D;
  float* ks = reinterpret_cast<float*>(sm);
  float* vs = reinterpret_cast<float*>(sm + lay.v);
  float* os = reinterpret_cast<float*>(sm + lay.obs);
  float* qs = reinterpret_cast<float*>(sm + lay.q);
  float* part = reinterpret_cast<float*>(sm + lay.part);       // [kObsGroups][rows]
  uint32_t* key = reinterpret_cast<uint32_t*>(sm + lay.key);
  int32_t* list = reinterpret_cast<int32_t*>(sm + lay.list);
  int32_t* pos = reinterpret_cast<int32_t*>(sm + lay.pos);
  auto fetch = [](const float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
  };
  pick_init(ps);
  pdl_wait();

  // ------------------------------------------------------------------ rows into shared memory
#pragma unroll 2
  for (int v = tid; v < cand * PIECES; v += kStepThreads) {
    const int r = v / PIECES, c = v % PIECES;
    fetch(ks + r * KF + c * 4, (r < stored ? kc + (size_t)r * D : kn + (size_t)(r - stored) * D) + c * 4);
  }
  if (evicts) {
#pragma unroll 1
    for (int v = tid; v < kMaxObs * PIECES; v += kStepThreads) {
      const int r = v / PIECES, c = v % PIECES;                // rows past the last repeat it and weigh nothing
      fetch(os + v * 4, qn + (size_t)obs_row(a, min(r, a.n_obs_rows - 1)) * D + c * 4);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll 2
  for (int v = tid; v < cand * PIECES; v += kStepThreads) {
    const int r = v / PIECES, c = v % PIECES;
    fetch(vs + v * 4, (r < stored ? vc + (size_t)r * D : vn + (size_t)(r - stored) * D) + c * 4);
  }
  const int q_first = rank * sp.tiles * kRows;
#pragma unroll 1
  for (int v = tid; v < sp.tiles * kRows * PIECES; v += kStepThreads) {
    const int r = v / PIECES, c = v % PIECES;
    fetch(qs + v * 4, qn + (size_t)min(q_first + r, n_new - 1) * D + c * 4);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const float cs = a.sm_scale * kLog2e;         // log2 units

  // ------------------------------------------------------------------ scores and list
  if (evicts) {
#pragma unroll 1
    for (int j = tid; j < cand; j += kStepThreads) pos[j] = j < stored ? a.pos_plane[off + j] : a.pos_base + (j - stored);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const int o0 = (warp % kObsGroups) * kRows, kw = warp / kObsGroups;
    float z[kTurns][kRows];
    {
      float2 acc[kTurns][kRows];                // even and odd dimensions apart
#pragma unroll
      for (int t = 0; t < kTurns; ++t)
#pragma unroll
        for (int i = 0; i < kRows; ++i) acc[t][i] = make_float2(0.f, 0.f);
      const float4* kp[kTurns];
#pragma unroll
      for (int t = 0; t < kTurns; ++t)
        kp[t] = reinterpret_cast<const float4*>(ks + min((t * kKeyWarps + kw) * kKeys + lane, cand - 1) * KF);
#pragma unroll 2
      for (int c = 0; c < PIECES; ++c) {
        float4 kf[kTurns];
#pragma unroll
        for (int t = 0; t < kTurns; ++t) kf[t] = kp[t][c];
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          const float4 qq = *reinterpret_cast<const float4*>(os + (o0 + i) * D + c * 4);
#pragma unroll
          for (int t = 0; t < kTurns; ++t) {
            acc[t][i] = fma2(make_float2(qq.x, qq.y), make_float2(kf[t].x, kf[t].y), acc[t][i]);
            acc[t][i] = fma2(make_float2(qq.z, qq.w), make_float2(kf[t].z, kf[t].w), acc[t][i]);
          }
        }
      }
#pragma unroll
      for (int t = 0; t < kTurns; ++t)
#pragma unroll
        for (int i = 0; i < kRows; ++i)
          z[t][i] = (t * kKeyWarps + kw) * kKeys + lane < cand ? (acc[t][i].x + acc[t][i].y) * cs : -INFINITY;
    }
    // the warp's own (max, sum-exp) of its rows; the exponentials stay in registers
    float m[kRows], l[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      m[i] = z[0][i];
#pragma unroll
      for (int t = 1; t < kTurns; ++t) m[i] = fmaxf(m[i], z[t][i]);
    }
    reduce8(m, [](float x, float y) { return fmaxf(x, y); });
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const float ref = m[i] == -INFINITY ? 0.f : m[i];        // a warp without keys
      l[i] = 0.f;
#pragma unroll
      for (int t = 0; t < kTurns; ++t) {
        z[t][i] = exp2f(z[t][i] - ref);
        l[i] += z[t][i];
      }
    }
    reduce8(l, [](float x, float y) { return x + y; });
#pragma unroll
    for (int i = 0; i < kRows; ++i)
      if (lane == i) stats[kw][o0 + i] = make_float2(m[i], l[i]);
    __syncthreads();
    float f[kRows];                             // exp2(m_warp - m) / l of the whole head, per row
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const float2 s0 = stats[0][o0 + i], s1 = stats[1][o0 + i];
      const float top = fmaxf(s0.x, s1.x);
      const float sum = s0.y * exp2f(s0.x - top) + s1.y * exp2f(s1.x - top);
      f[i] = o0 + i < a.n_obs_rows ? exp2f(m[i] - top) / sum : 0.f;
    }
#pragma unroll
    for (int t = 0; t < kTurns; ++t) {
      const int j = (t * kKeyWarps + kw) * kKeys + lane;
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < kRows; ++i) s = fmaf(z[t][i], f[i], s);
      if (j < cand) part[(size_t)(warp % kObsGroups) * sp.rows + j] = s;
    }
    __syncthreads();
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll 1
    for (int j = tid; j < cand; j += kStepThreads) {
      float s = 0.f;
#pragma unroll
      for (int g = 0; g < kObsGroups; ++g) s += part[(size_t)g * sp.rows + j];
      const bool fixed = is_protected(a, ctx, j);
      const uint32_t k = fixed ? 0xffffffffu : order_key(s);
      key[j] = k;
      if (!fixed) { lo = min(lo, k); hi = max(hi, k); }
    }
    pick<(kTurns * kKeyWarps * kKeys + kStepThreads - 1) / kStepThreads>(a, ps, key, list, cand, n_keep, lo, hi);
  } else {
#pragma unroll 1
    for (int j = tid; j < n_keep; j += kStepThreads) list[j] = j;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // this CTA has read what it needs of the cache: its loads have landed, so no memory ordering is asked for
  if (sp.ctas > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

  // ------------------------------------------------------------------ attention over the list
  const int splits = 1 << sp.log_splits, tile = warp >> sp.log_splits, split = warp & (splits - 1);
  float m[kRows], l[kRows];
  float2 o[kRows][PAIRS];
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    m[i] = kNoLogit;
    l[i] = 0.f;                                 // this lane's share
#pragma unroll
    for (int p = 0; p < PAIRS; ++p) o[i][p] = make_float2(0.f, 0.f);
  }
  if (q_first + tile * kRows < n_new) {
    const float* qt = qs + (size_t)tile * kRows * D;
#pragma unroll 1
    for (int j0 = split * kKeys; j0 < n_keep; j0 += splits * kKeys) {
      const int live = min(kKeys, n_keep - j0);
      const int src = list[j0 + min(lane, live - 1)];
      float x[kRows];
      {
        float2 acc[kRows];
#pragma unroll
        for (int i = 0; i < kRows; ++i) acc[i] = make_float2(0.f, 0.f);
        const float4* kp = reinterpret_cast<const float4*>(ks + src * KF);
#pragma unroll 4
        for (int c = 0; c < PIECES; ++c) {
          const float4 kf = kp[c];
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            const float4 qq = *reinterpret_cast<const float4*>(qt + i * D + c * 4);
            acc[i] = fma2(make_float2(qq.x, qq.y), make_float2(kf.x, kf.y), acc[i]);
            acc[i] = fma2(make_float2(qq.z, qq.w), make_float2(kf.z, kf.w), acc[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < kRows; ++i) x[i] = lane < live ? (acc[i].x + acc[i].y) * cs : -INFINITY;
      }
      float mt[kRows];
#pragma unroll
      for (int i = 0; i < kRows; ++i) mt[i] = x[i];
      reduce8(mt, [](float u, float w) { return fmaxf(u, w); });
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        mt[i] = fmaxf(mt[i], m[i]);
        const float corr = exp2f(m[i] - mt[i]), p = exp2f(x[i] - mt[i]);   // corr: 0 in the first turn
        m[i] = mt[i];
        l[i] = fmaf(l[i], corr, p);
        prob[warp][i][lane] = p;
#pragma unroll
        for (int u = 0; u < PAIRS; ++u) o[i][u] = mul2(o[i][u], make_float2(corr, corr));
      }
      __syncwarp();
#pragma unroll 2
      for (int jj = 0; jj < live; jj += 4) {    // probabilities past the last key are 0
        float2 vf[4][PAIRS];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float* vrow = vs + (size_t)list[j0 + min(jj + u, live - 1)] * D;
#pragma unroll
          for (int p = 0; p < PAIRS; ++p) vf[u][p] = *reinterpret_cast<const float2*>(vrow + 2 * lane + 64 * p);
        }
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          const float4 w = *reinterpret_cast<const float4*>(&prob[warp][i][jj]);
#pragma unroll
          for (int p = 0; p < PAIRS; ++p) {
            o[i][p] = fma2(make_float2(w.x, w.x), vf[0][p], o[i][p]);
            o[i][p] = fma2(make_float2(w.y, w.y), vf[1][p], o[i][p]);
            o[i][p] = fma2(make_float2(w.z, w.z), vf[2][p], o[i][p]);
            o[i][p] = fma2(make_float2(w.w, w.w), vf[3][p], o[i][p]);
          }
        }
      }
      __syncwarp();
    }
  }

  // ------------------------------------------------------------------ survivors to their places in the cache
  if (sp.ctas > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  {
    const int share = (n_keep + sp.ctas - 1) / sp.ctas, r0 = rank * share, r1 = min(n_keep, r0 + share);
#pragma unroll 2
    for (int v = r0 * PIECES + tid; v < r1 * PIECES; v += kStepThreads) {
      const int r = v / PIECES, c = v % PIECES, src = list[r];
      // stored rows that stay where they are need not be touched
      if ((src != r || src >= stored) && dbg_ok(src >= r && src < cand && r < a.cap[ctx], a.status, 14)) {
        *reinterpret_cast<float4*>(kc + (size_t)r * D + c * 4) = *reinterpret_cast<const float4*>(ks + src * KF + c * 4);
        *reinterpret_cast<float4*>(vc + (size_t)r * D + c * 4) = *reinterpret_cast<const float4*>(vs + src * D + c * 4);
        if (c == 0) a.pos_plane[off + r] = evicts ? pos[src] : a.pos_base + (src - stored);
      }
    }
  }

  // ------------------------------------------------------------------ merge of the warps that share a query tile
  reduce8(l, [](float x, float y) { return x + y; });
  __syncthreads();                              // nothing reads the keys any more
  float* ob = ks + (size_t)warp * kRows * D;
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    if (lane == i) row_ml[warp][i] = make_float2(m[i], l[i]);
#pragma unroll
    for (int p = 0; p < PAIRS; ++p) *reinterpret_cast<float2*>(ob + i * D + 2 * lane + 64 * p) = o[i][p];
  }
  __syncthreads();
  // a form per number of warps, so that all loads of a row are in flight at once
  auto combine = [&](auto splits_c) {
    constexpr int S = decltype(splits_c)::value;
#pragma unroll 1
    for (int v = tid; v < sp.tiles * kRows * PIECES; v += kStepThreads) {
      const int row = v / PIECES, c = v % PIECES, r = row % kRows, w0 = row / kRows * S;
      if (q_first + row >= n_new) break;
      float2 ml[S];
      float4 f[S], acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float top = -INFINITY, sum = 0.f;
#pragma unroll
      for (int w = 0; w < S; ++w) {
        ml[w] = row_ml[w0 + w][r];
        f[w] = *reinterpret_cast<const float4*>(ks + ((size_t)(w0 + w) * kRows + r) * D + c * 4);
      }
#pragma unroll
      for (int w = 0; w < S; ++w) top = fmaxf(top, ml[w].x);
#pragma unroll
      for (int w = 0; w < S; ++w) {
        const float wt = exp2f(ml[w].x - top);  // 0 for a warp without keys
        sum = fmaf(wt, ml[w].y, sum);
        acc.x = fmaf(wt, f[w].x, acc.x);
        acc.y = fmaf(wt, f[w].y, acc.y);
        acc.z = fmaf(wt, f[w].z, acc.z);
        acc.w = fmaf(wt, f[w].w, acc.w);
      }
      const float inv = 1.f / sum;
      *reinterpret_cast<float4*>(out + ((size_t)bh * n_new + q_first + row) * D + c * 4) =
          make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
    }
  };
  if (sp.log_splits == 3) combine(std::integral_constant<int, 8>());
  else if (sp.log_splits == 2) combine(std::integral_constant<int, 4>());
  else if (sp.log_splits == 1) combine(std::integral_constant<int, 2>());
  else combine(std::integral_constant<int, 1>());
}

template <int D>
int launch_t(const StepArgs& a, const void* q, const void* k_new, const void* v_new, void* out, cudaStream_t st) {
  const int heads = a.batch * a.n_heads, tiles = (a.n_new + kRows - 1) / kRows;
  const int cand = std::max(a.heads_of[0] ? a.cand[0] : 0, a.heads_of[1] ? a.cand[1] : 0);
  const int ranked = std::max(a.trig[0] ? a.cand[0] : 0, a.trig[1] ? a.cand[1] : 0);
  if (cand > (ranked ? kMaxCand : kMaxAppend) || (!ranked && a.n_new < kMinAppend) || tiles > kMaxTiles * kMaxCtas) return 0;
  StepShape s;
  s.rows = (cand + 3) / 4 * 4;
  const StepSizes sizes{D, a.n_new, a.heads_of, a.cand, a.kept, a.trig, sm_count()};
  auto go = [&](auto kern) {
    if (!allow_dynamic_smem(kern, kSmemCta)) return -1;
    const auto bytes = [](const StepShape& of) -> size_t { return Layout<D>(of.rows, of.tiles).total; };
    const auto places = [&](int ctas, size_t smem) { return cluster_places(reinterpret_cast<const void*>(kern), ctas, kStepThreads, smem); };
    if (!step_shape_f32(sizes, s, tiles, bytes, places)) return 0;
    return launch_step<float>(kern, a, s, bytes(s), q, k_new, v_new, out, st);
  };
  if (ranked <= 2 * kKeyWarps * kKeys) return go(step_small_f32_kernel<D, 2>);
  if constexpr (D == 64) {                      // at head_dim 128 shared memory holds fewer rows than four turns rank
    if (ranked > 4 * kKeyWarps * kKeys) return go(step_small_f32_kernel<D, kMaxTurns>);
  }
  return go(step_small_f32_kernel<D, 4>);
}

}  // namespace

int launch_step_small_f32(const StepArgs& a, const void* q, const void* k_new, const void* v_new, void* out, cudaStream_t st) {
  return a.head_dim == 128 ? launch_t<128>(a, q, k_new, v_new, out, st) : launch_t<64>(a, q, k_new, v_new, out, st);
}

}  // namespace hack
