// Final-scale merge of contextual heads (the sentence after Eq. 10): the entries that the last
// step discards are folded into their nearest retained counterparts by similarity-weighted
// averaging.  Reading implemented here (the paper leaves all of it open): nearness = cosine
// similarity between keys, counterpart = the retained key with the largest similarity (lowest index
// among equals), weight w = max(similarity, 0), and for a retained entry c with assigned set E_c
//   k_c <- (k_c + sum_e w_e k_e) / (1 + sum_e w_e),   v_c likewise with the same weights.
// bf16 caches only.  Around the compaction of that step:
//   before it (the discarded rows are still in place):
//     merge_evicted_index_kernel  complement of the ascending kept list, per head
//     merge_prepare_kernel        copies the discarded K, V rows to scratch planes and takes the
//                                 inverse norms of the discarded and of the retained keys
//   after it (the retained rows are contiguous in the cache plane):
//     merge_assign_kernel         S = E K^T on tcgen05, discarded rows on the TMEM lanes: a thread
//                                 owns one discarded key and keeps the running arg-max of
//                                 S[e, c] / |k_c| over the retained tiles
//     merge_apply_kernel          a CTA sifts the assignments for its 64 retained rows, a warp adds the
//                                 entries assigned to its 8 in ascending order (no atomics: the
//                                 result does not depend on scheduling)
// Every mbarrier wait is bounded; on expiry the CTA raises the status word and winds down.
#include <cuda.h>

#include <type_traits>

#include "hack_internal.h"
#include "tc_ptx.cuh"

namespace hack {
namespace {

using namespace ptx;

constexpr int kIdxThreads = 1024;
constexpr int kPrepThreads = 256;
constexpr int kPrepRows = 8;             // entries per warp
constexpr int kAssignThreads = 192;
constexpr int kTileM = 128;              // discarded rows per CTA, retained rows per tile
constexpr int kRing = 2;
constexpr int kApplyThreads = 256;
constexpr int kApplyRowsPerWarp = 8;     // retained rows per warp (64 per CTA)
constexpr int kApplyChunk = 4096;        // discarded entries a CTA looks through at a time
constexpr int kApplyHits = 256;          // entries a warp lists before it works them off
constexpr uint32_t kMergeDrainSpins = 1u << 22;

// ---------------------------------------------------------------- complement of the kept list
// The kept list becomes a bitmap in shared memory, a window of candidates at a time; a thread owns one
// word of 32 candidates, a prefix sum over the words' zero bits gives every word its place.
__global__ void __launch_bounds__(kIdxThreads)
merge_evicted_index_kernel(const StepArgs a, const MergeScratch ms, const int32_t* __restrict__ idx) {
  pdl_wait();
  const int bh = blockIdx.x;
  if (!a.is_ctx[bh % a.n_heads]) return;
  const int cand = a.cand[1], kept = a.kept[1];
  const int32_t* list = idx + (size_t)bh * a.kept_stride;
  int32_t* out = ms.ev_idx + (size_t)bh * ms.stride;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ uint32_t bits[kIdxThreads];
  __shared__ int warp_sums[32];
  int placed = 0;                                             // entries of the windows before this one
  for (int w0 = 0; w0 < cand; w0 += 32 * kIdxThreads) {
    bits[tid] = 0;
    __syncthreads();
    for (int r = tid; r < kept; r += kIdxThreads) {
      const int j = list[r] - w0;
      if (j >= 0 && j < 32 * kIdxThreads) atomicOr(&bits[j >> 5], 1u << (j & 31));
    }
    __syncthreads();
    const int left = cand - (w0 + 32 * tid);                  // candidates from this word on
    uint32_t gone = left >= 32 ? ~bits[tid] : left > 0 ? ~bits[tid] & ((1u << left) - 1u) : 0u;
    const int n = __popc(gone);
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < 32; ++w) {
      const int x = warp_sums[w];
      if (w < warp) before += x;
      total += x;
    }
    int pos = placed + before + incl - n;
    while (gone) {
      out[pos++] = w0 + 32 * tid + __ffs(gone) - 1;
      gone &= gone - 1;
    }
    placed += total;
    __syncthreads();
  }
}

// ---------------------------------------------------------------- scratch copies and inverse norms
// Bound by memory latency: a warp takes kPrepRows entries and has their rows in flight together (one
// entry per warp: 39 us for 16 heads of 6 200 candidates x 128, now 24).
template <int D>
__global__ void __launch_bounds__(kPrepThreads)
merge_prepare_kernel(const StepArgs a, const MergeScratch ms, const int32_t* __restrict__ idx,
                     const __nv_bfloat16* __restrict__ k_new, const __nv_bfloat16* __restrict__ v_new) {
  pdl_wait();
  const int bh = blockIdx.y;
  if (!a.is_ctx[bh % a.n_heads]) return;
  const int stored = a.stored[1], kept = a.kept[1], n_evict = a.cand[1] - kept;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = (blockIdx.x * (kPrepThreads / 32) + warp) * kPrepRows;
  const int n = min(kPrepRows, n_evict + kept - r0);
  if (n <= 0) return;
  constexpr int E = D / 32;                                   // bf16 elements per lane
  using Vec = typename std::conditional<E == 4, uint2, uint32_t>::type;
  int mine = 0;                                               // lane u holds entry r0 + u
  if (lane < n) {
    const int r = r0 + lane;
    mine = r < n_evict ? ms.ev_idx[(size_t)bh * ms.stride + r] : idx[(size_t)bh * a.kept_stride + (r - n_evict)];
  }
  Vec kv[kPrepRows] = {}, vv[kPrepRows] = {};
#pragma unroll
  for (int u = 0; u < kPrepRows; ++u) {
    const int j = __shfl_sync(0xffffffffu, mine, u);
    if (u < n) {
      const size_t src_row = j < stored ? (size_t)a.row_off[bh] + j : (size_t)bh * a.n_new + (j - stored);
      kv[u] = reinterpret_cast<const Vec*>((j < stored ? static_cast<const __nv_bfloat16*>(a.k_plane) : k_new) + src_row * D)[lane];
      if (r0 + u < n_evict)
        vv[u] = reinterpret_cast<const Vec*>((j < stored ? static_cast<const __nv_bfloat16*>(a.v_plane) : v_new) + src_row * D)[lane];
    }
  }
  float s[kPrepRows];
#pragma unroll
  for (int u = 0; u < kPrepRows; ++u) {
    const __nv_bfloat16* ke = reinterpret_cast<const __nv_bfloat16*>(&kv[u]);
    s[u] = 0.f;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const float x = __bfloat162float(ke[i]);
      s[u] = fmaf(x, x, s[u]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int u = 0; u < kPrepRows; ++u) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
#pragma unroll
  for (int u = 0; u < kPrepRows; ++u) {
    const int r = r0 + u;
    if (u >= n) break;
    const float inv = s[u] > 0.f ? 1.f / sqrtf(s[u]) : 0.f;
    if (r < n_evict) {
      const size_t dst = ((size_t)bh * ms.stride + r) * D;
      reinterpret_cast<Vec*>(ms.ev_k + dst)[lane] = kv[u];
      reinterpret_cast<Vec*>(ms.ev_v + dst)[lane] = vv[u];
      if (lane == 0) ms.ev_inv_norm[(size_t)bh * ms.stride + r] = inv;
    } else if (lane == 0) {
      ms.kept_inv_norm[(size_t)bh * a.kept_stride + (r - n_evict)] = inv;
    }
  }
}

// ---------------------------------------------------------------- nearest retained key on the tensor cores
struct AssignBars {
  uint64_t e_full;
  uint64_t k_full[kRing], k_empty[kRing];
  uint64_t acc_full[2], acc_free[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
};

__device__ __forceinline__ bool merge_wait(uint64_t* bar, uint32_t parity, AssignBars* b, int* status, int code, long long limit) {
  const uint32_t addr = smem_u32(bar);
  const long long t0 = clock64();
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait(addr, parity)) return true;
    if ((it & 63u) == 63u) {
      if (*reinterpret_cast<volatile int*>(&b->abort_flag)) return false;
      if (clock64() - t0 > limit) break;
    }
  }
  *reinterpret_cast<volatile int*>(&b->abort_flag) = 1;
  atomicExch(status, code);
  return false;
}

template <int D>
__global__ void __launch_bounds__(kAssignThreads)
merge_assign_kernel(const __grid_constant__ CUtensorMap tm_e, const __grid_constant__ CUtensorMap tm_k,
                    const StepArgs a, const MergeScratch ms) {
  constexpr int SUB = D / 64;
  constexpr uint32_t SUB_BYTES = kTileM * 128;
  constexpr uint32_t TILE_BYTES = SUB * SUB_BYTES;

  pdl_wait();
  const int bh = blockIdx.y, eb = blockIdx.x;
  if (!a.is_ctx[bh % a.n_heads]) return;
  const int kept = a.kept[1], n_evict = a.cand[1] - kept;
  if (eb * kTileM >= n_evict) return;
  const int n_kt = (kept + kTileM - 1) / kTileM;

  extern __shared__ unsigned char smem_dyn[];
  const uint32_t raw = smem_u32(smem_dyn);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_dyn + (base - raw);
  const uint32_t e_sm = base;
  const uint32_t k_sm = base + TILE_BYTES;
  AssignBars* bars = reinterpret_cast<AssignBars*>(sm + (1 + kRing) * TILE_BYTES);
  __shared__ __align__(16) float inv_c[4][2][kTileM];        // 1 / |k_c| of the retained tile in accumulator b

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    mbar_init(smem_u32(&bars->e_full), 1);
    for (int s = 0; s < kRing; ++s) { mbar_init(smem_u32(&bars->k_full[s]), 1); mbar_init(smem_u32(&bars->k_empty[s]), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&bars->acc_full[b]), 1); mbar_init(smem_u32(&bars->acc_free[b]), kTileM / 32); }
    mbar_init(smem_u32(&bars->drain), 1);
    bars->abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bars->tmem_base), 2 * kTileM);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      prefetch_tensormap(&tm_e);
      prefetch_tensormap(&tm_k);
      {
        const uint32_t bar = smem_u32(&bars->e_full);
        mbar_expect_tx(bar, TILE_BYTES);
        for (int s = 0; s < SUB; ++s) tma_load_2d(e_sm + s * SUB_BYTES, &tm_e, s * 64, bh * ms.stride + eb * kTileM, bar);
      }
      int issued = 0;
      bool ok = true;
      for (int t = 0; t < n_kt; ++t) {
        const int s = t % kRing;
        ok = merge_wait(&bars->k_empty[s], ((t / kRing) & 1) ^ 1, bars, a.status, 41, a.wait_cycles);
        if (!ok) break;
        const uint32_t bar = smem_u32(&bars->k_full[s]);
        mbar_expect_tx(bar, TILE_BYTES);
        for (int x = 0; x < SUB; ++x)
          tma_load_2d(k_sm + s * TILE_BYTES + x * SUB_BYTES, &tm_k, x * 64, a.row_off[bh] + t * kTileM, bar);
        ++issued;
      }
      if (!ok) {
        for (uint32_t it = 0; it < kMergeDrainSpins && !mbar_try_wait(smem_u32(&bars->e_full), 0); ++it) {}
        for (int i = max(0, issued - kRing); i < issued; ++i) {
          const uint32_t bar = smem_u32(&bars->k_full[i % kRing]);
          for (uint32_t it = 0; it < kMergeDrainSpins && !mbar_try_wait(bar, (i / kRing) & 1); ++it) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t IDESC = idesc_bf16_f32(kTileM, kTileM, 0);     // A = discarded keys, B = retained keys, K-major
      const uint64_t e_desc = smem_desc_sw128(e_sm, 16, 1024);
      bool ok = merge_wait(&bars->e_full, 0, bars, a.status, 42, a.wait_cycles);
      for (int t = 0; t < n_kt && ok; ++t) {
        const int s = t % kRing, b = t & 1;
        ok = merge_wait(&bars->k_full[s], (t / kRing) & 1, bars, a.status, 43, a.wait_cycles);
        if (ok) ok = merge_wait(&bars->acc_free[b], ((t >> 1) & 1) ^ 1, bars, a.status, 44, a.wait_cycles);
        if (!ok) break;
        tc_fence_after();
        const uint64_t k_desc = smem_desc_sw128(k_sm + s * TILE_BYTES, 16, 1024);
        if constexpr (D == 128) mma_ss_chain8(tmem + b * kTileM, e_desc, k_desc, IDESC, 0);
        else mma_ss_chain4(tmem + b * kTileM, e_desc, k_desc, IDESC, 0);
        mma_commit(smem_u32(&bars->k_empty[s]));
        mma_commit(smem_u32(&bars->acc_full[b]));
      }
    }
  } else {
    // ------------------------------------------------------------------ consumers
    const int quad = warp & 3;                                // TMEM lane quadrant this warp may read
    const int my_row = eb * kTileM + quad * 32 + lane;        // discarded entry this thread owns
    const uint32_t t_lane = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    // Bound by the latency of a reading warp's chain of instructions (0.9 us per tile and CTA, 1.3 with two on the SM):
    // the largest of 32 columns is formed as a tree, the 32 columns that hold the best one so far are kept
    // without a branch, and which of them it is is looked up once, at the end.  The next columns and norms are
    // on their way meanwhile.  (Four columns at a time, looked up at once: 62 us, now 55.  Two tiles of discarded rows that share
    // the retained tiles, or eight reading warps per tile: no faster.)
    float best = -INFINITY;
    int arg = 0;                                              // first of the 32 columns with the best one ...
    float2 won[16];                                           // ... and those columns
#pragma unroll
    for (int i = 0; i < 16; ++i) won[i] = make_float2(-INFINITY, -INFINITY);
    int last = 0;
    bool ok = true, single = false;
    // Every warp keeps its own copy of a tile's norms, so that the warps do not meet inside the loop.
    float inv[4];
    auto fetch = [&](int t) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = t * kTileM + u * 32 + lane;
        inv[u] = c < kept ? ms.kept_inv_norm[(size_t)bh * a.kept_stride + c] : 0.f;
      }
    };
    fetch(0);
    for (int t = 0; t < n_kt; ++t) {
      const int b = t & 1;
      float* inv_tile = inv_c[warp - 2][b];
#pragma unroll
      for (int u = 0; u < 4; ++u) inv_tile[u * 32 + lane] = inv[u];
      __syncwarp();
      fetch(t + 1);
      ok = __all_sync(0xffffffffu, merge_wait(&bars->acc_full[b], (t >> 1) & 1, bars, a.status, 45, a.wait_cycles));
      if (!ok) break;
      tc_fence_after();
      const int n_valid = min(kTileM, kept - t * kTileM);
      uint32_t acc2[2][32];                                    // the next 32 columns are on their way under these
      tmem_ld32(t_lane + b * kTileM, acc2[0]);
#pragma unroll
      for (int ch = 0; ch < kTileM / 32; ++ch) {
        uint32_t* acc = acc2[ch & 1];
        tmem_wait_ld();
        if (ch < kTileM / 32 - 1) {
          tmem_ld32(t_lane + b * kTileM + (ch + 1) * 32, acc2[(ch + 1) & 1]);
        } else {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&bars->acc_free[b]));
        }
        if (n_valid == kTileM) {
          float2 v[16];
          float top4[4];
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const float4 ic = *reinterpret_cast<const float4*>(&inv_tile[ch * 32 + 2 * i]);
            v[i] = mul2(make_float2(__uint_as_float(acc[2 * i]), __uint_as_float(acc[2 * i + 1])), make_float2(ic.x, ic.y));
            v[i + 1] = mul2(make_float2(__uint_as_float(acc[2 * i + 2]), __uint_as_float(acc[2 * i + 3])), make_float2(ic.z, ic.w));
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            top4[u] = fmaxf(v[4 * u].x, v[4 * u].y);
#pragma unroll
            for (int i = 1; i < 4; ++i) top4[u] = max3(top4[u], v[4 * u + i].x, v[4 * u + i].y);
          }
          const float top = fmaxf(fmaxf(top4[0], top4[1]), fmaxf(top4[2], top4[3]));
          // strict comparison, and of the equal columns the lowest: the lowest index wins among equals
          const bool more = top > best;
          best = more ? top : best;
          arg = more ? t * kTileM + ch * 32 : arg;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            won[i].x = more ? v[i].x : won[i].x;
            won[i].y = more ? v[i].y : won[i].y;
          }
        } else if (ch * 32 < n_valid) {
          if (ch == 0) {                                      // the last tile, a column at a time: from here on arg is the column itself
#pragma unroll
            for (int i = 15; i >= 0; --i) {
              if (won[i].y == best) last = arg + 2 * i + 1;
              if (won[i].x == best) last = arg + 2 * i;
            }
            arg = last;
            single = true;
          }
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float val = __uint_as_float(acc[i]) * inv_tile[ch * 32 + i];
            if (ch * 32 + i < n_valid && val > best) {
              best = val;
              arg = t * kTileM + ch * 32 + i;
            }
          }
        }
      }
    }
    if (!single) {
#pragma unroll
      for (int i = 15; i >= 0; --i) {
        if (won[i].y == best) last = arg + 2 * i + 1;
        if (won[i].x == best) last = arg + 2 * i;
      }
      arg = last;
    }
    if (ok && my_row < n_evict) {
      const size_t o = (size_t)bh * ms.stride + my_row;
      ms.assign[o] = arg;
      ms.weight[o] = fmaxf(best * ms.ev_inv_norm[o], 0.f);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (lane == 0 && bars->abort_flag) {             // what was issued gets a bounded chance to end, so that tensor memory can be freed
      mma_commit(smem_u32(&bars->drain));
      for (uint32_t it = 0; it < kMergeDrainSpins && !mbar_try_wait(smem_u32(&bars->drain), 0); ++it) {}
    }
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 2 * kTileM);
  }
}

// ---------------------------------------------------------------- weighted average into the retained rows
// A warp owns kApplyRowsPerWarp consecutive retained rows.  The discarded entries are sifted twice: every warp
// looks through an eighth of them and lists those assigned to any row of the CTA, then every warp looks through these
// lists for its own rows.  The entries found are fetched four at a time and added to the rows' fp32 accumulators in
// shared memory.  Entries are taken in ascending order, so a row's sum has one fixed order of additions.
// Bound by latency.  (With every warp walking all entries, 32 passes of a shuffled prefix sum for 4 096 entries, 16 heads x
// 2 104 retained rows took 42.7 us; now 34.8.)
template <int D>
__global__ void __launch_bounds__(kApplyThreads, 2)
merge_apply_kernel(const StepArgs a, const MergeScratch ms) {
  pdl_wait();
  const int bh = blockIdx.y;
  if (!a.is_ctx[bh % a.n_heads]) return;
  const int kept = a.kept[1], n_evict = a.cand[1] - kept;
  constexpr int E = D / 32;
  constexpr int R = kApplyRowsPerWarp;
  constexpr int kWarps = kApplyThreads / 32;
  using Vec = typename std::conditional<E == 4, uint2, uint32_t>::type;
  extern __shared__ __align__(16) unsigned char apply_smem[];
  float* acc_all = reinterpret_cast<float*>(apply_smem);                 // [warp][row][K | V][D]
  float* den_all = acc_all + kWarps * R * 2 * D;                          // [warp][row]
  constexpr int kPart = kApplyChunk / kWarps;                             // entries of a chunk that a warp sifts
  int* s_entry = reinterpret_cast<int*>(den_all + kWarps * R);            // [warp][kPart]: entry * rows of the CTA + row
  float* s_weight = reinterpret_cast<float*>(s_entry + kApplyChunk);      // [warp][kPart]
  int* s_hits = reinterpret_cast<int*>(s_weight + kApplyChunk);           // [warp][kApplyHits]: places in s_entry
  int* s_found = s_hits + kWarps * kApplyHits;                            // [warp]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  const int b0 = blockIdx.x * kWarps * R, c0 = b0 + warp * R;
  float* acc = acc_all + warp * R * 2 * D;
  float* den = den_all + warp * R;
  for (int i = lane; i < R * 2 * D; i += 32) acc[i] = 0.f;
  if (lane < R) den[lane] = 0.f;
  int* hits = s_hits + warp * kApplyHits;                       // entries of this chunk assigned to this warp's rows
  // adds the listed entries, four at a time: their rows are fetched together (the latencies overlap), then added in order
  auto flush = [&](int base, int n_hits) {
    for (int h0 = 0; h0 < n_hits; h0 += 4) {
      Vec kv[4], vv[4];
      int at[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (h0 + u < n_hits) {
          at[u] = hits[h0 + u];
          const size_t row = ((size_t)bh * ms.stride + base + s_entry[at[u]] / (kWarps * R)) * D;
          kv[u] = reinterpret_cast<const Vec*>(ms.ev_k + row)[lane];
          vv[u] = reinterpret_cast<const Vec*>(ms.ev_v + row)[lane];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (h0 + u < n_hits) {
          const int r = s_entry[at[u]] % R;                     // (a warp's rows start at a multiple of R)
          const float w = s_weight[at[u]];
          const __nv_bfloat16* ke = reinterpret_cast<const __nv_bfloat16*>(&kv[u]);
          const __nv_bfloat16* ve = reinterpret_cast<const __nv_bfloat16*>(&vv[u]);
          float* ak = acc + (r * 2) * D + lane * E;
          float* av = ak + D;
#pragma unroll
          for (int x = 0; x < E; ++x) {
            ak[x] = fmaf(w, __bfloat162float(ke[x]), ak[x]);
            av[x] = fmaf(w, __bfloat162float(ve[x]), av[x]);
          }
          if (lane == 0) den[r] += w;
        }
      }
    }
    __syncwarp();
  };
  for (int base = 0; base < n_evict; base += kApplyChunk) {
    const int n = min(kApplyChunk, n_evict - base);
    __syncthreads();                                            // the lists of the chunk before have been read
    int found = 0;
#pragma unroll 1
    for (int i0 = warp * kPart; i0 < min(n, (warp + 1) * kPart); i0 += 256) {
      // (kPart is a multiple of 256: a group never reaches into the next warp's part)
      uint32_t row[8];
      float w[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + u * 32 + lane;
        row[u] = i < n ? (uint32_t)(ms.assign[(size_t)bh * ms.stride + base + i] - b0) : 0xffffffffu;
        w[u] = i < n ? ms.weight[(size_t)bh * ms.stride + base + i] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const bool mine = row[u] < (uint32_t)(kWarps * R);
        const uint32_t some = __ballot_sync(0xffffffffu, mine);
        if (mine) {
          const int at = warp * kPart + found + __popc(some & below);
          s_entry[at] = (i0 + u * 32 + lane) * (kWarps * R) + (int)row[u];
          s_weight[at] = w[u];
        }
        found += __popc(some);
      }
    }
    if (lane == 0) s_found[warp] = found;
    __syncthreads();
    if (c0 >= kept) continue;
    // this warp's rows, in ascending order of the entries; its list is worked off when it fills and at the end
    int n_hits = 0;
#pragma unroll 1
    for (int part = 0; part < kWarps; ++part) {
      const int listed = s_found[part];
#pragma unroll 1
      for (int i0 = 0; i0 < listed; i0 += 32) {
        const int at = part * kPart + i0 + lane;
        const bool mine = i0 + lane < listed && s_entry[at] % (kWarps * R) / R == warp;
        const uint32_t some = __ballot_sync(0xffffffffu, mine);
        if (n_hits + 32 > kApplyHits) {
          __syncwarp();
          flush(base, n_hits);
          n_hits = 0;
        }
        if (mine) hits[n_hits + __popc(some & below)] = at;
        n_hits += __popc(some);
      }
    }
    __syncwarp();
    flush(base, n_hits);
  }
  __syncwarp();
  // the rows that received something: all of them are fetched before any is written back
  Vec kv[R], vv[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (c0 + r < kept && den[r] != 0.f) {
      const size_t row = ((size_t)a.row_off[bh] + c0 + r) * D;
      kv[r] = reinterpret_cast<const Vec*>(static_cast<const __nv_bfloat16*>(a.k_plane) + row)[lane];
      vv[r] = reinterpret_cast<const Vec*>(static_cast<const __nv_bfloat16*>(a.v_plane) + row)[lane];
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (c0 + r < kept && den[r] != 0.f) {                      // else nothing was assigned: the row keeps its bits
      const float inv = 1.f / (1.f + den[r]);
      __nv_bfloat16* ke = reinterpret_cast<__nv_bfloat16*>(&kv[r]);
      __nv_bfloat16* ve = reinterpret_cast<__nv_bfloat16*>(&vv[r]);
      const float* ak = acc + (r * 2) * D + lane * E;
      const float* av = ak + D;
#pragma unroll
      for (int x = 0; x < E; ++x) {
        ke[x] = __float2bfloat16_rn((__bfloat162float(ke[x]) + ak[x]) * inv);
        ve[x] = __float2bfloat16_rn((__bfloat162float(ve[x]) + av[x]) * inv);
      }
      const size_t row = ((size_t)a.row_off[bh] + c0 + r) * D;
      reinterpret_cast<Vec*>(static_cast<__nv_bfloat16*>(a.k_plane) + row)[lane] = kv[r];
      reinterpret_cast<Vec*>(static_cast<__nv_bfloat16*>(a.v_plane) + row)[lane] = vv[r];
    }
  }
}

template <int D>
size_t apply_smem_bytes() {
  return ((size_t)(kApplyThreads / 32) * (kApplyRowsPerWarp * (2 * D + 1) + kApplyHits + 1) + 2 * kApplyChunk) * sizeof(float);
}

template <int D>
size_t assign_smem_bytes() {
  return 1024 + (1 + kRing) * (size_t)(D / 64) * kTileM * 128 + sizeof(AssignBars) + 64;
}

}  // namespace

int launch_merge_prepare(const StepArgs& a, const MergeScratch& ms, const int32_t* idx, bool listed, const void* k_new,
                         const void* v_new, cudaStream_t st) {
  const int bh = a.batch * a.n_heads;
  const int rows = a.cand[1];                                  // discarded + retained entries of a contextual head
  if (!listed) launch_k(merge_evicted_index_kernel, bh, kIdxThreads, 0, st, a, ms, idx);
  constexpr int kEntries = kPrepThreads / 32 * kPrepRows;      // per CTA
  const dim3 grid((rows + kEntries - 1) / kEntries, bh);
  const __nv_bfloat16* kn = static_cast<const __nv_bfloat16*>(k_new);
  const __nv_bfloat16* vn = static_cast<const __nv_bfloat16*>(v_new);
  if (a.head_dim == 128) launch_k(merge_prepare_kernel<128>, grid, kPrepThreads, 0, st, a, ms, idx, kn, vn);
  else launch_k(merge_prepare_kernel<64>, grid, kPrepThreads, 0, st, a, ms, idx, kn, vn);
  return launched(listed ? 1 : 2);
}

int launch_merge_finish(const StepArgs& a, const MergeScratch& ms, cudaStream_t st) {
  const int bh = a.batch * a.n_heads;
  const int kept = a.kept[1], n_evict = a.cand[1] - kept;
  const CUtensorMap& te = *static_cast<const CUtensorMap*>(ms.ev_map);
  const CUtensorMap& tk = *static_cast<const CUtensorMap*>(a.k_map);
  const dim3 g_assign((n_evict + kTileM - 1) / kTileM, bh);
  constexpr int kRowsPerCta = (kApplyThreads / 32) * kApplyRowsPerWarp;
  const dim3 g_apply((kept + kRowsPerCta - 1) / kRowsPerCta, bh);
  if (a.head_dim == 128) {
    if (!allow_dynamic_smem(merge_assign_kernel<128>, assign_smem_bytes<128>())) return -1;
    launch_k(merge_assign_kernel<128>, g_assign, kAssignThreads, assign_smem_bytes<128>(), st, te, tk, a, ms);
    if (!allow_dynamic_smem(merge_apply_kernel<128>, apply_smem_bytes<128>())) return -1;
    launch_k(merge_apply_kernel<128>, g_apply, kApplyThreads, apply_smem_bytes<128>(), st, a, ms);
  } else {
    if (!allow_dynamic_smem(merge_assign_kernel<64>, assign_smem_bytes<64>())) return -1;
    launch_k(merge_assign_kernel<64>, g_assign, kAssignThreads, assign_smem_bytes<64>(), st, te, tk, a, ms);
    if (!allow_dynamic_smem(merge_apply_kernel<64>, apply_smem_bytes<64>())) return -1;
    launch_k(merge_apply_kernel<64>, g_apply, kApplyThreads, apply_smem_bytes<64>(), st, a, ms);
  }
  return launched(2);
}

}  // namespace hack
