// Attention variance of every head (Eq. 6, offline head classification) for bf16 caches:
//   sigma = sum_j Var_i A[i, j],  A = Softmax(sm_scale * Q K^T), rows i = the step's queries,
//   columns j = the head's cached keys, variance over the queries (population variance).
//
// The row statistics of the softmax (reference maximum m_i and sum l_i of every query) come from the
// attention kernel, which has them anyway; this file turns them into the column statistics.  A CTA
// owns two blocks of 128 keys of one head and walks over all query tiles:
//   warp 0    : TMA producer (the key blocks once, the query tiles through a ring)
//   warp 1    : tcgen05.mma issuer; S^T = K_blk Q_tile^T, keys on the 128 TMEM lanes, queries on
//               128 columns, two accumulators per key block so that the next MMA runs under the read-out
//   warps 2-9 : consumers of the first key block, warps 10-17 of the second; two threads own key r: each reads
//               its 64 of the 128 logits with tcgen05.ld, forms p = exp2(c z - c m_i - log2 l_i) and adds p and
//               p^2 to two registers
// so the sums over the queries stay inside a thread and nothing of size N x T is stored.  At the
// end the two have Var_i A[i, j] = sum p^2 / N - (sum p / N)^2 of their key; the CTA adds its 128
// variances and a second, tiny kernel adds the blocks of a head in a fixed order.  Bound by the special-function unit:
// 2 048 cycles for the two tiles of a step.  With one thread per key (two warps per scheduler, each waiting for its own
// tcgen05.ld and barriers) 32 heads x 4 096 queries x 10 521 keys took 472 us, some 3 150 cycles a step; now 451 us.
// Two blocks per CTA halve the query traffic: with one block per CTA (two CTAs per SM) the launch ran at the
// L2's rate of about 21 bytes per clock and SM.  32 heads x 4 096 queries x 10 521 keys x 128: 514 -> 482 us, short last blocks
// last in the order of the CTAs: -> 472 us.
// Every mbarrier wait is bounded; on expiry the CTA raises the status word and winds down.
#include <cuda.h>

#include "hack_internal.h"
#include "tc_ptx.cuh"

namespace hack {
namespace {

using namespace ptx;

constexpr int kVarSets = 2;             // key blocks per CTA
constexpr int kVarParts = 2;            // threads per key, each with its part of a tile's queries
constexpr int kVarWarps = 4 * kVarSets * kVarParts;   // consumers
constexpr int kVarThreads = 64 + 32 * kVarWarps;
constexpr int kVarTile = 128;            // keys per block, queries per tile
constexpr int kVarPart = kVarTile / kVarParts;
constexpr int kQStages = 3;
constexpr uint32_t kVarDrainSpins = 1u << 22;

struct VarBars {
  uint64_t k_full;
  uint64_t q_full[kQStages], q_empty[kQStages];
  uint64_t acc_full[kVarSets][2], acc_free[kVarSets][2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
};

__device__ __forceinline__ bool var_wait(uint64_t* bar, uint32_t parity, VarBars* b, int* status, int code, long long limit) {
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
__global__ void __launch_bounds__(kVarThreads, 1)
attn_colstats_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const StepArgs a, const float* __restrict__ row_stats, float* __restrict__ block_var,
                     int max_blocks) {
  constexpr int SUB = D / 64;
  constexpr uint32_t SUB_BYTES = kVarTile * 128;
  constexpr uint32_t TILE_BYTES = SUB * SUB_BYTES;

  pdl_wait();
  // All heads' first blocks come first and the last ones, which may be one block instead of two, last: 32 heads of 83 blocks
  // are 1 344 CTAs on 148 SMs, and a tenth round for twelve of them is short this way.
  const int bh = blockIdx.x, kb0 = blockIdx.y * kVarSets;
  const int len = a.kept[a.is_ctx[bh % a.n_heads]];
  if (kb0 * kVarTile >= len) return;
  const int n_sets = (kb0 + 1) * kVarTile < len ? 2 : 1;
  const int n_qt = (a.n_new + kVarTile - 1) / kVarTile;
  const float c = a.sm_scale * 1.4426950408889634f;

  extern __shared__ unsigned char smem_dyn[];
  const uint32_t raw = smem_u32(smem_dyn);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_dyn + (base - raw);
  const uint32_t k_sm = base;
  const uint32_t q_sm = base + kVarSets * TILE_BYTES;
  VarBars* bars = reinterpret_cast<VarBars*>(sm + (kVarSets + kQStages) * TILE_BYTES);
  __shared__ __align__(16) float stat[kVarWarps][2][kVarPart];   // -c m_i - log2 l_i of the query tile in accumulator b
  __shared__ float red[4 * kVarSets];
  __shared__ float2 other[kVarSets][kVarTile];                      // sums of the second thread of every key

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    mbar_init(smem_u32(&bars->k_full), 1);
    for (int s = 0; s < kQStages; ++s) { mbar_init(smem_u32(&bars->q_full[s]), 1); mbar_init(smem_u32(&bars->q_empty[s]), 1); }
    for (int i = 0; i < kVarSets; ++i)
      for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&bars->acc_full[i][b]), 1); mbar_init(smem_u32(&bars->acc_free[i][b]), 4 * kVarParts); }
    mbar_init(smem_u32(&bars->drain), 1);
    bars->abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bars->tmem_base), 2 * kVarSets * kVarTile);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      prefetch_tensormap(&tm_q);
      prefetch_tensormap(&tm_k);
      {
        const uint32_t bar = smem_u32(&bars->k_full);
        mbar_expect_tx(bar, n_sets * TILE_BYTES);
        for (int i = 0; i < n_sets; ++i)
          for (int s = 0; s < SUB; ++s)
            tma_load_2d(k_sm + i * TILE_BYTES + s * SUB_BYTES, &tm_k, s * 64, a.row_off[bh] + (kb0 + i) * kVarTile, bar);
      }
      int issued = 0;
      bool ok = true;
      for (int t = 0; t < n_qt; ++t) {
        const int s = t % kQStages;
        ok = var_wait(&bars->q_empty[s], ((t / kQStages) & 1) ^ 1, bars, a.status, 31, a.wait_cycles);
        if (!ok) break;
        const uint32_t bar = smem_u32(&bars->q_full[s]);
        mbar_expect_tx(bar, TILE_BYTES);
        for (int x = 0; x < SUB; ++x)
          tma_load_2d(q_sm + s * TILE_BYTES + x * SUB_BYTES, &tm_q, x * 64, bh * a.n_new + t * kVarTile, bar);
        ++issued;
      }
      if (!ok) {
        // give the copies already in flight a bounded chance to land before the CTA leaves
        for (uint32_t it = 0; it < kVarDrainSpins && !mbar_try_wait(smem_u32(&bars->k_full), 0); ++it) {}
        for (int i = max(0, issued - kQStages); i < issued; ++i) {
          const uint32_t bar = smem_u32(&bars->q_full[i % kQStages]);
          for (uint32_t it = 0; it < kVarDrainSpins && !mbar_try_wait(bar, (i / kQStages) & 1); ++it) {}
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t IDESC = idesc_bf16_f32(kVarTile, kVarTile, 0);      // A = keys, B = queries, both K-major
      bool ok = var_wait(&bars->k_full, 0, bars, a.status, 32, a.wait_cycles);
      for (int t = 0; t < n_qt && ok; ++t) {
        const int s = t % kQStages, b = t & 1;
        ok = var_wait(&bars->q_full[s], (t / kQStages) & 1, bars, a.status, 33, a.wait_cycles);
        const uint64_t q_desc = smem_desc_sw128(q_sm + s * TILE_BYTES, 16, 1024);
        for (int i = 0; i < n_sets && ok; ++i) {
          ok = var_wait(&bars->acc_free[i][b], ((t >> 1) & 1) ^ 1, bars, a.status, 34, a.wait_cycles);
          if (!ok) break;
          tc_fence_after();
          const uint64_t k_desc = smem_desc_sw128(k_sm + i * TILE_BYTES, 16, 1024);
          const uint32_t acc = tmem + (2 * i + b) * kVarTile;
          if constexpr (D == 128) mma_ss_chain8(acc, k_desc, q_desc, IDESC, 0);
          else mma_ss_chain4(acc, k_desc, q_desc, IDESC, 0);
          mma_commit(smem_u32(&bars->acc_full[i][b]));
        }
        if (ok) mma_commit(smem_u32(&bars->q_empty[s]));
      }
    }
  } else if ((warp - 2) / (4 * kVarParts) < n_sets) {
    // ------------------------------------------------------------------ consumers
    const int set = (warp - 2) / (4 * kVarParts), part = (warp - 2) / 4 % kVarParts, kb = kb0 + set;
    const int quad = warp & 3;                                // TMEM lane quadrant this warp may read
    const int key_row = quad * 32 + lane;                     // key of the block this thread owns
    const uint32_t t_lane = tmem + (static_cast<uint32_t>(quad * 32) << 16) + 2 * set * kVarTile + part * kVarPart;
    float2 sum_p[2] = {}, sum_p2[2] = {};                     // queries apart by their index modulo 4
    bool ok = true;
    // Statistics of a tile's queries, fetched one tile ahead; every warp keeps its own copy, so that the
    // warps do not meet inside the loop.  Queries past the end of the scale get weight 0: exp2(-inf) = 0.
    float2 ml[kVarPart / 32];
    auto fetch = [&](int t) {
#pragma unroll
      for (int u = 0; u < kVarPart / 32; ++u) {
        const int qi = t * kVarTile + part * kVarPart + u * 32 + lane;
        ml[u] = qi < a.n_new ? *reinterpret_cast<const float2*>(row_stats + ((size_t)bh * a.n_new + qi) * 2) : make_float2(INFINITY, 1.f);
      }
    };
    fetch(0);
    for (int t = 0; t < n_qt; ++t) {
      const int b = t & 1;
      float* st_tile = stat[warp - 2][b];
      // p = exp2(c z - c m - log2 l): the division is in the exponent
#pragma unroll
      for (int u = 0; u < kVarPart / 32; ++u) st_tile[u * 32 + lane] = -ml[u].x * c - __log2f(ml[u].y);
      __syncwarp();
      fetch(t + 1);
      ok = __all_sync(0xffffffffu, var_wait(&bars->acc_full[set][b], (t >> 1) & 1, bars, a.status, 35, a.wait_cycles));
      if (!ok) break;
      tc_fence_after();
      // the next 32 logits are on their way while the exponentials of these are formed
      uint32_t acc[2][32];
      tmem_ld32(t_lane + b * kVarTile, acc[0]);
#pragma unroll
      for (int ch = 0; ch < kVarPart / 32; ++ch) {
        tmem_wait_ld();
        if (ch + 1 < kVarPart / 32) {
          tmem_ld32(t_lane + b * kVarTile + (ch + 1) * 32, acc[(ch + 1) & 1]);
        } else {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&bars->acc_free[set][b]));
        }
        const uint32_t* z = acc[ch & 1];
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const float4 st = *reinterpret_cast<const float4*>(&st_tile[ch * 32 + i]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float2 x = fma2(make_float2(__uint_as_float(z[i + 2 * h]), __uint_as_float(z[i + 2 * h + 1])), make_float2(c, c),
                                  h == 0 ? make_float2(st.x, st.y) : make_float2(st.z, st.w));
            const float2 pr = make_float2(ex2(x.x), ex2(x.y));
            sum_p[h] = add2(sum_p[h], pr);
            sum_p2[h] = fma2(pr, pr, sum_p2[h]);
          }
        }
      }
    }
    // Var_i A[i, j] of this thread's key; keys past the end of the head count nothing (their sums
    // come from rows of another head and may have overflowed)
    const float inv_n = 1.f / (float)a.n_new;
    const float2 s1 = add2(sum_p[0], sum_p[1]), s2 = add2(sum_p2[0], sum_p2[1]);
    float sp = s1.x + s1.y, sp2 = s2.x + s2.y;
    if (part == 1) other[set][key_row] = make_float2(sp, ok ? sp2 : -1.f);   // < 0: this warp gave up
    asm volatile("bar.sync %0, %1;" ::"r"(1 + set), "n"(128 * kVarParts) : "memory");
    float var = 0.f;
    if (part == 0) {
      const float2 o = other[set][key_row];
      sp += o.x;
      sp2 += o.y;
      ok = __all_sync(0xffffffffu, ok && !(o.y < 0.f));
      if (ok && kb * kVarTile + key_row < len) {
        const float mean = sp * inv_n;
        var = fmaxf(fmaf(-mean, mean, sp2 * inv_n), 0.f);
      }
#pragma unroll
      for (int o2 = 16; o2 > 0; o2 >>= 1) var += __shfl_xor_sync(0xffffffffu, var, o2);
      if (lane == 0) red[4 * set + (warp - 2) % 4] = ok ? var : NAN;         // a warp that gave up poisons the block's sum
    }
    asm volatile("bar.sync %0, %1;" ::"r"(1 + set), "n"(128 * kVarParts) : "memory");
    if (part == 0 && (warp - 2) % 4 == 0 && lane == 0 && ok)
      block_var[(size_t)bh * max_blocks + kb] = (red[4 * set] + red[4 * set + 1]) + (red[4 * set + 2] + red[4 * set + 3]);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (lane == 0 && bars->abort_flag) {             // what was issued gets a bounded chance to end, so that tensor memory can be freed
      mma_commit(smem_u32(&bars->drain));
      for (uint32_t it = 0; it < kVarDrainSpins && !mbar_try_wait(smem_u32(&bars->drain), 0); ++it) {}
    }
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 2 * kVarSets * kVarTile);
  }
}

// sigma of one head = sum of its key blocks' variances, added in block order by one warp.
__global__ void __launch_bounds__(32)
attn_variance_finish_kernel(const StepArgs a, const float* __restrict__ block_var, int max_blocks,
                            float* __restrict__ sigma) {
  pdl_wait();
  const int bh = blockIdx.x, lane = threadIdx.x;
  const int len = a.kept[a.is_ctx[bh % a.n_heads]];
  const int n_blocks = (len + kVarTile - 1) / kVarTile;
  float s = 0.f;
  for (int kb = lane; kb < n_blocks; kb += 32) s += block_var[(size_t)bh * max_blocks + kb];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) sigma[bh] = s;
}

template <int D>
size_t var_smem_bytes() {
  return 1024 + (kVarSets + kQStages) * (size_t)(D / 64) * kVarTile * 128 + sizeof(VarBars) + 64;
}

}  // namespace

int launch_attention_variance(const StepArgs& a, const void* q, const float* row_stats, float* block_var,
                              int max_blocks, float* sigma, cudaStream_t st) {
  CUtensorMap tm_q;
  if (!make_rows_map(&tm_q, q, (uint64_t)a.batch * a.n_heads * a.n_new, a.head_dim)) {
    set_error("attention variance: cuTensorMapEncodeTiled failed for the queries");
    return -1;
  }
  const CUtensorMap& tk = *static_cast<const CUtensorMap*>(a.k_map);
  const int bh = a.batch * a.n_heads;
  const int longest = a.kept[0] > a.kept[1] ? a.kept[0] : a.kept[1];
  const int n_blocks = (longest + kVarTile - 1) / kVarTile;
  if (n_blocks > max_blocks) {
    set_error("attention variance: cache longer than the scratch area");
    return -1;
  }
  const dim3 grid(bh, (n_blocks + kVarSets - 1) / kVarSets);
  if (a.head_dim == 128) {
    if (!allow_dynamic_smem(attn_colstats_kernel<128>, var_smem_bytes<128>())) return -1;
    launch_k(attn_colstats_kernel<128>, grid, kVarThreads, var_smem_bytes<128>(), st, tm_q, tk, a, row_stats, block_var, max_blocks);
  } else {
    if (!allow_dynamic_smem(attn_colstats_kernel<64>, var_smem_bytes<64>())) return -1;
    launch_k(attn_colstats_kernel<64>, grid, kVarThreads, var_smem_bytes<64>(), st, tm_q, tk, a, row_stats, block_var, max_blocks);
  }
  launch_k(attn_variance_finish_kernel, bh, 32, 0, st, a, block_var, max_blocks, sigma);
  return launched(2);
}

}  // namespace hack
