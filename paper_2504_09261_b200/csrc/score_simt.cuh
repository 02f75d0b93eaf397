// The SIMT scoring body (Eq. 9 and the TOPK argument of Eq. 10-11) shared by the cache-based fp32
// path (score_kernels.cu) and the entry point without allocation (score_noalloc.cu).
//
// Pass 1: a CTA of 128 threads takes 128 candidate keys of one row-block, stages them and the (at
// most 32) observation rows in shared memory, forms the logits, stores them and publishes the
// (max, sum-exp) of every observation row over the chunk.  Pass 2: the chunk statistics of a
// row-block are merged into the statistics of the full softmax and every column is reduced:
// s_j = sum_i exp(z_ij - m_i) / l_i.  The callers differ only in where a key row, an observation
// row, a logit and a score live; they pass those as small functors.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "tc_ptx.cuh"

namespace hack {
namespace simt {

constexpr int kObs = 32;       // observation rows the kernels are built for
constexpr int kChunk = 128;    // candidate keys per CTA in pass 1 (= threads per CTA)

template <typename T> struct Elem;
template <> struct Elem<float> {
  static constexpr int kPerVec = 4;  // elements per 16 bytes
  __device__ static void unpack(const uint4& v, float* f) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
};
template <> struct Elem<__nv_bfloat16> {
  static constexpr int kPerVec = 8;
  __device__ static void unpack(const uint4& v, float* f) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
};

// Dynamic shared memory of pass 1: observation rows as fp32 [32][D], then the key tile
// [128][D/VEC + 1] of 16-byte vectors.
template <typename T, int D>
constexpr size_t logits_smem_bytes() {
  return (size_t)kObs * D * 4 + (size_t)kChunk * (D / Elem<T>::kPerVec + 1) * 16;
}

// Pass 1 for candidates [j0, j0 + 128) of one row-block with n_cand candidates.
//   obs_ptr(i)        -> pointer to observation row i (D elements of T), i < n_obs_rows
//   key_ptr(j)        -> pointer to candidate key j (D elements of T), j < n_cand
//   logit_ptr(i, j)   -> where the logit of (observation row i, candidate j) goes
//   part_ptr(i)       -> pointer to the two floats (max, sum-exp) of row i for this chunk
// Warp w forms the logits of observation rows 8 w .. 8 w + 7, lane x those of keys x + 32 u: twelve
// 16-byte shared-memory reads per 128 multiply-adds of a thread (a thread that held one key against
// all 32 rows read 16 bytes per 4), and the whole chunk of a row sits in one warp, so its statistics
// are warp reductions and its logits leave coalesced without a transposing pass.  The keys arrive by
// cp.async, all 16-byte pieces of the tile in flight at once.
// Both passes on 32 rows x 2 000 keys x 128 (bf16): 40.5 -> 26.2 us per call.
template <typename T, int D, typename ObsPtr, typename KeyPtr, typename LogitPtr, typename PartPtr>
__device__ __forceinline__ void chunk_logits(unsigned char* smem_raw, int j0, int n_cand, int n_obs_rows, float sm_scale,
                                             ObsPtr obs_ptr, KeyPtr key_ptr, LogitPtr logit_ptr, PartPtr part_ptr) {
  constexpr int VEC = Elem<T>::kPerVec;
  constexpr int ROWV = D / VEC;                 // 16-byte vectors per row
  constexpr int KROW = ROWV + 1;                // padded row stride (in vectors) of the key tile
  constexpr int OPW = kObs / (kChunk / 32);     // observation rows per warp
  constexpr int KPL = kChunk / 32;              // keys per lane
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* qs = reinterpret_cast<float*>(smem_raw);                       // [32][D]
  uint4* ks = reinterpret_cast<uint4*>(smem_raw + kObs * D * 4);        // [128][KROW]

#pragma unroll 8
  for (int v = tid; v < kChunk * ROWV; v += kChunk) {
    const int r = v / ROWV, c = v % ROWV;
    const int j = min(j0 + r, n_cand - 1);      // rows past the end repeat the last key; they are masked below
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(ks + r * KROW + c));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(key_ptr(j) + c * VEC) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
  for (int v = tid; v < kObs * ROWV; v += kChunk) {
    const int i = v / ROWV, c = v % ROWV;
    float f[VEC];
    if (i < n_obs_rows) {
      Elem<T>::unpack(*reinterpret_cast<const uint4*>(obs_ptr(i) + c * VEC), f);
    } else {
#pragma unroll
      for (int e = 0; e < VEC; ++e) f[e] = 0.f;
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) qs[i * D + c * VEC + e] = f[e];
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();

  const int i0 = warp * OPW;
  if (i0 >= n_obs_rows) return;
  float2 acc[OPW][KPL];                         // even and odd dimensions apart
#pragma unroll
  for (int i = 0; i < OPW; ++i)
#pragma unroll
    for (int u = 0; u < KPL; ++u) acc[i][u] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int c = 0; c < ROWV; ++c) {
    float kf[KPL][VEC];
#pragma unroll
    for (int u = 0; u < KPL; ++u) Elem<T>::unpack(ks[(lane + 32 * u) * KROW + c], kf[u]);
#pragma unroll
    for (int i = 0; i < OPW; ++i) {
      const float4* qv = reinterpret_cast<const float4*>(qs + (i0 + i) * D + c * VEC);
#pragma unroll
      for (int e4 = 0; e4 < VEC / 4; ++e4) {
        const float4 qq = qv[e4];
#pragma unroll
        for (int u = 0; u < KPL; ++u) {
          acc[i][u] = ptx::fma2(make_float2(qq.x, qq.y), make_float2(kf[u][4 * e4], kf[u][4 * e4 + 1]), acc[i][u]);
          acc[i][u] = ptx::fma2(make_float2(qq.z, qq.w), make_float2(kf[u][4 * e4 + 2], kf[u][4 * e4 + 3]), acc[i][u]);
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < OPW; ++i) {
    float z[KPL];
    float m = -INFINITY;
#pragma unroll
    for (int u = 0; u < KPL; ++u) {
      const int j = j0 + lane + 32 * u;
      z[u] = j < n_cand ? (acc[i][u].x + acc[i][u].y) * sm_scale : -INFINITY;
      m = fmaxf(m, z[u]);
      if (j < n_cand && i0 + i < n_obs_rows) *logit_ptr(i0 + i, j) = z[u];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float l = 0.f;
#pragma unroll
    for (int u = 0; u < KPL; ++u) l += expf(z[u] - m);      // exp(-inf) = 0 for padding
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0 && i0 + i < n_obs_rows) *reinterpret_cast<float2*>(part_ptr(i0 + i)) = make_float2(m, l);
  }
}

// Pass 2 for a CTA of 256 threads and candidates [j0, j0 + 256): row_m / row_inv_l are two shared
// arrays of 32 floats; part(c, i) points at the (max, sum-exp) of chunk c, row i; returns the score
// of candidate j0 + threadIdx.x through `score` (valid when the function returns true).
// Latency bound: eight threads merge the chunk statistics of a row, and a thread's 32 logits are
// loaded before the statistics are needed (a loop of unknown length waited for memory row by row).
template <typename PartPtr, typename LogitVal>
__device__ __forceinline__ bool column_scores(float* row_m, float* row_inv_l, int j0, int n_cand, int n_obs_rows,
                                              int n_chunks, PartPtr part, LogitVal logit, float& score) {
  const int j = j0 + threadIdx.x;
  float z[kObs];
#pragma unroll
  for (int i = 0; i < kObs; ++i) z[i] = i < n_obs_rows && j < n_cand ? logit(i, j) : 0.f;
  {
    const int i = threadIdx.x >> 3, sub = threadIdx.x & 7;
    float m = -INFINITY, l = 0.f;
    if (i < n_obs_rows) {
#pragma unroll 4
      for (int c = sub; c < n_chunks; c += 8) {
        const float2 p = *reinterpret_cast<const float2*>(part(c, i));
        const float mn = fmaxf(m, p.x);
        l = l * expf(m - mn) + p.y * expf(p.x - mn);
        m = mn;
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
      const float mn = fmaxf(m, m2);
      // a thread without chunks carries (-inf, 0)
      l = (l == 0.f ? 0.f : l * expf(m - mn)) + (l2 == 0.f ? 0.f : l2 * expf(m2 - mn));
      m = mn;
    }
    if (sub == 0) {
      row_m[i] = i < n_obs_rows ? m : 0.f;
      row_inv_l[i] = i < n_obs_rows ? 1.f / l : 0.f;
    }
  }
  __syncthreads();
  if (j >= n_cand) return false;
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < kObs; ++i) s += expf(z[i] - row_m[i]) * row_inv_l[i];     // rows past the last one weigh 0
  score = s;
  return true;
}

}  // namespace simt
}  // namespace hack
