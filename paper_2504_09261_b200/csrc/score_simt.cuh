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

// ---------------------------------------------------------------- one launch
// A cluster of up to eight CTAs owns one row-block.  Each CTA forms the logits of its chunks of 128
// candidates and keeps them in registers, the CTAs exchange the (max, sum-exp) of the observation rows
// through distributed shared memory, and every CTA reduces its own columns: no logits in memory and
// no second launch.
//  * fp32, one chunk per CTA: FMA pipe.  Warp w has observation rows 4 w .. 4 w + 3, a lane the keys
//    lane + 32 u.  16 rows x 640 candidates x 128: 9.0 us against 11.0 in two launches.
//  * bf16, up to four chunks per CTA: warp-level matrix instructions (fp32 accumulation), a warp has 16
//    keys of a chunk against all rows.  32 rows x 2 000 candidates x 128: 10.5 us against 26.0.
constexpr int kFusedThreads = 256;
constexpr int kFusedWarps = kFusedThreads / 32;
constexpr int kFusedCluster = 8;

__device__ __forceinline__ uint32_t fused_rank(int cl) {
  uint32_t rank = 0;
  if (cl > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  return rank;
}
__device__ __forceinline__ void fused_sync(int cl) {
  if (cl > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  else __syncthreads();
}
// pub holds the CTA's (max, sum-exp) of every row; row_stat receives (max, 1 / sum) of the row-block.
__device__ __forceinline__ void fused_merge(const float2* pub, float2* row_stat, int cl, int n_obs_rows) {
  fused_sync(cl);
  const int tid = threadIdx.x;
  if (tid < kObs) {
    float2 got[kFusedCluster];
#pragma unroll
    for (int r = 0; r < kFusedCluster; ++r) {
      got[r] = make_float2(-INFINITY, 0.f);
      if (r < cl) {
        uint32_t addr;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(ptx::smem_u32(&pub[tid])), "r"(r));
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(got[r].x), "=f"(got[r].y) : "r"(addr) : "memory");
      }
    }
    float top = -INFINITY, sum = 0.f;
#pragma unroll
    for (int r = 0; r < kFusedCluster; ++r) top = fmaxf(top, got[r].x);
#pragma unroll
    for (int r = 0; r < kFusedCluster; ++r) sum += got[r].y == 0.f ? 0.f : got[r].y * expf(got[r].x - top);
    row_stat[tid] = tid < n_obs_rows ? make_float2(top, 1.f / sum) : make_float2(0.f, 0.f);   // padding rows weigh nothing
  }
  __syncthreads();
  // this CTA has read its peers' statistics; it leaves (fused_leave) once they have read its own
  if (cl > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void fused_leave(int cl) {
  if (cl > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}

template <int D>
constexpr size_t fused_f32_smem() { return (size_t)kObs * D * 4 + (size_t)kChunk * (D + 4) * 4; }

//   store(j, s): the score of candidate j
template <int D, typename ObsPtr, typename KeyPtr, typename Store>
__device__ __forceinline__ void cluster_scores_f32(unsigned char* smem_raw, int cl, int n_cand, int n_obs_rows, float sm_scale,
                                                   ObsPtr obs_ptr, KeyPtr key_ptr, Store store) {
  constexpr int ROWV = D / 4, KROW = ROWV + 1, OPW = kObs / kFusedWarps, KPL = kChunk / 32;
  __shared__ float2 pub[kObs], row_stat[kObs];
  __shared__ float part[kFusedWarps][kChunk];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float4* qs = reinterpret_cast<float4*>(smem_raw);                     // [32][ROWV]
  float4* ks = qs + kObs * ROWV;                                        // [128][KROW]
  const int j0 = (int)fused_rank(cl) * kChunk, i0 = warp * OPW;

  float z[OPW][KPL];
#pragma unroll
  for (int i = 0; i < OPW; ++i)
#pragma unroll
    for (int u = 0; u < KPL; ++u) z[i][u] = -INFINITY;
  if (j0 < n_cand) {
    auto fetch = [](const float4* dst, const float* src, int bytes) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
    };
#pragma unroll 4
    for (int v = tid; v < kChunk * ROWV; v += kFusedThreads) {
      const int r = v / ROWV, c = v % ROWV;
      // rows past the end repeat the last key; they are masked below
      fetch(ks + r * KROW + c, key_ptr(min(j0 + r, n_cand - 1)) + c * 4, 16);
    }
#pragma unroll
    for (int v = tid; v < kObs * ROWV; v += kFusedThreads) {
      const int i = v / ROWV, c = v % ROWV;
      fetch(qs + v, obs_ptr(min(i, n_obs_rows - 1)) + c * 4, i < n_obs_rows ? 16 : 0);    // 0: zeros
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float2 acc[OPW][KPL];                       // even and odd dimensions apart
#pragma unroll
    for (int i = 0; i < OPW; ++i)
#pragma unroll
      for (int u = 0; u < KPL; ++u) acc[i][u] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int c = 0; c < ROWV; ++c) {
      float4 kf[KPL];
#pragma unroll
      for (int u = 0; u < KPL; ++u) kf[u] = ks[(lane + 32 * u) * KROW + c];
#pragma unroll
      for (int i = 0; i < OPW; ++i) {
        const float4 qq = qs[(i0 + i) * ROWV + c];
#pragma unroll
        for (int u = 0; u < KPL; ++u) {
          acc[i][u] = ptx::fma2(make_float2(qq.x, qq.y), make_float2(kf[u].x, kf[u].y), acc[i][u]);
          acc[i][u] = ptx::fma2(make_float2(qq.z, qq.w), make_float2(kf[u].z, kf[u].w), acc[i][u]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < OPW; ++i)
#pragma unroll
      for (int u = 0; u < KPL; ++u)
        if (j0 + lane + 32 * u < n_cand) z[i][u] = (acc[i][u].x + acc[i][u].y) * sm_scale;
  }
#pragma unroll
  for (int i = 0; i < OPW; ++i) {
    float m = fmaxf(fmaxf(z[i][0], z[i][1]), fmaxf(z[i][2], z[i][3])), l = 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (m > -INFINITY) {
#pragma unroll
      for (int u = 0; u < KPL; ++u) l += expf(z[i][u] - m);             // exp(-inf) = 0 for padding
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) pub[i0 + i] = make_float2(m, l);
  }
  fused_merge(pub, row_stat, cl, n_obs_rows);
  float sum[KPL] = {};
#pragma unroll
  for (int i = 0; i < OPW; ++i) {
    const float2 st = row_stat[i0 + i];
#pragma unroll
    for (int u = 0; u < KPL; ++u) sum[u] += expf(z[i][u] - st.x) * st.y;
  }
#pragma unroll
  for (int u = 0; u < KPL; ++u) part[warp][lane + 32 * u] = sum[u];
  __syncthreads();
  if (tid < kChunk && j0 + tid < n_cand) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kFusedWarps; ++w) v += part[w][tid];
    store(j0 + tid, v);
  }
  fused_leave(cl);
}

template <int D, int PER>
constexpr size_t fused_bf16_smem() { return (size_t)(kObs + PER * kChunk) * D * 2; }

template <int D, int PER, typename ObsPtr, typename KeyPtr, typename Store>
__device__ __forceinline__ void cluster_scores_bf16(unsigned char* smem_raw, int cl, int n_cand, int n_obs_rows, float sm_scale,
                                                    ObsPtr obs_ptr, KeyPtr key_ptr, Store store) {
  constexpr int PIECES = D / 8;                 // 16-byte pieces per row
  __shared__ float2 pub[kObs], row_stat[kObs], warp_stat[kFusedWarps][kObs];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t q_sm = ptx::smem_u32(smem_raw), k_sm = q_sm + kObs * D * 2;
  const int first = (int)fused_rank(cl) * PER * kChunk;
  // piece c of row r: the pieces of eight consecutive rows fall into different banks
  auto at = [](int r, int c) { return (uint32_t)r * (D * 2) + (uint32_t)((c ^ (r & 7)) << 4); };
  auto fetch = [](uint32_t dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
  };
#pragma unroll
  for (int v = tid; v < kObs * PIECES; v += kFusedThreads) {
    const int i = v / PIECES, c = v % PIECES;
    fetch(q_sm + at(i, c), obs_ptr(min(i, n_obs_rows - 1)) + c * 8, i < n_obs_rows ? 16 : 0);    // 0: zeros
  }
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    if (first + p * kChunk < n_cand) {
#pragma unroll 4
      for (int v = tid; v < kChunk * PIECES; v += kFusedThreads) {
        const int r = v / PIECES, c = v % PIECES;
        // rows past the end repeat the last key; they are masked below
        fetch(k_sm + p * kChunk * D * 2 + at(r, c), key_ptr(min(first + p * kChunk + r, n_cand - 1)) + c * 8, 16);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");     // a group per chunk: its logits are formed while the next ones arrive
  }
  // z[p][n][e]: key 16 warp + lane / 4 + 8 (e / 2) of chunk p, observation row 8 n + 2 (lane % 4) + e % 2
  float z[PER][4][4];
  const int key = 16 * warp + (lane >> 2);
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int j0 = first + p * kChunk;
    if (PER - 1 - p == 3) asm volatile("cp.async.wait_group 3;" ::: "memory");
    else if (PER - 1 - p == 2) asm volatile("cp.async.wait_group 2;" ::: "memory");
    else if (PER - 1 - p == 1) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int n = 0; n < 4; ++n) z[p][n][0] = z[p][n][1] = z[p][n][2] = z[p][n][3] = 0.f;
    if (j0 < n_cand) {
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) {
        uint32_t ka[4], qb[4];
        ptx::ldsm4(k_sm + p * kChunk * D * 2 + at(16 * warp + (lane & 15), 2 * kk + (lane >> 4)), ka);
#pragma unroll
        for (int h = 0; h < 2; ++h) {           // observation rows 16 h .. 16 h + 15
          ptx::ldsm4(q_sm + at(16 * h + (lane & 7) + ((lane >> 4) << 3), 2 * kk + ((lane >> 3) & 1)), qb);
          ptx::mma16816(z[p][2 * h], ka, qb[0], qb[1]);
          ptx::mma16816(z[p][2 * h + 1], ka, qb[2], qb[3]);
        }
      }
    }
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) z[p][n][e] = j0 + key + 8 * (e >> 1) < n_cand ? z[p][n][e] * sm_scale : -INFINITY;
  }
#pragma unroll
  for (int n = 0; n < 4; ++n)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      float m = -INFINITY, l = 0.f;
#pragma unroll
      for (int p = 0; p < PER; ++p) m = fmaxf(m, fmaxf(z[p][n][x], z[p][n][x + 2]));
#pragma unroll
      for (int o = 16; o >= 4; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (m > -INFINITY) {
#pragma unroll
        for (int p = 0; p < PER; ++p) l += expf(z[p][n][x] - m) + expf(z[p][n][x + 2] - m);    // exp(-inf) = 0 for padding
      }
#pragma unroll
      for (int o = 16; o >= 4; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane < 4) warp_stat[warp][8 * n + 2 * lane + x] = make_float2(m, l);
    }
  __syncthreads();
  if (tid < kObs) {
    float m = -INFINITY, l = 0.f;
#pragma unroll
    for (int w = 0; w < kFusedWarps; ++w) m = fmaxf(m, warp_stat[w][tid].x);
#pragma unroll
    for (int w = 0; w < kFusedWarps; ++w) l += warp_stat[w][tid].y == 0.f ? 0.f : warp_stat[w][tid].y * expf(warp_stat[w][tid].x - m);
    pub[tid] = make_float2(m, l);
  }
  fused_merge(pub, row_stat, cl, n_obs_rows);
  float s[PER][2] = {};
#pragma unroll
  for (int n = 0; n < 4; ++n)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const float2 st = row_stat[8 * n + 2 * (lane & 3) + x];
#pragma unroll
      for (int p = 0; p < PER; ++p)
#pragma unroll
        for (int h = 0; h < 2; ++h) s[p][h] += expf(z[p][n][x + 2 * h] - st.x) * st.y;
    }
#pragma unroll
  for (int p = 0; p < PER; ++p)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      s[p][h] += __shfl_xor_sync(0xffffffffu, s[p][h], 1);
      s[p][h] += __shfl_xor_sync(0xffffffffu, s[p][h], 2);
      const int j = first + p * kChunk + key + 8 * h;
      if ((lane & 3) == 0 && j < n_cand) store(j, s[p][h]);
    }
  fused_leave(cl);
}

// CTAs per row-block (0: two launches) and chunks per CTA of the one-launch form.  fp32: one chunk per
// CTA, and one CTA per SM or few CTAs per row-block (past that the two launches stream more: 32 rows x
// 1 024 candidates x 64 10.3 us against 11.1).
// bf16, head_dim 128: as many chunks per CTA as leave one CTA per SM, if four do (32 rows x 2 000 candidates 11.2 us with
// two, 9.7 with four; at head_dim 64 7.7 and 8.7).  A group of copies per chunk: 16 rows x 4 000 candidates 18.5 -> 17.3.
inline int fused_cluster(int n_cand, int rows, bool bf16, int head_dim, int sms, int& per) {
  const int n = (n_cand + kChunk - 1) / kChunk;
  per = (n + kFusedCluster - 1) / kFusedCluster;
  if (bf16) {
    if (per > 4) return 0;
    if (per == 3) per = 4;
    if (head_dim == 128 && rows * ((n + 3) / 4) <= sms)
      while (per < 4 && rows * ((n + per - 1) / per) > sms) per *= 2;
    return (n + per - 1) / per;
  }
  return per == 1 && (rows * n <= sms || n <= 4) ? n : 0;
}
// Launch with programmatic stream serialisation and clusters of `cl` CTAs along x.
template <typename... KArgs, typename... Args>
inline void launch_cluster(void (*kern)(KArgs...), int cl, int rows, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cl, rows);
  cfg.blockDim = dim3(kFusedThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cl;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// ---------------------------------------------------------------- two launches, any number of candidates
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
