// Attention of the scale's queries over the compacted per-head cache (Eq. 4 on the compressed
// cache) of fp32 caches, plain fp32 arithmetic on the CUDA cores: the exact-precision path (fp32
// workloads forbid TF32 at the required 1e-5).
//
// Bound: the FMA pipe.  A CTA serves 32 query rows of one head; its four groups of 64 threads walk
// every fourth tile of 32 keys with a streaming softmax of their own and are merged at the end, so
// that a launch with few query tiles (256 queries x 16 heads are 128 CTAs) still has eight warps per
// SM at work.  With one CTA per SM the length of a launch is a matter of whole CTAs: the heads with
// the longer cache go first, clusters of 2 or 4 CTAs split the keys of a query tile further (merged
// through distributed shared memory) where there are fewer tiles than SMs, and where there are more and the last
// round would be nearly empty every CTA takes the same number of rounds, parts of query tiles at either end of
// its share, which the last CTA to finish one adds up (16 heads x 1 024 queries x 128, 1 717 and 224 keys: 310 -> 272 us
// a step, 576 queries 176 -> 139).
// Inside a group a thread forms 4 x 4 logits and 4 x D/8 outputs: eight 16-byte
// shared-memory reads per 64 multiply-adds in Q K^T, twenty per 256 in P V, every read without bank
// conflicts (rows are padded) and served in two cycles: with the four lanes of a quad on four different rows
// (3.05 cycles a read) the shared-memory pipe was busy 0.79 of the time, 3 % slower.  What is left: packed multiply-adds of
// an outer product issue at 0.68 of the pipe's rate (three 64-bit operands), measured in registers alone.
// Both products run on packed pairs (fma.rn.f32x2).  The key buffer is refilled under the P V product
// and the value buffer under the next Q K^T product (cp.async).
// (The earlier form, four threads per query row that each held a quarter of it, read 16 bytes of
// shared memory per 4 multiply-adds with a four-way bank conflict.  Decoding loop of two layers of 16
// heads x 128, 2 240 tokens, stage calls: 13.8 -> 1.66 ms; one layer of 16 heads x 64, 680 tokens:
// 0.531 -> 0.308 ms.)
#include "hack_internal.h"
#include "launch_plans.h"
#include "tc_ptx.cuh"

namespace hack {
namespace {

using ptx::fma2;
using namespace simt;

constexpr int kThreads = kGroups * 64;

// 32 rows of D floats from global memory (rows at or past n_rows read as zero) into padded rows by
// cp.async (the caller commits and waits); `nthr` threads take part.
template <int D>
__device__ __forceinline__ void stage_rows(float* dst, const float* src, int n_rows, int t, int nthr) {
  constexpr int LD = D + 4, V = D / 4;
#pragma unroll 4
  for (int v = t; v < 32 * V; v += nthr) {
    const int r = v / V, c = v % V;
    const int bytes = r < n_rows ? 16 : 0;                 // 0: the 16 bytes are filled with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst + r * LD + c * 4)),
                 "l"(src + (size_t)(r < n_rows ? r : 0) * D + c * 4), "r"(bytes) : "memory");
  }
}

__device__ __forceinline__ void commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int D>
constexpr size_t simt_smem_bytes() {
  // query rows, then per group a key tile, a value tile and a probability tile
  return sizeof(float) * ((size_t)kBQ * (D + 4) + kGroups * (2 * (size_t)kBK * (D + 4) + kBQ * (kBK + 8)));
}

// One query tile per CTA, or per cluster, or equal shares (a form of its own: its bookkeeping costs the others registers;
// at head_dim 64, with two CTAs on an SM, it spills 24 bytes, which the plain form does not).
enum { kOne, kClustered, kShared };

template <int D, int MODE>
__global__ void __launch_bounds__(kThreads, D == 64 && MODE != kClustered ? 2 : 1)
attend_simt_kernel(const StepArgs a, const float* __restrict__ q, float* __restrict__ out,
                   const int32_t* __restrict__ order, int cluster, const Shares sh) {
  constexpr bool kCluster = MODE == kClustered, kShares = MODE == kShared;
  const int cl = kCluster ? cluster : 1;
  constexpr int LD = D + 4, LP = kBK + 8;
  constexpr int CV = D / 32;                      // float4 columns per thread
  const int rank = blockIdx.x % cl;
  const int tid = threadIdx.x, grp = tid >> 6, gt = tid & 63;
  // rows ty + 8 i; keys tx + 8 j; columns 4 tx + 32 c.  Four consecutive lanes are two of either: a 16-byte
  // read in which every four lanes ask for at most two pieces is served in two cycles instead of four.
  const int lane = tid & 31;
  const int ty = 4 * (gt >> 5) + ((lane & 1) | (lane >> 2 & 2)), tx = (lane >> 1 & 3) | (lane >> 2 & 4);

  extern __shared__ __align__(16) float smem[];
  float* qs = smem;
  float* ks = qs + kBQ * LD + grp * (2 * kBK * LD + kBQ * LP);
  float* vs = ks + kBK * LD;
  float* ps = vs + kBK * LD;

  auto group_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + grp) : "memory"); };

  pdl_wait();
  // This CTA's share: a query tile (a cluster its keys), or the tiles and parts of tiles in its half rounds.
  const int begin = kShares ? blockIdx.x * sh.span : 0, end = kShares ? min(begin + sh.span, sh.total) : 1;
  int tile = 0;
  if (kShares) {
    const int per = 2 * sh.rounds[0] + 1, part = sh.n_first * per;
    tile = begin < part ? begin / per : sh.n_first + (begin - part) / (2 * sh.rounds[1] + 1);
  }
#pragma unroll 1
  for (int at = begin; at < end; ++tile) {
    // rounds [r0, r1) of the tile
    int r0 = 0, r1 = 1 << 20, t0 = 0;
    bool whole = true;
    if (!kShares) {
      at = end;
    } else {
      t0 = tile_begin(sh, tile);
      const int t1 = tile_begin(sh, tile + 1);
      r0 = (at - t0) / 2;
      r1 = (min(end, t1) - t0) / 2;
      whole = r0 == 0 && r1 == (t1 - t0) / 2;
      at = t1;
      if (r0 == r1) continue;
    }
    const int bh = order[kShares ? tile / sh.n_qt : blockIdx.y];   // tables written when the cache was created
    const int len = a.kept[a.is_ctx[bh % a.n_heads]];
    const int q0 = (kShares ? tile % sh.n_qt : blockIdx.x / cl) * kBQ;
    const int n_tiles = min((len + kBK - 1) / kBK, kShares ? r1 * kGroups : 1 << 30);
    const int first = (kShares ? r0 : rank) * kGroups + grp, stride = cl * kGroups;   // key tiles of this group
    const float* kp = static_cast<const float*>(a.k_plane) + (size_t)a.row_off[bh] * D;
    const float* vp = static_cast<const float*>(a.v_plane) + (size_t)a.row_off[bh] * D;
    stage_rows<D>(qs, q + ((size_t)bh * a.n_new + q0) * D, a.n_new - q0, tid, kThreads);
    if (first < n_tiles) stage_rows<D>(ks, kp + (size_t)first * kBK * D, len - first * kBK, gt, 64);
    commit();
    if (first < n_tiles) stage_rows<D>(vs, vp + (size_t)first * kBK * D, len - first * kBK, gt, 64);
    commit();
    wait_group<1>();
    __syncthreads();

    float2 o[4][CV][2];
    float m[4], l[4];                               // l: this thread's share of the row sum
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      m[i] = kNoLogit;
      l[i] = 0.f;
#pragma unroll
      for (int c = 0; c < CV; ++c) o[i][c][0] = o[i][c][1] = make_float2(0.f, 0.f);
    }

    for (int t = first; t < n_tiles; t += stride) {
      // logits: s[i][j] of query row ty + 8 i and key tx + 8 j, even and odd dimensions in the two halves
      float2 s[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = make_float2(0.f, 0.f);
#pragma unroll (D == 128 || MODE == kOne ? 8 : 4)
      for (int d = 0; d < D; d += 4) {
        float4 qf[4], kf[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) qf[i] = *reinterpret_cast<const float4*>(qs + (ty + 8 * i) * LD + d);
#pragma unroll
        for (int j = 0; j < 4; ++j) kf[j] = *reinterpret_cast<const float4*>(ks + (tx + 8 * j) * LD + d);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            s[i][j] = fma2(make_float2(qf[i].x, qf[i].y), make_float2(kf[j].x, kf[j].y), s[i][j]);
            s[i][j] = fma2(make_float2(qf[i].z, qf[i].w), make_float2(kf[j].z, kf[j].w), s[i][j]);
          }
      }
      group_sync();                                 // both warps are done with the key tile
      if (t + stride < n_tiles)
        stage_rows<D>(ks, kp + (size_t)(t + stride) * kBK * D, len - (t + stride) * kBK, gt, 64);
      commit();

      float corr[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float z[4];
        float mt = m[i];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          z[j] = t * kBK + tx + 8 * j < len ? (s[i][j].x + s[i][j].y) * a.sm_scale : -INFINITY;
          mt = fmaxf(mt, z[j]);
        }
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 16));
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 2));
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 4));
        corr[i] = expf(m[i] - mt);                  // exp(-inf) = 0 in the first tile
        m[i] = mt;
        float add = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float p = expf(z[j] - mt);
          add += p;
          ps[(ty + 8 * i) * LP + tx + 8 * j] = p;
        }
        l[i] = l[i] * corr[i] + add;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < CV; ++c)
#pragma unroll
          for (int h = 0; h < 2; ++h) { o[i][c][h].x *= corr[i]; o[i][c][h].y *= corr[i]; }
      wait_group<1>();                              // the value tile has landed (the next keys may still be on their way)
      group_sync();                                 // ... for both warps; also orders this warp's probability rows

#pragma unroll 2
      for (int j = 0; j < kBK; j += 4) {
        float4 pf[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) pf[i] = *reinterpret_cast<const float4*>(ps + (ty + 8 * i) * LP + j);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float4 vf[CV];
#pragma unroll
          for (int c = 0; c < CV; ++c) vf[c] = *reinterpret_cast<const float4*>(vs + (j + u) * LD + 4 * tx + 32 * c);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float pu = u == 0 ? pf[i].x : u == 1 ? pf[i].y : u == 2 ? pf[i].z : pf[i].w;
            const float2 pp = make_float2(pu, pu);
#pragma unroll
            for (int c = 0; c < CV; ++c) {
              o[i][c][0] = fma2(pp, make_float2(vf[c].x, vf[c].y), o[i][c][0]);
              o[i][c][1] = fma2(pp, make_float2(vf[c].z, vf[c].w), o[i][c][1]);
            }
          }
        }
      }
      group_sync();                                 // both warps are done with the value tile
      if (t + stride < n_tiles)
        stage_rows<D>(vs, vp + (size_t)(t + stride) * kBK * D, len - (t + stride) * kBK, gt, 64);
      commit();
      wait_group<1>();                              // the next key tile has landed
      group_sync();
    }
    wait_group<0>();

    // merge of the groups: unnormalised outputs and (max, sum) of every row through shared memory
    // (a group's own key tile holds its 32 x D outputs, its probability tile the row statistics); the CTAs
    // of a cluster each finish a share of the rows
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float li = l[i];
      li += __shfl_xor_sync(0xffffffffu, li, 16);
      li += __shfl_xor_sync(0xffffffffu, li, 2);
      li += __shfl_xor_sync(0xffffffffu, li, 4);
      if (tx == 0) *reinterpret_cast<float2*>(ps + (ty + 8 * i) * 2) = make_float2(m[i], li);
#pragma unroll
      for (int c = 0; c < CV; ++c)
        *reinterpret_cast<float4*>(ks + (ty + 8 * i) * LD + 4 * tx + 32 * c) =
            make_float4(o[i][c][0].x, o[i][c][0].y, o[i][c][1].x, o[i][c][1].y);
    }
    if (kCluster) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
    constexpr int GSTRIDE = 2 * kBK * LD + kBQ * LP;
    const float* g0 = qs + kBQ * LD;
    const int rows = kBQ / cl;
    // Part of a tile: its sums go to one of this CTA's two places in memory, the first if its share begins in the tile.
    constexpr int kPlace = kBQ * (D + 2);
    float* const part_sum = a.simt_partial + (size_t)(2 * blockIdx.x + (begin < t0 ? 1 : 0)) * kPlace;
    for (int v = tid; v < rows * (D / 4); v += kThreads) {
      const int r = rank * rows + v / (D / 4), c = v % (D / 4);
      if (q0 + r >= a.n_new) continue;
      float top = -INFINITY, sum = 0.f;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int cta = 0; cta < cl; ++cta) {
        uint32_t base = 0;
        if (kCluster) asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(base) : "r"(ptx::smem_u32(g0)), "r"(cta));
        float2 st[kGroups];
        float4 f[kGroups];
        float mx = top;
#pragma unroll
        for (int g = 0; g < kGroups; ++g) {
          const int at_st = g * GSTRIDE + 2 * kBK * LD + r * 2, at_f = g * GSTRIDE + r * LD + c * 4;
          if (kCluster) {
            asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(st[g].x), "=f"(st[g].y) : "r"(base + 4u * at_st) : "memory");
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(f[g].x), "=f"(f[g].y), "=f"(f[g].z), "=f"(f[g].w) : "r"(base + 4u * at_f) : "memory");
          } else {
            st[g] = *reinterpret_cast<const float2*>(g0 + at_st);
            f[g] = *reinterpret_cast<const float4*>(g0 + at_f);
          }
          mx = fmaxf(mx, st[g].x);
        }
        const float keep = expf(top - mx);          // 0 for the first CTA; every CTA before a later one has keys
        top = mx;
        sum *= keep;
        acc.x *= keep; acc.y *= keep; acc.z *= keep; acc.w *= keep;
#pragma unroll
        for (int g = 0; g < kGroups; ++g) {
          const float w = expf(st[g].x - top);      // 0 for a group without keys
          sum = fmaf(w, st[g].y, sum);
          acc.x = fmaf(w, f[g].x, acc.x);
          acc.y = fmaf(w, f[g].y, acc.y);
          acc.z = fmaf(w, f[g].z, acc.z);
          acc.w = fmaf(w, f[g].w, acc.w);
        }
      }
      if (kShares && !whole) {
        __stcg(reinterpret_cast<float4*>(part_sum + r * D + c * 4), acc);
        if (c == 0) __stcg(reinterpret_cast<float2*>(part_sum + kBQ * D + 2 * r), make_float2(top, sum));
        continue;
      }
      const float inv = 1.f / sum;
      *reinterpret_cast<float4*>(out + ((size_t)bh * a.n_new + q0 + r) * D + c * 4) =
          make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
    }
    if (kShares && !whole) {
      // the CTA that is the last to finish a part of the tile adds the parts up, in the order of their keys
      __shared__ int last;
      const int t1 = tile_begin(sh, tile + 1);
      const int c0 = t0 / sh.span, c1 = (t1 - 1) / sh.span;
      // the CTA's part of this tile: none where its half rounds hold no round
      auto has = [&](int cta) { return (max(cta * sh.span, t0) - t0) / 2 < (min((cta + 1) * sh.span, t1) - t0) / 2; };
      __threadfence();
      __syncthreads();
      if (tid == 0) {
        int parts = 0;
        for (int cta = c0; cta <= c1; ++cta) parts += has(cta);
        last = atomicAdd(a.simt_arrived + tile, 1) == parts - 1;
        if (last) a.simt_arrived[tile] = 0;
      }
      __syncthreads();
      if (last) {
        __threadfence();
        for (int v = tid; v < kBQ * (D / 4); v += kThreads) {
          const int r = v / (D / 4), c = v % (D / 4);
          if (q0 + r >= a.n_new) continue;
          float top = -INFINITY, sum = 0.f;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int cta = c0; cta <= c1; ++cta) {
            if (!has(cta)) continue;
            const float* p = a.simt_partial + (size_t)(2 * cta + (cta * sh.span < t0 ? 1 : 0)) * kPlace;
            const float2 st = __ldcg(reinterpret_cast<const float2*>(p + kBQ * D + 2 * r));
            const float4 f = __ldcg(reinterpret_cast<const float4*>(p + r * D + c * 4));
            const float mx = fmaxf(top, st.x), keep = expf(top - mx), w = expf(st.x - mx);
            top = mx;
            sum = fmaf(w, st.y, sum * keep);
            acc.x = fmaf(w, f.x, acc.x * keep);
            acc.y = fmaf(w, f.y, acc.y * keep);
            acc.z = fmaf(w, f.z, acc.z * keep);
            acc.w = fmaf(w, f.w, acc.w * keep);
          }
          const float inv = 1.f / sum;
          *reinterpret_cast<float4*>(out + ((size_t)bh * a.n_new + q0 + r) * D + c * 4) =
              make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        }
      }
    }
    if (kShares) __syncthreads();                   // the next tile's loads overwrite what was merged
  }
  // no CTA leaves while another may still read its shared memory
  if (kCluster) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

template <int D>
int launch_t(const StepArgs& a, const void* q, void* out, cudaStream_t st) {
  const int n_qt = (a.n_new + kBQ - 1) / kBQ, heads = a.batch * a.n_heads;
  const SimtPlan plan = simt_plan(D, a.n_new, a.kept, a.heads_of, sm_count());
  const Shares& sh = plan.sh;
  const int cl = plan.cluster;
  const int32_t* order = a.head_order + (a.kept[1] > a.kept[0] ? heads : 0);
  auto kern = cl > 1 ? attend_simt_kernel<D, kClustered> : plan.shared ? attend_simt_kernel<D, kShared> : attend_simt_kernel<D, kOne>;
  if (!allow_dynamic_smem(kern, simt_smem_bytes<D>())) return -1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = plan.shared ? dim3(plan.ctas) : dim3(n_qt * cl, heads);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = simt_smem_bytes<D>();
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cl;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cl > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kern, a, static_cast<const float*>(q), static_cast<float*>(out), order, cl, sh);
  return launched(1);
}

}  // namespace

// Two parts of a tile per CTA; a counter per query tile.
size_t simt_partial_floats(int head_dim) { return (size_t)2 * sm_count() * (head_dim == 64 ? 2 : 1) * kBQ * (head_dim + 2); }
size_t simt_arrived_words(int heads, int max_new) { return (size_t)heads * ((max_new + kBQ - 1) / kBQ); }

int launch_attend_simt(const StepArgs& a, const void* q, void* out, cudaStream_t st) {
  return a.head_dim == 64 ? launch_t<64>(a, q, out, st) : launch_t<128>(a, q, out, st);
}

}  // namespace hack
