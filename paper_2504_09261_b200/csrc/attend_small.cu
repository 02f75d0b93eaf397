// Attention of small scales in the launch that also appends the new scale's K/V rows to the per-head
// cache (Eq. 3): over [cache rows ; new rows] (Eq. 4).  Such steps are pure latency: two dependent
// launches and the set-up of a tcgen05 pipeline (128-row tiles, tensor memory) cost more than the
// arithmetic.
//
// fp32 caches, append_attend_small_kernel: one warp serves one query row.  Scores: lane <-> key (a lane walks its key's row with 16-byte
// loads, the query row is broadcast from shared memory); softmax statistics with warp shuffles;
// output: lane <-> a run of head dimensions, the probabilities are broadcast lane by lane and the
// value rows are read coalesced.  Keys below the stored length come from the cache planes, the
// others straight from the caller's K/V tensors, so nothing depends on the append, which the
// same CTAs perform afterwards on cache rows no one reads in this launch.
#include <algorithm>

#include "hack_internal.h"
#include "tc_ptx.cuh"

namespace hack {
namespace {

using ptx::ldsm4;
using ptx::ldsm4_trans;
using ptx::mma16816;

constexpr int kWarps = 8;                       // query rows per CTA

template <typename T> struct Row;
template <> struct Row<float> {
  static constexpr int kPerVec = 4;
  __device__ static void unpack(const uint4& v, float* f) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
  __device__ static float load1(const float* p) { return *p; }
  __device__ static void store1(float* p, float v) { *p = v; }
};
// DL consecutive elements starting at p (DL * sizeof(T) bytes, naturally aligned) as floats.
template <typename T, int DL>
__device__ __forceinline__ void load_run(const T* p, float* f) {
  if constexpr (DL == 4) { const float4 v = *reinterpret_cast<const float4*>(p); f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w; }
  else { const float2 v = *reinterpret_cast<const float2*>(p); f[0] = v.x; f[1] = v.y; }
}

template <typename T, int D>
__global__ void __launch_bounds__(kWarps * 32)
append_attend_small_kernel(const StepArgs a, const T* __restrict__ q, const T* __restrict__ k_new,
                           const T* __restrict__ v_new, T* __restrict__ out) {
  pdl_wait();
  constexpr int VEC = Row<T>::kPerVec;
  constexpr int DL = D / 32;                    // output dimensions per lane
  const int bh = blockIdx.y;
  const int ctx = a.is_ctx[bh % a.n_heads];
  const int stored = a.stored[ctx];
  const int total = stored + a.n_new;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qi = blockIdx.x * kWarps + warp;
  const size_t off = a.row_off[bh];
  const T* kc = static_cast<const T*>(a.k_plane) + off * D;
  const T* vc = static_cast<const T*>(a.v_plane) + off * D;
  const T* kn = k_new + (size_t)bh * a.n_new * D;
  const T* vn = v_new + (size_t)bh * a.n_new * D;

  __shared__ __align__(16) float qs[kWarps][D];
  if (qi < a.n_new) {
    const T* qp = q + ((size_t)bh * a.n_new + qi) * D;
    for (int d = lane; d < D; d += 32) qs[warp][d] = Row<T>::load1(qp + d);
  }
  __syncwarp();

  if (qi < a.n_new) {
    const float c = a.sm_scale * 1.4426950408889634f;          // work in log2 units
    float m = -INFINITY, l = 0.f;
    float o[DL];
#pragma unroll
    for (int i = 0; i < DL; ++i) o[i] = 0.f;
    for (int j0 = 0; j0 < total; j0 += 32) {
      const int j = j0 + lane;
      float z = -INFINITY;
      if (j < total) {
        const T* kr = j < stored ? kc + (size_t)j * D : kn + (size_t)(j - stored) * D;
        float acc = 0.f;
#pragma unroll
        for (int v = 0; v < D / VEC; ++v) {
          float kf[VEC];
          Row<T>::unpack(*reinterpret_cast<const uint4*>(kr + v * VEC), kf);
#pragma unroll
          for (int e = 0; e < VEC; e += 4) {
            const float4 qq = *reinterpret_cast<const float4*>(&qs[warp][v * VEC + e]);
            acc = fmaf(qq.x, kf[e], acc);
            acc = fmaf(qq.y, kf[e + 1], acc);
            acc = fmaf(qq.z, kf[e + 2], acc);
            acc = fmaf(qq.w, kf[e + 3], acc);
          }
        }
        z = acc * c;
      }
      float mt = z;
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, s));
      const float m_new = fmaxf(m, mt);
      const float corr = exp2f(m - m_new);                      // 0 in the first tile
      const float p = exp2f(z - m_new);                         // 0 for lanes past the end
      float ps = p;
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, s);
      l = l * corr + ps;
      m = m_new;
#pragma unroll
      for (int i = 0; i < DL; ++i) o[i] *= corr;
      // value rows in groups of eight, loads first: lanes past the end carry p = 0 and re-read the
      // last row, so no guard is needed
      const int n_in = min(32, total - j0);
      for (int u0 = 0; u0 < n_in; u0 += 8) {
        float vf[8][DL];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int ju = min(j0 + u0 + u, total - 1);
          const T* vr = (ju < stored ? vc + (size_t)ju * D : vn + (size_t)(ju - stored) * D) + lane * DL;
          load_run<T, DL>(vr, vf[u]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float pu = __shfl_sync(0xffffffffu, p, u0 + u);
#pragma unroll
          for (int i = 0; i < DL; ++i) o[i] = fmaf(pu, vf[u][i], o[i]);
        }
      }
    }
    const float inv = 1.f / l;
    T* op = out + ((size_t)bh * a.n_new + qi) * D + lane * DL;
#pragma unroll
    for (int i = 0; i < DL; ++i) Row<T>::store1(op + i, o[i] * inv);
  }

  // append: rows [stored, stored + n_new) of the cache take the new scale's rows; the CTAs of a
  // head share them, 16 bytes per thread
  constexpr int ROWV = D / VEC;                 // 16-byte pieces per row
  const int n_pieces = dbg_ok(stored + a.n_new <= a.cap[ctx], a.status, 6) ? a.n_new * ROWV : 0;
  const uint4* ksrc = reinterpret_cast<const uint4*>(kn);
  const uint4* vsrc = reinterpret_cast<const uint4*>(vn);
  uint4* kdst = reinterpret_cast<uint4*>(static_cast<T*>(a.k_plane) + (off + stored) * D);
  uint4* vdst = reinterpret_cast<uint4*>(static_cast<T*>(a.v_plane) + (off + stored) * D);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pieces; i += gridDim.x * blockDim.x) {
    kdst[i] = ksrc[i];
    vdst[i] = vsrc[i];
  }
  if (blockIdx.x == 0 && n_pieces > 0)
    for (int r = threadIdx.x; r < a.n_new; r += blockDim.x) a.pos_plane[off + stored + r] = a.pos_base + r;
}

// ------------------------------------------------------------------ bf16 caches
// A CTA serves 16 queries of one head with warp-level matrix instructions (mma.m16n8k16; a 128-row
// tcgen05 tile would be at most a quarter full here).  Its W warps take the keys in turns of 16 with
// a streaming softmax of their own and are merged at the end, so that up to 64 keys (W = 4; 128 with
// eight warps, launches of few CTAs) are one trip to memory: a warp fetches its 16 key and value rows (and the first time the queries) with cp.async,
// all of them in flight at once, and everything after that is registers and shared memory.  New rows
// go from there to the cache as well.  The probabilities enter the second product as a sum of two
// bf16 numbers (error 2^-17), so they are as good as the fp32 ones of a SIMT kernel.
// Head types with a.seg_new set read and append the caller's rows; the others attend over the cache as
// it is.  Bound: latency (launch, one trip to memory, a few hundred dependent instructions).  Step of 25
// queries and 55 keys, 256 heads x 64: 5.4 us; 16 queries, 30 keys, 240 heads x 64: 3.4 us;
// 16 queries, 21 keys, 32 heads x 128: 3.6 us (one warp per query row on the CUDA cores:
// 27.5, 10.5 and 5.5 us).
constexpr int kMmaRows = 16;                    // queries per CTA, keys per warp and turn

// Two fp32 numbers as a sum of two packed pairs of bf16.
__device__ __forceinline__ void split_bf16(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - __low2float(h), y - __high2float(h));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

template <int D, int W>
constexpr size_t mma_smem_bytes() {
  // queries, then per warp a key and a value tile; the warp's two tiles later hold its 16 x D outputs
  return (size_t)kMmaRows * D * 2 * (1 + 2 * W);
}

template <int D, int W>
__global__ void __launch_bounds__(W * 32)
append_attend_mma_kernel(const StepArgs a, const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k_new,
                         const __nv_bfloat16* __restrict__ v_new, __nv_bfloat16* __restrict__ out, int after_compression) {
  constexpr int PIECES = D / 8;                 // 16-byte pieces per row
  constexpr uint32_t ROWB = D * 2;
  constexpr uint32_t TILE = kMmaRows * ROWB;    // 16 rows
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ float2 row_ml[W][kMmaRows];

  const int bh = blockIdx.y, q0 = blockIdx.x * kMmaRows;
  const int ctx = a.is_ctx[bh % a.n_heads];     // written when the cache was created, like row_off
  const int total = a.kept[ctx], stored = a.seg_new[ctx] ? total - a.n_new : total;   // cache rows, then the caller's
  const size_t off = a.row_off[bh];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const __nv_bfloat16* kc = static_cast<const __nv_bfloat16*>(a.k_plane) + off * D;
  const __nv_bfloat16* vc = static_cast<const __nv_bfloat16*>(a.v_plane) + off * D;
  const __nv_bfloat16* kn = k_new + (size_t)bh * a.n_new * D;
  const __nv_bfloat16* vn = v_new + (size_t)bh * a.n_new * D;
  const __nv_bfloat16* qn = q + (size_t)bh * a.n_new * D;
  const uint32_t q_sm = ptx::smem_u32(sm), k_sm = q_sm + TILE + warp * 2 * TILE, v_sm = k_sm + TILE;
  // 16-byte piece c of row r: the pieces of eight consecutive rows fall into different banks
  auto at = [](int r, int c) { return (uint32_t)r * ROWB + (uint32_t)((c ^ (r & 7)) << 4); };
  auto fetch = [](uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  };
  // Behind the step's compression launch (which has itself waited for everything before it) heads that
  // the step does not compress wait for nothing.
  if (!after_compression || a.trig[ctx]) pdl_grid_wait();
  pdl_launch_dependents();

  // rows past the last query or key repeat the last one: their results are not stored or weigh nothing
#pragma unroll
  for (int v = tid; v < kMmaRows * PIECES; v += W * 32) {
    const int r = v / PIECES, c = v % PIECES;
    fetch(q_sm + at(r, c), qn + (size_t)min(q0 + r, a.n_new - 1) * D + c * 8);
  }
  const bool appends = blockIdx.x == 0 && total > stored && dbg_ok(total <= a.cap[ctx], a.status, 6);
  const float cs = a.sm_scale * 1.4426950408889634f;          // work in log2 units
  float m[2] = {kNoLogit, kNoLogit}, l[2] = {0.f, 0.f};     // rows lane / 4 and lane / 4 + 8; l: this thread's share
  float o[D / 8][4];
#pragma unroll
  for (int n = 0; n < D / 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
  uint32_t qa[D / 16][4];

  const int turns = (total + W * kMmaRows - 1) / (W * kMmaRows);
  for (int t = 0; t < turns; ++t) {
    const int j0 = (t * W + warp) * kMmaRows;
    const bool any = j0 < total;
    if (any) {
#pragma unroll
      for (int i = 0; i < kMmaRows * PIECES / 32; ++i) {
        const int v = lane + i * 32, r = v / PIECES, c = v % PIECES;
        const int j = min(j0 + r, total - 1);
        fetch(k_sm + at(r, c), (j < stored ? kc + (size_t)j * D : kn + (size_t)(j - stored) * D) + c * 8);
        fetch(v_sm + at(r, c), (j < stored ? vc + (size_t)j * D : vn + (size_t)(j - stored) * D) + c * 8);
      }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    if (t == 0) {
      __syncthreads();                          // the queries were fetched by all warps
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) ldsm4(q_sm + at(lane & 15, 2 * kk + (lane >> 4)), qa[kk]);
    } else {
      __syncwarp();
    }
    if (!any) break;
    float s[2][4] = {};
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
      uint32_t b[4];                            // keys 0-7 and 8-15, each with the two halves of the k-step
      ldsm4(k_sm + at((lane & 7) + ((lane >> 4) << 3), 2 * kk + ((lane >> 3) & 1)), b);
      mma16816(s[0], qa[kk], b[0], b[1]);
      mma16816(s[1], qa[kk], b[2], b[3]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float z[4];
      float mt = m[h];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = j0 + (e >> 1) * 8 + 2 * (lane & 3) + (e & 1);
        z[e] = j < total ? s[e >> 1][2 * h + (e & 1)] * cs : -INFINITY;
        mt = fmaxf(mt, z[e]);
      }
      mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 1));
      mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 2));
      const float corr = exp2f(m[h] - mt);                    // 0 in the first turn
      m[h] = mt;
      float add = 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float p = exp2f(z[e] - mt);
        s[e >> 1][2 * h + (e & 1)] = p;
        add += p;
      }
      l[h] = l[h] * corr + add;
      if (t > 0) {
#pragma unroll
        for (int n = 0; n < D / 8; ++n) { o[n][2 * h] *= corr; o[n][2 * h + 1] *= corr; }
      }
    }
    uint32_t ph[4], pl[4];
    split_bf16(s[0][0], s[0][1], ph[0], pl[0]);
    split_bf16(s[0][2], s[0][3], ph[1], pl[1]);
    split_bf16(s[1][0], s[1][1], ph[2], pl[2]);
    split_bf16(s[1][2], s[1][3], ph[3], pl[3]);
#pragma unroll
    for (int nn = 0; nn < D / 16; ++nn) {
      uint32_t b[4];                            // 16 dimensions: two n-tiles, each with both halves of the 16 keys
      ldsm4_trans(v_sm + at(lane & 15, 2 * nn + (lane >> 4)), b);
      mma16816(o[2 * nn], ph, b[0], b[1]);
      mma16816(o[2 * nn + 1], ph, b[2], b[3]);
      mma16816(o[2 * nn], pl, b[0], b[1]);
      mma16816(o[2 * nn + 1], pl, b[2], b[3]);
    }
    // append: the new rows of this turn go from shared memory to rows [stored, total) of the cache
    if (appends && j0 + kMmaRows > stored) {
      uint4* kd = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(a.k_plane) + off * D);
      uint4* vd = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(a.v_plane) + off * D);
      const unsigned char* kb = sm + TILE + warp * 2 * TILE;
#pragma unroll
      for (int i = 0; i < kMmaRows * PIECES / 32; ++i) {
        const int v = lane + i * 32, r = v / PIECES, c = v % PIECES, j = j0 + r;
        if (j >= stored && j < total) {
          kd[(size_t)j * PIECES + c] = *reinterpret_cast<const uint4*>(kb + at(r, c));
          vd[(size_t)j * PIECES + c] = *reinterpret_cast<const uint4*>(kb + TILE + at(r, c));
        }
      }
      const int j = j0 + lane;
      if (lane < kMmaRows && j >= stored && j < total) a.pos_plane[off + j] = a.pos_base + (j - stored);
    }
    __syncwarp();                               // the tiles are refilled, or hold the outputs below
  }

  // merge of the warps: unnormalised outputs in the warp's own tiles (pairs of columns spread over
  // the banks), (max, sum) of every row beside them
  const int g = lane >> 2;
  float* ob = reinterpret_cast<float*>(sm + TILE + warp * 2 * TILE);
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
#pragma unroll
  for (int v = tid; v < kMmaRows * PIECES; v += W * 32) {
    const int r = v / PIECES, c = v % PIECES;
    float2 ml[W];
    float top = -INFINITY;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      ml[w] = row_ml[w][r];
      top = fmaxf(top, ml[w].x);
    }
    float sum = 0.f, acc[8] = {};
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float wt = exp2f(ml[w].x - top);    // 0 for a warp without keys
      sum = fmaf(wt, ml[w].y, sum);
      const float* src = reinterpret_cast<const float*>(sm + TILE + w * 2 * TILE) + r * D;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 f = *reinterpret_cast<const float2*>(src + 2 * ((4 * c + e) ^ ((r & 3) << 2)));
        acc[2 * e] = fmaf(wt, f.x, acc[2 * e]);
        acc[2 * e + 1] = fmaf(wt, f.y, acc[2 * e + 1]);
      }
    }
    if (q0 + r < a.n_new) {
      const float inv = 1.f / sum;
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 hh = __floats2bfloat162_rn(acc[2 * e] * inv, acc[2 * e + 1] * inv);
        w[e] = *reinterpret_cast<const uint32_t*>(&hh);
      }
      *reinterpret_cast<uint4*>(out + ((size_t)bh * a.n_new + q0 + r) * D + c * 8) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  // the launch behind this one relies on everything ahead of this grid being complete once it is
  if (bh == 0 && blockIdx.x == 0 && tid == 0) pdl_grid_wait();
}

}  // namespace

// The small kernel against the tcgen05 one, by the time either takes in microseconds (measured over 21 to
// 256 heads, 25 to 121 queries and 55 to 286 keys): 2 and 1.75 (head_dim 128) or 0.72 (64) per turn of 64
// keys and CTA that an SM has to do, against 5.5 and 0.9 per 128 keys and wave of 128-row tiles.
// 36 queries, 57 keys, 32 heads x 128: 3.7 against 6.4; 64 queries, 121 keys: 5.5 against 6.7 with 32
// heads, 8.9 against 7.5 with 64; 36 queries, 66 keys, 240 heads x 64: 9.1 against 13.0.
bool attend_small_serves(const StepArgs& a) {
  if (!attend_tc_serves(a, HACK_BF16)) return true;
  const int heads = a.batch * a.n_heads, keys = a.kept[0] > a.kept[1] ? a.kept[0] : a.kept[1];
  if (heads > 65535) return false;              // the heads are the second dimension of its grid
  const float sms = (float)sm_count();
  const int ctas = heads * ((a.n_new + kMmaRows - 1) / kMmaRows);
  const int turns = (keys + 4 * kMmaRows - 1) / (4 * kMmaRows);
  const float load = ctas <= sms ? (turns + 1) / 2 : turns * (ctas / sms);
  const int tiles = heads * ((a.n_new + 127) / 128);
  const int waves = (tiles + sm_count() - 1) / sm_count();
  return 2.f + (a.head_dim == 128 ? 1.75f : 0.72f) * load < waves * (5.5f + 0.9f * ((keys + 127) / 128));
}

int launch_attend_small(const StepArgs& a, int dtype, const void* q, const void* k_new, const void* v_new, void* out,
                        cudaStream_t st, bool after_compression) {
  const int heads = a.batch * a.n_heads;
  if (dtype == HACK_F32) {
    const dim3 grid((a.n_new + kWarps - 1) / kWarps, heads), block(kWarps * 32);
    const float* qp = static_cast<const float*>(q);
    const float* kp = static_cast<const float*>(k_new);
    const float* vp = static_cast<const float*>(v_new);
    float* op = static_cast<float*>(out);
    if (a.head_dim == 64) launch_k(append_attend_small_kernel<float, 64>, grid, block, 0, st, a, qp, kp, vp, op);
    else launch_k(append_attend_small_kernel<float, 128>, grid, block, 0, st, a, qp, kp, vp, op);
  } else {
    const dim3 grid((a.n_new + kMmaRows - 1) / kMmaRows, heads);
    const __nv_bfloat16* qp = static_cast<const __nv_bfloat16*>(q);
    const __nv_bfloat16* kp = static_cast<const __nv_bfloat16*>(k_new);
    const __nv_bfloat16* vp = static_cast<const __nv_bfloat16*>(v_new);
    __nv_bfloat16* op = static_cast<__nv_bfloat16*>(out);
    auto go = [&](auto kern, int warps, size_t smem) {
      if (!allow_dynamic_smem(kern, smem)) return -1;
      launch_k(kern, grid, dim3(warps * 32), smem, st, a, qp, kp, vp, op, (int)after_compression);
      return launched(1);
    };
    // eight warps once a CTA of four would need a second trip to memory, while that leaves every CTA an SM
    // (64 queries, 121 keys, 32 heads x 128: 5.6 -> 5.4 us; 240 heads x 64, 36 queries, 66 keys: 9.0 -> 11.6)
    const bool wide = std::max(a.kept[0], a.kept[1]) > 4 * kMmaRows && (int)(grid.x * grid.y) <= sm_count();
    if (a.head_dim == 64)
      return wide ? go(append_attend_mma_kernel<64, 8>, 8, mma_smem_bytes<64, 8>()) : go(append_attend_mma_kernel<64, 4>, 4, mma_smem_bytes<64, 4>());
    return wide ? go(append_attend_mma_kernel<128, 8>, 8, mma_smem_bytes<128, 8>()) : go(append_attend_mma_kernel<128, 4>, 4, mma_smem_bytes<128, 4>());
  }
  return launched(1);
}

}  // namespace hack
