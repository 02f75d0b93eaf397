// What the one-launch forms of a small step that evicts (step_small.cu, step_small_f32.cu) share: the shape of
// a launch and the selection of a head's survivors by one block.
#pragma once

#include "hack_internal.h"
#include "launch_plans.h"

namespace hack {
namespace small_step {

constexpr int kRangeBins = 256;                 // bins of the selection's histogram; one more for protected rows

template <typename T, typename... KArgs>
int launch_step(void (*kern)(KArgs...), const StepArgs& a, const StepShape& s, size_t smem, const void* q, const void* k_new,
                const void* v_new, void* out, cudaStream_t st) {
  if (!allow_dynamic_smem(kern, kSmemCta)) return -1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s.ctas, a.batch * a.n_heads);
  cfg.blockDim = dim3(kStepThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = s.ctas;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = s.ctas > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kern, a, static_cast<const T*>(q), static_cast<const T*>(k_new), static_cast<const T*>(v_new),
                     static_cast<T*>(out), s);
  return launched(1);
}

#if defined(__CUDACC__)
__device__ __forceinline__ uint32_t order_key(float f) {     // larger float -> larger key, never the top one
  const uint32_t u = __float_as_uint(f);
  return min((u & 0x80000000u) ? ~u : (u | 0x80000000u), 0xfffffffeu);
}
// Protected candidates of structural heads carry the top key.
__device__ __forceinline__ bool is_protected(const StepArgs& a, int ctx, int j) {
  return ctx == 0 && (j < a.t_init || (a.protect_new && j >= a.stored[0]));
}

struct PickShared {
  int hist[kRangeBins + 32];
  uint32_t range[2];                            // least and greatest key
  int n_in;
  uint32_t words[kMaxRows / 32];
};
__device__ __forceinline__ void pick_init(PickShared& ps) {
#pragma unroll 1
  for (int i = threadIdx.x; i < kRangeBins + 32; i += kStepThreads) ps.hist[i] = 0;
  if (threadIdx.x == 0) { ps.range[0] = 0xffffffffu; ps.range[1] = 0u; ps.n_in = 0; }
}

// The ascending list of the n_keep greatest of the keys key[0, cand), ties to the lower candidate, by the
// whole block.  lo, hi: least and greatest unprotected key this thread has written.  The list is complete
// after the caller's next block barrier.  MINE: keys per thread.
template <int MINE>
__device__ __forceinline__ void pick(const StepArgs& a, PickShared& ps, const uint32_t* key, int32_t* list, int cand, int n_keep,
                                     uint32_t lo, uint32_t hi) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    atomicMin(&ps.range[0], lo);
    atomicMax(&ps.range[1], hi);
  }
  __syncthreads();
  // the n_keep greatest keys: one histogram over their range finds the bin of the last survivor, whose
  // entries are ranked by comparison; protected rows have a bin of their own above all others
  lo = ps.range[0];
  hi = ps.range[1];
  const int shift = hi <= lo ? 0 : max(0, 32 - __clz(hi - lo) - 8);
  auto bin_of = [&](uint32_t k) { return k == 0xffffffffu ? kRangeBins : (int)((k - lo) >> shift); };
  uint32_t mine[MINE];
#pragma unroll
  for (int u = 0; u < MINE; ++u) {
    const int j = tid + u * kStepThreads;
    mine[u] = j < cand ? key[j] : 0u;
    if (j < cand) atomicAdd(&ps.hist[bin_of(mine[u])], 1);
  }
  __syncthreads();
  int digit, need;                            // found by every warp for itself
  {
    constexpr int PER = (kRangeBins + 32) / 32;              // lane 0 has the top bins
    int c[PER], sum = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) { c[i] = ps.hist[kRangeBins + 31 - PER * lane - i]; sum += c[i]; }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += n;
    }
    int cum = incl - sum, d = 0, rest = 0;
    const bool here = cum < n_keep && n_keep <= incl;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      if (cum < n_keep && n_keep <= cum + c[i]) { d = kRangeBins + 31 - PER * lane - i; rest = n_keep - cum; }
      cum += c[i];
    }
    const int src = __ffs(__ballot_sync(0xffffffffu, here)) - 1;
    digit = __shfl_sync(0xffffffffu, d, src);
    need = __shfl_sync(0xffffffffu, rest, src);
  }
  int32_t* in = list;                         // the bin's entries, until the list is written
#pragma unroll
  for (int u = 0; u < MINE; ++u) {
    const int j = tid + u * kStepThreads;
    if (j < cand && bin_of(mine[u]) == digit) in[atomicAdd(&ps.n_in, 1)] = j;
  }
  __syncthreads();
  const int n_bin = ps.n_in;
  bool keep[MINE];
#pragma unroll
  for (int u = 0; u < MINE; ++u) {
    const int j = tid + u * kStepThreads;
    const int b = j < cand ? bin_of(mine[u]) : -1;
    keep[u] = b >= digit;
    if (b == digit && need < n_bin) {
      int above = 0;                          // ties go to the lower candidate
#pragma unroll 4
      for (int i = 0; i < n_bin; ++i) {
        const int o = in[i];
        const uint32_t k = key[o];
        above += k > mine[u] || (k == mine[u] && o < j);
      }
      keep[u] = above < need;
    }
    const uint32_t w = __ballot_sync(0xffffffffu, keep[u]);
    if (lane == 0) ps.words[u * kStepWarps + warp] = w;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < MINE; ++u) {
    const int me = u * kStepWarps + warp;
    const int before = __reduce_add_sync(0xffffffffu, lane < me ? __popc(ps.words[lane]) : 0);
    const int o = before + __popc(ps.words[me] & ((1u << lane) - 1));
    if (keep[u] && dbg_ok(o < n_keep, a.status, 12)) list[o] = tid + u * kStepThreads;
  }
}
#endif

}  // namespace small_step
}  // namespace hack
