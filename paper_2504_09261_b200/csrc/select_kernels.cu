// Budgeted per-head selection (Eq. 10 for contextual heads, Eq. 11 for structural heads).
//
// One CTA per (batch, head).  The n largest keys are found exactly with an 8-bit-digit radix
// select over the fp32 bit patterns (4 histogram passes in shared memory), ties at the threshold
// going to the lower candidate index; protected candidates of structural heads carry the maximal
// key so that they are always inside the kept set.  A final ordered pass turns the keep flags
// into an ascending index list with a block-wide prefix sum.
//
// Fast path (up to kSelThreads * kMaxPerThread candidates): every thread keeps a contiguous run
// of keys in registers, histogram updates are aggregated per warp before they touch shared
// memory (scores of one head share their leading bits, so plain atomics would serialise), the
// digit holding the wanted rank is located by one warp, and the index list is produced with a
// single block scan.  Longer candidate lists take the general path that re-reads the scores.
#include "hack_internal.h"
#include "launch_plans.h"

namespace hack {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kMaxPerThread = 16;

// Order-preserving map from fp32 bits to unsigned (larger float -> larger key).
__device__ __forceinline__ uint32_t orderable(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

struct HeadView {
  const float* s;
  int cand, stored, t_init, protect_new, structural;
  __device__ __forceinline__ uint32_t key(int j) const {
    if (structural && (j < t_init || (protect_new && j >= stored))) return 0xffffffffu;
    const uint32_t k = orderable(s[j]);
    return k == 0xffffffffu ? 0xfffffffeu : k;   // keep the top key for protected entries only
  }
};

// Exclusive prefix sum of one value per thread over the CTA; also returns the CTA total.
__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_sums, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += n;
  }
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int w = warp_sums[lane];
    int wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += n;
    }
    warp_sums[lane] = wi - w;
    if (lane == 31) warp_sums[32] = wi;
  }
  __syncthreads();
  const int res = warp_sums[warp] + incl - v;
  total = warp_sums[32];
  __syncthreads();
  return res;
}

// Warp 0 finds the digit d (scanning from 255 down) at which the running count reaches `need`:
// sum_{b > d} hist[b] < need <= sum_{b >= d} hist[b].  Returns through shared memory (sh_count: the entries of bin d, if asked for).
__device__ __forceinline__ void locate_digit(const int* hist, int need, int* sh_digit, int* sh_need, int* sh_count = nullptr) {
  const int lane = threadIdx.x & 31;
  // lane l owns bins 255 - 8l ... 248 - 8l (descending), so lane order == descending bin order
  int c[8];
  int sum = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) { c[i] = hist[255 - 8 * lane - i]; sum += c[i]; }
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += n;
  }
  const int before = incl - sum;               // keys in bins above this lane's bins
  if (before < need && need <= incl) {
    int cum = before;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (cum < need && need <= cum + c[i]) {
        *sh_digit = 255 - 8 * lane - i;
        *sh_need = need - cum;
        if (sh_count) *sh_count = c[i];
      }
      cum += c[i];
    }
  }
}

// The ascending list of one head into `out` (global or shared memory), by the whole CTA.
template <int E>
__device__ __forceinline__ void select_list(const StepArgs& a, const float* scores, int bh, int ctx, int32_t* out) {
  const int cand = a.cand[ctx], n_keep = a.kept[ctx];
  const int tid = threadIdx.x, lane = tid & 31;
  if (!a.trig[ctx] || n_keep >= cand) {           // nothing to evict: identity list
    for (int j = tid; j < cand; j += kSelThreads) out[j] = j;
    return;
  }
  HeadView hv{scores + (size_t)bh * a.cand_stride, cand, a.stored[ctx], a.t_init, a.protect_new, ctx == 0};

  __shared__ int hist[256];
  __shared__ int sh_digit, sh_need, sh_count;
  __shared__ int warp_sums[33];

  // thread t owns candidates [t*E, t*E + E)
  const int j0 = tid * E;
  uint32_t key[E];
#pragma unroll
  for (int e = 0; e < E; ++e) key[e] = (j0 + e < cand) ? hv.key(j0 + e) : 0u;

  uint32_t prefix = 0, mask = 0;
  int need = n_keep;                               // rank (from the top) still to be located
#pragma unroll 1
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const bool in = (j0 + e < cand) && ((key[e] & mask) == prefix);
      const uint32_t digit = in ? ((key[e] >> shift) & 255u) : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, digit);
      if (in && lane == __ffs(peers) - 1) atomicAdd(&hist[digit], __popc(peers));
    }
    __syncthreads();
    if (tid < 32) locate_digit(hist, need, &sh_digit, &sh_need, &sh_count);
    __syncthreads();
    prefix |= (uint32_t)sh_digit << shift;
    need = sh_need;
    mask |= 255u << shift;
    // every entry of the located bin survives: those above prefix and, at most `need`, those equal to it
    if (need == sh_count) break;
  }
  // prefix = key of the n_keep-th largest element (or its digits so far); `need` of the entries equal to it survive
  const uint32_t thr = prefix;
  int gt = 0, eq = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const bool in = j0 + e < cand;
    gt += in && key[e] > thr;
    eq += in && key[e] == thr;
  }
  int total;
  const int packed = block_exclusive_scan(gt | (eq << 16), warp_sums, total);
  int gt_before = packed & 0xffff, eq_before = packed >> 16;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const bool in = j0 + e < cand;
    if (in && key[e] > thr) {
      const int o = gt_before + min(eq_before, need);
      if (dbg_ok(o >= 0 && o < n_keep, a.status, 4)) out[o] = j0 + e;
      ++gt_before;
    } else if (in && key[e] == thr) {
      if (eq_before < need && dbg_ok(gt_before + eq_before < n_keep, a.status, 4)) out[gt_before + eq_before] = j0 + e;
      ++eq_before;
    }
  }
}

template <int E>
__global__ void __launch_bounds__(kSelThreads)
select_reg_kernel(const StepArgs a, const float* __restrict__ scores, int32_t* __restrict__ idx,
                  int32_t* __restrict__ kept_out) {
  pdl_wait();
  const int bh = blockIdx.x;
  const int ctx = a.is_ctx[bh % a.n_heads];
  if (threadIdx.x == 0 && kept_out) kept_out[bh] = a.kept[ctx];
  select_list<E>(a, scores, bh, ctx, idx + (size_t)bh * a.kept_stride);
}

// Selection and in-place compaction of small heads in one launch: the list stays in shared memory and
// the CTA moves the rows itself, kMoveRun 16-byte pieces of K and of V per thread and round.  Entry o
// of the list becomes row o; a round's destinations lie at or before its own cache sources and
// before those of every later round, so reading a round before writing it is enough.  Three launches of 3
// to 5 us that wait for each other become one where a head's rows are a few microseconds for one SM
// (kSmallMoveBytes); step of 16 fp32 heads x 64, 374 kept rows: 36.0 against 40.4 us, 34 rows 20.4 against 24.6.
// Where there are SMs to spare a cluster of up to four CTAs moves a head's rows (move_ctas); each forms the whole list for
// itself.
constexpr int kMoveRun = 4;

template <int E>
__global__ void __launch_bounds__(kSelThreads)
select_move_kernel(const StepArgs a, const float* __restrict__ scores, const uint4* __restrict__ k_new,
                   const uint4* __restrict__ v_new, int row_pieces, int cl) {
  pdl_wait();
  const int bh = blockIdx.x / cl, rank = blockIdx.x % cl;
  const int ctx = a.is_ctx[bh % a.n_heads];
  const int stored = a.stored[ctx], n_keep = a.kept[ctx];
  extern __shared__ int32_t list[];               // [largest kept length]
  select_list<E>(a, scores, bh, ctx, list);
  __syncthreads();
  const int tid = threadIdx.x;
  const size_t off = a.row_off[bh];
  uint4* kp = reinterpret_cast<uint4*>(a.k_plane) + off * row_pieces;
  uint4* vp = reinterpret_cast<uint4*>(a.v_plane) + off * row_pieces;
  const uint4* kn = k_new + (size_t)bh * a.n_new * row_pieces;
  const uint4* vn = v_new + (size_t)bh * a.n_new * row_pieces;
  int32_t* pos = a.pos_plane + off;
  const int piece = tid % row_pieces, rsub = tid / row_pieces, rows = kSelThreads / row_pieces;   // row_pieces divides kSelThreads
  // stored rows that stay where they are need not be touched
  for (int c0 = 0; c0 < n_keep; c0 += cl * rows * kMoveRun) {
    uint4 kv[kMoveRun], vv[kMoveRun];
    int p[kMoveRun];
    bool mv[kMoveRun];
#pragma unroll
    for (int u = 0; u < kMoveRun; ++u) {
      const int r = c0 + (u * cl + rank) * rows + rsub;
      mv[u] = false;
      if (r < n_keep) {
        const int src = list[r];
        if (src != r || src >= stored) {
          if (!dbg_ok(src >= r && src < stored + a.n_new && r < a.cap[ctx], a.status, 11)) continue;
          mv[u] = true;
          const size_t at = (size_t)(src < stored ? src : src - stored) * row_pieces + piece;
          kv[u] = src < stored ? kp[at] : kn[at];
          vv[u] = src < stored ? vp[at] : vn[at];
          if (piece == 0) p[u] = src < stored ? pos[src] : a.pos_base + (src - stored);
        }
      }
    }
    // every source of the round has been read (with memory ordering: the loads need not have landed in registers)
    if (cl > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
#pragma unroll
    for (int u = 0; u < kMoveRun; ++u) {
      if (mv[u]) {
        const int r = c0 + (u * cl + rank) * rows + rsub;
        kp[(size_t)r * row_pieces + piece] = kv[u];
        vp[(size_t)r * row_pieces + piece] = vv[u];
        if (piece == 0) pos[r] = p[u];
      }
    }
  }
}

// General path: any candidate count; keys are recomputed from the scores in every pass.
__global__ void __launch_bounds__(kSelThreads)
select_kernel(const StepArgs a, const float* __restrict__ scores, int32_t* __restrict__ idx,
              int32_t* __restrict__ kept_out) {
  pdl_wait();
  const int bh = blockIdx.x;
  const int ctx = a.is_ctx[bh % a.n_heads];
  const int cand = a.cand[ctx], n_keep = a.kept[ctx];
  int32_t* out = idx + (size_t)bh * a.kept_stride;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0 && kept_out) kept_out[bh] = n_keep;
  if (!a.trig[ctx] || n_keep >= cand) {
    for (int j = tid; j < cand; j += kSelThreads) out[j] = j;
    return;
  }
  HeadView hv{scores + (size_t)bh * a.cand_stride, cand, a.stored[ctx], a.t_init, a.protect_new, ctx == 0};

  __shared__ int hist[256];
  __shared__ int sh_digit, sh_need;
  __shared__ int warp_sums[33];

  uint32_t prefix = 0, mask = 0;
  int need = n_keep;
  const int rounds = (cand + kSelThreads - 1) / kSelThreads;
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    for (int r = 0; r < rounds; ++r) {
      const int j = r * kSelThreads + tid;
      uint32_t k = 0;
      const bool in = j < cand && (((k = hv.key(j)) & mask) == prefix);
      const uint32_t digit = in ? ((k >> shift) & 255u) : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, digit);
      if (in && lane == __ffs(peers) - 1) atomicAdd(&hist[digit], __popc(peers));
    }
    __syncthreads();
    if (tid < 32) locate_digit(hist, need, &sh_digit, &sh_need);
    __syncthreads();
    prefix |= (uint32_t)sh_digit << shift;
    need = sh_need;
    mask |= 255u << shift;
  }
  const uint32_t thr = prefix;
  int out_base = 0, eq_base = 0;
  for (int base = 0; base < cand; base += kSelThreads) {
    const int j = base + tid;
    uint32_t k = 0;
    const bool in = j < cand;
    if (in) k = hv.key(j);
    const int gt = in && k > thr;
    const int eq = in && k == thr;
    int total;
    const int packed = block_exclusive_scan(gt | (eq << 16), warp_sums, total);
    const int gt_before = packed & 0xffff, eq_before = eq_base + (packed >> 16);
    // entries equal to the threshold are kept while their running rank is below `need`
    const int pos = out_base + gt_before + min(eq_before, need) - min(eq_base, need);
    if ((gt || (eq && eq_before < need)) && dbg_ok(pos >= 0 && pos < n_keep, a.status, 5)) out[pos] = j;
    out_base += (total & 0xffff) + min(eq_base + (total >> 16), need) - min(eq_base, need);
    eq_base += total >> 16;
  }
}

}  // namespace

int launch_select_move(const StepArgs& a, int dtype, const float* scores, const void* k_new, const void* v_new, cudaStream_t st) {
  const int max_cand = a.cand[0] > a.cand[1] ? a.cand[0] : a.cand[1], max_keep = a.kept[0] > a.kept[1] ? a.kept[0] : a.kept[1];
  const int row_pieces = a.head_dim * (dtype == HACK_F32 ? 4 : 2) / 16;
  if (max_cand > 4 * kSelThreads || (size_t)max_keep * row_pieces * 32 > kSmallMoveBytes) return 0;
  const int heads = a.batch * a.n_heads;
  const simt::SimtPlan plan = simt::simt_plan(a.head_dim, a.n_new, a.kept, a.heads_of, sm_count());
  const int beside = dtype == HACK_F32 && a.head_dim == 64 && plan.cluster == 1 ? plan.ctas : 0;
  const int cl = move_ctas(heads, beside, sm_count(), [](int ctas) {
    return cluster_places(reinterpret_cast<const void*>(select_move_kernel<4>), ctas, kSelThreads, 4 * kSelThreads * sizeof(int32_t));
  });
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(heads * cl);
  cfg.blockDim = dim3(kSelThreads);
  cfg.dynamicSmemBytes = (size_t)max_cand * sizeof(int32_t);
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
  cudaLaunchKernelEx(&cfg, select_move_kernel<4>, a, scores, static_cast<const uint4*>(k_new), static_cast<const uint4*>(v_new), row_pieces, cl);
  return launched(1);
}

int launch_select(const StepArgs& a, const float* scores, int32_t* idx, int32_t* kept_out,
                  cudaStream_t st) {
  const int grid = a.batch * a.n_heads;
  const int max_cand = a.cand[0] > a.cand[1] ? a.cand[0] : a.cand[1];
  const int per_thread = (max_cand + kSelThreads - 1) / kSelThreads;
  if (per_thread <= 4) launch_k(select_reg_kernel<4>, grid, kSelThreads, 0, st, a, scores, idx, kept_out);
  else if (per_thread <= 8) launch_k(select_reg_kernel<8>, grid, kSelThreads, 0, st, a, scores, idx, kept_out);
  else if (per_thread <= 12) launch_k(select_reg_kernel<12>, grid, kSelThreads, 0, st, a, scores, idx, kept_out);
  else if (per_thread <= kMaxPerThread) launch_k(select_reg_kernel<kMaxPerThread>, grid, kSelThreads, 0, st, a, scores, idx, kept_out);
  else launch_k(select_kernel, grid, kSelThreads, 0, st, a, scores, idx, kept_out);
  return launched(1);
}

}  // namespace hack
