// Internal declarations shared by the host API and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "hack.h"

namespace hack {

constexpr int kMaxObs = 32;        // rows of the observation window the kernels are built for
constexpr int kScoreChunk = 128;   // candidate keys per CTA in the SIMT scoring pass

// Everything a kernel needs to know about one (layer, scale) step.  Passed by value.
// Per-type arrays are indexed by the head's mask byte: [0] structural, [1] contextual.
struct StepArgs {
  int n_heads, batch, head_dim;
  int n_new;            // N_k
  int stored[2];        // L before the step
  int cand[2];          // T' = L + N_k
  int kept[2];          // length after the step
  int cap[2];           // rows a head of this type owns in the planes (checked builds compare against it)
  int trig[2];          // compression triggered for this type
  int heads_of[2];      // (batch, head) pairs of this type in the layer
  int seg_new[2];       // tensor-core attention reads this type's new rows from the caller's K/V and
                        // appends them itself (the type keeps the whole new scale in this step)
  long long wait_cycles;   // limit of every bounded device-side wait of the step's kernels
  int n_obs_rows;       // min(N_obs, N_k)
  int obs_first, obs_span;      // observation row i = obs_first + floor(i * obs_span / n_obs_rows) ...
  const int32_t* obs_rows;      // ... unless the caller supplied the rows (device, [n_obs_rows])
  int obs_full;                 // every query observes: the scoring kernels run once per group of 32 rows
  int score_accumulate;         // the scores of this round are added to those already there
  float sm_scale;
  int t_init;           // tokens in the always-kept leading scales (structural heads)
  int protect_new;      // structural heads: the new scale's tokens are protected
  int pos_base;         // global position of the new scale's first token (T_{k-1})
  int cand_stride, kept_stride;
  const uint8_t* is_ctx;   // device, [n_heads] of this layer
  const int32_t* row_off;  // device, [batch*n_heads] first row of each head in the planes
  void* k_plane;           // device, [rows, head_dim] of this layer
  void* v_plane;
  int32_t* pos_plane;      // device, [rows]
  int* status;             // device status word
  int32_t* n_old;          // device, [batch*n_heads]: survivors that were already stored (compaction)
  // tensor-core attention only (host pointers to 128-byte tensor maps of this layer's planes)
  const void* k_map;
  const void* v_map;
  const int32_t* head_order;   // device, [2][batch*n_heads]: structural heads first, contextual heads first
  float* simt_partial;         // fp32 attention: device scratch of query tiles that CTAs share (simt_partial_floats) ...
  int32_t* simt_arrived;       // ... and their counters (simt_arrived_words), zero between launches
};

struct Scratch {
  float* logits;    // [batch*n_heads, kMaxObs, cand_stride]
  float* partials;  // [batch*n_heads, max_chunks, kMaxObs, 2]  (row max, row sum per chunk)
  int max_chunks;
};

// Scratch of the final-scale merge of contextual heads (bf16 caches): the rows the last step
// discards, their list, inverse key norms, and the counterpart and weight of every discarded row.
struct MergeScratch {
  int stride;                  // rows per (batch, head) in the arrays below
  __nv_bfloat16* ev_k;         // [b*H, stride, D] discarded key rows
  __nv_bfloat16* ev_v;         // [b*H, stride, D] discarded value rows
  int32_t* ev_idx;             // [b*H, stride] their candidate indices, ascending
  float* ev_inv_norm;          // [b*H, stride] 1 / |k_e|
  float* kept_inv_norm;        // [b*H, kept_stride] 1 / |k_c|
  int32_t* assign;             // [b*H, stride] retained row each discarded row is folded into
  float* weight;               // [b*H, stride] max(cosine similarity, 0)
  const void* ev_map;          // host pointer to the 128-byte tensor map over ev_k
};
// Before the compaction of the step (idx = the kept lists; listed: ms.ev_idx holds their complements already) and after it.
int launch_merge_prepare(const StepArgs& a, const MergeScratch& ms, const int32_t* idx, bool listed, const void* k_new,
                         const void* v_new, cudaStream_t st);
int launch_merge_finish(const StepArgs& a, const MergeScratch& ms, cudaStream_t st);

// Kernel launchers (each returns the number of kernels it enqueued, or -1 on a launch error).
int launch_score(const StepArgs& a, int dtype, const void* q, const void* k_new, float* scores,
                 const Scratch& s, cudaStream_t st);
// bf16 caches: the same scores with the logits formed on the tensor cores (two launches).
int launch_score_tc(const StepArgs& a, const void* q, const void* k_new, float* scores, const Scratch& s,
                    cudaStream_t st);
int launch_select(const StepArgs& a, const float* scores, int32_t* idx, int32_t* kept_out,
                  cudaStream_t st);
// Selection and compaction of a step in one launch, for heads of few rows.  1: launched; 0: outside what
// the kernel is for, take launch_select and launch_compact; -1: launch error.
int launch_select_move(const StepArgs& a, int dtype, const float* scores, const void* k_new, const void* v_new, cudaStream_t st);
// bf16 caches: scores only (scores != nullptr) or scoring, selection and in-place compaction of the step
// in one launch of one thread-block cluster per head.  Its CTAs if launched; 0: the step is outside what
// the kernel holds, take the separate launches; -1: launch error.  beside_us, behind_us: SM-microseconds
// of the attention launch behind this one that can run beside it, and that need its result.  shape: the
// launch shape of this step as found before (0: not yet), kept by the caller.  kept_list, gone_list: the lists of
// the contextual heads and their complements go there, ascending, and their rows stay where they are (a step that merges).
int launch_compress_cluster(const StepArgs& a, const void* q, const void* k_new, const void* v_new, float* scores,
                            cudaStream_t st, float beside_us = 0.f, float behind_us = 0.f, uint16_t* shape = nullptr,
                            int32_t* kept_list = nullptr, int32_t* gone_list = nullptr, int gone_stride = 0);
// idx == nullptr: every head appends (keeps all candidates).  idx_all: there is a list for every head; 0: for the contextual
// ones, and the stored rows that the others keep are in place already (a.trig[0] must be 0).
int launch_compact(const StepArgs& a, int dtype, const int32_t* idx, int idx_all, const void* k_new,
                   const void* v_new, cudaStream_t st);
int launch_attend(const StepArgs& a, int dtype, const void* q, void* out, cudaStream_t st);

int launch_attend_simt(const StepArgs& a, const void* q, void* out, cudaStream_t st);   // fp32 caches
// Its scratch of one cache, on the current device.
size_t simt_partial_floats(int head_dim);
size_t simt_arrived_words(int heads, int max_new);
// row_stats (optional, device [b*H, N_k, 2]): per query row the reference maximum m (raw logit
// units; within the lazy-rescaling margin of the true maximum) and l = sum_j exp2(c (z_j - m)).
// k_new / v_new (optional): the caller's K/V of this scale; head types with a.seg_new set then attend
// over [the N_k new rows read from k_new / v_new ; kept - N_k cache rows] and the kernel appends
// those rows to the cache, so no append or copy launch precedes it for them.  compression_ctas: CTAs
// of the step's compression launch when that is the launch ahead of this one in the stream (heads that
// do not depend on it then start beside it), 0 if it is not.
int launch_attend_tc(const StepArgs& a, const void* q, void* out, float* row_stats, const void* k_new,
                     const void* v_new, cudaStream_t st, int compression_ctas);
// Rough SM-microseconds of the tensor-core attention of one head type (two query tiles per CTA).
float attend_tc_sm_us(const StepArgs& a, int type);
constexpr long long kDefaultWaitCycles = 2000000000ll;   // about one second: no wait is legitimately longer
// Attention variance per (batch, head) over the compacted cache (Eq. 6) from the row statistics of
// launch_attend_tc; block_var: device scratch [b*H, max_blocks]; sigma: device [b*H].  bf16 only.
int launch_attention_variance(const StepArgs& a, const void* q, const float* row_stats, float* block_var,
                              int max_blocks, float* sigma, cudaStream_t st);
bool attend_tc_serves(const StepArgs& a, int dtype);   // the tensor-core kernel takes this step's attention
// 2-D bf16 tensor map (128 x 64 boxes, 128-byte swizzle) over rows x head_dim; false on failure.
bool make_rows_map(void* out_map, const void* base, uint64_t rows, int head_dim);

// Attention of a small step in one launch that appends as well.  bf16: any step that attend_small_serves
// (head types with a.seg_new read the caller's rows and append them; after_compression: the launch ahead in
// the stream is the step's compression launch).  fp32: steps that evict nothing, at most kSmallQueries new tokens.
int launch_attend_small(const StepArgs& a, int dtype, const void* q, const void* k_new, const void* v_new, void* out,
                        cudaStream_t st, bool after_compression = false);
bool attend_small_serves(const StepArgs& a);   // bf16: the small kernel is the one for this step's attention
constexpr int kSmallQueries = 31;

// A whole step (scores, selection, attention, compaction) in one launch, for heads that fit into shared memory:
// steps that evict and, fp32, some that do not.  1: launched; 0: outside what the kernels are for; -1: launch error.
int launch_step_small(const StepArgs& a, int dtype, const void* q, const void* k_new, const void* v_new, void* out, cudaStream_t st);
int launch_step_small_f32(const StepArgs& a, const void* q, const void* k_new, const void* v_new, void* out, cudaStream_t st);

// Start of a running softmax maximum.  Finite, so that logits of -inf (products that overflow) weigh nothing even
// where they are all that a tile, or the share of a warp, has: -inf - (-inf) is no number.
constexpr float kNoLogit = -3.402823466e38f;

constexpr int kTcMinQueries = 32;   // below this the small kernel serves every bf16 step

void set_error(const std::string& msg);
// Number of SMs of the current device (asked once per device); the grid heuristics size to it.
int sm_count();
// Clusters of `ctas` CTAs of a kernel that find a place at once on an empty chip (asked once per kernel, size and device; its
// opt-in to the shared memory comes first).
int cluster_places(const void* kern, int ctas, int threads, size_t smem);

// Every kernel of the step is launched with programmatic stream serialisation: its CTAs may start
// while the previous kernel of the stream drains, and stop at pdl_wait() until that kernel has
// completed and its writes are visible.  Nothing that another kernel produces or still reads is
// touched before pdl_wait().
template <typename... KArgs, typename... Args>
inline void launch_k(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}
// Checked build (-DHACK_DEBUG_CHECKS), the stand-in for a memory checker: every ragged index a
// kernel forms (a list entry, a row of a head, a candidate, a slot of the index list) is compared
// with its bound before it is used; on a violation the access is skipped and the code of the site
// goes to the status word (nothing traps), which hack_poll_status reports.  The planes of a checked
// build also carry a canary row behind every head, verified on the host by hack_debug_check.  In
// the normal build the test is constant-true and costs nothing.
constexpr int kDebugCodeBase = 100;     // status codes of the bounds checks start here
constexpr unsigned char kCanaryByte = 0x5A;
#if defined(__CUDACC__)
#if defined(HACK_DEBUG_CHECKS)
__device__ __forceinline__ bool dbg_ok(bool cond, int* status, int code) {
  if (!cond) atomicExch(status, kDebugCodeBase + code);
  return cond;
}
#else
__device__ __forceinline__ bool dbg_ok(bool, int*, int) { return true; }
#endif
// Query row that serves as observation row i (Eq. 9's subset Q~).
__device__ __forceinline__ int obs_row(const StepArgs& a, int i) {
  // (i < 32 and obs_span <= N_k: the product fits 32 bits, whose division is a third of a 64-bit one's work)
  return a.obs_rows ? a.obs_rows[i] : a.obs_first + (int)(((uint32_t)i * (uint32_t)a.obs_span) / (uint32_t)a.n_obs_rows);
}
__device__ __forceinline__ void pdl_grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() {
  pdl_grid_wait();
  pdl_launch_dependents();
}
#endif

// Opt-in to more than 48 KB of dynamic shared memory.  The attribute belongs to the (function,
// device) pair, so it is set once per pair, on the device that is current (thread safe).
// False (with the error text recorded) if the driver refuses; the pair is then asked again next time.
bool allow_dynamic_smem_impl(const void* kern, size_t bytes);
template <typename F>
inline bool allow_dynamic_smem(F* kern, size_t bytes) {
  return allow_dynamic_smem_impl(reinterpret_cast<const void*>(kern), bytes);
}

// After a kernel launch: n if it was accepted, else -1 with the CUDA error text recorded.
inline int launched(int n) {
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return n;
  set_error(std::string("kernel launch: ") + cudaGetErrorString(e));
  return -1;
}

}  // namespace hack
