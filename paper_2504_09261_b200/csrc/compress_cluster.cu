// Compression of one step in ONE launch for bf16 caches: subset-attention scores (Eq. 9), budgeted
// selection (Eq. 10 for contextual heads, Eq. 11 for structural heads) and in-place compaction of
// the ragged per-head cache (the gathers of Eq. 10-11).
//
// Every (batch, head) is independent of every other, so a thread-block cluster owns one head
// and nothing leaves the cluster between the first key load and the last row store.  The CTAs of
// the cluster split the head's candidate list into consecutive runs of 128-key chunks (a chunk
// never straddles the stored part and the new part of the list):
//
//   1. scores, pass 1: each CTA streams its chunks through a TMA ring and forms their logits
//      against the (at most 32) observation rows with tcgen05.mma, as score_tc.cu does, but every
//      chunk keeps its own accumulator [128 lanes x 32 columns] in tensor memory.  The ones that do not
//      fit take turns on two bounce accumulators; the logits of ranked chunks among them go to shared
//      memory, or, past that, are formed a second time in pass 2.
//      Thread r of a consumer set owns key r of a chunk and keeps (reference maximum, sum-exp) of half
//      of the softmax rows; the 32 keys of a warp are merged by exchanging halves between lanes.
//   2. the CTAs publish their row statistics in shared memory; after a cluster barrier every CTA
//      merges all of them, in rank order, through distributed shared memory.
//   3. scores, pass 2: the logits are read back from tensor / shared memory (no second key
//      load, no second MMA) and s_j = sum_i exp(z_ij - m_i) / l_i becomes an order-preserving
//      32-bit key in shared memory (protected candidates of structural heads carry the top key).  The new
//      scale of a head that keeps it whole ends with pass 1: it is neither ranked nor listed.
//   4. exact radix select over the cluster: digits of 12, 12 and 8 bits; every CTA builds the
//      histogram of its own keys (the first one while it forms them) and publishes it in groups of 16
//      bins; after a cluster barrier a thread adds one group over the cluster (4 bytes per CTA instead
//      of 32), and one warp reads the bins of the group that holds the wanted rank, which also gives
//      every CTA's counts and so its offset in the head's index list.  Once at most kBinMax entries are
//      left in the located bin they are ranked by comparison (a digit costs 1.3-2 us, the heads of a
//      launch need one to three of them, and the slowest head sets its time).  The select stops early if
//      all entries left survive.  Ties at the threshold go to the lowest indices.
//   5. ascending index list by ballot counts; every entry goes straight into the shared memory of the
//      CTA that will move it (the list never touches global memory).
//   6. compaction in rounds: entry o of the list becomes row o of the head.  In a round every CTA
//      takes a run of consecutive entries out of memory (a stored survivor comes from the head's
//      own rows, at or behind its destination; a surviving new row from the caller's K/V) into shared
//      memory, the cluster meets, and the run goes out with bulk stores.  The destinations of a round
//      lie at or before its own cache sources and before those of every later round: in place.
//      (Contextual heads of a step that merges: the list and its complement go to memory, nothing moves.)
//   7. heads that keep the whole new scale stop behind their stored survivors; the attention
//      launch reads their new rows from the caller's tensors and appends them itself.
//
// What bounds it is the chain of dependent round trips once the keys have arrived: a head of two chunks
// (head_dim 64, one CTA) takes 8.4 us, one of 50 chunks (head_dim 128, four CTAs) 35 us, of which 13 are
// the key stream.  (With the rows' statistics folded through shared memory, 16 histogram bins per thread
// and CTA read through distributed shared memory, and an exchange of counts behind the select: 13.2
// and 44 us; 7 us per digit where that traffic met the attention of the other heads.)  One CTA per
// head where the GPU is full of heads, two CTAs per SM where there are more heads than SMs: 256 heads of
// 680 candidates 51 -> 40 us per step, attention included.
// Its code runs once from front to back, right behind the attention kernel's, so every line of it comes in from L2:
// loops of unknown length are not unrolled, waits are small and a round's loads stand in one place (97 -> 69 KB of
// code; 21 heads x 128, 121 to 2 025 queries: 818 -> 798 us a layer, 256 heads x 64 37.9 -> 36.9 us a step).
// In score-only mode the kernel stops after step 3 and writes the fp32 scores (hack_score).
// Every mbarrier wait is bounded; a CTA whose wait gives up raises the status word, and the
// cluster agrees at the first exchange to skip the rest, so that every CTA still reaches every
// cluster barrier.  No load in this file uses cluster multicast.
#include <cuda.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "hack_internal.h"
#include "tc_ptx.cuh"

namespace hack {
namespace {

using namespace ptx;

constexpr int kWorkers = 256;              // warps 0-7: two sets of four, one warp per TMEM lane quadrant
constexpr int kCkThreads = kWorkers + 32;  // and one issuing warp (a consumer that also issues slowed the key stream by a fifth)
constexpr int kCkWarps = kCkThreads / 32;
constexpr int kIssueWarp = kWorkers / 32;
constexpr int kCkChunk = 128;
constexpr int kHalfObs = kMaxObs / 2;      // observation rows a consumer set takes in pass 1
constexpr int kMaxSlots = 16;              // accumulators of 32 columns in 512 columns of tensor memory
constexpr int kMaxSeq = 80;                // products per CTA: its chunks, and those formed a second time
constexpr int kMaxCluster = 8;
constexpr uint32_t kCkDrainSpins = 1u << 22;
constexpr int kMaxStages = 4;              // key tiles in flight per CTA (deeper rings measured no faster)
constexpr int kHistBins = 4096;            // bins of a 12-bit digit of the radix select
constexpr int kHistWords = kHistBins / 2;  // 16-bit counters, two per word
constexpr int kBinMax = 256;               // entries of the located bin that are ranked by comparison
constexpr int kMaxStageRows = 512;         // rows (K and V) in a CTA's staging buffers of the compaction
constexpr int kMoveBuffers = 3;            // staging buffers of the compaction: loads run two rounds ahead of the stores
constexpr size_t kSmemBudget = 227 * 1024; // dynamic shared memory a CTA may ask for ...
constexpr size_t kSmemShared = 112 * 1024; // ... and half an SM's, for two CTAs per SM
constexpr float kLazyMax = 16.0f;          // log2 units a logit may exceed a thread's reference maximum
static_assert(kHistBins == 16 * kWorkers, "a worker sums 16 bins of a histogram");
static_assert(kMaxSeq * kCkChunk < 65536, "16-bit counters per CTA");
static_assert(kBinMax < kCkThreads && 4 * (kBinMax + 1) <= kHistWords, "a thread per entry, two lists in a histogram's place");

struct CkParams {
  int cluster;                // CTAs per head
  int p_max;                  // most chunks of any CTA whose logits are read twice (sizes shared memory)
  int cpc_max;                // most chunks of any CTA
  int slots;                  // accumulators in tensor memory
  int direct;                 // chunks with an accumulator of their own; the others share the last two
  int n_over;                 // ranked chunks past the direct ones whose logits stay in shared memory; those of the rest are formed again
  int stages;                 // key tiles in the TMA ring (2 .. kMaxStages)
  int region_bytes;           // front region of shared memory: ring, observation rows, overflow logits, histograms; later the row staging
  int stage_rows;             // rows (K and V) a CTA stages in shared memory per round of the compaction
  int score_only;             // stop after the scores
  float* scores;              // [b*H, cand_stride] or nullptr
  int32_t* kept_list;         // contextual heads: their list goes here, [b*H, kept_stride], and the rest of the
  int32_t* gone_list;         // candidates here, [b*H, gone_stride], and no row is moved; or both nullptr
  int gone_stride;
  const uint4* k_new;         // caller's K/V of this scale (compaction of heads whose new rows compete)
  const uint4* v_new;
};

struct CkShared {
  uint64_t full[kMaxStages], empty[kMaxStages];
  uint64_t acc_full[kMaxSeq];
  uint64_t acc_free[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort_flag;
  int pub_abort;                              // read by the other CTAs of the cluster
  int digit, need_in_bin, bin_count;          // the located digit, the rank left inside its bin, the bin's count
  int bin_n, bin_gt;                          // this CTA's entries in the located bin; the head's above the threshold there
  int cnt_gt[kMaxCluster], cnt_eq[kMaxCluster];   // per CTA: keys above the threshold, keys in the located bin
  int warp_sums[2][kCkWarps + 3];
  float2 pub_stats[4][kMaxObs];               // per lane quadrant (max, sum-exp) of every observation row; read by the cluster
  float2 part[4][kMaxObs];                    // the same merged over the CTAs of the cluster
  float4 row_stat[kMaxObs / 2];               // (max, 1 / sum) of the whole head, two rows a piece
  uint32_t coarse[2][kWorkers];               // per 16 bins: their count << 16 | the count of all bins above them; read by the cluster
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Barrier of the cluster; for a cluster of one CTA the block's own (0.1 us instead of 0.7).
__device__ __forceinline__ void cluster_sync(int cl) {
  if (cl == 1) __syncthreads();
  else asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Execution barrier of the cluster without memory ordering: for a point that only has to come after
// every CTA's loads have landed (nothing written before it is read by another CTA after it).
__device__ __forceinline__ void cluster_sync_relaxed(int cl) {
  __syncthreads();
  if (cl > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
// Address of the same shared-memory object in the CTA of rank `rank`.
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ int ld_peer_i32(uint32_t addr) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_peer_f2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_peer_u64(uint32_t addr) {
  unsigned long long v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n) : "memory");
}
__device__ __forceinline__ void st_peer_i32(uint32_t addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// False once the limit has passed or another wait of the CTA has given up (in little code; one thread writes the status word
// at the end).
__device__ __forceinline__ bool ck_wait(uint64_t* bar, uint32_t parity, CkShared* sh, int code, long long limit) {
  const uint32_t addr = smem_u32(bar);
  // a limit of a few cycles (a test's way to make a wait run out) is taken literally: the barrier is
  // tested without blocking and the clock is read after every test
  const bool brief = limit < 65536;
  if (__builtin_expect(!brief && mbar_try_wait(addr, parity), 1)) return true;
  volatile int* const flag = &sh->abort_flag;
  const long long t0 = clock64();
#pragma unroll 1
  while (!(brief ? mbar_test_wait(addr, parity) : mbar_try_wait(addr, parity))) {
    if (*flag) return false;
    if (clock64() - t0 > limit) *flag = code;
  }
  return true;
}

// Order-preserving map from fp32 bits to unsigned (larger float -> larger key).
__device__ __forceinline__ uint32_t ck_orderable(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// One more entry in bin `digit` of a histogram of 16-bit counters, two per word (a CTA holds fewer
// than 65 536 keys).  Called by whole warps; lanes that fall into the same bin add once.
__device__ __forceinline__ void hist_add(uint32_t* hist, bool in, uint32_t digit) {
  const uint32_t peers = __match_any_sync(0xffffffffu, in ? digit : 0xffffffffu);
  if (in && (threadIdx.x & 31) == __ffs(peers) - 1)
    atomicAdd(&hist[digit >> 1], (uint32_t)__popc(peers) << (16 * (digit & 1)));
}

// (max, sum-exp) of two disjoint sets of keys; a set without keys is (-inf, 0).
__device__ __forceinline__ float2 merge_stats(float2 x, float2 y) {
  const float m = fmaxf(x.x, y.x);
  const float lx = x.y == 0.f ? 0.f : x.y * ex2(x.x - m), ly = y.y == 0.f ? 0.f : y.y * ex2(y.x - m);
  return make_float2(m, lx + ly);
}

// Sum over the CTA's warps of one value per warp: what the warps before this one hold, and the total.
// `sums` is free again after the next block barrier.
__device__ __forceinline__ int ck_warp_prefix(int v, int* sums, int& total) {
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) sums[warp] = v;
  __syncthreads();
  int before = 0;
  total = 0;
#pragma unroll
  for (int w = 0; w < kCkWarps; ++w) {
    const int x = sums[w];
    if (w < warp) before += x;
    total += x;
  }
  return before;
}
// Exclusive prefix sum of one value per thread over the CTA, and the total.
__device__ __forceinline__ int ck_block_scan(int v, int* sums, int& total) {
  const int lane = threadIdx.x & 31;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += n;
  }
  return ck_warp_prefix(__shfl_sync(0xffffffffu, incl, 31), sums, total) + incl - v;
}

// kAgain: some CTA holds ranked chunks whose logits are formed a second time (a form of its own: the code
// for it costs a launch of few chunks 0.3 us).
// kLists: a step that merges (kept_list, gone_list).
template <int D, bool kAgain, bool kLists = false>
__global__ void __launch_bounds__(kCkThreads, 2)
compress_cluster_kernel(const __grid_constant__ CUtensorMap tm_cache, const __grid_constant__ CUtensorMap tm_new,
                        const StepArgs a, const __nv_bfloat16* __restrict__ q, const CkParams p) {
  constexpr int SUB = D / 64;
  constexpr uint32_t K_SUB_BYTES = kCkChunk * 128;
  constexpr uint32_t Q_SUB_BYTES = kMaxObs * 128;
  constexpr uint32_t K_BYTES = SUB * K_SUB_BYTES;
  constexpr int PIECES = D * 2 / 16;                      // 16-byte pieces per row
  const int STAGES = p.stages;
  const uint32_t RING_BYTES = (uint32_t)STAGES * K_BYTES;

  // Nothing that another kernel writes is touched before the dependency wait below: the head-type
  // table is written when the cache is created, the step's lengths travel in the arguments.
  const int bh = blockIdx.y;
  const int ctx = a.is_ctx[bh % a.n_heads];
  if (!a.trig[ctx]) {                                     // the whole cluster leaves together
    pdl_wait();
    return;
  }
  const int CL = p.cluster;
  const int rank = CL > 1 ? (int)cluster_rank() : 0;
  const int stored = a.stored[ctx], n_new = a.n_new;
  // A structural head that keeps the whole new scale ranks its stored candidates only: the new keys
  // enter the softmax denominators and are then done with.
  const bool drop_new = ctx == 0 && a.protect_new && !p.scores;
  const int n_rows = drop_new ? a.kept[ctx] - n_new : a.kept[ctx];   // survivors this kernel lists and moves
  const int n_sc = (stored + kCkChunk - 1) / kCkChunk, n_nc = (n_new + kCkChunk - 1) / kCkChunk;
  // This CTA's chunks: first a consecutive run of ranked candidates, then (drop_new) of the others.
  const int n_ranked = drop_new ? n_sc : n_sc + n_nc;
  const int cpr = (n_ranked + CL - 1) / CL, cpt = drop_new ? (n_nc + CL - 1) / CL : 0;
  const int c_begin = rank * cpr, t_begin = rank * cpt;
  const int n_p = max(0, min(cpr, n_ranked - c_begin));
  const int n_run = n_p + (drop_new ? max(0, min(cpt, n_nc - t_begin)) : 0);      // <= p.cpc_max
  // Ranked chunks whose logits are kept: with an accumulator of their own, then in shared memory.  The
  // others go through the ring and the tensor pipe a second time once the statistics are known: product
  // number n_run + x is chunk n_held + x.
  const int n_held = kAgain ? min(n_p, p.direct + p.n_over) : n_p, n_seq = n_run + n_p - n_held;
  auto chunk_of = [&](int seq) { return !kAgain || seq < n_run ? seq : n_held + seq - n_run; };
  const float zscale = a.sm_scale * 1.4426950408889634f;  // logits in log2 units
  const long long wlim = a.wait_cycles;

  extern __shared__ unsigned char smem_dyn[];
  const uint32_t raw = smem_u32(smem_dyn);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_dyn + (base - raw);
  const uint32_t k_sm = base;
  const uint32_t q_sm = base + RING_BYTES;
  float* over = reinterpret_cast<float*>(sm + RING_BYTES + SUB * Q_SUB_BYTES);            // [n_over][32][128]
  uint32_t* hist32 = reinterpret_cast<uint32_t*>(over + (size_t)p.n_over * kMaxObs * kCkChunk);   // [2][kHistWords]
  const int S_ROWS = p.stage_rows;                          // rows a CTA holds in its staging buffers
  uint32_t* keys = reinterpret_cast<uint32_t*>(sm + p.region_bytes);                            // [p_max * 128]
  int32_t* pos_stage = reinterpret_cast<int32_t*>(keys + (size_t)p.p_max * kCkChunk);          // [S_ROWS]
  int32_t* src_all = pos_stage + S_ROWS;                    // [p_max * 128 + S_ROWS]: this CTA's list entries of every round
  CkShared* sh = reinterpret_cast<CkShared*>(src_all + (size_t)p.p_max * kCkChunk + S_ROWS);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // chunk behind local index i: does it come from the cache, and its index in its part of the list
  auto chunk_part = [&](int i, bool& from_cache) -> int {
    const int chunk = i < n_p ? c_begin + i : n_sc + t_begin + (i - n_p);
    from_cache = chunk < n_sc;
    return from_cache ? chunk : chunk - n_sc;
  };
  // candidate behind slot (local chunk i, key r): is it a live entry, and its candidate index
  auto slot_info = [&](int slot, int& j) -> bool {
    bool from_cache;
    const int part_row = chunk_part(slot >> 7, from_cache) * kCkChunk + (slot & 127);
    j = (from_cache ? 0 : stored) + part_row;
    return part_row < (from_cache ? stored : n_new);
  };

  int issued = 0;                                           // issuing thread: key tiles on their way
  auto load_tile = [&](int i) {
    bool from_cache;
    const int part = chunk_part(chunk_of(i), from_cache);
    const CUtensorMap* tm = from_cache ? &tm_cache : &tm_new;
    const int row = (from_cache ? a.row_off[bh] : bh * n_new) + part * kCkChunk;
    const int s = i % STAGES;
    const uint32_t bar = smem_u32(&sh->full[s]);
    mbar_expect_tx(bar, K_BYTES);
#pragma unroll
    for (int c = 0; c < SUB; ++c) tma_load_2d(k_sm + s * K_BYTES + c * K_SUB_BYTES, tm, c * 64, row, bar);
    ++issued;
  };
  if (warp == kIssueWarp && lane == 0) {
#pragma unroll 1
    for (int s = 0; s < STAGES; ++s) { mbar_init(smem_u32(&sh->full[s]), 1); mbar_init(smem_u32(&sh->empty[s]), 1); }
#pragma unroll 1
    for (int i = 0; i < n_seq; ++i) mbar_init(smem_u32(&sh->acc_full[i]), 1);
    mbar_init(smem_u32(&sh->acc_free[0]), kWorkers / 32);   // a warp arrives once
    mbar_init(smem_u32(&sh->acc_free[1]), kWorkers / 32);
    mbar_init(smem_u32(&sh->drain), 1);
    sh->abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async();
    prefetch_tensormap(&tm_cache);
    prefetch_tensormap(&tm_new);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&sh->tmem_base), kMaxObs * p.slots);
    tmem_relinquish();
  }
  pdl_grid_wait();     // everything above overlaps the tail of the previous kernel
  // the next launch may start once every CTA holds its tensor memory
  if (warp == 0) pdl_launch_dependents();
  if (warp == kIssueWarp) {
    // the first key tiles are on their way while the other warps fetch the observation rows
    if (lane == 0)
#pragma unroll 1
      for (int i = 0; i < min(STAGES, n_seq); ++i) load_tile(i);
    __syncwarp();
  } else {
    // observation rows into the swizzled B tile; unused rows are zero
    for (int v = tid; v < kMaxObs * (D / 8); v += kWorkers) {
      const int i = v / (D / 8), c = v % (D / 8);
      uint4 val = make_uint4(0, 0, 0, 0);
      if (i < a.n_obs_rows)
        val = *reinterpret_cast<const uint4*>(q + ((size_t)bh * n_new + obs_row(a, i)) * D + c * 8);
      const uint32_t off = (c / 8) * Q_SUB_BYTES + i * 128 + (((c % 8) ^ (i & 7)) << 4);
      *reinterpret_cast<uint4*>(sm + RING_BYTES + off) = val;
    }
    fence_proxy_async();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&sh->tmem_base);

  // ------------------------------------------------------------------ 1. scores, pass 1
  const int set = warp >> 2;
  const int key_row = (warp & 3) * 32 + lane;
  const uint32_t t_lane = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
  // Chunks past the `direct` ones take turns on the last two accumulators.
  auto acc_slot = [&](int i) { return i < p.direct ? i : p.slots - 2 + ((i - p.direct) & 1); };
  // Products [from, to) (issuing thread).
  bool issue_ok = true;
  auto issue = [&](int from, int to) {
    constexpr uint32_t IDESC = idesc_bf16_f32(kCkChunk, kMaxObs, 0);
    const uint64_t q_desc = smem_desc_sw128(q_sm, 16, 1024);
#pragma unroll 1
    for (int i = from; i < to && issue_ok; ++i) {
      const int s = i % STAGES;
      bool ok = ck_wait(&sh->full[s], (i / STAGES) & 1, sh, 52, wlim);
      // a shared accumulator is free again once all consumers have read the chunk before
      if (ok && i >= p.direct)
        ok = ck_wait(&sh->acc_free[(i - p.direct) & 1], (((i - p.direct) >> 1) & 1) ^ 1, sh, 53, wlim);
      if (ok) {
        tc_fence_after();
        const uint64_t k_desc = smem_desc_sw128(k_sm + s * K_BYTES, 16, 1024);
        const uint32_t acc = tmem + acc_slot(i) * kMaxObs;
        if constexpr (D == 128) mma_ss_chain8_b32rows(acc, k_desc, q_desc, IDESC, 0);
        else mma_ss_chain4(acc, k_desc, q_desc, IDESC, 0);
        mma_commit(smem_u32(&sh->empty[s]));
        mma_commit(smem_u32(&sh->acc_full[i]));
        // the tile of the product before this one is free: refill its stage
        const int f = i - 1 + STAGES;
        if (i > 0 && f < n_seq) {
          ok = ck_wait(&sh->empty[f % STAGES], (f / STAGES - 1) & 1, sh, 51, wlim);
          if (ok) load_tile(f);
        }
      }
      issue_ok = ok;
    }
  };
  // After a wait that gave up: what is in flight gets a bounded chance to finish before the ring is reused and tensor memory freed.
  auto drain = [&]() {
    mma_commit(smem_u32(&sh->drain));
#pragma unroll 1
    for (uint32_t it = 0; it < kCkDrainSpins && !mbar_try_wait(smem_u32(&sh->drain), 0); ++it) {}
#pragma unroll 1
    for (int i = max(0, issued - STAGES); i < issued; ++i) {
      const uint32_t bar = smem_u32(&sh->full[i % STAGES]);
#pragma unroll 1
      for (uint32_t it = 0; it < kCkDrainSpins && !mbar_try_wait(bar, (i / STAGES) & 1); ++it) {}
    }
  };
  if (warp == kIssueWarp) {
    if (lane == 0) issue(0, n_run);
    __syncwarp();
  } else {
    // Thread r of a set owns key r of every chunk and keeps (reference maximum, sum-exp) of the set's 16
    // rows (all 32 in one thread would not leave registers for two CTAs per SM).  The reference starts
    // at the thread's first logit and is raised only when a logit exceeds it by 2^kLazyMax, so that an
    // entry usually costs one exponential.
    float rm[kHalfObs], rl[kHalfObs];
#pragma unroll
    for (int i = 0; i < kHalfObs; ++i) { rm[i] = -INFINITY; rl[i] = 0.f; }
    bool ok = true, first = true;
#pragma unroll 1
    for (int i = 0; i < n_run; ++i) {
      ok = __all_sync(0xffffffffu, ck_wait(&sh->acc_full[i], 0, sh, 54, wlim));
      if (!ok) break;
      tc_fence_after();
      uint32_t acc[kHalfObs];
      tmem_ld16(t_lane + acc_slot(i) * kMaxObs + set * kHalfObs, acc);
      tmem_wait_ld();
      if (i >= p.direct) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sh->acc_free[(i - p.direct) & 1]));
        if (i < n_held) {
          float* dst = over + ((size_t)(i - p.direct) * kMaxObs + set * kHalfObs) * kCkChunk + key_row;
#pragma unroll
          for (int r = 0; r < kHalfObs; ++r) dst[r * kCkChunk] = __uint_as_float(acc[r]);
        }
      }
      int j;
      if (slot_info(i * kCkChunk + key_row, j)) {
        if (first) {
          first = false;
#pragma unroll
          for (int r = 0; r < kHalfObs; ++r) { rm[r] = __uint_as_float(acc[r]) * zscale; rl[r] = 1.f; }
        } else {
          float d[kHalfObs], top = -INFINITY;
#pragma unroll
          for (int r = 0; r < kHalfObs; ++r) {
            d[r] = fmaf(__uint_as_float(acc[r]), zscale, -rm[r]);
            top = fmaxf(top, d[r]);
          }
          if (top > kLazyMax) {
#pragma unroll
            for (int r = 0; r < kHalfObs; ++r) {
              const float z = __uint_as_float(acc[r]) * zscale;
              const float mn = fmaxf(rm[r], z);
              rl[r] = rl[r] * ex2(rm[r] - mn) + ex2(z - mn);
              rm[r] = mn;
            }
          } else {
#pragma unroll
            for (int r = 0; r < kHalfObs; ++r) rl[r] += ex2(d[r]);
          }
        }
      }
    }
    if (ok) {
      // merge over the warp's 32 keys: in every step a lane hands half of its rows to its partner, so
      // that lanes r and r + 16 end up with row r of the set; then those two are merged
#pragma unroll
      for (int o = kHalfObs / 2; o > 0; o >>= 1) {
        const bool hi = lane & o;
#pragma unroll
        for (int r = 0; r < o; ++r) {
          const float2 keep = hi ? make_float2(rm[r + o], rl[r + o]) : make_float2(rm[r], rl[r]);
          const float2 give = hi ? make_float2(rm[r], rl[r]) : make_float2(rm[r + o], rl[r + o]);
          const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, o), __shfl_xor_sync(0xffffffffu, give.y, o));
          const float2 m = merge_stats(keep, got);
          rm[r] = m.x;
          rl[r] = m.y;
        }
      }
      const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, rm[0], 16), __shfl_xor_sync(0xffffffffu, rl[0], 16));
      if (lane < kHalfObs) sh->pub_stats[warp & 3][set * kHalfObs + lane] = merge_stats(make_float2(rm[0], rl[0]), got);
    }
  }
  __syncthreads();
  if (tid == 0) sh->pub_abort = *reinterpret_cast<volatile int*>(&sh->abort_flag);
  // the two histograms of the radix select
  if (tid < kWorkers) {
    uint4* z = reinterpret_cast<uint4*>(hist32 + 8 * tid);
    z[0] = z[1] = make_uint4(0, 0, 0, 0);
    z[kHistWords / 4] = z[kHistWords / 4 + 1] = make_uint4(0, 0, 0, 0);
  }

  // ------------------------------------------------------------------ 2. row statistics of the whole head
  cluster_sync(CL);
  if (tid < 4 * kMaxObs) {
    float2 got[kMaxCluster];
#pragma unroll
    for (int r = 0; r < kMaxCluster; ++r)                   // all loads in flight at once
      if (r < CL) got[r] = ld_peer_f2(peer_addr(&sh->pub_stats[warp][lane], r));
    float2 st = got[0];
#pragma unroll
    for (int r = 1; r < kMaxCluster; ++r)
      if (r < CL) st = merge_stats(st, got[r]);
    sh->part[warp][lane] = st;
  }
  bool any_abort = false;
  if (lane < CL) any_abort = ld_peer_i32(peer_addr(&sh->pub_abort, lane)) != 0;
  const bool aborted = __any_sync(0xffffffffu, any_abort);  // the same in every CTA of the cluster
  __syncthreads();
  if (warp == 0) {
    float2 st = sh->part[0][lane];
#pragma unroll
    for (int w = 1; w < 4; ++w) st = merge_stats(st, sh->part[w][lane]);
    // rows past n_obs_rows are padding: weight 0, finite reference
    reinterpret_cast<float2*>(sh->row_stat)[lane] = lane < a.n_obs_rows ? make_float2(st.x, 1.f / st.y) : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const bool select = !aborted && !p.score_only && n_rows > 0;

  // ------------------------------------------------------------------ 3. scores, pass 2
  if (kAgain && warp == kIssueWarp) {
    if (lane == 0 && issue_ok && !aborted) issue(n_run, n_seq);
    __syncwarp();
  } else if (!aborted && warp != kIssueWarp) {
    const bool structural = ctx == 0;
    bool ok = true;
#pragma unroll 1
    for (int i = set; i < n_p; i += 2) {                    // a set takes every other chunk here
      const bool again = kAgain && i >= n_held;
      const int seq = n_run + i - n_held;                   // the product that forms this chunk a second time
      if (again) {
        ok = __all_sync(0xffffffffu, ck_wait(&sh->acc_full[seq], 0, sh, 55, wlim)) && ok;
        tc_fence_after();
      }
      float s = 0.f;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t acc[kHalfObs];
        if (i < p.direct || again) {
          tmem_ld16(t_lane + (again ? acc_slot(seq) : i) * kMaxObs + h * kHalfObs, acc);
          tmem_wait_ld();
          if (again && h == 1) {
            // the accumulator counts a release by every worker warp; the four of this set stand for all of them
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_n(smem_u32(&sh->acc_free[(seq - p.direct) & 1]), 2);
          }
        } else {
          const float* src = over + ((size_t)(i - p.direct) * kMaxObs + h * kHalfObs) * kCkChunk + key_row;
#pragma unroll
          for (int r = 0; r < kHalfObs; ++r) acc[r] = __float_as_uint(src[r * kCkChunk]);
        }
#pragma unroll
        for (int r = 0; r < kHalfObs; r += 2) {
          const float4 st = sh->row_stat[(h * kHalfObs + r) / 2];
          s = fmaf(ex2(fmaf(__uint_as_float(acc[r]), zscale, -st.x)), st.y, s);
          s = fmaf(ex2(fmaf(__uint_as_float(acc[r + 1]), zscale, -st.z)), st.w, s);
        }
      }
      int j = 0;
      const bool live = slot_info(i * kCkChunk + key_row, j);
      uint32_t key = 0;
      if (live) {
        if (p.scores && dbg_ok(j < a.cand_stride, a.status, 8)) p.scores[(size_t)bh * a.cand_stride + j] = s;
        if (structural && (j < a.t_init || (a.protect_new && j >= stored))) {
          key = 0xffffffffu;
        } else {
          key = ck_orderable(s);
          if (key == 0xffffffffu) key = 0xfffffffeu;          // the top key is for protected entries only
        }
      }
      keys[i * kCkChunk + key_row] = key;
      if (!p.score_only) hist_add(hist32, live, key >> 20);   // first digit of the radix select
    }
  }
  tc_fence_before();
  __syncthreads();
  // (whichever thread's wait it was; tiles of the second products may be on their way when another CTA gives up)
  if (warp == kIssueWarp && lane == 0 && (aborted || sh->abort_flag)) drain();

  if (select) {
    // ---------------------------------------------------------------- 4. radix select over the cluster
    // Digits of 12, 12 and 8 bits.  The local histogram of the first digit was filled while the keys
    // were formed; the select stops as soon as every entry left in the located bin survives, which
    // with 24 bits fixed is the usual case.  Before the cluster meets, every CTA adds its bins in groups
    // of 16 and forms the counts above each group; afterwards worker t adds the CL words of group t, the
    // one warp whose groups hold the wanted rank reads that group's bins, and it learns on the
    // way how many keys each CTA holds above the located bin and in it.
    const int n_slots = n_p * kCkChunk;
    uint32_t prefix = 0, mask = 0;
    int need = n_rows;
    if (tid < CL) sh->cnt_gt[tid] = 0;
    if (tid == 0) { sh->bin_n = 0; sh->bin_gt = 0; }
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 20 : (pass == 1 ? 8 : 0);
      const uint32_t dmask = pass == 2 ? 255u : 4095u;
      uint32_t* hist = hist32 + (pass & 1) * kHistWords;
      if (pass > 0) {
#pragma unroll 1
        for (int slot = tid; slot < n_slots; slot += kCkThreads) {
          int j;
          const uint32_t k = keys[slot];
          // few entries are left and they differ: plain additions
          if ((k & mask) == prefix && slot_info(slot, j)) {
            const uint32_t digit = (k >> shift) & dmask;
            atomicAdd(&hist[digit >> 1], 1u << (16 * (digit & 1)));
          }
        }
        __syncthreads();
      }
      int mine = 0;
      if (tid < kWorkers) {
        const uint4 h0 = *reinterpret_cast<const uint4*>(hist + 8 * tid), h1 = *reinterpret_cast<const uint4*>(hist + 8 * tid + 4);
        const uint32_t w = (h0.x + h0.y + h0.z + h0.w) + (h1.x + h1.y + h1.z + h1.w);   // two 16-bit sums: a CTA holds fewer than 65 536 keys
        mine = (int)((w & 0xffffu) + (w >> 16));
      }
      int total;
      const int below = ck_block_scan(mine, sh->warp_sums[pass & 1], total);
      if (tid < kWorkers) sh->coarse[pass & 1][tid] = (uint32_t)mine << 16 | (uint32_t)(total - below - mine);
      cluster_sync(CL);                                       // (orders the CTA's own threads as well)
      if (tid < kWorkers) {
        uint32_t g[kMaxCluster];
#pragma unroll
        for (int r = 0; r < kMaxCluster; ++r) {               // all loads in flight at once
          g[r] = 0;
          if (r < CL) g[r] = (uint32_t)ld_peer_i32(peer_addr(&sh->coarse[pass & 1][tid], r));
        }
        int above = 0, group = 0;
#pragma unroll
        for (int r = 0; r < kMaxCluster; ++r) { above += (int)(g[r] & 0xffffu); group += (int)(g[r] >> 16); }
        // exactly one group holds the wanted rank; its warp reads the group's bins, lane (r, u) word u of CTA r
        const uint32_t winner = __ballot_sync(0xffffffffu, above < need && need <= above + group);
        if (winner) {
          const int src = __ffs(winner) - 1;
          const int grp = (tid & ~31) + src;
          above = __shfl_sync(0xffffffffu, above, src);
          uint32_t lo[2] = {0, 0};                            // word lane & 7 of the CTAs lane >> 3 and 4 + (lane >> 3)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if ((lane >> 3) + 4 * h < CL)
              lo[h] = (uint32_t)ld_peer_i32(peer_addr(hist + 8 * grp + (lane & 7), (lane >> 3) + 4 * h));
          // bins 2 u and 2 u + 1 over the CTAs, each in a word of its own
          int c0 = (int)(lo[0] & 0xffffu) + (int)(lo[1] & 0xffffu), c1 = (int)(lo[0] >> 16) + (int)(lo[1] >> 16);
#pragma unroll
          for (int o = 8; o <= 16; o <<= 1) {
            c0 += __shfl_xor_sync(0xffffffffu, c0, o);
            c1 += __shfl_xor_sync(0xffffffffu, c1, o);
          }
          // entries in the words above this lane's (u = lane & 7), by a suffix sum over 8 lanes
          int suf = c0 + c1;
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) {
            const int n = __shfl_down_sync(0xffffffffu, suf, o, 8);
            if ((lane & 7) + o < 8) suf += n;
          }
          const int over1 = above + suf - c0 - c1, over0 = over1 + c1;
          const bool hit1 = over1 < need && need <= over1 + c1, hit0 = over0 < need && need <= over0 + c0;
          const int u = (__ffs(__ballot_sync(0xffffffffu, hit0 || hit1)) - 1) & 7;
          const bool odd = __shfl_sync(0xffffffffu, (int)hit1, u);
          if (lane == u) {
            sh->digit = 16 * grp + 2 * u + (odd ? 1 : 0);
            sh->need_in_bin = need - (odd ? over1 : over0);
            sh->bin_count = odd ? c1 : c0;
          }
          // per CTA: entries of this group above the located bin, and in it
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int w = lane & 7, b0 = (int)(lo[h] & 0xffffu), b1 = (int)(lo[h] >> 16);
            int gt = w > u ? b0 + b1 : (w == u && !odd) ? b1 : 0;
            int eq = w == u ? (odd ? b1 : b0) : 0;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
              gt += __shfl_xor_sync(0xffffffffu, gt, o);
              eq += __shfl_xor_sync(0xffffffffu, eq, o);
            }
            const int r = (lane >> 3) + 4 * h;
            if (w == 0 && r < CL) {
              sh->cnt_gt[r] += gt;
              sh->cnt_eq[r] = eq;
            }
          }
          __syncwarp();
          if (lane == src) {
#pragma unroll
            for (int r = 0; r < kMaxCluster; ++r)
              if (r < CL) sh->cnt_gt[r] += (int)(g[r] & 0xffffu);
          }
        }
      }
      // the first histogram is free: every CTA read it before it arrived at the barrier above
      if (pass == 1 && tid < kWorkers) {
        uint4* z = reinterpret_cast<uint4*>(hist32 + 8 * tid);
        z[0] = z[1] = make_uint4(0, 0, 0, 0);
      }
      __syncthreads();
      prefix |= (uint32_t)sh->digit << shift;
      need = sh->need_in_bin;
      mask |= dmask << shift;
      const int m = sh->bin_count;
      if (need == m) break;                                   // the same in every CTA of the cluster
      if (m <= kBinMax) {
        // Few entries left: they are ranked by comparing each with all of them.  An entry is its key and,
        // below it, its complemented index, so that among equals the lowest index ranks first.
        unsigned long long* own = reinterpret_cast<unsigned long long*>(hist32 + ((pass & 1) ^ 1) * kHistWords);
        unsigned long long* all = own + kBinMax;
#pragma unroll 1
        for (int slot = tid; slot < n_slots; slot += kCkThreads) {
          int j;
          const uint32_t k = keys[slot];
          if ((k & mask) == prefix && slot_info(slot, j)) own[atomicAdd(&sh->bin_n, 1)] = (unsigned long long)k << 32 | (uint32_t)~j;
        }
        cluster_sync(CL);
        unsigned long long mine_e = 0;
        int r = 0;                                            // the CTA that holds this thread's entry
        if (tid < m) {
          int e = tid;
          while (e >= sh->cnt_eq[r]) e -= sh->cnt_eq[r++];
          mine_e = CL == 1 ? own[e] : ld_peer_u64(peer_addr(&own[e], r));
          all[tid] = mine_e;
        } else if (tid == m) {
          all[tid] = 0;                                       // the last pair may read one past the end
        }
        __syncthreads();
        if (tid < CL) sh->cnt_eq[tid] = 0;
        int before = 0;
        if (tid < m) {
#pragma unroll 4
          for (int i = 0; i < m; i += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(all + i);
            before += (v.x > mine_e) + (v.y > mine_e);
          }
          if (before == need - 1) sh->digit = (int)(mine_e >> 32);
        }
        __syncthreads();
        prefix = (uint32_t)sh->digit;
        mask = 0xffffffffu;
        if (tid < m) {
          const uint32_t k = (uint32_t)(mine_e >> 32);
          if (k > prefix) { atomicAdd(&sh->cnt_gt[r], 1); atomicAdd(&sh->bin_gt, 1); }
          if (k == prefix) atomicAdd(&sh->cnt_eq[r], 1);
        }
        __syncthreads();
        need -= sh->bin_gt;
        break;
      }
      __syncthreads();                                        // before the next pass writes what was just read
    }
    // ---------------------------------------------------------------- 5. ascending index list
    // prefix = the fixed digits of the n_rows-th largest key; of the entries that agree with it in
    // those digits `need` survive (lowest indices; all of them when the select stopped early).  A warp
    // takes a run of consecutive slots, 32 at a time: the survivors' places are ballot counts.
    const uint32_t thr = prefix;
    int gt_before = 0, eq_before = 0;
#pragma unroll
    for (int r = 0; r < kMaxCluster; ++r)
      if (r < rank) { gt_before += sh->cnt_gt[r]; eq_before += sh->cnt_eq[r]; }
    const int n_groups = n_slots / 32, per = (n_groups + kCkWarps - 1) / kCkWarps;
    const int g_begin = min(n_groups, warp * per), g_end = min(n_groups, g_begin + per);
    int gt = 0, eq = 0;
#pragma unroll 1
    for (int g = g_begin; g < g_end; ++g) {
      const int slot = g * 32 + lane;
      int j;
      const bool live = slot_info(slot, j);
      const uint32_t k = keys[slot] & mask;
      gt += __popc(__ballot_sync(0xffffffffu, live && k > thr));
      eq += __popc(__ballot_sync(0xffffffffu, live && k == thr));
    }
    int total;
    const int packed = ck_warp_prefix(gt | (eq << 16), sh->warp_sums[0], total);
    gt_before += packed & 0xffff;
    eq_before += packed >> 16;
    // Entry o of the head's ascending list is candidate j.  Entry o becomes row o of the head, and
    // rows are compacted in rounds of CL * S consecutive entries, CTA `rk` of the cluster staging S
    // of them: the entry goes straight into that CTA's shared memory.
    // rounds: as few as the staging buffers (a third of the staging rows each) allow, of equal size
    const int s_cap = S_ROWS / kMoveBuffers;
    const int n_rounds = (n_rows + CL * s_cap - 1) / (CL * s_cap);
    const int S = (n_rows + CL * n_rounds - 1) / (CL * n_rounds), RS = CL * S;
    // o / S and o / RS by a multiplication: exact for o < 65 536 and divisors up to 65 536
    const uint32_t inv_s = 0xffffffffu / (uint32_t)S + 1u, inv_rs = 0xffffffffu / (uint32_t)RS + 1u;
    const uint32_t lower = (1u << lane) - 1u;
    const bool lists = kLists && ctx;
#pragma unroll 1
    for (int g = g_begin; g < g_end; ++g) {
      const int slot = g * 32 + lane;
      int j;
      const bool live = slot_info(slot, j);
      const uint32_t k = keys[slot] & mask;
      const bool is_gt = live && k > thr, is_eq = live && k == thr;
      const uint32_t m_gt = __ballot_sync(0xffffffffu, is_gt), m_eq = __ballot_sync(0xffffffffu, is_eq);
      const int eq_rank = eq_before + __popc(m_eq & lower);
      const int o = gt_before + __popc(m_gt & lower) + min(eq_rank, need);
      if (lists) {
        // (as many survivors as o are ahead of an entry, whether it is one itself or not)
        if (is_gt || (is_eq && eq_rank < need)) {
          if (dbg_ok(o >= 0 && o < a.kept_stride, a.status, 9)) p.kept_list[(size_t)bh * a.kept_stride + o] = j;
        } else if (live && dbg_ok(j - o >= 0 && j - o < p.gone_stride, a.status, 9)) {
          p.gone_list[(size_t)bh * p.gone_stride + (j - o)] = j;
        }
      } else if ((is_gt || (is_eq && eq_rank < need)) && dbg_ok(o >= 0 && o < n_rows, a.status, 9)) {
        const int t = RS == 1 ? o : (int)__umulhi((uint32_t)o, inv_rs), w = o - t * RS;
        const int rk = S == 1 ? w : (int)__umulhi((uint32_t)w, inv_s), lr = w - rk * S;
        st_peer_i32(peer_addr(&src_all[t * S + lr], rk), j);
      }
      gt_before += __popc(m_gt);
      eq_before += __popc(m_eq);
    }
    cluster_sync(CL);                                         // every CTA holds its part of the list

    // ---------------------------------------------------------------- 6. and 7. compaction in rounds
    // A stored survivor moves forward (its source is a row of the head at or behind its
    // destination), a surviving new row comes out of the caller's K/V.  In a round every CTA stages
    // its S entries in shared memory, the cluster meets, and the rows go out with bulk stores (the
    // destinations of a CTA are one contiguous run).  The destinations of a round lie at or before
    // its own cache sources and before the cache sources of every later round, so nothing is
    // overwritten before it has been read: in place, no second buffer.
    const size_t off = a.row_off[bh];
    uint4* kp = reinterpret_cast<uint4*>(a.k_plane) + off * PIECES;
    uint4* vp = reinterpret_cast<uint4*>(a.v_plane) + off * PIECES;
    int32_t* pos = a.pos_plane + off;
    const uint4* kn = p.k_new + (size_t)bh * n_new * PIECES;
    const uint4* vn = p.v_new + (size_t)bh * n_new * PIECES;
    constexpr uint32_t ROWB = PIECES * 16;
    // Staging buffer b holds S key rows, then S value rows.  The loads of round t + 2 are issued
    // while round t stores: a later round's sources lie behind every earlier round's destinations.
    const uint32_t buf_bytes = 2u * (uint32_t)s_cap * ROWB;
    auto slice_first = [&](int t) { return t * RS + rank * S; };
    auto slice_rows = [&](int t) { return max(0, min(S, n_rows - slice_first(t))); };
    // ascending entries with source >= destination: if the last stored row of the slice stays
    // where it is, so does every row of the slice
    auto slice_moves = [&](int t) {
      const int rows = slice_rows(t), last = src_all[t * S + max(rows, 1) - 1];
      return rows > 0 && !(last == slice_first(t) + rows - 1 && last < stored);
    };
    auto issue_loads = [&](int t) {
      if (t < n_rounds && slice_moves(t)) {
        const int first = slice_first(t), rows = slice_rows(t);
        const int32_t* srcs = src_all + t * S;
        const uint32_t kb = base + (uint32_t)(t % kMoveBuffers) * buf_bytes, vb = kb + (uint32_t)S * ROWB;
        int32_t* ps = pos_stage + (t % kMoveBuffers) * s_cap;
#pragma unroll 2
        for (int v = tid; v < rows * PIECES; v += kCkThreads) {
          const int lr = v / PIECES, piece = v % PIECES;
          int src = srcs[lr];
          // a checked build turns an entry outside [destination, candidates) into "stays where it is"
          if (!dbg_ok(src >= first + lr && src < stored + n_new && first + lr < a.cap[ctx], a.status, 10))
            src = first + lr < stored ? first + lr : stored;
          const uint4* ks = src < stored ? kp + (size_t)src * PIECES : kn + (size_t)(src - stored) * PIECES;
          const uint4* vs = src < stored ? vp + (size_t)src * PIECES : vn + (size_t)(src - stored) * PIECES;
          cp_async16(kb + (uint32_t)lr * ROWB + piece * 16, ks + piece);
          cp_async16(vb + (uint32_t)lr * ROWB + piece * 16, vs + piece);
        }
#pragma unroll 1
        for (int lr = tid; lr < rows; lr += kCkThreads) {
          const int src = srcs[lr];
          if (src < stored) cp_async4(smem_u32(&ps[lr]), pos + max(src, 0));
          else ps[lr] = a.pos_base + (src - stored);
        }
      }
      cp_async_commit();                                      // one group per round, empty or not
    };
    const int n_moves = lists ? 0 : n_rounds;
    // (the two rounds ahead of the first only issue their loads: one place in the code for them)
#pragma unroll 1
    for (int t = n_moves > 0 ? -2 : 0; t < n_moves; ++t) {
      if (t >= 0) {
        cp_async_wait_group<1>();                               // the loads of round t (all but the latest group) have landed
        fence_proxy_async();                                    // the bulk stores below read what these threads wrote
        cluster_sync_relaxed(CL);                               // every source of this round has been read
        const bool moving = slice_moves(t);
        if (moving) {
          const int first = slice_first(t), rows = slice_rows(t);
          const uint32_t kb = base + (uint32_t)(t % kMoveBuffers) * buf_bytes, vb = kb + (uint32_t)S * ROWB;
          if (tid == 0) {
            constexpr uint32_t kPiece = 32768;                  // bytes per bulk store
            const uint32_t bytes = (uint32_t)rows * ROWB;
#pragma unroll 1
            for (uint32_t o = 0; o < bytes; o += kPiece) {
              const uint32_t n = min(kPiece, bytes - o);
              bulk_store(reinterpret_cast<unsigned char*>(kp + (size_t)first * PIECES) + o, kb + o, n);
              bulk_store(reinterpret_cast<unsigned char*>(vp + (size_t)first * PIECES) + o, vb + o, n);
            }
          }
          const int32_t* ps = pos_stage + (t % kMoveBuffers) * s_cap;
#pragma unroll 1
          for (int lr = tid; lr < rows; lr += kCkThreads) pos[first + lr] = ps[lr];
        }
        if (tid == 0) {
          bulk_commit();                                        // one group per round, empty or not
          bulk_wait_read<1>();                                  // round t - 1 has left its buffer, which round t + 2 fills
        }
        __syncthreads();
      }
      issue_loads(t + 2);
    }
    if (tid == 0) bulk_wait_read<0>();                        // shared memory is read out before the CTA leaves
  } else if (kLists && ctx) {
    // After a wait that gave up: the launches behind this one read rows through the lists all the same, so these hold
    // candidates of the head, each of them once.
#pragma unroll 1
    for (int j = rank * kCkThreads + tid; j < stored + n_new; j += CL * kCkThreads) {
      if (j < n_rows) p.kept_list[(size_t)bh * a.kept_stride + j] = j;
      else p.gone_list[(size_t)bh * p.gone_stride + (j - n_rows)] = j;
    }
  }
  if (tid == 0 && sh->abort_flag) atomicExch(a.status, sh->abort_flag);
  // no CTA leaves while another may still read its shared memory (past the list nobody does)
  if (!select) cluster_sync(CL);
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kMaxObs * p.slots);
  }
}

// Shared memory of one CTA: the front region (ring, observation rows and overflow logits; the
// compaction later stages rows over all of it), keys, the two per-row staging arrays, barriers and
// exchange area.
template <int D>
size_t ck_smem_bytes(const CkParams& p) {
  const size_t rows = (size_t)p.stage_rows;
  return 1024 + (size_t)p.region_bytes + (size_t)p.p_max * kCkChunk * sizeof(uint32_t) +
         (2 * rows + (size_t)p.p_max * kCkChunk) * sizeof(int32_t) + sizeof(CkShared) + 64;
}

// Ring depth and staging rows for this launch: as many key tiles in flight as the CTA has chunks
// (more would never be used) and as the budget holds; the front region then grows to what is left
// of the budget, so that a round of the compaction stages as many rows as possible.  False if the
// budget does not hold the launch.
template <int D>
bool ck_size(CkParams& p, size_t budget) {
  const size_t k_bytes = (size_t)(D / 64) * kCkChunk * 128;
  const size_t row_bytes = 2 * (size_t)D * 2;                // a key row and a value row
  const size_t over_bytes = (size_t)kMaxObs * kCkChunk * sizeof(float);
  const size_t q_hist = (size_t)(D / 64) * kMaxObs * 128 + 2 * kHistWords * sizeof(uint32_t);
  p.stage_rows = kMaxStageRows;
  p.region_bytes = 0;
  const size_t other = ck_smem_bytes<D>(p);                   // everything but the front region
  const size_t room = budget > other ? budget - other : 0;
  // logits past the accumulators stay in shared memory as far as they fit beside three key tiles
  const size_t ring_min = std::min(3, std::max(p.cpc_max, 2)) * k_bytes;
  p.n_over = std::max(0, std::min(p.p_max - p.direct, room > q_hist + ring_min ? (int)((room - q_hist - ring_min) / over_bytes) : 0));
  const size_t q_over = q_hist + (size_t)p.n_over * over_bytes;
  const int fit = room > q_over ? (int)((room - q_over) / k_bytes) : 0;
  p.stages = std::max(2, std::min({fit, kMaxStages, std::max(p.cpc_max, 2)}));
  const size_t need = p.stages * k_bytes + q_over;
  const size_t region = std::max(need, std::min(room, (size_t)kMaxStageRows * row_bytes)) / 1024 * 1024;
  p.region_bytes = (int)std::max(region, (need + 1023) / 1024 * 1024);
  p.stage_rows = (int)std::min<size_t>(kMaxStageRows, p.region_bytes / row_bytes);
  return ck_smem_bytes<D>(p) <= budget;
}

template <int D>
cudaLaunchConfig_t ck_config(const StepArgs& a, const CkParams& p, cudaLaunchAttribute* attr, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.cluster, a.batch * a.n_heads);
  cfg.blockDim = dim3(kCkThreads);
  cfg.dynamicSmemBytes = ck_smem_bytes<D>(p);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = p.cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

// Clusters of this shape the device runs at the same time (asked once per shape and device).  The
// occupancy queries count one CTA per SM for any kernel that allocates tensor memory, so the two that
// a shape for two CTAs per SM is made for (shared memory, registers and columns) are counted here.
template <int D>
int ck_active_clusters(const StepArgs& a, const CkParams& p, int per_sm) {
  if (p.cluster == 1) return per_sm * sm_count();
  struct Known { int dev, cluster; size_t smem; int n; };
  static std::mutex mu;
  static std::vector<Known> known;
  int dev = 0;
  cudaGetDevice(&dev);
  const size_t smem = ck_smem_bytes<D>(p);
  std::lock_guard<std::mutex> lock(mu);
  for (const Known& k : known)
    if (k.dev == dev && k.cluster == p.cluster && k.smem == smem) return per_sm * k.n;
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = ck_config<D>(a, p, attr, nullptr);
  cfg.numAttrs = 2;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, compress_cluster_kernel<D, false>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  known.push_back({dev, p.cluster, smem, n});
  return per_sm * n;
}

// Chunks of the candidate lists of a launch, per head type: those whose logits are read twice, and those
// that only enter the softmax denominators (the new scale of a head that keeps it whole).
struct CkLists {
  int ranked[2], once[2];
  int rows[2];                                               // survivors that are moved
};

// Ranked chunks of the longest CTA whose logits are formed a second time.
int ck_again(const CkParams& p) { return std::max(0, p.p_max - p.direct - p.n_over); }

// Shape of a launch with `cl` CTAs per head and `per_sm` CTAs per SM.  Two CTAs per SM share its tensor
// memory (256 columns each) and shared memory; a CTA that takes all 512 columns asks for more than half
// of the shared memory, so that no second one can be placed beside it and wait for columns.
template <int D>
bool ck_shape(CkParams& p, const CkLists& n, int cl, int per_sm) {
  p.cluster = cl;
  p.p_max = 1;
  p.cpc_max = 1;
  for (int t = 0; t < 2; ++t) {
    const int ranked = (n.ranked[t] + cl - 1) / cl, once = (n.once[t] + cl - 1) / cl;
    p.p_max = std::max(p.p_max, ranked);
    p.cpc_max = std::max(p.cpc_max, ranked + once);
  }
  const int most = per_sm == 2 ? kMaxSlots / 2 : kMaxSlots;
  p.slots = 1;
  while (p.slots < std::min(p.cpc_max, most)) p.slots *= 2;
  p.direct = p.cpc_max <= p.slots ? p.slots : p.slots - 2;
  if (!ck_size<D>(p, per_sm == 2 ? kSmemShared : kSmemBudget)) return false;
  if (p.cpc_max + ck_again(p) > kMaxSeq) return false;
  return p.slots <= kMaxSlots / 2 || ck_smem_bytes<D>(p) > kSmemShared + 4096;
}

// Device time of one cluster in microseconds, fitted to clock stamps inside the kernel over launches of
// 1 to 50 chunks per head: 7 us of dependent round trips, 2 to 6 more where they cross CTAs (a cluster of
// eight also waits for eight SMs of one GPC); the key tiles of a CTA at no more than 75 GB/s and its share
// of the memory's rate; a read-out per ranked chunk; the row moves.  CTAs that share an SM slow each
// other down.
template <int D>
float ck_cluster_us(const CkParams& p, const CkLists& n, int cl, bool crowded, float ctas) {
  const float tile_us = std::max(D / 128 * 0.43f + (D == 64 ? 0.25f : 0.f), ctas * kCkChunk * D * 2 / 6.0e6f);
  float most = 0.f;
  for (int t = 0; t < 2; ++t) {
    const int ranked = (n.ranked[t] + cl - 1) / cl, once = (n.once[t] + cl - 1) / cl;
    const int again = std::max(0, ranked - p.direct - p.n_over);
    const float move = (float)n.rows[t] / cl * D * 8 / 65000.f;      // a key and a value row in, the same out, at 65 GB/s
    most = std::max(most, (ranked + once + again) * tile_us + ranked * 0.3f + again * 0.2f + move);
  }
  const float fixed = cl == 1 ? 7.f : 8.4f + 0.35f * cl + (cl > 6 ? 2.f : 0.f);
  return fixed + (crowded ? 1.5f : 1.f) * most;
}

template <int D>
int launch_t(const StepArgs& a, const CUtensorMap& tm_cache, const CUtensorMap& tm_new, const void* q, CkParams p,
             const CkLists& lists, int n_clusters, float beside_us, float behind_us, uint16_t* shape, cudaStream_t st) {
  // the opt-in is made once per (kernel, device), so it asks for the most any launch can need
  if (!allow_dynamic_smem(compress_cluster_kernel<D, false>, kSmemBudget) ||
      !allow_dynamic_smem(compress_cluster_kernel<D, true>, kSmemBudget) ||
      !allow_dynamic_smem(compress_cluster_kernel<D, true, true>, kSmemBudget))
    return -1;
  // CTAs per head and per SM: the step ends when this launch and the attention that needs it are done,
  // and not before the SMs have done all the work there is (larger clusters finish sooner and keep
  // more SMs from the attention that could run beside them).  A late launch also leaves the attention behind
  // it a worse last round, hence the last term.  Measured per step (CTAs per head: us): 32 heads x 128,
  // 2 304 queries 2: 144, 3: 131, 4: 133, 6: 144; 64 heads 1: 268, 2: 239, 3: 247, 4: 250; 240 heads x 64,
  // 1 024 queries, one CTA per head: 127 with one per SM, 113 with two.
  const float sms = (float)sm_count();
  float best = 0.f;
  int best_cl = 0, best_per_sm = 0;
  if (shape && *shape) {                                     // found when this step came by before
    best_cl = *shape & 0xff;
    best_per_sm = *shape >> 8;
  }
  for (int per_sm = 1; per_sm <= 2 && !(shape && *shape); ++per_sm)
    for (int cl = 1; cl <= kMaxCluster; ++cl) {
      if (!ck_shape<D>(p, lists, cl, per_sm)) continue;
      // Clusters of an odd size that are placed while the launch ahead drains do not pack as tightly as on an empty chip:
      // of 44 clusters of 3, where 45 fit, one to three often started only when the first ones had ended, 12 us
      // late.  So a fifteenth of their places is not counted on: 45 heads x 128, 529 queries 42.7 -> 33.8 us a step, 43
      // heads 33.6 -> 31.1, 26 heads 32.3 -> 27.3; 42 and 24 heads are as fast with 3 and 5 CTAs as with any other number.
      // Even sizes need no reserve (33 heads, clusters of 4: 30.0, with one 31.0; 74 heads, of 2: 40.6, with one 47.4).
      const int fit = ck_active_clusters<D>(a, p, per_sm);
      const int active = per_sm == 1 && cl > 1 && cl % 2 == 1 ? fit - (fit + 14) / 15 : fit;
      if (active < 1) continue;
      if (D == 128 && per_sm == 2 && n_clusters * cl <= sms) continue;    // the CTAs spread over as many SMs, and attention takes a whole one
      const int waves = (n_clusters + active - 1) / active;
      const int at_once = std::min(n_clusters, active);
      const float us = waves * ck_cluster_us<D>(p, lists, cl, per_sm == 2 && at_once * cl > sms, (float)at_once * cl);
      const float sm_us = n_clusters * cl * us / (waves * per_sm);
      const float cost = std::max(us + behind_us / sms, (sm_us + beside_us + behind_us) / sms) + 0.6f * us;
      if (!best_cl || cost < best) {
        best = cost;
        best_cl = cl;
        best_per_sm = per_sm;
      }
    }
  if (!best_cl) return 0;
  if (shape) *shape = (uint16_t)(best_per_sm << 8 | best_cl);
  ck_shape<D>(p, lists, best_cl, best_per_sm);
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = ck_config<D>(a, p, attr, st);
  cudaLaunchKernelEx(&cfg, p.kept_list ? compress_cluster_kernel<D, true, true> : ck_again(p) > 0 ? compress_cluster_kernel<D, true> : compress_cluster_kernel<D, false>, tm_cache, tm_new, a, static_cast<const __nv_bfloat16*>(q), p);
  return launched(n_clusters * p.cluster);
}

}  // namespace

// Scores only (scores != nullptr) or the whole compression of the step.  Returns the working CTAs of
// its one launch, -1 on a launch error, or 0 when this step is outside what the kernel holds
// (candidate lists far beyond 8 x 40 chunks per head, the every-query scoring rounds): the caller then
// takes the separate scoring, selection and compaction launches.
int launch_compress_cluster(const StepArgs& a, const void* q, const void* k_new, const void* v_new, float* scores,
                            cudaStream_t st, float beside_us, float behind_us, uint16_t* shape, int32_t* kept_list, int32_t* gone_list,
                            int gone_stride) {
  if (!a.k_map || a.obs_full || a.score_accumulate) return 0;
  if (!a.trig[0] && !a.trig[1]) return 0;
  CkParams p{};
  p.score_only = scores != nullptr;
  p.scores = scores;
  p.kept_list = kept_list;
  p.gone_list = gone_list;
  p.gone_stride = gone_stride;
  p.k_new = static_cast<const uint4*>(k_new);
  p.v_new = static_cast<const uint4*>(v_new);
  CkLists lists = {};
  const int n_new_chunks = (a.n_new + kCkChunk - 1) / kCkChunk;
  for (int t = 0; t < 2; ++t)
    if (a.trig[t] && a.heads_of[t] > 0) {
      const bool drop_new = t == 0 && a.protect_new && !scores;
      lists.ranked[t] = (a.stored[t] + kCkChunk - 1) / kCkChunk + (drop_new ? 0 : n_new_chunks);
      lists.once[t] = drop_new ? n_new_chunks : 0;
      lists.rows[t] = scores || (t == 1 && kept_list) ? 0 : a.kept[t] - (drop_new ? a.n_new : 0);
    }
  // clusters that do work: the heads of the triggered types
  const int n_clusters = std::max(1, a.heads_of[0] * a.trig[0] + a.heads_of[1] * a.trig[1]);
  CUtensorMap tm_new;
  if (!make_rows_map(&tm_new, k_new, (uint64_t)a.batch * a.n_heads * a.n_new, a.head_dim)) {
    set_error("compression: cuTensorMapEncodeTiled failed for the new scale's keys");
    return -1;
  }
  const CUtensorMap& tm_cache = *static_cast<const CUtensorMap*>(a.k_map);
  return a.head_dim == 128 ? launch_t<128>(a, tm_cache, tm_new, q, p, lists, n_clusters, beside_us, behind_us, shape, st)
                           : launch_t<64>(a, tm_cache, tm_new, q, p, lists, n_clusters, beside_us, behind_us, shape, st);
}

}  // namespace hack
