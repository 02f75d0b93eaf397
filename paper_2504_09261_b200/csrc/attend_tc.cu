// Attention over the compacted per-head cache on the 5th-generation tensor cores (bf16 inputs,
// fp32 accumulation): O = Softmax(sm_scale * Q K^T) V with ragged per-head lengths (Eq. 4 on the
// compressed cache).
//
// One CTA serves one (batch, head) and up to two 128-row query tiles, which take turns on the
// tensor pipe so that the softmax of one tile overlaps the MMAs of the other (T = 2); or, at head_dim
// 64, short caches and an odd number of tiles, one tile on half an SM (T = 1: no warps 8-11, half the tensor memory).  A unit of work
// is a head and its one or two tiles (heads whose keys are one block: several rounds of them); where there are
// more units than CTAs run at once, a CTA that nears the end of its unit takes over one that has not
// been launched yet (cluster launch control): its loads and first products run under the last softmax and the
// epilogue of the unit before, and tensor memory, barriers and registers are set up once.
//   warp  0     : issuer of the Q K^T products; also owns the TMEM allocation
//   warp  1     : TMA producer (K and V tiles of 128 cache rows through rings)
//   warp  2     : issuer of the P V products (a single issuing thread for both products was the
//                 bottleneck of the CTA: 0.212 -> 0.174 ms on the largest launch)
//   warp  3     : appends the new scale's rows to the cache with bulk copies (heads that keep it whole)
//   warps 4-7   : softmax of tile 0 (thread r owns query row r: one TMEM lane, no shuffles)
//   warps 8-11  : softmax of tile 1
//   The first warpgroup hands most of its registers to the softmax warpgroups (setmaxnreg) so that
//   a whole 128-column score row lives in registers.
//
// What shapes the kernel (all measured on the device):
//  * The thread that issues the MMAs needs instruction-issue slots of its scheduler; many busy
//    softmax warps starve it (with four always-ready warps per scheduler one tcgen05.mma took
//    over 200 cycles to issue against about 70 to execute).  Hence one thread per query row (two
//    softmax warps per scheduler, normally only one of them active) rather than more, lighter
//    threads, and as few softmax instructions as possible: scale / sum / max work runs on packed
//    or 3-input instructions.
//  * The instruction cache: with every wait and every loop of the issuing warps unrolled the units made 91 KB of
//    code and the warps waited for instructions 1.8 cycles per issue instead of 0.5 (6 % slower).  Waits are small,
//    the issuers' loops rolled, rare code is out of the way of the loop over the blocks.
//  * Work for padding: the last block of a segment is formed and weighted in groups of 32 keys.
// Measured (a step with its compression, before -> with units, groups of 32 and rolled loops): 240 heads x 64,
// 1 024 queries, 1 045 keys 115 -> 110 us (94 on whole SMs); 256 heads x 64, 256 queries, 612 keys 38.9 -> 37.4; 32 heads x 128,
// 4 096 queries, 4 208 and 2 104 keys 191 -> 187.
// TMEM (512 columns): S [0,128)  P0 [128,192)  P1 [192,256)  O0 [256,256+D)  O1 [256+D,256+2D).
// There is ONE logit buffer, which the two tiles use in turn, and a probability buffer per tile.  A
// softmax thread reads its whole logit row into registers first and hands the buffer back at once
// (s_free), so the next Q K^T product (the other tile's, or with one tile per CTA this tile's next
// block) runs while it computes; the probabilities go to the tile's own buffer, from where the
// second MMA takes them, so that no product waits for another to release columns it writes.  With
// one buffer per tile holding first the logits and then the probabilities (the earlier form), each
// tile was a serial chain softmax -> P V -> Q K^T -> softmax of about 3 400 cycles per 128 keys,
// and the two tiles only interleaved; now the tensor pipe and the exponentials each run at their own
// rate.  K tiles are K-major operands, V tiles MN-major operands, both 128-byte swizzled as TMA
// writes them.  Softmax keeps a running maximum that is only raised (and O rescaled in TMEM) when
// a row's maximum grows by more than 2^32, so rescaling is rare after the first tile.
// (Tried and dropped: logits in two buffers of 64 keys per tile.  The 128 x 64 x 16 MMA re-reads the
// whole Q operand from shared memory for half the keys and takes nearly as long as the
// 128 x 128 x 16 one: the last-scale launch of the 10 521-token workload went from 0.233 to 0.301 ms.)
// The keys and values of a head come in two segments: len_b rows of the new scale taken straight from
// the caller's K/V tensors (second pair of tensor maps), then len_a rows of the head's cache.
// Heads that keep the whole new scale (steps without eviction; structural heads, whose latest scale
// is protected, Eq. 11) are served that way before the new rows are in the cache: the append
// (Eq. 3) is done by warp 3 of the same CTAs with bulk copies through a small staging buffer, each
// CTA of a head taking a slice of the rows; nothing in this launch reads the rows they write.
// Behind the step's compression launch each head waits (griddepcontrol.wait) only for what that
// launch gives it: heads of a type the step does not compress for nothing, heads that keep the whole
// new scale for their stored survivors, which come last, and only evicting contextual heads for
// everything.  Their CTAs lead the grid and start on the SMs the compression leaves free.
// A thread writes its output row from tensor memory, a whole 32-byte sector an instruction: the query tile's shared
// memory is free for the next unit's queries as soon as the last Q K^T product has read it.  (Tried: the output
// of a unit under the first block of the next one, in the wait for P: 1 to 2 % slower, the loop carries the code.
// Last units cut into pieces of their keys that the last one to finish adds up: 6 us per piece for the
// exchange through memory, more than the shorter last round gains.)
// Every mbarrier wait is bounded; on expiry the CTA raises the status word, drains what it has in
// flight, frees its TMEM and returns.
#include <cuda.h>

#include <algorithm>
#include <limits>
#include <type_traits>

#include "hack_internal.h"
#include "tc_ptx.cuh"

namespace hack {
namespace {

using namespace ptx;

constexpr int kBM = 128;                 // query rows per tile
constexpr int kBN = 128;                 // cache rows per K/V tile
constexpr int kMmaWarp = 0, kProducerWarp = 1, kPvWarp = 2, kAppendWarp = 3;   // an issuer is the oldest warp of its scheduler
// A CTA of T tiles: four warps that issue and four softmax warps per tile.  Registers are moved from the
// former to the latter: T = 2: 2*128*224 + 128*56 = 384*168 registers; T = 1: 128*200 + 128*56 = 256*128,
// half an SM's, like its tensor memory and shared memory: two such CTAs per SM.
template <int T> struct Shape;
template <> struct Shape<2> {
  static constexpr int kThreads = 384, kCtasPerSm = 1, kSoftmaxRegs = 224, kOtherRegs = 56;
  static constexpr uint32_t kTmemCols = 512, kOutCol = 256, kCopyChunk = 16384;   // kCopyChunk: bytes per bulk copy of the append
};
template <> struct Shape<1> {
  static constexpr int kThreads = 256, kCtasPerSm = 2, kSoftmaxRegs = 200, kOtherRegs = 56;
  static constexpr uint32_t kTmemCols = 256, kOutCol = 192, kCopyChunk = 8192;
};
constexpr int kKStages = 2;
constexpr int kVStages = 2;
constexpr uint32_t kSpinLimit = 1u << 22;          // polls while draining after an abort
constexpr uint32_t kWaitPolls = 1u << 28;          // polls of a wait without a clock, minutes
constexpr float kRescaleThreshold = 32.0f;   // log2 units: p <= 2^32, far inside the bf16 / fp32 range

struct TcParams {
  int n_new;
  int first_type, first_heads;           // the head type at the front of head_order and its heads
  int first_units;                       // its units; the other type's follow
  int units_per_head[2];                 // per head type
  int tiles_per_cta[2];                  // per head type: query tiles of a round (2, or 1)
  int rounds[2];                         // per head type: rounds of a unit (1 unless the keys are one block)
  int steal;                             // more units than CTAs run at once: a CTA goes on with another one
  int len_a[2], len_b[2];                // per head type: rows read from the cache, rows read from the caller's K/V
  int append_new;                        // heads with len_b > 0 also store those rows behind their len_a cache rows
  int dep[2];                            // per head type: what lies behind the dependency wait (kDep*)
  int q_before_wait;                     // the queries may be read ahead of the dependency wait
  int pos_base;                          // global position of the new scale's first token
  int head_dim_pieces;                   // 16-byte pieces per row
  int cap[2];                            // rows a head of each type owns (checked builds)
  long long wait_cycles;                 // limit of the producer's waits ...
  long long unit_cycles;                 // ... but those for other roles to be done with a unit of work
  uint4* k_plane;                        // cache planes of this layer (append only)
  uint4* v_plane;
  int32_t* pos_plane;
  const uint4* k_new;                    // the caller's K/V (append only)
  const uint4* v_new;
  float scale_log2;                      // sm_scale * log2(e)
  const int32_t* row_off;
  const int32_t* head_order;             // the heads of first_type, then the others
  __nv_bfloat16* out;
  int out_sectors;                       // the output starts on a 32-byte boundary
  float* row_stats;                      // optional [b*H, N_k, 2]: reference maximum and sum of every softmax row
  int* status;
};

// What a head has to wait for when the launch ahead in the stream may still be running.
constexpr int kDepNothing = 0;           // nothing that launch touches: it compresses the other head type only
constexpr int kDepCache = 1;             // the cache rows (and the place of the append); the new rows are the caller's
constexpr int kDepAll = 2;

// A piece of work: one head, some of its query tiles (`rounds` rounds of up to two).
struct Unit { int bh, part, type, krow; };

struct Bars {
  uint4 answer;                                     // of cluster launch control
  Unit unit[2];                                     // units of even and odd count; bh < 0: there is no more
  uint64_t u_full[2], u_empty[2], asked;
  uint64_t q_full[2], q_free[2];
  uint64_t k_full[kKStages], k_empty[kKStages];
  uint64_t v_full[kVStages], v_empty[kVStages];
  uint64_t s_full[2], s_free, p_full[2], p_free[2];
  uint64_t copy_full[2];                            // append: a chunk of new rows has landed in its staging half
  uint64_t drain[2];                                // the issuers' last products
  int2 out_at[8];                                   // per softmax warp
  uint32_t tmem_base;
  int abort_code;                                   // of the wait that gave up
};

// Waits for a phase of a barrier; false once a wait of the CTA has given up.  In little code: the instruction cache bounds
// this kernel.  The producer keeps the time: whatever else stands still, one of its own waits soon does too, and while
// it waits for the launch ahead, whose time is not this launch's, nobody's counts.  (A clock in every wait that leaves that time
// out: 33.6 -> 35.0 us a step of 256 heads x 64.)  The status word is written at the end, by one thread.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, Bars* b, int code) {
  const uint32_t addr = smem_u32(bar);
  if (__builtin_expect(mbar_try_wait(addr, parity), 1)) return true;
  volatile int* const flag = &b->abort_code;
#pragma unroll 1
  for (uint32_t polls = kWaitPolls; !mbar_try_wait(addr, parity); --polls) {
    if (*flag) return false;
    if (polls == 0) *flag = code;
  }
  return true;
}
// The same with a limit in clock cycles.
__device__ __forceinline__ bool wait_timed(uint64_t* bar, uint32_t parity, Bars* b, int code, long long limit) {
  const uint32_t addr = smem_u32(bar);
  if (__builtin_expect(mbar_try_wait(addr, parity), 1)) return true;
  volatile int* const flag = &b->abort_code;
  const long long t0 = clock64();
#pragma unroll 1
  while (!mbar_try_wait(addr, parity)) {
    if (*flag) return false;
    if (clock64() - t0 > limit) *flag = code;
  }
  return true;
}

template <int D, int T>
__global__ void __launch_bounds__(Shape<T>::kThreads, Shape<T>::kCtasPerSm)
attend_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                 const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_kn,
                 const __grid_constant__ CUtensorMap tm_vn, const TcParams p) {
  constexpr int SUB = D / 64;                       // 64-column (128-byte) sub-tiles per row
  constexpr uint32_t SUB_BYTES = kBN * 128;         // one sub-tile: 128 rows x 128 bytes
  constexpr uint32_t TILE_BYTES = SUB * SUB_BYTES;
  constexpr uint32_t S_COL = 0, P_COL = 128, O_COL = Shape<T>::kOutCol;
  constexpr int kSoftmaxRegs = Shape<T>::kSoftmaxRegs, kOtherRegs = Shape<T>::kOtherRegs;
  constexpr uint32_t kCopyChunk = Shape<T>::kCopyChunk;
  static_assert(P_COL + T * 64 <= O_COL && O_COL + T * D <= Shape<T>::kTmemCols, "tensor memory plan");

  extern __shared__ unsigned char smem_dyn[];
  const uint32_t raw = smem_u32(smem_dyn);
  const uint32_t base = (raw + 1023u) & ~1023u;     // 128-byte swizzle needs 1024-byte alignment
  unsigned char* sm = smem_dyn + (base - raw);
  const uint32_t q_sm = base;
  const uint32_t k_sm = q_sm + T * TILE_BYTES;
  const uint32_t v_sm = k_sm + kKStages * TILE_BYTES;
  const uint32_t copy_sm = v_sm + kVStages * TILE_BYTES;           // 2 x kCopyChunk bytes: staging of the append
  Bars* bars = reinterpret_cast<Bars*>(sm + (T + kKStages + kVStages) * TILE_BYTES + 2 * kCopyChunk);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // Unit number x of the launch: those of the first head type, then those of the other one.
  auto make_unit = [&](int x) {
    Unit u;
    const bool second = x >= p.first_units;
    u.type = second ? 1 - p.first_type : p.first_type;
    const int at = second ? x - p.first_units : x, per = p.units_per_head[u.type];
    const int head = at / per;
    u.part = at - head * per;
    u.bh = p.head_order[(second ? p.first_heads : 0) + head];
    u.krow = p.row_off[u.bh];
    return u;
  };
  // A role takes unit number n of this CTA (one thread; the arrival gives the slot back).
  auto wait_unit = [&](int n) { return wait_bar(&bars->u_full[n & 1], (n >> 1) & 1, bars, 13); };
  auto read_unit = [&](int n) {
    const volatile Unit& v = bars->unit[n & 1];
    return Unit{v.bh, v.part, v.type, v.krow};
  };
  auto give_unit = [&](int n) { mbar_arrive(smem_u32(&bars->u_empty[n & 1])); };
  // Its rounds, and in a round: the first query row and the tiles
  auto rounds_of = [&](const Unit& u) {
    const int rows = p.tiles_per_cta[u.type] * kBM, left = p.n_new - u.part * p.rounds[u.type] * rows;
    return min(p.rounds[u.type], (left + rows - 1) / rows);
  };
  auto first_row = [&](const Unit& u, int r) { return (u.part * p.rounds[u.type] + r) * p.tiles_per_cta[u.type] * kBM; };
  auto tiles_of = [&](const Unit& u, int q0) { return T == 2 && p.tiles_per_cta[u.type] == 2 && q0 + kBM < p.n_new ? 2 : 1; };
  // Blocks of 128 keys: the caller's rows come first (they may not have to wait), then the cache's; a head
  // never attends over nothing.
  auto blocks_b = [&](const Unit& u) { return (p.len_b[u.type] + kBN - 1) / kBN; };
  auto blocks = [&](const Unit& u) { return blocks_b(u) + (p.len_a[u.type] + kBN - 1) / kBN; };
  // Keys of the last block of a segment of `len` rows in groups of 32, the unit in which the products and the
  // softmax leave out what is past the last key
  auto last_groups = [](int len) { return (((len - 1) & (kBN - 1)) >> 5) + 1; };
  // Loads of the producer: a tile of 128 rows (the queries of slot t, or K / V block j of the unit)
  auto load_tile = [&](uint32_t dst, const CUtensorMap* tm, int row, uint64_t* bar) {
    mbar_expect_tx(smem_u32(bar), TILE_BYTES);
#pragma unroll 1
    for (int c = 0; c < SUB; ++c) tma_load_2d(dst + c * SUB_BYTES, tm, c * 64, row, smem_u32(bar));
  };
  auto load_kv = [&](const Unit& u, int j, int nb, uint32_t slot, int kv) {
    const bool b = j < nb;
    load_tile((kv ? v_sm : k_sm) + slot * TILE_BYTES, kv ? (b ? &tm_vn : &tm_v) : (b ? &tm_kn : &tm_k),
              b ? u.bh * p.n_new + j * kBN : u.krow + (j - nb) * kBN, kv ? &bars->v_full[slot] : &bars->k_full[slot]);
  };

  if (warp == kProducerWarp && lane == 0) {
#pragma unroll 1
    for (int t = 0; t < 2; ++t) {
      mbar_init(smem_u32(&bars->u_full[t]), 1);
      mbar_init(smem_u32(&bars->u_empty[t]), 3 + 4 * T);   // two issuers, the append, the softmax warps
      mbar_init(smem_u32(&bars->q_full[t]), 1);
      mbar_init(smem_u32(&bars->q_free[t]), 1);
      mbar_init(smem_u32(&bars->s_full[t]), 1);
      mbar_init(smem_u32(&bars->p_full[t]), 4);     // one arrival per warp of the tile
      mbar_init(smem_u32(&bars->p_free[t]), 1);
    }
    for (int s = 0; s < kKStages; ++s) { mbar_init(smem_u32(&bars->k_full[s]), 1); mbar_init(smem_u32(&bars->k_empty[s]), 1); }
    for (int s = 0; s < kVStages; ++s) { mbar_init(smem_u32(&bars->v_full[s]), 1); mbar_init(smem_u32(&bars->v_empty[s]), 1); }
    mbar_init(smem_u32(&bars->asked), 1);
    mbar_init(smem_u32(&bars->s_free), 4);          // the four warps of the tile whose logits were in the buffer
    mbar_init(smem_u32(&bars->copy_full[0]), 1);
    mbar_init(smem_u32(&bars->copy_full[1]), 1);
    mbar_init(smem_u32(&bars->drain[0]), 1);
    mbar_init(smem_u32(&bars->drain[1]), 1);
    bars->abort_code = 0;
    fence_barrier_init();
    fence_proxy_async();
  }
  if (T == 2 && warp == kProducerWarp) {
    // The barriers are ready; the producer does not wait for the others, nor they for its wait for the launch ahead:
    // with all of them behind that wait, their code came in from L2 only then (3.0 instead of 2.1 us from the end of the
    // compression to the first logits).  Not on half an SM, whose other half may be a CTA of the launch ahead that
    // their polling slows down (240 heads x 64, 1 045 keys: 110 against 114 us a step).
    __syncwarp();
    asm volatile("bar.arrive 1, %0;" ::"n"(Shape<T>::kThreads) : "memory");
    reg_dec<kOtherRegs>();
  }
  if (warp == kProducerWarp && lane == 0) {
    // the producer starts the first loads at once: they run under the TMEM allocation, the
    // synchronisation and the register reallocation below
    const Unit u = make_unit(blockIdx.x);
    bars->unit[0] = u;
    mbar_arrive(smem_u32(&bars->u_full[0]));
    const int nb = blocks_b(u), dep = p.dep[u.type], q0 = first_row(u, 0), ntile = tiles_of(u, q0);
    // The queries, like the new rows, are the caller's input.  When the kernel ahead of this one in
    // the stream is the step's own compression launch, whatever produced them had completed before
    // that launch passed its own dependency wait, hence before any CTA of this launch started: they
    // are loaded ahead of the wait.
    auto load_queries = [&]() {
      for (int t = 0; t < ntile; ++t) load_tile(q_sm + t * TILE_BYTES, &tm_q, u.bh * p.n_new + q0 + t * kBM, &bars->q_full[t]);
    };
    if (p.q_before_wait) load_queries();
    if (dep == kDepAll || (dep == kDepCache && nb == 0)) pdl_grid_wait();
    if (!p.q_before_wait) load_queries();
    load_kv(u, 0, nb, 0, 0);
    load_kv(u, 0, nb, 0, 1);
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(&bars->tmem_base), Shape<T>::kTmemCols);
    tmem_relinquish();
    // the next launch may start once every CTA of this one holds its tensor memory: a CTA of the next
    // launch that took the columns first would wait for this grid, and this CTA for the columns
    pdl_launch_dependents();
  }
  tc_fence_before();
  if (T == 1) __syncthreads();
  else if (warp != kProducerWarp) asm volatile("bar.sync 1, %0;" ::"n"(Shape<T>::kThreads) : "memory");
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&bars->tmem_base);
  // Everything above overlaps the tail of the previous kernel.  What waits for that kernel is the
  // producer (and so everything behind the tiles it loads) and the append.

  // An issuer leaves when its last product has ended, or after a while: a softmax thread that gave up waits for none.
  auto drained = [&](uint64_t* bar) {
    mma_commit(smem_u32(bar));
#pragma unroll 1
    for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait(smem_u32(bar), 0); ++it) {}
  };
  if (warp == kPvWarp) {
    // ------------------------------------------------------------------ issuer of the P V products
    // (a thread of its own: one thread issuing both products was the bottleneck of the CTA)
    reg_dec<kOtherRegs>();
    if (lane == 0) {
      constexpr uint32_t IDESC_PV = idesc_bf16_f32(kBM, D, 1);         // A = P (TMEM), B = V (MN-major)
      const uint64_t v_desc0 = smem_desc_sw128(v_sm, SUB_BYTES, 1024);
      bool ok = true;
      uint32_t g = 0, odd = 0;                                         // V tiles used up; per tile: products so far, parity
#pragma unroll 1
      for (int n = 0; ok; ++n) {
        ok = wait_unit(n);
        if (!ok) break;
        const Unit u = read_unit(n);
        give_unit(n);
        if (u.bh < 0) break;
        const int nb = blocks_b(u), nblk = blocks(u), nr = rounds_of(u);
        const int kg_b = last_groups(p.len_b[u.type]), kg_a = last_groups(p.len_a[u.type]);
#pragma unroll 1
        for (int r = 0; r < nr && ok; ++r) {
          const int ntile = tiles_of(u, first_row(u, r));
#pragma unroll 1
          for (int j = 0; j < nblk && ok; ++j) {
            const uint32_t vs = (g + j) % kVStages;
            const uint64_t vd = v_desc0 + (uint64_t)((vs * TILE_BYTES) >> 4);
            const int kg = j == nb - 1 ? kg_b : j == nblk - 1 ? kg_a : 4;
#pragma unroll 1
            for (int t = 0; t < ntile; ++t) {
              // (what comes last is the wait whose end something waits for)
              if (t == 0 && r == 0) ok = wait_bar(&bars->v_full[vs], ((g + j) / kVStages) & 1, bars, 6);
              const uint32_t o = tmem + O_COL + t * D, pa = tmem + P_COL + t * 64;
              if (!ok || !wait_bar(&bars->p_full[t], (odd >> t) & 1, bars, 5)) { ok = false; break; }
              tc_fence_after();
              if (kg == 4) {
                mma_ts_chain4(o, pa, vd, IDESC_PV, j > 0);
                mma_ts_chain4(o, pa + 32, vd + 4 * 128, IDESC_PV, 1);
              } else {
#pragma unroll 1
                for (int k = 0; k < 2 * kg; ++k) mma_ts(o, pa + 8 * k, vd + k * 128, IDESC_PV, j > 0 || k > 0);
              }
              mma_commit(smem_u32(&bars->p_free[t]));           // P_t may be rewritten, O_t is up to date
              odd ^= 1u << t;
              if (t == ntile - 1 && r == nr - 1) mma_commit(smem_u32(&bars->v_empty[vs]));
            }
          }
        }
        g += nblk;
      }
      drained(&bars->drain[1]);
    }
  } else if (warp == kAppendWarp) {
    reg_dec<kOtherRegs>();
    // Eq. 3 for the heads that keep the whole new scale: its rows go behind the len_a cache rows.  The rows are
    // one contiguous run in the caller's tensor and in the cache plane; the units of the head share
    // them, and one thread moves a unit's slice with bulk copies through two staging halves
    // (global -> shared -> global), so the append costs no registers and no issue slots.
    bool ok = true;
    uint32_t chunks = 0;                             // chunk counter over planes and units
#pragma unroll 1
    for (int n = 0; ok; ++n) {
      ok = __all_sync(0xffffffffu, wait_unit(n));
      if (!ok) break;
      const Unit u = read_unit(n);
      __syncwarp();
      if (lane == 0) give_unit(n);
      if (u.bh < 0) break;
      const int len_a = p.len_a[u.type], len_b = p.len_b[u.type];
      if (!p.append_new || len_b == 0 || !dbg_ok(len_a >= 0 && len_a + len_b <= p.cap[u.type], p.status, 7)) continue;
      if (p.dep[u.type] != kDepNothing) pdl_grid_wait();
      const int per = (len_b + p.units_per_head[u.type] - 1) / p.units_per_head[u.type];
      const int r0 = u.part * per, r1 = min(len_b, r0 + per);
#pragma unroll 1
      for (int r = r0 + lane; r < r1; r += 32) p.pos_plane[u.krow + len_a + r] = p.pos_base + r;
      if (lane == 0 && r1 > r0) {
        const uint32_t row_bytes = (uint32_t)p.head_dim_pieces * 16;
        const size_t src_off = ((size_t)u.bh * p.n_new + r0) * row_bytes, dst_off = ((size_t)u.krow + len_a + r0) * row_bytes;
        const uint32_t total = (uint32_t)(r1 - r0) * row_bytes;
        const uint32_t n_chunks = (total + kCopyChunk - 1) / kCopyChunk;
#pragma unroll 1
        for (int plane = 0; plane < 2 && ok; ++plane) {
          const unsigned char* src = reinterpret_cast<const unsigned char*>(plane == 0 ? p.k_new : p.v_new) + src_off;
          unsigned char* dst = reinterpret_cast<unsigned char*>(plane == 0 ? p.k_plane : p.v_plane) + dst_off;
#pragma unroll 1
          for (uint32_t ch = 0; ch < n_chunks && ok; ++ch, ++chunks) {
            const uint32_t half = chunks & 1;
            const uint32_t bytes = min(kCopyChunk, total - ch * kCopyChunk);
            const uint32_t bar = smem_u32(&bars->copy_full[half]);
            bulk_wait_read<1>();                     // the store that last read this half (two chunks ago) is done with it
            mbar_expect_tx(bar, bytes);
            bulk_load(copy_sm + half * kCopyChunk, src + (size_t)ch * kCopyChunk, bytes, bar);
            ok = wait_timed(&bars->copy_full[half], (chunks >> 1) & 1, bars, 12, p.wait_cycles);
            if (!ok) {                               // the copy gets a bounded chance to land before the CTA leaves
#pragma unroll 1
              for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait(bar, (chunks >> 1) & 1); ++it) {}
              break;
            }
            bulk_store(dst + (size_t)ch * kCopyChunk, copy_sm + half * kCopyChunk, bytes);
            bulk_commit();
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
    }
    if (lane == 0) bulk_wait<0>();                   // every store has been performed before the CTA may leave
  } else if (warp == kProducerWarp) {
    // ------------------------------------------------------------------ TMA producer, and the CTA's next unit
    if (T == 1) reg_dec<kOtherRegs>();
    if (lane == 0) {
      bool ok = true, pending = false;              // pending: an answer of cluster launch control is on its way
      uint32_t g = 0, issued_k = 1, issued_v = 1;   // K / V tiles of the units before this one; tiles on their way so far
      uint32_t q_issued = 0, q_odd = 0, answers = 0;   // bit t: query slot t was filled, the parity of its fillings
      Unit u = bars->unit[0];
#pragma unroll 1
      for (int n = 0;; ++n) {
        const int nb = blocks_b(u), nblk = blocks(u), nr = rounds_of(u), dep = p.dep[u.type];
        if (n > 0 && (dep == kDepAll || (dep == kDepCache && nb == 0))) pdl_grid_wait();
        // K / V tiles of the unit in order, and the queries of round r ahead of step r's value tile
#pragma unroll 1
        for (int j = 0; j < max(nblk, nr) && ok; ++j) {
          if (dep == kDepCache && j == nb && j < nblk) pdl_grid_wait();   // the head's stored survivors are in place
          const bool fresh = n > 0 || j > 0;        // the first tiles and queries of the CTA are on their way already
          const uint32_t gs = g + j;
#pragma unroll 1
          for (int kv = 0; kv < 2 && ok; ++kv) {
            if (kv == 1 && j < nr) {
              const int q0 = first_row(u, j), ntile = tiles_of(u, q0);
#pragma unroll 1
              for (int t = 0; t < ntile && ok; ++t) {
                if (fresh) {
                  if (q_issued >> t & 1) ok = wait_timed(&bars->q_free[t], ((q_odd >> t) & 1) ^ 1, bars, 14, p.wait_cycles);
                  if (!ok) break;
                  load_tile(q_sm + t * TILE_BYTES, &tm_q, u.bh * p.n_new + q0 + t * kBM, &bars->q_full[t]);
                }
                q_issued |= 1u << t;
                q_odd ^= 1u << t;
              }
            }
            if (!ok || !fresh || j >= nblk) continue;
            const uint32_t sl = gs % kKStages;      // (both rings have the same depth)
            ok = wait_timed(kv ? &bars->v_empty[sl] : &bars->k_empty[sl], ((gs / kKStages) & 1) ^ 1, bars, 1 + kv, p.wait_cycles);
            if (!ok) break;
            load_kv(u, j, nb, sl, kv);
            if (kv) ++issued_v;
            else ++issued_k;
          }
        }
        if (!ok) break;
        g += nblk;
        Unit next{-1, 0, 0, 0};
        if (p.steal) {
          // The next unit is asked for behind the last load of this one: three blocks earlier, it would be kept
          // from CTAs that are idle by then (512 units of 5 blocks on 296 places: 43.0 against 37.4 us a step).
          mbar_expect_tx(smem_u32(&bars->asked), 16);
          clc_ask(smem_u32(&bars->answer), smem_u32(&bars->asked));
          pending = true;
          ok = wait_timed(&bars->asked, answers & 1, bars, 15, p.wait_cycles);
          if (!ok) break;
          pending = false;
          ++answers;
          const int x = clc_answer(smem_u32(&bars->answer));
          fence_proxy_async();                       // the next answer overwrites what was just read
          if (x >= 0) next = make_unit(x);
        }
        if (n > 0) ok = wait_timed(&bars->u_empty[(n + 1) & 1], (((n + 1) >> 1) & 1) ^ 1, bars, 16, p.unit_cycles);
        if (!ok) break;
        bars->unit[(n + 1) & 1] = next;
        mbar_arrive(smem_u32(&bars->u_full[(n + 1) & 1]));
        if (next.bh < 0) {                           // the roles leave on time as well
          ok = wait_timed(&bars->u_empty[n & 1], (n >> 1) & 1, bars, 17, p.unit_cycles);
          break;
        }
        u = next;
      }
      if (!ok) {
        // give the copies already in flight a bounded chance to land before the CTA leaves
        auto landed = [&](uint64_t* bar, uint32_t parity) {
          for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait(smem_u32(bar), parity); ++it) {}
        };
        if (pending) landed(&bars->asked, answers & 1);
#pragma unroll 1
        for (int t = 0; t < T; ++t)
          if (q_issued >> t & 1) landed(&bars->q_full[t], ((q_odd >> t) & 1) ^ 1);
#pragma unroll 1
        for (uint32_t i = 0; i < kKStages; ++i) {
          if (issued_k > i) landed(&bars->k_full[(issued_k - 1 - i) % kKStages], ((issued_k - 1 - i) / kKStages) & 1);
          if (issued_v > i) landed(&bars->v_full[(issued_v - 1 - i) % kVStages], ((issued_v - 1 - i) / kVStages) & 1);
        }
      }
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------------ issuer of the Q K^T products
    reg_dec<kOtherRegs>();
    if (lane == 0) {
      constexpr uint32_t IDESC_0 = idesc_bf16_f32(kBM, 0, 0);          // A = Q, B = K (both K-major); N is added
      // descriptors of the tile bases; a k-step only adds a constant to the address field
      const uint64_t q_desc0 = smem_desc_sw128(q_sm, 16, 1024), k_desc0 = smem_desc_sw128(k_sm, 16, 1024);
      bool ok = true;
      // S = Q_t K_j^T into the one logit buffer; `use` counts the products issued so far, and product
      // number use needs the logits of product use - 1 to have left the buffer (s_free phase use - 1).  The
      // next logits only wait for the buffer, not for the softmax of the tile or the end of a unit.
      uint32_t use = 0, g = 0, q_odd = 0;
#pragma unroll 1
      for (int n = 0; ok; ++n) {
        ok = wait_unit(n);
        if (!ok) break;
        const Unit u = read_unit(n);
        give_unit(n);
        if (u.bh < 0) break;
        const int nb = blocks_b(u), nblk = blocks(u), nr = rounds_of(u);
        const uint32_t idesc_b = IDESC_0 + ((uint32_t)(last_groups(p.len_b[u.type]) * 4) << 17);
        const uint32_t idesc_a = IDESC_0 + ((uint32_t)(last_groups(p.len_a[u.type]) * 4) << 17);
#pragma unroll 1
        for (int r = 0; r < nr && ok; ++r) {
          const int ntile = tiles_of(u, first_row(u, r));
#pragma unroll 1
          for (int j = 0; j < nblk && ok; ++j) {
            const uint32_t ks = (g + j) % kKStages;
            const uint64_t kd = k_desc0 + (uint64_t)((ks * TILE_BYTES) >> 4);
            const uint32_t idesc = j == nb - 1 ? idesc_b : j == nblk - 1 ? idesc_a : IDESC_0 + ((kBN >> 3) << 17);
#pragma unroll 1
            for (int t = 0; t < ntile; ++t) {
              if (j == 0) {
                ok = wait_bar(&bars->q_full[t], (q_odd >> t) & 1, bars, 3);
                q_odd ^= 1u << t;
              }
              if (ok && t == 0 && r == 0) ok = wait_bar(&bars->k_full[ks], ((g + j) / kKStages) & 1, bars, 4);
              const uint64_t qd = q_desc0 + (uint64_t)((t * TILE_BYTES) >> 4);
              if (!ok || !wait_bar(&bars->s_free, (use - 1) & 1, bars, 10)) { ok = false; break; }   // (a fresh barrier passes for odd)
              tc_fence_after();
              if constexpr (D == 128) mma_ss_chain8(tmem + S_COL, qd, kd, idesc, 0);
              else mma_ss_chain4(tmem + S_COL, qd, kd, idesc, 0);
              mma_commit(smem_u32(&bars->s_full[t]));
              ++use;
              if (j == nblk - 1) mma_commit(smem_u32(&bars->q_free[t]));
              if (t == ntile - 1 && r == nr - 1) mma_commit(smem_u32(&bars->k_empty[ks]));
            }
          }
        }
        g += nblk;
      }
      drained(&bars->drain[0]);
    }
  } else {
    // ------------------------------------------------------------------ softmax + epilogue
    reg_inc<kSoftmaxRegs>();
    const int t = (warp >> 2) - 1;                 // tile served by this warpgroup
    const int row = tid & 127;                     // query row inside the tile == TMEM lane
    const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t s_addr = tmem + lane_addr + S_COL;
    const uint32_t p_addr = tmem + lane_addr + P_COL + t * 64;
    const uint32_t o_addr = tmem + lane_addr + O_COL + t * D;
    const float c = p.scale_log2;
    float m_used = kNoLogit, l = 0.f;
    uint32_t cnt = 0;                              // blocks of this tile so far
    bool ok = true, pending = false;               // pending: a round's output is still in tensor memory
    volatile int2* const out_at = &bars->out_at[warp - 4];   // of the round in work or pending: first row of its head, row of the tile
    auto bar_all = [&](uint64_t* bar, uint32_t parity, int code) { return __all_sync(0xffffffffu, wait_bar(bar, parity, bars, code)) != 0; };
    // Output of the round that ended.  A thread writes its own row, 32 bytes (a whole sector) an instruction,
    // straight from tensor memory: through the query tile's shared memory and a tiled store, the next round's
    // queries could not be on their way meanwhile.
    auto flush = [&]() {
      ok = bar_all(&bars->p_free[t], (cnt - 1) & 1, 9);        // the round's last product
      if (!ok) return;
      pending = false;
      tc_fence_after();
      const float inv = 1.f / l;
      const int head_row = out_at->x, tile_row = out_at->y + row;
      const bool out_live = tile_row < p.n_new;
      const size_t out_row = (size_t)head_row + tile_row;
      if (p.row_stats && out_live) *reinterpret_cast<float2*>(p.row_stats + out_row * 2) = make_float2(m_used, l);
      unsigned char* dst = reinterpret_cast<unsigned char*>(p.out) + out_row * (D * 2);
#pragma unroll 1
      for (int ch = 0; ch < D / 16; ++ch) {
        uint32_t orr[16], w[8];
        tmem_ld16(o_addr + ch * 16, orr);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const __nv_bfloat162 hh = __floats2bfloat162_rn(__uint_as_float(orr[2 * e]) * inv, __uint_as_float(orr[2 * e + 1]) * inv);
          w[e] = *reinterpret_cast<const uint32_t*>(&hh);
        }
        if (out_live) st_global_32b(dst + ch * 32, w, p.out_sectors != 0);
      }
    };
    // What a block adds to the reference maximum, the sum and, if the maximum grew, the factor of what is there
    auto raise = [&](float mx, float& alpha) {
      const bool grow = (mx - m_used) * c > kRescaleThreshold;     // always true in the first block
      const bool any = __any_sync(0xffffffffu, grow);
      alpha = 1.f;
      if (any) {
        const float m_new = grow ? mx : m_used;
        alpha = grow ? ex2((m_used - m_new) * c) : 1.f;
        l *= alpha;
        m_used = m_new;
      }
      return any;
    };
    // The second MMA sees the probabilities rounded to bf16, the row sum does not.  With the
    // lazily raised reference maximum even a dominant key's probability is no power of two,
    // and its rounding error (up to 2^-9 of an output that can reach 4) would pass straight
    // into O.  The block's largest probability is therefore entered into the sum as rounded,
    // which makes the weight of a dominant key exact; what is left is bounded by the weight
    // of the other keys.  Same instructions as the loops use for that element, hence the same bits.
    auto top_rounding = [&](float mx, float nmc) {
      const float p_top = ex2(fmaf(mx, c, nmc));
      return __bfloat162float(__float2bfloat16_rn(p_top)) - p_top;
    };
    // P_t still feeds the product of the previous block, which also still adds to O_t
    auto wait_p = [&](bool rescale, float alpha) {
      ok = bar_all(&bars->p_free[t], (cnt - 1) & 1, 11);
      if (!ok) return;
      tc_fence_after();
      if (rescale) {
#pragma unroll 1
        for (int ch = 0; ch < D / 8; ++ch) {               // rare path: kept light on registers
          uint32_t orr[8];
          tmem_ld8(o_addr + ch * 8, orr);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 8; ++i) orr[i] = __float_as_uint(__uint_as_float(orr[i]) * alpha);
          tmem_st8(o_addr + ch * 8, orr);
        }
      }
    };
    auto give_p = [&]() {
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->p_full[t]));
      ++cnt;
    };
    // A block of keys, the first `valid` of them live, in G groups of 32: 4, or (the last block of a segment) 2.
    auto block = [&](auto groups_c, bool first, int valid) {
      constexpr int G = decltype(groups_c)::value, N = 32 * G;
      ok = bar_all(&bars->s_full[t], cnt & 1, 8);
      if (!ok) return;
      tc_fence_after();
      uint32_t sr[N];
#pragma unroll
      for (int ch = 0; ch < G; ++ch) tmem_ld32(s_addr + ch * 32, sr + ch * 32);
      tmem_wait_ld();
      // the logits are in registers: the buffer goes back to the MMA warp at once
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->s_free));
      if (__builtin_expect(valid < N, 0)) {
#pragma unroll
        for (int i = G == 4 ? 64 : 0; i < N; ++i)
          if (i >= valid) sr[i] = 0xff800000u;   // -inf
      }
      float mx4[G];
#pragma unroll
      for (int u = 0; u < G; ++u) {
        mx4[u] = -INFINITY;
#pragma unroll
        for (int i = 0; i < 16; ++i) mx4[u] = max3(mx4[u], __uint_as_float(sr[u * 32 + 2 * i]), __uint_as_float(sr[u * 32 + 2 * i + 1]));
      }
      const float mx = G == 4 ? fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[G - 2], mx4[G - 1])) : fmaxf(mx4[0], mx4[1]);
      float alpha;
      const bool any_grow = raise(mx, alpha);
      const float2 c2 = make_float2(c, c);
      const float2 nmc2 = make_float2(-m_used * c, -m_used * c);
      float2 sum4[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      uint32_t pk[N / 2];
#pragma unroll
      for (int i = 0; i < N / 2; ++i) {
        const float2 x = fma2(make_float2(__uint_as_float(sr[2 * i]), __uint_as_float(sr[2 * i + 1])), c2, nmc2);
        float2 pr;
        pr.x = ex2(x.x);
        pr.y = ex2(x.y);
        sum4[i & 3] = add2(sum4[i & 3], pr);
        const __nv_bfloat162 hh = __floats2bfloat162_rn(pr.x, pr.y);
        pk[i] = *reinterpret_cast<const uint32_t*>(&hh);
      }
      const float2 sum2 = add2(add2(sum4[0], sum4[1]), add2(sum4[2], sum4[3]));
      l += sum2.x + sum2.y;
      l += top_rounding(mx, nmc2.x);
      if (cnt > 0) {
        wait_p(any_grow && !first, alpha);
        if (!ok) return;
      }
#pragma unroll
      for (int ch = 0; ch < G / 2; ++ch) tmem_st32(p_addr + ch * 32, pk + ch * 32);
      give_p();
    };
    // (What a round needs is read where it is needed: registers that live through a block are scarce.)
    int n = 0, r = 0;
    ok = __all_sync(0xffffffffu, wait_unit(0)) != 0;
#pragma unroll 1
    while (ok) {
      int left = 0, then = 0;                      // keys left of the caller's rows or the cache's; the cache's to follow
      const Unit u = read_unit(n);
      if (u.bh >= 0) {
        if (r == rounds_of(u)) {
          __syncwarp();
          if (lane == 0) give_unit(n);
          ++n;
          r = 0;
          ok = __all_sync(0xffffffffu, wait_unit(n)) != 0;
          continue;
        }
        if (t >= tiles_of(u, first_row(u, r))) { ++r; continue; }
        left = p.len_b[u.type];
        then = p.len_a[u.type];
        if (left == 0) { left = then; then = 0; }
      }
      if (pending) flush();                        // the round before this one
      if (left == 0 || !ok) break;                 // (the end: there is no other round without keys)
      if (lane == 0) { out_at->x = u.bh * p.n_new; out_at->y = first_row(u, r) + t * kBM; }
      __syncwarp();
      ++r;
      m_used = kNoLogit;
      l = 0.f;
      pending = true;
      bool first = true;
#pragma unroll 1
      while (ok) {
        if (left > 64) block(std::integral_constant<int, 4>(), first, left);
        else block(std::integral_constant<int, 2>(), first, left);
        first = false;
        left -= kBN;
        if (left <= 0) {
          left = then;
          then = 0;
          if (left == 0) break;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, Shape<T>::kTmemCols);
  }
  if (tid == 0 && bars->abort_code) atomicExch(p.status, bars->abort_code);
  // The launch behind this one relies on everything ahead of it being complete once this grid is, so
  // no CTA leaves before the launch ahead has completed, whatever its heads depend on.
  if (tid == 0) pdl_grid_wait();
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(sym);
  }
  return fn;
}

template <int D, int T>
size_t tc_smem_bytes() {
  return 1024 + (T + kKStages + kVStages) * (size_t)(D / 64) * kBN * 128 + 2 * Shape<T>::kCopyChunk + sizeof(Bars) + 64;
}

}  // namespace

// 2-D bf16 tensor map over `rows` x `head_dim`, box = 128 rows x 64 columns, 128-byte swizzle.
bool make_rows_map(void* out_map, const void* base, uint64_t rows, int head_dim) {
  EncodeTiledFn fn = encode_fn();
  if (!fn || rows == 0) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)head_dim, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)head_dim * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)kBN};
  const cuuint32_t estr[2] = {1, 1};
  return fn(static_cast<CUtensorMap*>(out_map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims,
            strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {
template <int D, int T>
int launch_tc(int grid, cudaStream_t st, const CUtensorMap& tm_q, const CUtensorMap& tk, const CUtensorMap& tv,
              const CUtensorMap& tm_kn, const CUtensorMap& tm_vn, const TcParams& p) {
  // two tiles of head_dim 64 ask for as much as head_dim 128: one CTA per SM, it owns all of tensor memory
  const size_t smem = T == 2 ? tc_smem_bytes<128, 2>() : tc_smem_bytes<D, T>();
  if (!allow_dynamic_smem(attend_tc_kernel<D, T>, smem)) return -1;
  launch_k(attend_tc_kernel<D, T>, grid, Shape<T>::kThreads, smem, st, tm_q, tk, tv, tm_kn, tm_vn, p);
  return launched(1);
}
}  // namespace

float attend_tc_sm_us(const StepArgs& a, int type) {
  // 4.5 us around the steps of a CTA (of a unit: a CTA that goes on with another one hides part of it); a step of 128 keys
  // is bound by the exponentials at head_dim 64
  const float step_us = a.head_dim == 128 ? 1.6f : 1.2f;
  return (float)a.heads_of[type] * ((a.n_new + 2 * kBM - 1) / (2 * kBM)) * (4.5f + step_us * ((a.kept[type] + kBN - 1) / kBN));
}

int launch_attend_tc(const StepArgs& a, const void* q, void* out, float* row_stats, const void* k_new,
                     const void* v_new, cudaStream_t st, int compression_ctas) {
  CUtensorMap tm_q;
  if (!make_rows_map(&tm_q, q, (uint64_t)a.batch * a.n_heads * a.n_new, a.head_dim)) {
    set_error("attention: cuTensorMapEncodeTiled failed for the queries");
    return -1;
  }
  TcParams p;
  p.n_new = a.n_new;
  const CUtensorMap& tk = *static_cast<const CUtensorMap*>(a.k_map);
  const CUtensorMap& tv = *static_cast<const CUtensorMap*>(a.v_map);
  CUtensorMap tm_kn = tk, tm_vn = tv;       // placeholders unless a head type reads the caller's rows
  p.append_new = 0;
  for (int t = 0; t < 2; ++t) {
    const bool from_caller = k_new && v_new && a.seg_new[t];
    p.len_b[t] = from_caller ? a.n_new : 0;
    p.len_a[t] = a.kept[t] - p.len_b[t];
    if (from_caller) p.append_new = 1;
  }
  if (p.append_new) {
    const uint64_t rows = (uint64_t)a.batch * a.n_heads * a.n_new;
    if (!make_rows_map(&tm_kn, k_new, rows, a.head_dim) || !make_rows_map(&tm_vn, v_new, rows, a.head_dim)) {
      set_error("attention: cuTensorMapEncodeTiled failed for the new scale's keys or values");
      return -1;
    }
  }
  // Behind the step's compression launch a head type that the step does not compress waits for
  // nothing, one that keeps the whole new scale waits only for its stored survivors.  The type that
  // waits least goes first (its CTAs start on the SMs the compression leaves free), then the longer one.
  for (int t = 0; t < 2; ++t)
    p.dep[t] = compression_ctas == 0 ? kDepAll : !a.trig[t] ? kDepNothing : p.len_b[t] > 0 ? kDepCache : kDepAll;
  p.q_before_wait = compression_ctas > 0;
  p.first_type = p.dep[0] != p.dep[1] ? (p.dep[1] < p.dep[0]) : (a.kept[1] > a.kept[0]);
  p.first_heads = a.heads_of[p.first_type];
  // One query tile per CTA while that still fits one wave (twice the CTAs, no idle SMs), else two.  A
  // type that does not wait for the compression has the SMs that launch does not hold.
  const int n_tiles = (a.n_new + kBM - 1) / kBM;
  // head_dim 64: CTAs of one tile that take half an SM each.  They read every K/V tile twice as often as CTAs of two
  // tiles, but a head of an odd number of tiles leaves none of those half empty.  Halves and whole SMs behind a compression, us a
  // step: 240 heads, 3 tiles, 5 to 9 blocks of keys 48.1 to 73.7 and 51.2 to 77.3, 5 tiles, 8 blocks 84.0 and 85.5, but 4 tiles, 8
  // blocks 75.3 and 72.2, 8 tiles, 9 and 12 blocks 119.8 and 113.9, 150.5 and 141.8; where every tile finds an SM whole ones, whose warps
  // run ahead of the wait, are as fast or faster (34 heads, 3 tiles, 8 blocks 29.7 and 28.1, 4 tiles, 5 blocks 24.6 and 23.6).
  // Without one: 256 heads, 1 tile, 2 blocks 10.0 and 13.3, 2 tiles, 3 blocks 20.1 and 18.8, 64 heads, 8 tiles, 18 blocks 69.6 and 61.4.
  const int longest = (std::max(a.kept[0], a.kept[1]) + kBN - 1) / kBN;
  const bool halves = a.head_dim == 64 && n_tiles % 2 == 1 && n_tiles * (a.heads_of[0] + a.heads_of[1]) > sm_count() &&
                      longest <= (compression_ctas > 0 ? 12 : 4);
  const int slots = sm_count() * (halves ? 2 : 1);           // CTAs that run at once
  const bool apart = p.dep[p.first_type] == kDepNothing && p.dep[1 - p.first_type] != kDepNothing;   // one type runs after the other
  for (int t = 0; t < 2; ++t) {
    const int heads = apart ? a.heads_of[t] : a.heads_of[0] + a.heads_of[1];
    const int sms = sm_count() - (p.dep[t] == kDepNothing ? compression_ctas : 0);
    p.tiles_per_cta[t] = halves || n_tiles * heads <= sms ? 1 : 2;
    const int parts = (n_tiles + p.tiles_per_cta[t] - 1) / p.tiles_per_cta[t];
    p.rounds[t] = a.kept[t] <= kBN && (p.len_a[t] == 0 || p.len_b[t] == 0) ? std::min(parts, std::max(1, parts * a.heads_of[t] / slots)) : 1;
    p.units_per_head[t] = (parts + p.rounds[t] - 1) / p.rounds[t];
  }
  p.first_units = p.units_per_head[p.first_type] * p.first_heads;
  const int grid = p.first_units + p.units_per_head[1 - p.first_type] * a.heads_of[1 - p.first_type];
  p.steal = grid > slots - compression_ctas / (halves ? 2 : 1);
  p.pos_base = a.pos_base;
  p.head_dim_pieces = a.head_dim * 2 / 16;
  p.cap[0] = a.cap[0];
  p.cap[1] = a.cap[1];
  constexpr long long kMost = std::numeric_limits<long long>::max() / 4;
  p.wait_cycles = std::min(a.wait_cycles, kMost);
  // a block takes a role no more than eight waits
  long long unit_waits = 0;
  for (int t = 0; t < 2; ++t)
    unit_waits = std::max<long long>(unit_waits, 8ll * p.rounds[t] * ((p.len_a[t] + kBN - 1) / kBN + (p.len_b[t] + kBN - 1) / kBN + 1));
  p.unit_cycles = p.wait_cycles > kMost / unit_waits ? kMost : p.wait_cycles * unit_waits;
  p.k_plane = static_cast<uint4*>(a.k_plane);
  p.v_plane = static_cast<uint4*>(a.v_plane);
  p.pos_plane = a.pos_plane;
  p.k_new = static_cast<const uint4*>(k_new);
  p.v_new = static_cast<const uint4*>(v_new);
  p.scale_log2 = a.sm_scale * 1.4426950408889634f;
  p.row_off = a.row_off;
  p.head_order = a.head_order + (size_t)p.first_type * a.batch * a.n_heads;
  p.out = static_cast<__nv_bfloat16*>(out);
  p.out_sectors = reinterpret_cast<uintptr_t>(out) % 32 == 0;
  p.row_stats = row_stats;
  p.status = a.status;
  if (a.head_dim == 128) return launch_tc<128, 2>(grid, st, tm_q, tk, tv, tm_kn, tm_vn, p);
  return halves ? launch_tc<64, 1>(grid, st, tm_q, tk, tv, tm_kn, tm_vn, p)
                : launch_tc<64, 2>(grid, st, tm_q, tk, tv, tm_kn, tm_vn, p);
}

}  // namespace hack
