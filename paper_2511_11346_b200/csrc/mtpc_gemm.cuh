// Projection kernel of the MtPC head (Sec. 3.3): logits = h W^T on the tcgen05 tensor cores, with the softmax
// over the vocabulary, the evidence gather (log phi at the target byte) and the log-softmax of the sum-unit logits all done
// in the epilogue straight out of tensor memory. The [positions, n, r, v] logit tensor never exists in HBM, except when a
// training call or a draft of many positions asks the epilogue to keep it (logit_out).
//
// One persistent CTA per SM, 10 warps:
//   warp 0      TMA producer: per 64-wide K block, one 128-row tile of h and the v rows of one emission unit
//               (or one tile of sum-unit rows) into a ring of shared-memory stages (128-byte swizzle).
//   warp 1      allocates the 512 TMEM columns, issues tcgen05.mma (M=128, N=chunk, K=16) from one thread. Warps 0 and 1 run as wholes
//               and predicate what they issue (elect_one): short calls 1 to 6 % shorter than from branches of lane 0's own (300 factored
//               positions of 4 x 8 x 256, d = 1024: 45.6 -> 42.8 us, 500 of 8 x 16 x 320, d = 2048: 69.0 -> 67.7).
//   warps 2..9  epilogue (2..5 on sorted rows); warp w reads TMEM lanes 32*(w%4)..+31, one thread per position (row), so every
//               row-wise reduction over the vocabulary is an in-thread loop, shared by the two warps of the same lanes.
// The N axis of the GEMM is the flattened (slot i, unit k, byte b) row index of W_emit. A work item is 128
// positions x one "group": `group_units` consecutive emission units = a run of rows that starts at a unit
// boundary, covered by accumulator tiles of `tile_cols` columns. The log-likelihood mode uses 256-column tiles
// whatever v is (v=320: 4 units = 1280 rows = 5 tiles; v=256: 1 unit = 1 tile): a tile may then hold the end
// of one unit and the start of the next, and the epilogue carries its running max / sum across tiles and
// closes a unit whenever its v-th column has been consumed. Sum-unit rows form work items of their own
// (one tile of `sum_cols` columns). Accumulators live in a ring of TMEM slots, so the epilogue of one tile
// overlaps the MMAs of the next. Every barrier wait is bounded: when one runs out the CTA raises
// MTPC_STATUS_TIMEOUT in the status word, drains its copies, frees its TMEM and returns.
#pragma once
#include <cuda_bf16.h>
#include <math_constants.h>

#include "mtpc_group.cuh"
#include "mtpc_ptx.cuh"

namespace mtpc {

constexpr int kBlockM = 128;         // positions per tile (= TMEM lanes)
constexpr int kBlockK = 64;          // bf16 elements per 128-byte swizzled row
constexpr int kMaxStages = 16;
constexpr int kMaxSlots = 8;
constexpr int kTmemCols = 512;
constexpr int kGemmThreads = 192;
constexpr uint64_t kWaitLimitNs = 1000ull * 1000ull * 1000ull;   // 1 s per barrier wait (the default, and always the limit of the drain waits)
constexpr uint64_t kAwakeNs = 100ull * 1000ull;                  // limits below this: see first_wait
constexpr uint64_t kAbortSettleNs = 200ull * 1000ull;            // 0.2 ms: far longer than any copy or MMA in flight takes
constexpr int kABytes = kBlockM * kBlockK * 2;                   // 16 KB
constexpr uint32_t kStatusBadTarget = 1u, kStatusBadUniform = 2u, kStatusTimeout = 4u;

// kModeLogitsGrouped: rows sorted by SLOT (the acceptance stage after a many-position draft): a work item is a GroupTile
// whose `unit` is a slot and a run of group_units of the slot's r units; their logits and log-sum-exps are written out per
// staged row. (There are only about n + rows / 128 tiles: without the split over units a batch of 4096 windows of 16 slots
// is 45 items for 148 SMs, each r v columns long: 623 us against 213.)
enum { kModeLogprob = 0, kModeLogitsGrouped = 1 };

struct GemmParams {
  CUtensorMap tm_a;      // hidden  [T, d]        box 64 x 128
  CUtensorMap tm_emit;   // W_emit  [n*r*v, d]    box 64 x tile_cols
  CUtensorMap tm_sum;    // W_sum   [S*r, d]      box 64 x sum_cols
  int T, m_tiles, kblocks;
  int m_units;                       // M work units: m-tiles, or pairs of m-tiles when two CTAs share every MMA
  int m_block;                       // M work units per rasterisation block (see tile_coord)
  int n, r, v;
  int vv;                            // symbols that exist (<= v, > v - 16): the columns [vv, v) of every unit are padding
  int emit_units;                    // n * r
  int num_groups;                    // emission groups in this launch (0: sum tiles only)
  int group_units;                   // emission units per full group (the last group may hold fewer)
  int tile_cols;                     // accumulator width of an emission tile
  int num_sum_tiles;                 // sum tiles in this launch (0: emission groups only)
  int sum_cols, sum_rows;            // sum tile width; S * r
  int slot_stride, num_slots;
  int stages, stage_bytes;
  const int* targets;                // [T, n] or NULL (a draft: no evidence yet, the logits are kept)
  float* G;                          // [T, n, r]       log phi at the target
  float* logw;                       // [T, S*r]        log-softmaxed sum-unit weights
  const float* sum_bias;             // [S*r] or NULL   added to the sum-unit logits before their softmax
  float* lse_out;                    // [T, n, r] or NULL: log-sum-exp of every input unit, kept for the backward pass or a draft
  float* logit_out;                  // [T, n*r*v] fp32 with row pitch logit_pitch, or NULL: the emission logits themselves,
  size_t logit_pitch;                // kept for the backward pass or a draft (padding columns as -inf)
  const GroupTile* group_tiles;      // sorted rows: the work items, and ...
  const int* group_num_tiles;        // ... how many there are (device memory: written by the kernel that made them)
  unsigned* work_counter;            // zeroed here for the circuit kernel that hands out its windows through it, or NULL
  unsigned* status;
  uint64_t wait_limit_ns;            // limit of every pipeline wait (kWaitLimitNs unless a test shortened it)
};

struct GemmControl {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t tfull[kMaxSlots];
  uint64_t tempty[kMaxSlots];
  uint64_t drain;
  uint64_t wait_limit_ns;
  uint32_t tmem_base;
  volatile int abort;
};

__device__ __forceinline__ float fast_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float fast_lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
// The log-likelihood epilogue's exponentials never take a reference below this: its product with log2 e is rounded by 64 at most, so that what
// lies below has no mass and never overflows, also where a run of -inf or of huge negative logits is all that a warp has seen.
constexpr float kLowestRef = -0x1p30f;

__device__ __forceinline__ bool bounded_wait(uint32_t bar, uint32_t parity, GemmControl* ctl, unsigned* status) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  uint32_t it = 0;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((++it & 15u) == 0) {
      if (ctl->abort) return false;
      if (global_timer_ns() - t0 > ctl->wait_limit_ns) {
        ctl->abort = 1;
        atomicOr(status, kStatusTimeout);
        return false;
      }
    }
  }
}
// Lane 0 waits, the whole warp learns the outcome (keeps the warp converged for the .sync.aligned TMEM loads).
__device__ __forceinline__ bool bounded_wait_warp(uint32_t bar, uint32_t parity, GemmControl* ctl, unsigned* status,
                                                  int lane) {
  int ok = 1;
  if (lane == 0) ok = bounded_wait(bar, parity, ctl, status) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// The whole warp waits and learns the outcome, known to be the same in every lane. It sleeps in try_wait until the barrier's phase is over or for
// as long as the hardware lets it (a suspend-time hint of 50 ns does not shorten that), and then looks whether another role has given up. P: the
// kernel's parameters.
template <typename P>
__device__ __forceinline__ bool bounded_wait_all(uint32_t bar, uint32_t parity, GemmControl* ctl, const P& p) {
  constexpr unsigned all = 0xffffffffu;
  if (__all_sync(all, mbar_try_wait(bar, parity))) return true;
  const uint64_t t0 = global_timer_ns();
  while (true) {
    if (__any_sync(all, ctl->abort)) return false;
    if (__all_sync(all, mbar_try_wait(bar, parity))) return true;
    if (__any_sync(all, global_timer_ns() - t0 > p.wait_limit_ns)) {
      ctl->abort = 1;
      if (elect_one()) atomicOr(p.status, kStatusTimeout);
      return false;
    }
  }
}
// A sleep outlasts limits of microseconds, and a choice between sleeping and not at every wait costs GEMMs 1.5 % (5 x 401 positions of a training call
// 990 -> 1005 us). So with a limit that short the MMA issuer keeps awake for its first copies, and what it decides reaches the other roles by the
// abort flag.
template <typename P>
__device__ __forceinline__ bool first_wait(uint32_t bar, GemmControl* ctl, const P& p) {
  constexpr unsigned all = 0xffffffffu;
  if (p.wait_limit_ns >= kAwakeNs) return true;
  const uint64_t t0 = global_timer_ns();
  while (!__all_sync(all, mbar_test_wait(bar, 0))) {
    if (__any_sync(all, global_timer_ns() - t0 > p.wait_limit_ns)) {
      ctl->abort = 1;
      if (elect_one()) atomicOr(p.status, kStatusTimeout);
      return false;
    }
  }
  return true;
}
// A wait that decides nothing: for what may still be in flight when a CTA goes away.
__device__ __forceinline__ void drain_wait(uint32_t bar, uint32_t parity) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity) && global_timer_ns() - t0 < kWaitLimitNs) {}
}

// Warp 1 of a CTA whose roles have all ended and met: if a wait gave up in any of them, its MMAs may still be in flight, also where it had issued
// all it had to. They are waited for before tensor memory is freed and the CTA goes away. Pairs: the leader's (`issuer`), and then as long
// as any copy of either CTA takes, since the peer's are counted on the leader's barriers and cannot be awaited.
template <int CTAS>
__device__ __forceinline__ void drain_after_abort(GemmControl* ctl, bool issuer) {
  if (!__any_sync(0xffffffffu, ctl->abort)) return;
  if (issuer) {
    const uint32_t lead = elect_one();                          // the lane that issued them
    if (CTAS == 2) umma_commit_pair(lead, smem_u32(&ctl->drain));
    else umma_commit(lead, smem_u32(&ctl->drain));
    drain_wait(smem_u32(&ctl->drain), 0);
  }
  if (CTAS == 2) {
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < kAbortSettleNs) {}
  }
  __syncwarp();
}

struct TileCoord {
  int mt, is_sum, ntiles, cols, brow0, unit0, nunits;
  int arow, count;   // first row of the A operand and the rows that count (set by the caller for ungrouped items)
};
// A grouped item: `count` staged rows from `row0` on, against the tiles of group_units of the r units of the one slot whose
// logits they need; the runs of one row tile follow each other.
__device__ __forceinline__ TileCoord group_coord(const GemmParams& p, int item) {
  const int tile = item / p.num_groups, first = (item - tile * p.num_groups) * p.group_units;
  const GroupTile g = p.group_tiles[tile];
  TileCoord c;
  c.mt = 0;
  c.is_sum = 0;
  c.unit0 = g.unit * p.r + first;
  c.nunits = min(p.group_units, p.r - first);
  c.cols = p.tile_cols;
  c.brow0 = c.unit0 * p.v;
  c.ntiles = (c.nunits * p.v + p.tile_cols - 1) / p.tile_cols;
  c.arow = g.row0;
  c.count = g.count;
  return c;
}
// Work items (c.mt counts M work units: m-tiles, or pairs of m-tiles in the CTA-pair kernel). Emission items come
// first, in blocks of m_block units: inside a block the unit runs fastest and
// the group next, so the CTAs that run at the same time share a few groups' weights through L2 while the block's
// hidden states (m_block x 128 rows) stay L2-resident for every group; a block is finished before the next one
// starts, so the weights are streamed from HBM once per block and the hidden states once. Sum items follow,
// m-tile fastest (ItemWalk).
__device__ __forceinline__ TileCoord tile_coord(const GemmParams& p, int item) {
  TileCoord c;
  const int emit_items = p.num_groups * p.m_units;
  int g;
  if (item < emit_items) {
    const int per_block = p.m_block * p.num_groups;
    const int blk = item / per_block;
    const int rem = item - blk * per_block;
    const int m0 = blk * p.m_block;
    const int mcount = min(p.m_block, p.m_units - m0);   // only the last block can be short
    g = rem / mcount;
    c.mt = m0 + (rem - g * mcount);
  } else {
    const int rem = item - emit_items;
    g = p.num_groups + rem / p.m_units;
    c.mt = rem % p.m_units;
  }
  c.is_sum = g >= p.num_groups;
  if (c.is_sum) {
    c.ntiles = 1;
    c.cols = p.sum_cols;
    c.brow0 = (g - p.num_groups) * p.sum_cols;
    c.unit0 = g - p.num_groups;   // index of the sum tile
    c.nunits = 0;
  } else {
    c.unit0 = g * p.group_units;
    c.nunits = min(p.group_units, p.emit_units - c.unit0);
    c.cols = p.tile_cols;
    c.brow0 = c.unit0 * p.v;
    c.ntiles = (c.nunits * p.v + p.tile_cols - 1) / p.tile_cols;
  }
  return c;
}

// A worker's items. Emission items are dealt round-robin; the workers that get none in the last round take sum tiles instead, up to
// an emission item's worth each, and what then remains is dealt round-robin to all: neighbours in time share a sum tile's weights.
// (Dealt round-robin behind the emission items, 84 sum tiles of 693 positions of a contextual 8 x 32 x 320 head made the longest
// worker 16 tiles long; 15 now, 14.2 the mean. Runs of consecutive sum tiles per worker stream all their weights at once: 4096
// positions of a 16 x 32 x 256 tree head 3349 us a draft and its acceptance instead of 3116; 3271 before.)
struct ItemWalk {
  int worker, workers, emit_items, idle, quota_end, end;
  __device__ __forceinline__ int first_sum(bool after_quota) const {
    const int j = worker - (workers - idle);                          // >= 0: a worker with no emission item in the last round
    if (!after_quota && j >= 0 && emit_items + j < min(quota_end, end)) return emit_items + j;
    return quota_end + worker;
  }
  __device__ __forceinline__ int first() const { return worker < emit_items ? worker : first_sum(false); }
  __device__ __forceinline__ int next(int item) const {
    if (item < emit_items) return item + workers < emit_items ? item + workers : first_sum(false);
    if (item >= quota_end) return item + workers;
    return item + idle < min(quota_end, end) ? item + idle : first_sum(true);
  }
};
__device__ __forceinline__ ItemWalk item_walk(const GemmParams& p, int emit_items, int sum_items, int worker, int workers) {
  const int busy = emit_items % workers;
  ItemWalk w{worker, workers, emit_items, busy ? workers - busy : 0, 0, emit_items + sum_items};
  const long long room = static_cast<long long>(w.idle) * ((p.group_units * p.v + p.tile_cols - 1) / p.tile_cols);
  w.quota_end = emit_items + (room < sum_items ? static_cast<int>(room) : sum_items);
  return w;
}

// Padding columns of a unit (vocabulary not a multiple of 16) count as logit = -inf: never the maximum, no mass.
template <int N>
__device__ __forceinline__ void mask_padding(float (&x)[N], int col_in_unit, int vv) {
  if (col_in_unit + N > vv) {
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (col_in_unit + q >= vv) x[q] = -CUDART_INF_F;
  }
}
// x[i] for an i < N that differs from lane to lane.
template <int N>
__device__ __forceinline__ float select_column(const float (&x)[N], int i) {
  float a[N / 2];
#pragma unroll
  for (int q = 0; q < N / 2; ++q) a[q] = i & (N / 2) ? x[q + N / 2] : x[q];
#pragma unroll
  for (int step = N / 4; step >= 1; step /= 2)
#pragma unroll
    for (int q = 0; q < step; ++q) a[q] = i & step ? a[q + step] : a[q];
  return a[0];
}
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void issue_batch(uint32_t taddr, uint32_t (&r)[16]) { tmem_ld16_issue(taddr, r); }
__device__ __forceinline__ void issue_batch(uint32_t taddr, uint32_t (&r)[32]) { tmem_ld32_issue(taddr, r); }
__device__ __forceinline__ void wait_batch(uint32_t (&r)[16]) { tmem_ld_wait16(r); }
__device__ __forceinline__ void wait_batch(uint32_t (&r)[32]) { tmem_ld_wait32(r); }

// log-softmax over groups of R adjacent columns inside one 16-column batch (R in {1,2,4,8,16}).
template <int R>
__device__ __forceinline__ void sum_groups_in_batch(const float (&x)[16], float* dst, int col0, int sum_rows) {
#pragma unroll
  for (int g = 0; g < 16 / R; ++g) {
    float m = x[g * R];
#pragma unroll
    for (int q = 1; q < R; ++q) m = fmaxf(m, x[g * R + q]);
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < R; ++q) s += fast_ex2((x[g * R + q] - m) * kLog2e);
    const float lse = m + fast_lg2(s) * kLn2;
    if (col0 + g * R < sum_rows) {
#pragma unroll
      for (int q = 0; q < R; ++q) dst[col0 + g * R + q] = x[g * R + q] - lse;
    }
  }
}

// CTAS = 1: every CTA works alone (cta_group::1). CTAS = 2: the kernel is launched in clusters of two CTAs that share
// every MMA (cta_group::2, M = 256): the pair covers 256 positions, each CTA stages its own 128 rows of h and HALF of the
// weight tile (the leader, cluster rank 0, the first half of the tile's columns), so a CTA moves a third less data from
// L2 to shared memory per MMA; the leader's warp 1 issues the MMAs for both, each CTA's epilogue warps read their own
// 128 accumulator rows. Barriers: full[s] lives in the leader and counts the bytes of both CTAs' copies; empty[s] and
// tfull[slot] exist in both CTAs and are signalled together by the leader's commits; tempty[slot] lives in the leader
// and collects the arrivals of both CTAs' epilogue warps.
//
// Epilogue of the log-likelihood mode: eight warps, two on each quarter of the accumulator rows, which take its batches of COLS columns in turn
// (32, or 16 where v is no multiple of 32). Each keeps a maximum, a sum and the target's logit of a unit's columns that it has seen; at the end of
// the unit the second hands its three to the first (in shared memory behind the control block, by a pair of named barriers), which adds
// them up. One warp alone issued on a fifth of the cycles: batches of 16 columns took it 600 cycles where their exponentials take
// 128, so that short K was bound by it and every call ended with 5 us of it. (8 x 16 x 320, d = 256, 4000 positions 188 us; with 32 columns,
// a maximum by halves and no branch around the target 118;
// with two warps 102. 4 x 8 x 256, d = 256, 256 positions 10.9 -> 9.0 us; 8 x 16 x 256, d = 1024, 3000 positions 161 -> 149.)
__host__ __device__ constexpr int gemm_subs(int mode) { return mode == kModeLogprob ? 2 : 1; }
__host__ __device__ constexpr int gemm_threads(int mode) { return 64 + 128 * gemm_subs(mode); }
constexpr int kExchangeBytes = 4 * 3 * 32 * 4;
template <int MODE, int CTAS, int COLS>
__global__ void __launch_bounds__(gemm_threads(MODE), 1) mtpc_gemm_kernel(const __grid_constant__ GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t tiles_addr = (raw_addr + 1023u) & ~1023u;
  uint8_t* tiles = smem_raw + (tiles_addr - raw_addr);
  GemmControl* ctl = reinterpret_cast<GemmControl*>(tiles + static_cast<size_t>(p.stages) * p.stage_bytes);

  const int warp = static_cast<int>(warp_uniform(threadIdx.x >> 5));
  const int lane = threadIdx.x & 31;
  constexpr bool kGrouped = MODE == kModeLogitsGrouped;
  constexpr int kSubs = gemm_subs(MODE);
  if (kGrouped) grid_dependency_wait();   // the tiles are read below
  static_assert(!kGrouped || CTAS == 1, "grouped tiles are ragged: no pairing");
  const int emit_items = kGrouped ? static_cast<int>(warp_uniform(*p.group_num_tiles)) * p.num_groups : p.num_groups * p.m_units;
  const uint32_t cta_rank = CTAS == 2 ? warp_uniform(cluster_cta_rank()) : 0u;      // 0 = the pair's leader
  auto coord = [&](int item) {
    if (kGrouped) return group_coord(p, item);
    TileCoord c = tile_coord(p, item);
    c.arow = (c.mt * CTAS + static_cast<int>(cta_rank)) * kBlockM;
    c.count = min(kBlockM, p.T - c.arow);                             // <= 0: a pair's second CTA past the last position
    return c;
  };
  const int worker = CTAS == 2 ? static_cast<int>(blockIdx.x >> 1) : static_cast<int>(blockIdx.x);
  const int workers = CTAS == 2 ? static_cast<int>(gridDim.x >> 1) : static_cast<int>(gridDim.x);
  const ItemWalk walk = item_walk(p, emit_items, kGrouped ? 0 : p.num_sum_tiles * p.m_units, worker, workers);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int s = 0; s < p.num_slots; ++s) {
      mbar_init(smem_u32(&ctl->tfull[s]), 1);
      mbar_init(smem_u32(&ctl->tempty[s]), 4 * CTAS * kSubs);
    }
    mbar_init(smem_u32(&ctl->drain), 1);
    ctl->abort = 0;
    ctl->wait_limit_ns = p.wait_limit_ns;
    fence_mbar_init();
    tma_prefetch_desc(&p.tm_a);
    tma_prefetch_desc(&p.tm_emit);
    tma_prefetch_desc(&p.tm_sum);
  }
  if (warp == 1) {
    if (CTAS == 2) {
      tmem_alloc_pair(smem_u32(&ctl->tmem_base), kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(&ctl->tmem_base), kTmemCols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (CTAS == 2) cluster_sync_all();   // the peer's barriers are initialised before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(ctl->tmem_base);
  grid_dependency_wait();     // barriers and tensor memory were set up while the kernel before this one finished
  grid_launch_dependents();   // (after the wait: kernels behind this one read a head's static tables early) they wait for this grid's results
  if (p.work_counter != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *p.work_counter = 0;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    const uint32_t lead = elect_one(), expects = cta_rank == 0 ? lead : 0u;
    uint32_t stage = 0, phase = 0, issued = 0;
    bool ok = true;
    const uint32_t own_full = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
    const uint32_t full0 = CTAS == 2 ? warp_uniform(cluster_map_shared(own_full, 0)) : own_full;   // the leader's barriers
    for (int item = walk.first(); item < walk.end && ok; item = walk.next(item)) {
      const TileCoord tc = coord(item);
      const CUtensorMap* tmb = tc.is_sum ? &p.tm_sum : &p.tm_emit;
      const int brows = tc.cols / CTAS;                                 // weight rows this CTA stages per tile
      const uint32_t bytes = CTAS * (kABytes + brows * (kBlockK * 2));   // of both CTAs' copies when paired
      const int arow = kGrouped ? static_cast<int>(warp_uniform(tc.arow)) : tc.arow;
      const int brow0 = kGrouped ? static_cast<int>(warp_uniform(tc.brow0)) : tc.brow0;
      for (int t = 0; t < tc.ntiles && ok; ++t) {
        const int brow = brow0 + t * tc.cols + static_cast<int>(cta_rank) * brows;
        for (int k = 0; k < p.kblocks * kBlockK; k += kBlockK) {
          if (!bounded_wait_all(empty0 + 8 * stage, phase ^ 1u, ctl, p)) { ok = false; break; }
          const uint32_t full = full0 + 8 * stage, a_dst = tiles_addr + stage * p.stage_bytes;
          mbar_arrive_expect_tx(expects, own_full + 8 * stage, bytes);
          if (CTAS == 2) {
            tma_load_2d_pair(lead, a_dst, &p.tm_a, full, k, arow);
            tma_load_2d_pair(lead, a_dst + kABytes, tmb, full, k, brow);
          } else {
            tma_load_2d(lead, a_dst, &p.tm_a, full, k, arow);
            tma_load_2d(lead, a_dst + kABytes, tmb, full, k, brow);
          }
          ++issued;
          if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
        }
      }
    }
    // The CTA must not go away with copies in flight. After a full run they have all landed already (the MMA warp
    // consumed them); after an abort, by this warp or by another one, give them a bounded chance to land.
    if (CTAS == 1 || cta_rank == 0) {
      for (uint32_t s = 0; s < static_cast<uint32_t>(p.stages) && s < issued; ++s)
        drain_wait(own_full + 8 * s, ((issued - 1 - s) / p.stages) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (cta_rank == 0) {
      const uint32_t lead = elect_one();
      uint32_t stage = 0, phase = 0, use = 0;
      bool ok = walk.first() >= walk.end || first_wait(smem_u32(&ctl->full[0]), ctl, p);
      const uint64_t a_desc0 = umma_smem_desc_sw128(tiles_addr), b_desc0 = umma_smem_desc_sw128(tiles_addr + kABytes);
      const uint32_t stage_step = p.stage_bytes >> 4, full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
      auto commit = [&](uint32_t bar) {                        // pairs: in both CTAs
        if (CTAS == 2) umma_commit_pair(lead, bar);
        else umma_commit(lead, bar);
      };
      for (int item = walk.first(); item < walk.end && ok; item = walk.next(item)) {
        const TileCoord tc = coord(item);
        const uint32_t idesc = umma_idesc_bf16(kBlockM * CTAS, tc.cols);
        for (int t = 0; t < tc.ntiles && ok; ++t, ++use) {
          const uint32_t slot = use % p.num_slots;
          if (!bounded_wait_all(smem_u32(&ctl->tempty[slot]), ((use / p.num_slots) & 1u) ^ 1u, ctl, p)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + slot * p.slot_stride;
          for (int kb = 0; kb < p.kblocks; ++kb) {
            if (!bounded_wait_all(full0 + 8 * stage, phase, ctl, p)) { ok = false; break; }
            tc_fence_after();
            const uint64_t a_desc = a_desc0 + stage * stage_step, b_desc = b_desc0 + stage * stage_step;
#pragma unroll
            for (int kk = 0; kk < kBlockK / 16; ++kk) {   // +32 bytes per K=16 step inside the swizzled row
              if (CTAS == 2) umma_bf16_pair(lead, d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
              else umma_bf16(lead, d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
            }
            commit(empty0 + 8 * stage);                   // frees the stage
            if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
          }
          if (!ok) break;
          commit(smem_u32(&ctl->tfull[slot]));            // the accumulators are ready
        }
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue
    const int quarter = warp & 3, sub = (warp - 2) >> 2;
    const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    uint32_t use = 0;
    bool ok = true;
    // a drained accumulator slot is handed back to the MMA issuer: the leader's, also from the peer's epilogue warps
    auto release_slot = [&](uint32_t slot) {
      if (CTAS == 2) mbar_arrive_cluster(cluster_map_shared(smem_u32(&ctl->tempty[slot]), 0));
      else mbar_arrive(smem_u32(&ctl->tempty[slot]));
    };
    bool handed = false;                                       // (of two warps, the second: the first has a unit's share to read)
    float* share = reinterpret_cast<float*>(ctl + 1) + quarter * 96 + lane;
    // After a wait that gave up a warp reads, stores and releases nothing more; it only meets its partner at the barriers of the units left.
    auto meet = [&](int units) {
      for (; units > 0; --units) {
        if (sub == 1) {
          if (handed) pair_sync(5 + quarter);
          pair_arrive(1 + quarter);
          handed = true;
        } else {
          pair_sync(1 + quarter);
          pair_arrive(5 + quarter);
        }
      }
    };
    for (int item = walk.first(); item < walk.end && (ok || kSubs == 2); item = walk.next(item)) {
      const TileCoord tc = coord(item);
      const int row = tc.arow + quarter * 32 + lane;
      const bool valid = quarter * 32 + lane < tc.count;
      const int nbatch = tc.cols / 16;

      if (tc.is_sum) {
        // ---- sum-unit logits -> log omega (Sec. 3.3): log-softmax over groups of r adjacent columns
        const uint32_t slot = use % p.num_slots;
        ok = ok && bounded_wait_warp(smem_u32(&ctl->tfull[slot]), (use / p.num_slots) & 1u, ctl, p.status, lane);
        if (!ok) continue;
        tc_fence_after();
        const uint32_t tcol = lane_base + slot * p.slot_stride;
        const int col_base = tc.unit0 * p.sum_cols;
        float* dst = p.logw + static_cast<size_t>(valid ? row : 0) * p.sum_rows;
        if (p.r <= 16) {
          for (int b = sub; b < nbatch; b += kSubs) {
            float x[16];
            tmem_ld16(tcol + b * 16, x);
            if (valid) {
              const int col0 = col_base + b * 16;
              if (p.sum_bias != nullptr) {
#pragma unroll
                for (int q = 0; q < 16; ++q)
                  if (col0 + q < p.sum_rows) x[q] += p.sum_bias[col0 + q];
              }
              switch (p.r) {
                case 1: sum_groups_in_batch<1>(x, dst, col0, p.sum_rows); break;
                case 2: sum_groups_in_batch<2>(x, dst, col0, p.sum_rows); break;
                case 4: sum_groups_in_batch<4>(x, dst, col0, p.sum_rows); break;
                case 8: sum_groups_in_batch<8>(x, dst, col0, p.sum_rows); break;
                default: sum_groups_in_batch<16>(x, dst, col0, p.sum_rows); break;
              }
            }
          }
        } else {
          const int bpg = p.r / 16;   // batches per group
          for (int g = sub; g < tc.cols / p.r; g += kSubs) {
            float m = -CUDART_INF_F, s = 0.f;
            const int gcol = col_base + g * p.r;
            const bool biased = p.sum_bias != nullptr && gcol < p.sum_rows;
            for (int b = 0; b < bpg; ++b) {
              float x[16];
              tmem_ld16(tcol + (g * bpg + b) * 16, x);
              if (biased) {
#pragma unroll
                for (int q = 0; q < 16; ++q) x[q] += p.sum_bias[gcol + b * 16 + q];
              }
              float bm = x[0];
#pragma unroll
              for (int q = 1; q < 16; ++q) bm = fmaxf(bm, x[q]);
              const float mn = fmaxf(m, bm);
              s *= fast_ex2((m - mn) * kLog2e);
#pragma unroll
              for (int q = 0; q < 16; ++q) s += fast_ex2((x[q] - mn) * kLog2e);
              m = mn;
            }
            const float lse = m + fast_lg2(s) * kLn2;
            for (int b = 0; b < bpg; ++b) {
              float x[16];
              tmem_ld16(tcol + (g * bpg + b) * 16, x);
              if (biased) {
#pragma unroll
                for (int q = 0; q < 16; ++q) x[q] += p.sum_bias[gcol + b * 16 + q];
              }
              if (valid && gcol < p.sum_rows) {
#pragma unroll
                for (int q = 0; q < 16; ++q) x[q] -= lse;
                // r is a multiple of 16 here, so the rows of log omega (S r floats) and this offset are 64-byte aligned
                st_global_v8(dst + gcol + b * 16, x);
                st_global_v8(dst + gcol + b * 16 + 8, x + 8);
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) release_slot(slot);
        use += 1;
        continue;
      }

      if (MODE == kModeLogitsGrouped) {
        // ---- the slot's logits and unit log-sum-exps per staged row (logit_out [rows, r v], lse_out [rows, r]): what the
        // acceptance stage needs to form the circuit's conditional of the first rejected byte
        const int k0 = tc.unit0 % p.r;                            // the item's first unit of the slot
        int col = 0, k = 0;                                       // column inside the item's nunits v columns; unit index
        float m = -CUDART_INF_F, s = 0.f;
        for (int t = 0; t < tc.ntiles && ok; ++t, ++use) {
          const uint32_t slot = use % p.num_slots;
          if (!bounded_wait_warp(smem_u32(&ctl->tfull[slot]), (use / p.num_slots) & 1u, ctl, p.status, lane)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t tcol = lane_base + slot * p.slot_stride;
          for (int b = 0; b < nbatch && k < tc.nunits; ++b) {
            float x[16];
            tmem_ld16(tcol + b * 16, x);
            mask_padding(x, col - k * p.v, p.vv);
            if (valid) {
              float* l = p.logit_out + static_cast<size_t>(row) * p.logit_pitch + k0 * p.v + col;
              st_global_v8(l, x);
              st_global_v8(l + 8, x + 8);
            }
            float bm = x[0];
#pragma unroll
            for (int q = 1; q < 16; ++q) bm = fmaxf(bm, x[q]);
            const float mn = fmaxf(m, bm);
            const float mn2 = mn * kLog2e;
            s *= fast_ex2((m - mn) * kLog2e);
#pragma unroll
            for (int q = 0; q < 16; ++q) s += fast_ex2(fmaf(x[q], kLog2e, -mn2));
            m = mn;
            col += 16;
            if (col == (k + 1) * p.v) {
              if (valid) p.lse_out[static_cast<size_t>(row) * p.r + k0 + k] = m + fast_lg2(s) * kLn2;
              ++k;
              m = -CUDART_INF_F; s = 0.f;
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) release_slot(slot);
        }
        if (!ok) break;
      } else {
        // ---- log phi at the target byte: online log-sum-exp over the v columns of each unit + gather. The
        // running (m, s) and the gathered logit live across tile boundaries; a unit is closed when its v-th
        // column has been passed. Two warps share a row (one on sorted rows, which never come here).
        static_assert(kGrouped || kSubs == 2, "a unit's columns are dealt to two warps");
        const int* tgts = (valid && p.targets != nullptr) ? p.targets + static_cast<size_t>(row) * p.n : nullptr;
        const int units_end = tc.unit0 + tc.nunits;
        int unit = tc.unit0, col_in_unit = 0;
        int slot_i = unit / p.r, k = unit - slot_i * p.r;
        float m = -CUDART_INF_F, s = 0.f, tval = 0.f;
        int tgt = tgts != nullptr ? tgts[slot_i] : -1;
        // ---- unit (slot_i, k) complete
        auto close_unit = [&] {
          if (sub == 1) {
            if (handed) pair_sync(5 + quarter);                          // the share before this one has been read
            share[0] = m;
            share[32] = s;
            share[64] = tval;
            pair_arrive(1 + quarter);
            handed = true;
          } else {
            pair_sync(1 + quarter);
            const float m2 = share[0], s2 = share[32];
            tval += share[64];                                           // (one of the two has seen the target's column)
            pair_arrive(5 + quarter);
            // the same bits whichever warp had the unit's first batch, which depends on where in an item the unit lies
            const float ref = fmaxf(m, kLowestRef), ref2 = fmaxf(m2, kLowestRef), rn = fmaxf(ref, ref2);
            s = __fadd_rn(__fmul_rn(s, fast_ex2((ref - rn) * kLog2e)), __fmul_rn(s2, fast_ex2((ref2 - rn) * kLog2e)));
            m = fmaxf(m, m2);
            // a unit that lies below the lowest reference as a whole: less than half an ulp above its maximum (-inf, NaN: NaN)
            const float lse = m >= kLowestRef ? fmaf(fast_lg2(s), kLn2, m) : fmaf(m - m, s, m);
            if (valid) {
              const size_t at = (static_cast<size_t>(row) * p.n + slot_i) * p.r + k;
              if (p.lse_out != nullptr) p.lse_out[at] = lse;
              if (tgts != nullptr) {
                p.G[at] = tgt < 0 ? 0.f : tgt >= p.vv ? CUDART_NAN_F : tval - lse;      // < 0: a marginalised byte, the input unit sums to 1
                if (tgt >= p.vv) atomicOr(p.status, kStatusBadTarget);
              }
            }
          }
          col_in_unit = 0;
          m = -CUDART_INF_F; s = 0.f; tval = 0.f;
          if (++unit < units_end && ++k == p.r) {
            k = 0;
            ++slot_i;
            if (tgts != nullptr) tgt = tgts[slot_i];
          }
        };
        // past one batch of columns, whoever's it was; false once the item's last unit has been closed
        auto pass_batch = [&]() -> bool {
          col_in_unit += COLS;
          if (col_in_unit != p.v) return true;
          close_unit();
          return unit < units_end;
        };
        for (int t = 0; t < tc.ntiles; ++t, ++use) {
          const uint32_t slot = use % p.num_slots;
          ok = ok && bounded_wait_warp(smem_u32(&ctl->tfull[slot]), (use / p.num_slots) & 1u, ctl, p.status, lane);
          if (!ok) {
            meet(units_end - unit);
            break;
          }
          tc_fence_after();
          const uint32_t tcol = lane_base + slot * p.slot_stride;
          // one batch of accumulator columns of this row
          auto consume = [&](const uint32_t (&raw)[COLS], int b) {
            float x[COLS];
#pragma unroll
            for (int q = 0; q < COLS; ++q) x[q] = __uint_as_float(raw[q]);
            mask_padding(x, col_in_unit, p.vv);
            if (p.logit_out != nullptr) {                                // row of W_emit = column of the logit matrix
              float* l = p.logit_out + static_cast<size_t>(row) * p.logit_pitch + tc.brow0 + t * tc.cols + b * COLS;
              if (valid) {
#pragma unroll
                for (int q = 0; q < COLS; q += 8) st_global_v8(l + q, x + q);   // 64-byte aligned: v and the tile widths are multiples of 16
              }
            }
            float bm[COLS / 2];
#pragma unroll
            for (int q = 0; q < COLS / 2; ++q) bm[q] = fmaxf(x[q], x[q + COLS / 2]);
#pragma unroll
            for (int step = COLS / 4; step >= 1; step /= 2)
#pragma unroll
              for (int q = 0; q < step; ++q) bm[q] = fmaxf(bm[q], bm[q + step]);
            const float ref = fmaxf(m, kLowestRef);
            m = fmaxf(m, bm[0]);
            const float rn = fmaxf(m, kLowestRef);
            const float2 l2 = make_float2(kLog2e, kLog2e), nr = make_float2(-rn * kLog2e, -rn * kLog2e);
            float2 sa = make_float2(s * fast_ex2((ref - rn) * kLog2e), 0.f), sb = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = 0; q < COLS; q += 2) {
              const float2 y = __ffma2_rn(make_float2(x[q], x[q + 1]), l2, nr);
              const float2 e = make_float2(fast_ex2(y.x), fast_ex2(y.y));
              if (q & 2) sb = __fadd2_rn(sb, e);
              else sa = __fadd2_rn(sa, e);
            }
            s = (sa.x + sa.y) + (sb.x + sb.y);
            const int rel = tgt - col_in_unit;
            const float at_rel = select_column(x, rel);                  // (a branch around it costs more than it saves)
            tval = static_cast<unsigned>(rel) < COLS ? at_rel : tval;
          };
          // this warp's batch b and the ones that it passes on the way
          auto take = [&](const uint32_t (&raw)[COLS], int b) -> bool {
            if (sub == 1 && !pass_batch()) return false;
            consume(raw, b);
            if (!pass_batch()) return false;
            return sub == 1 || pass_batch();
          };
          // The load of the next batch is in flight while this one goes through the exponentials (two register buffers).
          const int batches = tc.cols / COLS;
          uint32_t ra[COLS], rb[COLS];
          issue_batch(tcol + sub * COLS, ra);
          wait_batch(ra);
          for (int b = sub;;) {
            const bool more_b = b + kSubs < batches;
            if (more_b) issue_batch(tcol + (b + kSubs) * COLS, rb);
            const bool go_a = take(ra, b);
            if (more_b) wait_batch(rb);
            if (!go_a || !more_b) break;
            b += kSubs;
            const bool more_a = b + kSubs < batches;
            if (more_a) issue_batch(tcol + (b + kSubs) * COLS, ra);
            const bool go_b = take(rb, b);
            if (more_a) wait_batch(ra);
            if (!go_b || !more_a) break;
            b += kSubs;
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) release_slot(slot);
        }
      }
    }
    if (handed) pair_sync(5 + quarter);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) drain_after_abort<CTAS>(ctl, cta_rank == 0);
  if (CTAS == 2) {
    // A CTA of a pair may leave only when its partner no longer needs it (MMAs read both CTAs' shared memory and write
    // both CTAs' tensor memory; copies and arrivals cross over).
    __syncthreads();      // every warp converged again before the cluster-wide barrier
    cluster_sync_all();
  }
  if (warp == 1) {
    tc_fence_after();
    if (CTAS == 2) tmem_dealloc_pair(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

}  // namespace mtpc
