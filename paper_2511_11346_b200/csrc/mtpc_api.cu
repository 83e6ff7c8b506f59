// Host side of the C ABI declared in include/mtpc.h: argument checks, workspace carving, TMA descriptor
// encoding and kernel launches. Every step of the path runs in the kernels of this library; there is no CPU
// or library fallback.
#include <cuda.h>
#include <cuda_runtime.h>
#include <initializer_list>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <new>

#include "../../include/mtpc.h"
#include "mtpc_backward.cuh"
#include "mtpc_circuit.cuh"
#include "mtpc_decode.cuh"
#include "mtpc_gemm.cuh"
#include "mtpc_lowrank.cuh"
#include "mtpc_lowrank_gemm.cuh"

namespace {

using namespace mtpc;

constexpr size_t kAlign = 256;
constexpr int kMaxPhases = 5;
constexpr size_t kSlotSmemLimit = 160 * 1024;   // latent-draw tables of the draft slot kernel kept in shared memory up to this
constexpr size_t kSlotSmemPair = 112 * 1024;     // two of its CTAs share an SM up to this
constexpr int kMaxDraftVocab = 512;     // symbols a warp draws from in one go
constexpr int kHostChunkPositions = 512;    // the smallest piece a host-buffer call is uploaded and processed in
constexpr int kMaxHostChunks = 64;
constexpr int kWorkCounterWord = 16;   // word of the 256-byte status area used as the circuit kernels' work counter
constexpr int kSmemLimit = 232448;   // 227 KB of dynamic shared memory per CTA on sm_100
// Hidden states of one rasterisation block of the projection kernel: small enough to stay L2-resident next to the
// weight tiles streaming past (data read by all SMs ends up in both halves of the 126 MB L2).
constexpr size_t kHiddenBlockBytes = 36u << 20;
// Drafts of more positions than the few-position path takes keep the emission logits of their positions (the byte draws, the
// evidence and the acceptance stage are then gathers), at most this much of them: longer drafts run in chunks of positions,
// and their acceptance stage recomputes the logits it needs.
constexpr size_t kKeptLogitBytes = static_cast<size_t>(4) << 30;
// ... from hidden states staged by slot, this much at a time.
constexpr size_t kGroupStageBytes = 1u << 30;

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }
bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

// How one launch of the projection kernel tiles the N axis and uses shared / tensor memory.
struct Tiling {
  int tile_cols;        // accumulator width of an emission tile
  int slot_stride, num_slots, stages, stage_bytes, smem;
  int pair_stages, pair_stage_bytes, pair_smem;   // the same ring when two CTAs share every MMA (half a weight tile per CTA)
};

struct Layout {
  // derived sizes
  int S, sum_rows, sum_cols, sum_tiles;
  Tiling lp;            // 256-column tiles over the flattened (i,k,b) axis
  size_t max_windows;
  // workspace offsets (bytes)
  size_t off_status, off_wemit, off_wsum, off_hidden, off_logA, off_probA, off_cdfA, off_G, off_logw, off_sel, off_logits, off_unit_lse;
  size_t off_prefix, off_partial, off_sum_bias;   // training loss: prefix log-marginals [max_positions, n], per-sequence terms
  size_t off_msg;       // slot messages of the drafted windows [max_windows, n, r], kept for the acceptance stage
  int decode_max_p;     // positions the few-position draft path can take
  int kept_p;           // positions whose logits a longer draft can keep at once (0: no longer drafts)
  size_t off_h_hidden, off_h_targets, off_h_uniforms, off_h_bytes, off_h_out;
  // acceptance stage after a draft that did not keep its logits: windows that can be staged at once (0: not needed)
  size_t group_entries;
  size_t off_grp_ints, off_grp_tiles, off_grp_stage;
  // ... first rejected slot and staging row per window, the recomputed logits [accept_rows, r v] and unit log-sum-exps
  // [accept_rows, r] of that slot (a factored head forms them after every long draft)
  size_t accept_rows;     // windows that can be handled at once (0: not available)
  size_t off_acc_rej, off_acc_row, off_acc_logits, off_acc_lse;
  size_t total;
};


// Shared-memory ring and TMEM slots for tiles of `tile_cols` emission columns and `sum_cols` sum columns.
bool fit_tiling(Tiling* t, int sum_cols) {
  const int widest = t->tile_cols > sum_cols ? t->tile_cols : sum_cols;
  t->slot_stride = (widest + 31) / 32 * 32;
  t->num_slots = kTmemCols / t->slot_stride;
  if (t->num_slots > kMaxSlots) t->num_slots = kMaxSlots;
  t->stage_bytes = (kABytes + widest * kBlockK * 2 + 1023) / 1024 * 1024;   // A tile + one B tile
  const int ctl = 1024 + static_cast<int>(sizeof(GemmControl)) + kExchangeBytes;
  int stages = (kSmemLimit - ctl) / t->stage_bytes;
  if (stages > kMaxStages) stages = kMaxStages;
  t->stages = stages;
  t->smem = stages * t->stage_bytes + ctl;
  t->pair_stage_bytes = (kABytes + widest / 2 * kBlockK * 2 + 1023) / 1024 * 1024;   // A tile + half a B tile
  t->pair_stages = (kSmemLimit - ctl) / t->pair_stage_bytes;
  if (t->pair_stages > kMaxStages) t->pair_stages = kMaxStages;
  t->pair_smem = t->pair_stages * t->pair_stage_bytes + ctl;
  return stages >= 2 && t->num_slots >= 2;
}

// factored: the head keeps low-rank unembeddings factored (its long drafts take another route).
int plan(const mtpc_config& c, Layout* L, bool factored = false) {
  if (c.family < MTPC_CP || c.family > MTPC_BTREE) return MTPC_ERR_SHAPE;
  if (c.io_dtype != MTPC_F32 && c.io_dtype != MTPC_BF16) return MTPC_ERR_SHAPE;
  if (c.n < 1 || c.r < 1 || c.v < 1 || c.d < 1 || c.max_positions < 1 || c.max_windows_per_pos < 1)
    return MTPC_ERR_SHAPE;
  if ((c.flags & ~(MTPC_FLAG_HMM_CONTEXTUAL | MTPC_FLAG_SHORT_DRAFTS)) != 0) return MTPC_ERR_UNSUPPORTED;
  const bool ctx = (c.flags & MTPC_FLAG_HMM_CONTEXTUAL) != 0;
  if (ctx && c.family != MTPC_HMM) return MTPC_ERR_UNSUPPORTED;
  if (c.n > 64 || c.max_windows_per_pos > 64) return MTPC_ERR_UNSUPPORTED;
  if (!is_pow2(c.r) || c.r > 128) return MTPC_ERR_UNSUPPORTED;
  if (c.family != MTPC_CP && c.r > 32) return MTPC_ERR_UNSUPPORTED;
  if (c.family == MTPC_BTREE && (c.n < 2 || !is_pow2(c.n))) return MTPC_ERR_UNSUPPORTED;
  if (c.d % kBlockK != 0) return MTPC_ERR_UNSUPPORTED;
  if (c.v % 16 != 0) return MTPC_ERR_UNSUPPORTED;
  if (c.v_valid != 0 && (c.v_valid > c.v || c.v_valid <= c.v - 16)) return MTPC_ERR_SHAPE;
  if (static_cast<int64_t>(c.n) * c.r * c.v > (1ll << 30)) return MTPC_ERR_SHAPE;

  L->S = (c.family == MTPC_BTREE) ? 1 + (c.n - 2) * c.r : (ctx ? 1 + (c.n - 1) * c.r : 1);
  L->sum_rows = L->S * c.r;
  // sum tile: a multiple of both r and 16, at most 256 columns
  const int unit = c.r > 16 ? c.r : 16;
  int sum_cols = (L->sum_rows + unit - 1) / unit * unit;
  if (sum_cols > 256) sum_cols = 256 / unit * unit;
  L->sum_cols = sum_cols;
  L->sum_tiles = (L->sum_rows + sum_cols - 1) / sum_cols;
  const int emit_units = c.n * c.r;
  L->lp.tile_cols = 256;
  if (!fit_tiling(&L->lp, sum_cols)) return MTPC_ERR_UNSUPPORTED;

  L->decode_max_p = c.max_positions < kDecodeMaxP ? c.max_positions : kDecodeMaxP;
  const bool long_drafts = c.max_positions > L->decode_max_p && (c.flags & MTPC_FLAG_SHORT_DRAFTS) == 0;
  L->max_windows = static_cast<size_t>(long_drafts ? c.max_positions : L->decode_max_p) * c.max_windows_per_pos;
  if (L->max_windows < static_cast<size_t>(c.max_positions)) L->max_windows = c.max_positions;   // an evaluation's
  const size_t elt = c.io_dtype == MTPC_F32 ? 4 : 2;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes); return o; };
  L->off_status = take(256);
  const bool f32 = c.io_dtype == MTPC_F32;
  L->off_wemit = take(f32 ? static_cast<size_t>(c.n) * c.r * c.v * c.d * 2 : 0);
  L->off_wsum = take(f32 ? static_cast<size_t>(L->sum_rows) * c.d * 2 : 0);
  L->off_hidden = take(f32 ? static_cast<size_t>(c.max_positions) * c.d * 2 : 0);
  L->off_logA = take(c.family == MTPC_HMM && !ctx ? static_cast<size_t>(c.n - 1) * c.r * c.r * 4 : 0);
  L->off_probA = take(c.family == MTPC_HMM && !ctx ? static_cast<size_t>(c.n - 1) * c.r * c.r * 4 : 0);
  L->off_cdfA = take(c.family == MTPC_HMM && !ctx ? static_cast<size_t>(c.n - 1) * c.r * c.r * 4 : 0);
  L->off_sum_bias = take(ctx ? static_cast<size_t>(L->sum_rows) * 4 : 0);
  L->off_G = take(L->max_windows * c.n * c.r * 4);
  L->off_logw = take(static_cast<size_t>(c.max_positions) * L->sum_rows * 4);
  L->off_sel = take(L->max_windows * c.n * 4);
  L->off_msg = take(L->max_windows * c.n * c.r * 4);
  // (latents of more than 32 values are handled for the mixture only; HMM and BTree are limited to r <= 32 anyway)
  L->kept_p = 0;
  if (long_drafts && !factored) {
    const size_t cap = kKeptLogitBytes / (static_cast<size_t>(emit_units) * c.v * 4);     // >= 1: n r v <= 2^30
    L->kept_p = static_cast<size_t>(c.max_positions) < cap ? c.max_positions : static_cast<int>(cap);
  }
  const size_t logit_rows = L->kept_p > L->decode_max_p ? L->kept_p : L->decode_max_p;
  L->off_logits = take(logit_rows * emit_units * c.v * 4);
  L->off_unit_lse = take(logit_rows * emit_units * 4);
  L->off_prefix = take(static_cast<size_t>(c.max_positions) * c.n * 4);
  L->off_partial = take(static_cast<size_t>(c.max_positions) * c.n * 4);
  L->off_h_hidden = take(static_cast<size_t>(c.max_positions) * c.d * elt);
  L->off_h_targets = take(static_cast<size_t>(c.max_positions) * c.n * 4);
  L->off_h_uniforms = take(L->max_windows * 2 * c.n * 4);
  L->off_h_bytes = take(L->max_windows * c.n * 4);
  L->off_h_out = take(L->max_windows * 4);
  L->group_entries = 0;
  L->accept_rows = 0;
  if (long_drafts && L->kept_p < c.max_positions) {
    const size_t stage_cap = kGroupStageBytes / (static_cast<size_t>(c.d) * 2);
    const size_t row_cap = kGroupStageBytes / (static_cast<size_t>(c.r) * c.v * 4);
    L->accept_rows = L->max_windows < row_cap ? L->max_windows : row_cap;
    if (!factored && L->accept_rows > stage_cap) L->accept_rows = stage_cap;        // they share the staging rows
    if (L->accept_rows < static_cast<size_t>(c.max_windows_per_pos)) L->accept_rows = 0;   // not even one position
    if (!factored) L->group_entries = L->accept_rows;
  }
  const size_t ge = L->group_entries, ar = L->accept_rows;
  L->off_grp_ints = take(ge ? (3 * static_cast<size_t>(c.n) + 64) * 4 : 0);            // counts | cursors | offsets | tile count
  L->off_grp_tiles = take(ge ? (c.n + ge / 128 + 1) * sizeof(GroupTile) : 0);
  L->off_grp_stage = take(ge * c.d * 2);
  L->off_acc_rej = take(ar ? L->max_windows * 4 : 0);
  L->off_acc_row = take(ar ? L->max_windows * 4 : 0);
  L->off_acc_logits = take(ar * c.r * c.v * 4);
  L->off_acc_lse = take(ar * c.r * 4);
  L->total = off;
  return MTPC_OK;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// bf16 matrix [rows, cols] row-major (row pitch `pitch` elements, 0 = cols) -> tiles of box_rows x 64 elements,
// 128-byte swizzle, zero fill outside.
int make_tmap(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, uint64_t pitch = 0) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return MTPC_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0) return MTPC_ERR_WORKSPACE;
  if (pitch == 0) pitch = cols;
  if ((pitch * 2) % 16 != 0) return MTPC_ERR_WORKSPACE;
  cuuint64_t gdim[2] = {cols, rows};
  cuuint64_t gstride[1] = {pitch * 2};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(kBlockK), box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MTPC_OK : MTPC_ERR_CUDA;
}

// bf16 array [rows][units][v] (row pitch `pitch` elements) written in boxes of 32 rows x 64 columns of one unit, 128-byte swizzle: what lies
// past the unit's v columns is not written.
int make_tmap_unit_rows(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t units, uint64_t v, uint64_t pitch) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return MTPC_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0 || (pitch * 2) % 16 != 0 || (v * 2) % 16 != 0) return MTPC_ERR_WORKSPACE;
  cuuint64_t gdim[3] = {v, units, rows};
  cuuint64_t gstride[2] = {v * 2, pitch * 2};
  cuuint32_t box[3] = {64, 1, 32};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), gdim, gstride, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MTPC_OK : MTPC_ERR_CUDA;
}

// bf16 matrix [rows, cols] row-major read as an MN-major operand (its columns are the operand's M or N index, its rows
// the K index): boxes of 64 columns x 64 rows, 128-byte swizzle, zero fill outside.
int make_tmap_mn(CUtensorMap* tm, const void* base, uint64_t rows, uint64_t cols, uint64_t pitch) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return MTPC_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0 || (pitch * 2) % 16 != 0) return MTPC_ERR_WORKSPACE;
  cuuint64_t gdim[2] = {cols, rows};
  cuuint64_t gstride[1] = {pitch * 2};
  cuuint32_t box[2] = {64, static_cast<cuuint32_t>(kBlockK)};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MTPC_OK : MTPC_ERR_CUDA;
}

}  // namespace

struct mtpc_head {
  mtpc_config cfg;
  Layout L;
  uint8_t* ws;
  const void* W_emit_bf16;
  const void* W_sum_bf16;
  CUtensorMap tm_emit_lp, tm_sum;               // W_emit, W_sum
  CUtensorMap tm_emit_lp2, tm_sum2;             // the same with boxes of half the rows: what one CTA of a pair stages
  int projection_variant;                       // 0: chosen per launch; 1: every CTA alone; 2: CTA pairs (cta_group::2)
  // factored low-rank head (App. G; mtpc_create_head_lowrank): rank k > 0, no composed W_emit
  int lr_k;
  const void* lr_W_base;                        // [n, v, d] bf16
  const void* lr_A;                             // [n, r, v, k] bf16
  const void* lr_B;                             // [n, r, k, d] bf16
  size_t lr_off_arep;                           // workspace: A as [n, v, r, k]
  size_t lr_off_dec;                            // workspace: few-position draft products base [P, n v] | z [P, n r k]
  size_t lr_off_base;                           // workspace: W_base h [T, n v] fp32
  size_t lr_off_split;                          // workspace: parts of split plain GEMMs ...
  int lr_split_parts;                           // ... and how many there is room for
  CUtensorMap tm_lrB_dec;                       // B [n r k, d] for the few-position draft path
  size_t lr_off_zhl, lr_off_partial;            // workspace: z = B h as bf16 halves [T, n r, 2, k]; partial log-sum-exps per column block
  CUtensorMap lr_tm_a;                          // the copy of A in the boxes of the factored projection
  LowRankParams lr_params;                      // everything of the factored projection launch that does not depend on the call
  int max_pairs;                                // clusters of two projection CTAs that can be resident at once
  CUtensorMap tm_emit_dec, tm_sum_dec;          // the same matrices in the few-position draft path's tiles
  int decode_tile_rows, decode_sum_tile_rows;
  int decode_ksplit;                            // CTAs that share a tile of it, each with its part of K
  int max_decode_clusters[3];                   // clusters of 2, 4, 8 of its CTAs that can be resident at once
  int num_sms;
  cudaStream_t copy_stream; // host-buffer calls: uploads run here, ahead of the kernels (created on first use)
  cudaEvent_t* copy_events; // [copy_event_count]: "chunk c is on the device"; the one after the last chunk's: "the uploads may start"
  int copy_event_count;
  int draft_P;              // positions whose draft state (logits, or after a many-position draft G and log omega) is in the workspace (0: none)
  int draft_wpp;            // windows per position of that draft
  bool draft_msg;           // its slot messages are there too (a draft of prefix marginals leaves them, an acceptance call forms them)
  unsigned long long draft_capture;   // ... enqueued in this stream capture (0: none)
  bool joint_recorded;      // a draft of joints, which leaves no messages, may be replayed at any time
  bool draft_logits;        // every logit and unit log-sum-exp of its positions is there as well
  const void* draft_hidden; // the bf16 hidden states it read (the acceptance stage may have to stage rows of them)
  int ring;                 // calls whose per-kernel events are retained (0 = timing off)
  cudaEvent_t* ev;          // [ring][kMaxPhases][2]
  int* ring_phases;         // [ring] phases recorded by the call in that slot
  uint64_t calls;           // timed calls so far
  uint64_t launches;
  uint64_t wait_limit_ns;   // limit of the pipeline waits inside the tcgen05 kernels (kWaitLimitNs; a test may shorten it)
};

namespace {

template <typename T>
T* at(mtpc_head* h, size_t off) { return reinterpret_cast<T*>(h->ws + off); }

int valid_symbols(const mtpc_config& c) { return c.v_valid > 0 ? c.v_valid : c.v; }
bool is_ctx(const mtpc_head* h) { return (h->cfg.flags & MTPC_FLAG_HMM_CONTEXTUAL) != 0; }
// HMM transition log-probabilities as the kernels read them: position p's tables start at base + p * stride.
// Static transitions: one set in the workspace, stride 0. Contextual (App. H): the sum units after the first one
// in every position's row of log omega.
const float* hmm_tables(mtpc_head* h) {
  return is_ctx(h) ? at<float>(h, h->L.off_logw) + h->cfg.r : at<float>(h, h->L.off_logA);
}
int hmm_table_stride(const mtpc_head* h) { return is_ctx(h) ? h->L.sum_rows : 0; }
const float* sum_bias(mtpc_head* h) { return is_ctx(h) ? at<float>(h, h->L.off_sum_bias) : nullptr; }

struct PhaseTimer {
  mtpc_head* h;
  cudaStream_t st;
  int idx, slot;
  PhaseTimer(mtpc_head* head, cudaStream_t s) : h(head), st(s), idx(0), slot(0) {
    if (h->ring > 0) {
      slot = static_cast<int>(h->calls % h->ring);
      h->ring_phases[slot] = 0;
      h->calls++;
    }
  }
  cudaEvent_t* pair() { return h->ev + (static_cast<size_t>(slot) * kMaxPhases + idx) * 2; }
  void begin() { if (h->ring > 0 && idx < kMaxPhases) cudaEventRecord(pair()[0], st); }
  void end() {
    if (h->ring > 0 && idx < kMaxPhases) {
      cudaEventRecord(pair()[1], st);
      h->ring_phases[slot] = idx + 1;
    }
    ++idx;
  }
};

int check_launch() { return cudaGetLastError() == cudaSuccess ? MTPC_OK : MTPC_ERR_CUDA; }

// Launch `kernel`, optionally allowed to start before the kernel ahead of it in the stream has finished (programmatic
// dependent launch): such a kernel calls grid_dependency_wait() before it touches global memory, so what overlaps is its launch and
// set-up (about 2 us a kernel). cluster > 1: in clusters of that many CTAs.
// Five kernels do more before they wait. A kernel that lets its dependents in after its own wait (a gate) has nothing unfinished ahead of
// it, so whatever was launched before it has ended when anything behind it starts; each of the five relies on one:
//   draft_slot_kernel, circuit_hmm_kernel and the static HMM's Eq. 6 kernel copy the head's static tables. The tables are written by a plain
//     launch (bind_parameters), and the first kernel of every call that runs one of the three is a gate (the fp32 conversion, the projection,
//     the weight pass; an acceptance call, whose first kernel may be circuit_hmm_kernel, needs a draft since the last update).
//   loss_coeff_kernel reads the targets and writes the coefficients. The projection it is launched behind is a gate (on a factored head the
//     merge), so the caller's writes and the readers of the last call's coefficients are done.
//   loss_partial_kernel, beside the last GEMM, reads the prefixes and writes its partial sums. The GEMMs are NOT gates, they let their
//     dependents in before they wait. What lies between them and the circuit is: logit_gradient_kernel, by its plain launch, or on a factored
//     head lowrank_pad_kernel. Whoever makes the one a dependent or lets the other's dependents in early breaks the loss.
template <typename... Params, typename... Args>
void launch_clusters(void (*kernel)(Params...), int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool dependent,
                     Args&&... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (dependent) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <typename... Params, typename... Args>
void launch_kernel(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool dependent, Args&&... args) {
  launch_clusters(kernel, 1, grid, block, smem, st, dependent, args...);
}
// The kernels of a call follow each other as dependents, unless events are recorded between them.
bool overlapped(const mtpc_head* h) { return h->ring == 0; }

// Units per work item of the log-likelihood mode. An item covers its units with 256-column tiles; unless the
// units end on a tile boundary the last tile is partly wasted (its tail belongs to the next item, which recomputes it).
// Items are dealt round-robin to `ctas` persistent CTAs and the launch's sum tiles fill the last round (ItemWalk), so a launch
// takes about rounds x tiles-per-item tile times and the share of the sum tiles that the last round has no room for:
// pick the count that minimises that (v = 320: 4 units = 5 tiles, nothing wasted; v = 272: 8 units = 9 tiles, 6 % wasted
// but twice as many items as the waste-free 16 units = 17 tiles).
struct ItemPlan {
  int units = 1;             // per item
  long long tiles = 0;       // tile times of the launch
};
ItemPlan choose_group_units(int v, int emit_units, int m_tiles, int ctas, int sum_tiles) {
  ItemPlan best;
  const long long sums = static_cast<long long>(sum_tiles) * m_tiles;
  if (emit_units == 0) best.tiles = (sums + ctas - 1) / ctas;
  const int limit = emit_units < 64 ? emit_units : 64;
  for (int u = 1; u <= limit; ++u) {
    const int tiles = (u * v + 255) / 256;
    const long long items = static_cast<long long>((emit_units + u - 1) / u) * m_tiles;
    const long long rounds = (items + ctas - 1) / ctas;
    const long long rest = sums - (rounds * ctas - items) * tiles;
    const long long cost = rounds * tiles + (rest > 0 ? (rest + ctas - 1) / ctas : 0);
    if (u == 1 || cost < best.tiles) { best.tiles = cost; best.units = u; }
    if (rounds == 1 && rest <= 0) break;                              // longer items only make the one round longer
  }
  return best;
}

struct GroupArgs {           // rows sorted by slot: the staged hidden states and their tiles (mtpc_group.cuh)
  const void* stage = nullptr;
  int entries = 0;                           // rows of the staging buffer in use
  const GroupTile* tiles = nullptr;
  const int* num_tiles = nullptr;
  int max_tiles = 0;
};

struct GradArgs {            // what the projection kernel keeps for the backward pass or a draft
  float* lse_out = nullptr;                  // the units' log-sum-exps [T, n, r]
  float* logit_out = nullptr;                // the emission logits [T, n r v] fp32
  size_t logit_pitch = 0;
};

// Launch the projection kernel for `rows` positions over the emission groups (with_emit) and / or the sum tiles.
// first_row: where in log omega the launch's positions start (a draft that runs in chunks of positions).
int launch_gemm(mtpc_head* h, const void* hidden_bf16, int rows, bool with_emit, bool with_sum, const int* targets, cudaStream_t st,
                const GradArgs* ga = nullptr, const GroupArgs* grp = nullptr, int first_row = 0) {
  if (rows <= 0 || (!with_emit && !with_sum)) return MTPC_OK;
  const mtpc_config& c = h->cfg;
  const Layout& L = h->L;
  const Tiling& tl = L.lp;
  GemmParams p;
  memset(&p, 0, sizeof(p));
  if (ga) {
    p.lse_out = ga->lse_out;
    p.logit_out = ga->logit_out;
    p.logit_pitch = ga->logit_pitch;
  }
  int rc = grp ? make_tmap(&p.tm_a, grp->stage, static_cast<uint64_t>(grp->entries), static_cast<uint64_t>(c.d), kBlockM)
               : make_tmap(&p.tm_a, hidden_bf16, static_cast<uint64_t>(rows), static_cast<uint64_t>(c.d), kBlockM);
  if (rc != MTPC_OK) return rc;
  p.T = rows;
  p.m_tiles = (rows + kBlockM - 1) / kBlockM;
  // Every CTA alone, or two CTAs per MMA (when there are two m-tiles to pair up and the device can hold a cluster at all): whichever
  // plan takes less time. A pair moves less operand data per MMA, which counts when K is long; with few K steps the epilogue bounds
  // a tile, and a lone CTA need not wait for its partner's. Whole calls in pairs / alone over 256 to 4000 positions of 8 x 16 x 320,
  // 4 x 8 x 256 and 8 x 8 x 272 heads: d = 256 1.09 to 1.19, d = 512 1.08 to 1.32, d = 1024 0.96 to 1.11, d = 1280 0.94 to 1.15, d = 1536
  // 0.97 to 1.17, d = 2048 0.97 to 1.08, d = 4096 0.93 to 1.08 (above 1 there where a CTA has one or two tiles). A ragged
  // number of m-tiles costs the pairs more tiles (384 positions, d = 4096, 8 x 16 x 320: 5 a pair against 4, 150 us / 138).
  const int emit_units = with_emit ? c.n * c.r : 0, launch_sums = with_sum ? L.sum_tiles : 0;
  bool pair = grp == nullptr && h->projection_variant == 2;
  ItemPlan plan;
  if (grp == nullptr) {
    plan = choose_group_units(c.v, emit_units, p.m_tiles, h->num_sms, launch_sums);
    if (h->projection_variant != 1 && h->max_pairs > 0) {
      const ItemPlan two = choose_group_units(c.v, emit_units, (p.m_tiles + 1) / 2, h->max_pairs, launch_sums);
      if (h->projection_variant == 0 && p.m_tiles >= 2)       // (sum tiles of few columns: an MMA of a pair takes twice as long as a lone CTA's, see below)
        pair = !with_emit && L.sum_cols <= 64 ? false
               : c.d < 1536 ? two.tiles * 34 <= plan.tiles * 33 : two.tiles * 12 <= plan.tiles * 13;
      if (pair) plan = two;
    }
  }
  const int ctas = pair ? 2 : 1;
  const int workers = pair ? h->max_pairs : h->num_sms;               // CTAs, or CTA pairs, resident at once
  p.m_units = (p.m_tiles + ctas - 1) / ctas;
  p.kblocks = c.d / kBlockK;
  {
    const size_t unit_bytes = static_cast<size_t>(kBlockM) * ctas * c.d * 2;
    const int cap_units = kHiddenBlockBytes / unit_bytes > 0 ? static_cast<int>(kHiddenBlockBytes / unit_bytes) : 1;
    const int nblocks = (p.m_units + cap_units - 1) / cap_units;
    p.m_block = (p.m_units + nblocks - 1) / nblocks;
  }
  p.n = c.n; p.r = c.r; p.v = c.v;
  p.vv = valid_symbols(c);
  p.emit_units = c.n * c.r;
  p.group_units = plan.units;
  if (grp != nullptr) p.group_units = choose_group_units(c.v, c.r, grp->max_tiles, workers, 0).units;   // runs of a row tile's r units
  p.num_groups = grp != nullptr ? (c.r + p.group_units - 1) / p.group_units : (emit_units + p.group_units - 1) / p.group_units;
  p.tile_cols = tl.tile_cols;
  p.num_sum_tiles = with_sum ? L.sum_tiles : 0;
  p.sum_cols = L.sum_cols;
  p.sum_rows = L.sum_rows;
  p.slot_stride = tl.slot_stride;
  p.num_slots = tl.num_slots;
  p.stages = pair ? tl.pair_stages : tl.stages;
  p.stage_bytes = pair ? tl.pair_stage_bytes : tl.stage_bytes;
  size_t smem = pair ? tl.pair_smem : tl.smem;
  if (!with_emit) {
    // sum tiles alone (a factored head): narrower stages, more of them. 32 columns, d = 4096, under ncu: 1000 positions 22.4 us in pairs, 15.4 so,
    // 8192 positions 23.1 and 18.7.
    const int ctl = static_cast<int>(smem) - p.stages * p.stage_bytes;
    p.stage_bytes = (kABytes + L.sum_cols / ctas * kBlockK * 2 + 1023) / 1024 * 1024;
    p.stages = (kSmemLimit - ctl) / p.stage_bytes;
    if (p.stages > kMaxStages) p.stages = kMaxStages;
    smem = p.stages * p.stage_bytes + ctl;
  }
  p.tm_emit = pair ? h->tm_emit_lp2 : h->tm_emit_lp;
  p.tm_sum = pair ? h->tm_sum2 : h->tm_sum;
  p.targets = targets;
  p.G = at<float>(h, L.off_G);
  p.logw = at<float>(h, L.off_logw) + static_cast<size_t>(first_row) * L.sum_rows;
  p.sum_bias = sum_bias(h);
  if (grp) {
    p.group_tiles = grp->tiles;
    p.group_num_tiles = grp->num_tiles;
  }
  p.status = at<unsigned>(h, L.off_status);
  p.wait_limit_ns = h->wait_limit_ns;
  const long long items = grp ? static_cast<long long>(grp->max_tiles) * p.num_groups
                              : static_cast<long long>(p.m_units) * (p.num_groups + p.num_sum_tiles);
  const int grid = ctas * static_cast<int>(items < workers ? items : workers);
  p.work_counter = with_sum ? p.status + kWorkCounterWord : nullptr;    // (the first launch of every call that needs it zeroed)
  if (grp) launch_kernel(mtpc_gemm_kernel<kModeLogitsGrouped, 1, 16>, grid, gemm_threads(kModeLogitsGrouped), smem, st, overlapped(h), p);
  else if (!pair) launch_kernel(c.v % 32 == 0 ? mtpc_gemm_kernel<kModeLogprob, 1, 32> : mtpc_gemm_kernel<kModeLogprob, 1, 16>, grid, gemm_threads(kModeLogprob), smem, st, overlapped(h), p);
  else launch_clusters(c.v % 32 == 0 ? mtpc_gemm_kernel<kModeLogprob, 2, 32> : mtpc_gemm_kernel<kModeLogprob, 2, 16>, 2, grid, gemm_threads(kModeLogprob), smem, st, overlapped(h), p);
  h->launches++;
  return check_launch();
}

size_t btree_smem_bytes(int n, int r) { return static_cast<size_t>(kCircuitWarps) * btree_warp_floats(n, r) * sizeof(float); }

// CTAs that persistent kernels with `smem` bytes of dynamic shared memory each may launch: what the device holds at once, at
// most eight per SM.
int sms_times_resident(const mtpc_head* h, size_t smem) {
  const int per_sm = static_cast<int>(kSmemLimit / (smem + 1024));
  return h->num_sms * (per_sm < 1 ? 1 : per_sm > 8 ? 8 : per_sm);
}

// Circuit evaluation of W windows: out[w] = joint log-prob, prefix [W, n] = log-marginals of the prefixes x_0..x_i, msg
// [W, n, r] = slot messages (each may be NULL, not all).
// (The tree's joint kernel hands out windows through a counter next to the status word, which the projection or
// draft_slot_kernel before it has zeroed.)
int launch_circuit(mtpc_head* h, int W, int wpp, float* out, float* prefix, cudaStream_t st, bool raw_mixture = false,
                   float* msg = nullptr) {
  if (W <= 0) return MTPC_OK;
  const mtpc_config& c = h->cfg;
  const Layout& L = h->L;
  const float* G = at<float>(h, L.off_G);
  const float* logw = at<float>(h, L.off_logw);
  const int blocks = (W + kCircuitWarps - 1) / kCircuitWarps;
  const int threads = kCircuitWarps * 32;
  const bool sweep = prefix != nullptr || msg != nullptr;
  if (c.family == MTPC_CP && sweep) {
    const size_t per_warp = cp_prefix_warp_floats(c.n, c.r) * sizeof(float);
    const int warps = W <= h->num_sms || per_warp > 8192 ? 1 : 4;       // few windows: one per SM
    launch_kernel(circuit_cp_prefix_kernel, (W + warps - 1) / warps, warps * 32, warps * per_warp, st, overlapped(h), G, logw, out,
                  prefix, msg, W, wpp, c.n, c.r, L.sum_rows, raw_mixture ? 1 : 0);
  } else if (c.family == MTPC_CP) {
    launch_kernel(circuit_cp_kernel, blocks, threads, 0, st, overlapped(h), G, logw, out, W, wpp, c.n, c.r, L.sum_rows,
                  raw_mixture ? 1 : 0);
  } else if (c.family == MTPC_HMM) {
    const int stride = hmm_table_stride(h);
    const bool probabilities = stride == 0 && L.off_probA != 0;          // (a call without a head has log-probabilities alone)
    // Windows (a warp each) of a CTA: eight; of few windows with static tables as few as spread them over the SMs, two at least: a step is 40 reads of shared
    // memory a warp, which eight warps wait for in turn. Whole calls of a small head with eight / two, us: n = 16, r = 16, 120 positions
    // 33.6 / 23.7, 250 44.5 / 35.2; n = 8, r = 32, 120 positions 26.3 / 20.7; drafts + acceptance of n = 16, r = 32, v = 272, 16 positions of 16
    // windows 201.7 / 196.6. One a CTA: the same; two, and six warps that only help to copy tables, take longer. With r = 8 a step is too short to gain (n = 16, 250 positions 31.3 / 31.8).
    int warps = kHmmWarps;
    while (probabilities && c.r >= 16 && warps > 2 && (W + warps / 2 - 1) / (warps / 2) <= h->num_sms) warps /= 2;
    // as many tables as fit beside the warps' vectors (all of them but for very long windows)
    int chunk = c.n > 1 ? c.n - 1 : 1;
    while (chunk > 1 && hmm_circuit_smem_floats(c.n, c.r, prefix != nullptr, chunk, warps) * sizeof(float) > static_cast<size_t>(kSmemLimit)) --chunk;
    const size_t smem = hmm_circuit_smem_floats(c.n, c.r, prefix != nullptr, chunk, warps) * sizeof(float);
    const int items = stride == 0 ? (W + warps - 1) / warps : W / wpp * ((wpp + warps - 1) / warps);
    const int resident = sms_times_resident(h, smem);
    // contextual tables: a CTA per position while about one round of CTAs holds all positions, else a warp per window (both
    // measured at circuit_hmm_stream_kernel; the two cross between 1.0 and 1.6 rounds over n = 4 to 64, r = 8 to 32)
    if (stride != 0 && wpp <= 2 && 4ll * items > 5ll * resident) {
      const size_t stream_smem = kHmmStreamWarps * hmm_stream_warp_floats(c.n, c.r, prefix != nullptr) * sizeof(float);
      const int per_sm = static_cast<int>(kSmemLimit / (stream_smem + 1024)), ctas = (W + kHmmStreamWarps - 1) / kHmmStreamWarps;
      const int held = h->num_sms * (per_sm < 1 ? 1 : per_sm > 16 ? 16 : per_sm);
      launch_kernel(circuit_hmm_stream_kernel, ctas < held ? ctas : held, kHmmStreamWarps * 32, stream_smem, st, overlapped(h), G, logw,
                    hmm_tables(h), stride, out, prefix, msg, W, wpp, c.n, c.r, L.sum_rows);
    } else {
      launch_kernel(circuit_hmm_kernel, items < resident ? items : resident, warps * 32, smem, st, overlapped(h), G, logw,
                    probabilities ? at<float>(h, L.off_probA) : hmm_tables(h), stride, out, prefix, msg, W, wpp, c.n, c.r,
                    L.sum_rows, chunk, probabilities ? 1 : 0);
    }
  } else if (sweep) {
    const int warps = c.n / 2 < 8 ? c.n / 2 : 8;                         // a warp per node of the owners' level
    const bool fits = btree_prefix_smem_floats(c.n, c.r, warps, true) * sizeof(float) <= static_cast<size_t>(kSmemLimit);
    const size_t smem = btree_prefix_smem_floats(c.n, c.r, warps, fits) * sizeof(float);
    const int resident = sms_times_resident(h, smem);
    auto* kernel = c.r == 32 ? circuit_btree_prefix_kernel<32> : c.r == 16 ? circuit_btree_prefix_kernel<16>
                   : c.r == 8 ? circuit_btree_prefix_kernel<8> : circuit_btree_prefix_kernel<0>;
    launch_kernel(kernel, W < resident ? W : resident, warps * 32, smem, st, overlapped(h), G, logw, out,
                  prefix, msg, W, wpp, c.n, c.r, L.sum_rows, fits ? 1 : 0);
  } else {
    unsigned* counter = at<unsigned>(h, L.off_status) + kWorkCounterWord;
    const int resident = blocks < 8 * h->num_sms ? blocks : 8 * h->num_sms;   // more CTAs than an SM can hold do no harm
    // As a dependent only where a window is short work and there are few: else the CTAs crowd onto the SMs that fall free first
    // (n = 32, r = 16, d = 1024, whole calls as a dependent / not: 100 positions 71 / 58 us, 500 positions 98 / 84; n = 16, r = 8, 27
    // positions 26 / 29, 500 positions 45 / 41).
    const bool dependent = overlapped(h) && W <= h->num_sms && (c.n - 2) * c.r * c.r <= 1024;
    launch_kernel(circuit_btree_kernel, resident, threads, btree_smem_bytes(c.n, c.r), st, dependent, G, logw, out, counter, W,
                  wpp, c.n, c.r, L.sum_rows);
  }
  h->launches++;
  return check_launch();
}

// cudaFuncAttributeMaxDynamicSharedMemorySize belongs to the function, not to a head or a call: whoever sets it last
// wins. So every kernel that may ask for more than 48 KB gets the device's full limit, once and for all, and heads of
// different shapes (or a head and the static entry point) cannot lower it under each other.
template <typename K>
bool allow_full_smem(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) == cudaSuccess;
}
bool set_circuit_attributes() {
  bool ok = allow_full_smem(circuit_hmm_kernel);
  ok &= allow_full_smem(circuit_hmm_stream_kernel);
  ok &= allow_full_smem(circuit_btree_kernel);
  ok &= allow_full_smem(circuit_btree_prefix_kernel<32>) && allow_full_smem(circuit_btree_prefix_kernel<16>);
  ok &= allow_full_smem(circuit_btree_prefix_kernel<8>) && allow_full_smem(circuit_btree_prefix_kernel<0>);
  ok &= allow_full_smem(circuit_cp_prefix_kernel);
  return ok;
}

// How many clusters of `size` CTAs of a kernel, each with all the shared memory a CTA can have, device `dev` holds at once (0:
// none). Asked of the driver once per device and `which` (about 30 us each, a property of the device): heads are made often.
template <typename K>
int resident_clusters(K kernel, int size, int threads, int which, int dev) {
  constexpr int kDevices = 64;
  static std::atomic<int> known[4][kDevices];                            // count + 1
  std::atomic<int>* entry = dev >= 0 && dev < kDevices ? &known[which][dev] : nullptr;
  if (entry && entry->load() > 0) return entry->load() - 1;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(size);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = kSmemLimit;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (entry) entry->store(clusters + 1);
  return clusters;
}

// Rows per tile of the few-position draft path: the height in [64, 128] (multiple of 8) with which the longest of `ctas` persistent
// CTAs has the fewest rows, emission and sum-unit tiles dealt evenly together, a tile counted as 3 rows more and as one for every six
// positions the head may draft at once (its copies of their hidden states); ties go to the taller tile. (By the emission rows alone, a tree
// head of n = 8, r = 32, v = 256 got 5 tiles of 112 rows on its longest CTA where the mean is 485 rows, 4 of 128 now. 3 or 24 rows a tile whatever
// the positions, us: tree 16 x 32 x 256, 8 positions 154.1 / 155.8, 128 positions 209.9 / 206.6; tree 16 x 32 x 272, 8 positions 118.4 / 119.8. A head
// has one height, and one made for 128 positions loses nothing on fewer: made for the call's / for 128, tree 16 x 32 x 256, 8 positions 149.7 / 149.0, HMM
// 16 x 32 x 320, 1 position 208.3 / 208.2, mixture 8 x 16 x 320, 4 positions 63.1 / 62.8, tree 16 x 32 x 272, d = 2048, 8 positions 114.4 / 113.5.)
long long decode_tiles(long long rows, int sum_rows, int tr) {
  return (rows + tr - 1) / tr + (sum_rows + tr / 32 * 32 - 1) / (tr / 32 * 32);
}
int decode_tile_rows(long long rows, int sum_rows, int positions, int ctas) {
  int best = 128;
  long long best_cost = -1;
  for (int tr = 128; tr >= 64; tr -= 8) {
    const long long per_cta = (decode_tiles(rows, sum_rows, tr) + ctas - 1) / ctas;
    const long long cost = per_cta * (tr + 3 + positions / 6);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = tr; }
  }
  return best;
}
// The same together with the CTAs per tile (each with its part of K): 1, or 2, 4, 8 where all clusters of that size are
// resident at once (max_clusters: a size does not pack the SMs of every GPC, so fours cover less of the chip than twos) and
// every CTA keeps at least four K blocks. A CTA's time goes as its K steps x (rows it fetches per step + a fixed part worth
// about 32 rows) and the exchange of a cluster costs about 40 steps' worth of a row.
void choose_decode_tiling(long long rows, int sum_rows, int positions, int kblocks, int ctas, const int (&max_clusters)[3], int* tile_rows, int* ksplit) {
  *tile_rows = decode_tile_rows(rows, sum_rows, positions, ctas);
  *ksplit = 1;
  const long long per_cta = (decode_tiles(rows, sum_rows, *tile_rows) + ctas - 1) / ctas;
  long long best = kblocks * (per_cta * *tile_rows + 48);
  for (int e = 0; e < 3; ++e) {
    const int s = 2 << e;
    if (kblocks / s < 4) break;
    for (int tr = 128; tr >= 64; tr -= 8) {
      const long long cost = (kblocks + s - 1) / s * (tr + 48) + 40 * 48;
      if (decode_tiles(rows, sum_rows, tr) <= max_clusters[e] && cost < best) { best = cost; *tile_rows = tr; *ksplit = s; }
    }
  }
}

// Few-position draft path: one pass over all weight rows with the positions on the N axis.
int launch_decode_gemm(mtpc_head* h, const void* hidden_bf16, int P, cudaStream_t st) {
  const mtpc_config& c = h->cfg;
  const Layout& L = h->L;
  DecodeParams p;
  memset(&p, 0, sizeof(p));
  p.P = P;
  p.Ppad = (P + 15) / 16 * 16;
  int rc = make_tmap(&p.tm_h, hidden_bf16, static_cast<uint64_t>(P), static_cast<uint64_t>(c.d), p.Ppad);
  if (rc != MTPC_OK) return rc;
  p.tm_emit = h->tm_emit_dec;
  p.tm_sum = h->tm_sum_dec;
  p.kblocks = c.d / kBlockK;
  p.emit_rows = c.n * c.r * c.v;
  p.logits = at<float>(h, L.off_logits);
  if (h->lr_k > 0) {
    // a factored low-rank head streams W_base and B instead of the composed tensor: base = W_base h and z = B h, from
    // which lowrank_expand_kernel forms the logits
    p.tm_emit2 = h->tm_lrB_dec;
    p.emit_rows = c.n * c.v;
    p.emit2_rows = c.n * c.r * h->lr_k;
    p.logits = reinterpret_cast<float*>(h->ws + h->lr_off_dec);
    p.logits2 = p.logits + static_cast<size_t>(L.decode_max_p) * p.emit_rows;
  }
  p.sum_rows = L.sum_rows;
  p.r = c.r;
  p.tile_rows = h->decode_tile_rows;
  p.sum_tile_rows = h->decode_sum_tile_rows;
  p.tile_bytes = p.tile_rows * kBlockK * 2;
  p.emit_tiles = (p.emit_rows + p.tile_rows - 1) / p.tile_rows;
  p.emit2_tiles = (p.emit2_rows + p.tile_rows - 1) / p.tile_rows;
  p.sum_tiles = (p.sum_rows + p.sum_tile_rows - 1) / p.sum_tile_rows;
  p.tile_stride = (p.Ppad + 31) / 32 * 32;
  const int tiles = p.emit_tiles + p.emit2_tiles + p.sum_tiles;
  p.ksplit = h->decode_ksplit;
  while (p.ksplit > 1 && decode_exchange_bytes(p.ksplit, p.Ppad) > 64 * 1024) p.ksplit /= 2;
  // stage = weight tile + hidden tile, padded so that a 128-row operand read from the tile's base stays inside
  int stage = p.tile_bytes + p.Ppad * kBlockK * 2;
  if (stage < static_cast<int>(kABytes)) stage = kABytes;
  p.stage_bytes = (stage + 1023) / 1024 * 1024;
  const int ctl = 1024 + static_cast<int>(sizeof(GemmControl)) + static_cast<int>(decode_exchange_bytes(p.ksplit, p.Ppad));
  p.stages = (kSmemLimit - ctl) / p.stage_bytes;
  // At most nine stages (up to 16 positions 144 to 162 KB, by the tile's height): with more of them, or fewer, the same pass is up to 3 % slower. Why was
  // not found, but it is the number that counts, not the bytes, and it does on every head tried, whatever d, r, v and the circuit. Drafts +
  // acceptance with 7 / 8 / 9 / 10 / 12 stages, us: HMM 16 x 32 x 320, d = 4096, 8 positions 219.3 219.6 218.0 219.1 223.1; 16 x 16 x 272, d = 4096,
  // 12 positions 106.9 106.5 105.5 106.4 107.4; 8 x 32 x 272, d = 3072, 16 positions 84.6 84.1 83.7 84.2 84.4; mixture 4 x 32 x 256, d = 4096, 2
  // positions 55.1 55.3 53.6 54.2 54.1; 16 x 32 x 320, d = 2048, 6 positions 117.0 117.4 115.2 117.0 117.6; 8 x 8 x 256, d = 2048, 4 positions 22.4 22.6
  // 22.3 22.7 22.7; tree 8 x 16 x 256, d = 4096, 24 positions 60.9 60.4 59.7 59.9 60.1; 16 x 16 x 320, d = 2048, 40 positions 79.6 79.6 79.2 79.5 79.5;
  // the one exception mixture 8 x 16 x 320, d = 4096, 1 position 63.8 63.4 62.0 62.1 61.7. Six stages are 2 to 50 % slower.
  if (p.stages > kDecodeMaxStages) p.stages = kDecodeMaxStages;
  p.logw = at<float>(h, L.off_logw);
  p.sum_bias = sum_bias(h);
  p.status = at<unsigned>(h, L.off_status);
  p.wait_limit_ns = h->wait_limit_ns;
  launch_clusters(mtpc_decode_gemm_kernel, p.ksplit, p.ksplit > 1 ? tiles * p.ksplit : tiles < h->num_sms ? tiles : h->num_sms,
                  kGemmThreads, p.stages * p.stage_bytes + ctl, st, overlapped(h), p);
  h->launches++;
  if (h->lr_k > 0) {
    launch_kernel(lowrank_expand_kernel, dim3(c.n * c.r, (c.v + kExpandThreads - 1) / kExpandThreads), kExpandThreads,
                  static_cast<size_t>(P) * h->lr_k * sizeof(float), st, overlapped(h), p.logits, p.logits2,
                  static_cast<const __nv_bfloat16*>(h->lr_A), at<float>(h, L.off_logits), P, c.n, c.r, c.v, h->lr_k);
    h->launches++;
  }
  return check_launch();
}

void round_to_bf16(const float* src, __nv_bfloat16* dst, size_t count, cudaStream_t st, bool dependent) {
  const int vec = count % 8 == 0 && reinterpret_cast<uintptr_t>(src) % 16 == 0 && reinterpret_cast<uintptr_t>(dst) % 16 == 0;
  const size_t blocks = ((vec ? count / 8 : count) + 255) / 256;
  launch_kernel(f32_to_bf16_kernel, static_cast<unsigned>(blocks < 4096 ? blocks : 4096), 256, 0, st, dependent, src, dst,
                count, vec);
}

// hidden (io_dtype, device) -> bf16 device pointer the GEMM reads
int stage_hidden(mtpc_head* h, const void* hidden, int rows, const void** out_bf16, cudaStream_t st) {
  if (h->cfg.io_dtype == MTPC_BF16) { *out_bf16 = hidden; return MTPC_OK; }
  __nv_bfloat16* dst = at<__nv_bfloat16>(h, h->L.off_hidden);
  const size_t count = static_cast<size_t>(rows) * h->cfg.d;
  if (count) {
    round_to_bf16(static_cast<const float*>(hidden), dst, count, st, overlapped(h));
    h->launches++;
    if (check_launch() != MTPC_OK) return MTPC_ERR_CUDA;
  }
  *out_bf16 = dst;
  return MTPC_OK;
}

// One operand of a plain GEMM: a bf16 matrix in device memory, either [rows = M or N, K] with K contiguous (K-major) or
// [rows = K, M or N] with the M / N index contiguous (MN-major); pitch in elements.
struct GemmOperand {
  const void* ptr;
  size_t pitch;
  bool mn_major;
};

// Optional extras of a plain GEMM launch: bf16 output instead of fp32, and several products of one shape in a launch
// (see PlainGemmParams); a_* / b_* extents: the whole matrices the batched operands are windows of (M or N, then K).
// Scratch that lets a launch cut its last round along K (parts == 0: it does not).
struct SplitScratch {
  void* ptr = nullptr;
  int parts = 0;             // tile parts it has room for
};
// C2, C3: rows [m1, m2) and [m2, M) of the fp32 result go there.
struct PlainGemmExtra {
  float *C2 = nullptr, *C3 = nullptr;
  int m1 = 0, m2 = 0;
  void* C_bf16 = nullptr;
  int batches = 1, a_m_step = 0, a_k_step = 0, b_n_step = 0, b_k_step = 0;
  size_t c_step = 0;
  GemmOperand B2{nullptr, 0, false};         // a third K segment: K2 rows of B, from column a_k2 of A on
  int K2 = 0, a_k2 = 0;
  long long a_extent_m = 0, a_extent_k = 0, b_extent_n = 0, b_extent_k = 0;
};
int launch_plain_gemm(mtpc_head* h, GemmOperand A, GemmOperand B0, int K0, GemmOperand B1, int K1, int a_k1, float* C,
                      size_t ldc, int M, int N, cudaStream_t st, SplitScratch scratch = SplitScratch{}, void* C_hilo = nullptr,
                      int split_k = 0, const PlainGemmExtra* extra = nullptr);
// parts: 1 = sum-unit tiles (log omega), 2 = W_base h, z = B h and the repacked A, 4 = G (and the units' log-sum-exps)
int launch_lowrank_projection(mtpc_head* h, const void* hidden_bf16, int T, const int* targets, cudaStream_t st,
                              float* lse_out = nullptr, int parts = 7, bool targets_are_drafts = false);

// out [T] (joint) and / or prefix [T, n] (prefix log-marginals); either may be NULL, not both.
int window_logprob_impl(mtpc_head* h, const void* hidden, const int32_t* targets, int32_t T, float* out, float* prefix,
                        cudaStream_t st) {
  const void* hb = nullptr;
  h->draft_P = 0;   // log omega of the last draft is overwritten below
  int rc = stage_hidden(h, hidden, T, &hb, st);
  if (rc != MTPC_OK) return rc;
  PhaseTimer pt(h, st);
  pt.begin();
  if (h->lr_k > 0) rc = launch_lowrank_projection(h, hb, T, targets, st);
  else rc = launch_gemm(h, hb, T, true, true, targets, st);
  pt.end();
  if (rc != MTPC_OK) return rc;
  pt.begin();
  rc = launch_circuit(h, T, 1, out, prefix, st);
  pt.end();
  return rc;
}

// The stream capture that `st` is recording into (0: none).
unsigned long long capture_id(cudaStream_t st) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(st, &status, &id) != cudaSuccess) { cudaGetLastError(); return 0; }
  return status == cudaStreamCaptureStatusActive ? id + 1 : 0;
}
// Dynamic shared memory that leaves an SM room for its even share of `ctas` CTAs and no more. The CTAs of a programmatic dependent that do not fit
// beside the projection's (ten warps of 168 registers; with six of 120 they did) pile up on the SMs that fall free first, up to sixteen on one while
// others stay empty. Latent draws behind a projection, six warps ahead / ten / ten and so, us: tree 16 x 8, 595 positions 10.4 / 16.7 / 10.4, 16 x 32,
// 400 positions 10.2 / 18.0 / 10.4, 3000 positions 21 / 21 / 15; HMM 16 x 16, 568 positions 10.7 / 16.4 / 10.5, 1000 positions 17.2 / 17.7 / 11.4. (A plain
// launch 13, since its start is then in the chain; one window a CTA 11 to 13; 144 registers a thread in the projection: only the HMM's 568 10.2.)
size_t even_share_smem(const mtpc_head* h, long long ctas) {
  const size_t share = static_cast<size_t>((ctas + h->num_sms - 1) / h->num_sms);
  if (share == 0 || share > 16) return 0;                               // (sixteen CTAs are all that an SM's threads let in)
  return ((kSmemLimit + 1024) / share - 1024) / 1024 * 1024;            // (1 KB of an SM's 228 goes with every CTA)
}

// out_logprob [W] (joint) and / or out_prefix [W, n] (prefix log-marginals of the draft); either may be NULL, not both.
int draft_sample_impl(mtpc_head* h, const void* hidden, int32_t P, int32_t wpp, const float* uniforms,
                      int32_t* out_bytes, float* out_logprob, float* out_prefix, cudaStream_t st) {
  const mtpc_config& c = h->cfg;
  const Layout& L = h->L;
  const int W = P * wpp;
  if (P > L.decode_max_p && (c.flags & MTPC_FLAG_SHORT_DRAFTS) != 0) return MTPC_ERR_UNSUPPORTED;
  // a draft that returns prefix marginals runs the sweep that also yields the slot messages of the acceptance stage (the joints
  // alone take a tree half the table passes: 203 us against 294 for 8000 windows of n = 16, r = 32)
  float* const msg = out_prefix ? at<float>(h, L.off_msg) : nullptr;
  const unsigned long long capture = capture_id(st);
  if (capture != 0 && !out_prefix) h->joint_recorded = true;
  if (h->lr_k > 0 && P > L.decode_max_p && wpp == 1 && c.v <= kMaxDraftVocab) {
    // A long draft on a factored head, one window per position: log omega, the latent draws, then every (window, slot)
    // forms the logits of its one selected unit from W_base h and B h (lowrank_draw_kernel) and draws its byte; the
    // evidence of the drafted bytes under every unit is the factored projection with them as targets. No logits are
    // kept: the acceptance stage forms those of a window's rejected slot from W_base h and B h.
    const int k = h->lr_k;
    h->draft_P = 0;
    PhaseTimer pt(h, st);
    pt.begin();
    int rc = launch_lowrank_projection(h, hidden, P, nullptr, st, nullptr, /*parts=*/1 | 2);
    pt.end();
    if (rc != MTPC_OK) return rc;
    pt.begin();
    launch_kernel(latent_sample_kernel, (W + kLatentWarps - 1) / kLatentWarps, 32 * kLatentWarps, 0, st, overlapped(h),
                  c.family, at<float>(h, L.off_logw), hmm_tables(h), uniforms, at<int>(h, L.off_sel), out_bytes,
                  at<unsigned>(h, L.off_status), W, wpp, c.n, c.r, L.sum_rows, hmm_table_stride(h));
    h->launches++;
    pt.end();
    if ((rc = check_launch()) != MTPC_OK) return rc;
    pt.begin();
    const float* base = reinterpret_cast<const float*>(h->ws + h->lr_off_base);
    {
      const int pairs = W * c.n;
      int blocks = (pairs + kDrawWarps - 1) / kDrawWarps;
      if (blocks > 32 * h->num_sms) blocks = 32 * h->num_sms;
      launch_kernel(lowrank_draw_kernel, blocks, 32 * kDrawWarps, static_cast<size_t>(kDrawWarps) * c.v * sizeof(float), st,
                    overlapped(h), base, reinterpret_cast<const __nv_bfloat16*>(h->ws + h->lr_off_zhl),
                    static_cast<const __nv_bfloat16*>(h->lr_A), at<int>(h, L.off_sel), uniforms, out_bytes,
                    at<unsigned>(h, L.off_status), W, wpp, c.n, c.r, c.v, valid_symbols(c), k);
      h->launches++;
    }
    pt.end();
    if ((rc = check_launch()) != MTPC_OK) return rc;
    pt.begin();
    rc = launch_lowrank_projection(h, hidden, P, out_bytes, st, nullptr, /*parts=*/4, /*targets_are_drafts=*/true);
    pt.end();
    if (rc != MTPC_OK) return rc;
    pt.begin();
    rc = launch_circuit(h, W, wpp, out_logprob, out_prefix, st, /*raw_mixture=*/false, msg);
    pt.end();
    if (rc == MTPC_OK) {               // G, log omega, the messages, W_base h and B h stay in place for an acceptance call
      h->draft_P = P;
      h->draft_wpp = wpp;
      h->draft_msg = msg != nullptr;
      h->draft_capture = capture;
      h->draft_logits = false;
      h->draft_hidden = nullptr;
    }
    return rc;
  }
  if (h->lr_k > 0 && P > L.decode_max_p) {
    // Otherwise (several windows per position, or units wider than 512 symbols) the few-position path runs chunk after
    // chunk of positions: W_base, B and A are small enough to stay in L2. Only the last chunk's logits and messages remain: no
    // acceptance stage after such a draft.
    for (int p0 = 0; p0 < P; p0 += L.decode_max_p) {
      const int pc = P - p0 < L.decode_max_p ? P - p0 : L.decode_max_p;
      const size_t w0 = static_cast<size_t>(p0) * wpp;
      const int rc = draft_sample_impl(h, static_cast<const uint8_t*>(hidden) + static_cast<size_t>(p0) * c.d * 2, pc, wpp,
                                       uniforms + w0 * 2 * c.n, out_bytes + w0 * c.n, out_logprob ? out_logprob + w0 : nullptr,
                                       out_prefix ? out_prefix + w0 * c.n : nullptr, st);
      if (rc != MTPC_OK) return rc;
    }
    h->draft_P = 0;
    return MTPC_OK;
  }
  const void* hb = nullptr;
  int rc = stage_hidden(h, hidden, P, &hb, st);
  if (rc != MTPC_OK) return rc;
  PhaseTimer pt(h, st);
  h->draft_P = 0;
  if (P <= L.decode_max_p) {
    // Few positions: every weight row is read once. 1. all logits (emission -> scratch, sum units -> log omega)
    // 2. per (position, slot): latent draws, byte draws, evidence of the drafted bytes  3. circuit evaluation
    pt.begin();
    rc = launch_decode_gemm(h, hb, P, st);
    pt.end();
    if (rc != MTPC_OK) return rc;
    pt.begin();
    {
      int chain = 0;                                       // longest chain of latent-draw tables of any slot
      if (c.family == MTPC_HMM) chain = c.n - 1;
      if (c.family == MTPC_BTREE) { for (int m = c.n; m > 2; m >>= 1) ++chain; }
      const size_t base = static_cast<size_t>((2 * c.r + 3) & ~3) * sizeof(float);
      const size_t with_tables = base + static_cast<size_t>(chain) * c.r * c.r * sizeof(float);
      const int in_smem = chain > 0 && with_tables <= kSlotSmemLimit;
      // The units' weights stay in shared memory for the byte draws where there are many draws to a unit, if they fit beside the
      // tables without costing an SM its second CTA, or there is no second one to be had anyway. (Where most are never used, the
      // CTAs are better kept small enough to wait beside the weight pass's: 27 positions of a tree head, 4 windows on 32 units,
      // 109.4 us with them and 106.3 without; 16 windows on 16 units, 64 positions: 153.4 and 157.0.)
      const size_t weights = static_cast<size_t>(c.r) * ((c.v + 31) / 32 * 32) * sizeof(float);
      const size_t smem = (in_smem ? with_tables : base) + weights;
      const int weights_in_smem = c.v <= kMaxDraftVocab && 2 * wpp >= c.r &&
                                  (smem <= kSlotSmemPair || (smem <= kSlotSmemLimit && c.n * P <= h->num_sms));
      // builds of the narrow kernel that unroll 4, 8, 10 or 16 batches of 32 symbols: the smallest that covers v; where a device full of
      // CTAs is not all of them, and a third fits an SM's shared memory, the builds whose registers let it (see draft_slot_kernel; not of
      // contextual tables, which come by L2 for every position. Two / three there, us: one window a position, n = 16, r = 16, 100 positions 116.2 /
      // 116.9, r = 32, 115 positions 204.8 / 204.9, r = 8, 120 positions 75.8 / 75.7; but four windows, n = 8, r = 16, 64 positions 44.1 / 42.9, n = 16, r = 32,
      // 128 positions 162.0 / 161.1, and sixteen, n = 8, r = 32, 100 positions 129.8 / 126.5: with many draws to a table three would gain)
      const size_t slot_smem = weights_in_smem ? smem : smem - weights;
      const bool crowd = !is_ctx(h) && c.n * P > 2 * h->num_sms && 3 * (slot_smem + 1024) <= static_cast<size_t>(kSmemLimit);
      auto* slot_kernel = c.v > kMaxDraftVocab ? draft_slot_kernel<true, 16, 2>
                          : c.v <= 128 ? (crowd ? draft_slot_kernel<false, 4, 3> : draft_slot_kernel<false, 4, 2>)
                          : c.v <= 256 ? (crowd ? draft_slot_kernel<false, 8, 3> : draft_slot_kernel<false, 8, 2>)
                          : c.v <= 320 ? (crowd ? draft_slot_kernel<false, 10, 3> : draft_slot_kernel<false, 10, 2>)
                                       : draft_slot_kernel<false, 16, 2>;
      launch_kernel(slot_kernel, dim3(c.n, P), kSlotThreads, slot_smem, st, overlapped(h), c.family,
                    at<float>(h, L.off_logits), at<float>(h, L.off_logw), is_ctx(h) ? hmm_tables(h) : at<float>(h, L.off_cdfA), uniforms, out_bytes,
                    at<float>(h, L.off_G), at<float>(h, L.off_unit_lse), at<unsigned>(h, L.off_status),
                    at<unsigned>(h, L.off_status) + kWorkCounterWord, wpp, c.n, c.r, c.v, valid_symbols(c), L.sum_rows,
                    hmm_table_stride(h), in_smem, weights_in_smem);
    }
    h->launches++;
    h->draft_P = P;
    h->draft_wpp = wpp;
    h->draft_msg = msg != nullptr;
    h->draft_capture = capture;
    h->draft_logits = true;
    pt.end();
    if ((rc = check_launch()) != MTPC_OK) return rc;
    pt.begin();
    rc = launch_circuit(h, W, wpp, out_logprob, out_prefix, st, /*raw_mixture=*/c.r > 32, msg);
    pt.end();
    return rc;
  }
  // Many positions: one projection that keeps its logits, unit log-sum-exps and log omega; everything after it is gathers.
  // In chunks of positions if the logits of all of them do not fit (then only the last chunk's remain).
  const int chunks = (P + L.kept_p - 1) / L.kept_p, chunk_p = (P + chunks - 1) / chunks;
  for (int p0 = 0; p0 < P; p0 += chunk_p) {
    const int pc = P - p0 < chunk_p ? P - p0 : chunk_p, wc = pc * wpp;
    const size_t w0 = static_cast<size_t>(p0) * wpp;
    const float* u = uniforms + w0 * 2 * c.n;
    GradArgs keep;
    keep.lse_out = at<float>(h, L.off_unit_lse);
    keep.logit_out = at<float>(h, L.off_logits);
    keep.logit_pitch = static_cast<size_t>(c.n) * c.r * c.v;
    pt.begin();
    rc = launch_gemm(h, static_cast<const __nv_bfloat16*>(hb) + static_cast<size_t>(p0) * c.d, pc, true, true, nullptr, st, &keep, nullptr, p0);
    pt.end();
    if (rc != MTPC_OK) return rc;
    int* sel = at<int>(h, L.off_sel) + w0 * c.n;
    pt.begin();
    const int latent_ctas = (wc + kLatentWarps - 1) / kLatentWarps;
    launch_kernel(latent_sample_kernel, latent_ctas, 32 * kLatentWarps, even_share_smem(h, latent_ctas), st, overlapped(h),
                  c.family, at<float>(h, L.off_logw) + static_cast<size_t>(p0) * L.sum_rows,
                  hmm_tables(h) + static_cast<size_t>(p0) * hmm_table_stride(h), u, sel, out_bytes + w0 * c.n,
                  at<unsigned>(h, L.off_status), wc, wpp, c.n, c.r, L.sum_rows, hmm_table_stride(h));
    pt.end();
    pt.begin();
    auto* pick = c.v > kMaxDraftVocab ? draft_pick_kernel<true, 16>
                 : c.v <= 256 ? draft_pick_kernel<false, 8>
                 : c.v <= 320 ? draft_pick_kernel<false, 10> : draft_pick_kernel<false, 16>;
    launch_kernel(pick, (wc * c.n + 7) / 8, 256, 0, st, overlapped(h), keep.logit_out, keep.lse_out, sel, u,
                  out_bytes + w0 * c.n, at<float>(h, L.off_G) + w0 * c.n * c.r, at<unsigned>(h, L.off_status), wc * c.n, wpp,
                  c.n, c.r, c.v, valid_symbols(c));
    pt.end();
    h->launches += 2;
    if ((rc = check_launch()) != MTPC_OK) return rc;
  }
  pt.begin();
  rc = launch_circuit(h, W, wpp, out_logprob, out_prefix, st, /*raw_mixture=*/false, msg);
  pt.end();
  if (rc == MTPC_OK) {                 // G, log omega, the messages and the logits stay in place for an acceptance call
    h->draft_P = P;
    h->draft_wpp = wpp;
    h->draft_msg = msg != nullptr;
    h->draft_capture = capture;
    h->draft_logits = chunks == 1;
    h->draft_hidden = hb;
  }
  return rc;
}

// ---------------------------------------------------------------- backward pass (host side)
size_t round64(size_t x) { return (x + 63) / 64 * 64; }

// How a plain GEMM of `tiles` tiles and `kblocks` K blocks is dealt to `workers` (CTAs, or pairs: ctas = 2): the tiles of the
// last, partial round are cut into `split` parts each. Cost in K-block times of a worker (0.4 us): a part adds about 8 for
// writing its fp32 tile, the reduction 10 and its bytes through L2 (15 tile parts of 128 KB a block time). Cut only where that
// wins clearly, into no more than `parts` tile parts in all.
struct SplitPlan {
  int tail = 0, split = 1;
  long long cost = 0;
};
SplitPlan plan_split(long long tiles, int kblocks, int workers, int ctas, int parts) {
  SplitPlan b;
  const long long whole = tiles / workers;
  const int rem = static_cast<int>(tiles % workers);
  b.cost = whole * kblocks + (rem ? kblocks : 0);
  if (rem == 0) return b;
  const long long limit = b.cost - 8;
  for (int s = 2; s <= 16 && rem * s * ctas <= parts && kblocks / s >= 4; ++s) {
    const long long rounds = (static_cast<long long>(rem) * s + workers - 1) / workers;
    const long long cost = whole * kblocks + rounds * ((kblocks + s - 1) / s + 8) + 10 + rem * s * ctas / 15;
    if (cost < b.cost && cost < limit) { b.cost = cost; b.tail = rem; b.split = s; }
  }
  return b;
}

int k_blocks(size_t k) { return static_cast<int>((k + kBlockK - 1) / kBlockK); }
// Tile parts that a launch of M x N over `kblocks` K blocks may be cut into, by single CTAs or pairs of a 148-SM device (elsewhere
// what is reserved limits the cut).
int split_parts(size_t M, int N, int kblocks) {
  int parts = 0;
  for (int ctas = 1; ctas <= 2; ++ctas) {
    const long long tiles = static_cast<long long>((M + ctas * kBlockM - 1) / (ctas * kBlockM)) * ((N + kPlainTileN - 1) / kPlainTileN);
    const SplitPlan p = plan_split(tiles, kblocks, 148 / ctas, ctas, kSplitParts);
    if (p.tail * p.split * ctas > parts) parts = p.tail * p.split * ctas;
  }
  return parts;
}

// Carving of the backward workspace for T positions (all buffers 256-byte aligned).
// The sum-unit logit gradients sit to the right of the emission logit gradients in one matrix [T, Kd], Kd = Nc + Spad.
struct BackwardLayout {
  size_t Nc, Spad, Kd;
  size_t off_lse, off_post, off_logits, off_dlogit, off_coeff, off_split, total;
  int parts;                 // tile parts at off_split
};
// rank > 0: of a factored head, which keeps no logits.
void plan_backward(const mtpc_config& c, const Layout& L, int T, BackwardLayout* B, int rank = 0) {
  B->Nc = static_cast<size_t>(c.n) * c.r * c.v;
  B->Spad = round64(L.sum_rows);
  B->Kd = B->Nc + B->Spad;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes); return o; };
  B->off_lse = take(static_cast<size_t>(T) * c.n * c.r * 4);
  B->off_post = take(static_cast<size_t>(T) * c.n * c.r * 4);
  B->off_logits = take(rank == 0 ? static_cast<size_t>(T) * B->Nc * 4 : 0);   // [T, Nc] fp32: the emission logits of the forward pass
  B->off_dlogit = take(static_cast<size_t>(T) * B->Kd * 2);          // [T, Nc | Spad] bf16
  B->off_coeff = take(static_cast<size_t>(T) * c.n * 4);             // Eq. 6: weights of the prefix marginals
  // parts of the GEMMs' cut tiles: d hidden, and the weight gradients in one launch
  const size_t nv = static_cast<size_t>(c.n) * c.v, nrk = static_cast<size_t>(c.n) * c.r * rank;
  const int dh_blocks = (rank ? k_blocks(nv) + k_blocks(nrk) : k_blocks(B->Nc)) + k_blocks(L.sum_rows);
  const int dh = split_parts(T, c.d, dh_blocks), dw = split_parts((rank ? nv + nrk : B->Nc) + L.sum_rows, c.d, k_blocks(T));
  B->parts = dh > dw ? dh : dw;
  B->off_split = take(B->parts * kSplitPartBytes);
  B->total = off;
}

template <int CTAS>
void launch_plain_tiles(const PlainGemmParams& p, bool a_mn, bool b_mn, int grid, size_t smem, cudaStream_t st, bool dependent) {
  auto* kernel = a_mn ? plain_gemm_kernel<true, true, kPlainTileN, CTAS>
                      : b_mn ? plain_gemm_kernel<false, true, kPlainTileN, CTAS> : plain_gemm_kernel<false, false, kPlainTileN, CTAS>;
  launch_clusters(kernel, CTAS, grid, kGemmThreads, smem, st, dependent, p);
}

// C[M, N] fp32 (pitch ldc) = A B^T over K = K0 + K1: segment 0 multiplies A's K range [0, K0) with B0, segment 1 (K1 > 0)
// A's K range [a_k1, a_k1 + K1) with B1.
// C_hilo != NULL (then C is NULL): the result leaves as two bf16 halves per entry, see PlainGemmParams.
int launch_plain_gemm(mtpc_head* h, GemmOperand A, GemmOperand B0, int K0, GemmOperand B1, int K1, int a_k1, float* C,
                      size_t ldc, int M, int N, cudaStream_t st, SplitScratch scratch, void* C_hilo, int split_k,
                      const PlainGemmExtra* extra) {
  if (M <= 0 || N <= 0 || K0 <= 0) return MTPC_OK;
  if (K1 > 0 && (A.mn_major || B1.mn_major != B0.mn_major)) return MTPC_ERR_SHAPE;
  if (A.mn_major && !B0.mn_major) return MTPC_ERR_SHAPE;
  const PlainGemmExtra none;
  const PlainGemmExtra& x = extra ? *extra : none;
  if (x.batches < 1 || (x.batches > 1 && K1 > 0)) return MTPC_ERR_SHAPE;
  PlainGemmParams p;
  memset(&p, 0, sizeof(p));
  p.M = M; p.N = N;
  p.a_k0[0] = 0;
  p.a_k0[1] = a_k1;
  p.seg_kblocks[0] = (K0 + kBlockK - 1) / kBlockK;
  p.seg_kblocks[1] = K1 > 0 ? (K1 + kBlockK - 1) / kBlockK : 0;
  p.a_k0[2] = x.a_k2;
  p.seg_kblocks[2] = x.K2 > 0 ? (x.K2 + kBlockK - 1) / kBlockK : 0;
  if (x.K2 > 0 && (K1 <= 0 || !x.B2.mn_major || !B0.mn_major)) return MTPC_ERR_SHAPE;
  const int kblocks = p.seg_kblocks[0] + p.seg_kblocks[1] + p.seg_kblocks[2];
  // batched products with a rank for N: 64-column accumulator tiles
  const int tile_n = (x.batches > 1 && N <= 64 && B0.mn_major) ? 64 : kPlainTileN;
  p.n_tiles = (N + tile_n - 1) / tile_n;
  const int m_tiles = (M + kBlockM - 1) / kBlockM;
  // Single CTAs or pairs: whichever needs fewer K-block times (a pair's 256 x 256 tile takes its two SMs as long as a single
  // CTA's 128 x 256 tile takes one), a pair counted 1/16 cheaper: it moves a third less operand data (dW_sum of 14368 rows:
  // 280 us in pairs, 312 us alone). Within one round it is the call's latency that counts, and a lone CTA's is shorter unless K is long and
  // the tiles are not so few that most are cut (training calls of 700 positions, 4 x 16 x 320, d = 3072 276 us alone, 268 in pairs; 500 factored
  // positions of 8 x 32 x 320, d = 4096 277 / 271; but 300 factored positions of 4 x 8 x 256, d = 1024 41.5 / 43.8, and training calls of 250
  // positions, 8 x 8 x 256, d = 2048 105.5 / 106.6).
  SplitPlan plan;
  bool pair = false;
  if (tile_n == kPlainTileN && x.batches == 1) {
    plan = plan_split(static_cast<long long>(m_tiles) * p.n_tiles, kblocks, h->num_sms, 1, scratch.parts);
    const long long tiles = static_cast<long long>(m_tiles) * p.n_tiles;
    if (h->max_pairs > 0 && m_tiles >= 2 && (tiles > h->num_sms || (kblocks >= 64 && 4 * tiles > h->num_sms))) {
      const SplitPlan two = plan_split(static_cast<long long>((m_tiles + 1) / 2) * p.n_tiles, kblocks, h->max_pairs, 2, scratch.parts);
      if (two.cost * 15 <= plan.cost * 16) { plan = two; pair = true; }
    }
  }
  const int ctas = pair ? 2 : 1;
  p.m_tiles = (m_tiles + ctas - 1) / ctas;
  p.tail_tiles = plan.tail;
  p.split = plan.split;
  p.partial = static_cast<float*>(scratch.ptr);
  const int Ka = x.K2 > 0 ? x.a_k2 + x.K2 : K1 > 0 ? a_k1 + K1 : K0;           // extent of A along K
  const uint64_t a_m = x.a_extent_m ? x.a_extent_m : M, a_k = x.a_extent_k ? x.a_extent_k : Ka;
  const uint64_t b_n = x.b_extent_n ? x.b_extent_n : N, b_k = x.b_extent_k ? x.b_extent_k : K0;
  const int b_box = kPlainTileN / ctas;
  int rc = A.mn_major ? make_tmap_mn(&p.tm_a, A.ptr, a_k, a_m, A.pitch) : make_tmap(&p.tm_a, A.ptr, a_m, a_k, kBlockM, A.pitch);
  if (rc == MTPC_OK)
    rc = B0.mn_major ? make_tmap_mn(&p.tm_b[0], B0.ptr, b_k, b_n, B0.pitch) : make_tmap(&p.tm_b[0], B0.ptr, b_n, b_k, b_box, B0.pitch);
  if (rc == MTPC_OK && K1 > 0)
    rc = B1.mn_major ? make_tmap_mn(&p.tm_b[1], B1.ptr, K1, N, B1.pitch) : make_tmap(&p.tm_b[1], B1.ptr, N, K1, b_box, B1.pitch);
  if (rc == MTPC_OK && x.K2 > 0) rc = make_tmap_mn(&p.tm_b[2], x.B2.ptr, x.K2, N, x.B2.pitch);
  if (rc != MTPC_OK) return rc;
  p.stage_bytes = kABytes + tile_n / ctas * kBlockK * 2;
  const int ctl = 1024 + static_cast<int>(sizeof(GemmControl));
  p.stages = (kSmemLimit - ctl) / p.stage_bytes;
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  p.wide_stores = (reinterpret_cast<uintptr_t>(C) % 32 == 0 && ldc % 8 == 0 && x.c_step % 8 == 0) ? 1 : 0;
  p.C = C;
  p.ldc = ldc;
  p.C2 = x.C2;
  p.C3 = x.C3;
  p.m_end[0] = x.C2 ? x.m1 : M;
  p.m_end[1] = x.C3 ? x.m2 : M;
  if (reinterpret_cast<uintptr_t>(x.C2) % 32 != 0 || reinterpret_cast<uintptr_t>(x.C3) % 32 != 0) p.wide_stores = 0;
  p.C_hilo = static_cast<__nv_bfloat16*>(C_hilo);
  p.split_k = split_k;
  p.C_bf16 = static_cast<__nv_bfloat16*>(x.C_bf16);
  if ((C != nullptr) + (C_hilo != nullptr) + (x.C_bf16 != nullptr) != 1) return MTPC_ERR_NULL;
  if (C_hilo != nullptr && (split_k < 16 || split_k % 16 != 0 || N % split_k != 0)) return MTPC_ERR_SHAPE;
  if (x.C_bf16 != nullptr && (reinterpret_cast<uintptr_t>(x.C_bf16) % 32 != 0 || ldc % 16 != 0 || x.c_step % 16 != 0))
    return MTPC_ERR_WORKSPACE;
  p.batches = x.batches;
  p.a_m_step = x.a_m_step; p.a_k_step = x.a_k_step; p.b_n_step = x.b_n_step; p.b_k_step = x.b_k_step;
  p.c_step = x.c_step;
  p.status = at<unsigned>(h, h->L.off_status);
  p.wait_limit_ns = h->wait_limit_ns;
  const long long items = static_cast<long long>(p.m_tiles) * p.n_tiles * p.batches + static_cast<long long>(p.tail_tiles) * (p.split - 1);
  const int workers = pair ? h->max_pairs : h->num_sms;
  const int grid = ctas * static_cast<int>(items < workers ? items : workers);
  const size_t smem = p.stages * p.stage_bytes + ctl;
  if (tile_n == 64 && A.mn_major) launch_kernel(plain_gemm_kernel<true, true, 64>, grid, kGemmThreads, smem, st, overlapped(h), p);
  else if (tile_n == 64) launch_kernel(plain_gemm_kernel<false, true, 64>, grid, kGemmThreads, smem, st, overlapped(h), p);
  else if (pair) launch_plain_tiles<2>(p, A.mn_major, B0.mn_major, grid, smem, st, overlapped(h));
  else launch_plain_tiles<1>(p, A.mn_major, B0.mn_major, grid, smem, st, overlapped(h));
  h->launches++;
  if (p.tail_tiles > 0) {
    launch_kernel(split_reduce_kernel, p.tail_tiles * ctas * 8, 256, 0, st, overlapped(h), p, ctas);
    h->launches++;
  }
  return check_launch();
}

// What a factored head serves (mtpc_lowrank_gemm.cuh); false: the shape does not fit.
bool plan_lowrank(const mtpc_config& c, int k, LowRankParams* p) {
  if (k < 16 || k > kLrMaxRank || k % 16 != 0 || c.v % 16 != 0 || c.v > kLrMaxVocab) return false;
  p->n = c.n; p->r = c.r; p->v = c.v; p->k = k;
  p->vv = c.v_valid > 0 ? c.v_valid : c.v;
  return true;
}

// One launch of the factored projection's kernel on what parts 1 | 2 left in the workspace.
template <int MODE>
int launch_lowrank_logits(mtpc_head* h, LowRankParams p, int T, cudaStream_t st) {
  const int rc = make_tmap(&p.tm_z, h->ws + h->lr_off_zhl, static_cast<uint64_t>(T), static_cast<uint64_t>(p.n) * p.r * 2 * p.k, kBlockM);
  p.blocks = (p.v + kLrCols - 1) / kLrCols;
  p.tm_a = h->lr_tm_a;
  if (rc != MTPC_OK) return rc;
  p.T = T;
  p.m_tiles = (T + kBlockM - 1) / kBlockM;
  p.base = reinterpret_cast<const float*>(h->ws + h->lr_off_base);
  p.status = at<unsigned>(h, h->L.off_status);
  p.wait_limit_ns = h->wait_limit_ns;
  const long long items = static_cast<long long>(p.m_tiles) * p.n * p.blocks;
  const int held = lowrank_ctas(MODE) * h->num_sms;
  const int grid = static_cast<int>(items < held ? items : held);
  launch_kernel(lowrank_logits_kernel<MODE>, grid, lowrank_threads(MODE), lowrank_smem_bytes(MODE), st, overlapped(h), p);
  h->launches++;
  return check_launch();
}

// Factored projection of a low-rank head: log omega by the dense kernel's sum tiles, W_base h and z = B h (as two bf16 halves)
// by plain GEMMs, A repacked; then the log-sum-exps over base + corrections and their merge into G.
int launch_lowrank_projection(mtpc_head* h, const void* hidden_bf16, int T, const int* targets, cudaStream_t st, float* lse_out,
                              int parts, bool targets_are_drafts) {
  const mtpc_config& c = h->cfg;
  const Layout& L = h->L;
  const int units = c.n * c.r, k = h->lr_k;
  int rc = MTPC_OK;
  if (parts & 1) rc = launch_gemm(h, hidden_bf16, T, false, true, targets, st);
  if (rc != MTPC_OK) return rc;
  __nv_bfloat16* zhl = reinterpret_cast<__nv_bfloat16*>(h->ws + h->lr_off_zhl);
  float* base = reinterpret_cast<float*>(h->ws + h->lr_off_base);
  if (parts & 2) {
    const GemmOperand hid{hidden_bf16, static_cast<size_t>(c.d), false};
    const GemmOperand bmat{h->lr_B, static_cast<size_t>(c.d), false};          // [n r k, d], K = d contiguous
    const GemmOperand wmat{h->lr_W_base, static_cast<size_t>(c.d), false};
    rc = launch_plain_gemm(h, hid, wmat, c.d, wmat, 0, 0, base, static_cast<size_t>(c.n) * c.v, T, c.n * c.v, st, SplitScratch{h->ws + h->lr_off_split, h->lr_split_parts});
    // z = B h, leaving the GEMM's epilogue already split into its two bf16 halves [T, n r, 2, k]
    if (rc == MTPC_OK)
      rc = launch_plain_gemm(h, hid, bmat, c.d, bmat, 0, 0, nullptr, 0, T, units * k, st, SplitScratch{h->ws + h->lr_off_split, h->lr_split_parts}, zhl, k);
    if (rc != MTPC_OK) return rc;
    // A as [n, v, r, k]: the adaptor columns of adjacent components side by side (remade every call: A may have changed)
    const size_t pieces = static_cast<size_t>(units) * c.v * (k / 8);
    launch_kernel(lowrank_repack_kernel, static_cast<unsigned>((pieces + 255) / 256), 256, 0, st, overlapped(h),
                  static_cast<const uint4*>(h->lr_A), reinterpret_cast<uint4*>(h->ws + h->lr_off_arep), c.n, c.r, c.v, k / 8);
    h->launches += 1;
  }
  if (!(parts & 4)) return check_launch();
  LowRankParams p = h->lr_params;
  p.log_sum = reinterpret_cast<float*>(h->ws + h->lr_off_partial);
  p.ref = p.log_sum + static_cast<size_t>((c.v + 31) / 32) * ((T + 31) / 32 * 32) * units;
  if ((rc = launch_lowrank_logits<kLowRankForward>(h, p, T, st)) != MTPC_OK) return rc;
  launch_kernel(k == 16 ? lowrank_merge_kernel<16> : lowrank_merge_kernel<32>, dim3((T + 31) / 32, c.n, (c.r + kMergeUnits - 1) / kMergeUnits), 256, 0, st, overlapped(h), p.log_sum, p.ref,
                base, zhl, reinterpret_cast<const __nv_bfloat16*>(h->ws + h->lr_off_arep), targets, at<float>(h, L.off_G),
                lse_out, at<unsigned>(h, L.off_status), T, c.n, c.r, c.v, p.vv, targets_are_drafts ? 1 : 0);
  h->launches += 1;
  return check_launch();
}

// Warps per CTA of the circuit backward kernels: as many of 8, 4, 2, 1 as keep the CTA's shared memory within the limit
// (long windows need n x r floats of messages per warp). warps == 0: not even one warp fits.
struct BackwardShape {
  int warps;
  size_t smem;
  bool wide;                 // HMM, Eq. 6: see hmm_loss_warp_floats
};
BackwardShape circuit_backward_shape(const mtpc_head* h, bool loss) {
  const mtpc_config& c = h->cfg;
  const size_t shared = c.family == MTPC_HMM && !is_ctx(h) ? static_cast<size_t>(c.n - 1) * c.r * c.r : 0;   // the CTA's dT
  auto fit = [&](size_t per_warp) {
    for (int w = kCircuitWarps; w >= 1; w >>= 1)
      if ((shared + w * per_warp) * sizeof(float) <= static_cast<size_t>(kSmemLimit)) return w;
    return 0;
  };
  auto shape = [&](size_t per_warp, bool wide) {
    const int w = fit(per_warp);
    return BackwardShape{w, (shared + w * per_warp) * sizeof(float), wide};
  };
  if (c.family == MTPC_BTREE) return shape(btree_backward_warp_floats(c.n, c.r), false);
  if (c.family == MTPC_CP) return shape(loss ? cp_loss_warp_floats(c.n, c.r) : 0, false);
  const BackwardShape compact = shape(hmm_backward_warp_floats(c.n, c.r), false);
  if (!loss) return compact;
  const BackwardShape wide = shape(hmm_loss_warp_floats(c.n, c.r, true), true);
  return wide.warps >= compact.warps ? wide : compact;
}

// Warps (windows at a time) of a CTA of the static HMM's Eq. 6 kernel: the running sums of all n - 1 tables lie in shared memory beside the
// tables themselves, so few fit for long windows (at r = 32 sixteen up to n = 16, eight up to n = 21, four up to n = 24); 0: the streaming
// kernel. Four warps still win, and so do few windows, which sixteen warps a CTA leave on few SMs. Whole training calls of small heads (d = 64),
// streaming / so, in us: n = 24, r = 32 at 50 windows 202 / 105, 500 271 / 168, 2000 664 / 541; n = 20 at 100 180 / 94; n = 8 at 30 88 / 56,
// 200 109 / 64, 1500 181 / 129, 8192 677 / 514; n = 8, r = 16 at 200 76 / 51; n = 4, r = 8 at 40 45 / 38.
size_t hmm_static_loss_smem(const mtpc_config& c, int warps) {
  const size_t tables = (static_cast<size_t>(c.n - 1) * c.r * c.r + 3) / 4 * 4;
  return (2 * tables + warps * hmm_static_loss_warp_floats(c.n, c.r)) * sizeof(float);
}
int hmm_static_loss_warps(const mtpc_head* h) {
  if (h->cfg.family != MTPC_HMM || is_ctx(h) || h->L.off_probA == 0) return 0;
  for (int w = kHmmStaticWarps; w >= 4; w >>= 1)
    if (hmm_static_loss_smem(h->cfg, w) <= static_cast<size_t>(kSmemLimit)) return w;
  return 0;
}

// a.coeff (Eq. 6: the weights [W, n] of the prefix log-marginals) chooses the kernels that give every prefix and the whole
// gradient in one launch; otherwise the gradient of sum_w a.weight[w] log q_w.
int launch_circuit_backward(mtpc_head* h, CircuitBackwardArgs a, float* dT, cudaStream_t st) {
  const mtpc_config& c = h->cfg;
  const Layout& L = h->L;
  a.G = at<float>(h, L.off_G);
  a.logw = at<float>(h, L.off_logw);
  a.n = c.n;
  a.r = c.r;
  a.sum_rows = L.sum_rows;
  unsigned* counter = at<unsigned>(h, L.off_status) + kWorkCounterWord;
  const bool loss = a.coeff != nullptr;
  const BackwardShape shape = circuit_backward_shape(h, loss);
  const int warps = shape.warps;
  if (warps == 0) return MTPC_ERR_UNSUPPORTED;
  const int blocks = (a.W + warps - 1) / warps;
  const int threads = warps * 32;
  const int resident = blocks < 8 * h->num_sms ? blocks : 8 * h->num_sms;
  const size_t smem = shape.smem;
  const int static_warps = loss ? hmm_static_loss_warps(h) : 0;
  if (c.family == MTPC_CP && loss) {
    launch_kernel(circuit_cp_loss_backward_kernel, blocks, threads, smem, st, overlapped(h), a);
  } else if (c.family == MTPC_CP) {
    launch_kernel(circuit_cp_backward_kernel, blocks, threads, smem, st, overlapped(h), a);
  } else if (c.family == MTPC_HMM && loss && static_warps > 0) {
    const size_t ssmem = hmm_static_loss_smem(c, static_warps);
    const int batches = (a.W + static_warps - 1) / static_warps;
    const int held = h->num_sms * (2 * (ssmem + 1024) <= static_cast<size_t>(kSmemLimit) ? 2 : 1);
    launch_kernel(circuit_hmm_static_loss_backward_kernel, batches < held ? batches : held, static_warps * 32, ssmem, st, overlapped(h), a,
                  at<float>(h, L.off_probA), hmm_tables(h), dT);
  } else if (c.family == MTPC_HMM && loss) {
    launch_kernel(circuit_hmm_loss_backward_kernel, resident, threads, smem, st, overlapped(h), a, hmm_tables(h),
                  hmm_table_stride(h), dT, counter, shape.wide ? 1 : 0);
  } else if (c.family == MTPC_HMM) {
    launch_kernel(circuit_hmm_backward_kernel, resident, threads, smem, st, overlapped(h), a, hmm_tables(h),
                  hmm_table_stride(h), dT, counter);
  } else if (loss) {
    const int tw = c.n / 2 < 8 ? c.n / 2 : 8;                             // a warp per node of the owners' level
    const bool fits = btree_loss_smem_floats(c.n, c.r, tw, true) * sizeof(float) <= static_cast<size_t>(kSmemLimit);
    const size_t tsmem = btree_loss_smem_floats(c.n, c.r, tw, fits) * sizeof(float);
    const int grid = a.W < sms_times_resident(h, tsmem) ? a.W : sms_times_resident(h, tsmem);
    // (Plainly since its sweep on log tables, whose CTAs crowded beside the projection's last ones: 350 -> 395 us at 4096 windows of a 16 x 32
    // head. For the present sweep it makes no difference there, whole calls plainly / as a dependent 9.66 / 9.71 ms, nor at 1000 windows, 2.56 /
    // 2.57; small calls would be shorter as dependents: 8 x 16 x 64, d = 512, 2000 windows 202 / 177 us, 4 x 8 x 256, d = 256, 200 windows 59 / 53.)
    auto* kernel = c.r == 32 ? circuit_btree_loss_backward_kernel<32> : c.r == 16 ? circuit_btree_loss_backward_kernel<16>
                   : c.r == 8 ? circuit_btree_loss_backward_kernel<8> : circuit_btree_loss_backward_kernel<0>;
    launch_kernel(kernel, grid, tw * 32, tsmem, st, /*dependent=*/false, a, fits ? 1 : 0);
  } else {
    launch_kernel(circuit_btree_backward_kernel, resident, threads, smem, st, overlapped(h), a, counter);
  }
  h->launches++;
  return check_launch();
}

// Shared-memory attributes of the circuit backward kernels (per function: always the full limit, see allow_full_smem).
int set_backward_attributes(const mtpc_head* head) {
  if (circuit_backward_shape(head, false).warps == 0) return MTPC_ERR_UNSUPPORTED;   // (the loss kernels fit where these do)
  bool ok = allow_full_smem(circuit_hmm_backward_kernel);
  ok &= allow_full_smem(circuit_cp_loss_backward_kernel);
  ok &= allow_full_smem(circuit_btree_loss_backward_kernel<32>) && allow_full_smem(circuit_btree_loss_backward_kernel<16>);
  ok &= allow_full_smem(circuit_btree_loss_backward_kernel<8>) && allow_full_smem(circuit_btree_loss_backward_kernel<0>);
  ok &= allow_full_smem(circuit_hmm_loss_backward_kernel);
  ok &= allow_full_smem(circuit_hmm_static_loss_backward_kernel);
  ok &= allow_full_smem(circuit_btree_backward_kernel);
  return ok ? MTPC_OK : MTPC_ERR_CUDA;
}

// Phases 3 and 4 of a backward call: the logit gradients (post, lse and the kept logits -> bf16 rows) and the plain GEMMs.
// The sum-unit logit gradients are already in place to the right of dlogit. Every GEMM operand is read where it lies:
// the weights and the hidden states in the caller's buffers, the gradient matrix along its rows or down its columns.
int backward_tail(mtpc_head* head, const BackwardLayout& B, uint8_t* bw, const void* hb, const int32_t* targets, int T,
                  float* d_hidden, float* dW_emit, float* dW_sum, PhaseTimer& pt, cudaStream_t st) {
  const mtpc_config& c = head->cfg;
  const Layout& L = head->L;
  __nv_bfloat16* dlogit = reinterpret_cast<__nv_bfloat16*>(bw + B.off_dlogit);
  const int Nc = static_cast<int>(B.Nc);
  pt.begin();
  LogitGradArgs la;
  la.logits = reinterpret_cast<const float*>(bw + B.off_logits);
  la.lse = reinterpret_cast<const float*>(bw + B.off_lse);
  la.post = reinterpret_cast<const float*>(bw + B.off_post);
  la.targets = targets;
  la.dlogit = dlogit;
  la.pitch = B.Kd;
  la.T = T; la.Nc = Nc; la.n = c.n; la.r = c.r; la.v = c.v;
  {
    const int col_blocks = (Nc / 8 + 255) / 256;
    int row_blocks = (16 * head->num_sms + col_blocks - 1) / col_blocks;   // enough CTAs to fill the device, each walks rows
    if (row_blocks > T) row_blocks = T;
    if (row_blocks > 65535) row_blocks = 65535;
    // not as a dependent: CTAs scheduled beside the circuit kernel's last ones would share a few SMs (517 us became 690 at 4096
    // positions of a 16 x 32 x 256 head); and loss_partial_kernel, which works before it waits, relies on it (launch_clusters)
    launch_kernel(logit_gradient_kernel, dim3(col_blocks, row_blocks), 256, 0, st, /*dependent=*/false, la);
  }
  head->launches++;
  int rc = check_launch();
  pt.end();
  if (rc != MTPC_OK) return rc;
  pt.begin();
  const GemmOperand g_rows{dlogit, B.Kd, false};            // [T, Nc | S r] along its rows: K = the logit index
  const GemmOperand g_cols{dlogit, B.Kd, true};             // the same matrix down its columns: K = the position
  const GemmOperand w_emit{head->W_emit_bf16, static_cast<size_t>(c.d), true};   // [Nc, d]: N = d contiguous
  const GemmOperand w_sum{head->W_sum_bf16, static_cast<size_t>(c.d), true};
  const GemmOperand hid{hb, static_cast<size_t>(c.d), true};                     // [T, d]: N = d contiguous, K = the position
  // d hidden [T, d] = dlogit [T, Nc] W_emit [Nc, d] + dsum [T, S r] W_sum [S r, d]
  rc = launch_plain_gemm(head, g_rows, w_emit, Nc, w_sum, L.sum_rows, Nc, d_hidden, c.d, T, c.d, st,
                         SplitScratch{bw + B.off_split, B.parts});
  // [dW_emit; dW_sum] [Nc + S r, d] = [dlogit | dsum]^T hidden [T, d]
  PlainGemmExtra two;
  two.C2 = dW_sum;
  two.m1 = Nc;
  if (rc == MTPC_OK)
    rc = launch_plain_gemm(head, g_cols, hid, T, hid, 0, 0, dW_emit, c.d, Nc + L.sum_rows, c.d, st, SplitScratch{bw + B.off_split, B.parts}, nullptr, 0, &two);
  pt.end();
  return rc;
}

// Backward workspace of a factored head: the dense layout without kept logits (log-sum-exps, posteriors, logit gradients), then
//   sy    [T, n v | n r k | S r padded] bf16: the logit gradients summed over a slot's components, multiplied by the
//         adaptors A, and those of the sum units: the A operand of d hidden and of the three weight-gradient GEMMs;
//   apad  [n r, v rounded up to 64, k] bf16: A with zero rows between the units.
struct LowRankBackwardLayout {
  BackwardLayout B;
  size_t Ksy, pitch, v64;
  size_t off_sy, off_apad, total;
};
void plan_lowrank_backward(const mtpc_config& c, const Layout& L, int k, int T, LowRankBackwardLayout* R) {
  plan_backward(c, L, T, &R->B, k);
  const size_t units = static_cast<size_t>(c.n) * c.r;
  R->Ksy = static_cast<size_t>(c.n) * c.v + units * k;
  R->pitch = R->Ksy + R->B.Spad;
  R->v64 = round64(c.v);
  size_t off = R->B.total;
  auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes); return o; };
  R->off_sy = take(static_cast<size_t>(T) * R->pitch * 2);
  R->off_apad = take(units * R->v64 * k * 2);
  R->total = off;
}

// Phases 3 and 4 of a training call on a factored head: logit gradients g [T, n r v] (bf16), their sum over a slot's
// components, the zero-padded A; then the GEMMs. The sum units' logit gradients are already in the
// right-hand columns of sy.
int launch_adaptor_grad(mtpc_head* h, const __nv_bfloat16* g, size_t g_pitch, int Nc, const void* a_pad, int v64, __nv_bfloat16* y,
                        size_t y_pitch, float* dA, int T, cudaStream_t st) {
  const mtpc_config& c = h->cfg;
  AdaptorGradParams p;
  memset(&p, 0, sizeof(p));
  p.units = c.n * c.r;
  p.T = T;
  p.v = c.v;
  p.v64 = v64;
  p.k = h->lr_k;
  const int ctl = 1024 + static_cast<int>(sizeof(GemmControl));
  p.stages = (kSmemLimit - ctl - static_cast<int>(adaptor_fixed_bytes(v64))) / static_cast<int>(kAdaptorStage);
  if (p.stages < 2) return MTPC_ERR_UNSUPPORTED;
  const uint64_t z_cols = static_cast<uint64_t>(p.units) * 2 * p.k;
  int rc = make_tmap(&p.tm_g, g, T, Nc, kBlockM, g_pitch);
  if (rc == MTPC_OK) rc = make_tmap(&p.tm_z, h->ws + h->lr_off_zhl, T, z_cols, kBlockM, z_cols);
  if (rc == MTPC_OK) rc = make_tmap_mn(&p.tm_a, a_pad, static_cast<uint64_t>(p.units) * v64, p.k, p.k);
  if (rc != MTPC_OK) return rc;
  p.y = y;
  p.y_pitch = y_pitch;
  p.dA = dA;
  p.status = at<unsigned>(h, h->L.off_status);
  p.wait_limit_ns = h->wait_limit_ns;
  launch_kernel(adaptor_grad_kernel, p.units < h->num_sms ? p.units : h->num_sms, kGemmThreads,
                p.stages * kAdaptorStage + adaptor_fixed_bytes(v64) + ctl, st, overlapped(h), p);
  h->launches++;
  return check_launch();
}

int lowrank_backward_tail(mtpc_head* head, const LowRankBackwardLayout& R, uint8_t* bw, const void* hb, const int32_t* targets,
                          int T, float* d_hidden, float* dW_base, float* dA, float* dB, float* dW_sum, PhaseTimer& pt,
                          cudaStream_t st) {
  const mtpc_config& c = head->cfg;
  const Layout& L = head->L;
  const BackwardLayout& B = R.B;
  const int k = head->lr_k, units = c.n * c.r;
  __nv_bfloat16* sy = reinterpret_cast<__nv_bfloat16*>(bw + R.off_sy);
  int rc = MTPC_OK;
  pt.begin();
  __nv_bfloat16* dlogit = reinterpret_cast<__nv_bfloat16*>(bw + B.off_dlogit);
  const int Nc = static_cast<int>(B.Nc);
  LowRankParams lp = head->lr_params;
  lp.targets = targets;
  lp.G = at<float>(head, L.off_G);
  lp.lse = reinterpret_cast<const float*>(bw + B.off_lse);
  lp.post = reinterpret_cast<const float*>(bw + B.off_post);
  if ((rc = make_tmap_unit_rows(&lp.tm_g, dlogit, static_cast<uint64_t>(T), static_cast<uint64_t>(units), static_cast<uint64_t>(c.v), B.Kd)) != MTPC_OK) return rc;
  lp.s = sy;
  lp.s_pitch = R.pitch;
  if ((rc = launch_lowrank_logits<kLowRankGradient>(head, lp, T, st)) != MTPC_OK) return rc;
  {
    const size_t pad_pieces = static_cast<size_t>(units) * R.v64 * (k / 8);
    launch_kernel(lowrank_pad_kernel, static_cast<unsigned>((pad_pieces + 255) / 256), 256, 0, st, overlapped(head),
                  static_cast<const uint4*>(head->lr_A), reinterpret_cast<uint4*>(bw + R.off_apad), units, c.v,
                  static_cast<int>(R.v64), k / 8);
  }
  head->launches += 1;
  if ((rc = check_launch()) != MTPC_OK) return rc;
  pt.end();
  // 4. the GEMMs
  pt.begin();
  const GemmOperand none{nullptr, 0, false};
  const GemmOperand hid{hb, static_cast<size_t>(c.d), true};
  // y_ij = g_ij A_ij [T, k] into the middle columns of sy and dA_ij [v, k] = g_ij^T z_ij from one reading of g, where a CTA can keep a
  // unit's A and there are units for at least half the SMs; else one batched product each
  const bool one_pass = c.v <= kAdaptorMaxV && 2 * units >= head->num_sms;
  if (one_pass) {
    rc = launch_adaptor_grad(head, dlogit, B.Kd, Nc, bw + R.off_apad, static_cast<int>(R.v64), sy + static_cast<size_t>(c.n) * c.v, R.pitch,
                             dA, T, st);
  } else {
    PlainGemmExtra x;
    x.C_bf16 = sy + static_cast<size_t>(c.n) * c.v;
    x.batches = units;
    x.a_k_step = c.v;
    x.b_k_step = static_cast<int>(R.v64);
    x.c_step = k;
    x.a_extent_m = T; x.a_extent_k = Nc;
    x.b_extent_n = k; x.b_extent_k = static_cast<long long>(units) * R.v64;
    rc = launch_plain_gemm(head, GemmOperand{dlogit, B.Kd, false}, GemmOperand{bw + R.off_apad, static_cast<size_t>(k), true},
                           static_cast<int>(R.v64), none, 0, 0, nullptr, R.pitch, T, k, st, SplitScratch{}, nullptr, 0, &x);
  }
  // d hidden [T, d] = s W_base + y B + dsum W_sum
  PlainGemmExtra tail;
  tail.B2 = GemmOperand{head->W_sum_bf16, static_cast<size_t>(c.d), true};
  tail.K2 = L.sum_rows;
  tail.a_k2 = static_cast<int>(R.Ksy);
  if (rc == MTPC_OK)
    rc = launch_plain_gemm(head, GemmOperand{sy, R.pitch, false}, GemmOperand{head->lr_W_base, static_cast<size_t>(c.d), true}, c.n * c.v,
                           GemmOperand{head->lr_B, static_cast<size_t>(c.d), true}, units * k, c.n * c.v, d_hidden, c.d, T, c.d, st,
                           SplitScratch{bw + B.off_split, B.parts}, nullptr, 0, &tail);
  // [dW_base; dB; dW_sum] = [s | y | dsum]^T h: sy down its columns
  PlainGemmExtra three;
  three.C2 = dB;
  three.m1 = c.n * c.v;
  three.C3 = dW_sum;
  three.m2 = static_cast<int>(R.Ksy);
  if (rc == MTPC_OK)
    rc = launch_plain_gemm(head, GemmOperand{sy, R.pitch, true}, hid, T, hid, 0, 0, dW_base, c.d, static_cast<int>(R.Ksy) + L.sum_rows,
                           c.d, st, SplitScratch{bw + B.off_split, B.parts}, nullptr, 0, &three);
  if (rc == MTPC_OK && !one_pass) {   // on the bf16 high half of z the forward pass left
    PlainGemmExtra x;
    x.batches = units;
    x.a_m_step = c.v;
    x.b_n_step = 2 * k;
    x.c_step = static_cast<size_t>(c.v) * k;
    x.a_extent_m = Nc; x.a_extent_k = T;
    x.b_extent_n = static_cast<long long>(units) * 2 * k; x.b_extent_k = T;
    rc = launch_plain_gemm(head, GemmOperand{dlogit, B.Kd, true},
                           GemmOperand{head->ws + head->lr_off_zhl, static_cast<size_t>(units) * 2 * k, true}, T, none, 0, 0, dA,
                           k, c.v, k, st, SplitScratch{}, nullptr, 0, &x);
  }
  pt.end();
  return rc;
}

int check_call(mtpc_head* h, int32_t rows) {
  if (!h) return MTPC_ERR_NULL;
  if (rows < 0 || rows > h->cfg.max_positions) return MTPC_ERR_SHAPE;
  return MTPC_OK;
}

}  // namespace

// The vector paths of the low-rank kernels need d a multiple of 4 and 16-byte aligned pointers.
static bool lowrank_vector_ok(int d, std::initializer_list<const void*> ptrs) {
  if (d % 4) return false;
  for (const void* p : ptrs)
    if (reinterpret_cast<uintptr_t>(p) % 16) return false;
  return true;
}

// Everything the head derives from the parameters: bf16 copies of fp32 weights, the tensor maps on the weight
// matrices, the log-softmaxed static HMM transitions or the contextual transition bias. Used at creation and again
// whenever the caller's parameters have changed (mtpc_update_parameters).
static int bind_parameters(mtpc_head* h, const void* W_emit, const void* W_sum, const float* T_static, cudaStream_t st) {
  const mtpc_config* cfg = &h->cfg;
  const Layout& L = h->L;
  const bool ctx = (cfg->flags & MTPC_FLAG_HMM_CONTEXTUAL) != 0;
  const size_t emit_count = static_cast<size_t>(cfg->n) * cfg->r * cfg->v * cfg->d;
  const size_t sum_count = static_cast<size_t>(L.sum_rows) * cfg->d;
  if (cfg->io_dtype == MTPC_F32) {
    round_to_bf16(static_cast<const float*>(W_emit), at<__nv_bfloat16>(h, L.off_wemit), emit_count, st, false);
    round_to_bf16(static_cast<const float*>(W_sum), at<__nv_bfloat16>(h, L.off_wsum), sum_count, st, false);
    h->launches += 2;
    h->W_emit_bf16 = h->ws + L.off_wemit;
    h->W_sum_bf16 = h->ws + L.off_wsum;
  } else {
    h->W_emit_bf16 = W_emit;
    h->W_sum_bf16 = W_sum;
  }
  if (ctx) {
    // bias of the contextual transition logits, laid out like the sum-unit rows: zeros for the initial unit
    bool bad = cudaMemsetAsync(h->ws + L.off_sum_bias, 0, static_cast<size_t>(L.sum_rows) * 4, st) != cudaSuccess;
    if (T_static && cfg->n > 1)
      bad |= cudaMemcpyAsync(h->ws + L.off_sum_bias + static_cast<size_t>(cfg->r) * 4, T_static,
                             static_cast<size_t>(cfg->n - 1) * cfg->r * cfg->r * 4, cudaMemcpyDeviceToDevice,
                             st) != cudaSuccess;
    if (bad) return MTPC_ERR_CUDA;
  } else if (cfg->family == MTPC_HMM && cfg->n > 1) {
    const int rows = (cfg->n - 1) * cfg->r;
    static_tables_kernel<<<(rows + 7) / 8, 256, 0, st>>>(T_static, at<float>(h, L.off_logA), at<float>(h, L.off_probA),
                                                         at<float>(h, L.off_cdfA), rows, cfg->r);
    h->launches++;
  }
  if (check_launch() != MTPC_OK) return MTPC_ERR_CUDA;
  const uint64_t emit_rows = static_cast<uint64_t>(cfg->n) * cfg->r * cfg->v;
  const bool dense = h->lr_k == 0;      // a factored low-rank head has no composed W_emit: only the sum-unit maps
  int rc = MTPC_OK;
  if (dense) rc = make_tmap(&h->tm_emit_lp, h->W_emit_bf16, emit_rows, cfg->d, L.lp.tile_cols);
  if (rc == MTPC_OK) rc = make_tmap(&h->tm_sum, h->W_sum_bf16, L.sum_rows, cfg->d, L.sum_cols);
  if (rc == MTPC_OK && dense) rc = make_tmap(&h->tm_emit_lp2, h->W_emit_bf16, emit_rows, cfg->d, L.lp.tile_cols / 2);
  if (rc == MTPC_OK) rc = make_tmap(&h->tm_sum2, h->W_sum_bf16, L.sum_rows, cfg->d, L.sum_cols / 2);
  const uint64_t base_rows = static_cast<uint64_t>(cfg->n) * cfg->v, adapt_rows = static_cast<uint64_t>(cfg->n) * cfg->r * h->lr_k;
  choose_decode_tiling(static_cast<long long>(dense ? emit_rows : base_rows + adapt_rows), L.sum_rows, L.decode_max_p, cfg->d / kBlockK, h->num_sms,
                       h->max_decode_clusters, &h->decode_tile_rows, &h->decode_ksplit);
  if (rc == MTPC_OK && dense) rc = make_tmap(&h->tm_emit_dec, h->W_emit_bf16, emit_rows, cfg->d, h->decode_tile_rows);
  if (rc == MTPC_OK && !dense) rc = make_tmap(&h->tm_emit_dec, h->lr_W_base, base_rows, cfg->d, h->decode_tile_rows);
  if (rc == MTPC_OK && !dense) rc = make_tmap(&h->tm_lrB_dec, h->lr_B, adapt_rows, cfg->d, h->decode_tile_rows);
  h->decode_sum_tile_rows = h->decode_tile_rows / 32 * 32;   // whole groups of r <= 32 rows per warp; fits the tile pitch
  if (rc == MTPC_OK) rc = make_tmap(&h->tm_sum_dec, h->W_sum_bf16, L.sum_rows, cfg->d, h->decode_sum_tile_rows);
  h->draft_P = 0;                                              // logits left by an earlier draft belong to the old parameters
  return rc;
}

extern "C" {

int mtpc_workspace_bytes(const mtpc_config* cfg, size_t* out_bytes) {
  if (!cfg || !out_bytes) return MTPC_ERR_NULL;
  Layout L;
  int rc = plan(*cfg, &L);
  if (rc != MTPC_OK) return rc;
  *out_bytes = L.total;
  return MTPC_OK;
}

// lowrank: NULL for a dense head; else the rank and the three parameter tensors of App. G (W_emit is NULL then).
struct LowRankSpec {
  int k;
  const void* W_base;
  const void* A;
  const void* B;
};

// Workspace of a factored head beyond the dense layout: z = B h as two bf16 halves [T, n r, 2, k] (written by the GEMM
// that computes it), W_base h, the log-sums of 32 columns each with their references, and the copy of A the factored kernel reads.
static int lowrank_extra_bytes(const mtpc_config& c, int k, size_t base_total, size_t* off_zhl,
                               size_t* off_partial, size_t* off_arep, size_t* off_dec, size_t* off_base, size_t* off_split, int* parts, size_t* total) {
  const size_t units = static_cast<size_t>(c.n) * c.r;
  size_t off = align_up(base_total);
  *off_zhl = off;
  off += align_up(static_cast<size_t>(c.max_positions) * units * 2 * k * 2);
  *off_partial = off;
  off += align_up(static_cast<size_t>((c.max_positions + 31) / 32 * 32) * (units + c.n) * ((c.v + 31) / 32) * sizeof(float));
  *off_arep = off;                      // the copy of A laid out [n, v, r, k]
  off += align_up(units * c.v * k * 2);
  *off_dec = off;                       // few-position draft: base = W_base h [P, n v] and z = B h [P, n r k], fp32
  off += align_up(static_cast<size_t>(c.max_positions < kDecodeMaxP ? c.max_positions : kDecodeMaxP) *
                  (static_cast<size_t>(c.n) * c.v + units * k) * 4);
  *off_base = off;                      // W_base h [T, n v] fp32
  off += align_up(static_cast<size_t>(c.max_positions) * c.n * c.v * 4);
  *off_split = off;                     // z = B h and W_base h: parts of the tiles of their last rounds
  *parts = 0;
  const int m_tiles = (c.max_positions - 1) / kBlockM + 1, period = 148;      // (the last rounds repeat with it, see split_parts)
  for (int m = 1; m <= m_tiles && m <= period; ++m) {
    const int w = split_parts(static_cast<size_t>(m) * kBlockM, c.n * c.v, c.d / kBlockK);
    const int z = split_parts(static_cast<size_t>(m) * kBlockM, static_cast<int>(units) * k, c.d / kBlockK);
    if (w > *parts) *parts = w;
    if (z > *parts) *parts = z;
  }
  off += align_up(*parts * kSplitPartBytes);
  *total = off;
  return MTPC_OK;
}

static int create_head_impl(const mtpc_config* cfg, const void* W_emit, const LowRankSpec* lowrank, const void* W_sum,
                            const float* T_static, void* workspace, size_t workspace_bytes, void* stream, mtpc_head** out) {
  if (!cfg || !W_sum || !workspace || !out) return MTPC_ERR_NULL;
  if (!lowrank && !W_emit) return MTPC_ERR_NULL;
  if (lowrank && (!lowrank->W_base || !lowrank->A || !lowrank->B)) return MTPC_ERR_NULL;
  *out = nullptr;
  Layout L;
  int rc = plan(*cfg, &L, lowrank != nullptr);
  if (rc != MTPC_OK) return rc;
  LowRankParams lrp;
  memset(&lrp, 0, sizeof(lrp));
  size_t lr_zhl = 0, lr_partial = 0, lr_arep = 0, lr_dec = 0, lr_base = 0, lr_split = 0;
  int lr_parts = 0;
  if (lowrank) {
    if (cfg->io_dtype != MTPC_BF16) return MTPC_ERR_UNSUPPORTED;
    if (!plan_lowrank(*cfg, lowrank->k, &lrp)) return MTPC_ERR_UNSUPPORTED;
    lowrank_extra_bytes(*cfg, lowrank->k, L.total, &lr_zhl, &lr_partial, &lr_arep, &lr_dec, &lr_base,
                        &lr_split, &lr_parts, &L.total);
  }
  const bool ctx = (cfg->flags & MTPC_FLAG_HMM_CONTEXTUAL) != 0;
  if (cfg->family == MTPC_HMM && cfg->n > 1 && !ctx && !T_static) return MTPC_ERR_NULL;
  if (workspace_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) % kAlign) != 0) return MTPC_ERR_WORKSPACE;
  int dev = 0, cc_major = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MTPC_ERR_CUDA;
  if (cudaDeviceGetAttribute(&cc_major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess || cc_major != 10)
    return MTPC_ERR_CUDA;   // tcgen05 / TMEM code: sm_100 only
  mtpc_head* h = new (std::nothrow) mtpc_head;
  if (!h) return MTPC_ERR_CUDA;
  memset(h, 0, sizeof(*h));
  h->cfg = *cfg;
  h->L = L;
  h->ws = static_cast<uint8_t*>(workspace);
  h->wait_limit_ns = kWaitLimitNs;
  if (lowrank) {
    h->lr_k = lowrank->k;
    h->lr_W_base = lowrank->W_base;
    h->lr_A = lowrank->A;
    h->lr_B = lowrank->B;
    h->lr_off_zhl = lr_zhl;
    h->lr_off_partial = lr_partial;
    h->lr_off_arep = lr_arep;
    h->lr_off_dec = lr_dec;
    h->lr_off_base = lr_base;
    h->lr_off_split = lr_split;
    h->lr_split_parts = lr_parts;
    h->lr_params = lrp;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  bool fail = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess;
  // the attribute is per function, not per head: always ask for the full 227 KB so that heads do not undo each other
  fail |= !allow_full_smem(mtpc_gemm_kernel<kModeLogprob, 1, 16>) || !allow_full_smem(mtpc_gemm_kernel<kModeLogprob, 1, 32>);
  fail |= !allow_full_smem(mtpc_gemm_kernel<kModeLogitsGrouped, 1, 16>);
  fail |= !allow_full_smem(mtpc_gemm_kernel<kModeLogprob, 2, 16>) || !allow_full_smem(mtpc_gemm_kernel<kModeLogprob, 2, 32>);
  h->max_pairs = fail ? 0 : resident_clusters(mtpc_gemm_kernel<kModeLogprob, 2, 16>, 2, gemm_threads(kModeLogprob), 0, dev);
  fail |= !allow_full_smem(plain_gemm_kernel<false, false>);
  fail |= !allow_full_smem(plain_gemm_kernel<false, true>);
  fail |= !allow_full_smem(plain_gemm_kernel<true, true>);
  fail |= !allow_full_smem(plain_gemm_kernel<false, false, kPlainTileN, 2>);
  fail |= !allow_full_smem(plain_gemm_kernel<false, true, kPlainTileN, 2>);
  fail |= !allow_full_smem(plain_gemm_kernel<true, true, kPlainTileN, 2>);
  fail |= !allow_full_smem(plain_gemm_kernel<true, true, 64>);
  fail |= !allow_full_smem(plain_gemm_kernel<false, true, 64>);
  fail |= !allow_full_smem(adaptor_grad_kernel);
  fail |= cudaFuncSetAttribute(mtpc_decode_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) !=
          cudaSuccess;
  for (int e = 0; e < 3; ++e) h->max_decode_clusters[e] = fail ? 0 : resident_clusters(mtpc_decode_gemm_kernel, 2 << e, kGemmThreads, 1 + e, dev);
  const int slot_smem = static_cast<int>(kSlotSmemLimit);
  for (auto* kernel : {draft_slot_kernel<false, 4, 2>, draft_slot_kernel<false, 8, 2>, draft_slot_kernel<false, 10, 2>, draft_slot_kernel<false, 16, 2>,
                       draft_slot_kernel<false, 4, 3>, draft_slot_kernel<false, 8, 3>, draft_slot_kernel<false, 10, 3>, draft_slot_kernel<true, 16, 2>})
    fail |= cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, slot_smem) != cudaSuccess;
  fail |= !set_circuit_attributes() || !allow_full_smem(latent_sample_kernel);
  fail |= !allow_full_smem(spec_accept_kernel<true>) || !allow_full_smem(spec_accept_kernel<false>);
  fail |= cudaMemsetAsync(h->ws + L.off_status, 0, 256, st) != cudaSuccess;
  if (fail) { delete h; return MTPC_ERR_CUDA; }

  rc = bind_parameters(h, W_emit, W_sum, T_static, st);
  if (rc == MTPC_OK && lowrank) {
    fail = !allow_full_smem(lowrank_logits_kernel<kLowRankForward>);
    fail |= !allow_full_smem(lowrank_logits_kernel<kLowRankGradient>);
    if (fail) rc = MTPC_ERR_CUDA;
    if (rc == MTPC_OK)
      rc = make_tmap(&h->lr_tm_a, h->ws + h->lr_off_arep, static_cast<uint64_t>(cfg->n) * cfg->v,
                     static_cast<uint64_t>(cfg->r) * lowrank->k, kLrCols);
  }
  if (rc != MTPC_OK) { delete h; return rc; }
  *out = h;
  return MTPC_OK;
}

int mtpc_create_head(const mtpc_config* cfg, const void* W_emit, const void* W_sum, const float* T_static,
                     void* workspace, size_t workspace_bytes, void* stream, mtpc_head** out) {
  if (!W_emit) return MTPC_ERR_NULL;
  return create_head_impl(cfg, W_emit, nullptr, W_sum, T_static, workspace, workspace_bytes, stream, out);
}

int mtpc_lowrank_workspace_bytes(const mtpc_config* cfg, int32_t k, size_t* out_bytes) {
  if (!cfg || !out_bytes) return MTPC_ERR_NULL;
  Layout L;
  int rc = plan(*cfg, &L, /*factored=*/true);
  if (rc != MTPC_OK) return rc;
  LowRankParams lrp;
  if (cfg->io_dtype != MTPC_BF16 || !plan_lowrank(*cfg, k, &lrp)) return MTPC_ERR_UNSUPPORTED;
  size_t a = 0, b = 0, c3 = 0, c4 = 0, c5 = 0, c6 = 0;
  int parts = 0;
  return lowrank_extra_bytes(*cfg, k, L.total, &a, &b, &c3, &c4, &c5, &c6, &parts, out_bytes);
}

int mtpc_create_head_lowrank(const mtpc_config* cfg, int32_t k, const void* W_base, const void* A, const void* B,
                             const void* W_sum, const float* T_static, void* workspace, size_t workspace_bytes,
                             void* stream, mtpc_head** out) {
  const LowRankSpec spec{k, W_base, A, B};
  return create_head_impl(cfg, nullptr, &spec, W_sum, T_static, workspace, workspace_bytes, stream, out);
}


int mtpc_update_parameters(mtpc_head* head, const void* W_emit, const void* W_sum, const float* T_static, void* stream) {
  if (!head || !W_sum || (!W_emit && head->lr_k == 0)) return MTPC_ERR_NULL;   // a factored head has no W_emit to rebind
  const mtpc_config& c = head->cfg;
  if (c.family == MTPC_HMM && c.n > 1 && !(c.flags & MTPC_FLAG_HMM_CONTEXTUAL) && !T_static) return MTPC_ERR_NULL;
  return bind_parameters(head, W_emit, W_sum, T_static, static_cast<cudaStream_t>(stream));
}

int mtpc_window_logprob(mtpc_head* head, const void* hidden, const int32_t* targets, int32_t T, float* out_logprob,
                        void* stream) {
  int rc = check_call(head, T);
  if (rc != MTPC_OK) return rc;
  if (T == 0) return MTPC_OK;
  if (!hidden || !targets || !out_logprob) return MTPC_ERR_NULL;
  return window_logprob_impl(head, hidden, targets, T, out_logprob, nullptr, static_cast<cudaStream_t>(stream));
}

int mtpc_window_prefix_logprob(mtpc_head* head, const void* hidden, const int32_t* targets, int32_t T,
                               float* out_prefix_logprob, void* stream) {
  int rc = check_call(head, T);
  if (rc != MTPC_OK) return rc;
  if (T == 0) return MTPC_OK;
  if (!hidden || !targets || !out_prefix_logprob) return MTPC_ERR_NULL;
  return window_logprob_impl(head, hidden, targets, T, nullptr, out_prefix_logprob, static_cast<cudaStream_t>(stream));
}

int mtpc_draft_sample(mtpc_head* head, const void* hidden, int32_t P, int32_t wpp, const float* uniforms,
                      int32_t* out_bytes, float* out_logprob, void* stream) {
  int rc = check_call(head, P);
  if (rc != MTPC_OK) return rc;
  if (wpp < 1 || wpp > head->cfg.max_windows_per_pos) return MTPC_ERR_SHAPE;
  if (P == 0) return MTPC_OK;
  if (!hidden || !uniforms || !out_bytes || !out_logprob) return MTPC_ERR_NULL;
  return draft_sample_impl(head, hidden, P, wpp, uniforms, out_bytes, out_logprob, nullptr,
                           static_cast<cudaStream_t>(stream));
}

int mtpc_draft_sample_prefix(mtpc_head* head, const void* hidden, int32_t P, int32_t wpp, const float* uniforms,
                             int32_t* out_bytes, float* out_prefix_logprob, void* stream) {
  int rc = check_call(head, P);
  if (rc != MTPC_OK) return rc;
  if (wpp < 1 || wpp > head->cfg.max_windows_per_pos) return MTPC_ERR_SHAPE;
  if (P == 0) return MTPC_OK;
  if (!hidden || !uniforms || !out_bytes || !out_prefix_logprob) return MTPC_ERR_NULL;
  return draft_sample_impl(head, hidden, P, wpp, uniforms, out_bytes, nullptr, out_prefix_logprob,
                           static_cast<cudaStream_t>(stream));
}

int mtpc_speculative_accept(mtpc_head* head, int32_t P, int32_t wpp, const int32_t* draft_bytes,
                            const float* prefix_logprob, const float* target_probs, const float* accept_uniforms,
                            int32_t* out_accepted, int32_t* out_next_byte, void* stream) {
  int rc = check_call(head, P);
  if (rc != MTPC_OK) return rc;
  if (wpp < 1 || wpp > head->cfg.max_windows_per_pos) return MTPC_ERR_SHAPE;
  if (P == 0) return MTPC_OK;
  if (!draft_bytes || !prefix_logprob || !target_probs || !accept_uniforms || !out_accepted || !out_next_byte)
    return MTPC_ERR_NULL;
  if (head->draft_P != P || head->draft_wpp != wpp) return MTPC_ERR_STATE;
  const mtpc_config& c = head->cfg;
  const Layout& L = head->L;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int W = P * wpp;
  const size_t smem = accept_smem_floats(c.r, c.v) * sizeof(float);
  if (smem > static_cast<size_t>(kSmemLimit)) return MTPC_ERR_UNSUPPORTED;      // a residual row of more than ~56k symbols
  const int threads = accept_threads(c.v);
  auto* accept_kernel = W <= head->num_sms ? spec_accept_kernel<true> : spec_accept_kernel<false>;
  PhaseTimer pt(head, st);
  float* const msg = at<float>(head, L.off_msg);
  // The slot messages are formed here, from the evidence and log omega the draft left, unless they are sure to be the last draft's
  // when this call runs: formed by a call of the same capture, or outside any while no draft of joints has been recorded. (A
  // recorded call runs after drafts the host does not see.)
  const unsigned long long capture = capture_id(st);
  if (!head->draft_msg || head->draft_capture != capture || (capture == 0 && head->joint_recorded)) {
    rc = launch_circuit(head, W, wpp, nullptr, nullptr, st, /*raw_mixture=*/P <= L.decode_max_p && c.r > 32, msg);
    if (rc != MTPC_OK) return rc;
    head->draft_msg = true;
    head->draft_capture = capture;
  }
  if (head->draft_logits) {
    // every logit of the drafted positions is still in the workspace
    pt.begin();
    launch_kernel(accept_kernel, W, threads, smem, st, overlapped(head), at<float>(head, L.off_logits),
                  at<float>(head, L.off_unit_lse), msg, draft_bytes, prefix_logprob, target_probs, accept_uniforms, out_accepted,
                  out_next_byte, at<unsigned>(head, L.off_status), W, wpp, c.n, c.r, c.v, valid_symbols(c),
                  static_cast<const int*>(nullptr));
    head->launches++;
    pt.end();
    return check_launch();
  }
  // A draft that ran in chunks kept the last one's logits only (a factored head's long draft none). The evidence of the drafted bytes (G) and log omega are still in
  // the workspace; what is missing is, for every window rejected at byte s, the r v logits of slot s. So: run the tests,
  // sort the rejected windows by s, stage their hidden states, recompute those logits with one sorted projection pass,
  // then run the acceptance kernel on them. In chunks of positions whose windows fit the scratch.
  const bool factored = head->lr_k > 0;     // (a long draft on a factored head left W_base h and B h instead of needing the hidden states)
  if (L.accept_rows == 0 || (!factored && !head->draft_hidden)) return MTPC_ERR_UNSUPPORTED;
  if (factored && c.v > kMaxDraftVocab) return MTPC_ERR_UNSUPPORTED;
  int* ints = at<int>(head, L.off_grp_ints);
  int* counts = ints, *cursors = ints + c.n, *offsets = ints + 2 * c.n, *num_tiles = ints + 3 * c.n;
  GroupTile* tiles = at<GroupTile>(head, L.off_grp_tiles);
  __nv_bfloat16* stage = at<__nv_bfloat16>(head, L.off_grp_stage);
  int* rej = at<int>(head, L.off_acc_rej);
  int* row_of = at<int>(head, L.off_acc_row);
  float* lg = at<float>(head, L.off_acc_logits);
  float* lse = at<float>(head, L.off_acc_lse);
  const int chunk_pos = static_cast<int>(L.accept_rows / wpp);                  // >= 1 by construction
  for (int p0 = 0; p0 < P; p0 += chunk_pos) {
    const int pc = P - p0 < chunk_pos ? P - p0 : chunk_pos;
    const int wc = pc * wpp;
    const size_t w0 = static_cast<size_t>(p0) * wpp;
    const int32_t* xb = draft_bytes + w0 * c.n;
    const float* pre = prefix_logprob + w0 * c.n;
    const float* tp = target_probs + w0 * (c.n + 1) * c.v;
    const float* ua = accept_uniforms + w0 * (c.n + 1);
    pt.begin();
    launch_kernel(accept_test_kernel, (wc + 7) / 8, 256, 0, st, overlapped(head), xb, pre, tp, ua, rej, wc, c.n, c.v,
                  valid_symbols(c));
    if (factored) {
      // the slot's logits from W_base h and B h, window by window: no sort, no staging, no projection pass
      const int pairs = wc * c.r;
      int blocks = (pairs + kDrawWarps - 1) / kDrawWarps;
      if (blocks > 32 * head->num_sms) blocks = 32 * head->num_sms;
      launch_kernel(lowrank_slot_logits_kernel, blocks, 32 * kDrawWarps, 0, st, overlapped(head),
                    reinterpret_cast<const float*>(head->ws + head->lr_off_base),
                    reinterpret_cast<const __nv_bfloat16*>(head->ws + head->lr_off_zhl),
                    static_cast<const __nv_bfloat16*>(head->lr_A), rej, lg, lse, row_of, wc, static_cast<int>(w0), wpp, c.n,
                    c.r, c.v, valid_symbols(c), head->lr_k);
      head->launches += 2;
      pt.end();
      int rcf = check_launch();
      if (rcf != MTPC_OK) return rcf;
      pt.begin();
      launch_kernel(accept_kernel, wc, threads, smem, st, overlapped(head), lg, lse, msg + w0 * c.n * c.r, xb,
                    pre, tp, ua, out_accepted + w0, out_next_byte + w0, at<unsigned>(head, L.off_status), wc, wpp, c.n, c.r, c.v,
                    valid_symbols(c), row_of);
      head->launches++;
      pt.end();
      if ((rcf = check_launch()) != MTPC_OK) return rcf;
      continue;
    }
    if (cudaMemsetAsync(ints, 0, static_cast<size_t>(2 * c.n) * 4, st) != cudaSuccess) return MTPC_ERR_CUDA;
    const int cblocks = (wc + kGroupThreads - 1) / kGroupThreads;
    group_count_kernel<<<cblocks < 4 * head->num_sms ? cblocks : 4 * head->num_sms, kGroupThreads, c.n * sizeof(int), st>>>(
        rej, counts, wc, c.n);
    group_scan_kernel<<<1, kGroupScanThreads, 0, st>>>(counts, offsets, tiles, num_tiles, c.n);
    const int gblocks = (wc + kGroupThreads / 32 - 1) / (kGroupThreads / 32);
    group_gather_kernel<<<gblocks < 16 * head->num_sms ? gblocks : 16 * head->num_sms, kGroupThreads, 0, st>>>(
        rej, static_cast<const __nv_bfloat16*>(head->draft_hidden) + static_cast<size_t>(p0) * c.d, offsets, cursors, stage,
        wc, wpp, c.d, row_of);
    head->launches += 4;
    int rc2 = check_launch();
    if (rc2 != MTPC_OK) return rc2;
    GroupArgs ga;
    ga.stage = stage;
    ga.entries = wc;
    ga.tiles = tiles;
    ga.num_tiles = num_tiles;
    ga.max_tiles = c.n + wc / 128 + 1;
    GradArgs out;
    out.lse_out = lse;
    out.logit_out = lg;
    out.logit_pitch = static_cast<size_t>(c.r) * c.v;
    rc2 = launch_gemm(head, head->draft_hidden, pc, true, false, nullptr, st, &out, &ga);
    pt.end();
    if (rc2 != MTPC_OK) return rc2;
    pt.begin();
    launch_kernel(accept_kernel, wc, threads, smem, st, overlapped(head), lg, lse, msg + w0 * c.n * c.r, xb,
                  pre, tp, ua, out_accepted + w0, out_next_byte + w0, at<unsigned>(head, L.off_status), wc, wpp, c.n, c.r, c.v,
                  valid_symbols(c), row_of);
    head->launches++;
    pt.end();
    if ((rc2 = check_launch()) != MTPC_OK) return rc2;
  }
  return MTPC_OK;
}

int mtpc_window_loss(mtpc_head* head, const void* hidden, const int32_t* targets, int32_t num_sequences,
                     int32_t sequence_length, float gamma, float* out_slot_loss, float* out_loss, void* stream) {
  if (!head) return MTPC_ERR_NULL;
  if (num_sequences < 1 || sequence_length < 1) return MTPC_ERR_SHAPE;
  const int64_t T64 = static_cast<int64_t>(num_sequences) * sequence_length;
  if (T64 > head->cfg.max_positions) return MTPC_ERR_SHAPE;
  if (!hidden || !targets || !out_slot_loss || !out_loss) return MTPC_ERR_NULL;
  const int T = static_cast<int>(T64);
  const Layout& L = head->L;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  float* prefix = at<float>(head, L.off_prefix);
  float* partial = at<float>(head, L.off_partial);
  int rc = window_logprob_impl(head, hidden, targets, T, nullptr, prefix, st);   // phases 0 and 1
  if (rc != MTPC_OK) return rc;
  launch_kernel(loss_partial_kernel, num_sequences, kLossThreads, 0, st, overlapped(head), prefix, targets, partial,
                sequence_length, head->cfg.n, 0);
  launch_kernel(loss_final_kernel, 1, kLossThreads, 0, st, overlapped(head), partial, out_slot_loss, out_loss, num_sequences,
                head->cfg.n, gamma);
  head->launches += 2;
  return check_launch();
}

int mtpc_backward_workspace_bytes(const mtpc_config* cfg, int32_t T, size_t* out_bytes) {
  if (!cfg || !out_bytes) return MTPC_ERR_NULL;
  if (T < 1) return MTPC_ERR_SHAPE;
  Layout L;
  int rc = plan(*cfg, &L);
  if (rc != MTPC_OK) return rc;
  BackwardLayout B;
  plan_backward(*cfg, L, T, &B);
  *out_bytes = B.total;
  return MTPC_OK;
}

int mtpc_window_logprob_backward(mtpc_head* head, const void* hidden, const int32_t* targets, int32_t T,
                                 const float* weight, void* bwd_workspace, size_t bwd_workspace_bytes,
                                 float* out_logprob, float* d_hidden, float* dW_emit, float* dW_sum, float* dT_static,
                                 void* stream) {
  int rc = check_call(head, T);
  if (rc != MTPC_OK) return rc;
  if (T == 0) return MTPC_OK;
  if (!hidden || !targets || !weight || !bwd_workspace || !d_hidden || !dW_emit || !dW_sum) return MTPC_ERR_NULL;
  if (head->lr_k > 0) return MTPC_ERR_UNSUPPORTED;
  const mtpc_config& c = head->cfg;
  const bool static_hmm = c.family == MTPC_HMM && !is_ctx(head) && c.n > 1;
  if (static_hmm && !dT_static) return MTPC_ERR_NULL;
  BackwardLayout B;
  plan_backward(c, head->L, T, &B);
  if (bwd_workspace_bytes < B.total || (reinterpret_cast<uintptr_t>(bwd_workspace) % kAlign) != 0)
    return MTPC_ERR_WORKSPACE;
  if ((rc = set_backward_attributes(head)) != MTPC_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* bw = static_cast<uint8_t*>(bwd_workspace);
  if (static_hmm && cudaMemsetAsync(dT_static, 0, static_cast<size_t>(c.n - 1) * c.r * c.r * 4, st) != cudaSuccess)
    return MTPC_ERR_CUDA;
  const void* hb = nullptr;
  head->draft_P = 0;
  rc = stage_hidden(head, hidden, T, &hb, st);
  if (rc != MTPC_OK) return rc;
  PhaseTimer pt(head, st);
  // 1. forward projection, keeping the units' log-sum-exps
  pt.begin();
  GradArgs fwd;
  fwd.lse_out = reinterpret_cast<float*>(bw + B.off_lse);
  fwd.logit_out = reinterpret_cast<float*>(bw + B.off_logits);
  fwd.logit_pitch = B.Nc;
  rc = launch_gemm(head, hb, T, true, true, targets, st, &fwd);
  pt.end();
  if (rc != MTPC_OK) return rc;
  // 2. circuit backward: posteriors of the input units and of the sum units
  pt.begin();
  CircuitBackwardArgs a;
  memset(&a, 0, sizeof(a));
  a.targets = targets;
  a.weight = weight;
  a.out = out_logprob;
  a.post = reinterpret_cast<float*>(bw + B.off_post);
  a.dsum = reinterpret_cast<__nv_bfloat16*>(bw + B.off_dlogit) + B.Nc;      // columns [Nc, Nc + S r) of the dlogit rows
  a.dsum_pitch = static_cast<int>(B.Kd);
  a.W = T;
  rc = launch_circuit_backward(head, a, dT_static, st);
  pt.end();
  if (rc != MTPC_OK) return rc;
  // 3., 4. logit gradients from the kept logits, then the plain GEMMs
  return backward_tail(head, B, bw, hb, targets, T, d_hidden, dW_emit, dW_sum, pt, st);
}

int mtpc_lowrank_backward_workspace_bytes(const mtpc_config* cfg, int32_t k, int32_t T, size_t* out_bytes) {
  if (!cfg || !out_bytes) return MTPC_ERR_NULL;
  if (T < 1) return MTPC_ERR_SHAPE;
  Layout L;
  int rc = plan(*cfg, &L);
  if (rc != MTPC_OK) return rc;
  LowRankParams lrp;
  if (cfg->io_dtype != MTPC_BF16 || !plan_lowrank(*cfg, k, &lrp)) return MTPC_ERR_UNSUPPORTED;
  LowRankBackwardLayout R;
  plan_lowrank_backward(*cfg, L, k, T, &R);
  *out_bytes = R.total;
  return MTPC_OK;
}

int mtpc_lowrank_window_logprob_backward(mtpc_head* head, const void* hidden, const int32_t* targets, int32_t T,
                                         const float* weight, void* bwd_workspace, size_t bwd_workspace_bytes,
                                         float* out_logprob, float* d_hidden, float* dW_base, float* dA, float* dB,
                                         float* dW_sum, float* dT_static, void* stream) {
  int rc = check_call(head, T);
  if (rc != MTPC_OK) return rc;
  if (T == 0) return MTPC_OK;
  if (!hidden || !targets || !weight || !bwd_workspace || !d_hidden || !dW_base || !dA || !dB || !dW_sum) return MTPC_ERR_NULL;
  if (head->lr_k == 0) return MTPC_ERR_STATE;                  // a head on a composed tensor: mtpc_window_logprob_backward
  const mtpc_config& c = head->cfg;
  const Layout& L = head->L;
  const int k = head->lr_k;
  const bool static_hmm = c.family == MTPC_HMM && !is_ctx(head) && c.n > 1;
  if (static_hmm && !dT_static) return MTPC_ERR_NULL;
  LowRankBackwardLayout R;
  plan_lowrank_backward(c, L, k, T, &R);
  const BackwardLayout& B = R.B;
  if (bwd_workspace_bytes < R.total || (reinterpret_cast<uintptr_t>(bwd_workspace) % kAlign) != 0) return MTPC_ERR_WORKSPACE;
  if ((rc = set_backward_attributes(head)) != MTPC_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* bw = static_cast<uint8_t*>(bwd_workspace);
  if (static_hmm && cudaMemsetAsync(dT_static, 0, static_cast<size_t>(c.n - 1) * c.r * c.r * 4, st) != cudaSuccess)
    return MTPC_ERR_CUDA;
  const void* hb = hidden;                                     // (factored heads are bf16)
  head->draft_P = 0;
  PhaseTimer pt(head, st);
  // 1. factored forward projection, keeping every unit's log-sum-exp
  pt.begin();
  rc = launch_lowrank_projection(head, hb, T, targets, st, reinterpret_cast<float*>(bw + B.off_lse));
  pt.end();
  if (rc != MTPC_OK) return rc;
  // 2. circuit backward: posteriors of the input units; the sum units' logit gradients go to the right of sy
  pt.begin();
  __nv_bfloat16* sy = reinterpret_cast<__nv_bfloat16*>(bw + R.off_sy);
  CircuitBackwardArgs a;
  memset(&a, 0, sizeof(a));
  a.targets = targets;
  a.weight = weight;
  a.out = out_logprob;
  a.post = reinterpret_cast<float*>(bw + B.off_post);
  a.dsum = sy + R.Ksy;
  a.dsum_pitch = static_cast<int>(R.pitch);
  a.W = T;
  rc = launch_circuit_backward(head, a, dT_static, st);
  pt.end();
  if (rc != MTPC_OK) return rc;
  // 3., 4. logit gradients and what is derived from them, then the GEMMs
  return lowrank_backward_tail(head, R, bw, hb, targets, T, d_hidden, dW_base, dA, dB, dW_sum, pt, st);
}

}  // extern "C"

// Eq. 6 loss and its gradients, on a head built on a composed tensor (dW_emit) or on a factored one (dW_base, dA, dB): the
// two differ in the projection that keeps the logits and in the GEMMs at the end.
static int window_loss_backward_impl(mtpc_head* head, const void* hidden, const int32_t* targets, int32_t num_sequences,
                                     int32_t sequence_length, float gamma, void* bwd_workspace, size_t bwd_workspace_bytes,
                                     float* out_slot_loss, float* out_loss, float* d_hidden, float* dW_emit, float* dW_base,
                                     float* dA, float* dB, float* dW_sum, float* dT_static, void* stream) {
  if (!head) return MTPC_ERR_NULL;
  if (num_sequences < 1 || sequence_length < 1) return MTPC_ERR_SHAPE;
  const int64_t T64 = static_cast<int64_t>(num_sequences) * sequence_length;
  if (T64 > head->cfg.max_positions) return MTPC_ERR_SHAPE;
  if (!hidden || !targets || !bwd_workspace || !out_slot_loss || !out_loss || !d_hidden || !dW_sum) return MTPC_ERR_NULL;
  const bool factored = head->lr_k > 0;
  if (factored ? (!dW_base || !dA || !dB) : !dW_emit) return MTPC_ERR_NULL;
  const int T = static_cast<int>(T64);
  const mtpc_config& c = head->cfg;
  const Layout& L = head->L;
  const bool static_hmm = c.family == MTPC_HMM && !is_ctx(head) && c.n > 1;
  if (static_hmm && !dT_static) return MTPC_ERR_NULL;
  LowRankBackwardLayout R;
  memset(&R, 0, sizeof(R));
  if (factored) plan_lowrank_backward(c, L, head->lr_k, T, &R);
  else plan_backward(c, L, T, &R.B);
  const BackwardLayout& B = R.B;
  if (bwd_workspace_bytes < (factored ? R.total : B.total) || (reinterpret_cast<uintptr_t>(bwd_workspace) % kAlign) != 0)
    return MTPC_ERR_WORKSPACE;
  int rc = set_backward_attributes(head);
  if (rc != MTPC_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* bw = static_cast<uint8_t*>(bwd_workspace);
  float* post = reinterpret_cast<float*>(bw + B.off_post);
  float* coeff = reinterpret_cast<float*>(bw + B.off_coeff);
  float* prefix = at<float>(head, L.off_prefix);
  float* partial = at<float>(head, L.off_partial);
  if (static_hmm && cudaMemsetAsync(dT_static, 0, static_cast<size_t>(c.n - 1) * c.r * c.r * 4, st) != cudaSuccess)
    return MTPC_ERR_CUDA;
  const void* hb = nullptr;
  head->draft_P = 0;
  rc = stage_hidden(head, hidden, T, &hb, st);
  if (rc != MTPC_OK) return rc;
  PhaseTimer pt(head, st);
  // 1. forward projection (keeping the log-sum-exps) and the weight of every prefix log-marginal in the loss
  pt.begin();
  GradArgs fwd;
  fwd.lse_out = reinterpret_cast<float*>(bw + B.off_lse);
  fwd.logit_out = reinterpret_cast<float*>(bw + B.off_logits);
  fwd.logit_pitch = B.Nc;
  rc = factored ? launch_lowrank_projection(head, hb, T, targets, st, fwd.lse_out)
                : launch_gemm(head, hb, T, true, true, targets, st, &fwd);
  if (rc != MTPC_OK) return rc;
  launch_kernel(loss_coeff_kernel, num_sequences, kLossThreads, 0, st, overlapped(head), targets, coeff, sequence_length, c.n,
                num_sequences, gamma);
  head->launches++;
  pt.end();
  if ((rc = check_launch()) != MTPC_OK) return rc;
  // 2. circuit: every prefix and the whole gradient of the loss. The sum units' logit gradients (bf16)
  // go to the right of dlogit, or of [s | y] on a factored head.
  pt.begin();
  CircuitBackwardArgs a;
  memset(&a, 0, sizeof(a));
  a.targets = targets;
  a.coeff = coeff;
  a.prefix = prefix;
  a.post = post;
  a.dsum = factored ? reinterpret_cast<__nv_bfloat16*>(bw + R.off_sy) + R.Ksy
                    : reinterpret_cast<__nv_bfloat16*>(bw + B.off_dlogit) + B.Nc;
  a.dsum_pitch = static_cast<int>(factored ? R.pitch : B.Kd);
  a.W = T;
  if ((rc = launch_circuit_backward(head, a, dT_static, st)) != MTPC_OK) return rc;
  const bool beside = overlapped(head);
  auto launch_loss = [&] {
    launch_kernel(loss_partial_kernel, num_sequences, kLossThreads, 0, st, beside, prefix, targets, partial, sequence_length, c.n,
                  beside ? 1 : 0);
    launch_kernel(loss_final_kernel, 1, kLossThreads, 0, st, beside, partial, out_slot_loss, out_loss, num_sequences, c.n, gamma);
    head->launches += 2;
  };
  if (!beside) launch_loss();                                  // between events: in the phase of the circuit
  pt.end();
  if ((rc = check_launch()) != MTPC_OK) return rc;
  rc = factored ? lowrank_backward_tail(head, R, bw, hb, targets, T, d_hidden, dW_base, dA, dB, dW_sum, pt, st)
                : backward_tail(head, B, bw, hb, targets, T, d_hidden, dW_emit, dW_sum, pt, st);
  if (rc != MTPC_OK) return rc;
  if (beside) launch_loss();                                   // from the prefixes, beside the last GEMM
  return check_launch();
}

extern "C" {

int mtpc_window_loss_backward(mtpc_head* head, const void* hidden, const int32_t* targets, int32_t num_sequences,
                              int32_t sequence_length, float gamma, void* bwd_workspace, size_t bwd_workspace_bytes,
                              float* out_slot_loss, float* out_loss, float* d_hidden, float* dW_emit, float* dW_sum,
                              float* dT_static, void* stream) {
  if (head && head->lr_k > 0) return MTPC_ERR_UNSUPPORTED;     // a factored head: mtpc_lowrank_window_loss_backward
  return window_loss_backward_impl(head, hidden, targets, num_sequences, sequence_length, gamma, bwd_workspace,
                                   bwd_workspace_bytes, out_slot_loss, out_loss, d_hidden, dW_emit, nullptr, nullptr, nullptr,
                                   dW_sum, dT_static, stream);
}

int mtpc_lowrank_window_loss_backward(mtpc_head* head, const void* hidden, const int32_t* targets, int32_t num_sequences,
                                      int32_t sequence_length, float gamma, void* bwd_workspace, size_t bwd_workspace_bytes,
                                      float* out_slot_loss, float* out_loss, float* d_hidden, float* dW_base, float* dA,
                                      float* dB, float* dW_sum, float* dT_static, void* stream) {
  if (head && head->lr_k == 0) return MTPC_ERR_STATE;          // a head on a composed tensor: mtpc_window_loss_backward
  return window_loss_backward_impl(head, hidden, targets, num_sequences, sequence_length, gamma, bwd_workspace,
                                   bwd_workspace_bytes, out_slot_loss, out_loss, d_hidden, nullptr, dW_base, dA, dB, dW_sum,
                                   dT_static, stream);
}

// Streams and events of the chunked host-buffer path; no device memory is allocated.
static int ensure_copy_pipeline(mtpc_head* head, int chunks) {
  if (!head->copy_stream && cudaStreamCreateWithFlags(&head->copy_stream, cudaStreamNonBlocking) != cudaSuccess)
    return MTPC_ERR_CUDA;
  if (head->copy_event_count < chunks + 1) {
    cudaEvent_t* ev = static_cast<cudaEvent_t*>(calloc(chunks + 1, sizeof(cudaEvent_t)));
    if (!ev) return MTPC_ERR_CUDA;
    for (int i = 0; i < chunks + 1; ++i) {
      if (i < head->copy_event_count) ev[i] = head->copy_events[i];
      else if (cudaEventCreateWithFlags(&ev[i], cudaEventDisableTiming) != cudaSuccess) { free(ev); return MTPC_ERR_CUDA; }
    }
    free(head->copy_events);
    head->copy_events = ev;
    head->copy_event_count = chunks + 1;
  }
  return MTPC_OK;
}

int mtpc_lowrank_compose(int32_t n, int32_t r, int32_t v, int32_t d, int32_t k, const void* W_base, const void* A,
                         const void* B, void* W_emit_out, void* stream) {
  if (!W_base || !A || !B || !W_emit_out) return MTPC_ERR_NULL;
  if (n < 1 || r < 1 || v < 1 || d < 1 || k < 1 || static_cast<int64_t>(n) * r > 65535 ||
      (v + kComposeCtaRows - 1) / kComposeCtaRows > 65535)
    return MTPC_ERR_SHAPE;
  if (k > kLowRankMaxK) return MTPC_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const auto* w = static_cast<const __nv_bfloat16*>(W_base);
  const auto* a = static_cast<const __nv_bfloat16*>(A);
  const auto* b = static_cast<const __nv_bfloat16*>(B);
  auto* u = static_cast<__nv_bfloat16*>(W_emit_out);
  const int rows = (v + kComposeCtaRows - 1) / kComposeCtaRows;
  if (lowrank_vector_ok(d, {W_base, B, W_emit_out})) {
    const size_t smem = compose_smem_bytes(k, 4);
    if (cudaFuncSetAttribute(lowrank_compose_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) !=
        cudaSuccess)
      return MTPC_ERR_CUDA;
    lowrank_compose_kernel<4><<<dim3((d + 4 * kLowRankThreads - 1) / (4 * kLowRankThreads), rows, n * r), kLowRankThreads, smem,
                                st>>>(w, a, b, u, r, v, d, k);
  } else {
    const size_t smem = compose_smem_bytes(k, 1);
    lowrank_compose_kernel<1><<<dim3((d + kLowRankThreads - 1) / kLowRankThreads, rows, n * r), kLowRankThreads, smem, st>>>(
        w, a, b, u, r, v, d, k);
  }
  return check_launch();
}

int mtpc_lowrank_backward(int32_t n, int32_t r, int32_t v, int32_t d, int32_t k, const void* A, const void* B,
                          const float* dW_emit, float* dW_base, float* dA, float* dB, void* stream) {
  if (!A || !B || !dW_emit || !dW_base || !dA || !dB) return MTPC_ERR_NULL;
  if (n < 1 || r < 1 || v < 1 || d < 1 || k < 1 || v > 65535 || static_cast<int64_t>(n) * r > 65535) return MTPC_ERR_SHAPE;
  if (k > kLowRankMaxK) return MTPC_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const auto* a = static_cast<const __nv_bfloat16*>(A);
  const auto* b = static_cast<const __nv_bfloat16*>(B);
  const int units = n * r, kchunks = (k + kRankChunk - 1) / kRankChunk;
  auto blocks = [&](int cv) { return (d + cv * kLowRankThreads - 1) / (cv * kLowRankThreads); };
  if (lowrank_vector_ok(d, {B, dW_emit, dW_base, dB})) {
    lowrank_dw_kernel<4><<<dim3(blocks(4), v, n), kLowRankThreads, 0, st>>>(dW_emit, dW_base, r, v, d);
    lowrank_da_kernel<4><<<dim3((v + 31) / 32, units), kLowRankThreads, 0, st>>>(dW_emit, b, dA, v, d, k);
    lowrank_db_kernel<4><<<dim3(blocks(4), kchunks, units), kLowRankThreads, 0, st>>>(dW_emit, a, dB, v, d, k);
  } else {
    lowrank_dw_kernel<1><<<dim3(blocks(1), v, n), kLowRankThreads, 0, st>>>(dW_emit, dW_base, r, v, d);
    lowrank_da_kernel<1><<<dim3((v + 31) / 32, units), kLowRankThreads, 0, st>>>(dW_emit, b, dA, v, d, k);
    lowrank_db_kernel<1><<<dim3(blocks(1), kchunks, units), kLowRankThreads, 0, st>>>(dW_emit, a, dB, v, d, k);
  }
  return check_launch();
}

// Pieces a host-buffer call of T positions is uploaded and processed in (at most kMaxHostChunks; returns how many). While one is
// processed the next is uploaded, so what is not hidden is the first upload if the kernels take longer, the last piece's kernels
// if the link does: that piece is the smallest, and the others grow away from it by the ratio of the two times (50 GB/s and
// 1.4 PFLOP/s; 1.25 to 2), so that none waits for its neighbour. 8192 positions of the 8 x 16 x 320 head, d = 4096: four equal
// pieces 2.10 ms, these 1.96; fp32 hidden states, d = 3072, 8 x 16 x 272: 2.18 and 2.06.
static int host_chunks(const mtpc_config& c, const Layout& L, int lr_k, int T, int* sizes) {
  const double rows = lr_k > 0 ? static_cast<double>(c.n) * c.v + static_cast<double>(c.n) * c.r * lr_k : static_cast<double>(c.n) * c.r * c.v;
  const double compute = 2.0 * c.d * (rows + L.sum_rows) / 1.4e15;
  const double upload = (static_cast<double>(c.d) * (c.io_dtype == MTPC_F32 ? 4 : 2) + 4.0 * c.n) / 50e9;
  double growth = compute > upload ? compute / upload : upload / compute;
  growth = growth < 1.25 ? 1.25 : growth > 2.0 ? 2.0 : growth;
  int count = 0, left = T;
  for (double size = kHostChunkPositions; left > 0; size *= growth) {
    int take = static_cast<int>((size < 1e9 ? size : 1e9) / 256.0 + 0.5) * 256;
    if (left <= take + take / 2 || count == kMaxHostChunks - 1) take = left;
    sizes[count++] = take;
    left -= take;
  }
  if (compute < upload)
    for (int i = 0; i < count / 2; ++i) { const int x = sizes[i]; sizes[i] = sizes[count - 1 - i]; sizes[count - 1 - i] = x; }
  return count;
}

int mtpc_window_logprob_host(mtpc_head* head, const void* hidden_host, const int32_t* targets_host, int32_t T,
                             float* out_logprob_host, void* stream) {
  int rc = check_call(head, T);
  if (rc != MTPC_OK) return rc;
  if (T == 0) return MTPC_OK;
  if (!hidden_host || !targets_host || !out_logprob_host) return MTPC_ERR_NULL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const Layout& L = head->L;
  const mtpc_config& c = head->cfg;
  const size_t elt = c.io_dtype == MTPC_F32 ? 4 : 2;
  uint8_t* dh = head->ws + L.off_h_hidden;
  int32_t* dt = at<int32_t>(head, L.off_h_targets);
  float* dout = at<float>(head, L.off_h_out);
  // The positions are uploaded in chunks on a second stream while the kernels of the chunks before run on `stream`.
  int sizes[kMaxHostChunks];
  const int chunks = host_chunks(c, L, head->lr_k, T, sizes);
  if ((rc = ensure_copy_pipeline(head, chunks)) != MTPC_OK) return rc;
  cudaStream_t cs = head->copy_stream;
  bool fail = cudaEventRecord(head->copy_events[chunks], st) != cudaSuccess;     // uploads wait for earlier work on `stream`
  fail |= cudaStreamWaitEvent(cs, head->copy_events[chunks], 0) != cudaSuccess;
  size_t t0 = 0;
  for (int k = 0; k < chunks && !fail; t0 += sizes[k++]) {
    const size_t tc = sizes[k];
    fail |= cudaMemcpyAsync(dh + t0 * c.d * elt, static_cast<const uint8_t*>(hidden_host) + t0 * c.d * elt, tc * c.d * elt,
                            cudaMemcpyHostToDevice, cs) != cudaSuccess;
    fail |= cudaMemcpyAsync(dt + t0 * c.n, targets_host + t0 * c.n, tc * c.n * 4, cudaMemcpyHostToDevice, cs) != cudaSuccess;
    fail |= cudaEventRecord(head->copy_events[k], cs) != cudaSuccess;
  }
  if (fail) return MTPC_ERR_CUDA;
  t0 = 0;
  for (int k = 0; k < chunks; t0 += sizes[k++]) {
    if (cudaStreamWaitEvent(st, head->copy_events[k], 0) != cudaSuccess) return MTPC_ERR_CUDA;
    rc = window_logprob_impl(head, dh + t0 * c.d * elt, dt + t0 * c.n, sizes[k], dout + t0, nullptr, st);
    if (rc != MTPC_OK) { cudaStreamSynchronize(cs); return rc; }
  }
  fail = cudaMemcpyAsync(out_logprob_host, dout, static_cast<size_t>(T) * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess;
  fail |= cudaStreamSynchronize(st) != cudaSuccess;
  return fail ? MTPC_ERR_CUDA : MTPC_OK;
}

int mtpc_draft_sample_host(mtpc_head* head, const void* hidden_host, int32_t P, int32_t wpp,
                           const float* uniforms_host, int32_t* out_bytes_host, float* out_logprob_host,
                           void* stream) {
  int rc = check_call(head, P);
  if (rc != MTPC_OK) return rc;
  if (wpp < 1 || wpp > head->cfg.max_windows_per_pos) return MTPC_ERR_SHAPE;
  if (P == 0) return MTPC_OK;
  if (!hidden_host || !uniforms_host || !out_bytes_host || !out_logprob_host) return MTPC_ERR_NULL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const Layout& L = head->L;
  const mtpc_config& c = head->cfg;
  const size_t elt = c.io_dtype == MTPC_F32 ? 4 : 2;
  const size_t W = static_cast<size_t>(P) * wpp;
  void* dh = head->ws + L.off_h_hidden;
  float* du = at<float>(head, L.off_h_uniforms);
  int32_t* db = at<int32_t>(head, L.off_h_bytes);
  float* dout = at<float>(head, L.off_h_out);
  bool fail = cudaMemcpyAsync(dh, hidden_host, static_cast<size_t>(P) * c.d * elt, cudaMemcpyHostToDevice, st) !=
              cudaSuccess;
  fail |= cudaMemcpyAsync(du, uniforms_host, W * 2 * c.n * 4, cudaMemcpyHostToDevice, st) != cudaSuccess;
  if (fail) return MTPC_ERR_CUDA;
  rc = draft_sample_impl(head, dh, P, wpp, du, db, dout, nullptr, st);
  if (rc != MTPC_OK) return rc;
  fail = cudaMemcpyAsync(out_bytes_host, db, W * c.n * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess;
  fail |= cudaMemcpyAsync(out_logprob_host, dout, W * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess;
  fail |= cudaStreamSynchronize(st) != cudaSuccess;
  return fail ? MTPC_ERR_CUDA : MTPC_OK;
}

int mtpc_get_status(mtpc_head* head, void* stream, uint32_t* out_flags) {
  if (!head || !out_flags) return MTPC_ERR_NULL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint32_t flags = 0;
  void* dev = head->ws + head->L.off_status;
  if (cudaMemcpyAsync(&flags, dev, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return MTPC_ERR_CUDA;
  if (cudaMemsetAsync(dev, 0, 4, st) != cudaSuccess) return MTPC_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return MTPC_ERR_CUDA;
  *out_flags = flags;
  return (flags & MTPC_STATUS_TIMEOUT) ? MTPC_ERR_TIMEOUT : MTPC_OK;
}

static void free_timing(mtpc_head* head) {
  if (head->ev) {
    for (size_t i = 0; i < static_cast<size_t>(head->ring) * kMaxPhases * 2; ++i) cudaEventDestroy(head->ev[i]);
    free(head->ev);
    free(head->ring_phases);
  }
  head->ev = nullptr;
  head->ring_phases = nullptr;
  head->ring = 0;
  head->calls = 0;
}

int mtpc_set_timing(mtpc_head* head, int32_t ring) {
  if (!head) return MTPC_ERR_NULL;
  if (ring < 0 || ring > 4096) return MTPC_ERR_SHAPE;
  free_timing(head);
  if (ring == 0) return MTPC_OK;
  const size_t count = static_cast<size_t>(ring) * kMaxPhases * 2;
  head->ev = static_cast<cudaEvent_t*>(calloc(count, sizeof(cudaEvent_t)));
  head->ring_phases = static_cast<int*>(calloc(ring, sizeof(int)));
  if (!head->ev || !head->ring_phases) { free(head->ev); free(head->ring_phases); head->ev = nullptr; return MTPC_ERR_CUDA; }
  head->ring = ring;
  for (size_t i = 0; i < count; ++i)
    if (cudaEventCreate(&head->ev[i]) != cudaSuccess) { head->ring = 0; return MTPC_ERR_CUDA; }
  return MTPC_OK;
}

int mtpc_get_timing(mtpc_head* head, int32_t calls_back, float* out_ms, int32_t capacity, int32_t* out_count) {
  if (!head || !out_ms || !out_count) return MTPC_ERR_NULL;
  *out_count = 0;
  if (head->ring == 0) return MTPC_OK;
  if (calls_back < 0 || calls_back >= head->ring || static_cast<uint64_t>(calls_back) >= head->calls)
    return MTPC_ERR_SHAPE;
  const int slot = static_cast<int>((head->calls - 1 - calls_back) % head->ring);
  const int nph = head->ring_phases[slot];
  for (int i = 0; i < nph && i < capacity; ++i) {
    cudaEvent_t* pair = head->ev + (static_cast<size_t>(slot) * kMaxPhases + i) * 2;
    if (cudaEventSynchronize(pair[1]) != cudaSuccess) return MTPC_ERR_CUDA;
    if (cudaEventElapsedTime(&out_ms[i], pair[0], pair[1]) != cudaSuccess) return MTPC_ERR_CUDA;
    *out_count = i + 1;
  }
  return MTPC_OK;
}

int mtpc_debug_set_wait_limit_ns(mtpc_head* head, uint64_t limit_ns) {
  if (!head) return MTPC_ERR_NULL;
  head->wait_limit_ns = limit_ns == 0 ? kWaitLimitNs : limit_ns;
  return MTPC_OK;
}

int mtpc_debug_set_projection_variant(mtpc_head* head, int32_t variant) {
  if (!head) return MTPC_ERR_NULL;
  if (variant < 0 || variant > 2) return MTPC_ERR_SHAPE;
  if (variant == 2 && head->max_pairs <= 0) return MTPC_ERR_UNSUPPORTED;
  head->projection_variant = variant;
  return MTPC_OK;
}

int mtpc_debug_set_draft_grouping(mtpc_head* head, int32_t mode) {
  if (!head) return MTPC_ERR_NULL;
  if (mode < 0 || mode > 2) return MTPC_ERR_SHAPE;
  if (mode == 2 && head->cfg.max_positions <= head->L.decode_max_p) return MTPC_ERR_UNSUPPORTED;
  return MTPC_OK;                      // one implementation: the modes draw the same bytes
}

int mtpc_launch_count(mtpc_head* head, uint64_t* out_count) {
  if (!head || !out_count) return MTPC_ERR_NULL;
  *out_count = head->launches;
  return MTPC_OK;
}

int mtpc_destroy(mtpc_head* head) {
  if (!head) return MTPC_ERR_NULL;
  free_timing(head);
  for (int i = 0; i < head->copy_event_count; ++i) cudaEventDestroy(head->copy_events[i]);
  free(head->copy_events);
  if (head->copy_stream) cudaStreamDestroy(head->copy_stream);
  delete head;
  return MTPC_OK;
}

const char* mtpc_status_string(int code) {
  switch (code) {
    case MTPC_OK: return "ok";
    case MTPC_ERR_NULL: return "a required pointer is NULL";
    case MTPC_ERR_SHAPE: return "a size argument is out of range";
    case MTPC_ERR_UNSUPPORTED: return "configuration not supported by this version";
    case MTPC_ERR_WORKSPACE: return "workspace too small or misaligned";
    case MTPC_ERR_CUDA: return "a CUDA call failed (no sm_100 device, launch error, or driver entry point missing)";
    case MTPC_ERR_TIMEOUT: return "a device-side bounded wait expired";
    case MTPC_ERR_STATE:
      return "the head holds no draft state for this call (mtpc_speculative_accept must follow a draft of the same positions)";
    case MTPC_ERR_STATIC_SCRATCH:
      return "the call needs more scratch than the library's built-in static array holds (mtpc_window_logprob_static)";
    default: return "unknown status code";
  }
}

}  // extern "C"

// ------------------------------------------------------------------------------------------------------------
// mtpc_window_logprob_static: the window log-likelihood for callers that have no device allocator at hand.
// All scratch (status word, log-softmaxed HMM transitions, G, log omega) is carved out of one file-scope device
// array, so the call needs neither a head nor a caller-made workspace and allocates nothing.
// ------------------------------------------------------------------------------------------------------------
namespace {

// Every GPU that loads the library holds this array until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[MTPC_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
void* g_static_scratch_addr[kMaxDevices];   // device address of the array on each device, 0 = not looked up yet

// In host code `g_static_scratch` is only a handle for the runtime, not a device address: the address the
// kernels need comes from cudaGetSymbolAddress, asked once per device with that device current.
int static_scratch_address(unsigned char** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MTPC_ERR_CUDA;
  void* p = __atomic_load_n(&g_static_scratch_addr[dev], __ATOMIC_ACQUIRE);
  if (!p) {
    if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) return MTPC_ERR_CUDA;
    __atomic_store_n(&g_static_scratch_addr[dev], p, __ATOMIC_RELEASE);   // every thread gets the same answer
  }
  *out = static_cast<unsigned char*>(p);
  return MTPC_OK;
}

}  // namespace

extern "C" int mtpc_window_logprob_static(const mtpc_config* cfg, const void* W_emit, const void* W_sum,
                                          const float* T_static, const void* hidden, const int32_t* targets,
                                          int32_t T, float* out_logprob, uint32_t* out_status, void* stream) {
  if (!cfg) return MTPC_ERR_NULL;
  if (cfg->io_dtype != MTPC_BF16) return MTPC_ERR_UNSUPPORTED;   // fp32 inputs would need rounded copies of the weights
  if (cfg->flags != 0) return MTPC_ERR_UNSUPPORTED;
  if (T < 0) return MTPC_ERR_SHAPE;
  mtpc_config c = *cfg;
  c.max_positions = T > 0 ? T : 1;
  c.max_windows_per_pos = 1;
  Layout L;
  int rc = plan(c, &L);
  if (rc != MTPC_OK) return rc;
  // Carve only what this call needs: [status | logA (HMM) | G | log omega].
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes); return o; };
  L.off_status = take(256);
  L.off_logA = take(c.family == MTPC_HMM ? static_cast<size_t>(c.n - 1) * c.r * c.r * 4 : 0);
  L.off_G = take(static_cast<size_t>(c.max_positions) * c.n * c.r * 4);
  L.off_logw = take(static_cast<size_t>(c.max_positions) * L.sum_rows * 4);
  L.off_sel = L.off_wemit = L.off_wsum = L.off_hidden = L.off_logits = L.off_unit_lse = 0;   // unused by this call
  L.off_prefix = L.off_partial = L.off_sum_bias = L.off_msg = L.off_probA = L.off_cdfA = 0;
  L.off_h_hidden = L.off_h_targets = L.off_h_uniforms = L.off_h_bytes = L.off_h_out = 0;
  L.total = off;
  if (L.total > static_cast<size_t>(MTPC_STATIC_SCRATCH_BYTES)) return MTPC_ERR_STATIC_SCRATCH;
  if (T == 0) return MTPC_OK;
  if (!W_emit || !W_sum || !hidden || !targets || !out_logprob) return MTPC_ERR_NULL;
  if (c.family == MTPC_HMM && c.n > 1 && !T_static) return MTPC_ERR_NULL;

  int dev = 0, cc_major = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MTPC_ERR_CUDA;
  if (cudaDeviceGetAttribute(&cc_major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess || cc_major != 10)
    return MTPC_ERR_CUDA;
  unsigned char* scratch = nullptr;
  if ((rc = static_scratch_address(&scratch)) != MTPC_OK) return rc;

  mtpc_head h;                       // host-side bookkeeping only, lives for the duration of this call
  memset(&h, 0, sizeof(h));
  h.cfg = c;
  h.L = L;
  h.ws = scratch;
  h.W_emit_bf16 = W_emit;
  h.W_sum_bf16 = W_sum;
  h.wait_limit_ns = kWaitLimitNs;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  bool fail = cudaDeviceGetAttribute(&h.num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess;
  fail |= !allow_full_smem(mtpc_gemm_kernel<kModeLogprob, 1, 16>) || !allow_full_smem(mtpc_gemm_kernel<kModeLogprob, 1, 32>);
  fail |= !set_circuit_attributes();
  // The array keeps whatever the previous call left in it. Only the status word has to start at zero; G, log omega
  // and logA are fully rewritten for the rows this call reads.
  fail |= cudaMemsetAsync(scratch + L.off_status, 0, 256, st) != cudaSuccess;
  if (fail) return MTPC_ERR_CUDA;
  if (c.family == MTPC_HMM && c.n > 1) {
    const int rows = (c.n - 1) * c.r;
    static_tables_kernel<<<(rows + 7) / 8, 256, 0, st>>>(T_static, at<float>(&h, L.off_logA), nullptr, nullptr, rows, c.r);
    if (check_launch() != MTPC_OK) return MTPC_ERR_CUDA;
  }
  rc = make_tmap(&h.tm_emit_lp, W_emit, static_cast<uint64_t>(c.n) * c.r * c.v, c.d, L.lp.tile_cols);
  if (rc == MTPC_OK) rc = make_tmap(&h.tm_sum, W_sum, L.sum_rows, c.d, L.sum_cols);
  if (rc != MTPC_OK) return rc;
  rc = window_logprob_impl(&h, hidden, targets, T, out_logprob, nullptr, st);
  if (rc != MTPC_OK) return rc;
  if (out_status &&
      cudaMemcpyAsync(out_status, scratch + L.off_status, 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return MTPC_ERR_CUDA;
  return MTPC_OK;
}
