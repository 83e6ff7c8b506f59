// Draft path for few positions (decode-time speculative drafting, Algorithm 1): the cost is one pass over the
// emission weights, so the work is organised around streaming them from HBM exactly once.
//
//   mtpc_decode_gemm_kernel   logits[p, row] = W[row] . h_p for every weight row (emission and sum-unit rows) and
//                             every position p < P <= 128, with the roles of the operands swapped with respect
//                             to the training-shaped kernel: 128 weight rows sit on the M axis (TMEM lanes), the
//                             positions on the N axis (TMEM columns). Emission logits go to a small scratch
//                             [P, n*r*v] fp32 (P is tiny here, so this is a few MB against hundreds of MB of
//                             weights); sum-unit logits are log-softmaxed over their groups of r rows (= lanes,
//                             by warp shuffles) and written as log omega [P, S*r]. A mixture of more than 32
//                             components (CP, r = 64 or 128) spans several warps: its logits are written as they
//                             are, and the kernels that follow normalise them where they need to.
//                             Weight rows are cut into tiles of `tile_rows` <= 128 rows, chosen by the host so that
//                             the tiles divide evenly over the persistent CTAs; each CTA takes a contiguous run
//                             of tiles and walks K once per tile.
//   draft_slot_kernel         one CTA per (position, window slot i): log-sum-exp of the r input units of the
//                             slot, then per window (one warp each): latent draws down to the unit that owns
//                             slot i, the byte by inverse CDF of that unit's categorical, and the evidence
//                             G[w, i, k] = log phi_k(byte) for all k, which the circuit kernels then reduce.
#pragma once
#include "mtpc_circuit.cuh"
#include "mtpc_gemm.cuh"

namespace mtpc {

constexpr int kDecodeMaxP = 128;                   // positions per call on this path
constexpr int kDecodeMaxStages = 9;                // of the weight pass's ring (see launch_decode_gemm)
constexpr int kSlotThreads = 512;

struct DecodeParams {
  CUtensorMap tm_h;      // hidden [P, d]       box 64 x Ppad
  CUtensorMap tm_emit;   // W_emit [n*r*v, d]   box 64 x tile_rows
  CUtensorMap tm_sum;    // W_sum  [S*r, d]     box 64 x sum_tile_rows
  CUtensorMap tm_emit2;  // a second matrix of emission-like rows [emit2_rows, d], box 64 x tile_rows (a factored
                         // low-rank head: tm_emit = W_base, tm_emit2 = B); unused when emit2_tiles == 0
  int P, Ppad, kblocks;
  int emit_rows, sum_rows, r;
  int emit2_rows, emit2_tiles;
  int tile_rows;                 // rows of an emission tile (a multiple of 8, <= 128)
  int sum_tile_rows;             // rows of a sum tile (a multiple of 32, <= tile_rows rounded up to 32)
  int tile_bytes;                // shared-memory pitch of a weight tile
  int emit_tiles, sum_tiles;
  int tile_stride;               // TMEM columns per tile
  int stages, stage_bytes;
  int ksplit;                    // CTAs of a cluster that share a run of tiles, each with its part of K (1: no cluster)
  float* logits;         // [P, emit_rows]
  float* logits2;        // [P, emit2_rows]
  float* logw;           // [P, sum_rows]
  const float* sum_bias; // [sum_rows] or NULL: added to the sum-unit logits before their softmax
  unsigned* status;
  uint64_t wait_limit_ns;   // limit of every pipeline wait
};

// Tile `t` of the launch: emission tiles first, then those of the second matrix, then sum tiles.
struct DecodeTile {
  int is_sum, second, index, rows;   // which matrix, tile index within it, rows per tile
};
__device__ __forceinline__ DecodeTile decode_tile(const DecodeParams& p, int t) {
  DecodeTile d;
  d.is_sum = t >= p.emit_tiles + p.emit2_tiles;
  d.second = !d.is_sum && t >= p.emit_tiles;
  d.index = d.is_sum ? t - p.emit_tiles - p.emit2_tiles : (d.second ? t - p.emit_tiles : t);
  d.rows = d.is_sum ? p.sum_tile_rows : p.tile_rows;
  return d;
}

// The warps that issue copies and MMAs run as wholes (elect_one): four MMAs of N = 16 and their copies, issued from a branch of lane 0's own,
// took 650 cycles a K step and tile, more than the step's bytes where a CTA has one tile (draft + acceptance of 8 positions of a factored
// head, d = 4096: 32.7 -> 27.0 us; 4 x 8 x 256, d = 1024, 16 positions: 20.0 -> 17.4) and nearly as much where it has three (mixture
// 8 x 16 x 320, 1 position 65.7 -> 63.6, HMM 16 x 32 x 320, 8 positions 225.7 -> 221.5; 128 positions of the mixture 96.7 -> 89.3).
// A CTA walks its run of tiles one after the other. Shared-memory stage: the weight tile (the MMA reads 128 rows from its base: what
// lies beyond the tile's own rows is other data, and the TMEM lanes it produces are never read), then the hidden tile
// (Ppad rows x 128 bytes) followed by slack so that the 128-row read stays inside the stage. Tensor memory: two slots of tile_stride columns.
// ksplit > 1: where the tiles leave most SMs idle (a factored head's 4600 rows are 72 tiles) a cluster of ksplit CTAs takes a
// tile, each walking its part of K; the others hand their fp32 accumulators to the first one through its shared memory (behind
// the ring: [rank - 1][position quad][128 rows] of float4), which adds them in rank order and runs the epilogue.
// Every CTA then has one tile. The pass over 39 MB of weights (n = 8, r = 16, v = 320, d = 4096, rank 16) took 30 us as 72 CTAs
// of 64 K steps and half the SMs idle; draft + acceptance of 8 positions: 51 -> 38 us with clusters
// of two.
__host__ __device__ inline size_t decode_exchange_bytes(int ksplit, int Ppad) {
  return static_cast<size_t>(ksplit - 1) * kBlockM * Ppad * sizeof(float);
}
__global__ void __launch_bounds__(kGemmThreads, 1) mtpc_decode_gemm_kernel(const __grid_constant__ DecodeParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t tiles_addr = (raw_addr + 1023u) & ~1023u;
  uint8_t* tiles = smem_raw + (tiles_addr - raw_addr);
  uint8_t* exchange = tiles + static_cast<size_t>(p.stages) * p.stage_bytes;
  GemmControl* ctl = reinterpret_cast<GemmControl*>(exchange + decode_exchange_bytes(p.ksplit, p.Ppad));

  const int warp = static_cast<int>(warp_uniform(threadIdx.x >> 5));
  const int lane = threadIdx.x & 31;
  const int total_tiles = p.emit_tiles + p.emit2_tiles + p.sum_tiles;
  const int rank = p.ksplit > 1 ? static_cast<int>(warp_uniform(cluster_cta_rank())) : 0;
  const int group = static_cast<int>(blockIdx.x) / p.ksplit, groups = static_cast<int>(gridDim.x) / p.ksplit;
  const int tile_begin = static_cast<int>(static_cast<long long>(group) * total_tiles / groups);
  const int tile_end = static_cast<int>(static_cast<long long>(group + 1) * total_tiles / groups);
  const int kb0 = rank * p.kblocks / p.ksplit, kb1 = (rank + 1) * p.kblocks / p.ksplit;
  const uint32_t hidden_off = p.tile_bytes;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&ctl->full[s]), 1);
      mbar_init(smem_u32(&ctl->empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&ctl->tfull[s]), 1);
      mbar_init(smem_u32(&ctl->tempty[s]), 4);
    }
    mbar_init(smem_u32(&ctl->drain), 1);
    ctl->abort = 0;
    ctl->wait_limit_ns = p.wait_limit_ns;
    fence_mbar_init();
    tma_prefetch_desc(&p.tm_h);
    tma_prefetch_desc(&p.tm_emit);
    tma_prefetch_desc(&p.tm_sum);
    if (p.emit2_tiles > 0) tma_prefetch_desc(&p.tm_emit2);
  }
  if (warp == 0 && tile_begin < tile_end && p.ksplit == 1) {
    // the ring's first K blocks of weights on their way to L2 while the kernel before this one finishes (draft + acceptance, without / with it:
    // mixture 8 x 16 x 320, 1 position 63.1 / 62.1 us, tree 8 x 32 x 256, 27 positions 88.2 / 87.5; not where clusters share a tile, whose short
    // runs it lengthens: 26.6 / 26.8)
    const uint32_t lead = elect_one();
    const DecodeTile t = decode_tile(p, tile_begin);
    const CUtensorMap* map = t.is_sum ? &p.tm_sum : (t.second ? &p.tm_emit2 : &p.tm_emit);
    for (int kb = kb0; kb < min(kb1, kb0 + p.stages); ++kb) tma_prefetch_2d(lead, map, kb * kBlockK, t.index * t.rows);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&ctl->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  if (p.ksplit > 1) cluster_sync_all();   // every CTA of the cluster runs before one writes into another's shared memory
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(ctl->tmem_base);
  grid_dependency_wait();     // a draft that follows another call closely sets up its barriers while that one finishes
  grid_launch_dependents();   // (after the wait: the per-slot kernel reads static tables early) it waits for this grid's results

  const int quarter = warp & 3;
  const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
  // Tile `tile` of the launch, whose accumulators start at tensor-memory column `col`: logits or log omega of this warp's 32
  // rows. others: the accumulators of the cluster's other CTAs (NULL: none).
  auto finish_tile = [&](int tile, uint32_t col, const float4* others) {
    const DecodeTile t = decode_tile(p, tile);
    if (quarter * 32 >= t.rows) return;                            // warp-uniform: none of this warp's lanes is a row
    const int nrows = t.is_sum ? p.sum_rows : (t.second ? p.emit2_rows : p.emit_rows);
    float* dst = t.is_sum ? p.logw : (t.second ? p.logits2 : p.logits);
    const int local = quarter * 32 + lane;
    const int row = t.index * t.rows + local;
    const bool mine = local < t.rows && row < nrows;
    const float bias = (t.is_sum && p.sum_bias != nullptr && mine) ? p.sum_bias[row] : 0.f;
    for (int b = 0; b < (p.P + 15) / 16; ++b) {
      float x[16];
      tmem_ld16(lane_base + col + b * 16, x);
      if (others != nullptr) {
        for (int part = 0; part + 1 < p.ksplit; ++part) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float4 y = others[(part * (p.Ppad / 4) + b * 4 + c) * kBlockM + local];
            x[4 * c] += y.x;
            x[4 * c + 1] += y.y;
            x[4 * c + 2] += y.z;
            x[4 * c + 3] += y.w;
          }
        }
      }
      if (t.is_sum && p.r <= 32) {
#pragma unroll
        for (int c = 0; c < 16; ++c) x[c] += bias;
        // log-softmax over the r rows of a sum unit = r adjacent lanes (r a power of two <= 32); the 16
        // positions of the batch are reduced side by side so that the shuffles overlap
        float m[16], e[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) m[c] = x[c];
        for (int off = 1; off < p.r; off <<= 1) {
#pragma unroll
          for (int c = 0; c < 16; ++c) m[c] = fmaxf(m[c], __shfl_xor_sync(0xffffffffu, m[c], off));
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) e[c] = fast_ex2((x[c] - m[c]) * kLog2e);
        for (int off = 1; off < p.r; off <<= 1) {
#pragma unroll
          for (int c = 0; c < 16; ++c) e[c] += __shfl_xor_sync(0xffffffffu, e[c], off);
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) x[c] = x[c] - m[c] - fast_lg2(e[c]) * kLn2;
      }
      if (mine) {
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int pos = b * 16 + c;
          if (pos < p.P) dst[static_cast<size_t>(pos) * nrows + row] = x[c];   // 32 lanes -> 128 contiguous bytes
        }
      }
    }
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    const uint32_t lead = elect_one();
    uint32_t stage = 0, phase = 0, issued = 0;
    bool ok = true;
    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
    for (int tile = tile_begin; tile < tile_end && ok; ++tile) {
      const DecodeTile t = decode_tile(p, tile);
      const CUtensorMap* map = t.is_sum ? &p.tm_sum : (t.second ? &p.tm_emit2 : &p.tm_emit);
      const int row = t.index * t.rows;
      const uint32_t bytes = (t.rows + p.Ppad) * (kBlockK * 2);    // out-of-range rows are zero-filled and counted
      for (int k = kb0 * kBlockK; k < kb1 * kBlockK; k += kBlockK) {
        if (!bounded_wait_all(empty0 + 8 * stage, phase ^ 1u, ctl, p)) { ok = false; break; }
        const uint32_t full = full0 + 8 * stage, dst = tiles_addr + stage * p.stage_bytes;
        mbar_arrive_expect_tx(lead, full, bytes);
        tma_load_2d(lead, dst, map, full, k, row);
        tma_load_2d(lead, dst + hidden_off, &p.tm_h, full, k, 0);
        ++issued;
        if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
      }
    }
    // no copy may still be in flight when the CTA goes away (they have all landed unless some warp gave up)
    for (uint32_t s = 0; s < static_cast<uint32_t>(p.stages) && s < issued; ++s)
      drain_wait(full0 + 8 * s, ((issued - 1 - s) / p.stages) & 1u);
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer: D[row, p] = W[row, :] . h[p, :]
    const uint32_t lead = elect_one();
    uint32_t stage = 0, phase = 0, use = 0;
    bool ok = tile_begin >= tile_end || first_wait(smem_u32(&ctl->full[0]), ctl, p);
    const uint32_t idesc = umma_idesc_bf16(kBlockM, p.Ppad);
    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
    const uint32_t stage_step = p.stage_bytes >> 4;             // descriptors step in 16-byte units
    const uint64_t a_desc0 = umma_smem_desc_sw128(tiles_addr), b_desc0 = umma_smem_desc_sw128(tiles_addr + hidden_off);
    for (int tile = tile_begin; tile < tile_end && ok; ++tile, ++use) {
      const uint32_t slot = use & 1u;
      if (!bounded_wait_all(smem_u32(&ctl->tempty[slot]), ((use >> 1) & 1u) ^ 1u, ctl, p)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + slot * p.tile_stride;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!bounded_wait_all(full0 + 8 * stage, phase, ctl, p)) { ok = false; break; }
        tc_fence_after();
        const uint64_t a_desc = a_desc0 + stage * stage_step, b_desc = b_desc0 + stage * stage_step;
#pragma unroll
        for (int kk = 0; kk < kBlockK / 16; ++kk)
          umma_bf16(lead, d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, (kb != kb0 || kk != 0) ? 1u : 0u);
        umma_commit(lead, empty0 + 8 * stage);
        if (++stage == static_cast<uint32_t>(p.stages)) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      umma_commit(lead, smem_u32(&ctl->tfull[slot]));
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue: warp q owns lanes 32q .. 32q+31
    uint32_t use = 0;
    bool ok = true;
    for (int tile = tile_begin; tile < tile_end && ok; ++tile, ++use) {
      const uint32_t slot = use & 1u;
      if (!bounded_wait_warp(smem_u32(&ctl->tfull[slot]), (use >> 1) & 1u, ctl, p.status, lane)) {
        ok = false;
        break;
      }
      tc_fence_after();
      if (p.ksplit == 1) {
        finish_tile(tile, slot * p.tile_stride, nullptr);
      } else if (rank > 0) {
        // the cluster's one tile: the accumulators go to its first CTA
        const uint32_t dst0 = cluster_map_shared(smem_u32(exchange), 0) + (quarter * 32 + lane) * 16;
        for (int b = 0; b < (p.P + 15) / 16; ++b) {
          float x[16];
          tmem_ld16(lane_base + b * 16, x);
          const uint32_t dst = dst0 + ((rank - 1) * (p.Ppad / 4) + b * 4) * (kBlockM * 16);
#pragma unroll
          for (int c = 0; c < 4; ++c) st_cluster_v4(dst + c * (kBlockM * 16), x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctl->tempty[slot]));
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) drain_after_abort<1>(ctl, true);
  if (p.ksplit > 1) {
    cluster_sync_all();       // the other CTAs' accumulators have arrived
    if (rank == 0 && warp >= 2) {
      tc_fence_after();
      if (tile_begin < tile_end) finish_tile(tile_begin, 0, reinterpret_cast<const float4*>(exchange));
      tc_fence_before();
    }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---------------------------------------------------------------- per-(position, slot) sampling
// Inclusive warp scan (sum).
__device__ __forceinline__ float warp_scan_incl(float x, int lane) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float y = __shfl_up_sync(kFull, x, off);
    if (lane >= off) x += y;
  }
  return x;
}
// Categorical draw over r <= 32 log-probabilities held one per lane (lanes >= r hold anything): the smallest
// j with u < p_0 + ... + p_j, else r - 1. All lanes return the same index.
__device__ __forceinline__ int warp_inv_cdf_logp(float logp, int r, float u, int lane) {
  const float pr = lane < r ? expf(logp) : 0.f;
  const float cum = warp_scan_incl(pr, lane);
  const unsigned hit = __ballot_sync(kFull, lane < r && u < cum);
  return hit ? __ffs(hit) - 1 : r - 1;
}

// The tables of `rows` rows of r <= 32 static transition logits x, one warp per row: their log-softmax, and what a head keeps besides
// it (prob and cdf; NULL: a call without a head), the probabilities (the circuit's recursion) and their running sums, with which a draw
// is one comparison per lane and a ballot, and yields what warp_inv_cdf_logp yields. The sum runs in index order. (mtpc_update_parameters on n = 8,
// r = 8: 6.8 us as two kernels, one of them with a thread per row; 4.6 before there were tables to keep.)
__global__ void __launch_bounds__(256) static_tables_kernel(const float* __restrict__ x, float* __restrict__ logp,
                                                            float* __restrict__ prob, float* __restrict__ cdf, int rows, int r) {
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= rows) return;
  const float mine = lane < r ? x[static_cast<size_t>(row) * r + lane] : -CUDART_INF_F;
  float m = mine;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, off));
  const float e = expf(mine - m);
  float s = 0.f;
  for (int j = 0; j < r; ++j) s += __shfl_sync(kFull, e, j);
  const float lp = mine - (m + logf(s));
  if (lane < r) logp[static_cast<size_t>(row) * r + lane] = lp;
  if (prob == nullptr) return;
  const float cum = warp_scan_incl(lane < r ? expf(lp) : 0.f, lane);
  if (lane < r) {
    prob[static_cast<size_t>(row) * r + lane] = __expf(lp);
    cdf[static_cast<size_t>(row) * r + lane] = cum;
  }
}
__device__ __forceinline__ int warp_inv_cdf(float cum, int r, float u, int lane) {
  const unsigned hit = __ballot_sync(kFull, lane < r && u < cum);
  return hit ? __ffs(hit) - 1 : r - 1;
}

// The same draw over the softmax of r <= 128 unnormalised logits x[0..r): lane l owns the consecutive indices
// [l * per, (l + 1) * per), per = ceil(r / 32) <= 4; u * total < running sum, index order, no division.
__device__ __forceinline__ int warp_inv_cdf_logits_wide(const float* __restrict__ x, int r, float u, int lane) {
  const int per = (r + 31) / 32;
  const int k0 = lane * per;
  float xv[4];
  float m = -CUDART_INF_F;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    xv[q] = (q < per && k0 + q < r) ? x[k0 + q] : -CUDART_INF_F;
    m = fmaxf(m, xv[q]);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, off));
  float part = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    xv[q] = __expf(xv[q] - m);       // padding: exp(-inf) = 0
    part += xv[q];
  }
  const float incl = warp_scan_incl(part, lane);
  const float total = __shfl_sync(kFull, incl, 31);
  const float thr = u * total;
  const unsigned hit = __ballot_sync(kFull, thr < incl);
  if (!hit) return r - 1;
  const int src = __ffs(hit) - 1;
  const float before = __shfl_up_sync(kFull, incl, 1);
  int found = -1;
  if (lane == src) {
    float cum = lane == 0 ? 0.f : before;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (found < 0 && q < per && k0 + q < r) {
        cum += xv[q];
        if (thr < cum) found = k0 + q;
      }
    if (found < 0) found = min(k0 + per, r) - 1;
  }
  return __shfl_sync(kFull, found, src);
}

// Tables the latent draws of slot i walk through (Algorithm 1 at the sum units), in the order they are used.
// CP: none. HMM: the transitions into steps 1..i. BTree: the nodes on the path from the root (exclusive) down to
// the deepest internal node above token i.
__device__ __forceinline__ int slot_chain_length(int family, int n, int i) {
  if (family == 1) return i;
  if (family == 2) return 31 - __clz(n / 2 + (i >> 1));   // depth of the owner node n/2 - 1 + i/2 in heap order
  return 0;
}
// Global address of table `step` (0-based) of the chain. lw: this position's log omega; hmm: this position's
// (or the static) transition tables [n-1, r, r].
__device__ __forceinline__ const float* slot_chain_table(int family, const float* lw, const float* hmm, int n, int r,
                                                         int i, int step) {
  if (family == 1) return hmm + static_cast<size_t>(step) * r * r;
  const int code = n / 2 + (i >> 1);                       // owner + 1
  const int depth = 31 - __clz(code);
  const int node = (code >> (depth - 1 - step)) - 1;       // path node at level step + 1
  return lw + r + static_cast<size_t>(node - 1) * r * r;
}

constexpr int kSlotMaxPerLane = 16;   // symbols a lane holds at a time: 512 per warp pass
// Sum of exp(x[b] - m) over the symbols [c0, c0 + 512) that exist (b < vv); lane l takes l, l + 32, ... of the chunk.
__device__ __forceinline__ float warp_chunk_sum(const float* __restrict__ x, int c0, int vv, float m, int lane) {
  float xv[kSlotMaxPerLane];
#pragma unroll
  for (int q = 0; q < kSlotMaxPerLane; ++q) {
    const int b = c0 + lane + 32 * q;
    xv[q] = b < vv ? x[b] : -CUDART_INF_F;
  }
  float s = 0.f;
#pragma unroll
  for (int q = 0; q < kSlotMaxPerLane; ++q) s += __expf(xv[q] - m);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(kFull, s, off);
  return s;
}
// e[q] = p[q] for q < per (the widest loads that per allows; p is aligned for them), `fill` from p + limit on and in the rest of e.
template <int NQ>
__device__ __forceinline__ void load_run(const float* p, int per, int limit, float fill, float (&e)[NQ]) {
#pragma unroll
  for (int q = 0; q < NQ; ++q) e[q] = fill;
  if (per % 4 == 0) {
#pragma unroll
    for (int q = 0; q + 3 < NQ; q += 4)
      if (q < per && q < limit) {
        const float4 x = *reinterpret_cast<const float4*>(p + q);
        e[q] = x.x; e[q + 1] = x.y; e[q + 2] = x.z; e[q + 3] = x.w;
      }
  } else if (per % 2 == 0) {
#pragma unroll
    for (int q = 0; q + 1 < NQ; q += 2)
      if (q < per && q < limit) {
        const float2 x = *reinterpret_cast<const float2*>(p + q);
        e[q] = x.x; e[q + 1] = x.y;
      }
  } else {
#pragma unroll
    for (int q = 0; q < NQ; ++q)
      if (q < per && q < limit) e[q] = p[q];
  }
}
// Inverse CDF over weights held by a warp, lane l those of the consecutive symbols [b0, b0 + per), b0 = c0 + l per (0 beyond
// end and beyond per). The threshold is thr * (the weights' total) when `relative`, else thr itself. Returns the smallest symbol
// whose running sum exceeds it; the last one below end if rounding leaves none. All lanes return the same value.
template <int NQ>   // per <= NQ <= kSlotMaxPerLane: the steps that are unrolled
__device__ __forceinline__ int warp_inv_cdf_weights(const float (&ev)[NQ], int c0, int per, int end, float thr, bool relative, int lane) {
  float part = 0.f;
#pragma unroll
  for (int q = 0; q < NQ; ++q) part += ev[q];
  const float incl = warp_scan_incl(part, lane);
  if (relative) thr *= __shfl_sync(kFull, incl, 31);
  const unsigned hit = __ballot_sync(kFull, thr < incl);
  const float before = __shfl_up_sync(kFull, incl, 1);
  // the running sums never fall: the number of a lane's that the threshold is not below is the place of the first that it is
  float cum = lane == 0 ? 0.f : before;
  int passed = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    cum += ev[q];
    passed += thr < cum ? 0 : 1;
  }
  const int b0 = c0 + lane * per;
  const int found = min(b0 + min(passed, per), min(b0 + per, end) - 1);    // the lane's total passed the threshold: its last symbol
  return hit ? __shfl_sync(kFull, found, __ffs(hit) - 1) : min(c0 + 32 * per, end) - 1;
}
// The same over the 32 * per symbols starting at c0 of a unit of v, vv of them real, on the weights exp(x[b] - m).
template <int NQ>
__device__ __forceinline__ int warp_inv_cdf_chunk(const float* __restrict__ x, int c0, int per, int v, int vv, float m, float thr,
                                                  bool relative, int lane) {
  const int b0 = c0 + lane * per;
  float ev[NQ];
  load_run<NQ>(x + b0, per, v - b0, -CUDART_INF_F, ev);
#pragma unroll
  for (int q = 0; q < NQ; ++q) ev[q] = b0 + q < vv ? fast_ex2((ev[q] - m) * kLog2e) : 0.f;
  return warp_inv_cdf_weights<NQ>(ev, c0, per, vv, thr, relative, lane);
}

// hmm: HMM transition tables [n-1, r, r]; position p reads them at hmm + p * hmm_stride. Stride 0: one static set for all
// positions, as running sums of probabilities (static_tables_kernel); stride sum_rows with hmm = log omega + r: contextual
// tables (App. H) of log-probabilities.
// grid = (n, P), 16 warps. Shared memory: 2 * r floats (max and log-sum-exp of each unit of the slot); when weights_in_smem, the
// units' weights exp(logit - max), which the byte draws then read instead of the logits; when tables_in_smem, the chain's tables
// (slot_chain_length * r * r floats), fetched by cp.async while the log-sum-exps are computed, static ones while the kernel still
// waits for the one before it.
// The log-sum-exps also go to unit_lse_out [P, n, r], so that later calls can turn the retained logits into log phi.
// Bound by trips to memory that wait on one another, and by instructions where a device full of CTAs shares them: so a warp requests
// its first unit's logits, its first window's uniforms and the root weights before anything else, and the next unit's logits
// before it works on this one's. Loops that run once or twice stay rolled: at
// these durations fetching instructions counts. Time after the weight pass, per slot stage: mixture n = 16, r = 16, v = 320, 64
// positions of 16 windows 22 -> 15.5 us; HMM n = 16, r = 32, 8 positions 16.2 -> 9.8; tree n = 8, r = 32, 27 positions 10.4 -> 8.
// WIDE: vocabularies of more than 512 symbols (a separate build: the narrow one keeps a unit's logits in registers).
// CTAS: of them that an SM's registers hold. Two leave a warp everything in flight that it asks for; of more CTAs than the device then holds
// three an SM take less time, a few values spilled (draft + acceptance, two / three, us: mixture 16 x 16 x 320, 64 positions of 16 windows
// 137.1 / 134.4, 128 positions of one window, d = 1024, 71.9 / 67.4; tree 16 x 32 x 256, 128 positions 207.4 / 200.6), fewer CTAs more
// (HMM 16 x 16 x 256, d = 512, 1 position of 16 windows 32.2 / 33.7, tree 8 x 32 x 256, 27 positions 88.4 / 89.6).
template <bool WIDE, int NQ, int CTAS>   // NQ: batches of 32 symbols of a unit that are unrolled (v <= 32 NQ; WIDE: 16)
__global__ void __launch_bounds__(kSlotThreads, CTAS) draft_slot_kernel(
    int family, const float* __restrict__ logits, const float* __restrict__ logw, const float* __restrict__ hmm_tables,
    const float* __restrict__ uniforms, int* __restrict__ out_bytes, float* __restrict__ G,
    float* __restrict__ unit_lse_out, unsigned* status, unsigned* work_counter, int wpp, int n, int r, int v, int vv,
    int sum_rows, int hmm_stride, int tables_in_smem, int weights_in_smem) {
  extern __shared__ __align__(16) float sm[];
  grid_launch_dependents();
  const int per = (v + 31) / 32;             // consecutive symbols per lane in the CDF scan (<= NQ, narrow)
  float* weights = sm + ((2 * r + 3) & ~3);  // [r][32 per]
  float* tabs = weights + (weights_in_smem ? r * 32 * per : 0);
  const int chain = slot_chain_length(family, n, blockIdx.x);
  const bool early = tables_in_smem && family == 1 && hmm_stride == 0;      // static tables, complete before the call's first kernel lets this in
  if (early) fetch_floats(tabs, hmm_tables, chain * r * r, kSlotThreads);
  if (threadIdx.x < wpp) prefetch_l2(uniforms + (static_cast<size_t>(blockIdx.y) * wpp + threadIdx.x) * 2 * n);
  grid_dependency_wait();     // the logits and log omega come from the kernel before this one
  if (work_counter != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0)
    *work_counter = 0;        // the circuit kernel that follows hands out its windows through this counter
  float* unit_max = sm;
  float* unit_lse = sm + r;
  const int i = blockIdx.x;
  const int pos = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nwarps = kSlotThreads / 32;
  const int rr = r * r;
  const float* row = logits + (static_cast<size_t>(pos) * n + i) * r * v;   // [r, v] logits of this slot
  const float* lw = logw + static_cast<size_t>(pos) * sum_rows;
  const float* hmm = hmm_tables + static_cast<size_t>(pos) * hmm_stride;
  const int nlat = (family == 0) ? 1 : (family == 1 ? n : n - 1);           // latent draws of a window (n <= 64)

  constexpr int kVec = (NQ + 3) / 4;
  auto load_unit = [&](int k, float4 (&xv)[kVec]) {      // lane l: symbols [4 l, 4 l + 4), [128 + 4 l, ..), ..
#pragma unroll
    for (int q = 0; q < kVec; ++q) {
      const int b = 4 * (lane + 32 * q);
      xv[q] = b < v ? *reinterpret_cast<const float4*>(row + k * v + b)
                    : make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
    }
  };
  struct Draws { float u0, u1, byte; };                  // lane l: the window's latent uniforms l and 32 + l; its byte's
  auto load_draws = [&](int j) {
    const float* u = uniforms + (pos * wpp + j) * 2 * n;           // (at most 128 positions of 64 windows: 32 bits do)
    return Draws{lane < nlat ? u[lane] : 0.f, 32 + lane < nlat ? u[32 + lane] : 0.f, u[n + i]};
  };
  float4 next_unit[kVec];
  Draws next_draws{};
  if (!WIDE && warp < r) load_unit(warp, next_unit);
  if (warp < wpp) next_draws = load_draws(warp);
  const float root_logp = r <= 32 && lane < r ? lw[lane] : 0.f;

  if (tables_in_smem && !early) {
#pragma unroll 1
    for (int step = 0; step < chain; ++step)
      fetch_floats(tabs + step * rr, slot_chain_table(family, lw, hmm, n, r, i, step), rr, kSlotThreads);
  }
  if (tables_in_smem) cp_async_commit();

  // ---- log-sum-exp of every input unit of the slot (wide vocabularies: 512 symbols at a time, merged online)
  constexpr int kChunk = kSlotMaxPerLane * 32;
  for (int k = warp; k < r; k += nwarps) {
    float m = -CUDART_INF_F, s = 0.f;
    if (!WIDE) {
      float4 xv[kVec];
#pragma unroll
      for (int q = 0; q < kVec; ++q) xv[q] = next_unit[q];
      if (k + nwarps < r) load_unit(k + nwarps, next_unit);
#pragma unroll
      for (int q = 0; q < kVec; ++q) {
        const int b = 4 * (lane + 32 * q);
        if (b + 3 >= vv) {                       // [vv, v): padding symbols
          if (b >= vv) xv[q].x = -CUDART_INF_F;
          if (b + 1 >= vv) xv[q].y = -CUDART_INF_F;
          if (b + 2 >= vv) xv[q].z = -CUDART_INF_F;
          xv[q].w = -CUDART_INF_F;
        }
        m = fmaxf(fmaxf(m, fmaxf(xv[q].x, xv[q].y)), fmaxf(xv[q].z, xv[q].w));
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, off));
#pragma unroll
      for (int q = 0; q < kVec; ++q) {
        const int b = 4 * (lane + 32 * q);
        const float4 e = make_float4(fast_ex2((xv[q].x - m) * kLog2e), fast_ex2((xv[q].y - m) * kLog2e),
                                     fast_ex2((xv[q].z - m) * kLog2e), fast_ex2((xv[q].w - m) * kLog2e));
        s += (e.x + e.y) + (e.z + e.w);          // padding: 2^-inf = 0
        if (weights_in_smem && b < 32 * per) *reinterpret_cast<float4*>(weights + k * 32 * per + b) = e;
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(kFull, s, off);
    }
    for (int c0 = 0; WIDE && c0 < v; c0 += kChunk) {
      const float* x = row + static_cast<size_t>(k) * v;
      float xv[NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int b = c0 + lane + 32 * q;
        xv[q] = b < vv ? x[b] : -CUDART_INF_F;
      }
      float cm = xv[0];
#pragma unroll
      for (int q = 1; q < NQ; ++q) cm = fmaxf(cm, xv[q]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) cm = fmaxf(cm, __shfl_xor_sync(kFull, cm, off));
      const float mn = fmaxf(m, cm);           // finite from the first chunk on (symbol 0 always exists)
      float cs = 0.f;
#pragma unroll
      for (int q = 0; q < NQ; ++q) cs += __expf(xv[q] - mn);   // padding: exp(-inf) = 0
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) cs += __shfl_xor_sync(kFull, cs, off);
      s = s * __expf(m - mn) + cs;             // first chunk: 0 * exp(-inf) = 0
      m = mn;
    }
    if (lane == 0) {
      unit_max[k] = m;
      unit_lse[k] = m + __logf(s);
      unit_lse_out[(pos * n + i) * r + k] = unit_lse[k];   // kept for the acceptance stage
    }
  }
  const float root_cum = warp_scan_incl(lane < r && r <= 32 ? expf(root_logp) : 0.f, lane);
  if (tables_in_smem) cp_async_wait<0>();
  __syncthreads();

  for (int j = warp; j < wpp; j += nwarps) {
    const int slot = (pos * wpp + j) * n + i;
    const Draws d = next_draws;
    if (j + nwarps < wpp) next_draws = load_draws(j + nwarps);
    auto uniform = [&](int c) { return __shfl_sync(kFull, c < 32 ? d.u0 : d.u1, c & 31); };
    // ---- latent draws down to the unit that owns slot i; every uniform the window's latent draws use is checked
    const bool bad = __any_sync(kFull, !(d.u0 >= 0.f && d.u0 < 1.f) || !(d.u1 >= 0.f && d.u1 < 1.f) || !(d.byte >= 0.f && d.byte < 1.f));
    int byte = -1;
    if (bad) {
      if (lane == 0) atomicOr(status, 2u);
    } else {
      int z = r > 32 ? warp_inv_cdf_logits_wide(lw, r, uniform(0), lane)     // CP only; the mixture logits are unnormalised
                     : warp_inv_cdf(root_cum, r, uniform(0), lane);
      if (family == 1) {
        for (int st = 0; st < chain; ++st) {
          const float t = lane >= r ? 0.f : tables_in_smem ? tabs[st * rr + z * r + lane] : hmm[st * rr + z * r + lane];
          z = hmm_stride == 0 ? warp_inv_cdf(t, r, uniform(st + 1), lane) : warp_inv_cdf_logp(t, r, uniform(st + 1), lane);
        }
      } else if (family == 2) {
        const int code = n / 2 + (i >> 1);
        for (int st = 0; st < chain; ++st) {
          const int node = (code >> (chain - 1 - st)) - 1;
          const float t = lane >= r ? 0.f : tables_in_smem ? tabs[st * rr + z * r + lane] : lw[r + (node - 1) * rr + z * r + lane];
          z = warp_inv_cdf_logp(t, r, uniform(node), lane);
        }
      }
      const float* x = row + z * v;
      const float m = unit_max[z];
      if (!WIDE && weights_in_smem) {
        // ---- inverse CDF over the v bytes of unit z: lane l owns bytes [l*per, (l+1)*per)
        float ev[NQ];
        load_run<NQ>(weights + z * 32 * per + lane * per, per, per, 0.f, ev);
        byte = warp_inv_cdf_weights<NQ>(ev, 0, per, vv, d.byte, true, lane);
      } else if (!WIDE) {
        byte = warp_inv_cdf_chunk<NQ>(x, 0, per, v, vv, m, d.byte, true, lane);
      } else {
        // ---- wide vocabulary: 512 symbols at a time. First the total (chunk sums in fp32, added up in fp64), then
        // the chunk the threshold u * total falls into, then the draw inside that chunk.
        double total = 0.0;
        for (int c0 = 0; c0 < v; c0 += kChunk) total += static_cast<double>(warp_chunk_sum(x, c0, vv, m, lane));
        const double thr = static_cast<double>(d.byte) * total;
        double before = 0.0;
        byte = vv - 1;                           // rounding may leave no index: the last one
        for (int c0 = 0; c0 < v; c0 += kChunk) {
          const float cs = warp_chunk_sum(x, c0, vv, m, lane);
          if (thr < before + static_cast<double>(cs)) {
            byte = warp_inv_cdf_chunk<kSlotMaxPerLane>(x, c0, kSlotMaxPerLane, v, vv, m, static_cast<float>(thr - before), false, lane);
            break;
          }
          before += static_cast<double>(cs);
        }
      }
    }
    if (lane == 0) out_bytes[slot] = byte;
    // evidence of the drafted byte under every input unit of the slot; a draw that was refused (byte -1) has none:
    // NaN, so that the window's log-prob comes out as NaN rather than as the joint of its other bytes
    for (int k = lane; k < r; k += 32)
      G[slot * r + k] = byte < 0 ? CUDART_NAN_F : row[k * v + byte] - unit_lse[k];
  }
}

// ---------------------------------------------------------------- draft of many positions
// Latent draws (Algorithm 1 at the sum units), one warp per window, lane = latent value. Writes unit_sel[w, i] = the input unit
// chosen for token i and presets out_bytes to -1; a window with a uniform outside [0,1) gets -1 throughout. (One thread per
// window walking r entries per draw took 57 us for 4096 windows of a 16-leaf tree, 15 dependent draws each; this 14 us.)
constexpr int kLatentWarps = 4;
__global__ void __launch_bounds__(32 * kLatentWarps) latent_sample_kernel(
    int family, const float* __restrict__ logw, const float* __restrict__ logA, const float* __restrict__ uniforms,
    int* __restrict__ unit_sel, int* __restrict__ out_bytes, unsigned* status, int W, int wpp, int n, int r, int sum_rows,
    int logA_stride) {
  grid_dependency_wait();
  const int w = blockIdx.x * kLatentWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= W) return;
  const float* lw = logw + static_cast<size_t>(w / wpp) * sum_rows;
  const float* u = uniforms + static_cast<size_t>(w) * 2 * n;
  const int nlat = (family == 0) ? 1 : (family == 1 ? n : n - 1);
  // The drawn values stay in registers, lane l those of the latents l and 32 + l, and are read by shuffles.
  int lo = 0, hi = 0;
  auto value = [&](int j) {                        // of latent j, which may differ from lane to lane
    const int a = __shfl_sync(kFull, lo, j & 31), b = __shfl_sync(kFull, hi, j & 31);
    return j < 32 ? a : b;
  };
  bool bad = false;
  for (int c = lane; c < nlat; c += 32) bad |= !(u[c] >= 0.f && u[c] < 1.f);
  bad = __any_sync(kFull, bad);
  if (bad) {
    if (lane == 0) atomicOr(status, 2u);
  } else {
    int prev = r > 32 ? warp_inv_cdf_logits_wide(lw, r, u[0], lane) : warp_inv_cdf_logp(lane < r ? lw[lane] : 0.f, r, u[0], lane);
    if (lane == 0) lo = prev;
    for (int j = 1; j < nlat; ++j) {
      const int parent = family == 1 ? prev : value((j - 1) >> 1);
      const float* tab = family == 1 ? logA + static_cast<size_t>(w / wpp) * logA_stride + (static_cast<size_t>(j - 1) * r + parent) * r
                                     : lw + r + (static_cast<size_t>(j - 1) * r + parent) * r;
      prev = warp_inv_cdf_logp(lane < r ? tab[lane] : 0.f, r, u[j], lane);
      if (lane == (j & 31)) (j < 32 ? lo : hi) = prev;
    }
  }
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    const int z = value(i >= n || family == 0 ? 0 : family == 1 ? i : n / 2 - 1 + (i >> 1));
    if (i < n) {
      unit_sel[static_cast<size_t>(w) * n + i] = bad ? -1 : z;
      out_bytes[static_cast<size_t>(w) * n + i] = -1;
    }
  }
  grid_launch_dependents();
}

// Byte draws of a draft whose logits were kept by the projection kernel: one warp per (window, slot) draws the byte by inverse
// CDF from the logits of the unit the latent draw selected and gathers its evidence G[w, i, k] = log phi_k(byte) from the
// slot's r units. 4 v + 36 r bytes per pair; bound by three dependent trips to memory. (The projection of the drafted bytes'
// evidence, and a sampling projection on hidden states sorted by unit before it, are what keeping the logits replaces: 2232 +
// 217 + 74 us at 4096 positions of the n = 16, r = 32, v = 256 tree, against 206 us more for the projection that keeps them
// and 67 us here.)
template <bool WIDE, int NQ>   // units of more than 512 symbols: 512 at a time, as in draft_slot_kernel; else v <= 32 NQ
__global__ void __launch_bounds__(256) draft_pick_kernel(const float* __restrict__ logits, const float* __restrict__ unit_lse,
                                                         const int* __restrict__ unit_sel, const float* __restrict__ uniforms,
                                                         int* __restrict__ out_bytes, float* __restrict__ G, unsigned* status,
                                                         int pairs, int wpp, int n, int r, int v, int vv) {
  grid_dependency_wait();
  const int e = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (e >= pairs) return;
  const int w = e / n, i = e - w * n;
  const size_t unit0 = (static_cast<size_t>(w / wpp) * n + i) * r;
  const float* row = logits + unit0 * v;                   // [r, v] logits of this slot
  const int z = unit_sel[e];
  const float ub = uniforms[static_cast<size_t>(w) * 2 * n + n + i];
  int byte = -1;
  if (z >= 0) {
    if (!(ub >= 0.f && ub < 1.f)) {
      if (lane == 0) atomicOr(status, 2u);
    } else {
      const float* x = row + static_cast<size_t>(z) * v;
      const float m = unit_lse[unit0 + z];                 // the weights are then probabilities
      if (!WIDE) {
        byte = warp_inv_cdf_chunk<NQ>(x, 0, (v + 31) / 32, v, vv, m, ub, true, lane);
      } else {
        constexpr int kChunk = kSlotMaxPerLane * 32;
        double total = 0.0;
        for (int c0 = 0; c0 < v; c0 += kChunk) total += static_cast<double>(warp_chunk_sum(x, c0, vv, m, lane));
        const double thr = static_cast<double>(ub) * total;
        double before = 0.0;
        byte = vv - 1;                                     // rounding may leave no index: the last one
        for (int c0 = 0; c0 < v; c0 += kChunk) {
          const float cs = warp_chunk_sum(x, c0, vv, m, lane);
          if (thr < before + static_cast<double>(cs)) {
            byte = warp_inv_cdf_chunk<kSlotMaxPerLane>(x, c0, kSlotMaxPerLane, v, vv, m, static_cast<float>(thr - before), false, lane);
            break;
          }
          before += static_cast<double>(cs);
        }
      }
    }
  }
  if (lane == 0) out_bytes[e] = byte;
  for (int k = lane; k < r; k += 32)
    G[static_cast<size_t>(e) * r + k] = byte < 0 ? CUDART_NAN_F : row[static_cast<size_t>(k) * v + byte] - unit_lse[unit0 + k];
  grid_launch_dependents();
}

// ---------------------------------------------------------------- acceptance stage (Algorithm 3)
constexpr int kAcceptMaxThreads = 512;

// Shared memory of one CTA (= one window) of spec_accept_kernel, in floats: the residual weights of the v bytes; the log-weight
// of every input unit of the slot (r), whose space then holds the warps' partial sums.
__host__ __device__ inline size_t accept_smem_floats(int r, int v) { return static_cast<size_t>(v) + (r > 16 ? r : 16); }
// One thread per byte up to 512 of them.
inline int accept_threads(int v) { return v >= kAcceptMaxThreads ? kAcceptMaxThreads : (v + 31) / 32 * 32; }

// One CTA per drafted window w (position p = w / wpp). Inputs: the draft's bytes and prefix log-marginals, the target
// model's conditionals along the draft, one uniform per test plus one for the last byte; the logits and per-unit
// log-sum-exps of the slots, and the slot messages msg [W, n, r] the circuit kernels left in the workspace.
//   1. s = 0; while s < n: the draft's conditional of byte s is q_s = exp(prefix[s] - prefix[s-1]) (prefix[-1] = 0);
//      stop if alpha_s > p(x_s) / q_s, tested as alpha_s * q_s > p(x_s); else s += 1.
//   2. s == n: the extra byte is drawn from the target row n.
//      s <  n: it is drawn from max(0, p(.) - q(. | x_0..x_{s-1})) / Z. The circuit's conditional of slot s is a mixture of the
//      slot's r input units under softmax(msg[w, s, :]): q(b | ..) = sum_k exp(logit_k[b] + msg_k - LSE(msg) - lse_k).
//   Both draws are inverse-CDF on unnormalised weights (u * total < running sum, index order, no division).
// The call is a chain of dependent L2 round trips: every warp runs the tests (one ballot, no broadcast through shared
// memory), a thread then has all the logits of its byte in flight, and the scan over the bytes is one warp scan plus the
// warps' totals. With the recursions gone from it (they were one warp's serial chain through the tables) and launched as a
// programmatic dependent the kernel went from 59 to 6 us at HMM n = 16, 128 windows; 12 to 5 us for one mixture window; 569 to
// 49 us for 4096 tree windows of n = 16. row_of != NULL (logits recomputed after a long draft): `logits` [rows, r v] and `unit_lse` [rows, r] hold only the
// slot of each rejected window's first rejected byte, at row row_of[w].
// AHEAD: a thread asks for its byte's target probability and the logits of 32 units before the weights are formed, which takes two
// trips to memory out of the chain and twice the registers. 128 windows of an HMM, r = 32: 9.7 -> 6.8 us behind the circuit; 108 of a tree
// 7.5 -> 6.7; but 1024 windows of a mixture 11.7 -> 15.0, so only while every window has an SM to itself.
template <bool AHEAD>
__global__ void __launch_bounds__(kAcceptMaxThreads) spec_accept_kernel(
    const float* __restrict__ logits, const float* __restrict__ unit_lse, const float* __restrict__ msg,
    const int* __restrict__ bytes, const float* __restrict__ prefix, const float* __restrict__ target,
    const float* __restrict__ uniforms, int* __restrict__ out_accepted, int* __restrict__ out_next, unsigned* status, int W,
    int wpp, int n, int r, int v, int vv, const int* __restrict__ row_of) {
  extern __shared__ __align__(16) float sm[];
  grid_launch_dependents();
  // The window's rows of the target model, on their way to L2 meanwhile (another 0.3 to 1.1 us a step). All n + 1 of them, since which values and which
  // row the stage reads depends on the draft; beyond 32 KB that is more than it is worth (asked for / not, us: 32 windows of a mixture n = 16, v = 512 37.1 / 35.8,
  // v = 1024 62.7 / 61.6; 128 of n = 32, v = 320 42.7 / 42.5; of a tree n = 32, v = 512 109.0 / 108.7; only 4 of n = 64, v = 320 71.0 / 71.5).
  if (AHEAD) {
    const size_t row = static_cast<size_t>(n + 1) * v * sizeof(float);
    const char* rows = reinterpret_cast<const char*>(target) + blockIdx.x * row;
    if (row <= 32768)
      for (int at = threadIdx.x * 128; at < static_cast<int>(row); at += blockDim.x * 128) prefetch_l2(rows + at);
    if (threadIdx.x == 0) prefetch_l2(uniforms + static_cast<size_t>(blockIdx.x) * (n + 1));
  }
  grid_dependency_wait();   // the draft's outputs come from the kernels before this one
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int w = blockIdx.x;
  float* mres = sm;                                      // [v]
  float* cw = sm + v;                                    // [r], then the warps' totals
  const int pos = w / wpp;
  const int* x = bytes + static_cast<size_t>(w) * n;
  const float* pre = prefix + static_cast<size_t>(w) * n;
  const float* u = uniforms + static_cast<size_t>(w) * (n + 1);
  const float* tp = target + static_cast<size_t>(w) * (n + 1) * v;
  const float u_last = u[n];
  // ---- 1. acceptance tests: lane i runs the test of byte i; the first rejecting lane ends the accepted run
  bool bad_u = !(u_last >= 0.f && u_last < 1.f), bad_x = false;
  int s = n;
#pragma unroll 1
  for (int base = 0; base < n; base += 32) {
    const int i = base + lane;
    bool rej = false;
    if (i < n) {
      const int xi = x[i];
      const float ui = u[i], now = pre[i], before = i > 0 ? pre[i - 1] : 0.f;
      bad_u |= !(ui >= 0.f && ui < 1.f);
      const bool inside = static_cast<unsigned>(xi) < static_cast<unsigned>(vv);
      bad_x |= !inside;
      rej = inside && ui * __expf(now - before) > tp[static_cast<size_t>(i) * v + xi];
    }
    const unsigned m = __ballot_sync(kFull, rej);
    if (m && s == n) s = base + __ffs(m) - 1;
  }
  bad_u = __any_sync(kFull, bad_u);
  bad_x = __any_sync(kFull, bad_x);
  if (bad_u || bad_x) {                                  // the same for every warp
    if (threadIdx.x == 0) {
      atomicOr(status, bad_u ? 2u : 1u);
      out_accepted[w] = -1;
      out_next[w] = -1;
    }
    return;
  }
  // ---- 2. weights of the v bytes
  const float* trow = tp + static_cast<size_t>(s) * v;
  if (s == n) {
#pragma unroll 1
    for (int b = threadIdx.x; b < v; b += blockDim.x) mres[b] = b < vv ? trow[b] : 0.f;
  } else {
    const size_t lrow = row_of != nullptr ? static_cast<size_t>(row_of[w]) : static_cast<size_t>(pos) * n + s;
    const float* ulse = unit_lse + lrow * r;
    const float* lg = logits + lrow * r * v;             // [r, v] logits of slot s
    float ahead[AHEAD ? 32 : 1], t_ahead;
    if constexpr (AHEAD) {
      const int b = threadIdx.x < vv ? threadIdx.x : 0;
      t_ahead = trow[b];
#pragma unroll
      for (int e = 0; e < 16; ++e) ahead[e] = e < r ? lg[static_cast<size_t>(e) * v + b] : 0.f;
      if (r > 16) {
#pragma unroll
        for (int e = 16; e < 32; ++e) ahead[e] = lg[static_cast<size_t>(e) * v + b];
      }
    }
    if (wib == 0) {
      const float* mw = msg + (static_cast<size_t>(w) * n + s) * r;
      float c[4], l[4];
      float m = -CUDART_INF_F;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = lane + 32 * q;
        c[q] = k < r ? mw[k] : -CUDART_INF_F;
        l[q] = k < r ? ulse[k] : 0.f;
        m = fmaxf(m, c[q]);
      }
      m = warp_max_nan(m);
      float sum = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) sum += __expf(c[q] - m);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(kFull, sum, off);
      const float lse = m + __logf(sum);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (lane + 32 * q < r) cw[lane + 32 * q] = (c[q] - lse - l[q]) * kLog2e;
    }
    __syncthreads();
#pragma unroll 1
    for (int b = threadIdx.x; b < v; b += blockDim.x) {
      float res = 0.f;
      if (b < vv) {
        const bool first = AHEAD && b == threadIdx.x;
        const float t = first ? t_ahead : trow[b];
        float q0 = 0.f, q1 = 0.f;
        int k = 0;
        if constexpr (AHEAD) {
          if (first && r >= 16) {
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              q0 += fast_ex2(fmaf(ahead[e], kLog2e, cw[e]));
              q1 += fast_ex2(fmaf(ahead[e + 1], kLog2e, cw[e + 1]));
            }
            k = 16;
            if (r > 16) {
#pragma unroll
              for (int e = 16; e < 32; e += 2) {
                q0 += fast_ex2(fmaf(ahead[e], kLog2e, cw[e]));
                q1 += fast_ex2(fmaf(ahead[e + 1], kLog2e, cw[e + 1]));
              }
              k = 32;
            }
          } else if (first) {
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (e < r) q0 += fast_ex2(fmaf(ahead[e], kLog2e, cw[e]));
            k = r;
          }
        }
#pragma unroll 1
        for (; k + 16 <= r; k += 16) {                   // sixteen rows' logits in flight, two accumulation chains
          float xv[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) xv[e] = lg[static_cast<size_t>(k + e) * v + b];
#pragma unroll
          for (int e = 0; e < 16; e += 2) {
            q0 += fast_ex2(fmaf(xv[e], kLog2e, cw[k + e]));
            q1 += fast_ex2(fmaf(xv[e + 1], kLog2e, cw[k + e + 1]));
          }
        }
#pragma unroll 1
        for (; k < r; ++k) q0 += fast_ex2(fmaf(lg[static_cast<size_t>(k) * v + b], kLog2e, cw[k]));
        res = fmaxf(0.f, t - (q0 + q1));
      }
      mres[b] = res;                                     // padding symbols carry no mass
    }
  }
  __syncthreads();
  // ---- 3. inverse CDF over mres: thread t owns the bytes [t * per, (t + 1) * per)
  const int per = (v + blockDim.x - 1) / blockDim.x;
  const int b0 = threadIdx.x * per;
  float part = 0.f;
#pragma unroll 1
  for (int q = 0; q < per; ++q)
    if (b0 + q < v) part += mres[b0 + q];
  const float incl = warp_scan_incl(part, lane);
  if (lane == 31) cw[wib] = incl;
  __syncthreads();
  // every warp adds the warps' totals up in the same order, so exactly one of them finds the threshold inside its own run
  float total = 0.f;
#pragma unroll 1
  for (int q = 0; q < warps; ++q) total += cw[q];
  const float thr = u_last * total;
  float before = 0.f;
  int owner = -1;
#pragma unroll 1
  for (int q = 0; q < warps; ++q) {
    const float end = before + cw[q];
    if (thr < end) { owner = q; break; }
    before = end;
  }
  if (owner < 0) {                                       // rounding may leave no index: the last one
    if (threadIdx.x == 0) {
      out_accepted[w] = s;
      out_next[w] = vv - 1;
    }
    return;
  }
  if (wib != owner) return;
  const unsigned some = __ballot_sync(kFull, part > 0.f);
  unsigned hit = __ballot_sync(kFull, part > 0.f && thr < before + incl);
  if (!hit) hit = some ? 1u << (31 - __clz(some)) : 1u << 31;      // the run's last byte with mass
  const int src = __ffs(hit) - 1;
  const float prev = __shfl_up_sync(kFull, incl, 1);
  if (lane == src) {
    float cum = before + (lane == 0 ? 0.f : prev);
    int found = -1, last = min(b0 + per, vv) - 1;
#pragma unroll 1
    for (int q = 0; q < per && found < 0; ++q)
      if (b0 + q < vv && mres[b0 + q] > 0.f) {
        cum += mres[b0 + q];
        last = b0 + q;
        if (thr < cum) found = b0 + q;
      }
    out_accepted[w] = s;
    out_next[w] = found >= 0 ? found : min(last, vv - 1);
  }
}

// The tests of Algorithm 3 alone, one warp per window: first_rejected[w] = s if the draft is rejected at byte s < n, else -1
// (everything accepted, or inputs that the acceptance kernel will refuse). Decides which slot's logits the acceptance
// stage after a many-position draft has to recompute for the window.
__global__ void accept_test_kernel(const int* __restrict__ bytes, const float* __restrict__ prefix,
                                   const float* __restrict__ target, const float* __restrict__ uniforms,
                                   int* __restrict__ first_rejected, int W, int n, int v, int vv) {
  grid_dependency_wait();
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= W) return;
  const int* x = bytes + static_cast<size_t>(w) * n;
  const float* pre = prefix + static_cast<size_t>(w) * n;
  const float* u = uniforms + static_cast<size_t>(w) * (n + 1);
  const float* tp = target + static_cast<size_t>(w) * (n + 1) * v;
  bool bad = false;
  for (int c = lane; c <= n; c += 32) bad |= !(u[c] >= 0.f && u[c] < 1.f);
  for (int c = lane; c < n; c += 32) bad |= static_cast<unsigned>(x[c]) >= static_cast<unsigned>(vv);
  bad = __any_sync(kFull, bad);
  int s = n;
  if (!bad) {
    for (int base = 0; base < n && s == n; base += 32) {
      const int i = base + lane;
      bool rej = false;
      if (i < n) {
        const float q = __expf(pre[i] - (i > 0 ? pre[i - 1] : 0.f));
        rej = u[i] * q > tp[static_cast<size_t>(i) * v + x[i]];
      }
      const unsigned m = __ballot_sync(kFull, rej);
      if (m) s = base + __ffs(m) - 1;
    }
  }
  if (lane == 0) first_rejected[w] = (bad || s == n) ? -1 : s;
  grid_launch_dependents();
}

}  // namespace mtpc
